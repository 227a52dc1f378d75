"""The bounds behind Collision::tame and safe() of the 3-D step (lbm3d.cu): which
cells can send a population, or add to a sum, that leaves the fixed-point range +-8.

A population is s A A A + k'_x B C C + k'_y C B C + k'_z C C B with per axis the
factors below.  Whole factors are bounded here by sampling u, sums by taking each
neighbour at the worst of the kinds of cell that count as tame."""
import itertools

import numpy as np

VEL = list(itertools.product((0, 1, -1), repeat=3))


def factors(u):
    t = 1 / 3 + u * u
    return ({0: 1 - t, 1: (t + u) / 2, -1: (t - u) / 2}, {0: -2 * u, 1: u + 0.5, -1: u - 0.5},
            {0: 1 - u * u, 1: (u * u + u) / 2, -1: (u * u - u) / 2})


def largest(v):
    """Per factor and velocity the largest magnitude over |u| <= v."""
    at = [factors(u) for u in np.linspace(-v, v, 2001)]
    return [{e: max(abs(f[i][e]) for f in at) for e in (0, 1, -1)} for i in range(3)]


def bound(kinds, e):
    """Largest population of velocity e: kinds of cells (|u|, |s|, |k'_i|)."""
    s = k = 0.0
    for v, most, big in kinds:
        A, B, C = largest_of[v]
        s = max(s, most * A[e[0]] * A[e[1]] * A[e[2]])
        k = max(k, big * (B[e[0]] * C[e[1]] * C[e[2]] + C[e[0]] * B[e[1]] * C[e[2]] + C[e[0]] * C[e[1]] * B[e[2]]))
    return s + k


largest_of = {v: largest(v) for v in (0.2, 0.4)}


def test_tame_cells_of_a_field_add_up_in_range():
    kinds = [(0.2, 2.1, 0.3), (0.4, 1.1, 0.15)]
    total = sum(bound(kinds, e) for e in VEL)
    assert 7.5 < total < 7.9
    # and they are safe()
    assert all(safe_bound((v, v, v), m, k) < 7.9 for v, m, k in kinds)


def test_tame_cells_of_a_uniform_velocity_add_up_in_range():
    for u in itertools.product(np.linspace(-0.5, 0.5, 11), repeat=3):
        F = [factors(v) for v in u]
        s = sum(abs(F[0][0][a] * F[1][0][b] * F[2][0][c]) for a, b, c in VEL)
        k = sum(abs(F[0][1][a] * F[1][2][b] * F[2][2][c]) + abs(F[0][2][a] * F[1][1][b] * F[2][2][c])
                + abs(F[0][2][a] * F[1][2][b] * F[2][1][c]) for a, b, c in VEL)
        assert 4.0 * s + 0.4 * k < 7.9
    # and they are safe(), there with constants: |A| <= 2/3, |B| <= 1, |C| <= 1
    assert (2 / 3) ** 3 < 0.3 and 0.3 * 4.0 + 3 * 0.4 < 7.9


def safe_bound(u, most, big):
    """As in Collision::safe(): the largest factor of each axis."""
    v = np.abs(u)
    a = np.maximum(np.maximum(2 / 3, v * v - 2 / 3), (1 / 3 + v * v + v) / 2)
    b = np.maximum(2 * v, v + 0.5)
    c = np.maximum(np.maximum(1, v * v - 1), (v * v + v) / 2)
    return most * a.prod() + big * (b[0] * c[1] * c[2] + c[0] * b[1] * c[2] + c[0] * c[1] * b[2])


def test_safe_cells_send_populations_in_range():
    rng = np.random.default_rng(3)
    for _ in range(2000):
        u = rng.uniform(-2, 2, 3) * rng.choice([0.1, 1.0], 3)
        most, big = rng.uniform(0, 4), rng.uniform(0, 3)
        s, k = most * rng.choice([-1, 1]), big * rng.choice([-1, 1], 3)
        (Ax, Bx, Cx), (Ay, By, Cy), (Az, Bz, Cz) = (factors(v) for v in u)
        largest_sent = max(abs(s * Ax[a] * Ay[b] * Az[c] + k[0] * Bx[a] * Cy[b] * Cz[c] + k[1] * Cx[a] * By[b] * Cz[c]
                               + k[2] * Cx[a] * Cy[b] * Bz[c]) for a, b, c in VEL)
        assert largest_sent <= safe_bound(u, most, big) * (1 + 1e-12)
