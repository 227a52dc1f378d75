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


largest_of = {v: largest(v) for v in (0.2, 0.4, 0.5, 1.0)}


def test_tame_cells_of_a_field_add_up_in_range():
    kinds = [(0.2, 2.1, 0.3), (0.4, 1.1, 0.15)]
    total = sum(bound(kinds, e) for e in VEL)
    assert 7.5 < total < 7.9
    # and they are safe(): 0.3 |s| + 3 max |k'| below 7.9
    assert all(0.3 * m + 3 * b < 7.9 for _, m, b in kinds)


def test_tame_cells_of_a_uniform_velocity_add_up_in_range():
    for u in itertools.product(np.linspace(-0.5, 0.5, 11), repeat=3):
        F = [factors(v) for v in u]
        s = sum(abs(F[0][0][a] * F[1][0][b] * F[2][0][c]) for a, b, c in VEL)
        k = sum(abs(F[0][1][a] * F[1][2][b] * F[2][2][c]) + abs(F[0][2][a] * F[1][1][b] * F[2][2][c])
                + abs(F[0][2][a] * F[1][2][b] * F[2][1][c]) for a, b, c in VEL)
        assert 4.0 * s + 0.4 * k < 7.9
    assert 0.3 * 4 + 3 * 0.4 < 7.9


def test_safe_cells_send_populations_in_range():
    for v, per_s, per_k in ((0.5, 0.3, 3.0), (1.0, 1.6, 6.0)):
        A, B, C = largest_of[v]
        assert max(A.values()) ** 3 <= per_s
        assert 3 * max(B.values()) * max(C.values()) ** 2 <= per_k + 1e-12
