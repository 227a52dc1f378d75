"""Cells of the 3-D lattices that leave the valid range: their populations are
invalid, and so is every cell that one of them reaches, one cell a step, until
new fields are given (include/lbm3.h).

The region is exact, and cells far from it keep the bits they have without it: in
a step a cell depends on those up to two away (populations from its neighbours,
whose normals read theirs)."""
import numpy as np
import pytest

from paper_2504_09024_gb300 import lbm3

pytestmark = pytest.mark.gpu


def drop(nx, ny, nz):
    Z, Y, X = np.meshgrid(np.arange(nz) + 0.5, np.arange(ny) + 0.5, np.arange(nx) + 0.5, indexing="ij")
    zeta = np.minimum(X - nx / 4, 3 * nx / 4 - X) + 0.4 * np.sin(2 * np.pi * (Y / ny + Z / nz))
    phi = 0.5 + 0.5 * np.tanh(2 * zeta / 3.0)
    c = 0.3 / np.cosh(2 * zeta / 3.0) ** 2
    u = (0.03 * np.sin(2 * np.pi * Z / nz) + 0.01, 0.02 * np.cos(2 * np.pi * X / nx),
         0.02 * np.sin(2 * np.pi * Y / ny))
    return phi, c, u


def sim(shape, phi, c, field, u, launch):
    nx, ny, nz = shape
    g = lbm3.Sim3(nx, ny, nz, W=3.0, M_phi=0.05, D_s=0.08, u=(0, 0, 0) if field else (0.02, -0.013, 0.009),
                  velocity_field=field)
    g.init(phi, c, *(u if field else (None,) * 3))
    if launch:
        lbm3.lbm3_set_launch_shape(g.ctx, *launch)
    return g


def spread(bad):
    for axis in range(3):
        bad = bad | np.roll(bad, 1, axis) | np.roll(bad, -1, axis)
    return bad


# one cell, and two side by side (an even number of invalid senders to most of
# their neighbours in the very first step); on both sides of tile edges
@pytest.mark.parametrize("cells", [[(5, 9, 31)], [(5, 9, 30), (5, 9, 31)], [(0, 0, 0), (12, 19, 32)]])
@pytest.mark.parametrize("which", ["phi", "c"])
@pytest.mark.parametrize("field,launch", [(False, None), (True, None), (False, (6, 4)), (True, (10, 5)),
                                          (False, (18, 13))])
def test_invalid_cells_stay_invalid(cells, which, field, launch):
    shape = nx, ny, nz = 37, 23, 13
    phi, c, u = drop(*shape)
    clean = sim(shape, phi, c, field, u, launch)
    bad = np.zeros((nz, ny, nx), dtype=bool)
    for at in cells:
        bad[at] = True
        (phi if which == "phi" else c)[at] = 5.0
    # the initial normals near a wrong phi are others
    other = spread(bad) if which == "phi" else bad
    g = sim(shape, phi, c, field, u, launch)
    sent = int(bad.sum())
    for _ in range(10):
        f, p, s, want = g.fields(), g.pops(), g.sums(), clean.fields()
        for name, lattice in (("phi", "f"), ("c", "h")):
            assert np.array_equal(np.isnan(f[name]), bad), name
            assert np.array_equal(f[name][~(bad | other)], want[name][~(bad | other)]), name
            assert np.isnan(p[lattice]).sum() == 27 * sent
        assert s["nonfinite"] == 54 * sent
        sent = int(bad.sum())
        bad, other = spread(bad), spread(spread(other))
        g.step(1)
        clean.step(1)
    assert bad.sum() > 19 * 19 * 13
    # new fields start from a clean slate
    phi, c, u = drop(*shape)
    again, clean = sim(shape, phi, c, field, u, launch), g
    clean.init(phi, c, *(u if field else (None,) * 3))
    again.step(3)
    clean.step(3)
    assert np.array_equal(clean.fields()["phi"], again.fields()["phi"]) and clean.sums()["nonfinite"] == 0


def collided(shape, pops, u, W, M, D):
    """Outgoing f populations of a state in FP64, [27] arrays, and the length of grad phi."""
    nx, ny, nz = shape
    E = np.array([tuple(v) for v in lbm3.lbm3_velocities()])
    f = pops["f"]
    s = f.sum(0)
    j = [(E[:, i, None, None, None] * f).sum(0) for i in range(3)]
    w1 = {-1: 1 / 6, 0: 2 / 3, 1: 1 / 6}
    g = [0.0, 0.0, 0.0]
    for e in E:
        v = np.roll(s, tuple(-e[::-1]), (0, 1, 2))
        for i in range(3):
            g[i] = g[i] + 3 * w1[e[0]] * w1[e[1]] * w1[e[2]] * e[i] * v
    size = np.sqrt(sum(a * a for a in g))
    theta = 4 / W * (1 - s) * s
    k = []
    for i in range(3):
        a = j[i] - u[i] * s
        k.append(a + (M * theta * g[i] / np.maximum(size, 1e-30) - a) / (3 * M + 0.5))
    fac = []
    for v in u:
        t = 1 / 3 + v * v
        fac.append(({0: 1 - t, 1: (t + v) / 2, -1: (t - v) / 2}, {0: -2 * v, 1: v + 0.5, -1: v - 0.5},
                    {0: 1 - v * v, 1: (v * v + v) / 2, -1: (v * v - v) / 2}))
    (Ax, Bx, Cx), (Ay, By, Cy), (Az, Bz, Cz) = fac
    return E, s, size, np.array([s * Ax[a] * Ay[b] * Az[c] + k[0] * Bx[a] * Cy[b] * Cz[c] + k[1] * Cx[a] * By[b] * Cz[c]
                                 + k[2] * Cx[a] * Cy[b] * Bz[c] for a, b, c in E])


@pytest.mark.parametrize("launch", [None, (6, 4), (10, 3), (18, 9)])
def test_populations_that_leave_the_range(launch):
    """phi = 1 (no interface flux) in a diverging velocity, W = 0.004: in the second
    step theta reaches 80 and |k'| 23.  A population below -8 is invalid, one above 8
    is cut off, whatever its velocity.  FP32 normals: phi to 2^-24, its gradient
    above 1e-3, so k' to 23 * 4 * 2^-24 / 1e-3 = 6e-3 and populations to 1e-2."""
    shape = nx, ny, nz = 34, 21, 9
    Z, Y, X = np.meshgrid(np.arange(nz) + 0.5, np.arange(ny) + 0.5, np.arange(nx) + 0.5, indexing="ij")
    wave = 2 * np.pi * (X / nx + Y / ny + Z / nz)
    u = (0.1 * np.sin(2 * np.pi * X / nx), 0.1 * np.sin(2 * np.pi * Y / ny + 1.0), 0.05 * np.sin(wave))
    phi, c = np.full((nz, ny, nx), 1.0), np.full((nz, ny, nx), 0.001)
    W, M, D = 0.004, 1.0, 0.08
    g = lbm3.Sim3(nx, ny, nz, W=W, M_phi=M, D_s=D, velocity_field=True)
    g.init(phi, c, *u)
    if launch:
        lbm3.lbm3_set_launch_shape(g.ctx, *launch)
    g.step(1)
    E, s, size, want = collided(shape, g.pops(), u, W, M, D)
    g.step(1)
    got, f, sums = g.pops(), g.fields(), g.sums()
    sent = np.array([np.roll(got["f"][q], tuple(-E[q][::-1]), (0, 1, 2)) for q in range(27)])
    clear = size > 1e-3
    assert clear.mean() > 0.8
    low = high = still = 0
    for q in range(27):
        if not E[q].any():
            continue
        at = clear & (want[q] < -8 - 1e-2)
        assert np.isnan(sent[q][at]).all()
        low, still = low + at.sum(), still + (at.sum() if E[q][0] == 0 else 0)
        at = clear & (want[q] > 8 + 1e-2)
        assert (sent[q][at] == 8 - 2.0 ** -28).all()
        high = high + at.sum()
        at = clear & (np.abs(want[q]) < 8 - 1e-2)
        assert np.abs(sent[q][at] - want[q][at]).max() < 1e-2
    assert low > 200 and high > 200 and still > 200  # 326, 267 and 308 in FP64
    # the rest population takes the remainder, modulo the range
    left = (np.where(np.isnan(sent), -8.0, sent).sum(0) - s) / 16
    assert (left == np.round(left)).all()
    bad = np.isnan(got["f"]).any(0)
    assert np.array_equal(np.isnan(f["phi"]), bad) and not np.isnan(f["c"]).any()
    assert np.array_equal(f["phi"][~bad], got["f"].sum(0)[~bad]) and np.array_equal(f["c"], got["h"].sum(0))
    assert sums["nonfinite"] == np.isnan(got["f"]).sum() and sums["sum_phi"] == np.nansum(got["f"])
    # a cell that received one is invalid from then on
    g.step(1)
    assert np.isnan(g.fields()["phi"][spread(bad)]).all() and np.isnan(g.fields()["c"][spread(bad)]).all()


def timed(nx, u, spike=False, steps=False):
    """us of phi and c into device arrays (or of a step) after two steps with a velocity field
    of size u."""
    import torch
    z = torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5 - nx / 2
    r = torch.sqrt(z[:, None, None] ** 2 + z[None, :, None] ** 2 + z[None, None, :] ** 2)
    zeta = nx / 4 - r
    phi, c = 0.5 + 0.5 * torch.tanh(zeta / 2), 0.3 / torch.cosh(zeta / 2) ** 2
    if spike:
        phi[nx // 3, 5, 7] = 5.0
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        stream.wait_stream(torch.cuda.default_stream())
        g = lbm3.Sim3(nx, nx, nx, W=4.0, M_phi=0.05, D_s=0.08, velocity_field=True, stream=stream.cuda_stream)
        lbm3.lbm3_init_fields_device(g.ctx, phi, c, *(torch.full_like(phi, v) for v in (u if isinstance(u, tuple) else (u, -u, 0.0))))
        g.step(2)
        out = torch.empty((2,) + phi.shape, dtype=torch.float64, device="cuda")
        best = 1e30
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            if steps:
                g.step(1)
            else:
                lbm3.lbm3_get_fields_device(g.ctx, out[0], out[1])
            b.record()
            b.synchronize()
            best = min(best, 1e3 * a.elapsed_time(b))
    g.sums()
    g.close()
    return best


def test_outputs_of_fast_and_of_partly_invalid_runs_stay_cheap():
    """Populations are formed again only next to planes that call for it, and then once
    each: a velocity of 0.35 costs nothing, one invalid cell three planes of 128, and a
    velocity that no bound holds for (0.7) the populations of every cell once."""
    usual = timed(128, 0.05)
    assert timed(128, 0.35) < 3 * usual
    assert timed(128, 0.05, spike=True) < 5 * usual
    assert timed(128, 0.7) < 60 * usual


def test_a_fast_field_steps_as_quickly():
    """Beyond one cell a step along an axis (1.2) populations are still in range, and the
    step has nothing to settle at its end."""
    assert timed(128, (1.2, 0.0, 0.0), steps=True) < 1.5 * timed(128, (0.05, 0.0, 0.0), steps=True)


@pytest.mark.parametrize("shape", [(5, 5, 5), (33, 17, 9), (16, 8, 4)])
def test_sums_of_populations_that_leave_32_bits(shape):
    """A converging velocity of 0.45 where c is 3.9: the populations that meet in a
    cell are in range and their sum is not; c is the sum all the same."""
    nx, ny, nz = shape
    Z, Y, X = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    u = tuple(-0.45 * np.sign(a - n // 2) for a, n in ((X, nx), (Y, ny), (Z, nz)))
    phi, c = np.full((nz, ny, nx), 0.5), np.full((nz, ny, nx), 3.9)
    g = lbm3.Sim3(nx, ny, nz, W=4.0, M_phi=0.05, D_s=0.08, velocity_field=True)
    g.init(phi, c, *u)
    g.step(1)
    f, p, s = g.fields(), g.pops(), g.sums()
    assert f["c"].max() > 10.0
    assert np.array_equal(f["c"], p["h"].sum(0)) and np.array_equal(f["phi"], p["f"].sum(0))
    assert s["sum_c"] == p["h"].sum() and s["nonfinite"] == 0
