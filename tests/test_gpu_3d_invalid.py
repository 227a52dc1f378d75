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
