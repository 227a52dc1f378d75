"""The 3-D state is kept as the moments that a collision reads and populations
are formed again on request (lbm3d.cu).  Checked here: edges of the step's tiles
and segments against the FP64 oracle, the moments against the populations, and
cells that leave the valid range.

Tolerances: populations within 2e-6 + 5e-8 T of the oracle after T steps, as in
test_gpu_3d.py (errors of a few FP32 units in the last place of the largest
population a step); phi and c equal to the sums of the populations exactly (both
are whole numbers of 2^-28 below 2^53).
"""
import numpy as np
import pytest

import oracle
from paper_2504_09024_gb300 import lbm3

pytestmark = pytest.mark.gpu


def drop(nx, ny, nz, scale=1.0):
    Z, Y, X = np.meshgrid(np.arange(nz) + 0.5, np.arange(ny) + 0.5, np.arange(nx) + 0.5, indexing="ij")
    # two flat interfaces across x, bent by the other axes
    zeta = np.minimum(X - nx / 4, 3 * nx / 4 - X) + 0.4 * np.sin(2 * np.pi * (Y / ny + Z / nz))
    phi = 0.5 + 0.5 * np.tanh(2 * zeta / 3.0)
    c = 0.3 / np.cosh(2 * zeta / 3.0) ** 2
    u = (scale * (0.03 * np.sin(2 * np.pi * Z / nz) + 0.01), scale * 0.02 * np.cos(2 * np.pi * X / nx),
         scale * 0.02 * np.sin(2 * np.pi * Y / ny))
    return phi, c, u


def run(nx, ny, nz, field, steps, shape=None, scale=1.0):
    phi, c, u = drop(nx, ny, nz, scale)
    if not field:
        u = (0.02, -0.013, 0.009)
    g = lbm3.Sim3(nx, ny, nz, W=3.0, M_phi=0.05, D_s=0.08, u=(0, 0, 0) if field else u, velocity_field=field)
    g.init(phi, c, *(u if field else (None,) * 3))
    if shape:
        lbm3.lbm3_set_launch_shape(g.ctx, *shape)
    g.step(steps)
    return g, phi, c, u


@pytest.mark.parametrize("nx,ny,nz,shape,field", [
    (30, 16, 6, (18, 6), False),    # whole tiles
    (31, 17, 7, (18, 3), False),    # one column, row and plane over
    (29, 15, 5, (18, 4), True),     # one short
    (61, 9, 4, (10, 1), True),
    (60, 8, 1, (10, 1), False),     # one plane
    (33, 5, 2, (6, 2), True),
    (59, 31, 9, None, False),       # the library's own shapes
    (59, 31, 9, None, True),
])
def test_tile_edges_against_the_oracle(nx, ny, nz, shape, field):
    steps = 6
    g, phi, c, u = run(nx, ny, nz, field, steps, shape)
    o = oracle.Sim3(nx, ny, nz, W=3.0, M_phi=0.05, D_s=0.08)
    o.init(phi, c, *u)
    o.step(steps)
    index = {tuple(v): i for i, v in enumerate(oracle.velocities3())}
    perm = np.array([index[tuple(v)] for v in lbm3.lbm3_velocities()])
    got, want = g.pops(), o.pops()
    for name in ("f", "h"):
        assert np.abs(got[name] - want[name][perm]).max() <= 2e-6 + 5e-8 * steps, name


@pytest.mark.parametrize("steps", [0, 1, 5])
@pytest.mark.parametrize("field,scale", [(False, 1.0), (True, 1.0), (True, 14.0)])
def test_fields_and_sums_are_those_of_the_populations(field, scale, steps):
    """scale 14: velocities for which the step does not trust the sums alone."""
    g, _, _, _ = run(37, 21, 9, field, steps, scale=scale)
    p, f, s = g.pops(), g.fields(), g.sums()
    assert np.array_equal(p["f"].sum(0), f["phi"]) and np.array_equal(p["h"].sum(0), f["c"])
    assert s["sum_phi"] == f["phi"].sum() and s["sum_c"] == f["c"].sum() and s["nonfinite"] == 0


@pytest.mark.parametrize("value", [5.0, -1e9, float("nan"), float("inf")])
def test_an_invalid_cell_spreads_one_cell_a_step(value):
    nx, ny, nz = 33, 20, 11
    phi, c, _ = drop(nx, ny, nz)
    at = (5, 9, 31)
    phi[at] = value
    g = lbm3.Sim3(nx, ny, nz, W=3.0, M_phi=0.05, D_s=0.08, u=(0.02, -0.013, 0.009))
    g.init(phi, c)
    bad = np.zeros((nz, ny, nx), dtype=bool)
    bad[at] = True
    if not np.isfinite(value):  # the gradient of the neighbours is not finite either
        bad = None
    sent = 1
    for step in range(3):
        f, p, s = g.fields(), g.pops(), g.sums()
        if bad is None:
            assert np.isnan(f["phi"][at]) and np.isnan(p["f"][(slice(None),) + at]).all() and s["nonfinite"] >= 54
            break
        assert np.array_equal(np.isnan(f["phi"]), bad) and np.array_equal(np.isnan(f["c"]), bad)
        assert s["nonfinite"] == 54 * sent
        assert np.isnan(p["f"]).sum() + np.isnan(p["h"]).sum() == 54 * sent
        sent = int(bad.sum())
        for axis in range(3):
            bad = bad | np.roll(bad, 1, axis) | np.roll(bad, -1, axis)
        g.step(1)
    # new fields start from a clean slate
    phi, c, _ = drop(nx, ny, nz)
    g.init(phi, c)
    g.step(2)
    assert np.isfinite(g.fields()["phi"]).all() and g.sums()["nonfinite"] == 0
