"""The tile-parallel step in forms that take more than one launch a step or more than
one run a stream, and at every number of rows a tile: the bits of the sweep."""
import numpy as np
import pytest
import torch

from paper_2504_09024_gb300 import lbm, workloads as W

pytestmark = pytest.mark.gpu


def start(run, nx, ny):
    phi, c = W.drop_fields(nx, ny, max(1.5, min(nx, ny) / 3.0), 4.0, xc=nx / 2 + 0.31, c0=0.3)
    run.init(phi, c, np.full_like(phi, 0.01), np.zeros_like(phi))


def physics(k, nx, ny):
    return W.Physics(nx=nx, ny=ny, walls_y=k % 2, M_phi=0.02, D_s=0.02 + 0.001 * k, sigma_o=5e-3, beta=0.02 * (k % 20))


# 150 runs: three tables of at most 64, so three launches a step; 40 runs: three on
# each of the 16 side streams of the chains form
@pytest.mark.parametrize("runs,form", [(150, lbm.LBM_BATCH_PERSISTENT), (40, lbm.LBM_BATCH_CHAINS)])
def test_many_small_runs(runs, form):
    grids = [((33, 17), (40, 21), (64, 9))[k % 3] for k in range(runs)]
    out = []
    for shape in (None, (64, 16)):
        b = lbm.Batch([physics(k, *g) for k, g in enumerate(grids)])
        b.set_form(form)
        if shape:
            b.set_launch_shape(*shape)
        for r, g in zip(b.runs, grids):
            start(r, *g)
        b.step(37)  # graphs of 32, 4 and 1 steps
        b.step(3)
        b.sync()
        out.append([r.pops() for r in b.runs])
        b.close()
    for k, (p, q) in enumerate(zip(*out)):
        for name in p:
            np.testing.assert_array_equal(p[name], q[name], err_msg=f"run {k} {name}")


def rows_of(nx, ny, sms):
    """The library's rows a tile: the fewest that leave one tile to an SM, else that fit
    three to an SM, else 8."""
    tiles = {r: -(-nx // 32) * -(-ny // r) for r in range(4, 9)}
    for most in (sms, 3 * sms):
        for r in range(4, 9):
            if tiles[r] <= most:
                return r
    return 8


@pytest.mark.parametrize("rows", [4, 5, 6, 7, 8])
@pytest.mark.parametrize("walls,dtype", [(0, lbm.LBM_F32), (1, lbm.LBM_F16S)])
def test_every_number_of_rows(rows, walls, dtype):
    """A ragged grid of this GPU's for which the library takes that many rows."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nx, ny = next((x, y) for x in range(129, 700, 31) for y in range(50, 300, 9)
                  if rows_of(x, y, sms) == rows and x % 32 and y % rows and -(-x // 32) * -(-y // 8) <= 14 * sms)
    out = []
    for shape in (None, (128, 16)):
        p = W.Physics(nx=nx, ny=ny, walls_y=walls, u_wall=0.02 * walls, M_phi=0.02, D_s=0.02, sigma_o=5e-3, beta=0.3)
        s = lbm.Sim(p, dtype=dtype, kernel=lbm.LBM_KERNEL_TMA)
        if shape:
            s.set_launch_shape(*shape)
        start(s, nx, ny)
        s.step(13)
        out.append(s.pops())
        s.close()
    for name in out[0]:
        np.testing.assert_array_equal(out[0][name], out[1][name], err_msg=name)
