"""The tile-parallel step, which contexts with no launch shape set take on
small grids, gives the bits of the sweep at every launch shape."""
import numpy as np
import pytest

from paper_2504_09024_gb300 import lbm, workloads as W

pytestmark = pytest.mark.gpu


def run(nx, ny, dtype, walls, fixed_u, ratio, steps, shape=None):
    phys = W.Physics(nx=nx, ny=ny, walls_y=walls, mode=int(fixed_u), u_wall=0.02 * walls, M_phi=0.02,
                     D_s=0.02, nu_a=0.1 * ratio, rho_a=ratio, sigma_o=5e-3, beta=0.3)
    phi, c = W.drop_fields(nx, ny, max(1.5, min(nx, ny) / 3.0), 4.0, xc=nx / 2 + 0.31, yc=ny / 2 + 0.17,
                           c_of_theta=lambda t: 0.3 + 0.15 * np.cos(t))
    ux = W.shear_profile(nx, ny, 0.02)[0] if walls else np.full_like(phi, 0.01)
    s = lbm.Sim(phys, dtype=dtype, kernel=lbm.LBM_KERNEL_TMA)
    if shape:
        s.set_launch_shape(*shape)
    s.init(phi, c, ux, np.full_like(phi, 0.004 * (1 - walls)))
    s.step(steps)
    out = s.pops()
    s.close()
    return out


# tiles of 32 columns and of 4 rows, or 8 where the 4-row tiles outnumber the
# resident blocks (1031 x 61: 528 of them): whole and ragged in both
# directions, narrower than a tile, shorter than the halo
@pytest.mark.parametrize("nx,ny", [(4, 4), (5, 7), (32, 8), (33, 17), (63, 4), (100, 61), (1031, 61)])
@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("dtype,fixed_u,ratio", [
    (lbm.LBM_F32, False, 1.0), (lbm.LBM_F32, False, 2.0), (lbm.LBM_F32, True, 1.0),
    (lbm.LBM_F16S, False, 1.0), (lbm.LBM_BF16S, True, 1.0)])
def test_tile_step_equals_sweep(nx, ny, walls, dtype, fixed_u, ratio):
    a = run(nx, ny, dtype, walls, fixed_u, ratio, 41)
    b = run(nx, ny, dtype, walls, fixed_u, ratio, 41, shape=(128, 16))
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)


def test_library_shape_fills_one_wave():
    """Beyond the tile-parallel range the chosen sweep shape covers the grid
    in one wave of resident blocks."""
    s = lbm.Sim(W.Physics(nx=2048, ny=1024))
    bx, seg = lbm.lbm_get_launch_shape(s.ctx)
    assert bx in (64, 128, 192) and seg >= 4
    assert -(-2048 // (bx - 4)) * -(-1024 // seg) <= 152 * 6
    s.close()


@pytest.mark.parametrize("grids", [[(100, 60), (72, 44), (64, 5)], [(1031, 61)] * 6 + [(300, 40)] * 3])
@pytest.mark.parametrize("fixed_u", [False, True])
def test_batch_shapes_agree_bitwise(grids, fixed_u):
    """Batches at the library's shape (the tile-parallel step here: 4 and 8
    rows a tile), in both forms, give the bits of the sweep at a set shape."""
    out = []
    for form, shape in ((lbm.LBM_BATCH_PERSISTENT, None), (lbm.LBM_BATCH_CHAINS, None),
                        (lbm.LBM_BATCH_PERSISTENT, (192, 24)), (lbm.LBM_BATCH_PERSISTENT, (64, 16))):
        physics = [W.Physics(nx=nx, ny=ny, walls_y=0 if fixed_u else k % 2, mode=int(fixed_u), M_phi=0.02,
                             D_s=0.02 + 0.01 * k, sigma_o=5e-3, beta=0.05 * k)
                   for k, (nx, ny) in enumerate(grids)]
        b = lbm.Batch(physics)
        b.set_form(form)
        if shape:
            b.set_launch_shape(*shape)
        for r, (nx, ny) in zip(b.runs, grids):
            phi, c = W.drop_fields(nx, ny, max(1.5, min(nx, ny) / 3.0), 4.0, xc=nx / 2 + 0.31, c0=0.3)
            r.init(phi, c, np.full_like(phi, 0.01), np.zeros_like(phi))
        b.step(37)
        b.sync()
        out.append([r.pops() for r in b.runs])
        b.close()
    for other in out[1:]:
        for p, q in zip(out[0], other):
            for k in p:
                np.testing.assert_array_equal(p[k], q[k], err_msg=k)


def test_two_cells_per_thread_on_the_librarys_shape():
    """A width the library chose gives way where two cells per thread do not
    have it; one the user set does not."""
    phys = W.Physics(nx=100, ny=60)
    b = lbm.Batch([phys, phys])
    lbm.lbm_set_cells_per_thread(b.runs[0].ctx, 2)
    b.set_cells_per_thread(2)
    assert b.launch_shape()[0] in (128, 192)
    b.set_cells_per_thread(1)
    b.set_launch_shape(64, 16)
    with pytest.raises(lbm.LBMError):
        b.set_cells_per_thread(2)
    b.close()


def test_batch_stall_hook_on_the_tile_step():
    """The bounded wait of the tile-parallel step, in a batch and alone."""
    phys = W.Physics(nx=100, ny=60)
    phi, c = W.drop_fields(100, 60, 14.0, 4.0, c0=0.3)
    z = np.zeros_like(phi)
    b = lbm.Batch([phys, phys])
    s = lbm.Sim(phys, kernel=lbm.LBM_KERNEL_TMA)
    for r in (b.runs[0], b.runs[1], s):
        r.init(phi, c, z, z)
    for r, obj in ((b.runs[1], b), (s, s)):
        lbm.lbm_debug_stall_next_step(r.ctx)
        obj.step(1)
        with pytest.raises(lbm.LBMError) as e:
            obj.sync()
        assert e.value.code == lbm.LBM_ERR_TIMEOUT
        r.init(phi, c, z, z)
        obj.step(3)
        obj.sync()
        assert np.isfinite(r.fields()["phi"]).all()
    s.close()
    b.close()


@pytest.mark.parametrize("nx,ny", [(201, 101), (399, 203), (257, 127)])  # 5, 6 and 7 rows a tile
@pytest.mark.parametrize("walls,dtype", [(0, lbm.LBM_F32), (1, lbm.LBM_F32), (1, lbm.LBM_F16S)])
def test_tile_step_of_other_heights_equals_sweep(nx, ny, walls, dtype):
    a = run(nx, ny, dtype, walls, False, 1.0, 20)
    b = run(nx, ny, dtype, walls, False, 1.0, 20, shape=(128, 16))
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
