"""Diagnostics and the count of drops at the edges of their kernels' tiles.

The diagnostics are compared with the same sums in FP64 numpy over the fields that
the library returns; both see the same values, so what differs is the rounding of
FP64 sums: 1e-9 relative (2e-9 for the drop indicator, which the library takes from
phi in units of 2^-29).  The count of drops is a whole number and compared with
scipy's labels.
"""
import numpy as np
import pytest

from paper_2504_09024_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu


def sim_of(nx, ny, walls, phi, dtype=lbm.LBM_F32, mode=0):
    p = wl.Physics(nx=nx, ny=ny, walls_y=walls, mode=mode, W=4.0, M_phi=0.05, D_s=0.05,
                   u_wall=0.01 if walls else 0.0, sigma_o=1e-3, beta=0.3)
    s = lbm.Sim(p, dtype=dtype)
    y = (np.arange(ny) + 0.5)[:, None] + np.zeros((ny, nx))
    s.init(phi, np.full_like(phi, 0.1), 0.01 * (2 * y / ny - 1), np.full_like(phi, 0.002))
    return s


def disc(nx, ny, cx, cy, r, W=4.0):
    x, y = np.arange(nx) + 0.5, np.arange(ny) + 0.5
    dx = (x - cx + nx / 2) % nx - nx / 2
    dy = (y - cy + ny / 2) % ny - ny / 2
    return 0.5 + 0.5 * np.tanh(2 * (r - np.hypot(dx[None, :], dy[:, None])) / W)


@pytest.mark.parametrize("nx,ny,walls,mode,dtype", [
    (32, 8, 0, 0, lbm.LBM_F32), (33, 9, 1, 0, lbm.LBM_F32), (31, 7, 0, 1, lbm.LBM_F32),
    (100, 61, 1, 0, lbm.LBM_F16S), (4, 4, 0, 0, lbm.LBM_F32), (300, 40, 0, 0, lbm.LBM_BF16S)])
def test_diagnostics_are_those_of_the_fields(nx, ny, walls, mode, dtype):
    s = sim_of(nx, ny, walls, disc(nx, ny, 0.1 * nx, 0.4 * ny, 0.3 * min(nx, ny)), dtype, mode)
    s.step(3)
    d, f = s.diagnostics(), s.fields()
    w = np.clip(f["phi"], 0.0, 1.0)
    x, y = np.arange(nx) + 0.5, np.arange(ny) + 0.5

    def centre(t, n, axis):
        a = 2 * np.pi * t / n
        m = w.sum(axis)
        return np.arctan2((m * np.sin(a)).sum(), (m * np.cos(a)).sum()) % (2 * np.pi) * n / (2 * np.pi)

    xc = centre(x, nx, 0)
    yc = (w.sum(1) * y).sum() / w.sum() if walls else centre(y, ny, 1)
    dx = (x - xc + nx / 2) % nx - nx / 2
    dy = y - yc if walls else (y - yc + ny / 2) % ny - ny / 2
    xx, yy = (w * dx[None, :] ** 2).sum() / w.sum(), (w * dy[:, None] ** 2).sum() / w.sum()
    xy = (w * dx[None, :] * dy[:, None]).sum() / w.sum()
    root = np.sqrt(max(0.25 * (xx - yy) ** 2 + xy * xy, 0.0))
    want = {"sum_phi": f["phi"].sum(), "sum_c": f["c"].sum(), "xc": xc, "yc": yc,
            "umax": np.sqrt(f["ux"] ** 2 + f["uy"] ** 2).max()}
    for k, v in want.items():
        assert abs(d[k] - v) <= 2e-9 * abs(v), (k, d[k], v)
    # L^2 + B^2 and L^2 - B^2 are 16 times the trace and 32 times the root
    L2, B2 = d["L"] ** 2, d["B"] ** 2
    assert abs(L2 + B2 - 16 * (xx + yy)) <= 2e-9 * 16 * (xx + yy)
    assert abs(L2 - B2 - 32 * root) <= 2e-8 * 16 * (xx + yy)
    assert d["nonfinite"] == 0 and d["sigma_neg"] == 0


def test_diagnostics_leave_invalid_cells_out_and_count_them():
    import torch
    nx, ny = 70, 21
    phi, c = disc(nx, ny, 20, 10, 6), np.full((ny, nx), 0.1)
    c[3, 5], c[4, 40] = 0.99, 0.98  # 1 + 0.3 log(1 - c) < 0
    phi[9, 33] = np.nan
    s = sim_of(nx, ny, 0, phi, mode=1)
    # fields on the device take any c; those from the host are checked
    t = [torch.from_numpy(v).cuda() for v in (phi, c, np.zeros_like(phi), np.zeros_like(phi))]
    torch.cuda.synchronize()
    lbm.lbm_init_fields_device(s.ctx, *t)
    d, f = s.diagnostics(), s.fields()
    bad = ~(np.isfinite(f["phi"]) & np.isfinite(f["c"]) & np.isfinite(f["ux"]))
    assert d["nonfinite"] == bad.sum() >= 1
    with np.errstate(divide="ignore", invalid="ignore"):
        assert d["sigma_neg"] == (1 + 0.3 * np.log(1 - f["c"][~bad]) < 0).sum() >= 2
    assert abs(d["sum_phi"] - f["phi"][~bad].sum()) <= 1e-9 * nx * ny


@pytest.mark.parametrize("nx,ny,walls,kind", [
    (64, 16, 0, "noise"), (65, 17, 1, "noise"), (131, 40, 0, "noise"), (4, 5, 0, "noise"), (97, 33, 0, "full"),
    (97, 33, 1, "empty"), (90, 64, 0, "spiral"), (256, 128, 1, "noise"), (33, 9, 0, "stripes")])
def test_count_of_drops(nx, ny, walls, kind):
    from scipy import ndimage
    rng = np.random.default_rng(nx * ny)
    if kind == "noise":
        inside = rng.random((ny, nx)) < 0.58
    elif kind == "spiral":  # one winding set: the longest chains of runs
        y, x = np.mgrid[0:ny, 0:nx]
        inside = (y % 4 == 0) & (x > 0) | (x == 1) & (y % 8 < 5) | (x == nx - 2) & ((y + 4) % 8 < 5)
    elif kind == "stripes":
        inside = np.arange(nx)[None, :] % 2 + np.zeros((ny, nx), int) > 0
    else:
        inside = np.full((ny, nx), kind == "full")
    s = sim_of(nx, ny, walls, np.where(inside, 1.0, 0.0), mode=1)
    lab, n = ndimage.label(inside)
    parent = list(range(n + 1))

    def find(a):
        while parent[a] != a:
            a = parent[a]
        return a

    pairs = list(zip(lab[:, 0], lab[:, -1])) + ([] if walls else list(zip(lab[0], lab[-1])))
    for a, b in pairs:
        if a and b:
            parent[find(a)] = find(b)
    want = len({find(a) for a in range(1, n + 1)})
    for _ in range(3):
        assert s.components(0.5) == want
