"""Autotuners time what they are given: a tuned run or batch is not slower than one
left alone.

Medians of nine alternating timings of 320 steps each (milliseconds, so the spread of
one side is below 1 %); 5 % are allowed for the few steps the tuner itself measures."""
import numpy as np
import pytest
import torch

from paper_2504_09024_gb300 import lbm, lbm3, workloads as W

pytestmark = pytest.mark.gpu


def median_us(objects, stream, steps=320):
    times = [[] for _ in objects]
    with torch.cuda.stream(stream):
        for k in range(10):
            for o, t in zip(objects, times):
                o.step(steps)
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                o.step(steps)
                b.record()
                b.synchronize()
                if k:
                    t.append(1e3 * a.elapsed_time(b) / steps)
    return [float(np.median(t)) for t in times]


def physics(nx, ny):
    return W.Physics(nx=nx, ny=ny, M_phi=0.02, D_s=0.02, sigma_o=5e-3, beta=0.3)


def start(run, nx, ny):
    phi, c = W.drop_fields(nx, ny, min(nx, ny) / 4.0, 4.0, c0=0.3)
    run.init(phi, c, np.zeros_like(phi), np.zeros_like(phi))


# grids for which the library takes 5 to 7 rows a tile on 152 SMs
@pytest.mark.parametrize("nx,ny", [(500, 140), (360, 180), (400, 200)])
def test_a_tuned_run_is_not_slower(nx, ny):
    s = torch.cuda.Stream()
    runs = [lbm.Sim(physics(nx, ny), stream=s.cuda_stream) for _ in range(2)]
    for r in runs:
        start(r, nx, ny)
    runs[1].autotune(steps=64)
    alone, tuned = median_us(runs, s)
    assert tuned < 1.05 * alone
    for r in runs:
        r.close()


@pytest.mark.parametrize("grids", [[(300, 130)] * 2, [(200, 100)] * 3 + [(150, 61)]])
def test_a_tuned_batch_is_not_slower(grids):
    s = torch.cuda.Stream()
    batches = [lbm.Batch([physics(*g) for g in grids], stream=s.cuda_stream) for _ in range(2)]
    for b in batches:
        for r, g in zip(b.runs, grids):
            start(r, *g)
    batches[1].autotune(steps=64)
    alone, tuned = median_us(batches, s)
    assert tuned < 1.05 * alone
    for b in batches:
        b.close()


def test_the_3d_tuner_times_the_shape_it_is_given():
    """Three heights of tile, five of segment (4, 8, 16, 32 and all 40 planes), and the
    shape that was set, which is none of those; one warm-up step each."""
    g = lbm3.Sim3(40, 30, 40)
    lbm3.lbm3_set_launch_shape(g.ctx, 10, 13)
    lbm3.lbm3_autotune(g.ctx, 3)
    assert g.t == (3 * 5 + 1) * (3 + 1)
    lbm3.lbm3_set_launch_shape(g.ctx, 18, 40)
    before = g.t
    lbm3.lbm3_autotune(g.ctx, 3)
    assert g.t - before == 3 * 5 * (3 + 1)
    g.close()


@pytest.mark.parametrize("shape", [(256, 256, 256), (150, 97, 61)])
def test_a_tuned_3d_run_is_not_slower(shape):
    nx, ny, nz = shape
    s = torch.cuda.Stream()
    runs = [lbm3.Sim3(nx, ny, nz, u=(0.02, -0.013, 0.009), stream=s.cuda_stream) for _ in range(2)]
    lbm3.lbm3_autotune(runs[1].ctx, 20)
    z = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for r in runs:
        lbm3.lbm3_init_fields_device(r.ctx, z, z, None, None, None)
    alone, tuned = median_us(runs, s, steps=40)
    assert tuned < 1.05 * alone
    for r in runs:
        r.close()
