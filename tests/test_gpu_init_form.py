"""The stored form of a new state (sum of a cell's nine slots in fixed point, and each
slot less its weight's share of the sum) has the bits that FP64 arithmetic gives: the
slots added in their order, and one fused multiply-add a slot."""
import os

import numpy as np
import pytest

from paper_2504_09024_gb300 import lbm, workloads as W

pytestmark = pytest.mark.gpu

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WEIGHTS = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, dtype=np.float32)


def populations(kind, shape, rng):
    """[9][ny][nx] float32 values: a population of each sort that a state has."""
    w = WEIGHTS[:, None, None]
    if kind == "interface":  # a profile with its flux
        phi = 1 / (1 + np.exp(-rng.uniform(-8, 8, shape)))
        return (w * phi * (1 + 0.05 * rng.standard_normal((9,) + shape))).astype(np.float32)
    if kind == "bulk":       # weights times a value, each rounded
        return (w.astype(np.float64) * rng.choice([1.0, 0.3, 0.999999, 1.04, 1e-3], shape)).astype(np.float32)
    if kind == "tail":       # a tail that dies out, zeros of both signs among it
        v = w * 10.0 ** rng.uniform(-44, -9, shape)
        return (v * rng.choice([0.0, -0.0, 1.0, 1.0, 1.3], (9,) + shape)).astype(np.float32)
    if kind == "foot":       # the foot of a profile: sums of a fixed-point unit to a few thousand
        return (w * 10.0 ** rng.uniform(-10, -5, shape) * (1 + 0.1 * rng.standard_normal((9,) + shape))).astype(np.float32)
    if kind == "ties":       # sums at and next to half a unit: slot 8 carries what is missing
        f = (w * rng.uniform(0.1, 1.0, shape)).astype(np.float32)
        units = f[:8].astype(np.float64).sum(0) * 2.0 ** 29
        off = rng.choice([0.0, 1.0, -1.0], shape) * 2.0 ** rng.uniform(-30, -10, shape)
        f[8] = (0.5 + off - (units - np.floor(units))) / 2.0 ** 29
        return f
    return rng.uniform(-0.2, 0.2, (9,) + shape).astype(np.float32)  # anything with a sum in range


def stored(f):
    """Sum (whole numbers) and deviations of the slots f in FP64; scale 2^29."""
    slots = np.stack([np.roll(f[q], (-EY[q], -EX[q]), (0, 1)) for q in range(9)])  # periodic
    s = np.zeros(f.shape[1:])
    for q in range(9):
        s = s + slots[q].astype(np.float64)
    S = np.rint(s * 2.0 ** 29)
    # the fused multiply-add: the product has 55 bits and the difference fits 64 where
    # slots are multiples of 2^-64, as they are wherever S is not 0
    wide = slots[1:].astype(np.longdouble) - WEIGHTS[1:, None, None].astype(np.longdouble) * (S.astype(np.longdouble) / 2 ** 29)
    return S, wide.astype(np.float64).astype(np.float32)


@pytest.mark.parametrize("kind", ["interface", "bulk", "foot", "tail", "ties", "any"])
def test_stored_form_has_the_bits_of_fp64(kind, tmp_path):
    nx, ny = 509, 257
    rng = np.random.default_rng(7)
    f, h = populations(kind, (ny, nx), rng), populations(kind, (ny, nx), rng)
    s = lbm.Sim(W.Physics(nx=nx, ny=ny, walls_y=0, M_phi=0.05, D_s=0.05, sigma_o=1e-3, beta=0.3, c_max=1.0))
    z = np.zeros((ny, nx))
    s.init(z, z, z, z)
    lbm.lbm_set_populations(s.ctx, f.astype(np.float64), h.astype(np.float64), None)
    path = os.path.join(tmp_path, "state")
    lbm.lbm_save_state(s.ctx, path)
    raw = np.fromfile(path, dtype=np.uint8)
    s.close()
    # planes of 4 ghost columns, nx columns, 4 ghost columns, padded to 32
    pitch = -(-(nx + 8) // 32) * 32
    state = raw[-4 * 27 * ny * pitch:].view(np.float32).reshape(27, ny, pitch)[:, :, 4:4 + nx]
    for base, values in ((0, f), (9, h)):
        S, d = stored(values)
        assert np.array_equal(np.ascontiguousarray(state[base]).view(np.int32), S.astype(np.int32))
        got = np.ascontiguousarray(state[base + 1:base + 9])
        assert np.array_equal(got.view(np.int32), d.view(np.int32))
