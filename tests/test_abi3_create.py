"""lbm3_create chooses a launch shape before it touches the device, and that takes
no time that grows with the box: a legal box of 2^30 planes is refused here, without
a GPU, as quickly as a small one."""
import ctypes
import time

import pytest

from paper_2504_09024_gb300 import build as B
from paper_2504_09024_gb300 import lbm, lbm3


def has_gpu():
    try:
        import torch
        return torch.cuda.is_available()
    except ImportError:
        return False


@pytest.mark.skipif(has_gpu(), reason="would allocate the 80 GB of the box")
@pytest.mark.parametrize("size", [(1, 1, 1 << 30), (3, 2, 178956970), (16, 16, 16)])
def test_choice_of_launch_shape_takes_no_time(size):
    B.build()
    lib = lbm3.load()
    p = lbm3.lbm3_params()
    assert lib.lbm3_params_default(ctypes.byref(p)) == lbm.LBM_OK
    p.nx, p.ny, p.nz = size
    ctx = ctypes.c_void_p()
    t = time.perf_counter()
    rc = lib.lbm3_create(ctypes.byref(p), None, ctypes.byref(ctx))
    took = time.perf_counter() - t
    assert rc == lbm.LBM_ERR_CUDA and not ctx.value
    assert took < 1.0
