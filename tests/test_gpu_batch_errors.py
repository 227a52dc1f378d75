"""A batch reports what went wrong on the device in one of its runs."""
import numpy as np
import pytest

from paper_2504_09024_gb300 import lbm, workloads as W

pytestmark = pytest.mark.gpu


def test_batch_sync_reports_a_timeout_of_one_of_its_runs():
    """A run of a batch launches kernels with bounded waits on its own, too (its fields
    and diagnostics, or a step taken alone: the one that the test hook can make fail)."""
    phys = W.Physics(nx=100, ny=60)
    phi, c = W.drop_fields(100, 60, 14.0, 4.0, c0=0.3)
    z = np.zeros_like(phi)
    b = lbm.Batch([phys, phys, phys])
    for r in b.runs:
        r.init(phi, c, z, z)
    b.sync()
    lbm.lbm_debug_stall_next_step(b.runs[2].ctx)
    b.runs[2].step(1)
    with pytest.raises(lbm.LBMError) as e:
        b.sync()
    assert e.value.code == lbm.LBM_ERR_TIMEOUT
    # reported once, to whoever asks first
    b.runs[2].sync()
    lbm.lbm_debug_stall_next_step(b.runs[1].ctx)
    b.runs[1].step(1)
    with pytest.raises(lbm.LBMError):
        b.runs[1].sync()
    b.sync()
    for r in b.runs:
        r.init(phi, c, z, z)
    b.step(3)
    b.sync()
    want = b.runs[0].fields()
    for r in b.runs[1:]:
        got = r.fields()
        assert all(np.array_equal(got[k], want[k]) for k in want)
    b.close()
