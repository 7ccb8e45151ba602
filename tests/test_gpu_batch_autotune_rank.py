"""vc_batch_autotune times what a solve runs by the schedule.  Where the resident loop takes the
FP32 sweeps that is the refinement, which a tuning of 2 iterations and of 40 times very differently
(the graph of sweeps, timed before, would also be run); the schedule it leaves must still give the
same solve, and the cut iteration limit must not stay behind."""
import pytest
import torch

from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu


def test_resident_batches_are_tuned_on_the_refinement():
    native = native_or_skip()
    b = native.Batch(inputs.batch_params(64, 2))
    ref = b.value_iterate(tol=1e-6)
    assert max(s["correction_sweeps"] for s in ref[3]) > 2 * 4
    n = native.kernel_launches()
    b.autotune(sweeps=4)
    # 18 schedules, timed twice: 10 launches each before the iterations, none of the sweep graph's
    assert native.kernel_launches() - n == 36 * 10
    got = b.value_iterate(tol=1e-6)
    assert all(torch.equal(x, y) for x, y in zip(ref[:1], got[:1]))
    assert [s["sweeps"] for s in ref[3]] == [s["sweeps"] for s in got[3]]
    assert all(s["certified"] == 1 for s in got[3])
    assert [s["rounds"] for s in ref[3]] == [s["rounds"] for s in got[3]]
    assert max(s["correction_sweeps"] for s in got[3]) > 2 * 4
    b.close()
