"""The autotuner ranks what a solve runs: on a small stored matrix a sweep of the resident loop takes
less than half of a launched one with its residual and stopping test, so after tuning the solves
use it (a handful of launches), whichever schedule single sweeps keep and with or without a sliced
copy; pinning a schedule goes back to that schedule's own way.  Results never change."""
import pytest
import torch

from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fmt", ["csr_f32", "csr_bf16"])
@pytest.mark.parametrize("sliced", [False, True])
def test_solves_use_the_faster_loop(fmt, sliced):
    native = native_or_skip()
    m = native.MDP.build(inputs.make_params(3, 3, 4, 0.95, seed=3), fmt=fmt, padded=True, sliced=sliced)

    def solve():
        n = native.kernel_launches()
        V, _, pi, st = m.value_iterate(tol=1e-6, fp32_only=True)
        return V, pi, st["sweeps"], native.kernel_launches() - n

    ref = solve()
    assert ref[2] > 100 and (ref[3] > 100) == sliced  # a sliced handle starts with the launched ring
    m.autotune(reps=5)
    got = solve()
    assert got[3] < 10
    assert torch.equal(ref[0], got[0]) and torch.equal(ref[1], got[1]) and ref[2] == got[2]
    V = torch.rand(m.S, device="cuda") * 50
    want = m.bellman32(V, torch.empty_like(V)).clone()
    launched = []
    for k in range(m.schedules()):
        m.use_schedule(k)
        info = m.info()
        out = solve()
        launched.append(out[3] > 100)
        assert launched[-1] == (info["csr_sliced"] == 1 or info["csr_pipelined"] == 0)
        assert torch.equal(ref[0], out[0]) and torch.equal(m.bellman32(V, torch.empty_like(V)), want)
    assert any(launched) and not all(launched)
    m.close()
