"""A resident kernel ends its launch after some 4 ms (8 M cycles), so that kernels of other streams
get their turn: long solves take launches in proportion to their time, and where a launch ends
changes no result (the points differ from run to run, the values must not)."""
import pytest
import torch

from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu

MS = 8.0  # 8 M cycles at 1 GHz: no launch is longer
SLOW = dict(tol=1e-9, fp32_only=True, want_v64=False, raise_on_nonconvergence=False)


def _count(native, call):
    n = native.kernel_launches()
    out = call()
    return out, native.kernel_launches() - n


@pytest.mark.parametrize("H,C,Q,fmt,sweeps", [(3, 3, 19, "implicit", 40000), (5, 3, 15, "implicit", 16000),
                                              (6, 4, 10, "implicit", 8000), (5, 3, 15, "csr_f32", 12000)])
@pytest.mark.parametrize("self_loop", [False, True])
def test_value_iteration(H, C, Q, fmt, sweeps, self_loop):
    native = native_or_skip()
    m = native.MDP.build(inputs.make_params(H, C, Q, 0.9999, seed=4), fmt=fmt)
    (V, _, _, st), n = _count(native, lambda: m.value_iterate(max_sweeps=sweeps, self_loop=self_loop, want_pi=False, **SLOW))
    assert st["ms_fp32"] > MS
    assert st["ms_fp32"] / MS <= n <= st["ms_fp32"]
    # the same sweeps in two calls, and (stored rows) by the launched kernels
    k = st["sweeps"]  # fewer than allowed where the FP32 floor ends the loop
    half = m.value_iterate(max_sweeps=k // 3, self_loop=self_loop, **SLOW)[0]
    rest = m.value_iterate(V=half, max_sweeps=k - k // 3, self_loop=self_loop, **SLOW)
    assert torch.equal(rest[0], V) and rest[3]["residual"] == st["residual"]
    if fmt != "implicit":
        m.set_wait_limit(1 << 22)
        assert torch.equal(m.value_iterate(max_sweeps=sweeps, self_loop=self_loop, **SLOW)[0], V)
    m.close()


def test_batch():
    native = native_or_skip()
    b = native.Batch([inputs.make_params(H, C, Q, 0.9999, seed=i) for i, (H, C, Q) in
                      enumerate([(5, 3, 15), (4, 6, 6), (2, 6, 12), (4, 5, 7)])])
    kw = dict(tol=1e-9, fp32_only=True, raise_on_nonconvergence=False)
    t = [torch.cuda.Event(enable_timing=True) for _ in range(2)]

    def solve():
        t[0].record()
        out = b.value_iterate(max_sweeps=9000, **kw)
        t[1].record()
        torch.cuda.synchronize()
        return out

    out, n = _count(native, solve)
    assert t[0].elapsed_time(t[1]) > MS and n >= t[0].elapsed_time(t[1]) / MS
    half = b.value_iterate(max_sweeps=2700, **kw)[0]
    assert torch.equal(b.value_iterate(V=half, max_sweeps=6300, **kw)[0], out[0])
    b.close()


def test_correction_solve():
    """An adjoint system of long rows: some 60 ms of BiCGSTAB, several launches in one call."""
    native = native_or_skip()
    m = native.MDP.build(inputs.make_params(3, 40, 3, 0.9, seed=3))
    _, V64, pi, _ = m.value_iterate(tol=1e-6)
    rho = torch.full((m.S,), 1.0 / m.S, dtype=torch.float64, device="cuda")
    dJ, lam, gs = m.value_grad(V64, pi, rho, tol=1e-9, want_lambda=True)
    assert gs["residual64"] < 1e-9
    dJ2, lam2, _ = m.value_grad(V64, pi, rho, tol=1e-9, want_lambda=True)
    assert torch.equal(dJ, dJ2) and torch.equal(lam, lam2)
    m.close()
