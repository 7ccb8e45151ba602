"""The resident FP32 loop against its own sweeps: k sweeps in one call equal k one-sweep calls
bit for bit (values, residual, sweep count), over the layouts that pick another kernel --
rows of odd and even queue lengths (8- and 16-byte items), every host bound, one CTA and
many, value arrays that are only 8-byte aligned -- and resuming a stopped loop continues it."""
import pytest

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu

# (H, C, Q): S on both sides of the one-CTA limit (8,192) and of one item per thread
SHAPES = [(1, 1, 0), (1, 1, 1), (2, 3, 3), (3, 3, 4), (4, 4, 5), (4, 4, 6), (4, 4, 7), (5, 2, 16), (5, 3, 15),
          (6, 3, 2), (7, 2, 4), (8, 2, 3), (9, 1, 9), (12, 1, 1)]


@pytest.mark.parametrize("H,C,Q", SHAPES)
@pytest.mark.parametrize("shift", [0, 2])
def test_loop_equals_its_sweeps(H, C, Q, shift):
    native = native_or_skip()
    import torch

    from paper_2012_12419_gb300 import inputs

    m = native.MDP.build(inputs.make_params(H, C, Q, 0.95, seed=11))
    g = torch.Generator(device="cuda").manual_seed(2)
    start = torch.rand(m.S + shift, device="cuda", generator=g)[shift:] * 40
    for k in (1, 2, 67):  # 67: past the 64 slots of the residual ring
        V, _, pi, st = m.value_iterate(V=start.clone() if shift == 0 else _shifted(start, shift), tol=1e-30,
                                       max_sweeps=k, fp32_only=True, want_v64=False, raise_on_nonconvergence=False)
        a, b = start.clone(), torch.empty_like(start)
        for _ in range(k):
            m.bellman32(a, b)
            a, b = b, a
        assert torch.equal(V, a) and st["sweeps"] == k
        assert st["residual"] == float((a - b).abs().max())
        pi_ref, _ = m.extract_policy(a)
        assert torch.equal(pi, pi_ref)
    half, _, _, _ = m.value_iterate(V=start.clone(), tol=1e-30, max_sweeps=30, fp32_only=True,
                                    raise_on_nonconvergence=False)
    rest, _, _, _ = m.value_iterate(V=half, tol=1e-30, max_sweeps=37, fp32_only=True, raise_on_nonconvergence=False)
    assert torch.equal(rest, V)
    m.close()


def _shifted(t, shift):
    import torch

    buf = torch.empty(t.numel() + shift, device="cuda")
    buf[shift:] = t
    return buf[shift:]
