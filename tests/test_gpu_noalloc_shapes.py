"""The no-allocation sweep in two launches against the handle's sweep, bit for bit, over its
dispatch: items of four and two states, arrays that are only 8-byte aligned, blocks of two and of
eight warps, every host bound; called twice in a row, so the residual's words must come back
clean."""
import pytest

from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,C,Q", [(1, 1, 0), (2, 3, 3), (4, 4, 6), (5, 4, 11), (6, 4, 9), (6, 4, 10), (8, 2, 3), (9, 1, 5)])
@pytest.mark.parametrize("shift", [0, 2])
def test_sweep_equals_the_handles(H, C, Q, shift):
    native = native_or_skip()
    import torch

    p = inputs.make_params(H, C, Q, 0.95, seed=H + Q)
    m = native.MDP.build(p)
    g = torch.Generator(device="cuda").manual_seed(4)
    V = torch.rand(m.S + shift, device="cuda", generator=g)[shift:] * 40
    want, wpi = torch.empty(m.S, device="cuda"), torch.empty(m.S, dtype=torch.int32, device="cuda")
    m.bellman32(V.clone(), want, wpi)
    out = torch.empty(m.S + shift, device="cuda")[shift:]
    pi, res = torch.empty_like(wpi), torch.empty(1, device="cuda")
    for _ in range(2):
        out.fill_(-1.0)
        native.bellman32_noalloc(p, V, out, pi, res)
        assert torch.equal(out, want) and torch.equal(pi, wpi)
        assert float(res) == float((want - V).abs().max())
    native.bellman32_noalloc(p, want, out, None, None)
    m.bellman32(want.clone(), V)
    assert torch.equal(out, V)
    m.close()
