"""The resident batched loop against the single-instance loop, bit for bit: both run the items
of vc_implicit.cuh, so every instance's FP32 values and sweep count must equal its own solve.

The lists mix host counts 1..5, rows of odd and even queue lengths (items of 4 and of 2),
instances smaller than a warp's share and larger than the whole-instance path's limit, several
discounts (instances end at different sweeps and the work is cut again), one instance alone,
and a host count that sends the batch to the graph loop."""
import pytest

from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu

SIZES = {
    "mixed": [(1, 1, 1), (5, 3, 8), (2, 6, 12), (4, 5, 7), (3, 2, 4), (5, 4, 11), (2, 2, 3), (4, 6, 6), (1, 3, 0)],
    "one": [(5, 4, 9)],
    "graph": [(6, 2, 10), (3, 3, 5), (5, 3, 8), (4, 5, 7)],
}


@pytest.mark.parametrize("name", list(SIZES))
@pytest.mark.parametrize("self_loop", [False, True])
def test_batch_equals_single_solves(name, self_loop):
    native = native_or_skip()
    import torch

    gammas = (0.9, 0.95, 0.99)
    ps = [inputs.make_params(H, C, Q, gammas[i % 3], seed=50 + i) for i, (H, C, Q) in enumerate(SIZES[name])]
    b = native.Batch(ps)
    assert b.small_instances()["count"] < len(ps)  # at least one instance needs the loop
    g = torch.Generator(device="cuda").manual_seed(1)
    start = torch.rand(b.total, device="cuda", generator=g) * 10
    for most in (1, 2, 5, 1_000_000):
        V, _, pi, st, _ = b.value_iterate(V=start.clone(), tol=1e-6, max_sweeps=most, fp32_only=True,
                                          raise_on_nonconvergence=False, self_loop=self_loop)
        for i, p in enumerate(ps):
            lo, hi = int(b.offsets[i]), int(b.offsets[i + 1])
            m = native.MDP.build(p)
            W, _, pj, sj = m.value_iterate(V=start[lo:hi].clone(), tol=1e-6, max_sweeps=most, fp32_only=True,
                                           want_v64=False, raise_on_nonconvergence=False, self_loop=self_loop)
            assert torch.equal(V[lo:hi], W) and torch.equal(pi[lo:hi], pj), (i, most)
            assert st[i]["sweeps"] == sj["sweeps"] and (st[i]["termination"] == 2) == (sj["status"] != native.VC_OK)
            m.close()
    b.close()
