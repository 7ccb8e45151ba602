"""Small instances that outlast the large ones: the resident batched loop leaves those of at most
4,096 states to the whole-instance kernel once no larger one is active.  Values and sweep counts must
be those of each instance's own solve, bit for bit, whether an even or an odd number of sweeps was
done before, with instances at the limit and just above it, a loop that max_sweeps ends in either
part, and the path switched off or limited."""
import pytest
import torch

from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu

# (H, C, Q, gamma): 640, 4,096 and 4,608 states that converge slowly, 20,000 quickly; 18,432 last
SLOW = [(3, 3, 4, 0.99), (3, 7, 3, 0.99), (2, 15, 8, 0.985), (1, 1, 0, 0.99)]
CASES = {"above": SLOW + [(4, 4, 15, 0.9)], "below": SLOW[:2] + [(4, 4, 15, 0.9)], "late": SLOW[:1] + [(4, 4, 15, 0.9), (5, 3, 8, 0.995)]}


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("self_loop", [False, True])
def test_equal_to_single_solves(case, self_loop):
    native = native_or_skip()
    ps = [inputs.make_params(H, C, Q, g, seed=30 + i) for i, (H, C, Q, g) in enumerate(CASES[case])]
    b = native.Batch(ps)
    kw = dict(tol=1e-6, fp32_only=True, raise_on_nonconvergence=False, self_loop=self_loop)
    singles = [native.MDP.build(p) for p in ps]
    for limit in (1 << 20, 0, 1000):
        b.set_small_instances(limit)
        for most in (1_000_000, 1, 150, 151):
            V, _, _, st, _ = b.value_iterate(max_sweeps=most, **kw)
            for i, m in enumerate(singles):
                W, _, _, sj = m.value_iterate(max_sweeps=most, **kw)
                assert torch.equal(V[int(b.offsets[i]):int(b.offsets[i + 1])], W), (limit, most, i)
                assert st[i]["sweeps"] == sj["sweeps"], (limit, most, i)
    # warm start: the quick one is done at once and the rest goes over after a sweep or none
    V, V64, pi, st, _ = b.value_iterate(V=V.clone(), tol=1e-6, self_loop=self_loop)
    assert all(s["certified"] == 1 for s in st)
    for m in singles:
        m.close()
    b.close()
