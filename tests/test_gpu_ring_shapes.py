"""Every launch shape of the sliced ring sweep, by the number of actions (units of one and of two
actions, odd counts, and the count at which 24 warps claim units as far ahead as allowed): with
one slice a tile (which fits every ring here) all shapes are offered that one action a unit allows, and
each gives the direct sliced kernel's sweep bit
for bit, for rows of a model and of a user's matrix, both value types and both backups."""
import pytest
import torch

from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip
from test_gpu_csr_loop import _rows

pytestmark = pytest.mark.gpu

# warps per CTA of the planner's shapes, and the tiles a claim may run ahead (kSlots - 2)
WARPS, AHEAD = (12, 16, 10, 24, 8, 8), 10


@pytest.mark.parametrize("source", ["model", "user"])
@pytest.mark.parametrize("A", [2, 3, 4, 5, 8])
@pytest.mark.parametrize("bf16", [False, True])
def test_shapes_agree(source, A, bf16):
    native = native_or_skip()
    fmt = "csr_bf16" if bf16 else "csr_f32"
    if source == "model":
        C = {2: 60, 3: 30, 4: 9, 5: 6, 8: 2}[A]
        m = native.MDP.build(inputs.make_params(A - 1, C, 9, 0.95, seed=A), fmt=fmt, sliced=True)
    else:
        m = native.MDP.from_csr(20011, A, *_rows(20011, A, 9, A, bf16), 0.95).slice()
    V = torch.rand(m.S, device="cuda") * 50
    kw = dict(tol=1e-30, fp32_only=True, want_v64=False, raise_on_nonconvergence=False)
    ref, tried = None, 0
    for k in reversed(range(m.schedules())):  # the direct sliced kernel comes last
        m.use_schedule(k)
        info = m.info()
        if not info["csr_sliced"]:
            break
        out = [m.bellman32(V, torch.empty_like(V))]
        pi = torch.empty(m.S, dtype=torch.int32, device="cuda")
        out += [m.bellman32(V, torch.empty_like(V), pi), pi]
        out += [m.value_iterate(V=V.clone(), max_sweeps=3, self_loop=sl, **kw)[0] for sl in (False, True)]
        if ref is None:
            assert not info["csr_pipelined"]
            ref = out
        assert all(torch.equal(a, b) for a, b in zip(ref, out)), (k, info)
        tried += info["csr_pipelined"] == 1 and info["csr_tile_states"] == 32
    assert tried == sum(1 for w in WARPS if w <= AHEAD * A)
    m.close()
