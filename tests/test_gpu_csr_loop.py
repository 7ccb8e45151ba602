"""The resident FP32 loop over stored matrices against the launched sweeps, bit for bit.

A handle whose waits were capped keeps the launched kernels (``set_wait_limit`` with the default
number of polls), so one handle gives both: values, policy, residual and sweep count must be
equal.  Rows: ragged, empty and infeasible ones, an own-state entry, single and long rows; every
lane count per state; state counts that are no multiple of a chunk; one CTA and many; both value
types, both backups; and a stopped loop that goes on."""
import pytest

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu

DEFAULT_POLLS = 1 << 22


def _rows(S, A, K, seed, bf16):
    import torch

    g = torch.Generator(device="cuda").manual_seed(seed)
    rows = S * A
    n = torch.randint(1, K + 1, (rows,), generator=g, device="cuda")
    bad = torch.rand(rows, generator=g, device="cuda") < 0.2
    bad[::A] = False
    n[bad] = 0
    col = torch.randint(0, S, (rows, K), generator=g, device="cuda")
    col[:, 0] = torch.arange(rows, device="cuda") // A  # the row's own state
    col = col.sort(1).values
    live = torch.arange(K, device="cuda") < n[:, None]
    w = torch.where(live, torch.rand((rows, K), generator=g, device="cuda", dtype=torch.float64) + 0.05, 0.0)
    val = (w / w.sum(1, keepdim=True).clamp_min(1e-300)).to(torch.bfloat16 if bf16 else torch.float32)
    R = torch.rand(rows, generator=g, device="cuda") * 2 - 1
    R[bad] = float("-inf")
    row_ptr = torch.zeros(rows + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(n, 0, out=row_ptr[1:])
    return row_ptr, col[live].to(torch.int32), val[live], R


@pytest.mark.parametrize("S,A,K", [(1, 1, 1), (3, 2, 2), (31, 1, 7), (33, 3, 16), (1001, 5, 17), (4099, 4, 12),
                                   (20011, 9, 5), (3001, 17, 33), (2003, 32, 4), (60013, 2, 40)])
@pytest.mark.parametrize("bf16", [False, True])
def test_loop_equals_launched_sweeps(S, A, K, bf16):
    native = native_or_skip()
    import torch

    m = native.MDP.from_csr(S, A, *_rows(S, A, K, S + A, bf16), 0.95)
    g = torch.Generator(device="cuda").manual_seed(3)
    start = torch.rand(S, device="cuda", generator=g) * 40
    for self_loop in (False, True):
        for k in (1, 2, 67):  # 67: past the 64 slots of the residual ring
            out = []
            for polls in (-1, DEFAULT_POLLS):
                m.set_wait_limit(polls)
                V, _, pi, st = m.value_iterate(V=start.clone(), tol=1e-30, max_sweeps=k, fp32_only=True,
                                               want_v64=False, raise_on_nonconvergence=False, self_loop=self_loop)
                out.append((V, pi, st["sweeps"], st["residual"]))
            assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
            assert out[0][2:] == out[1][2:]
    m.set_wait_limit(-1)
    kw = dict(tol=1e-30, fp32_only=True, want_v64=False, raise_on_nonconvergence=False, self_loop=True)
    half = m.value_iterate(V=start.clone(), max_sweeps=30, **kw)[0]
    assert torch.equal(m.value_iterate(V=half, max_sweeps=37, **kw)[0], out[0][0])
    m.close()


@pytest.mark.parametrize("fmt,padded", [("csr_f32", True), ("csr_f32", False), ("csr_bf16", True)])
@pytest.mark.parametrize("H,C,Q", [(3, 3, 4), (5, 3, 6), (7, 2, 4)])
def test_model_rows(H, C, Q, fmt, padded):
    native = native_or_skip()
    import torch

    from paper_2012_12419_gb300 import inputs

    m = native.MDP.build(inputs.make_params(H, C, Q, 0.95, seed=9), fmt=fmt, padded=padded)
    for self_loop in (False, True):
        out = []
        for polls in (-1, DEFAULT_POLLS):
            m.set_wait_limit(polls)
            V, V64, pi, st = m.value_iterate(tol=1e-6, self_loop=self_loop)
            out.append((V, V64, pi, st["sweeps"]))
        assert all(torch.equal(x, y) for x, y in zip(out[0][:3], out[1][:3])) and out[0][3] == out[1][3]
    m.close()
