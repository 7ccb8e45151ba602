"""The resident BiCGSTAB kernel at the edges of its dispatch, against FP64 residuals.

``evaluate_policy`` returns once max|T_pi V - V| < tol in FP64 (k_resid64), so its values are
within tol / (1 - gamma) of V_pi.  Both of two evaluations with different correction solvers
(BiCGSTAB against FP64 fixed-point sweeps of torch on the exported rows) therefore agree within
2 tol / (1 - gamma), plus FP64 rounding of the rows' FP32 probabilities (the stored rows are
what both use).  Sizes: one CTA and the first grids beyond it, ragged row counts, both widths of
the two-pass product (Q odd / even) with H below, at and above 8 hosts.
"""
import numpy as np
import pytest
import torch

from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu


def _user(S, A, K, seed, bf16=False):
    g = torch.Generator(device="cuda").manual_seed(seed)
    col = torch.randint(0, S, (S * A, K), generator=g, device="cuda").sort(1).values
    w = torch.rand((S * A, K), generator=g, device="cuda", dtype=torch.float64) + 0.05
    val = (w / w.sum(1, keepdim=True)).to(torch.bfloat16 if bf16 else torch.float32)
    R = torch.rand(S * A, generator=g, device="cuda") * 2 - 1
    rp = torch.arange(S * A + 1, device="cuda", dtype=torch.int64) * K
    return rp, col.to(torch.int32).reshape(-1), val.reshape(-1), R


@pytest.mark.parametrize("S,A,K,bf16", [(1, 1, 1, False), (33, 2, 3, False), (2048, 3, 5, False), (2049, 3, 9, False),
                                        (20001, 2, 17, False), (20001, 2, 17, True), (310001, 2, 8, False)])
def test_stored_rows(S, A, K, bf16):
    native = native_or_skip()
    gamma, tol = 0.95, 1e-10
    rp, col, val, R = _user(S, A, K, S + K, bf16)
    m = native.MDP.from_csr(S, A, rp, col, val, R, gamma)
    pi = (torch.arange(S, device="cuda") % A).to(torch.int32)
    V, n = m.evaluate_policy(pi, tol=tol)
    rows = torch.arange(S, device="cuda") * A + pi
    c = col.reshape(-1, K)[rows].long()
    p = val.reshape(-1, K).to(torch.float64)[rows]
    if bf16:
        p = p * (1 / p.sum(1, keepdim=True)).to(torch.float32).to(torch.float64)
    r = R.to(torch.float64)[rows]
    W = torch.zeros(S, dtype=torch.float64, device="cuda")
    for _ in range(700):  # 0.95^700 / (1 - 0.95) < 1e-13
        W = r + gamma * (p * W[c]).sum(1)
    assert float((V - W).abs().max()) <= 2 * tol / (1 - gamma)
    assert n > 0
    m.close()


# H, C, Q: 1 host; one CTA; the two-pass product with Q odd (items of 4), Q even (items of 2)
# and more than 8 hosts (items of 2 and the wide host bound)
@pytest.mark.parametrize("H,C,Q", [(1, 1, 1), (2, 2, 5), (3, 3, 4), (3, 6, 5), (5, 4, 14), (5, 4, 15), (6, 4, 6), (7, 3, 15), (7, 3, 20),
                                   (8, 3, 5), (9, 3, 2)])
def test_model_products(H, C, Q):
    native = native_or_skip()
    gamma, tol = 0.95, 1e-10
    p = inputs.make_params(H, C, Q, gamma, seed=H + C + Q)
    m = native.MDP.build(p, fmt="implicit")
    pi = m.greedy_policy()
    V, n = m.evaluate_policy(pi, tol=tol)
    V2, n2 = m.evaluate_policy(pi, tol=tol)
    assert torch.equal(V, V2) and n == n2  # fixed order: bitwise reproducible
    # the FP64 Bellman backup of the policy's values: T V >= V up to the residual, and equal to
    # it where the backup's argmax is the policy's own action
    T, arg, _, _ = m.bellman64(V)
    same = arg == pi
    assert float((V - T).max()) <= tol
    assert bool(same.any())
    assert float((T - V)[same].abs().max()) <= tol
    m.close()
