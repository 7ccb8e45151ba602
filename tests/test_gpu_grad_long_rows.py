"""Transposed rows longer than a lane orders alone (32 entries): hosts of many slots, whose departures
all lead to the empty host, at the limit and far beyond it, next to short rows in the same slice.
dJ against the oracle's dense adjoint solve with the bound derived in test_gpu_grad_slices (S 1e-10
relative), and bitwise equal when repeated: the rows are filled in an order that varies, so only
complete and correctly ordered rows give the same sums twice."""
import numpy as np
import pytest

import oracle
from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,C,Q", [(1, 14, 1), (1, 15, 1), (1, 16, 0), (1, 31, 0), (1, 200, 1), (1, 1000, 0), (2, 20, 0)])
def test_gradient_matches_the_dense_adjoint(H, C, Q):
    native = native_or_skip()
    import torch

    p = inputs.make_params(H, C, Q, 0.9, seed=50 + C)
    Vs, pis, _, _ = oracle.solve(p, tol=1e-12)
    S = len(Vs)
    rho = np.full(S, 1.0 / S)
    want = oracle.grad_dense(p, Vs, pis, rho)
    m = native.MDP.build(p)
    dev = lambda x, t: torch.tensor(np.asarray(x), device="cuda", dtype=t)  # noqa: E731
    args = dev(Vs, torch.float64), dev(pis, torch.int32), dev(rho, torch.float64)
    dJ, lam, _ = m.value_grad(*args, tol=1e-13, want_lambda=True)
    assert np.max(np.abs(dJ.cpu().numpy() - want)) <= S * 1e-10 * np.max(np.abs(want))
    for _ in range(3):
        dJ2, lam2, _ = m.value_grad(*args, tol=1e-13, want_lambda=True)
        assert torch.equal(dJ, dJ2) and torch.equal(lam, lam2)
    m.close()
