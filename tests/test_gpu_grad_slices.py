"""The adjoint's sliced transpose, the contraction's sums and the model's row tally at their
edges: state counts below, at and across the slices of 32 rows, host bounds of each
instantiation (4, 8, 16).

dJ against the oracle's dense adjoint solve.  value_grad stops at max|(I - gamma P^T) lam - rho| <
1e-13, so lam is within 1e-13 S / (1 - gamma) of the exact one in the 1-norm; a derivative's
coefficients are at most max|dR| + gamma max|dV| sum|dp|, below 2 max|dJ| / max(rho) here, hence
a bound of S 1e-10 relative to the largest derivative."""
import numpy as np
import pytest

import oracle
from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 0), (1, 1, 3), (1, 2, 5), (2, 3, 2), (3, 2, 4), (4, 2, 1), (5, 1, 2), (8, 1, 0), (9, 1, 0)]


@pytest.mark.parametrize("H,C,Q", SHAPES)
def test_gradient_matches_the_dense_adjoint(H, C, Q):
    native = native_or_skip()
    import torch

    p = inputs.make_params(H, C, Q, 0.95, seed=30 + H)
    Vs, pis, _, _ = oracle.solve(p, tol=1e-12)
    S = len(Vs)
    rho = np.full(S, 1.0 / S)
    want = oracle.grad_dense(p, Vs, pis, rho)
    m = native.MDP.build(p)
    dev = lambda x, t: torch.tensor(np.asarray(x), device="cuda", dtype=t)  # noqa: E731
    args = dev(Vs, torch.float64), dev(pis, torch.int32), dev(rho, torch.float64)
    dJ, _, gs = m.value_grad(*args, tol=1e-13)
    assert np.max(np.abs(dJ.cpu().numpy() - want)) <= S * 1e-10 * np.max(np.abs(want))
    assert gs["J"] == pytest.approx(float(rho @ Vs), rel=1e-13)
    assert float(native.objective(args[0], args[2])) == pytest.approx(float(rho @ Vs), rel=1e-13)
    dJ2, _, _ = m.value_grad(*args, tol=1e-13)
    assert torch.equal(dJ, dJ2)  # fixed orders throughout
    m.close()


@pytest.mark.parametrize("H,C,Q", SHAPES + [(6, 2, 3)])
def test_implicit_tally_equals_the_stored_rows(H, C, Q):
    native = native_or_skip()
    p = inputs.make_params(H, C, Q, 0.95, seed=30 + H)
    a, b = native.MDP.build(p), native.MDP.build(p, fmt="csr_f32")
    for key in ("nnz_logical", "feasible_rows"):
        assert a.info()[key] == b.info()[key]
    a.close()
    b.close()
