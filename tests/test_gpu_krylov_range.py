"""Dot products of the correction solve beyond FP32's range.

Scaling rewards and tolerance by a power of two commutes with every rounding of the solve as
long as nothing over- or underflows, so the values scale exactly and the product count stays.  At
2^62 each state's square (2^124) still fits FP32 and the sum over a CTA's states (130 and 2,040
here, one CTA for the smallest) does not: the sums have to carry FP64's range.
"""
import pytest
import torch

from gpu_common import native_or_skip
from test_gpu_krylov_resident import _user

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,A,K", [(2000, 2, 6), (20001, 2, 8), (310001, 1, 5)])
def test_scaled_rewards(S, A, K):
    native = native_or_skip()
    gamma, tol, base, up = 0.95, 1e-8, 2.0**30, 2.0**32
    rp, col, val, R = _user(S, A, K, S + K)
    pi = (torch.arange(S, device="cuda") % A).to(torch.int32)
    out = []
    for scale in (base, base * up):
        m = native.MDP.from_csr(S, A, rp, col, val, R * scale, gamma)
        out.append(m.evaluate_policy(pi, tol=tol * scale))
        m.close()
    assert out[0][1] == out[1][1] > 0
    assert torch.equal(out[0][0] * up, out[1][0])
