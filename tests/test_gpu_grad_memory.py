"""Temporary device memory of the gradient, from the device pool's high-water mark: 16 bytes an entry
of the padded transpose (its padding at most 2.2 times the entries for rows of this shape), the rows'
own arrays (24 bytes a state) and 64 MB of scratch, not a second copy of the transpose."""
import ctypes

import pytest
import torch

from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu

USED_MEM_HIGH = 8  # CUmemPool_attribute


def test_peak_of_the_pool():
    native = native_or_skip()
    m = native.MDP.build(inputs.make_params(6, 5, 10, 0.9, seed=4))
    _, V64, pi, _ = m.value_iterate(tol=1e-6)
    rho = torch.full((m.S,), 1.0 / m.S, dtype=torch.float64, device="cuda")
    cu = ctypes.CDLL("libcuda.so.1")
    pool, v = ctypes.c_void_p(), ctypes.c_uint64(0)
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), ctypes.c_int(torch.cuda.current_device())) == 0
    torch.cuda.synchronize()
    assert cu.cuMemPoolSetAttribute(pool, USED_MEM_HIGH, ctypes.byref(v)) == 0
    gs = m.value_grad(V64, pi, rho, tol=1e-9)[2]
    assert cu.cuMemPoolGetAttribute(pool, USED_MEM_HIGH, ctypes.byref(v)) == 0
    bound = 16 * 2.2 * gs["nnz_transpose"] + 24 * m.S + (64 << 20)
    assert 16 * gs["nnz_transpose"] < v.value <= bound < 28 * 1.9 * gs["nnz_transpose"]
    m.close()
