"""The bounded waits of the resident kernels run out without a GPU fault: capped at 0 polls from
the host, a grid-barrier wait of the implicit loop, of the correction solve (a policy's evaluation,
the adjoint of the gradient) and of the batched loop, and a staging wait of the stored-matrix loop,
ends its call with VC_ERR_TIMEOUT; the same handle then gives the results of an untouched one, bit
for bit.  The last two are reached in the bounds-checking build only (a child process): in the
normal one a cap keeps a stored matrix on the launched sweeps and a batch has no cap."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BIG = inputs.make_params(5, 3, 15, 0.95, seed=7)  # 32,768 states: many CTAs in both loops


def _refused(native, call):
    with pytest.raises(native.VcError) as e:
        call()
    assert e.value.code == native.VC_ERR_TIMEOUT


@pytest.mark.parametrize("self_loop", [False, True])
def test_implicit_loop(self_loop):
    native = native_or_skip()
    m = native.MDP.build(BIG)
    ref = m.value_iterate(tol=1e-6, self_loop=self_loop)
    m.set_wait_limit(0)
    _refused(native, lambda: m.value_iterate(tol=1e-6, self_loop=self_loop, fp32_only=True))
    m.set_wait_limit(-1)
    got = m.value_iterate(tol=1e-6, self_loop=self_loop)
    assert all(torch.equal(a, b) for a, b in zip(ref[:3], got[:3])) and ref[3]["sweeps"] == got[3]["sweeps"]
    m.close()


def test_correction_solve_and_adjoint():
    native = native_or_skip()
    m = native.MDP.build(BIG)
    pi = m.greedy_policy()
    rho = torch.full((m.S,), 1.0 / m.S, dtype=torch.float64, device="cuda")
    V, n = m.evaluate_policy(pi, tol=1e-8)
    dJ, _, _ = m.value_grad(V, pi, rho, tol=1e-9)
    m.set_wait_limit(0)
    _refused(native, lambda: m.evaluate_policy(pi, tol=1e-8))
    _refused(native, lambda: m.value_grad(V, pi, rho, tol=1e-9))
    m.set_wait_limit(-1)
    V2, n2 = m.evaluate_policy(pi, tol=1e-8)
    assert torch.equal(V, V2) and n == n2
    assert torch.equal(dJ, m.value_grad(V, pi, rho, tol=1e-9)[0])
    m.close()


SCRIPT = r"""
import ctypes
import sys
import torch
sys.path.insert(0, ROOT)
from paper_2012_12419_gb300 import inputs, native

L = native.load(build_if_missing=True)
assert L._name.endswith("libvcmdp_debug.so"), L._name


def refused(call):
    try:
        call()
    except native.VcError as e:
        assert e.code == native.VC_ERR_TIMEOUT, e
        return
    raise AssertionError("the capped wait did not give up")


for fmt in ("csr_f32", "csr_bf16"):
    m = native.MDP.build(inputs.make_params(5, 3, 15, 0.95, seed=7), fmt=fmt, padded=True)
    ref = m.value_iterate(tol=1e-6, fp32_only=True)
    m.set_wait_limit(0)
    refused(lambda: m.value_iterate(tol=1e-6, fp32_only=True))
    m.set_wait_limit(-1)
    got = m.value_iterate(tol=1e-6, fp32_only=True)
    assert torch.equal(ref[0], got[0]) and ref[3]["sweeps"] == got[3]["sweeps"]
    m.close()
b = native.Batch([inputs.make_params(H, C, Q, 0.95, seed=i) for i, (H, C, Q) in
                  enumerate([(5, 3, 15), (3, 3, 4), (4, 5, 7), (2, 6, 12)])])
for sl in (False, True):
    ref = b.value_iterate(tol=1e-6, self_loop=sl)
    assert L.vc_debug_batch_wait_limit(b._h, ctypes.c_int64(0)) == 0
    refused(lambda: b.value_iterate(tol=1e-6, self_loop=sl))
    assert L.vc_debug_batch_wait_limit(b._h, ctypes.c_int64(-1)) == 0
    got = b.value_iterate(tol=1e-6, self_loop=sl)
    assert all(torch.equal(x, y) for x, y in zip(ref[:3], got[:3]))
    assert [s["sweeps"] for s in ref[3]] == [s["sweeps"] for s in got[3]]
b.close()
print("wait limits ok")
""".replace("ROOT", repr(ROOT))


def test_stored_matrix_and_batched_loops():
    env = dict(os.environ, VC_DEBUG_BOUNDS="1")
    r = subprocess.run([sys.executable, "-c", SCRIPT], env=env, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "wait limits ok" in r.stdout
