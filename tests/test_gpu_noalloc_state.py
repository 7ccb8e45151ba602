"""The no-allocation sweep owes nothing to what an earlier call left behind: with its residual words
overwritten (a hook of the bounds-checking build, in a child process) the next call still returns
max|V_out - V|, for a ticket below, at and beyond the grid and a residual larger than its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import ctypes
import sys
import torch
sys.path.insert(0, ROOT)
from paper_2012_12419_gb300 import inputs, native

L = native.load(build_if_missing=True)
assert L._name.endswith("libvcmdp_debug.so"), L._name
for H, C, Q in ((1, 1, 1), (3, 3, 4), (5, 3, 15)):
    p = inputs.make_params(H, C, Q, 0.95, seed=7)
    S = inputs.num_states(H, C, Q)
    V = torch.rand(S, device="cuda") * 50
    out = torch.empty_like(V)
    for residual in (0, 0x7F7FFFFF):
        for ticket in (0, 1, 7, 100000, 0xFFFFFFFF):
            torch.cuda.synchronize()
            assert L.vc_debug_noalloc_words(ctypes.c_uint32(residual), ctypes.c_uint32(ticket)) == 0
            for _ in range(2):
                res = torch.full((1,), -1.0, device="cuda")
                native.bellman32_noalloc(p, V, out, None, res)
                torch.cuda.synchronize()
                assert res.item() == (out - V).abs().max().item(), (H, C, Q, residual, ticket, res.item())
print("noalloc state ok")
""".replace("ROOT", repr(ROOT))


def test_residual_words_are_cleared_by_the_call():
    env = dict(os.environ, VC_DEBUG_BOUNDS="1")
    r = subprocess.run([sys.executable, "-c", SCRIPT], env=env, capture_output=True, text=True, timeout=1200)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "noalloc state ok" in r.stdout
