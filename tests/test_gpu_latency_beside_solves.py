"""A control loop's sweep beside long solves: with two threads solving without pause on streams of
their own, a no-allocation sweep on a third stream waits for the launch that runs and no longer.
A launch lasts at most 8 ms (8 M cycles at 1 GHz or more), the sweep's two kernels may each meet one,
and the host reads in between: 40 ms.  (Queued on the device without turns, the solves' launches let
it wait for the rest of a solve: 250 ms.)  The solves' results are those of a thread alone."""
import threading
import time

import pytest
import torch

from paper_2012_12419_gb300 import inputs

from gpu_common import native_or_skip

pytestmark = pytest.mark.gpu


def test_latency_of_a_sweep():
    native = native_or_skip()
    solve = dict(tol=1e-9, max_sweeps=20000, fp32_only=True, want_v64=False, want_pi=False, raise_on_nonconvergence=False)
    ms = [native.MDP.build(inputs.make_params(6, 4, 10, 0.9999, seed=i)) for i in range(2)]
    refs = [m.value_iterate(**solve)[0] for m in ms]
    p = inputs.make_params(4, 4, 6, 0.95, seed=1)
    V = torch.rand(inputs.num_states(4, 4, 6), device="cuda")
    W, r = torch.empty_like(V), torch.empty(1, device="cuda")
    native.bellman32_noalloc(p, V, W, None, r)
    torch.cuda.synchronize()
    stop, wrong, solves = threading.Event(), [], [0, 0]

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            while not stop.is_set():
                out = ms[i].value_iterate(**solve)[0]
                if not torch.equal(out, refs[i]):
                    wrong.append(i)
                solves[i] += 1

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    time.sleep(0.3)
    waits = []
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        for _ in range(100):
            t0 = time.perf_counter()
            native.bellman32_noalloc(p, V, W, None, r)
            while not st.query():
                time.sleep(0.0002)
            waits.append(1e3 * (time.perf_counter() - t0))
            time.sleep(0.004)
    stop.set()
    for t in threads:
        t.join()
    assert not wrong and min(solves) > 0
    assert max(waits) <= 40.0, sorted(waits)[-10:]
    for m in ms:
        m.close()
