"""The partial sums of the resident BiCGSTAB kernel under every order in which two CTAs can run.

A stage stores a CTA's partials in a set of the buffer, passes one grid barrier and reads all
CTAs' partials; a product adds a barrier of its own before its stage (V and T), the x / r update
before stage X none.  The set of each stage comes from the kernel's own header, compiled here;
a search over the interleavings of two CTAs then checks that every read finds the partials of its
own stage and iteration.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2012_12419_gb300", "csrc")
STAGES = ("kKrInit", "kKrV", "kKrT", "kKrX")


def _sets(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "sets.cu"
    src.write_text('#include <stdio.h>\n#include "vc_krylov.cuh"\nint main() {\n'
                   + "".join(f'    printf("%d ", vc::kr_part_set(vc::{s}));\n' for s in STAGES)
                   + '    printf("%d\\n", vc::kKrPartSets);\n}\n')
    exe = tmp_path / "sets"
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", CSRC, "-I",
                        os.path.join(ROOT, "include"), str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    v = [int(x) for x in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()]
    assert all(0 <= s < v[-1] for s in v[:-1])
    return dict(zip(STAGES, v))


def _program(sets, iterations=3):
    """One CTA's steps: ("w" | "r", set, token) and ("b",) for a grid barrier."""
    def reduce(stage, it):
        token = (stage, it)
        return [("w", sets[stage], token), ("b",), ("r", sets[stage], token)]

    steps = reduce("kKrInit", 0)
    for it in range(iterations):
        steps += [("b",)] + reduce("kKrV", it) + [("b",)] + reduce("kKrT", it) + reduce("kKrX", it)
    return steps


def _misread(steps):
    """First wrong read over all interleavings of two CTAs, or None."""
    nbar = [0]
    for s in steps:
        nbar.append(nbar[-1] + (s[0] == "b"))
    start = (0, 0, ((), ()))  # program counters, what each CTA last stored per set
    seen, todo = {start}, [start]
    while todo:
        pc0, pc1, mem = todo.pop()
        for me in (0, 1):
            pc, other = (pc0, pc1) if me == 0 else (pc1, pc0)
            if pc == len(steps):
                continue
            kind = steps[pc][0]
            now = list(mem)
            if kind == "b":
                # passes once the other CTA has arrived: it stands at this barrier or beyond it
                if nbar[other] < nbar[pc] or (nbar[other] == nbar[pc] and (other == len(steps) or steps[other][0] != "b")):
                    continue
            elif kind == "w":
                now[me] = tuple(sorted({**dict(mem[me]), steps[pc][1]: steps[pc][2]}.items()))
            else:
                for cta in (0, 1):
                    got = dict(mem[cta]).get(steps[pc][1])
                    if got != steps[pc][2]:
                        return steps[pc], got
            nxt = (pc0 + (me == 0), pc1 + (me == 1), tuple(now))
            if nxt not in seen:
                seen.add(nxt)
                todo.append(nxt)
    return None


def test_search_finds_a_shared_set():
    """One set for every stage is what the search has to reject: T's late readers meet X's writers."""
    bad = _misread(_program(dict.fromkeys(STAGES, 0)))
    assert bad is not None and bad[0][2][0] == "kKrT" and bad[1][0] == "kKrX"


def test_partials_survive_every_interleaving(tmp_path):
    assert _misread(_program(_sets(tmp_path))) is None
