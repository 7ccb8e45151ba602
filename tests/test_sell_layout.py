"""Region offsets of slice records, from the sweeps' own header compiled for the host: the offsets
that a sweep forms from a stored record must be those the record was laid out with, whatever its
length -- for a record in global memory also beyond 2^31 bytes (one row of 16.8 M entries is
enough), for one in shared memory up to what a ring can hold."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2012_12419_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include "vc_sell.cuh"
int main() {
    const long long all[] = {0, 1, 7, 400, 16777215, 16777216, 16800000, 67108864, 2147483647};
    for (long long rows : all)
        for (int A : {1, 5, 31})
            for (int scale = 0; scale < 2; scale++) {
                int32_t hdr[32] = {};
                hdr[A] = (int32_t)rows;
                const unsigned char* rec = reinterpret_cast<const unsigned char*>(hdr);
                const vc::RecLayout L = vc::rec_layout(A, rows, scale ? 2 : 4, scale != 0);
                const auto p = vc::rec_at<long long>(rec, A, scale != 0);
                if (p.rows != rows || p.scale != L.scale || p.col != L.col || p.val != L.val) {
                    printf("rows %lld A %d scale %d: %lld %lld\n", rows, A, scale, (long long)p.val, L.val);
                    return 1;
                }
                if (rows > 400) continue;
                const auto q = vc::rec_at<int>(rec, A, scale != 0);
                if (q.rows != rows || q.scale != L.scale || q.col != L.col || q.val != L.val) return 2;
            }
    return 0;
}
"""


def test_record_offsets(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "rec.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "rec"
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
