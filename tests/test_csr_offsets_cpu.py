"""The offsets with which a sparse row is cut into runs and chunks, up to 2^32 - 1
nonzeros: the functions the kernels use, compiled for the host (no GPU needed)."""
import os
import shutil
import subprocess

import pytest

from test_build_cpu import CSRC, ROOT

PROGRAM = r"""
#include "gfp_internal.h"
#include <cstdio>
using namespace gfp;
int main()
{
    const uint64_t top = 1ull << 32;
    uint64_t ns[400], count = 0;
    for (uint64_t d = 0; d < 130; ++d) {
        ns[count++] = d;
        ns[count++] = top - 1 - d;
        ns[count++] = (top >> 1) + d;
    }
    for (uint64_t i = 0; i < count; ++i)
        for (int S = 2; S <= 8; S *= 2) {
            const uint32_t n = (uint32_t)ns[i];
            uint64_t at = 0;   // the runs cover [0, n) in order, in steps of eight, evenly
            for (int sub = 0; sub < S; ++sub) {
                uint32_t x, y;
                csr_run(n, S, sub, x, y);
                if (x != at || y < x || y > n || (y < n && (y - x) % 8) ||
                    (uint64_t)(y - x) > n / S + (sub == S - 1 ? 72 : 8)) {
                    printf("n %u S %d sub %d: %u %u\n", n, S, sub, x, y);
                    return 1;
                }
                at = y;
            }
            if (at != n) return 2;
        }
    for (uint32_t d = 1; d <= 200; ++d) {   // the last chunks of the longest row
        uint32_t steps = 0;
        for (uint32_t q = CSR_NNZ_MAX - d; q < CSR_NNZ_MAX; q += 32)
            if (++steps > 10) return 3;
        if (steps != (d + 31) / 32) return 4;
    }
    return 0;
}
"""


def test_runs_and_chunks_up_to_2_32(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "offsets.cpp", tmp_path / "offsets"
    src.write_text(PROGRAM)
    inc = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-I", inc, "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                        str(src), "-o", str(exe), "-ldl"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, (r.returncode, r.stdout)
