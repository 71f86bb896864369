"""Blocks of the reduction jobs (csrc/exa_reduce.h), compiled for the host: every element is covered, up to the
largest 32-bit counts."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_16265_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
MAIN = r'''
#include <cstdio>
#include "exa_reduce.h"
using namespace exa_red;
int main() {
    const int big = 0x7fffffff;
    for (int sms : {100, 152})
    for (int kind : {PERM, SEG, WSEG, CSUM, CHUNK, BSEG, FILL})
        for (int n : {1, 7, 8, 9, 255, 256, 257, 511, 512, 513, 8192, 8193, 152 * 2 * 512 - 1, 152 * 2 * 512, 152 * 2 * 2048 - 1,
                      152 * 2 * 2048, 1000000007, big - 4096, big - 2047, big - 31, big - 7, big}) {
            Job j;
            j.kind = kind;
            j.n = n;
            j.lo = kind == FILL ? n / 3 : 0;
            const long long b = plan(j, sms);
            long long per = kind == PERM ? (j.wide ? 2048 : 512) : kind == SEG ? (j.wide ? 512 : 256)
                            : kind == WSEG || kind == CSUM ? 8 : kind == FILL ? 8192 : 1;
            const long long first = kind == FILL ? j.lo / 32 * 32 : 0;  // whole mask words
            if ((kind == PERM && j.wide != (n >= 2LL * sms * 2048)) || (kind == SEG && j.wide != (n >= 2LL * sms * 512))) return 2;
            if (b < 1 || first + b * per < n || first + (b - 1) * per >= n) { std::printf("kind %d n %d: %lld\n", kind, n, b); return 1; }
        }
    return 0;
}
'''


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_blocks_cover_every_element(tmp_path):
    src = tmp_path / "plan.cu"
    src.write_text(MAIN)
    exe = tmp_path / "plan"
    subprocess.run([NVCC, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
