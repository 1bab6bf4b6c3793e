"""CPU test of the grid-stride loop that the 64-bit histogram takes its keys by: every
index of [0, n) once, up to the largest n (2^32 - 1), where the next index of a step
does not fit 32 bits.  The loop is compiled for the host from the kernels' own header."""
from __future__ import annotations

import subprocess

import pytest

from paper_1008_2849_gb300 import build

# For every thread of a grid of `gsize` threads with `loads` keys each a step: its last
# steps' indices near n, which must be in order and below n; the steps in all, and of
# the indices from `tail` on how often each is taken.
PROGRAM = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "rs_device.cuh"
int main(int, char** a) {
    const uint32_t gsize = strtoul(a[1], 0, 0), loads = strtoul(a[2], 0, 0);
    const uint32_t n = strtoul(a[3], 0, 0);
    const uint32_t tail = n > 3 * loads * gsize ? n - 3 * loads * gsize : 0;
    std::vector<unsigned char> taken(n - tail, 0);
    uint64_t all = 0;
    for (uint32_t t = 0; t < gsize; ++t) {
        uint64_t steps = 0, before = 0;
        const uint64_t most = (uint64_t)n / (loads * gsize) + 1;
        bool bad = false;
        rs::strided(t, loads * gsize, n, [&](uint32_t i, uint32_t left) {
            if (++steps > most || (steps > 1 && i <= before) || left != n - i) bad = true;
            if (bad) { puts("out of order"); exit(1); }
            before = i;
            if (left > loads * gsize && i + loads * gsize <= tail) {
                all += loads;
                return;
            }
            for (uint32_t u = 0; u < loads; ++u)
                if (u * gsize < left) {
                    ++all;
                    const uint32_t at = i + u * gsize;
                    if (at >= tail) ++taken[at - tail];
                }
        });
    }
    for (unsigned char c : taken) if (c != 1) { puts("not once"); return 1; }
    if (all != n) { puts("count"); return 1; }
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("strided")
    src = d / "strided.cu"
    src.write_text(PROGRAM)
    exe = d / "strided"
    subprocess.run([build.nvcc(), "-O2", "-std=c++17", "--expt-extended-lambda", *build.ARCH, "-I",
                    build.CSRC, str(src), "-o", str(exe), "-cudart", "static"], check=True)
    return str(exe)


@pytest.mark.parametrize("gsize,loads", [(152 * 1024, 4), (304 * 512, 4)])
@pytest.mark.parametrize("n", [1, 1000, (1 << 32) - 622_592, (1 << 32) - 622_591,
                               (1 << 32) - 400_000, (1 << 32) - 155_649, (1 << 32) - 2,
                               (1 << 32) - 1])
def test_strided_takes_every_index_once(program, gsize, loads, n):
    res = subprocess.run([program, str(gsize), str(loads), str(n)], capture_output=True, text=True,
                         timeout=300)
    assert res.returncode == 0, res.stdout
