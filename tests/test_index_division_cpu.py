"""The kernels' division by a fixed extent equals integer division over its whole range.

FastDiv (lbpc_internal.h) replaces n / d for 0 <= n < 2^31, 1 <= d < 2^31 by one high product.
Compiled as host code; every divisor up to 4096, the neighbours of powers of two and seeded
ones up to 2^31 - 1, each at the multiples of d and their predecessors, where a wrong
reciprocal shows first, and at the ends of the range.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdint>
#include <cstdio>
#include "lbpc_internal.h"
static uint64_t st = 12345;
static uint32_t rnd() { st = st * 6364136223846793005ULL + 1442695040888963407ULL; return st >> 33; }
static long bad = 0;
static void check(uint32_t d) {
    const lbpc::FastDiv f = lbpc::fast_div((int)d);
    const uint32_t top = 0x7fffffffu;
    for (int i = 0; i < 40; i++) {
        const uint32_t m = rnd() / d * d;
        const uint32_t ns[6] = {0, m, m ? m - 1 : 0, top, top - top % d, top / d * d ? top / d * d - 1 : 0};
        for (uint32_t n : ns) bad += f.div(n) != n / d;
    }
}
int main() {
    for (uint32_t d = 1; d <= 4096; d++) check(d);
    for (int b = 1; b < 31; b++) { check((1u << b) - 1); check(1u << b); check((1u << b) + 1); }
    check(0x7fffffffu);
    for (int i = 0; i < 20000; i++) check(1 + rnd() % 0x7fffffffu);
    printf("%ld\n", bad);
    return 0;
}
"""


def test_fast_division_is_exact(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "div.cu", tmp_path / "div"
    src.write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_1703_02652_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert out.strip() == "0"
