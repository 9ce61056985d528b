"""Bits of a record taken as an index by the grouping passes, on the CPU: the function's own text, compiled
for the host with CUDA's funnel shifts spelled out, is defined and exact for every shift that a plan can ask
for -- up to 64, where a record fills its word and its prefix is not split."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <stdint.h>
#include <stdio.h>
#define __device__ static
#define __forceinline__ inline
// CUDA's definitions: the shift taken mod 32, or clamped to 32
static uint32_t __funnelshift_r(uint32_t lo, uint32_t hi, uint32_t s) {
    return (uint32_t)(((((uint64_t)hi) << 32) | lo) >> (s & 31u));
}
static uint32_t __funnelshift_rc(uint32_t lo, uint32_t hi, uint32_t s) {
    return (uint32_t)(((((uint64_t)hi) << 32) | lo) >> (s < 32u ? s : 32u));
}
%s
int main() {
    const uint64_t xs[] = {0ull, 1ull, ~0ull, 0x123456789abcdef0ull, 0x8000000000000001ull, 0xffffffff00000000ull};
    for (uint64_t x : xs)
        for (volatile int s = 0; s <= 64; s++) {
            const uint32_t want = s < 64 ? (uint32_t)(x >> s) : 0u, got = low_bits_at(x, s);
            if (got != want) {
                printf("x %%llx s %%d: %%x, not %%x\n", (unsigned long long)x, s, got, want);
                return 1;
            }
        }
    return 0;
}
"""


@pytest.mark.skipif(not shutil.which("g++"), reason="needs g++")
def test_every_shift(tmp_path):
    text = open(os.path.join(ROOT, "paper_2010_10055_gb300", "csrc", "bucket.cuh")).read()
    fn = re.search(r"__device__ __forceinline__ uint32_t low_bits_at\(.*?\n}\n", text, re.S).group(0)
    src, exe = tmp_path / "bits.cpp", tmp_path / "bits"
    src.write_text(MAIN % fn)
    subprocess.run(["g++", "-O0", "-std=c++17", "-fsanitize=undefined", "-fsanitize-undefined-trap-on-error",
                    str(src), "-o", str(exe)], check=True)
    p = subprocess.run([str(exe)], capture_output=True, text=True)
    assert p.returncode == 0, p.stdout or p.returncode
