"""window_to_double_seldom (tc_ptx.cuh), the rounding of the Cholesky's epilogue, on
the host against window_to_double: the same bits for every window and exponent."""
import shutil
import subprocess

import pytest

from test_fixed_point_cpu import HEADER

HARNESS = r"""
#include <cstdio>
#include <cstdint>
#include <cstring>
#include <random>
#define __host__
#define __device__
#define __forceinline__ inline
%s
int main() {
    std::mt19937_64 g(5);
    long bad = 0, n = 0;
    auto check = [&](long long x, int sc) {
        const double a = window_to_double(x, sc), b = window_to_double_seldom(x, sc);
        bad += memcmp(&a, &b, 8) != 0;
        ++n;
    };
    const long long top = (1LL << 62) + (1LL << 55);
    for (int i = 0; i < 3000000; ++i) {
        long long x = (long long)(g() >> (1 + g() %% 63));
        if (i %% 5 == 0) x = (1LL << (g() %% 63)) + (long long)(g() %% 5) - 2;  // near a power of two
        if (x > top || x < 0) x = top;
        if (g() & 1) x = -x;
        const int sc = i %% 3 ? (int)(g() %% 200) - 100 : (int)(g() %% 2400) - 1200;
        check(x, sc);
    }
    for (long long x : {0LL, 1LL, -1LL, (1LL << 53) - 1, (1LL << 53) + 1, (1LL << 32) - 1, 1LL << 32, top, -top})
        for (int sc = -1200; sc <= 1200; ++sc) check(x, sc);
    printf("%%ld of %%ld\n", bad, n);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no g++")
def test_the_same_bits(tmp_path):
    src = open(HEADER).read()
    a = src.index("__host__ __device__ __forceinline__ int clz64_any")
    b = src.index("// The four FP32 levels of a 4-slice product")
    cpp, exe = tmp_path / "w.cpp", tmp_path / "w"
    cpp.write_text(HARNESS % src[a:b])
    subprocess.run(["g++", "-O2", "-std=c++17", str(cpp), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
