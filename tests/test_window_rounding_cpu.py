"""sgemm_window (tc_ptx.cuh), the recombined window of the NK_F64 products, on the host
against 128-bit integers: V / 2^drop to nearest (halves up), V = sum D_t 2^(8 (7 - t)), for
every drop that window_drop gives and levels up to their bounds."""
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
    std::mt19937_64 g(7);
    long bad = 0, n = 0;
    for (int i = 0; i < 2000000; ++i) {
        const long long K = 1 + (long long)(g() %% (i %% 3 ? 4096 : 65792));
        const int drop = window_drop(K);
        const long long top = K * 255 < (1LL << 24) ? K * 255 : (1LL << 24);
        int d[7];
        __int128 V = 0;
        for (int t = 0; t < 7; ++t) {
            d[t] = (int)((long long)(g() %% (2 * top + 1)) - top);
            if (i %% 5 == 0 && t < 5) d[t] = 0;
            V += (__int128)d[t] << (8 * (6 - t));
        }
        const __int128 half = drop ? (__int128)1 << (drop - 1) : 0;
        const long long want = (long long)((V + half) >> drop);
        bad += sgemm_window(d, drop) != want;
        ++n;
    }
    printf("%%ld of %%ld\n", bad, n);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no g++")
def test_to_nearest(tmp_path):
    src = open(HEADER).read()
    a = src.index("__host__ __device__ __forceinline__ long long sgemm_window(")
    b = src.index("// x 2^sc for |x| < 2^63 as FP64, rounded to nearest")
    cpp, exe = tmp_path / "w.cpp", tmp_path / "w"
    cpp.write_text(HARNESS % src[a:b])
    subprocess.run(["g++", "-O2", "-std=c++17", str(cpp), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
