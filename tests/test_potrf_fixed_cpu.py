"""The fixed-point arithmetic of k_potrf64 (k_tc.cu) on the host: L D L^T of 64 x 64
positive definite blocks, column by column with the kernel's own routines, compared
with the block in extended precision.  Pivots that are powers of four sit at the end
of the reciprocal's range (1 / M = 4).

Tolerance: a product enters an entry to 2^-59 of sqrt(a_ii a_jj), u and its quotient
are held to 2^-60 of that, and there are at most 64 of each: 64 (2^-59 + 2 2^-60) =
2^-52, taken twice."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SOURCE = os.path.join(os.path.dirname(HERE), "paper_2112_10526_gb300", "csrc", "k_tc.cu")

HARNESS = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <random>
#include <vector>
#define __host__
#define __device__
#define __forceinline__ inline
struct int2 { int x, y; };
static int2 make_int2(int x, int y) { return int2{x, y}; }
%s
static const int n = 64;
static std::mt19937_64 gen(3);
static double uni() { return (double)(gen() >> 11) / 9007199254740992.0; }

// worst error of L D L^T against a, relative to sqrt(a_ii a_jj)
static double factor(const std::vector<double> &a) {
    std::vector<long long> v(n * n);
    std::vector<int> ke(n);
    for (int i = 0; i < n; ++i) {
        int x;
        std::frexp(a[i * n + i], &x);
        ke[i] = (x + 1) >> 1;
    }
    for (int i = 0; i < n; ++i)
        for (int j = 0; j <= i; ++j) v[i * n + j] = llrint(std::ldexp(a[i * n + j], 60 - ke[i] - ke[j]));
    std::vector<long double> L(n * n, 0.0L);
    for (int c = 0; c < n; ++c) {
        const long long d = v[c * n + c];
        const int f = (__builtin_clzll(d) - 4) >> 1;
        const int2 y = halves((long long)fixed_reciprocal((unsigned long long)d << (2 * f)));
        std::vector<int2> u(n), l(n);
        for (int r = c + 1; r < n; ++r) {
            u[r] = halves(v[r * n + c] << (f + 2));
            l[r] = halves(mul62(u[r], y));
        }
        for (int r = c + 1; r < n; ++r)
            for (int q = c + 1; q <= r; ++q) v[r * n + q] -= mul62(u[r], l[q]);
        const long double rs = 1.0L / sqrtl((long double)d);
        for (int r = c; r < n; ++r) L[r * n + c] = ldexpl((long double)v[r * n + c] * rs, ke[r] - 30);
    }
    double worst = 0.0;
    for (int i = 0; i < n; ++i)
        for (int j = 0; j <= i; ++j) {
            long double s = 0.0L;
            for (int k = 0; k <= j; ++k) s += L[i * n + k] * L[j * n + k];
            const double e = std::fabs((double)(s - (long double)a[i * n + j])) / std::sqrt(a[i * n + i] * a[j * n + j]);
            if (!(e <= worst)) worst = e;
        }
    return worst;
}

// A Gram matrix whose columns before `at` are only on the diagonal, so that
// column `at` comes to its turn as it is, with the diagonal entry `pivot`.
static std::vector<double> block(int at, double pivot) {
    std::vector<double> b(n * 2 * n), a(n * n, 0.0);
    for (double &x : b) x = uni() - 0.5;
    for (int i = 0; i < n; ++i)
        for (int j = 0; j <= i; ++j) {
            double s = 0.0;
            for (int k = 0; k < 2 * n; ++k) s += b[i * 2 * n + k] * b[j * 2 * n + k];
            a[i * n + j] = i == j || j >= at ? s : 0.0;
        }
    const double scale = std::sqrt(pivot / a[at * n + at]);
    for (int i = 0; i < n; ++i)
        for (int j = 0; j <= i; ++j) a[i * n + j] *= (i == at ? scale : 1.0) * (j == at ? scale : 1.0);
    a[at * n + at] = pivot;
    return a;
}

int main() {
    double worst = 0.0;
    for (int at : {0, 1, 30, 31, 32, 62, 63})
        for (double pivot : {1.0, 0.25, 4.0, 0x1p-40, 0x1p+40, 2.0, 1.0 + 0x1p-52, 1.0 - 0x1p-53, 0.25 + 0x1p-54, 3.0}) {
            const double e = factor(block(at, pivot));
            if (!(e <= worst)) worst = e;
            if (!(e <= 0x1p-51)) printf("column %%d, pivot %%.17g: %%g\n", at, pivot, e);
        }
    printf("worst %%g\n", worst);
    return !(worst <= 0x1p-51);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no g++")
def test_blocks_with_pivots_at_the_ends_of_the_range(tmp_path):
    src = open(SOURCE).read()
    a = src.index("__host__ __device__ __forceinline__ float rcp_approx")
    b = src.index("__host__ __device__ constexpr int tri_from")
    cpp, exe = tmp_path / "p.cpp", tmp_path / "p"
    cpp.write_text(HARNESS % src[a:b])
    subprocess.run(["g++", "-O2", "-std=c++17", str(cpp), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
