"""The NK_F64 factorisation and its triangular solves (launch_cholesky_tc and
launch_cholesky_solve_tc, `exact`) on matrices whose roundings all go one way.

fwd, bwd: L = I and one row, or column, of a 1 and otherwise 0.9 2^-53, which a single
chain of n / 32 or n / 8 additions drops term by term: the sum of n terms comes back to
(terms of a group + groups + 40) 2^-53, the groups those of the kernels (16 terms and n /
512, 32 and n / 256; 40 for the lanes, warps, the block's solve and the data).

panel: rows of one large entry and 63 of 2^-8 of it, against rows of large ones, with
digits of 255: the update's error in units of 2^-53 sqrt(a_ii a_jj) is at most 18 / 8
(the bound of a panel, 17 m_i m_j, and its addition, on |l_i| |l_j| = 8 m_i m_j), the
diagonal block's and the data's roundings 2 more."""
import os
import shutil
import subprocess
import tempfile

import pytest
import torch

pytestmark = pytest.mark.gpu

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_10526_gb300")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
#include "../../include/nk.h"
#include "nk_internal.h"

// L (lower triangle of A) and x = A^-1 b
static int solve(int64_t n, std::vector<double> &A, std::vector<double> &b) {
    double *dA, *db;
    int *info, h[2] = {-1, -1};
    void *ws;
    if (cudaMalloc(&dA, n * n * 8) || cudaMalloc(&db, n * 8) || cudaMalloc(&info, 8) ||
        cudaMalloc(&ws, nk::tc_chol_ws_bytes(n)))
        return 2;
    cudaMemcpy(dA, A.data(), n * n * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(db, b.data(), n * 8, cudaMemcpyHostToDevice);
    cudaMemset(info, 0, 8);
    if (nk::launch_cholesky_tc(dA, n, info, info + 1, ws, nullptr, nullptr, true) != cudaSuccess) return 3;
    if (nk::launch_cholesky_solve_tc(dA, n, ws, db, info + 1, nullptr, true) != cudaSuccess) return 4;
    if (cudaMemcpy(h, info, 8, cudaMemcpyDeviceToHost) != cudaSuccess || h[0] || h[1]) return 5;
    cudaMemcpy(A.data(), dA, n * n * 8, cudaMemcpyDeviceToHost);
    cudaMemcpy(b.data(), db, n * 8, cudaMemcpyDeviceToHost);
    cudaFree(dA);
    cudaFree(db);
    cudaFree(info);
    cudaFree(ws);
    return 0;
}

int main(int argc, char **argv) {
    const double u = 0x1p-53, q = 0.9 * u;
    if (!strcmp(argv[1], "panel")) {
        const int64_t n = 128;
        const double big = ldexp((double)((1LL << 52) + (1LL << 45) - 1), -53);
        const double small = ldexp((double)((1LL << 53) - 17), -61);
        std::vector<double> l(64 * 64), A(n * n, 0.0), b(n, 1.0);
        for (int r = 0; r < 64; ++r)
            for (int c = 0; c < 64; ++c) l[r * 64 + c] = r % 2 || c == r / 2 ? big : small;
        for (int i = 0; i < 64; ++i) A[i * n + i] = 1.0;
        for (int r = 0; r < 64; ++r) {
            for (int c = 0; c < 64; ++c) A[(64 + r) * n + c] = l[r * 64 + c];
            for (int s = 0; s <= r; ++s) {
                long double v = 0.0L;
                for (int c = 0; c < 64; ++c) v += (long double)l[r * 64 + c] * l[s * 64 + c];
                A[(64 + r) * n + 64 + s] = (double)(r == s ? 1.25L * v : v);
            }
        }
        std::vector<double> L = A;
        if (int e = solve(n, L, b)) return e;
        double worst = 0;
        for (int i = 0; i < n; ++i)
            for (int j = 0; j <= i; ++j) {
                long double v = 0.0L;
                for (int c = 0; c <= j; ++c) v += (long double)L[i * n + c] * L[j * n + c];
                worst = fmax(worst, (double)(fabsl(v - A[i * n + j]) / sqrt(A[i * n + i] * A[j * n + j]) / u));
            }
        printf("worst %g u\n", worst);
        return worst <= 18.0 / 8 + 2 ? 0 : 1;
    }
    const int64_t n = 8192;
    std::vector<double> A(n * n, 0.0), b(n, 1.0);
    for (int64_t i = 0; i < n; ++i) A[i * n + i] = 1.0;
    long double want;
    double got, tol;
    if (!strcmp(argv[1], "fwd")) {  // the last row
        for (int64_t c = 0; c < n - 1; ++c) A[(n - 1) * n + c] = c ? q : 1.0;
        A[n * n - 1] = 2.0;
        b[n - 1] = 0.0;
        if (int e = solve(n, A, b)) return e;
        got = b[n - 1], want = -(1.0L + (n - 2) * (long double)q);
        tol = (16 + n / 512 + 40) * u;
    } else {  // the first column
        for (int64_t r = 1; r < n; ++r) A[r * n] = r == n - 64 ? 1.0 : q;
        A[(n - 64) * (n + 1)] = 2.0;
        for (int64_t r = 1; r < n - 64; ++r) A[(n - 64) * n + r] = q;
        for (int64_t r = n - 63; r < n; ++r) A[r * n + n - 64] = q;
        b[0] = 0.0;
        if (int e = solve(n, A, b)) return e;
        got = b[0], want = -(1.0L + (n - 2) * (long double)q);
        tol = (32 + n / 256 + 40) * u;
    }
    printf("%.17g: off by %g u\n", got, (double)((got - want) / u));
    return fabsl(got - want) <= tol ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def program():
    if shutil.which("nvcc") is None:
        pytest.skip("needs nvcc")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "c.cu"), os.path.join(d, "c")
        with open(src, "w") as f:
            f.write(PROGRAM)
        r = subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I",
                            os.path.join(PKG, "csrc"), "-I", os.path.join(os.path.dirname(PKG), "include"), src,
                            os.path.join(PKG, "libnk.so"), "-o", exe, "-Xlinker", f"-rpath={PKG}"],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        yield exe


@pytest.mark.parametrize("what", ["fwd", "bwd", "panel"])
def test_roundings_that_go_one_way(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
