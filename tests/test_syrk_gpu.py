"""S = scale X^T X + eps I on the tensor cores (launch_syrk_tc), entry by entry against
sums in extended precision: edges of its tiles, chunks and segments of rows, columns of
very different scales, of rare large entries, of zeros and with a NaN.

Tolerance, relative to sqrt(S_ii S_jj): with r = (power of two of the largest entry) /
rms of a column, the slices' rounding and the products left out err by 2^-57 (r_i + r_j)
+ 5 2^-64 r_i r_j; columns of r > 16 are summed in FP64, 16 chains a pair: (rows / 16 + 6)
2^-53.  The sums, the scale and the shift: 4 2^-53."""
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
#include <random>
#include <vector>
#include "../../include/nk.h"
#include "nk_internal.h"

int main(int argc, char **argv) {
    const int64_t rows = atoll(argv[1]), n = atoll(argv[2]);
    std::mt19937_64 g(rows * 1000 + n);
    std::normal_distribution<double> normal;
    std::vector<double> X(rows * n);
    int64_t nan_col = -1;
    for (int64_t c = 0; c < n; ++c)
        for (int64_t r = 0; r < rows; ++r) {
            double v = normal(g);
            if (n > 4) {
                if (c %% 7 == 1) v = (g() %% 1000 < 1 ? 1.998 : -0.002);   // a spin that flips in 1 of 1000
                if (c %% 7 == 3) v = 1e-3 * v + (g() %% 333 == 0 ? v : 0);
                if (c %% 7 == 4) v *= 1e130;
                if (c %% 7 == 5) v *= 1e-130;
                if (c == 6) v = 0.0;
                if (c == 9) {
                    nan_col = c;
                    if (r == rows / 2) v = NAN;
                }
            }
            X[r * n + c] = v;
        }
    double *dX, *dC;
    int *err;
    void *ws;
    std::vector<double> C(n * n, -7.0);
    if (cudaMalloc(&dX, X.size() * 8) || cudaMalloc(&dC, C.size() * 8) || cudaMalloc(&err, 4) ||
        cudaMalloc(&ws, nk::tc_syrk_ws_bytes(rows, n)))
        return 2;
    cudaMemcpy(dX, X.data(), X.size() * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(dC, C.data(), C.size() * 8, cudaMemcpyHostToDevice);
    cudaMemset(err, 0, 4);
    const double scale = 1.0 / (double)rows, eps = 1e-3;
    if (nk::launch_syrk_tc(dX, rows, n, scale, eps, dC, err, ws, nullptr) != cudaSuccess) return 3;
    int code = -1;
    if (cudaMemcpy(&code, err, 4, cudaMemcpyDeviceToHost) != cudaSuccess || code != 0) return 4;
    cudaMemcpy(C.data(), dC, C.size() * 8, cudaMemcpyDeviceToHost);
    std::vector<long double> ss(n, 0.0L);
    std::vector<double> rr(n, 1.0);
    for (int64_t c = 0; c < n; ++c) {
        double m = 0;
        for (int64_t r = 0; r < rows; ++r) ss[c] += (long double)X[r * n + c] * X[r * n + c], m = fmax(m, fabs(X[r * n + c]));
        int e = 0;
        std::frexp(m, &e);
        if (m > 0) rr[c] = (double)(ldexpl(1.0L, e) / sqrtl(ss[c] / rows));
    }
    int bad = 0;
    double worst = 0;
    for (int64_t i = 0; i < n; ++i)
        for (int64_t j = 0; j < n; ++j) {
            const double got = C[i * n + j];
            bool ok;
            if (j > i) {
                ok = got == -7.0;  // untouched
            } else if (i == nan_col || j == nan_col) {
                ok = std::isnan(got);
            } else {
                long double s = 0.0L;
                for (int64_t r = 0; r < rows; ++r) s += (long double)X[r * n + i] * X[r * n + j];
                s = s * scale + (i == j ? eps : 0.0);
                const long double size = sqrtl(ss[i] * ss[j]) * scale + (i == j ? eps : 0.0);
                // at the limit of 16 either of the two forms may be taken
                const double sums = (rows / 16 + 6) * 0x1p-53;
                const double cut = 0x1p-57 * (rr[i] + rr[j]) + 5 * 0x1p-64 * rr[i] * rr[j];
                const double tol = 4 * 0x1p-53 + (rr[i] > 16.5 || rr[j] > 16.5 ? sums : rr[i] > 15.5 || rr[j] > 15.5 ? fmax(sums, cut) : cut);
                const double e = size > 0 ? (double)(fabsl((long double)got - s) / size) : (got == 0.0 ? 0.0 : 1.0);
                ok = e <= tol;
                worst = fmax(worst, e);
            }
            if (!ok && bad++ < 10) printf("%%lld %%lld: %%.17g\n", (long long)i, (long long)j, got);
        }
    printf("worst %%g\n", worst);
    return bad ? 1 : 0;
}
""".replace("%%", "%")


@pytest.fixture(scope="module")
def program():
    if shutil.which("nvcc") is None:
        pytest.skip("needs nvcc")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "s.cu"), os.path.join(d, "s")
        with open(src, "w") as f:
            f.write(PROGRAM)
        r = subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I",
                            os.path.join(PKG, "csrc"), "-I", os.path.join(os.path.dirname(PKG), "include"), src,
                            os.path.join(PKG, "libnk.so"), "-o", exe, "-Xlinker", f"-rpath={PKG}"],
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        yield exe


@pytest.mark.parametrize("rows,n", [(1, 1), (64, 31), (65, 33), (1000, 127), (4096, 129), (4096, 300), (3001, 257)])
def test_entries(program, rows, n):
    r = subprocess.run([program, str(rows), str(n)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("rows,n", [((1 << 19) + 1, 3), (1200000, 4)])
def test_segments_of_rows(program, rows, n):
    r = subprocess.run([program, str(rows), str(n)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
