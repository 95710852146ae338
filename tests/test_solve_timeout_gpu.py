"""Time-outs in the direct solves reach the caller in both precisions.  The waits
themselves are tested in test_wait_timeout_gpu; here the host code of the library
(nk_api.cu) is compiled with a stand-in for the triangular solves that reports code 7
at once, as a wait that ran out would, and linked to the rest of the library."""
import os
import shutil
import subprocess
import tempfile

import pytest
import torch

pytestmark = pytest.mark.gpu

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_10526_gb300")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#define launch_cholesky_solve_tc stand_in_solve
#include "nk_api.cu"

__global__ void k_report(int *err) { *err = 7; }
namespace nk {
cudaError_t stand_in_solve(const double *, int64_t, const void *, double *, int *err, cudaStream_t st, bool) {
    k_report<<<1, 1, 0, st>>>(err);
    return cudaGetLastError();
}
}

template <class T>
static T *up(const std::vector<T> &h) {
    T *d = nullptr;
    cudaMalloc(&d, h.size() * sizeof(T));
    cudaMemcpy(d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice);
    return d;
}

int main() {
    const int N = 4, M = 3, Ns = 32, Np = N + M + N * M;
    std::vector<double> p(Np), F(Np, 1.0);
    std::vector<int8_t> s(Ns * N);
    for (int i = 0; i < Np; ++i) p[i] = 0.1 * ((i * 7) % 5 - 2);
    for (int i = 0; i < Ns * N; ++i) s[i] = (i * i / 3) % 2 ? 1 : -1;
    nk_ctx *ctx = nullptr;
    if (nk_ctx_create(0, &ctx) != NK_OK) return 2;
    nk_rbm rbm{N, M, up(p)};
    int8_t *ds = up(s);
    double *dF = up(F), *dd = up(F);
    int bad = 0;
    auto expect = [&](const char *what, long long got, long long want) {
        if (got != want) printf("%s: %lld, expected %lld\n", what, got, want), ++bad;
    };
    int32_t code = -1;
    for (int solver : {NK_SOLVER_CHOLESKY, NK_SOLVER_CHOLESKY_SAMPLESPACE}) {
        expect("f64", nk_sr_solve(ctx, &rbm, NK_F64, ds, Ns, dF, solver, 0.1, 1e-6, 10, dd, nullptr, nullptr, nullptr),
               NK_OK);
        nk_ctx_error(ctx, &code, nullptr);
        expect("its code", code, 7);
        nk_ctx_error(ctx, &code, nullptr);
        expect("the code once read", code, 0);
        expect("mixed",
               nk_sr_solve(ctx, &rbm, NK_MIXED, ds, Ns, dF, solver, 0.1, 1e-6, 10, dd, nullptr, nullptr, nullptr),
               NK_ERR_TIMEOUT);
    }
    std::vector<int32_t> e = {0, 1, 1, 2, 2, 3, 3, 0};
    nk_ham ham{};
    ham.kind = NK_TFIM;
    ham.J = ham.h = 1.0;
    ham.n_edges = 4;
    ham.edges = up(e);
    nk_sr_stats *st = nullptr, hs;
    cudaMalloc(&st, sizeof *st);
    for (int prec : {NK_F64, NK_MIXED}) {
        nk_chains ch{Ns, ds, 0, nullptr};
        nk_sr_cfg cfg{};
        cfg.precision = prec;
        cfg.solver = NK_SOLVER_CHOLESKY;
        cfg.n_samples = 1;
        cfg.diag_shift = 0.1;
        expect("step", nk_sr_step(ctx, &rbm, &ham, &ch, &cfg, st, nullptr, nullptr, nullptr), NK_OK);
        cudaMemcpy(&hs, st, sizeof hs, cudaMemcpyDeviceToHost);
        expect("its status", (long long)hs.solver_status, -7);
        nk_ctx_error(ctx, &code, nullptr);
        expect("the step's code", code, 7);
    }
    nk_ctx_destroy(ctx);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="needs nvcc")
def test_a_time_out_is_reported():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    with tempfile.TemporaryDirectory() as d:
        src, exe = os.path.join(d, "t.cu"), os.path.join(d, "t")
        with open(src, "w") as f:
            f.write(PROGRAM)
        r = subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17",
                            "--expt-relaxed-constexpr", "-I", os.path.join(PKG, "csrc"), "-I",
                            os.path.join(os.path.dirname(PKG), "include"), src, os.path.join(PKG, "libnk.so"), "-o",
                            exe, "-Xlinker", f"-rpath={PKG}"], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
        assert r.returncode == 0, r.stdout + r.stderr
