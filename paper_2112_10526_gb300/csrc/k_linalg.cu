// FP64 linear algebra of the VMC step: sample statistics, Jacobian products
// (vjp / jvp, App. B.1), the stored centred Jacobian, QGT products and
// Gram matrices (App. B.2 / B.3), and the CG / SGD vector kernels.
//
// Every reduction runs in a fixed order (split-K partials summed in split
// order, tree reductions with a fixed shape), so results are bitwise
// reproducible from run to run.

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "nk_common.cuh"
#include "nk_internal.h"

namespace nk {

namespace {

// ------------------------------------------------------ tile GEMM engine ---
// C(m, n) = sum_{k in split} A(m, k) B(n, k) in FP64: 16 x 16 tile per block,
// one output per thread, K staged 32 at a time in shared memory with the next
// 32 already in registers.  The loaders say whether k (kContig = true) or m/n
// is the contiguous index in memory so that the staging loads coalesce either
// way.
// The FP64 pipe of this part (2 lanes a clock and SM) bounds every shape, so
// the tile is as small as the block: nothing is computed for padding beyond
// 15 rows and columns, and a small product still spreads over many SMs (64 x
// 64 tiles with 4 x 4 outputs a thread, on one SM: 296 us for a 17 x 17 x 256
// product, 244 us for 46 x 38 x 1025).  Products large enough for the tensor
// cores do not come here (f64_on_tensor).

constexpr int kGT = 16, kGK = 32;

template <class LA, class LB, class EP>
__global__ void __launch_bounds__(256) k_gemm16(int64_t Md, int64_t Nd, int64_t Kd, int64_t kchunk,
                                                LA la, LB lb, EP ep) {
    __shared__ double As[kGK][kGT + 1];
    __shared__ double Bs[kGK][kGT + 1];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t m0 = (int64_t)blockIdx.x * kGT, n0 = (int64_t)blockIdx.y * kGT;
    if (!ep.active(m0, n0)) return;
    const int split = blockIdx.z;
    const int64_t kb = (int64_t)split * kchunk;
    const int64_t ke = kb + kchunk < Kd ? kb + kchunk : Kd;
    // the two elements of each operand that this thread stages
    int ka[2], ra[2], kbb[2], rb[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int e = threadIdx.x + 256 * u;
        ka[u] = LA::kContig ? (e & 31) : (e >> 4);
        ra[u] = LA::kContig ? (e >> 5) : (e & 15);
        kbb[u] = LB::kContig ? (e & 31) : (e >> 4);
        rb[u] = LB::kContig ? (e >> 5) : (e & 15);
    }
    double av[2], bv[2];
    auto fetch = [&](int64_t k0) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            av[u] = (m0 + ra[u] < Md && k0 + ka[u] < ke) ? la(m0 + ra[u], k0 + ka[u]) : 0.0;
            bv[u] = (n0 + rb[u] < Nd && k0 + kbb[u] < ke) ? lb(n0 + rb[u], k0 + kbb[u]) : 0.0;
        }
    };
    double acc = 0.0;
    fetch(kb);
    for (int64_t k0 = kb; k0 < ke; k0 += kGK) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            As[ka[u]][ra[u]] = av[u];
            Bs[kbb[u]][rb[u]] = bv[u];
        }
        __syncthreads();
        if (k0 + kGK < ke) fetch(k0 + kGK);
        const int kn = (int)(ke - k0 < kGK ? ke - k0 : kGK);
        if (kn == kGK) {
#pragma unroll 8
            for (int kk = 0; kk < kGK; ++kk) acc = fma(As[kk][ty], Bs[kk][tx], acc);
        } else {
            for (int kk = 0; kk < kn; ++kk) acc = fma(As[kk][ty], Bs[kk][tx], acc);
        }
        __syncthreads();
    }
    const int64_t m = m0 + ty, n = n0 + tx;
    if (m < Md && n < Nd) ep(m, n, split, acc);
}

template <class LA, class LB, class EP>
cudaError_t gemm16(int64_t Md, int64_t Nd, int64_t Kd, int splits, LA la, LB lb, EP ep, cudaStream_t st) {
    if (Md <= 0 || Nd <= 0) return cudaSuccess;
    if (splits < 1) splits = 1;
    const int64_t kchunk = (Kd + splits - 1) / splits;
    dim3 grid((unsigned)((Md + kGT - 1) / kGT), (unsigned)((Nd + kGT - 1) / kGT), (unsigned)splits);
    (k_gemm16<<<grid, 256, 0, st>>>(Md, Nd, Kd, kchunk > 0 ? kchunk : 1, la, lb, ep), nk::note_launch());
    return cudaGetLastError();
}

// -------------------------------------------------------- vjp: J^T g -------
// Augmented GEMM P[j][i] = sum_k A'(k, j) g_k B'(k, i) with A' = [T, 1] and
// B' = [S, 1]: P[j<M][i<N] is the W block, P[j][N] the b block and P[M][i]
// the a block of J^T g.

struct VjpA {  // A'(j, k) = T_kj (j < M) or 1
    static constexpr bool kContig = false;
    const double *T;
    int M;
    __device__ double operator()(int64_t j, int64_t k) const { return j < M ? T[(size_t)k * M + j] : 1.0; }
};

struct AugSg_kn {  // g'_k B'(i, k), g'_k = scale (g_k - shift), B' = s_ki (i < N) or 1, i contiguous
    static constexpr bool kContig = false;
    const int8_t *s;
    const double *g, *shift;
    double scale;
    int N;
    __device__ double operator()(int64_t i, int64_t k) const {
        const double gk = scale * (g[k] - (shift ? *shift : 0.0));
        return i < N ? (double)s[(size_t)k * N + i] * gk : gk;
    }
};

struct EpPartial {
    double *P;
    int64_t ld, plane;
    __device__ bool active(int64_t, int64_t) const { return true; }
    __device__ void operator()(int64_t m, int64_t n, int split, double v) const {
        P[(size_t)split * plane + (size_t)m * ld + n] = v;
    }
};

// sum of n values `stride` apart: eight loads and four chains in flight (the
// sum waits on memory and on dependent FP64 adds).
__device__ __forceinline__ double sum_strided(const double *__restrict__ p, int64_t stride, int n) {
    double q[4] = {0.0, 0.0, 0.0, 0.0};
    int b = 0;
    for (; b + 7 < n; b += 8) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = p[(size_t)(b + u) * stride];
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] += v[u] + v[u + 4];
    }
    for (; b < n; ++b) q[b & 3] += p[(size_t)b * stride];
    return (q[0] + q[1]) + (q[2] + q[3]);
}

__global__ void k_vjp_reduce(int N, int M, int splits, const double *__restrict__ P,
                             double *__restrict__ out) {
    const int64_t plane = (int64_t)(M + 1) * (N + 1);
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= plane) return;
    const int j = (int)(idx / (N + 1)), i = (int)(idx % (N + 1));
    if (j == M && i == N) return;
    const double s = sum_strided(P + idx, plane, splits);
    if (j == M)
        out[i] = s;
    else if (i == N)
        out[N + j] = s;
    else
        out[N + M + (size_t)j * N + i] = s;
}

// Splits of the K = Ns range: about four blocks per SM (the FP64 pipe is full
// with two), at least 8 samples each and at most 32 partial planes (their sum
// waits on memory: 19 us for 128 planes).
int vjp_splits(int N, int M, int64_t Ns) {
    const int64_t tiles = (int64_t)((M + 1 + kGT - 1) / kGT) * ((N + 1 + kGT - 1) / kGT);
    int64_t sp = (608 + tiles - 1) / tiles;
    const int64_t maxsp = (Ns + 7) / 8;
    if (sp > maxsp) sp = maxsp;
    if (sp > 32) sp = 32;
    if (sp < 1) sp = 1;
    return (int)sp;
}

// --------------------------------------------------------- jvp: J v --------
// U[k][j] = sum_i B'(k, i) V'(j, i) with V' = [[V_W, v_b], [v_a, 0]], then
// w_k = sum_j A'(k, j) U[k][j].

struct AugS_k {  // A(k, i) = s_ki or 1, i (the K index) contiguous
    static constexpr bool kContig = true;
    const int8_t *s;
    int N;
    __device__ double operator()(int64_t k, int64_t i) const {
        return i < N ? (double)s[(size_t)k * N + i] : 1.0;
    }
};

struct VAug {
    static constexpr bool kContig = true;
    const double *v;
    int N, M;
    __device__ double operator()(int64_t j, int64_t i) const {
        if (j < M) return i < N ? v[N + M + (size_t)j * N + i] : v[N + j];
        return i < N ? v[i] : 0.0;
    }
};

struct EpStore {
    double *C;
    int64_t ld;
    __device__ bool active(int64_t, int64_t) const { return true; }
    __device__ void operator()(int64_t m, int64_t n, int, double v) const {
        C[(size_t)m * ld + n] = v;
    }
};

__global__ void k_rowdot_aug(int M, int64_t Ns, const double *__restrict__ T,
                             const double *__restrict__ U, double *__restrict__ w) {
    const int lane = threadIdx.x & 31;
    const int64_t k = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (k >= Ns) return;
    double acc = 0.0;
    for (int j = lane; j <= M; j += 32)
        acc += (j < M ? T[(size_t)k * M + j] : 1.0) * U[(size_t)k * (M + 1) + j];
    acc = warp_sum(acc);
    if (lane == 0) w[k] = acc;
}

// ------------------------------------------------------- Jacobian rows -----

__global__ void k_jacobian_rows(int N, int M, const int8_t *__restrict__ s,
                                const double *__restrict__ T, int64_t row0, int64_t rows,
                                const double *__restrict__ mean, double *__restrict__ O) {
    const int64_t Np = (int64_t)N + M + (int64_t)M * N;
    const int64_t r = blockIdx.y;
    if (r >= rows) return;
    const int64_t k = row0 + r;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < Np;
         p += (int64_t)gridDim.x * blockDim.x) {
        double v;
        if (p < N)
            v = (double)s[(size_t)k * N + p];
        else if (p < N + M)
            v = T[(size_t)k * M + (p - N)];
        else {
            const int64_t q = p - N - M;
            const int64_t j = q / N, i = q % N;
            v = T[(size_t)k * M + j] * (double)s[(size_t)k * N + i];
        }
        if (mean) v -= mean[p];
        O[(size_t)r * Np + p] = v;
    }
}

// ------------------------------------------------------------- GEMV -------

__global__ void k_gemv_rows(const double *__restrict__ A, int64_t rows, int64_t cols,
                            const double *__restrict__ x, double *__restrict__ y) {
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= rows) return;
    double acc = 0.0;
    for (int64_t c = lane; c < cols; c += 32) acc += A[(size_t)r * cols + c] * x[c];
    acc = warp_sum(acc);
    if (lane == 0) y[r] = acc;
}

// Rows per partial sum: about four blocks of 256 columns per SM, at most 32
// partials (or 256 rows each), at least 16 rows.
int64_t gemv_t_rows(int64_t rows, int64_t cols) {
    const int64_t bc = (cols + 255) / 256;
    int64_t parts = 608 / (bc > 0 ? bc : 1);
    if (parts > 32) parts = 32;
    if (parts < (rows + 255) / 256) parts = (rows + 255) / 256;
    const int64_t r = (rows + parts - 1) / parts;
    return r < 16 ? 16 : r;
}

// partial[b][c] = sum over rows of chunk b (nr rows) of A[r][c] x[r]
__global__ void k_gemv_t_partial(const double *__restrict__ A, int64_t rows, int64_t cols, int64_t nr,
                                 const double *__restrict__ x, double *__restrict__ partial) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.y * nr;
    if (c >= cols) return;
    const int64_t r1 = r0 + nr < rows ? r0 + nr : rows;
    double p = 0.0, q = 0.0;
    int64_t r = r0;
#pragma unroll 4
    for (; r + 1 < r1; r += 2) {
        p = fma(A[(size_t)r * cols + c], x[r], p);
        q = fma(A[(size_t)(r + 1) * cols + c], x[r + 1], q);
    }
    if (r < r1) p = fma(A[(size_t)r * cols + c], x[r], p);
    partial[(size_t)blockIdx.y * cols + c] = p + q;
}

__global__ void k_sum_partials(int64_t cols, int nparts, const double *__restrict__ partial,
                               double scale, double *__restrict__ y) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cols) return;
    y[c] = scale * sum_strided(partial + c, cols, nparts);
}

// ----------------------------------------------------------- SYRK (J^T J) --

struct ColMajorA {  // A(p, k) = dJ[k][p], p contiguous
    static constexpr bool kContig = false;
    const double *A;
    int64_t ld;
    __device__ double operator()(int64_t p, int64_t k) const { return A[(size_t)k * ld + p]; }
};

struct EpSyrk {
    double *C;
    int64_t n;
    double scale, eps;
    __device__ bool active(int64_t m0, int64_t n0) const { return n0 <= m0 + kGT - 1; }
    __device__ void operator()(int64_t m, int64_t q, int, double v) const {
        if (q > m) return;
        const double r = v * scale + (m == q ? eps : 0.0);
        C[(size_t)m * n + q] = r;
        C[(size_t)q * n + m] = r;
    }
};

// ---------------------------------------------------- sample-space Gram ---
// K_raw[k][l] = g_s + g_t + g_t g_s with g_s = s_k.s_l (exact integer) and
// g_t = t_k.t_l (FP64): the Gram of the Jacobian rows O_k = [s_k, t_k,
// t_k (x) s_k] without forming them.

__global__ void __launch_bounds__(256) k_gram_raw(int N, int M, int64_t Ns,
                                                  const int8_t *__restrict__ s,
                                                  const double *__restrict__ T,
                                                  double *__restrict__ K) {
    __shared__ double As[16][64 + 1];
    __shared__ double Bs[16][64 + 1];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t m0 = (int64_t)blockIdx.y * 64, n0 = (int64_t)blockIdx.x * 64;
    if (n0 > m0 + 63) return;  // lower triangle of tiles only
    int gs[4][4] = {};
    double gt[4][4] = {};
    for (int i0 = 0; i0 < N; i0 += 16) {
        for (int e = threadIdx.x; e < 1024; e += 256) {
            const int kk = e & 15, r = e >> 4;
            const int i = i0 + kk;
            As[kk][r] = (m0 + r < Ns && i < N) ? (double)s[(size_t)(m0 + r) * N + i] : 0.0;
            Bs[kk][r] = (n0 + r < Ns && i < N) ? (double)s[(size_t)(n0 + r) * N + i] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk)
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    gs[u][v] += (int)As[kk][ty * 4 + u] * (int)Bs[kk][tx * 4 + v];
        __syncthreads();
    }
    for (int j0 = 0; j0 < M; j0 += 16) {
        for (int e = threadIdx.x; e < 1024; e += 256) {
            const int kk = e & 15, r = e >> 4;
            const int j = j0 + kk;
            As[kk][r] = (m0 + r < Ns && j < M) ? T[(size_t)(m0 + r) * M + j] : 0.0;
            Bs[kk][r] = (n0 + r < Ns && j < M) ? T[(size_t)(n0 + r) * M + j] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            double av[4], bv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                av[u] = As[kk][ty * 4 + u];
                bv[u] = Bs[kk][tx * 4 + u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) gt[u][v] = fma(av[u], bv[v], gt[u][v]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int64_t k = m0 + ty * 4 + u;
        if (k >= Ns) continue;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int64_t l = n0 + tx * 4 + v;
            if (l >= Ns || l > k) continue;
            const double g = (double)gs[u][v] + gt[u][v] + gt[u][v] * (double)gs[u][v];
            K[(size_t)k * Ns + l] = g;
            K[(size_t)l * Ns + k] = g;
        }
    }
}

__global__ void k_row_mean(int64_t n, const double *__restrict__ K, double *__restrict__ r) {
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= n) return;
    double acc = 0.0;
    for (int64_t c = lane; c < n; c += 32) acc += K[(size_t)row * n + c];
    acc = warp_sum(acc);
    if (lane == 0) r[row] = acc / (double)n;
}

// Single block: rbar = mean(r) into r[n].
__global__ void k_mean_into(int64_t n, double *__restrict__ r) {
    __shared__ double red[32];
    double acc = 0.0;
    for (int64_t c = threadIdx.x; c < n; c += blockDim.x) acc += r[c];
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        v = warp_sum(v);
        if (threadIdx.x == 0) r[n] = v / (double)n;
    }
}

constexpr int kCenterRows = 16;

// K_kl <- (K_kl - r_k - r_l + rbar) / n (+ eps on the diagonal), written
// as fma(K_kl - r_l, 1/n, (rbar - r_k) / n): two FP64 operations per entry
// (the FP64 pipe bounds this kernel, not HBM).  16 rows in blockIdx.y (grid-
// stride), 256 columns per block in blockIdx.x; lower_only leaves the part
// above the diagonal untouched.  A row a block was bound by starting 262144
// blocks: 372 us for the lower half of 8192 rows, 197 so.
__global__ void k_double_center(int64_t n, double *__restrict__ K, const double *__restrict__ r,
                                const double *__restrict__ bk, double inv_n, double eps, int lower_only) {
    const int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= n) return;
    const double rl = r[l];
    for (int64_t k0 = (int64_t)blockIdx.y * kCenterRows; k0 < n; k0 += (int64_t)gridDim.y * kCenterRows) {
        if (lower_only && (int64_t)blockIdx.x * blockDim.x >= k0 + kCenterRows) continue;  // block-uniform
#pragma unroll 8
        for (int u = 0; u < kCenterRows; ++u) {
            const int64_t k = k0 + u;
            if (k < n && !(lower_only && l > k)) {
                double v = fma(K[(size_t)k * n + l] - rl, inv_n, bk[k]);
                if (k == l) v += eps;
                K[(size_t)k * n + l] = v;
            }
        }
    }
}

// bk[k] = (rbar - r_k) / n, the per-row part of the double centring.
__global__ void k_center_rows(int64_t n, const double *__restrict__ r, double inv_n, double *__restrict__ bk) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) bk[k] = (r[n] - r[k]) * inv_n;
}


// ------------------------------------------------------------ statistics ---

__device__ __forceinline__ void neumaier_add(double &s, double &c, double x) {
    double r, e;
    two_sum(s, x, r, e);
    s = r;
    c += e;
}

__device__ __forceinline__ void comp_merge(double &s, double &c, double s2, double c2) {
    double r, e;
    two_sum(s, s2, r, e);
    s = r;
    c = c + c2 + e;
}

// The statistics run on one cluster of eight blocks: the compensated sums cost
// 7 FP64 operations a sample and one SM retires 2 lanes a clock (91 us for
// 16384 samples, 650 us for 65536 on a single block of 1024 threads).  Their
// partial sums meet in distributed shared memory.  256 threads a block: with
// 1024 the sum over a block (8 FP64 operations a level, quantity and warp) took
// longer than the samples; one warp a quantity sums the block (1024 samples: 23.7
// us, 29.8 with every warp's own sum first).
constexpr int kStatCtas = 8, kStatThreads = 256;

// Compensated sums of nq quantities over all threads of the cluster, in a
// fixed order (lanes, warps, blocks); every thread returns the totals in s.
template <int nq>
__device__ void cluster_comp_sum(double (&s)[nq], double (&c)[nq]) {
    static_assert(kStatThreads == 256 && kStatCtas == 8, "sums of eight");
    __shared__ double2 part[nq][kStatThreads];
    __shared__ double2 tot[nq];
    __shared__ double all[nq];
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < nq; ++q) part[q][threadIdx.x] = make_double2(s[q], c[q]);
    __syncthreads();
    // warp q sums quantity q over the block (eight threads a lane first: 96 FP64
    // instructions where every warp's own sum took 40), then over the blocks
    if (warp < nq) {
        double2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = part[warp][32 * u + lane];
#pragma unroll
        for (int h = 4; h > 0; h >>= 1)
#pragma unroll
            for (int u = 0; u < h; ++u) comp_merge(v[u].x, v[u].y, v[u + h].x, v[u + h].y);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            comp_merge(v[0].x, v[0].y, __shfl_down_sync(0xffffffffu, v[0].x, o),
                       __shfl_down_sync(0xffffffffu, v[0].y, o));
        if (lane == 0) tot[warp] = v[0];
    }
    cl.sync();
    if (warp < nq) {
        double2 v = *cl.map_shared_rank(&tot[warp], lane & 7);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1)
            comp_merge(v.x, v.y, __shfl_down_sync(0xffffffffu, v.x, o), __shfl_down_sync(0xffffffffu, v.y, o));
        if (lane == 0) all[warp] = v.x + v.y;
    }
    cl.sync();  // the totals are read before they are written again
#pragma unroll
    for (int q = 0; q < nq; ++q) s[q] = all[q];
}

__global__ void __cluster_dims__(kStatCtas, 1, 1) __launch_bounds__(kStatThreads)
    k_stats(const double *__restrict__ e, int64_t Ns, int n_chains, double *__restrict__ out) {
    const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
    double s1[1] = {0.0}, c1[1] = {0.0};
    for (int64_t k = gid; k < Ns; k += step) neumaier_add(s1[0], c1[0], e[k]);
    cluster_comp_sum(s1, c1);
    const double mean = s1[0] / (double)Ns;
    // sum (e - mean)^2, and over the chains the sums of (m - mean) and (m -
    // mean)^2, m the chain's mean
    double s[3] = {0.0, 0.0, 0.0}, c[3] = {0.0, 0.0, 0.0};
    for (int64_t k = gid; k < Ns; k += step) {
        const double d = e[k] - mean;
        neumaier_add(s[0], c[0], d * d);
    }
    const int64_t per = n_chains > 0 ? Ns / n_chains : 0;
    const bool chains = n_chains > 1 && per >= 2 && per * n_chains == Ns;
    if (chains && per <= 32) {  // a thread per chain
        for (int64_t ch = gid; ch < n_chains; ch += step) {
            double a = 0.0, ac = 0.0;
            for (int64_t q = 0; q < per; ++q) neumaier_add(a, ac, e[ch * per + q]);
            const double d = (a + ac) / (double)per - mean;
            neumaier_add(s[1], c[1], d);
            neumaier_add(s[2], c[2], d * d);
        }
    } else if (chains) {  // a warp per chain
        const int lane = threadIdx.x & 31;
        for (int64_t ch = gid >> 5; ch < n_chains; ch += step >> 5) {
            double a = 0.0, ac = 0.0;
            for (int64_t q = lane; q < per; q += 32) neumaier_add(a, ac, e[ch * per + q]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                comp_merge(a, ac, __shfl_down_sync(0xffffffffu, a, o), __shfl_down_sync(0xffffffffu, ac, o));
            if (lane == 0) {
                const double d = (a + ac) / (double)per - mean;
                neumaier_add(s[1], c[1], d);
                neumaier_add(s[2], c[2], d * d);
            }
        }
    }
    if (chains) {
        cluster_comp_sum(s, c);
    } else {
        double sv[1] = {s[0]}, cv[1] = {c[0]};
        cluster_comp_sum(sv, cv);
        s[0] = sv[0];
    }
    if (gid == 0) {
        const double var = s[0] / (double)Ns;
        double err = sqrt(var / (double)Ns);
        if (chains) {
            // variance of the chain means about their own mean
            const double cm = s[1] / (double)n_chains, v = s[2] / (double)n_chains - cm * cm;
            err = sqrt((v < 0.0 ? 0.0 : v) / (double)n_chains);
        }
        out[0] = mean;
        out[1] = var;
        out[2] = err;
    }
}

// -------------------------------------------------------------- vectors ---

__global__ void k_axpby(int64_t n, double alpha, const double *__restrict__ x, double beta,
                        double *__restrict__ y) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = beta == 0.0 ? alpha * x[i] : alpha * x[i] + beta * y[i];
}

constexpr int kDotBlock = 256;

int dot_blocks(int64_t n) {
    int64_t b = (n + kDotBlock * 8 - 1) / (kDotBlock * 8);
    if (b > 1024) b = 1024;
    if (b < 1) b = 1;
    return (int)b;
}

__global__ void k_dot_partial(int64_t n, const double *__restrict__ x, const double *__restrict__ y,
                              double *__restrict__ partial) {
    __shared__ double red[kDotBlock / 32];
    double acc = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        acc += x[i] * (y ? y[i] : 1.0);
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < kDotBlock / 32 ? red[threadIdx.x] : 0.0;
        v = warp_sum(v);
        if (threadIdx.x == 0) partial[blockIdx.x] = v;
    }
}

__global__ void k_dot_final(int nb, const double *__restrict__ partial, double scale,
                            double *__restrict__ out) {
    __shared__ double red[32];
    double acc = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) acc += partial[i];
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
        v = warp_sum(v);
        if (threadIdx.x == 0) *out = v * scale;
    }
}

__global__ void k_sub_scalar_scale(int64_t n, double *__restrict__ x, const double *__restrict__ m,
                                   double scale) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = (x[i] - *m) * scale;
}

__global__ void k_fill(int64_t n, double v, double *__restrict__ x) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = v;
}

__global__ void k_cg_xr(int64_t n, const double *__restrict__ rr, const double *__restrict__ pAp,
                        const double *__restrict__ p, const double *__restrict__ Ap,
                        double *__restrict__ x, double *__restrict__ r, const int *__restrict__ done) {
    if (*done) return;
    const double alpha = *rr / *pAp;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        x[i] += alpha * p[i];
        r[i] -= alpha * Ap[i];
    }
}

__global__ void k_cg_p(int64_t n, const double *__restrict__ rr_new,
                       const double *__restrict__ rr_old, const double *__restrict__ r,
                       double *__restrict__ p, const int *__restrict__ done) {
    if (*done) return;
    const double beta = *rr_new / *rr_old;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = r[i] + beta * p[i];
}

// Counts the iteration just taken (unless already converged), tests the
// residual and keeps rr_keep = rr for the next iteration.
__global__ void k_cg_check(const double *__restrict__ rr, const double *__restrict__ ff, double tol,
                           int *__restrict__ done, int *__restrict__ iters,
                           double *__restrict__ rr_keep) {
    if (*done) return;
    *iters += 1;
    *rr_keep = *rr;
    if (*rr <= tol * tol * *ff) *done = 1;
}

__global__ void k_sgd(int64_t n, double lr, const double *__restrict__ d, double *__restrict__ p) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] -= lr * d[i];
}

__global__ void k_force_g(int64_t Ns, const double *__restrict__ e, const double *__restrict__ st,
                          double *__restrict__ g) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < Ns) g[k] = 2.0 * (e[k] - st[0]) / (double)Ns;
}

__global__ void k_write_sr_stats(const double *__restrict__ st3, const unsigned long long *acc, int C,
                                 double n_proposals, const double *__restrict__ ff,
                                 const double *__restrict__ dd, const int *__restrict__ it,
                                 const double *__restrict__ rr, const int *__restrict__ status,
                                 nk_sr_stats *__restrict__ out) {
    __shared__ unsigned long long red[256];
    unsigned long long a = 0;
    for (int c = threadIdx.x; c < C; c += blockDim.x) a += acc[c];
    red[threadIdx.x] = a;
    __syncthreads();
    for (int w = blockDim.x >> 1; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out->energy = st3[0];
        out->variance = st3[1];
        out->error = st3[2];
        out->acceptance = n_proposals > 0 ? (double)red[0] / n_proposals : 0.0;
        out->cg_iters = it ? (double)*it : 0.0;
        out->cg_residual = (rr && ff && *ff > 0) ? sqrt(*rr / *ff) : 0.0;
        out->f_norm = ff ? sqrt(*ff) : 0.0;
        out->delta_norm = dd ? sqrt(*dd) : 0.0;
        // status[0]: Cholesky breakdown pivot, status[1]: tensor-core time-out
        out->solver_status = status ? (status[1] ? -(double)status[1] : (double)status[0]) : 0.0;
    }
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// r holds n + 1 row means (the last the grand mean) followed by room for n
// per-row coefficients.
void launch_double_center(int64_t n, double *K, double *r, double eps, bool lower_only, cudaStream_t st) {
    double *bk = r + n + 1;
    (k_center_rows<<<nblk(n, 256), 256, 0, st>>>(n, r, 1.0 / (double)n, bk), nk::note_launch());
    const unsigned rows = nblk(n, kCenterRows);
    const dim3 grid(nblk(n, 256), rows < 65535 ? rows : 65535);
    (k_double_center<<<grid, 256, 0, st>>>(n, K, r, bk, 1.0 / (double)n, eps, lower_only ? 1 : 0),
     nk::note_launch());
}

}  // namespace

// ============================================================ launchers ====

cudaError_t launch_stats(const double *e, int64_t Ns, int n_chains, double *out, cudaStream_t st) {
    (k_stats<<<kStatCtas, kStatThreads, 0, st>>>(e, Ns, n_chains, out), nk::note_launch());
    return cudaGetLastError();
}

size_t vjp_partial_doubles(int N, int M, int64_t Ns) {
    return (size_t)vjp_splits(N, M, Ns) * (size_t)(M + 1) * (size_t)(N + 1);
}

cudaError_t launch_vjp(int N, int M, int64_t Ns, const int8_t *s, const double *T, const double *g,
                       double g_scale, const double *g_shift, double *partial, double *out,
                       cudaStream_t st) {
    const int sp = vjp_splits(N, M, Ns);
    VjpA la{T, M};
    AugSg_kn lb{s, g, g_shift, g_scale, N};
    const int64_t plane = (int64_t)(M + 1) * (N + 1);
    EpPartial ep{partial, N + 1, plane};
    const int slot = prof_begin(NK_PROF_JVP_VJP, st);
    cudaError_t err = gemm16(M + 1, N + 1, Ns, sp, la, lb, ep, st);
    if (err != cudaSuccess) return err;
    (k_vjp_reduce<<<nblk(plane, 256), 256, 0, st>>>(N, M, sp, partial, out), nk::note_launch());
    prof_end(slot, st, 2.0 * (double)Ns * (N + 1) * (double)(M + 1));
    return cudaGetLastError();
}

cudaError_t launch_jvp(int N, int M, int64_t Ns, const int8_t *s, const double *T, const double *v,
                       double *U, double *out, cudaStream_t st) {
    AugS_k la{s, N};
    VAug lb{v, N, M};
    EpStore ep{U, M + 1};
    const int slot = prof_begin(NK_PROF_JVP_VJP, st);
    cudaError_t err = gemm16(Ns, M + 1, N + 1, 1, la, lb, ep, st);
    if (err != cudaSuccess) return err;
    (k_rowdot_aug<<<nblk(Ns, 8), 256, 0, st>>>(M, Ns, T, U, out), nk::note_launch());
    prof_end(slot, st, 2.0 * (double)Ns * (N + 1) * (double)(M + 1) + 2.0 * (double)Ns * (M + 1));
    return cudaGetLastError();
}


cudaError_t launch_jacobian_rows(int N, int M, const int8_t *s, const double *T, int64_t row0,
                                 int64_t rows, const double *mean, double *O, cudaStream_t st) {
    if (rows <= 0) return cudaSuccess;
    const int64_t Np = (int64_t)N + M + (int64_t)M * N;
    int64_t gx = (Np + 255) / 256;
    if (gx > 64) gx = 64;
    for (int64_t r = 0; r < rows; r += 65535) {
        const int64_t rr = rows - r < 65535 ? rows - r : 65535;
        dim3 grid((unsigned)gx, (unsigned)rr);
        (k_jacobian_rows<<<grid, 256, 0, st>>>(N, M, s, T, row0 + r, rr, mean,
                                              O + (size_t)r * Np), nk::note_launch());
    }
    return cudaGetLastError();
}

cudaError_t launch_gemv_rows(const double *A, int64_t rows, int64_t cols, const double *x,
                             double *y, cudaStream_t st) {
    if (rows <= 0) return cudaSuccess;
    (k_gemv_rows<<<nblk(rows, 8), 256, 0, st>>>(A, rows, cols, x, y), nk::note_launch());
    return cudaGetLastError();
}

size_t gemv_t_partial_doubles(int64_t rows, int64_t cols) {
    const int64_t nr = gemv_t_rows(rows, cols);
    return (size_t)((rows + nr - 1) / nr) * (size_t)cols;
}

cudaError_t launch_gemv_t(const double *A, int64_t rows, int64_t cols, const double *x,
                          double scale, double *partial, double *y, cudaStream_t st) {
    const int64_t nr = gemv_t_rows(rows, cols), nb = (rows + nr - 1) / nr;
    for (int64_t b0 = 0; b0 < nb; b0 += 65535) {
        const int64_t bb = nb - b0 < 65535 ? nb - b0 : 65535;
        dim3 grid(nblk(cols, 256), (unsigned)bb);
        (k_gemv_t_partial<<<grid, 256, 0, st>>>(A + (size_t)b0 * nr * cols, rows - b0 * nr, cols, nr, x + b0 * nr,
                                               partial + (size_t)b0 * cols), nk::note_launch());
    }
    (k_sum_partials<<<nblk(cols, 256), 256, 0, st>>>(cols, (int)nb, partial, scale, y), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_syrk_t(const double *A, int64_t rows, int64_t cols, double scale, double eps,
                          double *C, cudaStream_t st) {
    ColMajorA la{A, cols};
    EpSyrk ep{C, cols, scale, eps};
    return gemm16(cols, cols, rows, 1, la, la, ep, st);
}

cudaError_t launch_gram_samplespace(int N, int M, int64_t Ns, const int8_t *s, const double *T,
                                    double eps, double *K, double *rowmean, cudaStream_t st) {
    dim3 grid((unsigned)((Ns + 63) / 64), (unsigned)((Ns + 63) / 64));
    const int slot = prof_begin(NK_PROF_GRAM, st);
    (k_gram_raw<<<grid, 256, 0, st>>>(N, M, Ns, s, T, K), nk::note_launch());
    prof_end(slot, st, (double)Ns * (Ns + 1) * (double)(N + M));
    (k_row_mean<<<nblk(Ns, 8), 256, 0, st>>>(Ns, K, rowmean), nk::note_launch());
    (k_mean_into<<<1, 1024, 0, st>>>(Ns, rowmean), nk::note_launch());
    launch_double_center(Ns, K, rowmean, eps, false, st);
    return cudaGetLastError();
}

// The tensor-core Cholesky reads only the lower triangle.
cudaError_t launch_center_gram(int64_t Ns, double *K, double *rowmean, double eps, cudaStream_t st) {
    (k_row_mean<<<nblk(Ns, 8), 256, 0, st>>>(Ns, K, rowmean), nk::note_launch());
    (k_mean_into<<<1, 1024, 0, st>>>(Ns, rowmean), nk::note_launch());
    launch_double_center(Ns, K, rowmean, eps, true, st);
    return cudaGetLastError();
}

cudaError_t launch_axpby(int64_t n, double alpha, const double *x, double beta, double *y,
                         cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    (k_axpby<<<nblk(n, 256), 256, 0, st>>>(n, alpha, x, beta, y), nk::note_launch());
    return cudaGetLastError();
}

size_t dot_partial_doubles(int64_t n) { return (size_t)dot_blocks(n); }

cudaError_t launch_dot(int64_t n, const double *x, const double *y, double *partial, double *out,
                       cudaStream_t st) {
    const int nb = dot_blocks(n);
    (k_dot_partial<<<nb, kDotBlock, 0, st>>>(n, x, y, partial), nk::note_launch());
    (k_dot_final<<<1, 1024, 0, st>>>(nb, partial, 1.0, out), nk::note_launch());
    return cudaGetLastError();
}

// x <- (x - mean(x)) * scale; partial holds dot_partial_doubles(n) + 1 doubles.
cudaError_t launch_center(int64_t n, double *x, double *partial, double scale, cudaStream_t st) {
    const int nb = dot_blocks(n);
    (k_dot_partial<<<nb, kDotBlock, 0, st>>>(n, x, nullptr, partial), nk::note_launch());
    (k_dot_final<<<1, 1024, 0, st>>>(nb, partial, 1.0 / (double)n, partial + nb), nk::note_launch());
    (k_sub_scalar_scale<<<nblk(n, 256), 256, 0, st>>>(n, x, partial + nb, scale), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_fill(int64_t n, double v, double *x, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    (k_fill<<<nblk(n, 256), 256, 0, st>>>(n, v, x), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_cg_update_xr(int64_t n, const double *rr, const double *pAp, const double *p,
                                const double *Ap, double *x, double *r, const int *done,
                                cudaStream_t st) {
    (k_cg_xr<<<nblk(n, 256), 256, 0, st>>>(n, rr, pAp, p, Ap, x, r, done), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_cg_update_p(int64_t n, const double *rr_new, const double *rr_old,
                               const double *r, double *p, const int *done, cudaStream_t st) {
    (k_cg_p<<<nblk(n, 256), 256, 0, st>>>(n, rr_new, rr_old, r, p, done), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_cg_check(const double *rr, const double *ff, double tol, int *done, int *iters,
                            double *rr_keep, cudaStream_t st) {
    (k_cg_check<<<1, 1, 0, st>>>(rr, ff, tol, done, iters, rr_keep), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_sgd(int64_t n, double lr, const double *delta, double *params,
                       cudaStream_t st) {
    (k_sgd<<<nblk(n, 256), 256, 0, st>>>(n, lr, delta, params), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_make_force_g(int64_t Ns, const double *eloc, const double *stats, double *g,
                                cudaStream_t st) {
    (k_force_g<<<nblk(Ns, 256), 256, 0, st>>>(Ns, eloc, stats, g), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_write_sr_stats(const double *stats3, const unsigned long long *acc, int C,
                                  double n_proposals, const double *ff, const double *dd,
                                  const int *cg_iters, const double *cg_rr, const int *status,
                                  nk_sr_stats *out, cudaStream_t st) {
    (k_write_sr_stats<<<1, 256, 0, st>>>(stats3, acc, C, n_proposals, ff, dd, cg_iters, cg_rr, status, out), nk::note_launch());
    return cudaGetLastError();
}

}  // namespace nk
