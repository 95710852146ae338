// RBM kernels: flip-ratio tables, ln psi, chain initialisation, Metropolis
// sweeps and local energies.
//
// Model (NetKet 3, Sec. 3.2, Table tab:nk.models, RBM):
//   ln psi(s) = sum_i a_i s_i + sum_j ln cosh theta_j,  theta = b + W s.
//
// Flip-ratio identity used by the sweep and local-energy kernels.  With
// t_j = tanh theta_j and s_i = +-1, cosh(theta - d) = cosh theta cosh d
// (1 - tanh theta tanh d) gives, for flipping site i (d_j = 2 W_ji s_i):
//   ln psi(s^(i)) - ln psi(s) = -2 a_i s_i + K_i + sum_j ln(1 - s_i t_j tau_ji)
// with tau_ji = tanh(2 W_ji), K_i = sum_j ln cosh(2 W_ji); and for swapping an
// antiparallel pair (i, k) (d_j = 2 s_i (W_ji - W_jk)):
//   ln psi(s^(ik)) - ln psi(s) = -2 s_i (a_i - a_k) + K_e + sum_j ln(1 - s_i t_j tau_ej)
// with tau_ej = tanh(2 (W_ji - W_jk)), K_e = sum_j ln cosh(2 (W_ji - W_jk)).
// The sum of logs is taken as the log of one renormalised product, so a
// ratio costs one FMA and one multiply per hidden unit.  After an accepted
// move t_j becomes tanh(theta_j - d_j) = (t_j - s_i tau_j) / (1 - s_i t_j tau_j).

#include <cuda_runtime.h>

#include <type_traits>

#include "nk_common.cuh"
#include "nk_internal.h"
#include "tanh64.cuh"
#include "tc_ptx.cuh"

namespace nk {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------- tables ---

__global__ void k_transpose_W(int N, int M, const double *__restrict__ W, double *__restrict__ Wt) {
    __shared__ double tile[32][33];
    int j0 = blockIdx.y * 32, i0 = blockIdx.x * 32;
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        int j = j0 + r, i = i0 + threadIdx.x;
        if (j < M && i < N) tile[r][threadIdx.x] = W[(size_t)j * N + i];
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        int i = i0 + r, j = j0 + threadIdx.x;
        if (i < N && j < M) Wt[(size_t)i * M + j] = tile[threadIdx.x][r];
    }
}

// x in [-1, 1] as 2^62 x to nearest; +-1 and every FP64 number down to 1/512 are
// exact, so that a factor 1 - t tau of saturated units is 0 as it is in FP64 (one
// ulp less than 1 instead made it 2^-52, which the cosh(2 W) of large weights
// multiplies to anything).  A NaN reads as 1: k_eloc carries it on by itself, and
// the table's NaNs stand in K as well.
__device__ __forceinline__ long long to_fixed62(double x) {
    int b;
    unsigned long long m;
    bool neg;
    split_bits(x, b, m, neg);
    const int sh = b - 1013;  // m 2^(b - 1075 + 62)
    const unsigned long long y = sh >= 0 ? (sh > 10 ? 1ULL << 62 : m << sh)
                                         : (sh <= -54 ? 0ULL : (m >> (-sh)) + ((m >> (-sh - 1)) & 1ULL));
    return neg ? -(long long)y : (long long)y;
}

template <typename R>
__device__ __forceinline__ typename TauOf<R>::type to_tau(double x);
template <>
__device__ __forceinline__ float to_tau<float>(double x) {
    return (float)x;
}
template <>
__device__ __forceinline__ long long to_tau<double>(double x) {
    return to_fixed62(x);
}

// The exponent of every unit's weights (column j of Wt; |W| < 2^e, 0 for zero
// weights, 100000 with an infinity or a NaN) and Wt in place as the integers
// (y >> 30, y & (2^30 - 1)), y = rint(W 2^(59 - e)): the integers of the wide
// slices of k_slice_rows_h5, so that activations summed from either are the
// same to the last bit.  Units whose exponent is flagged (infinities, NaNs,
// magnitudes near the ends of the FP64 range) keep their FP64 weights.
__global__ void __launch_bounds__(256) k_fix_weights(int N, int M, double *__restrict__ Wt, int *__restrict__ eW) {
    const int c = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int j = blockIdx.x * 32 + c;
    int ex = -100000;
    if (j < M)
        for (int i = y; i < N; i += 8) {
            int b;
            unsigned long long m;
            bool neg;
            split_bits(Wt[(size_t)i * M + j], b, m, neg);
            if (m) ex = max(ex, b == 2047 ? 100000 : b - 1022);
        }
    __shared__ int red[8][32];
    red[y][c] = ex;
    __syncthreads();
    for (int q = 0; q < 8; ++q) ex = max(ex, red[q][c]);
    const int e = ex == -100000 ? 0 : ex;
    if (j >= M) return;
    if (y == 0) eW[j] = e;
    if (flagged_exp(e)) return;
    for (int i = y; i < N; i += 8) {
        int b;
        unsigned long long m;
        bool neg;
        split_bits(Wt[(size_t)i * M + j], b, m, neg);
        long long v = 0;
        if (m) {
            const int sh = b - 1075 + 59 - e;
            const unsigned long long u =
                sh >= 0 ? m << sh : (sh <= -64 ? 0ULL : (m >> (-sh)) + ((m >> (-sh - 1)) & 1ULL));
            v = neg ? -(long long)u : (long long)u;
        }
        reinterpret_cast<int2 *>(Wt)[(size_t)i * M + j] = make_int2((int)(v >> 30), (int)(v & 0x3FFFFFFF));
    }
}

// theta_j = b_j + sum_i W_ji s_i from the integers of k_fix_weights (exact sum,
// rounded once): two 64-bit multiply-adds a site on the integer pipe.  drop =
// theta_drop(N).
__host__ __device__ inline int theta_drop(int N) { return window_drop(8LL * N); }

__device__ __forceinline__ double fixed_theta(const Tables<double> &T, const int8_t *sv, int j, int drop) {
    const int e = T.eW[j];
    double v;
    if (flagged_exp(e)) {
        v = 0.0;
        for (int i = 0; i < T.N; ++i) v = fma((double)sv[i], T.Wt[(size_t)i * T.M + j], v);
    } else {
        const int2 *w = reinterpret_cast<const int2 *>(T.Wt) + j;
        long long hi = 0, lo = 0;
#pragma unroll 4
        for (int i = 0; i < T.N; ++i) {
            const int2 y = __ldg(w + (size_t)i * T.M);
            const int s = sv[i];
            hi += (long long)s * y.x;
            lo += (long long)s * y.y;
        }
        v = window_to_double((long long)((unsigned long long)hi << (30 - drop)) + (lo >> drop), e - 59 + drop);
    }
    return v + T.b[j];
}

// One block per site (or edge): tau row, its transpose and K by a fixed-order
// block reduction.
template <typename R>
__global__ void k_tau_rows(int N, int M, int nrows, const double *__restrict__ Wt,
                           const int32_t *__restrict__ edges, typename TauOf<R>::type *__restrict__ tau,
                           typename TauOf<R>::type *__restrict__ tauT, R *__restrict__ K, float *__restrict__ tauf,
                           double *__restrict__ D) {
    int r = blockIdx.x;
    if (r >= nrows) return;
    const double *w0, *w1 = nullptr;
    if (edges) {
        const int i = edges[2 * r], k = edges[2 * r + 1];
        if ((unsigned)i >= (unsigned)N || (unsigned)k >= (unsigned)N) return;  // never used
        w0 = Wt + (size_t)i * M;
        w1 = Wt + (size_t)k * M;
    } else {
        w0 = Wt + (size_t)r * M;
    }
    double part = 0.0;
    for (int j = threadIdx.x; j < M; j += blockDim.x) {
        double d = w1 ? (w0[j] - w1[j]) : w0[j];
        const double v = tanh64(2.0 * d);
        if (tau) tau[(size_t)r * M + j] = to_tau<R>(v);
        if (tauT) tauT[(size_t)j * nrows + r] = to_tau<R>(v);
        if (tauf) {
            tauf[(size_t)r * M + j] = (float)v;
            D[(size_t)r * M + j] = 2.0 * d;
        }
        part += lncosh(2.0 * d);
    }
    __shared__ double red[32];
    part = warp_sum(part);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x < 32) {
        int nw = blockDim.x >> 5;
        double v = threadIdx.x < nw ? red[threadIdx.x] : 0.0;
        v = warp_sum(v);
        if (threadIdx.x == 0) K[r] = (R)v;
    }
}

// ------------------------------------------------------------------ ln psi ---

// One warp per configuration; theta rebuilt in FP64 from the transposed W.
__global__ void k_logpsi(int N, int M, const double *__restrict__ a, const double *__restrict__ b,
                         const double *__restrict__ Wt, const int8_t *__restrict__ s, int64_t B,
                         double *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char sm[];
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int64_t k = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    if (k >= B) return;
    int8_t *sv = reinterpret_cast<int8_t *>(sm) + (size_t)warp * ((N + 15) & ~15);
    for (int i = lane; i < N; i += 32) sv[i] = s[(size_t)k * N + i];
    __syncwarp();
    double part = 0.0;
    for (int i = lane; i < N; i += 32) part += a[i] * (double)sv[i];
    for (int j = lane; j < M; j += 32) {
        double th = b[j];
        for (int i = 0; i < N; ++i) th = fma(Wt[(size_t)i * M + j], (double)sv[i], th);
        part += lncosh(th);
    }
    part = warp_sum(part);
    if (lane == 0) out[k] = part;
}

// ln psi from a precomputed theta [B][M]: one warp per configuration.
__global__ void k_logpsi_theta(int N, int M, const double *__restrict__ a, const double *__restrict__ theta,
                               const int8_t *__restrict__ s, int64_t B, double *__restrict__ out) {
    const int lane = threadIdx.x & 31;
    const int64_t k = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (k >= B) return;
    double part = 0.0;
    for (int i = lane; i < N; i += 32) part += a[i] * (double)s[(size_t)k * N + i];
    for (int j = lane; j < M; j += 32) part += lncosh(theta[(size_t)k * M + j]);
    part = warp_sum(part);
    if (lane == 0) out[k] = part;
}

__global__ void k_tanh_inplace(int64_t n, double *__restrict__ x, bool lib) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = lib ? tanh(x[i]) : tanh64(x[i]);
}

// ------------------------------------------------------------- chain init ---

__global__ void k_chain_init(int N, int C, int rule, unsigned long long seed, unsigned stream_id,
                             int8_t *__restrict__ s) {
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    int8_t *sc = s + (size_t)c * N;
    if (rule == NK_RULE_LOCAL) {
        for (int blk = 0; blk * 256 < N; ++blk) {
            Philox4 y = philox4x64_10((unsigned long long)blk, (unsigned long long)c, stream_id, 1ULL,
                                      seed, 0ULL);
            for (int bit = 0; bit < 256 && blk * 256 + bit < N; ++bit)
                sc[blk * 256 + bit] = ((y.v[bit >> 6] >> (bit & 63)) & 1ULL) ? 1 : -1;
        }
    } else {
        for (int i = 0; i < N; ++i) sc[i] = i < N / 2 ? 1 : -1;
        for (int i = N - 1; i >= 1; --i) {
            Philox4 y = philox4x64_10((unsigned long long)i, (unsigned long long)c, stream_id, 1ULL,
                                      seed, 0ULL);
            int j = pick_index(y.v[0], i + 1);
            int8_t tmp = sc[i];
            sc[i] = sc[j];
            sc[j] = tmp;
        }
    }
}

// ------------------------------------------------------ ratio products ---

// prod over j = j0, j0 + step, ... < M of (1 - si t_j tau[j * tstride]) as
// mantissa x 2^exp.  Four independent running products (each renormalised
// every RenormEvery factors) keep several loads and multiplies in flight.
__device__ __forceinline__ Prod<float> strided_product(const float *__restrict__ t, const float *__restrict__ tau,
                                                       size_t tstride, float si, int j0, int step, int M) {
    using R = float;
    R m0 = R(1), m1 = R(1), m2 = R(1), m3 = R(1);
    int e = 0, cnt = 0;
    int j = j0;
    for (; j + 3 * step < M; j += 4 * step) {
        m0 *= R(1) - si * t[j] * tau[(size_t)j * tstride];
        m1 *= R(1) - si * t[j + step] * tau[(size_t)(j + step) * tstride];
        m2 *= R(1) - si * t[j + 2 * step] * tau[(size_t)(j + 2 * step) * tstride];
        m3 *= R(1) - si * t[j + 3 * step] * tau[(size_t)(j + 3 * step) * tstride];
        if (++cnt == RenormEvery<R>::value) {
            Prod<R> q0{m0, 0}, q1{m1, 0}, q2{m2, 0}, q3{m3, 0};
            renorm(q0);
            renorm(q1);
            renorm(q2);
            renorm(q3);
            m0 = q0.m;
            m1 = q1.m;
            m2 = q2.m;
            m3 = q3.m;
            e += q0.e + q1.e + q2.e + q3.e;
            cnt = 0;
        }
    }
    for (; j < M; j += step) m0 *= R(1) - si * t[j] * tau[(size_t)j * tstride];
    Prod<R> p{m0, e};
    renorm(p);
    p.m *= m1;
    renorm(p);
    p.m *= m2;
    renorm(p);
    p.m *= m3;
    renorm(p);
    return p;
}

// The same product for NK_F64 from 2^62 t and 2^62 tau in 64-bit integers: a
// factor 1 - s t tau is 2^60 -+ the high half of a product, good to 2^-60, and
// the running mantissa (leading one at bit 63) takes two factors and one
// normalisation a step.  An FP64 multiply-add or multiply costs 64 clocks a warp
// and scheduler, a 64-bit high product about 11: 30 clocks a factor against 192
// (multiply, multiply-add, multiply).
struct FixProd {
    unsigned long long m;
    int e;
};
__device__ __forceinline__ unsigned long long fixed_factor(long long t, long long tau, bool up) {
    const long long p = __mul64hi(t, tau) * 4;  // 2^62 t tau
    return (1ULL << 62) - (unsigned long long)(up ? p : -p);  // 2^62 (1 - s t tau), in [0, 2^63]
}
__device__ __forceinline__ void fixed_mul(FixProd &a, unsigned long long f, int point) {
    const unsigned long long r = __umul64hi(a.m, f);  // 2^(point - 1) of the product
    const int z = __clz((int)(r >> 32));
    a.m = r << z;
    a.e += 64 - point - z;
}
__device__ __forceinline__ Prod<double> fixed_value(const FixProd &a) {
    // m 2^-63 2^e, as a mantissa in [1/2, 1)
    return Prod<double>{window_to_double((long long)(a.m >> 1), -63), a.e + 1};
}

// The product where a factor is small or 0: one at a time, normalised over all 64
// bits.
__device__ __noinline__ Prod<double> strided_product_small(const long long *__restrict__ t,
                                                           const long long *__restrict__ tau, size_t tstride, bool up,
                                                           int j0, int step, int M) {
    FixProd a{1ULL << 63, 0};
    for (int j = j0; j < M; j += step) {
        const unsigned long long r = __umul64hi(a.m, fixed_factor(t[j], tau[(size_t)j * tstride], up));
        const int z = min(__clzll((long long)r), 63);
        a.m = r << z;
        a.e += 2 - z;
    }
    return fixed_value(a);
}

// Two factors go into the product through the high half of theirs, which keeps 2^-60:
// enough down to 2^-8, where FP64 itself has 2^-49 left of a factor.  The smallest is
// noted, and the product done over one by one if it was below (a pair of 2^-20 would
// keep 22 bits; |W| from 1 on, units that a flip turns over).
__device__ __forceinline__ Prod<double> strided_product(const long long *__restrict__ t,
                                                        const long long *__restrict__ tau, size_t tstride, double si,
                                                        int j0, int step, int M) {
    const bool up = si > 0.0;
    FixProd a{1ULL << 63, 0}, b{1ULL << 63, 0};
    unsigned least = 1u << 20;
    int j = j0;
    for (; j + 3 * step < M; j += 4 * step) {
        const unsigned long long f0 = fixed_factor(t[j], tau[(size_t)j * tstride], up);
        const unsigned long long f1 = fixed_factor(t[j + step], tau[(size_t)(j + step) * tstride], up);
        const unsigned long long f2 = fixed_factor(t[j + 2 * step], tau[(size_t)(j + 2 * step) * tstride], up);
        const unsigned long long f3 = fixed_factor(t[j + 3 * step], tau[(size_t)(j + 3 * step) * tstride], up);
        const unsigned long long p0 = __umul64hi(f0, f1), p1 = __umul64hi(f2, f3);  // 2^60 of the products
        least = min(least, min((unsigned)(p0 >> 32), (unsigned)(p1 >> 32)));
        fixed_mul(a, p0, 60);
        fixed_mul(b, p1, 60);
    }
    for (; j < M; j += step) {
        const unsigned long long f = fixed_factor(t[j], tau[(size_t)j * tstride], up);
        least = min(least, (unsigned)(f >> 34));
        fixed_mul(a, f, 62);
    }
    if (least < 1u << 20) return strided_product_small(t, tau, tstride, up, j0, step, M);
    fixed_mul(a, b.m, 63);
    a.e += b.e;
    return fixed_value(a);
}

// Lanes over hidden units, four consecutive units per lane (16-byte loads of
// t and tau): prod over this lane's units of (1 - si t_j tau_j).  Needs
// M % 4 == 0 and 16-byte aligned rows.  kSharedTau: the tau row is in shared
// memory (plain loads instead of the read-only global path); the arithmetic
// is the same either way.
template <bool kSharedTau>
__device__ __forceinline__ float4 load_tau4(const float *tau) {
    if (kSharedTau) return *reinterpret_cast<const float4 *>(tau);
    return __ldg(reinterpret_cast<const float4 *>(tau));
}

// frexp of a positive running product: m = f 2^k, f in [0.5, 1), from the
// exponent bits (zero and subnormal m are left as they are, k = 0; the
// products here are renormalised every 8 factors in (0, 2)).
__device__ __forceinline__ float renorm_bits(float m, int &e) {
    const int b = __float_as_int(m);
    const int be = (b >> 23) & 0xFF;
    e += be ? be - 126 : 0;
    return be ? __int_as_float((b & 0x807FFFFF) | 0x3F000000) : m;
}

// A lane's tau row in groups g of four 16-byte loads (units j0 + 512 g + 128
// u, u < 4), for g = 0 .. full - 1: f(uv, g) runs on each group in order,
// while a ring of four keeps the loads of the next three groups in flight
// (large M reads the row from L2, one round trip per group otherwise).
// Returns full.
template <class F>
__device__ __forceinline__ int tau_ring4(const float *__restrict__ tau, int j0, int full, F &&f) {
    float4 r0[4], r1[4], r2[4], r3[4];
    auto load = [&](float4 (&r)[4], int g) {
#pragma unroll
        for (int u = 0; u < 4; ++u) r[u] = __ldg(reinterpret_cast<const float4 *>(tau + j0 + g * 512 + u * 128));
    };
    if (0 < full) load(r0, 0);
    if (1 < full) load(r1, 1);
    if (2 < full) load(r2, 2);
    int g = 0;
    for (; g + 3 < full; g += 4) {
        load(r3, g + 3);
        f(r0, g);
        if (g + 4 < full) load(r0, g + 4);
        f(r1, g + 1);
        if (g + 5 < full) load(r1, g + 5);
        f(r2, g + 2);
        if (g + 6 < full) load(r2, g + 6);
        f(r3, g + 3);
    }
    // up to three groups left, already in r0 / r1 / r2
    if (g < full) f(r0, g++);
    if (g < full) f(r1, g++);
    if (g < full) f(r2, g++);
    return g;
}

// groups of four units (j + 384 < M) of the lane starting at unit j
__device__ __forceinline__ int lane_groups(int M, int j) { return M - j - 3 * 128 > 0 ? (M - j - 3 * 128 + 511) / 512 : 0; }

// kPos: s_i = +1 (factors 1 - t tau), else s_i = -1 (1 + t tau), the sign
// in the FMA operand; the running products are renormalised by their
// exponent bits.
template <bool kSharedTau, bool kRing, bool kPos>
__device__ __forceinline__ Prod<float> lane_product4_signed(const float *__restrict__ t, const float *__restrict__ tau,
                                                            int lane, int M) {
    float m0 = 1.f, m1 = 1.f;
    int e = 0;
    int j = 4 * lane;
    // Large M: the ring of tau_ring4 (the products and renormalisations run
    // in the order of the plain loop below, so the result is the same).
    if (kRing && !kSharedTau && M >= 6 * 512) {
        const int j0 = j;
        j += 512 * tau_ring4(tau, j0, lane_groups(M, j0), [&](const float4 (&uv)[4], int g) {
            float4 tv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) tv[u] = *reinterpret_cast<const float4 *>(t + j0 + g * 512 + u * 128);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                m0 *= fmaf(kPos ? -tv[u].x : tv[u].x, uv[u].x, 1.f) * fmaf(kPos ? -tv[u].y : tv[u].y, uv[u].y, 1.f);
                m1 *= fmaf(kPos ? -tv[u].z : tv[u].z, uv[u].z, 1.f) * fmaf(kPos ? -tv[u].w : tv[u].w, uv[u].w, 1.f);
            }
            m0 = renorm_bits(m0, e);
            m1 = renorm_bits(m1, e);
        });
    }
    // groups of four 16-byte loads in flight (large M reads the tau row from L2),
    // renormalised after each group as before
    for (; j + 3 * 128 < M; j += 4 * 128) {
        float4 uv[4], tv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) uv[u] = load_tau4<kSharedTau>(tau + j + u * 128);
#pragma unroll
        for (int u = 0; u < 4; ++u) tv[u] = *reinterpret_cast<const float4 *>(t + j + u * 128);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            m0 *= fmaf(kPos ? -tv[u].x : tv[u].x, uv[u].x, 1.f) * fmaf(kPos ? -tv[u].y : tv[u].y, uv[u].y, 1.f);
            m1 *= fmaf(kPos ? -tv[u].z : tv[u].z, uv[u].z, 1.f) * fmaf(kPos ? -tv[u].w : tv[u].w, uv[u].w, 1.f);
        }
        m0 = renorm_bits(m0, e);
        m1 = renorm_bits(m1, e);
    }
    for (; j < M; j += 128) {
        const float4 tv = *reinterpret_cast<const float4 *>(t + j);
        const float4 uv = load_tau4<kSharedTau>(tau + j);
        m0 *= fmaf(kPos ? -tv.x : tv.x, uv.x, 1.f) * fmaf(kPos ? -tv.y : tv.y, uv.y, 1.f);
        m1 *= fmaf(kPos ? -tv.z : tv.z, uv.z, 1.f) * fmaf(kPos ? -tv.w : tv.w, uv.w, 1.f);
    }
    Prod<float> p{m0, e};
    renorm(p);
    p.m *= m1;
    renorm(p);
    return p;
}

template <bool kSharedTau = false, bool kRing = false>
__device__ __forceinline__ Prod<float> lane_product4(const float *__restrict__ t, const float *__restrict__ tau,
                                                     float si, int lane, int M) {
    return si > 0.f ? lane_product4_signed<kSharedTau, kRing, true>(t, tau, lane, M)
                    : lane_product4_signed<kSharedTau, kRing, false>(t, tau, lane, M);
}

template <bool kRing>
__device__ __forceinline__ Prod<float> unit_lanes_product(const float *t, const float *tau, float si, int lane, int M,
                                                          bool vec4) {
    return vec4 ? lane_product4<false, kRing>(t, tau, si, lane, M)
                : strided_product(t, tau, 1, si, lane, 32, M);
}

// frexp by the exponent bits where they are those of a normal number.
__device__ __forceinline__ void renorm_fast(Prod<float> &p) {
    const int b = __float_as_int(p.m), be = (b >> 23) & 0xFF;
    if (be - 1u < 254u) {
        p.e += be - 126;
        p.m = __int_as_float((b & 0x807FFFFF) | 0x3F000000);
    } else {
        renorm(p);
    }
}

// tanh(theta) of a unit after a flip: (t - s tau) / (1 - s t tau), s = +1 (kPos) or
// -1, as a product with the approximate reciprocal, in four instructions: the value of
// __fdividef here, whose div.approx.f32 the PTX ISA manual defines as a * (1 / b) for b
// in [2^-126, 2^126] (the denominator is 0 or at least 2^-48, and below 2).
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
template <bool kPos>
__device__ __forceinline__ float flipped(float t, float tau) {
    return kPos ? (t - tau) * rcp_approx(fmaf(-t, tau, 1.f)) : (t + tau) * rcp_approx(fmaf(t, tau, 1.f));
}

// lane_product4 on t and a tau row already held in registers: chunk u is units j
// = 4 lane + 128 u .. j + 3 (zero past M).  The groups, renormalisations and tail
// are those of lane_product4, in the same order, so the result is identical.
template <int kC>
__device__ __forceinline__ Prod<float> lane_product4_regs(const float4 (&tv)[kC], const float4 (&uv)[kC], float si,
                                                          int lane, int M) {
    float m0 = 1.f, m1 = 1.f;
    int e = 0, G = 0;
    const int j = 4 * lane;
#pragma unroll
    for (int g = 0; g < kC / 4; ++g) {
        if (j + 512 * g + 3 * 128 < M) {
#pragma unroll
            for (int u = 4 * g; u < 4 * g + 4; ++u) {
                m0 *= fmaf(-si * tv[u].x, uv[u].x, 1.f) * fmaf(-si * tv[u].y, uv[u].y, 1.f);
                m1 *= fmaf(-si * tv[u].z, uv[u].z, 1.f) * fmaf(-si * tv[u].w, uv[u].w, 1.f);
            }
            m0 = renorm_bits(m0, e);
            m1 = renorm_bits(m1, e);
            ++G;
        }
    }
#pragma unroll
    for (int u = 0; u < kC; ++u) {
        if (u >= 4 * G && j + 128 * u < M) {
            m0 *= fmaf(-si * tv[u].x, uv[u].x, 1.f) * fmaf(-si * tv[u].y, uv[u].y, 1.f);
            m1 *= fmaf(-si * tv[u].z, uv[u].z, 1.f) * fmaf(-si * tv[u].w, uv[u].w, 1.f);
        }
    }
    Prod<float> p{m0, e};
    renorm_fast(p);
    p.m *= m1;
    renorm_fast(p);
    return p;
}

// ------------------------------------------------------------------ sweep ---

// Edge e of the list joins two sites of [0, N) holding different spins, after
// the spins of sites i and k are flipped (i = k = -1: as they are).
__device__ __forceinline__ bool antiparallel(const int32_t *__restrict__ edges, int e, int N, const int8_t *sv,
                                             int i, int k) {
    const int a = edges[2 * e], b = edges[2 * e + 1];
    if ((unsigned)a >= (unsigned)N || (unsigned)b >= (unsigned)N) return false;
    const int sa = (a == i || a == k) ? -sv[a] : sv[a], sb = (b == i || b == k) ? -sv[b] : sv[b];
    return sa != sb;
}

// MetropolisHamiltonian proposal of a Heisenberg-type Hamiltonian (Sec. 3.4):
// the connected configurations are the swaps across the n(s) antiparallel
// edges; the proposal is the r-th of them in edge order, r = floor(hi n(s) /
// 2^32), and n(s') is counted on the swapped state.  Warp-uniform results;
// e_sel = -1 when n(s) = 0.
__device__ __forceinline__ void hamiltonian_pick(const int32_t *__restrict__ edges, int E, int N, const int8_t *sv,
                                                 unsigned hi, int lane, int &e_sel, int &ns, int &nsp) {
    ns = 0;
    nsp = 0;
    e_sel = -1;
    for (int e0 = 0; e0 < E; e0 += 32) {
        const int e = e0 + lane;
        ns += __popc(__ballot_sync(kFull, e < E && antiparallel(edges, e, N, sv, -1, -1)));
    }
    if (ns == 0) return;
    int r = (int)(((unsigned long long)hi * (unsigned long long)ns) >> 32);  // r < ns
    for (int e0 = 0; e0 < E; e0 += 32) {
        const int e = e0 + lane;
        const bool f = e < E && antiparallel(edges, e, N, sv, -1, -1);
        const unsigned m = __ballot_sync(kFull, f);
        const int cnt = __popc(m);
        if (r < cnt) {  // warp-uniform
            const bool hit = f && __popc(m & ((1u << lane) - 1u)) == r;
            e_sel = e0 + __ffs(__ballot_sync(kFull, hit)) - 1;
            break;
        }
        r -= cnt;
    }
    if (e_sel < 0) {
        ns = 0;
        return;
    }
    const int i = edges[2 * e_sel], k = edges[2 * e_sel + 1];
    for (int e0 = 0; e0 < E; e0 += 32) {
        const int e = e0 + lane;
        nsp += __popc(__ballot_sync(kFull, e < E && antiparallel(edges, e, N, sv, i, k)));
    }
}

template <typename R>
struct SweepK {
    Tables<R> t;
    SweepArgs a;
    int warp_bytes, t_bytes;
    bool vec4;  // FP32 with M % 4 == 0: 16-byte loads in the ratio products
};

// One warp per chain.  Hidden units are spread over the lanes (j = lane,
// lane + 32, ...); t = tanh theta and the spins live in shared memory.  The
// 32 lanes evaluate the Philox blocks of 32 consecutive proposals at once and
// broadcast them one per proposal.  kHam: the Hamiltonian rule, whose edge
// depends on the state (a separate instantiation keeps the registers of the
// local and exchange rules as they are).
// kRing: the FP32 form with the pipelined tau loads (M >= 3072), given the
// registers of 3 blocks of 4 warps per SM (what shared memory allows there);
// otherwise the registers of 7 blocks, for the small-M occupancy.
template <bool kHam, bool kRing>
__global__ void __launch_bounds__(128, kRing ? 3 : 7) k_sweep(SweepK<float> P) {
    using R = float;
    extern __shared__ __align__(16) unsigned char sm[];
    const Tables<R> &T = P.t;
    const SweepArgs &A = P.a;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * (blockDim.x >> 5) + warp;
    if (c >= A.C) return;
    const int N = T.N, M = T.M;
    R *t = reinterpret_cast<R *>(sm + (size_t)warp * P.warp_bytes);
    int8_t *sv = reinterpret_cast<int8_t *>(sm + (size_t)warp * P.warp_bytes + P.t_bytes);
    for (int i = lane; i < N; i += 32) sv[i] = A.s[(size_t)c * N + i];
    __syncwarp();
    unsigned long long acc = 0;
    const int n_sweeps = A.n_discard + A.n_samples;
    using Acc = R;  // precision of the accept arithmetic
    for (int w = 0; w < n_sweeps; ++w) {
        // From-scratch FP64 theta = b + W s (rebuilt here, or given by the
        // tensor-core product); t = tanh theta and the ln cosh terms of ln psi
        // in FP32 lanes (the FP64 pipe of this part runs at 1/64 of the FP32
        // rate).
        double lp = 0.0;
        for (int j = lane; j < M; j += 32) {
            double th;
            if (A.theta_in) {
                th = A.theta_in[(size_t)c * (A.theta_ld > 0 ? A.theta_ld : M) + j];
            } else {
                th = T.b[j];
                for (int i = 0; i < N; ++i) th = fma(T.Wt[(size_t)i * M + j], (double)sv[i], th);
            }
            const float thf = (float)th;
            t[j] = tanhf(thf);
            lp += (double)lncosh(thf);
        }
        for (int i = lane; i < N; i += 32) lp += T.a[i] * (double)sv[i];
        lp = warp_sum(lp);
        __syncwarp();
        const unsigned long long qbase = (unsigned long long)(A.sweep0 + w) * (unsigned long long)N;
        // Lane l prepares proposal q0 + l of each batch of 32: its Philox
        // block, ln u, the site / edge, K and the visible-bias difference, so
        // that a proposal only broadcasts them.
        // The accept decision is taken in FP32 (ln u and the ratio).
        int b_i = 0, b_k = -1, b_row = 0, b_ok = 1;
        unsigned b_hi = 0;
        R b_K = R(0);
        Acc b_aa = Acc(0), b_lu = Acc(0);
        for (int q = 0; q < N; ++q) {
            if ((q & 31) == 0) {
                Philox4 y = philox4x64_10(qbase + (unsigned long long)(q + lane), (unsigned long long)c,
                                          (unsigned long long)A.stream_id, 0ULL, A.seed, 0ULL);
                b_lu = logf((float)uniform53(y.v[1]));
                if (A.rule == NK_RULE_LOCAL) {
                    b_i = pick_index(y.v[0], N);
                    b_k = -1;
                    b_row = b_i;
                    b_K = T.K_site[b_i];
                    b_aa = (Acc)T.a[b_i];
                } else if (kHam) {
                    b_hi = (unsigned)(y.v[0] >> 32);  // the edge depends on the state
                } else {
                    const int e = pick_index(y.v[0], T.E);
                    const int i0 = A.edges[2 * e], k0 = A.edges[2 * e + 1];
                    // an edge outside [0, N) is never a move (bounds guard)
                    b_ok = (unsigned)i0 < (unsigned)N && (unsigned)k0 < (unsigned)N;
                    b_i = b_ok ? i0 : 0;
                    b_k = b_ok ? k0 : 0;
                    b_row = e;
                    b_K = T.K_edge[e];
                    b_aa = b_ok ? (Acc)(T.a[b_i] - T.a[b_k]) : Acc(0);
                }
            }
            const int src = q & 31;
            int i = __shfl_sync(kFull, b_i, src), k = __shfl_sync(kFull, b_k, src);
            int row = __shfl_sync(kFull, b_row, src);
            R K = __shfl_sync(kFull, b_K, src);
            Acc aa = __shfl_sync(kFull, b_aa, src);
            const Acc lu = __shfl_sync(kFull, b_lu, src);
            const size_t slot = ((size_t)c * A.dec_stride + A.dec_offset + w) * N + q;
            const R *tau;
            Acc corr = Acc(0);  // ln g(s|s') - ln g(s'|s)
            if (A.rule == NK_RULE_LOCAL) {
                tau = T.tau_site + (size_t)row * M;
            } else if (kHam) {
                int e, ns, nsp;
                hamiltonian_pick(A.edges, T.E, N, sv, __shfl_sync(kFull, b_hi, src), lane, e, ns, nsp);
                if (e < 0) {
                    if (lane == 0 && A.decisions) A.decisions[slot] = 2;
                    continue;
                }
                i = A.edges[2 * e];
                k = A.edges[2 * e + 1];
                row = e;
                K = T.K_edge[e];
                aa = (Acc)(T.a[i] - T.a[k]);
                corr = logf((float)ns) - logf((float)nsp);
                tau = T.tau_edge + (size_t)row * M;
            } else {
                if (!__shfl_sync(kFull, b_ok, src) || sv[i] == sv[k]) {
                    if (lane == 0 && A.decisions) A.decisions[slot] = 2;
                    continue;
                }
                tau = T.tau_edge + (size_t)row * M;
            }
            const Acc d0 = Acc(-2) * aa * (Acc)sv[i];
            const R si = (R)sv[i];
            Prod<R> pr = unit_lanes_product<kRing>(t, tau, si, lane, M, P.vec4);
            pr = warp_prod_normalised(pr);
            const Acc delta = d0 + (Acc)(K + prod_log(pr));
            const bool accept = lu < Acc(2) * delta + corr;
            if (lane == 0 && A.decisions) A.decisions[slot] = accept ? 1 : 0;
            if (accept) {
                if (P.vec4) {
                    // FP32 path: 16-byte accesses, fast division (t is rebuilt
                    // exactly from theta after every sweep)
                    float *tf = reinterpret_cast<float *>(t);
                    const float *uf = reinterpret_cast<const float *>(tau);
                    auto update = [&](auto pos) {
                        constexpr bool kPos = decltype(pos)::value;
                        auto upd = [&](float4 tv, const float4 &uv, int j) {
                            *reinterpret_cast<float4 *>(tf + j) =
                                make_float4(flipped<kPos>(tv.x, uv.x), flipped<kPos>(tv.y, uv.y),
                                            flipped<kPos>(tv.z, uv.z), flipped<kPos>(tv.w, uv.w));
                        };
                        // the row again in groups of four 16-byte loads (one round
                        // trip per group where it has left L1)
                        int j = 4 * lane;
                        for (; j + 3 * 128 < M; j += 4 * 128) {
                            float4 uv[4], tv[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u)
                                uv[u] = __ldg(reinterpret_cast<const float4 *>(uf + j + u * 128));
#pragma unroll
                            for (int u = 0; u < 4; ++u) tv[u] = *reinterpret_cast<const float4 *>(tf + j + u * 128);
#pragma unroll
                            for (int u = 0; u < 4; ++u) upd(tv[u], uv[u], j + u * 128);
                        }
                        for (; j < M; j += 128)
                            upd(*reinterpret_cast<const float4 *>(tf + j),
                                __ldg(reinterpret_cast<const float4 *>(uf + j)), j);
                    };
                    if (si > R(0))
                        update(std::true_type{});
                    else
                        update(std::false_type{});
                } else {
                    for (int j = lane; j < M; j += 32) {
                        const R tj = t[j], tv = si * tau[j];
                        t[j] = (tj - tv) / (R(1) - tj * tv);
                    }
                }
                __syncwarp();
                if (lane == 0) {
                    sv[i] = (int8_t)-sv[i];
                    if (k >= 0) sv[k] = (int8_t)-sv[k];
                }
                lp += (double)delta;
                ++acc;
            }
            __syncwarp();
        }
        if (w >= A.n_discard) {
            const size_t row = (size_t)c * A.out_stride + A.out_offset + (w - A.n_discard);
            for (int i = lane; i < N; i += 32) A.samples[row * N + i] = sv[i];
            if (lane == 0 && A.logpsi) A.logpsi[row] = lp;
        }
        __syncwarp();
    }
    for (int i = lane; i < N; i += 32) A.s[(size_t)c * N + i] = sv[i];
    if (lane == 0 && A.n_accepted) A.n_accepted[c] += acc;
}

// NK_F64 sweeps, every proposal screened in FP32.  The FP64 pipe retires 2
// lanes a clock and SM and a dependent FP64 operation takes about 64 clocks, so
// the FP64 product and logarithm of a proposal (3.7 us each at M = 16) cost far
// more than the FP32 ones, and only their comparison with
// ln u matters.  Per proposal the warp takes ln of the ratio product from
// FP32 t = tanh(theta) and tau, with a bound on its error from the smallest
// factor f_min >= 2^-6: each factor 1 - s t tau errs by less than 2^-22 (t:
// theta rounded, 2^-25, and tanhf, 2^-23; tau 2^-25; the FMA 2^-24), its
// logarithm by 2^-22 / f_min, the products and the sum of the lanes'
// logarithms by 2^-21 / f_min a unit, and the lanes' logarithms, the threshold
// ln u / 2 - K + a-part and the Hastings term by 2^-13 + 2^-21 (|sum| + |ln u /
// 2 - K| + |a-part|) in all: 2^-20 M / f_min and these are the bound.
// A proposal whose two sides differ by more than the bound is decided.  The
// others take the differences ln cosh(theta') - ln cosh(theta) themselves,
// first in FP32 (each errs by 2^-22 (|theta| + |theta'| + 2) at most, whatever
// the factor, which settles nearly all proposals with a small factor), then,
// still undecided (about one in a thousand at M = 200), in FP64.  The
// decisions are those of FP64 either way, also where t and tau round to 1 and
// the FP64 product form (which this replaces) loses its digits.  theta itself stays in FP64: it
// is rebuilt at every sweep, moved by one addition a unit on an accepted
// move, and ln psi of a sample is taken from it directly.
// 16-site chain, 16 chains, 80 sweeps: 4.76 ms with every proposal in FP64, 0.59
// by the form of it with the units in registers.
template <bool kHam>
__global__ void __launch_bounds__(128) k_sweep_screened(SweepK<double> P) {
    extern __shared__ __align__(16) unsigned char sm[];
    const Tables<double> &T = P.t;
    const SweepArgs &A = P.a;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * (blockDim.x >> 5) + warp;
    if (c >= A.C) return;
    const int N = T.N, M = T.M;
    unsigned char *base = sm + (size_t)warp * P.warp_bytes;
    double *th = reinterpret_cast<double *>(base);                        // [M]
    float *t = reinterpret_cast<float *>(base + (size_t)P.t_bytes);       // [M]
    int8_t *sv = reinterpret_cast<int8_t *>(base + (size_t)P.t_bytes + P.t_bytes / 2);
    const bool local = A.rule == NK_RULE_LOCAL;
    const double *Dtab = local ? T.D_site : T.D_edge;
    const float *tabf = local ? T.tauf_site : T.tauf_edge;
    for (int i = lane; i < N; i += 32) sv[i] = A.s[(size_t)c * N + i];
    __syncwarp();
    unsigned long long acc = 0;
    const int n_sweeps = A.n_discard + A.n_samples, drop = theta_drop(N);
    for (int w = 0; w < n_sweeps; ++w) {
        // theta = b + W s from scratch, t = tanh theta
        for (int j = lane; j < M; j += 32) {
            double v;
            if (A.theta_in) {
                v = A.theta_in[(size_t)c * (A.theta_ld > 0 ? A.theta_ld : M) + j];
            } else {
                v = fixed_theta(T, sv, j, drop);
            }
            th[j] = v;
            t[j] = tanhf((float)v);
        }
        __syncwarp();
        const unsigned long long qbase = (unsigned long long)(A.sweep0 + w) * (unsigned long long)N;
        // lane l prepares proposal q0 + l of each batch of 32
        int b_i = 0, b_k = -1, b_row = 0, b_ok = 1;
        unsigned b_hi = 0;
        double b_K = 0.0, b_aa = 0.0, b_u = 1.0;
        float b_h = 0.f, b_a2 = 0.f;  // ln u / 2 - K (ln u / 2 for kHam), 2 a-part
        for (int q = 0; q < N; ++q) {
            const int src = q & 31;
            if (src == 0) {
                Philox4 y = philox4x64_10(qbase + (unsigned long long)(q + lane), (unsigned long long)c,
                                          (unsigned long long)A.stream_id, 0ULL, A.seed, 0ULL);
                b_u = uniform53(y.v[1]);
                if (local) {
                    b_i = pick_index(y.v[0], N);
                    b_k = -1;
                    b_row = b_i;
                    b_K = T.K_site[b_i];
                    b_aa = T.a[b_i];
                } else if (kHam) {
                    b_hi = (unsigned)(y.v[0] >> 32);  // the edge depends on the state
                } else {
                    const int e = pick_index(y.v[0], T.E);
                    const int i0 = A.edges[2 * e], k0 = A.edges[2 * e + 1];
                    // an edge outside [0, N) is never a move (bounds guard)
                    b_ok = (unsigned)i0 < (unsigned)N && (unsigned)k0 < (unsigned)N;
                    b_i = b_ok ? i0 : 0;
                    b_k = b_ok ? k0 : 0;
                    b_row = e;
                    b_K = T.K_edge[e];
                    b_aa = b_ok ? T.a[b_i] - T.a[b_k] : 0.0;
                }
                b_h = 0.5f * logf((float)b_u) - (kHam ? 0.f : (float)b_K);
                b_a2 = (float)(2.0 * b_aa);
            }
            int i = __shfl_sync(kFull, b_i, src), k = __shfl_sync(kFull, b_k, src);
            int row = __shfl_sync(kFull, b_row, src);
            float h = __shfl_sync(kFull, b_h, src), a2 = __shfl_sync(kFull, b_a2, src);
            const size_t slot = ((size_t)c * A.dec_stride + A.dec_offset + w) * N + q;
            double K, aa = 0.0;
            int n_s = 1, n_sp = 1;
            if (!kHam) K = __shfl_sync(kFull, b_K, src);
            if (kHam) {
                int e, ns, nsp;
                hamiltonian_pick(A.edges, T.E, N, sv, __shfl_sync(kFull, b_hi, src), lane, e, ns, nsp);
                if (e < 0) {
                    if (lane == 0 && A.decisions) A.decisions[slot] = 2;
                    continue;
                }
                i = A.edges[2 * e];
                k = A.edges[2 * e + 1];
                row = e;
                K = T.K_edge[e];
                aa = T.a[i] - T.a[k];
                h -= (float)K + 0.5f * (logf((float)ns) - logf((float)nsp));  // ln g(s|s') - ln g(s'|s)
                a2 = (float)(2.0 * aa);
                n_s = ns;
                n_sp = nsp;
            } else if (!local && (!__shfl_sync(kFull, b_ok, src) || sv[i] == sv[k])) {
                if (lane == 0 && A.decisions) A.decisions[slot] = 2;
                continue;
            }
            const float si = (float)sv[i];
            // accepted iff sum_j ln(1 - s t_j tau_j) > ln u / 2 - K + 2 (a-part) s (- corr / 2)
            const float thr = fmaf(a2, si, h);
            const float *uf = tabf + (size_t)row * M;
            float m0 = 1.f, m1 = 1.f, mn = 1.f;
            int ex = 0, j = lane;
            for (; j + 7 * 32 < M; j += 8 * 32) {
                float f[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) f[u] = __ldg(uf + j + 32 * u);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    f[u] = fmaf(-si * t[j + 32 * u], f[u], 1.f);
                    mn = fminf(mn, f[u]);
                }
                m0 = renorm_bits(m0 * ((f[0] * f[1]) * (f[2] * f[3])), ex);
                m1 = renorm_bits(m1 * ((f[4] * f[5]) * (f[6] * f[7])), ex);
            }
            for (; j < M; j += 32) {  // at most 7 more
                const float f = fmaf(-si * t[j], __ldg(uf + j), 1.f);
                mn = fminf(mn, f);
                m0 *= f;
            }
            float sum = (__log2f(m0 * m1) + (float)ex) * 0.69314718f;
            sum = warp_sum(sum);
            mn = __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(fmaxf(mn, 0.f))));
            const float margin = __fdividef((float)M * 9.5367432e-7f, mn) +
                                 4.7683716e-7f * (fabsf(sum) + fabsf(h) + fabsf(a2)) + 1.2207031e-4f;
            bool accept;
            const double *D = Dtab + (size_t)row * M;
            if (mn >= 0.015625f && fabsf(sum - thr) > margin) {
                accept = sum > thr;
            } else {
                // factors too small to trust, or undecided: the ln cosh terms
                // themselves, first in FP32
                const double sd = (double)sv[i];
                const float thr2 = fmaf(a2, si, h + (float)K);
                float d2 = 0.f, w2 = 0.f;
                for (int j2 = lane; j2 < M; j2 += 32) {
                    const float x = (float)th[j2], y = (float)fma(-sd, D[j2], th[j2]);
                    d2 += lncosh(y) - lncosh(x);
                    w2 += fabsf(x) + fabsf(y);
                }
                d2 = warp_sum(d2);
                w2 = warp_sum(w2);
                const float margin2 = 4.7683716e-7f * (w2 + 2.f * (float)M + fabsf(d2) + fabsf(h) + fabsf((float)K) +
                                                       fabsf(a2)) + 1.2207031e-4f;
                if (fabsf(d2 - thr2) > margin2) {
                    accept = d2 > thr2;
                } else {
                    double d3 = 0.0;
                    for (int j3 = lane; j3 < M; j3 += 32) d3 += lncosh(fma(-sd, D[j3], th[j3])) - lncosh(th[j3]);
                    d3 = warp_sum(d3);
                    const double av = kHam ? aa : __shfl_sync(kFull, b_aa, src);
                    const double corr = kHam ? log((double)n_s) - log((double)n_sp) : 0.0;
                    accept = log(__shfl_sync(kFull, b_u, src)) < 2.0 * (d3 - 2.0 * av * sd) + corr;
                }
            }
            if (lane == 0 && A.decisions) A.decisions[slot] = accept ? 1 : 0;
            if (accept) {
                const double sd = (double)sv[i];
                for (int j = lane; j < M; j += 32) {
                    const double v = fma(-sd, D[j], th[j]);
                    th[j] = v;
                    t[j] = tanhf((float)v);
                }
                __syncwarp();
                if (lane == 0) {
                    sv[i] = (int8_t)-sv[i];
                    if (k >= 0) sv[k] = (int8_t)-sv[k];
                }
                ++acc;
            }
            __syncwarp();
        }
        if (w >= A.n_discard) {
            const size_t row = (size_t)c * A.out_stride + A.out_offset + (w - A.n_discard);
            for (int i = lane; i < N; i += 32) A.samples[row * N + i] = sv[i];
            if (A.logpsi) {
                double lp = 0.0;
                for (int j = lane; j < M; j += 32) lp += lncosh(th[j]);
                for (int i = lane; i < N; i += 32) lp += T.a[i] * (double)sv[i];
                lp = warp_sum(lp);
                if (lane == 0) A.logpsi[row] = lp;
            }
        }
        __syncwarp();
    }
    for (int i = lane; i < N; i += 32) A.s[(size_t)c * N + i] = sv[i];
    if (lane == 0 && A.n_accepted) A.n_accepted[c] += acc;
}

// k_sweep_screened for the local and exchange rules with M <= 32 kU: theta
// and t in registers (lane l holds units l, l + 32, ...), the rows of the next
// proposal loaded while the current one is decided.  Few chains wait on the
// chain of one proposal after the other, so with kSpec the moved t is computed
// beside the decision instead of after it (the FP64 pipe and the exponentials
// then run for rejected proposals too, which costs nothing until it has more
// than two chains per scheduler to serve).  Same arithmetic, bounds and
// fallbacks as k_sweep_screened.
template <int kU, bool kSpec>
__global__ void __launch_bounds__(128) k_sweep_screened_regs(SweepK<double> P) {
    extern __shared__ __align__(16) unsigned char sm[];
    const Tables<double> &T = P.t;
    const SweepArgs &A = P.a;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * (blockDim.x >> 5) + warp;
    if (c >= A.C) return;
    const int N = T.N, M = T.M;
    int8_t *sv = reinterpret_cast<int8_t *>(sm + (size_t)warp * P.warp_bytes);
    const bool local = A.rule == NK_RULE_LOCAL;
    const double *Dtab = local ? T.D_site : T.D_edge;
    const float *tabf = local ? T.tauf_site : T.tauf_edge;
    for (int i = lane; i < N; i += 32) sv[i] = A.s[(size_t)c * N + i];
    __syncwarp();
    unsigned long long acc = 0;
    const int n_sweeps = A.n_discard + A.n_samples, drop = theta_drop(N);
    bool in[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) in[u] = lane + 32 * u < M;
    double th[kU];
    float t[kU];
    for (int w = 0; w < n_sweeps; ++w) {
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int j = lane + 32 * u;
            double v = 0.0;
            if (in[u]) {
                if (A.theta_in) {
                    v = A.theta_in[(size_t)c * (A.theta_ld > 0 ? A.theta_ld : M) + j];
                } else {
                    v = fixed_theta(T, sv, j, drop);
                }
            }
            th[u] = v;
            t[u] = tanhf((float)v);  // 0 past M: a factor 1
        }
        const unsigned long long qbase = (unsigned long long)(A.sweep0 + w) * (unsigned long long)N;
        for (int q0 = 0; q0 < N; q0 += 32) {
            // lane l prepares proposal q0 + l
            const Philox4 y = philox4x64_10(qbase + (unsigned long long)(q0 + lane), (unsigned long long)c,
                                            (unsigned long long)A.stream_id, 0ULL, A.seed, 0ULL);
            const double b_u = uniform53(y.v[1]);
            int b_i, b_k = -1, b_row, b_ok = 1;
            double b_K, b_aa;
            if (local) {
                b_i = b_row = pick_index(y.v[0], N);
                b_K = T.K_site[b_i];
                b_aa = T.a[b_i];
            } else {
                b_row = pick_index(y.v[0], T.E);
                const int i0 = A.edges[2 * b_row], k0 = A.edges[2 * b_row + 1];
                // an edge outside [0, N) is never a move (bounds guard)
                b_ok = (unsigned)i0 < (unsigned)N && (unsigned)k0 < (unsigned)N;
                b_i = b_ok ? i0 : 0;
                b_k = b_ok ? k0 : 0;
                b_K = T.K_edge[b_row];
                b_aa = b_ok ? T.a[b_i] - T.a[b_k] : 0.0;
            }
            const float b_h = 0.5f * logf((float)b_u) - (float)b_K, b_a2 = (float)(2.0 * b_aa);
            const int nq = N - q0 < 32 ? N - q0 : 32;
            float uf[kU];
            double D[kU];
            auto fetch = [&](int row) {
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const size_t at = (size_t)row * M + lane + 32 * u;
                    uf[u] = in[u] ? __ldg(tabf + at) : 0.f;
                    D[u] = in[u] ? __ldg(Dtab + at) : 0.0;
                }
            };
            fetch(__shfl_sync(kFull, b_row, 0));
            for (int src = 0; src < nq; ++src) {
                const int i = __shfl_sync(kFull, b_i, src), k = __shfl_sync(kFull, b_k, src);
                const float h = __shfl_sync(kFull, b_h, src), a2 = __shfl_sync(kFull, b_a2, src);
                const int next = __shfl_sync(kFull, b_row, src + 1 < nq ? src + 1 : src);
                float u0[kU];
                double D0[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    u0[u] = uf[u];
                    D0[u] = D[u];
                }
                fetch(next);
                const int si8 = sv[i];
                const size_t slot = ((size_t)c * A.dec_stride + A.dec_offset + w) * N + q0 + src;
                if (!local && (!__shfl_sync(kFull, b_ok, src) || si8 == sv[k])) {
                    if (lane == 0 && A.decisions) A.decisions[slot] = 2;
                    continue;
                }
                const float si = (float)si8;
                const double sd = si8 > 0 ? 1.0 : -1.0;
                const float thr = fmaf(a2, si, h);
                float m = 1.f, mn = 1.f;
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const float f = fmaf(-si * t[u], u0[u], 1.f);
                    mn = fminf(mn, f);
                    m *= f;
                }
                double th2[kU];
                float t2[kU];
                if (kSpec) {
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        th2[u] = fma(-sd, D0[u], th[u]);
                        t2[u] = tanhf((float)th2[u]);
                    }
                }
                const float sum = warp_sum(__log2f(m)) * 0.69314718f;
                mn = __uint_as_float(__reduce_min_sync(kFull, __float_as_uint(fmaxf(mn, 0.f))));
                // |sum - thr| above the bound, both sides times f_min
                const float slack = 4.7683716e-7f * (fabsf(sum) + fabsf(h) + fabsf(a2)) + 1.2207031e-4f;
                bool accept;
                if (mn >= 0.015625f && (fabsf(sum - thr) - slack) * mn > (float)M * 9.5367432e-7f) {
                    accept = sum > thr;
                } else {
                    const float K = (float)__shfl_sync(kFull, b_K, src), thr2 = fmaf(a2, si, h + K);
                    float d2 = 0.f, w2 = 0.f;
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        const float x = (float)th[u], z = (float)fma(-sd, D0[u], th[u]);
                        d2 += lncosh(z) - lncosh(x);
                        w2 += fabsf(x) + fabsf(z);
                    }
                    d2 = warp_sum(d2);
                    w2 = warp_sum(w2);
                    const float margin2 = 4.7683716e-7f * (w2 + 2.f * (float)M + fabsf(d2) + fabsf(h) + fabsf(K) +
                                                           fabsf(a2)) + 1.2207031e-4f;
                    if (fabsf(d2 - thr2) > margin2) {
                        accept = d2 > thr2;
                    } else {
                        double d3 = 0.0;
#pragma unroll
                        for (int u = 0; u < kU; ++u)
                            if (in[u]) d3 += lncosh(fma(-sd, D0[u], th[u])) - lncosh(th[u]);
                        d3 = warp_sum(d3);
                        accept = log(__shfl_sync(kFull, b_u, src)) <
                                 2.0 * (d3 - 2.0 * __shfl_sync(kFull, b_aa, src) * sd);
                    }
                }
                if (lane == 0 && A.decisions) A.decisions[slot] = accept ? 1 : 0;
                if (accept) {
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        th[u] = kSpec ? th2[u] : fma(-sd, D0[u], th[u]);
                        t[u] = kSpec ? t2[u] : tanhf((float)th[u]);
                    }
                    if (lane == 0) {
                        sv[i] = (int8_t)-si8;
                        if (k >= 0) sv[k] = (int8_t)si8;
                    }
                    ++acc;
                    __syncwarp();
                }
            }
        }
        if (w >= A.n_discard) {
            const size_t row = (size_t)c * A.out_stride + A.out_offset + (w - A.n_discard);
            for (int i = lane; i < N; i += 32) A.samples[row * N + i] = sv[i];
            if (A.logpsi) {
                double lp = 0.0;
#pragma unroll
                for (int u = 0; u < kU; ++u)
                    if (in[u]) lp += lncosh(th[u]);
                for (int i = lane; i < N; i += 32) lp += T.a[i] * (double)sv[i];
                lp = warp_sum(lp);
                if (lane == 0) A.logpsi[row] = lp;
            }
        }
    }
    for (int i = lane; i < N; i += 32) A.s[(size_t)c * N + i] = sv[i];
    if (lane == 0 && A.n_accepted) A.n_accepted[c] += acc;
}

// FP32 sweeps of the local and exchange rules at few units (M % 4 == 0, M <=
// 128 kC): t = tanh(theta) in registers, the rows of flip ratios of the next
// kSweepAhead proposals on their way into a ring in shared memory (cp.async; a
// lane reads back only the 16-byte chunks it copied).  The proposals come from
// Philox alone, so the rows are known ahead; an exchange row is fetched if its
// spins differ at that time (and loaded on demand if they have come to differ
// since).  A chain then waits for nothing but its own arithmetic: with 1024
// chains there are two warps a scheduler, and the row's L2 round trip and the
// shared-memory round trips of t were most of a proposal.  The arithmetic and
// the order of every product are those of k_sweep, so the decisions are
// identical.  ln psi is summed only where it is asked for.
// 10 x 10 lattice, M = 200, 1024 chains: 66 us a sweep with the row loaded when
// its proposal came up, 55 now: some 160 instructions a proposal at 6.5 cycles
// each, the latency of one dependent on the next.
constexpr int kSweepAhead = 4;

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int n>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(n) : "memory");
}

template <int kC>
__global__ void __launch_bounds__(128) k_sweep_rows(SweepK<float> P) {
    extern __shared__ __align__(16) unsigned char sm[];
    const Tables<float> &T = P.t;
    const SweepArgs &A = P.a;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * (blockDim.x >> 5) + warp;
    if (c >= A.C) return;
    const int N = T.N, M = T.M;
    unsigned char *base = sm + (size_t)warp * P.warp_bytes;
    float *ring = reinterpret_cast<float *>(base);  // [kSweepAhead][M]
    int4 *prop_i = reinterpret_cast<int4 *>(base + (size_t)kSweepAhead * P.t_bytes);  // [32]
    float4 *prop_f = reinterpret_cast<float4 *>(prop_i + 32);                         // [32]
    int8_t *sv = reinterpret_cast<int8_t *>(prop_f + 32);
    const bool local = A.rule == NK_RULE_LOCAL;
    const float *tab = local ? T.tau_site : T.tau_edge;
    for (int i = lane; i < N; i += 32) sv[i] = A.s[(size_t)c * N + i];
    __syncwarp();
    unsigned long long acc = 0;
    const int n_sweeps = A.n_discard + A.n_samples;
    for (int w = 0; w < n_sweeps; ++w) {
        const bool want_lp = A.logpsi != nullptr && w >= A.n_discard;
        uint8_t *decisions =
            A.decisions ? A.decisions + ((size_t)c * A.dec_stride + A.dec_offset + w) * N : nullptr;
        const double *th = A.theta_in + (size_t)c * (A.theta_ld > 0 ? A.theta_ld : M);
        float4 t[kC];
#pragma unroll
        for (int u = 0; u < kC; ++u) {
            const int j = 4 * lane + 128 * u;
            t[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (j < M) {
                const double2 a = *reinterpret_cast<const double2 *>(th + j);
                const double2 b = *reinterpret_cast<const double2 *>(th + j + 2);
                t[u] = make_float4(tanhf((float)a.x), tanhf((float)a.y), tanhf((float)b.x), tanhf((float)b.y));
            }
        }
        double lp = 0.0;
        if (want_lp) {
            for (int j = lane; j < M; j += 32) lp += (double)lncosh((float)th[j]);
            for (int i = lane; i < N; i += 32) lp += T.a[i] * (double)sv[i];
            lp = warp_sum(lp);
        }
        const unsigned long long qbase = (unsigned long long)(A.sweep0 + w) * (unsigned long long)N;
        for (int q0 = 0; q0 < N; q0 += 32) {
            // lane l prepares proposal q0 + l
            const Philox4 y = philox4x64_10(qbase + (unsigned long long)(q0 + lane), (unsigned long long)c,
                                            (unsigned long long)A.stream_id, 0ULL, A.seed, 0ULL);
            const float b_lu = logf((float)uniform53(y.v[1]));
            int4 pi;    // site i (-1: never a move), site k (-1: single flip), row, -
            float4 pf;  // ln u, K, a-part, -
            if (local) {
                const int i = pick_index(y.v[0], N);
                pi = make_int4(i, -1, i, 0);
                pf = make_float4(b_lu, T.K_site[i], (float)T.a[i], 0.f);
            } else {
                const int row = pick_index(y.v[0], T.E);
                const int i0 = A.edges[2 * row], k0 = A.edges[2 * row + 1];
                // an edge outside [0, N) is never a move (bounds guard)
                const bool in = (unsigned)i0 < (unsigned)N && (unsigned)k0 < (unsigned)N;
                pi = make_int4(in ? i0 : -1, k0, row, 0);
                pf = make_float4(b_lu, T.K_edge[row], in ? (float)(T.a[i0] - T.a[k0]) : 0.f, 0.f);
            }
            // handed on through shared memory: two loads a proposal instead of
            // seven shuffles
            __syncwarp();
            prop_i[lane] = pi;
            prop_f[lane] = pf;
            __syncwarp();
            const int nq = N - q0 < 32 ? N - q0 : 32;
            unsigned fetched = 0;  // bit src: the row of proposal src is in (or on its way to) the ring
            auto prefetch = [&](int src) {
                if (src < nq) {
                    const int4 p = prop_i[src];
                    if (local || (p.x >= 0 && sv[p.x] != sv[p.y])) {  // warp-uniform
                        const float *row_p = tab + (size_t)p.z * M;
                        float *dst = ring + (size_t)(src % kSweepAhead) * (P.t_bytes / 4);
#pragma unroll
                        for (int u = 0; u < kC; ++u) {
                            const int j = 4 * lane + 128 * u;
                            if (j < M) cp_async16(dst + j, row_p + j);
                        }
                        fetched |= 1u << src;
                    }
                }
                cp_async_commit();  // one group a proposal, empty or not
            };
#pragma unroll
            for (int src = 0; src < kSweepAhead - 1; ++src) prefetch(src);
            for (int src = 0; src < nq; ++src) {
                prefetch(src + kSweepAhead - 1);
                // this proposal's row has landed (those of the later ones may be under
                // way), also if it is no move any more: its slot is refilled next
                cp_async_wait<kSweepAhead - 1>();
                const int4 p = prop_i[src];
                const int i = p.x, k = p.y;
                const int si8 = i >= 0 ? sv[i] : 0;
                if (!local && (i < 0 || si8 == sv[k])) {
                    if (decisions && lane == 0) decisions[q0 + src] = 2;
                    continue;
                }
                float4 uv[kC];
                if ((fetched >> src) & 1u) {
                    const float *row_s = ring + (size_t)(src % kSweepAhead) * (P.t_bytes / 4);
#pragma unroll
                    for (int u = 0; u < kC; ++u) {
                        const int j = 4 * lane + 128 * u;
                        uv[u] = j < M ? *reinterpret_cast<const float4 *>(row_s + j) : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                } else {
                    const float *row_p = tab + (size_t)p.z * M;
#pragma unroll
                    for (int u = 0; u < kC; ++u) {
                        const int j = 4 * lane + 128 * u;
                        uv[u] = j < M ? __ldg(reinterpret_cast<const float4 *>(row_p + j))
                                      : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
                const float si = (float)si8;
                const float4 pf = prop_f[src];
                const float d0 = -2.f * pf.z * si;
                Prod<float> pr = lane_product4_regs<kC>(t, uv, si, lane, M);
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) {  // as warp_prod_normalised
                    pr.m *= __shfl_xor_sync(kFull, pr.m, off);
                    pr.e += __shfl_xor_sync(kFull, pr.e, off);
                }
                renorm_fast(pr);
                const float delta = d0 + (pf.y + prod_log(pr));
                const bool accept = pf.x < 2.f * delta;
                if (decisions && lane == 0) decisions[q0 + src] = accept ? 1 : 0;
                if (accept) {
#pragma unroll
                    for (int u = 0; u < kC; ++u)
                        t[u] = make_float4(flipped<true>(t[u].x, si * uv[u].x), flipped<true>(t[u].y, si * uv[u].y),
                                           flipped<true>(t[u].z, si * uv[u].z), flipped<true>(t[u].w, si * uv[u].w));
                    if (lane == 0) {
                        sv[i] = (int8_t)-si8;
                        if (!local) sv[k] = (int8_t)si8;  // it held -s_i
                    }
                    if (want_lp) lp += (double)delta;
                    ++acc;
                    __syncwarp();
                }
            }
            cp_async_wait<0>();  // the ring's slots start over with the next batch
        }
        if (w >= A.n_discard) {
            const size_t row = (size_t)c * A.out_stride + A.out_offset + (w - A.n_discard);
            for (int i = lane; i < N; i += 32) A.samples[row * N + i] = sv[i];
            if (lane == 0 && A.logpsi) A.logpsi[row] = lp;
        }
        __syncwarp();
    }
    for (int i = lane; i < N; i += 32) A.s[(size_t)c * N + i] = sv[i];
    if (lane == 0 && A.n_accepted) A.n_accepted[c] += acc;
}

// FP32 sweeps of the local and exchange rules at many units (M % 4 == 0, M <= 128
// kU), theta given: a block of two warps per chain.  Thread (l, h) = (16 warp +
// lane / 2, lane % 2) does the part of lane l of k_sweep that goes into its running
// product m_h: units 4 l + 2 h + 128 u and the next, in the same order, so that
// every product, renormalisation and decision is the same.  Its t = tanh(theta)
// stays in registers; the row of flip ratios comes into shared memory once, by
// cp.async while the move before it is worked on, and serves both the product and
// the update.  The moves of a batch of 32 proposals are found by ballot; the next
// one is guessed from the spins as they are (an accepted move changes the few
// proposals that share a site with it: then the row is fetched on demand).
// k_sweep had a warp per chain, t in shared memory (12 chains an SM at M = 4608)
// and read the row twice from L2: 12 TB/s of it, and three warps a scheduler.
// 24 x 24 lattice, M = 4608, 8192 chains: 6.8 ms a sweep there, 5.3 here.
template <int kU>
__global__ void __launch_bounds__(64, kU <= 16 ? (kU <= 8 ? 16 : 12) : (kU <= 24 ? 9 : (kU <= 40 ? 6 : 4))) k_sweep_pair(SweepK<float> P) {
    extern __shared__ __align__(16) unsigned char sm[];
    const Tables<float> &T = P.t;
    const SweepArgs &A = P.a;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = blockIdx.x;
    const int N = T.N, M = T.M, words = (N + 31) / 32;
    float *ring = reinterpret_cast<float *>(sm);                              // [2][M]
    float2 *xch = reinterpret_cast<float2 *>(sm + 2 * (size_t)P.t_bytes);     // [32] (product, exponent)
    uint32_t *sb = reinterpret_cast<uint32_t *>(xch + 32) + warp * words;     // bit i: spin i is up (a copy per warp)
    const int l = 16 * warp + (lane >> 1), h = lane & 1, j0 = 4 * l + 2 * h;
    const bool local = A.rule == NK_RULE_LOCAL;
    const float *tab = local ? T.tau_site : T.tau_edge;
    constexpr int kLoose = 2;  // groups of four chunks that may be cut short
    for (int w = 0; w < words; ++w) {
        const int i = 32 * w + lane;
        const unsigned up = __ballot_sync(kFull, i < N && A.s[(size_t)c * N + i] > 0);
        if (lane == 0) sb[w] = up;
    }
    __syncwarp();
    auto spin = [&](int i) { return (sb[i >> 5] >> (i & 31)) & 1u; };
    unsigned long long acc = 0;
    const int n_sweeps = A.n_discard + A.n_samples;
    for (int w = 0; w < n_sweeps; ++w) {
        const bool want_lp = warp == 0 && A.logpsi != nullptr && w >= A.n_discard;
        uint8_t *decisions = A.decisions && warp == 0
                                 ? A.decisions + ((size_t)c * A.dec_stride + A.dec_offset + w) * N
                                 : nullptr;
        const double *th = A.theta_in + (size_t)c * (A.theta_ld > 0 ? A.theta_ld : M);
        float2 t[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int j = j0 + 128 * u;
            t[u] = make_float2(0.f, 0.f);
            if (j < M) {
                const double2 a = *reinterpret_cast<const double2 *>(th + j);
                t[u] = make_float2(tanhf((float)a.x), tanhf((float)a.y));
            }
        }
        double lp = 0.0;
        if (want_lp) {
            for (int j = lane; j < M; j += 32) lp += (double)lncosh((float)th[j]);
            for (int i = lane; i < N; i += 32) lp += T.a[i] * (spin(i) ? 1.0 : -1.0);
            lp = warp_sum(lp);
        }
        const unsigned long long qbase = (unsigned long long)(A.sweep0 + w) * (unsigned long long)N;
        // lane l's proposal q0 + l: sites (i < 0: never a move), row, ln u, K and
        // the visible-bias difference
        struct Batch {
            int i, k, row;
            float lu, K, aa;
        };
        auto draw = [&](int q0) {
            Batch b{-1, -1, 0, 0.f, 0.f, 0.f};
            const Philox4 y = philox4x64_10(qbase + (unsigned long long)(q0 + lane), (unsigned long long)c,
                                            (unsigned long long)A.stream_id, 0ULL, A.seed, 0ULL);
            if (q0 + lane >= N) return b;
            b.lu = logf((float)uniform53(y.v[1]));
            if (local) {
                b.i = b.row = pick_index(y.v[0], N);
                b.K = T.K_site[b.i];
                b.aa = (float)T.a[b.i];
            } else {
                b.row = pick_index(y.v[0], T.E);
                const int i0 = A.edges[2 * b.row], k0 = A.edges[2 * b.row + 1];
                // an edge outside [0, N) is never a move (bounds guard)
                if ((unsigned)i0 < (unsigned)N && (unsigned)k0 < (unsigned)N) {
                    b.i = i0;
                    b.k = k0;
                    b.aa = (float)(T.a[i0] - T.a[k0]);
                }
                b.K = T.K_edge[b.row];
            }
            return b;
        };
        auto is_move = [&](const Batch &b) { return b.i >= 0 && (local || spin(b.i) != spin(b.k)); };
        auto fetch = [&](int row, int buf) {
            const float *src = tab + (size_t)row * M + 4 * tid;
            const uint32_t dst = smem_u32(ring) + (uint32_t)buf * (uint32_t)P.t_bytes + 16u * (uint32_t)tid;
#pragma unroll
            for (int v = 0; v < kU / 2; ++v)
                if (v + 2 * kLoose < kU / 2 || 4 * tid + 256 * v < M)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 1024u * v), "l"(src + 256 * v)
                                 : "memory");
            cp_async_commit();
        };
        Batch cur = draw(0), nxt = draw(32);
        int q0 = 0, pos = -1;         // the batch and the last proposal of it that was dealt with
        int ahead_q = -1, buf = 0;    // the proposal whose row is on its way to buffer buf
        for (;;) {
            const unsigned later = pos < 0 ? kFull : ~((2u << pos) - 1u);
            const unsigned mask = __ballot_sync(kFull, is_move(cur)) & later;
            const int src = mask ? __ffs(mask) - 1 : 32;
            if (decisions && lane > pos && lane < src && q0 + lane < N) decisions[q0 + lane] = 2;
            if (src == 32) {  // the batch is done
                q0 += 32;
                if (q0 >= N) break;
                cur = nxt;
                nxt = draw(q0 + 32);
                pos = -1;
                continue;
            }
            pos = src;
            const int i = __shfl_sync(kFull, cur.i, src), k = __shfl_sync(kFull, cur.k, src);
            if (ahead_q != q0 + src) {  // guessed wrongly, or the first of the sweep
                cp_async_wait<0>();
                fetch(__shfl_sync(kFull, cur.row, src), buf);
            }
            cp_async_wait<0>();
            __syncthreads();  // the row is there for both warps; both are done with the other buffer
            const float *row_s = ring + (size_t)buf * (P.t_bytes / 4) + j0;
            {
                const unsigned rest = src == 31 ? 0u : mask & ~((2u << src) - 1u);
                const unsigned then = __ballot_sync(kFull, is_move(nxt));
                if (rest | then) {
                    const int at = __ffs(rest ? rest : then) - 1;
                    ahead_q = q0 + at + (rest ? 0 : 32);
                    buf ^= 1;
                    fetch(__shfl_sync(kFull, rest ? cur.row : nxt.row, at), buf);
                } else {
                    ahead_q = -1;
                    buf ^= 1;
                }
            }
            const bool up = spin(i);
            const float si = up ? 1.f : -1.f;
            // the running product m_h of lane l
            float m = 1.f;
            int e = 0;
            auto product = [&](auto pos_tag) {
                constexpr bool kPos = decltype(pos_tag)::value;
                auto mul = [&](int u) {
                    const float2 v = *reinterpret_cast<const float2 *>(row_s + 128 * u);
                    m *= fmaf(kPos ? -t[u].x : t[u].x, v.x, 1.f) * fmaf(kPos ? -t[u].y : t[u].y, v.y, 1.f);
                };
#pragma unroll
                for (int g = 0; g < kU / 4; ++g) {
                    if (g + kLoose < kU / 4 || 4 * l + 512 * g + 3 * 128 < M) {
#pragma unroll
                        for (int u = 4 * g; u < 4 * g + 4; ++u) mul(u);
                        m = renorm_bits(m, e);
                    } else {
#pragma unroll
                        for (int u = 4 * g; u < 4 * g + 3; ++u)
                            if (4 * l + 128 * u < M) mul(u);
                    }
                }
            };
            if (up)
                product(std::true_type{});
            else
                product(std::false_type{});
            const float mo = __shfl_xor_sync(kFull, m, 1);
            Prod<float> pr{h ? mo : m, e + __shfl_xor_sync(kFull, e, 1)};
            renorm_fast(pr);
            pr.m *= h ? m : mo;
            renorm_fast(pr);
            // over the lanes l as warp_prod_normalised: 16 across the warps, then 8 .. 1
            if (h == 0) xch[l] = make_float2(pr.m, __int_as_float(pr.e));
            __syncthreads();
            {
                const float2 o = xch[l ^ 16];
                pr.m *= o.x;
                pr.e += __float_as_int(o.y);
            }
#pragma unroll
            for (int off = 16; off > 1; off >>= 1) {
                pr.m *= __shfl_xor_sync(kFull, pr.m, off);
                pr.e += __shfl_xor_sync(kFull, pr.e, off);
            }
            renorm_fast(pr);
            const float d0 = -2.f * __shfl_sync(kFull, cur.aa, src) * si;
            const float delta = d0 + (__shfl_sync(kFull, cur.K, src) + prod_log(pr));
            const bool accept = __shfl_sync(kFull, cur.lu, src) < 2.f * delta;
            if (decisions && lane == 0) decisions[q0 + src] = accept ? 1 : 0;
            if (accept) {
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    if (u + 4 * kLoose < kU || 4 * l + 128 * u < M) {
                        const float2 v = *reinterpret_cast<const float2 *>(row_s + 128 * u);
                        t[u] = make_float2(flipped<true>(t[u].x, si * v.x), flipped<true>(t[u].y, si * v.y));
                    }
                }
                __syncwarp();
                if (lane == 0) {
                    sb[i >> 5] ^= 1u << (i & 31);
                    if (k >= 0) sb[k >> 5] ^= 1u << (k & 31);
                }
                __syncwarp();
                if (want_lp) lp += (double)delta;
                ++acc;
            }
        }
        cp_async_wait<0>();  // (a guess that turned out to be no move)
        __syncthreads();
        if (w >= A.n_discard) {
            const size_t row = (size_t)c * A.out_stride + A.out_offset + (w - A.n_discard);
            for (int i = tid; i < N; i += 64) A.samples[row * N + i] = spin(i) ? 1 : -1;
            if (tid == 0 && A.logpsi) A.logpsi[row] = lp;
        }
    }
    for (int i = tid; i < N; i += 64) A.s[(size_t)c * N + i] = spin(i) ? 1 : -1;
    if (tid == 0 && A.n_accepted) A.n_accepted[c] += acc;
}

// ----------------------------------------------------------- local energy ---

template <typename R>
struct ElocK {
    Tables<R> t;
    ElocArgs a;
    int warp_bytes, t_bytes, s_bytes;
    int units;  // 1: lanes over hidden units (large M), 0: lanes over connections
};

// One warp per sample.  theta and t are rebuilt from s; the connected
// configurations are spread over the lanes (sites for the Ising field term,
// antiparallel edges for the Heisenberg exchange term), each lane running
// over all hidden units with the unit-major tables.
template <typename R>
__global__ void __launch_bounds__(128) k_eloc(ElocK<R> P) {
    extern __shared__ __align__(16) unsigned char sm[];
    const Tables<R> &T = P.t;
    const ElocArgs &A = P.a;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t k = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    if (k >= A.Ns) return;
    const int N = T.N, M = T.M, E = T.E;
    unsigned char *base = sm + (size_t)warp * P.warp_bytes;
    using Tau = typename TauOf<R>::type;
    Tau *t = reinterpret_cast<Tau *>(base);
    int8_t *sv = reinterpret_cast<int8_t *>(base + P.t_bytes);
    int *list = reinterpret_cast<int *>(base + P.t_bytes + P.s_bytes);
    for (int i = lane; i < N; i += 32) sv[i] = A.s[(size_t)k * N + i];
    __syncwarp();
    bool nan = false;
    for (int j = lane; j < M; j += 32) {
        double th;
        if (A.theta_in) {
            th = A.theta_in[(size_t)k * M + j];
        } else if constexpr (sizeof(R) == 8) {
            th = fixed_theta(T, sv, j, theta_drop(N));
        } else {
            th = T.b[j];
            for (int i = 0; i < N; ++i) th = fma(T.Wt[(size_t)i * M + j], (double)sv[i], th);
        }
        const double tj = A.lib_tanh ? tanh(th) : tanh64(th);
        t[j] = to_tau<R>(tj);
        if (sizeof(R) == 8) nan |= tj != tj;
        if (A.t_out) A.t_out[(size_t)k * M + j] = tj;
    }
    // a NaN among the activations, which the integers of NK_F64 cannot hold, is
    // added to every ratio's logarithm
    const double poison =
        sizeof(R) == 8 && __any_sync(kFull, nan) ? __longlong_as_double(0x7FF8000000000000LL) : 0.0;
    // edges [0, E1) couple with J, the next-nearest ones [E1, E) with J2
    const int E1 = E - A.E2;
    double diag = 0.0;
    for (int e = lane; e < E; e += 32) {
        const int i = T.edges[2 * e], kk = T.edges[2 * e + 1];
        if ((unsigned)i < (unsigned)N && (unsigned)kk < (unsigned)N)
            diag += (e < E1 ? A.J : A.J2) * (double)sv[i] * (double)sv[kk];
    }
    __syncwarp();
    double off = 0.0;
    if (A.kind == NK_TFIM && P.units) {
        // large M: lanes over hidden units, one warp reduction per site
        for (int i = 0; i < N; ++i) {
            const R si = (R)sv[i];
            Prod<R> pr = strided_product(t, T.tau_site + (size_t)i * M, 1, si, lane, 32, M);
            pr = warp_prod(pr);
            const double delta = -2.0 * T.a[i] * (double)si + (double)(T.K_site[i] + prod_log(pr)) + poison;
            if (lane == 0) off += -A.h * exp(delta);
        }
    } else if (A.kind == NK_TFIM) {
        // small M: lanes over sites, each over all hidden units
        for (int i = lane; i < N; i += 32) {
            const R si = (R)sv[i];
            Prod<R> pr = strided_product(t, T.tau_siteT + i, (size_t)N, si, 0, 1, M);
            const double delta = -2.0 * T.a[i] * (double)si + (double)(T.K_site[i] + prod_log(pr)) + poison;
            off += -A.h * exp(delta);
        }
    } else {
        // compact the antiparallel edges
        int n = 0;
        for (int e0 = 0; e0 < E; e0 += 32) {
            const int e = e0 + lane;
            bool f = false;
            if (e < E) {
                const int i = T.edges[2 * e], kk = T.edges[2 * e + 1];
                f = (unsigned)i < (unsigned)N && (unsigned)kk < (unsigned)N && sv[i] != sv[kk];
            }
            const unsigned mask = __ballot_sync(kFull, f);
            if (f) list[n + __popc(mask & ((1u << lane) - 1u))] = e;
            n += __popc(mask);
        }
        __syncwarp();
        // off-diagonal elements; the Marshall sign flips only the edges that
        // join the two sublattices (the nearest-neighbour class)
        const double hoff = A.marshall ? -2.0 * A.J : 2.0 * A.J, hoff2 = 2.0 * A.J2;
        if (P.units) {
            for (int idx = 0; idx < n; ++idx) {
                const int e = list[idx];
                const int i = T.edges[2 * e], kk = T.edges[2 * e + 1];
                const R si = (R)sv[i];
                Prod<R> pr = strided_product(t, T.tau_edge + (size_t)e * M, 1, si, lane, 32, M);
                pr = warp_prod(pr);
                const double delta =
                    -2.0 * (double)si * (T.a[i] - T.a[kk]) + (double)(T.K_edge[e] + prod_log(pr)) + poison;
                if (lane == 0) off += (e < E1 ? hoff : hoff2) * exp(delta);
            }
        } else {
            for (int idx = lane; idx < n; idx += 32) {
                const int e = list[idx];
                const int i = T.edges[2 * e], kk = T.edges[2 * e + 1];
                const R si = (R)sv[i];
                Prod<R> pr = strided_product(t, T.tau_edgeT + e, (size_t)E, si, 0, 1, M);
                const double delta =
                    -2.0 * (double)si * (T.a[i] - T.a[kk]) + (double)(T.K_edge[e] + prod_log(pr)) + poison;
                off += (e < E1 ? hoff : hoff2) * exp(delta);
            }
        }
    }
    const double tot = warp_sum(diag + off);
    if (lane == 0) A.eloc[k] = tot;
}

// ------------------------------------------- sample-batched local energy ---
// Large M (NK_MIXED, theta given): one CTA of eloc_warps(kU) warps holds
// tanh(theta) of kEG samples in shared memory; every warp takes connections
// (sites, or edges) in turn, loads each tau row once (16-byte loads, lanes
// over units) and applies it to all kEG samples, so the tau traffic per ratio
// term drops kEG-fold.  One warp reduction per (connection, sample).
constexpr int kEG = 8;
// Warps per CTA.  At M >= 4096 the t of kEG samples (147 KB at M = 4608)
// leaves room for one CTA per SM, and the kernel waits on shared-memory and
// fixed latencies: 32 warps instead of 16 took the 24 x 24 local energies
// from 62.1 to 52.1 ms a step.
__host__ __device__ constexpr int eloc_warps(int kU) { return kU == 4 ? 32 : 16; }

struct ElocBK {
    Tables<float> t;
    ElocArgs a;
    int t_ld, s_ld;
};

// kU tau loads in flight per lane: 4 where M is large enough that the
// shared-memory t of kEG samples allows one CTA per SM anyway (M >= 4096),
// else 2 (the extra registers of 4 would halve the resident CTAs).
template <int kU>
__global__ void __launch_bounds__(eloc_warps(kU) * 32) k_eloc_batched(ElocBK P) {
    constexpr int kEW = eloc_warps(kU);
    extern __shared__ __align__(16) unsigned char sm[];
    const Tables<float> &T = P.t;
    const ElocArgs &A = P.a;
    const int N = T.N, M = T.M, E = T.E, E1 = E - A.E2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t k0 = (int64_t)blockIdx.x * kEG;
    const int G = (int)(A.Ns - k0 < kEG ? A.Ns - k0 : kEG);
    float *t = reinterpret_cast<float *>(sm);                                    // [kEG][t_ld]
    int8_t *sv = reinterpret_cast<int8_t *>(sm + (size_t)kEG * P.t_ld * 4);      // [kEG][s_ld]
    double *part = reinterpret_cast<double *>(sm + (size_t)kEG * P.t_ld * 4 + (size_t)kEG * P.s_ld);  // [kEW][kEG]
    double *diag = part + kEW * kEG;                                              // [kEG]
    float *offw = reinterpret_cast<float *>(diag + kEG);                          // [kEW][kEG]
    for (int x = threadIdx.x; x < kEG * N; x += blockDim.x) {
        const int g = x / N, i = x % N;
        sv[g * P.s_ld + i] = g < G ? A.s[(size_t)(k0 + g) * N + i] : (int8_t)1;
    }
    for (int x = threadIdx.x; x < kEG * M; x += blockDim.x) {
        const int g = x / M, j = x % M;
        float tv = 0.f;
        if (g < G) {
            const double th = A.theta_in[(size_t)(k0 + g) * M + j];
            const double tj = A.lib_tanh ? tanh(th) : tanh64(th);
            tv = (float)tj;
            if (A.t_out) A.t_out[(size_t)(k0 + g) * M + j] = tj;
        }
        t[g * P.t_ld + j] = tv;
    }
    __syncthreads();
    // diagonal part: warp g sums J_e s_i s_k over the edges of sample g
    if (warp < G) {
        double d = 0.0;
        const int8_t *s = sv + warp * P.s_ld;
        for (int e = lane; e < E; e += 32) {
            const int i = T.edges[2 * e], kk = T.edges[2 * e + 1];
            if ((unsigned)i < (unsigned)N && (unsigned)kk < (unsigned)N)
                d += (e < E1 ? A.J : A.J2) * (double)s[i] * (double)s[kk];
        }
        d = warp_sum(d);
        if (lane == 0) diag[warp] = d;
    }
    // FP32 path: ratios, exponentials and the per-warp partial sums in FP32
    // lanes (each warp adds about nconn / kEW terms); the diagonal part and
    // the final sum stay in FP64.
    if (lane < kEG) offw[warp * kEG + lane] = 0.f;
    __syncwarp();
    const bool tfim = A.kind == NK_TFIM;
    const int nconn = tfim ? N : E;
    const float hoff = (float)(A.marshall ? -2.0 * A.J : 2.0 * A.J), hoff2 = (float)(2.0 * A.J2),
                hfield = (float)(-A.h);
    for (int c = warp; c < nconn; c += kEW) {
        int i, kk = -1;
        const float *tau;
        float K, aa;
        if (tfim) {
            i = c;
            tau = T.tau_site + (size_t)c * M;
            K = T.K_site[c];
            aa = (float)T.a[i];
        } else {
            i = T.edges[2 * c];
            kk = T.edges[2 * c + 1];
            if ((unsigned)i >= (unsigned)N || (unsigned)kk >= (unsigned)N) continue;
            tau = T.tau_edge + (size_t)c * M;
            K = T.K_edge[c];
            aa = (float)(T.a[i] - T.a[kk]);
        }
        unsigned active = 0;
#pragma unroll
        for (int g = 0; g < kEG; ++g)
            if (g < G && (tfim || sv[g * P.s_ld + i] != sv[g * P.s_ld + kk])) active |= 1u << g;
        if (!active) continue;
        // The active samples of this connection as slots 0 .. cnt - 1 (in
        // increasing sample order, so every product is formed as before):
        // the loops below stop at cnt, so inactive samples cost nothing.
        // Those with s_i = +1 come first: the factors 1 - t tau of the one kind and 1 +
        // t tau of the other then differ in the sign of an FMA's operand, and a sample
        // takes kU chunks and their renormalisations in one go: 24 x 24 lattice, M =
        // 4608, 65536 samples: 50.8 ms with a multiplication by the sign and the
        // samples inside each chunk, 45.7 so (M = 1600: 3.0 ms either way).
        unsigned ups = 0;
#pragma unroll
        for (int g = 0; g < kEG; ++g) ups |= (unsigned)(sv[g * P.s_ld + i] > 0) << g;
        const int cnt = __popc(active), cnt_up = __popc(active & ups);
        float m[kEG];
        int ex[kEG];
        float sg[kEG];
        const float *tg[kEG];
        int gs[kEG];
        unsigned rest = active & ups, down = active & ~ups;
#pragma unroll
        for (int q = 0; q < kEG; ++q) {
            if (!rest) rest = down, down = 0;
            const int g = rest ? __ffs(rest) - 1 : 0;
            rest &= rest - 1u;
            gs[q] = g;
            m[q] = 1.f;
            ex[q] = 0;
            sg[q] = (float)sv[g * P.s_ld + i];
            tg[q] = t + (size_t)g * P.t_ld;
        }
        // This lane's units j = 4 lane + 128 it, it = j >> 7: the tau loads
        // of kU iterations are issued together (the row comes from L2), and
        // the products are renormalised after every odd iteration.
        for (int j0 = 4 * lane; j0 < M; j0 += kU * 128) {
            float4 uv[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u)
                uv[u] = j0 + u * 128 < M ? __ldg(reinterpret_cast<const float4 *>(tau + j0 + u * 128))
                                         : make_float4(0.f, 0.f, 0.f, 0.f);
            auto multiply = [&](int q, auto up) {
                constexpr bool kUp = decltype(up)::value;
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int j = j0 + u * 128;
                    if (j >= M) break;
                    const float4 tv = *reinterpret_cast<const float4 *>(tg[q] + j);
                    m[q] *= fmaf(kUp ? -tv.x : tv.x, uv[u].x, 1.f) * fmaf(kUp ? -tv.y : tv.y, uv[u].y, 1.f) *
                            fmaf(kUp ? -tv.z : tv.z, uv[u].z, 1.f) * fmaf(kUp ? -tv.w : tv.w, uv[u].w, 1.f);
                    if (u & 1) m[q] = renorm_bits(m[q], ex[q]);  // kU is even
                }
            };
#pragma unroll
            for (int q = 0; q < kEG; ++q) {
                if (q >= cnt) break;
                if (q < cnt_up)
                    multiply(q, std::true_type{});
                else
                    multiply(q, std::false_type{});
            }
        }
#pragma unroll
        for (int q = 0; q < kEG; ++q) {
            if (q >= cnt) break;
            Prod<float> p{m[q], ex[q]};
            renorm(p);
            p = warp_prod_normalised(p);
            const float delta = -2.f * aa * sg[q] + (K + prod_log(p));
            if (lane == 0) {
                float &o = offw[warp * kEG + gs[q]];
                o = fmaf(tfim ? hfield : (c < E1 ? hoff : hoff2), expf(delta), o);
            }
        }
    }
    __syncwarp();
    if (lane == 0) {
#pragma unroll
        for (int g = 0; g < kEG; ++g) part[warp * kEG + g] = (double)offw[warp * kEG + g];
    }
    __syncthreads();
    if (threadIdx.x < G) {
        double tot = diag[threadIdx.x];
        for (int w = 0; w < kEW; ++w) tot += part[w * kEG + threadIdx.x];
        A.eloc[k0 + threadIdx.x] = tot;
    }
}

// --------------------------------------------------------- batched theta ---

// T[k][j] = tanh(b_j + sum_i W_ji s_ki): 16 x 16 output tile per block, one
// output per thread, FP64 FMA (bound by the FP64 pipe: see k_gemm16).
__global__ void __launch_bounds__(256) k_theta_tanh(int N, int M, const double *__restrict__ b,
                                                    const double *__restrict__ W,
                                                    const int8_t *__restrict__ s, int64_t B,
                                                    double *__restrict__ T) {
    __shared__ double Sa[32][16 + 1];
    __shared__ double Wb[32][16 + 1];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t k0 = (int64_t)blockIdx.x * 16;
    const int j0 = blockIdx.y * 16;
    double acc = 0.0;
    for (int i0 = 0; i0 < N; i0 += 32) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int e = threadIdx.x + 256 * u, ii = e & 31, rr = e >> 5;
            const int64_t kk = k0 + rr;
            const int jj = j0 + rr, ic = i0 + ii;
            Sa[ii][rr] = (kk < B && ic < N) ? (double)s[(size_t)kk * N + ic] : 0.0;
            Wb[ii][rr] = (jj < M && ic < N) ? W[(size_t)jj * N + ic] : 0.0;
        }
        __syncthreads();
        const int n = N - i0 < 32 ? N - i0 : 32;
        for (int ii = 0; ii < n; ++ii) acc = fma(Sa[ii][ty], Wb[ii][tx], acc);
        __syncthreads();
    }
    const int64_t kk = k0 + ty;
    const int jj = j0 + tx;
    if (kk < B && jj < M) T[(size_t)kk * M + jj] = tanh64(acc + b[jj]);
}

template <typename R>
static int align16(int x) {
    return (x + 15) & ~15;
}

}  // namespace

// ------------------------------------------------------------- launchers ---

template <typename R>
cudaError_t launch_tables(const Tables<R> &t, bool need_site, bool need_edge, cudaStream_t st) {
    dim3 tb(32, 8), tg((t.N + 31) / 32, (t.M + 31) / 32);
    (k_transpose_W<<<tg, tb, 0, st>>>(t.N, t.M, t.W, t.Wt), nk::note_launch());
    if (need_site)
        (k_tau_rows<R><<<t.N, 256, 0, st>>>(t.N, t.M, t.N, t.Wt, nullptr, t.tau_site, t.tau_siteT,
                                           t.K_site, t.tauf_site, t.D_site), nk::note_launch());
    if (need_edge && t.E > 0)
        (k_tau_rows<R><<<t.E, 256, 0, st>>>(t.N, t.M, t.E, t.Wt, t.edges, t.tau_edge, t.tau_edgeT,
                                           t.K_edge, t.tauf_edge, t.D_edge), nk::note_launch());
    if (t.eW)
        (k_fix_weights<<<(t.M + 31) / 32, 256, 0, st>>>(t.N, t.M, t.Wt, t.eW), nk::note_launch());
    return cudaGetLastError();
}

template cudaError_t launch_tables<double>(const Tables<double> &, bool, bool, cudaStream_t);
template cudaError_t launch_tables<float>(const Tables<float> &, bool, bool, cudaStream_t);

cudaError_t launch_logpsi(int N, int M, const double *a, const double *b, const double *Wt,
                          const int8_t *s, int64_t B, double *out, cudaStream_t st) {
    if (B <= 0) return cudaSuccess;
    const int wpb = 4;
    size_t smem = (size_t)wpb * ((N + 15) & ~15);
    unsigned grid = (unsigned)((B + wpb - 1) / wpb);
    (k_logpsi<<<grid, 32 * wpb, smem, st>>>(N, M, a, b, Wt, s, B, out), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_logpsi_theta(int N, int M, const double *a, const double *theta, const int8_t *s, int64_t B,
                                double *out, cudaStream_t st) {
    if (B <= 0) return cudaSuccess;
    (k_logpsi_theta<<<(unsigned)((B + 7) / 8), 256, 0, st>>>(N, M, a, theta, s, B, out), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_tanh_inplace(int64_t n, double *x, bool lib, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    (k_tanh_inplace<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, x, lib), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_chain_init(int N, int C, int rule, uint64_t seed, uint32_t stream_id,
                              int8_t *s, cudaStream_t st) {
    if (C <= 0) return cudaSuccess;
    (k_chain_init<<<(C + 127) / 128, 128, 0, st>>>(N, C, rule, seed, stream_id, s), nk::note_launch());
    return cudaGetLastError();
}

// The register sweep for up to kC chunks of 128 units.
template <int kC>
cudaError_t launch_sweep_rows(SweepK<float> P, cudaStream_t st) {
    P.warp_bytes = kSweepAhead * P.t_bytes + 1024 + align16<float>(P.t.N);
    // two warps a block spread few chains more evenly over the SMs
    const int wpb = P.a.C <= 4864 ? 2 : 4;
    const size_t smem = (size_t)wpb * P.warp_bytes;
    cudaError_t err = nk::allow_max_dynamic_smem((const void *)k_sweep_rows<kC>);
    if (err != cudaSuccess) return err;
    const unsigned grid = (unsigned)((P.a.C + wpb - 1) / wpb);
    const int slot = prof_begin(NK_PROF_SWEEP, st);
    (k_sweep_rows<kC><<<grid, 32 * wpb, smem, st>>>(P), nk::note_launch());
    prof_end(slot, st, (double)P.a.C * (P.a.n_discard + P.a.n_samples) * P.t.N * (double)P.t.M);
    return cudaGetLastError();
}

// The two-warp sweep for up to kU chunks of 128 units.
template <int kU>
cudaError_t launch_sweep_pair(const SweepK<float> &P, cudaStream_t st) {
    const size_t smem = 2 * (size_t)P.t_bytes + 256 + 2 * (size_t)((P.t.N + 31) / 32) * 4;
    cudaError_t err = nk::allow_max_dynamic_smem((const void *)k_sweep_pair<kU>);
    if (err != cudaSuccess) return err;
    const int slot = prof_begin(NK_PROF_SWEEP, st);
    (k_sweep_pair<kU><<<(unsigned)P.a.C, 64, smem, st>>>(P), nk::note_launch());
    prof_end(slot, st, (double)P.a.C * (P.a.n_discard + P.a.n_samples) * P.t.N * (double)P.t.M);
    return cudaGetLastError();
}

// NK_F64: the screened kernel.  Shared memory holds theta (FP64), t (FP32) and
// the spins of each chain.
template <int kU>
cudaError_t launch_sweep_screened_regs(SweepK<double> P, cudaStream_t st) {
    P.warp_bytes = align16<double>(P.t.N);
    // one chain per scheduler while there are few: their warps do not share it
    const int wpb = P.a.C <= 152 ? 1 : 4;
    const unsigned grid = (unsigned)((P.a.C + wpb - 1) / wpb);
    const int slot = prof_begin(NK_PROF_SWEEP, st);
    if (P.a.C <= 1216)
        (k_sweep_screened_regs<kU, true><<<grid, 32 * wpb, wpb * P.warp_bytes, st>>>(P), nk::note_launch());
    else
        (k_sweep_screened_regs<kU, false><<<grid, 32 * wpb, wpb * P.warp_bytes, st>>>(P), nk::note_launch());
    prof_end(slot, st, (double)P.a.C * (P.a.n_discard + P.a.n_samples) * P.t.N * (double)P.t.M);
    return cudaGetLastError();
}

cudaError_t launch_sweep_screened(const SweepK<double> &P0, cudaStream_t st) {
    if (P0.a.rule != NK_RULE_HAMILTONIAN && P0.t.M <= 128)
        return P0.t.M <= 32 ? launch_sweep_screened_regs<1>(P0, st)
                            : (P0.t.M <= 64 ? launch_sweep_screened_regs<2>(P0, st)
                                            : launch_sweep_screened_regs<4>(P0, st));
    SweepK<double> P = P0;
    P.t_bytes = align16<double>(P.t.M * 8 + 8) / 32 * 32 + 32;  // theta; half of it holds t
    P.warp_bytes = P.t_bytes + P.t_bytes / 2 + align16<double>(P.t.N);
    int wpb = 4;
    while (wpb > 1 && (size_t)wpb * P.warp_bytes > 200 * 1024) wpb >>= 1;
    const size_t smem = (size_t)wpb * P.warp_bytes;
    if (smem > 227 * 1024) return cudaErrorInvalidValue;
    const bool ham = P.a.rule == NK_RULE_HAMILTONIAN;
    cudaError_t err = nk::allow_max_dynamic_smem(ham ? (const void *)k_sweep_screened<true>
                                                     : (const void *)k_sweep_screened<false>);
    if (err != cudaSuccess) return err;
    const unsigned grid = (unsigned)((P.a.C + wpb - 1) / wpb);
    const int slot = prof_begin(NK_PROF_SWEEP, st);
    if (ham)
        (k_sweep_screened<true><<<grid, 32 * wpb, smem, st>>>(P), nk::note_launch());
    else
        (k_sweep_screened<false><<<grid, 32 * wpb, smem, st>>>(P), nk::note_launch());
    prof_end(slot, st, (double)P.a.C * (P.a.n_discard + P.a.n_samples) * P.t.N * (double)P.t.M);
    return cudaGetLastError();
}

// The arguments of a sweep with the defaults filled in.
template <typename R>
SweepK<R> sweep_args(const Tables<R> &t, const SweepArgs &a) {
    SweepK<R> P;
    P.t = t;
    P.a = a;
    if (P.a.out_stride <= 0) {
        P.a.out_stride = a.n_samples;
        P.a.out_offset = 0;
    }
    if (P.a.dec_stride <= 0) {
        P.a.dec_stride = a.n_discard + a.n_samples;
        P.a.dec_offset = 0;
    }
    P.t_bytes = align16<R>(t.M * (int)sizeof(R));
    P.warp_bytes = P.t_bytes + align16<R>(t.N);
    P.vec4 = sizeof(R) == 4 && (t.M % 4) == 0;
    return P;
}

template <>
cudaError_t launch_sweep<double>(const Tables<double> &t, const SweepArgs &a, cudaStream_t st) {
    if (a.C <= 0 || a.n_discard + a.n_samples <= 0) return cudaSuccess;
    return launch_sweep_screened(sweep_args(t, a), st);
}

template <>
cudaError_t launch_sweep<float>(const Tables<float> &t, const SweepArgs &a, cudaStream_t st) {
    if (a.C <= 0 || a.n_discard + a.n_samples <= 0) return cudaSuccess;
    const SweepK<float> P = sweep_args(t, a);
    // local and exchange rules with theta given: t in registers, a warp a chain (two
    // are slower there: M = 400, 1024 chains: 0.10 and 0.13 ms a sweep) ...
    const int chunks = (t.M + 127) / 128;
    const bool regs = P.vec4 && a.rule != NK_RULE_HAMILTONIAN && a.theta_in;
    if (regs && chunks <= 4)
        return chunks == 1 ? launch_sweep_rows<1>(P, st)
                           : (chunks == 2 ? launch_sweep_rows<2>(P, st) : launch_sweep_rows<4>(P, st));
    // ... or two: from 25 chunks of 128 units (M = 4608, 8192 chains: 5.3 ms a sweep,
    // 6.8 by k_sweep; 256 chains: 0.74 and 1.19), and below with at most eight chains
    // an SM (M = 2000, 512 chains: 0.21 and 0.31 ms; M = 1600, 8192 chains: 3.7 and 3.0)
    if (regs && chunks <= 48 && (chunks > 24 || a.C <= 1216))
        return chunks <= 8    ? launch_sweep_pair<8>(P, st)
               : chunks <= 16 ? launch_sweep_pair<16>(P, st)
               : chunks <= 24 ? launch_sweep_pair<24>(P, st)
               : chunks <= 32 ? launch_sweep_pair<32>(P, st)
               : chunks <= 40 ? launch_sweep_pair<40>(P, st)
                              : launch_sweep_pair<48>(P, st);
    int wpb = 4;
    while (wpb > 1 && (size_t)wpb * P.warp_bytes > 200 * 1024) wpb >>= 1;
    size_t smem = (size_t)wpb * P.warp_bytes;
    if (smem > 227 * 1024) return cudaErrorInvalidValue;
    const bool ham = a.rule == NK_RULE_HAMILTONIAN;
    const bool ring = P.vec4 && t.M >= 6 * 512;
    const void *fn = ham ? (ring ? (const void *)k_sweep<true, true> : (const void *)k_sweep<true, false>)
                         : (ring ? (const void *)k_sweep<false, true> : (const void *)k_sweep<false, false>);
    cudaError_t err = nk::allow_max_dynamic_smem(fn);
    if (err != cudaSuccess) return err;
    unsigned grid = (unsigned)((a.C + wpb - 1) / wpb);
    const int slot = prof_begin(NK_PROF_SWEEP, st);
    if (ham && ring)
        (k_sweep<true, true><<<grid, 32 * wpb, smem, st>>>(P), nk::note_launch());
    else if (ham)
        (k_sweep<true, false><<<grid, 32 * wpb, smem, st>>>(P), nk::note_launch());
    else if (ring)
        (k_sweep<false, true><<<grid, 32 * wpb, smem, st>>>(P), nk::note_launch());
    else
        (k_sweep<false, false><<<grid, 32 * wpb, smem, st>>>(P), nk::note_launch());
    prof_end(slot, st, (double)a.C * (a.n_discard + a.n_samples) * t.N * (double)t.M);
    return cudaGetLastError();
}

size_t eloc_batched_smem(int N, int M, int warps) {
    const size_t t_ld = (size_t)(M + 3) / 4 * 4, s_ld = (size_t)(N + 15) / 16 * 16;
    return (size_t)kEG * t_ld * 4 + (size_t)kEG * s_ld + (size_t)(warps * kEG + kEG) * 8 + (size_t)warps * kEG * 4;
}

template <typename R>
cudaError_t launch_eloc_batched(const Tables<R> &, const ElocArgs &, cudaStream_t) {
    return cudaErrorNotSupported;
}

template <>
cudaError_t launch_eloc_batched<float>(const Tables<float> &t, const ElocArgs &a, cudaStream_t st) {
    ElocBK P;
    P.t = t;
    P.a = a;
    P.t_ld = (t.M + 3) / 4 * 4;
    P.s_ld = (t.N + 15) / 16 * 16;
    const bool wide = t.M >= 4096;
    const int warps = wide ? eloc_warps(4) : eloc_warps(2);
    const size_t smem = eloc_batched_smem(t.N, t.M, warps);
    if (smem > 227 * 1024) return cudaErrorInvalidValue;
    const void *fn = wide ? (const void *)k_eloc_batched<4> : (const void *)k_eloc_batched<2>;
    cudaError_t err = nk::allow_max_dynamic_smem(fn);
    if (err != cudaSuccess) return err;
    const unsigned grid = (unsigned)((a.Ns + kEG - 1) / kEG);
    const int slot = prof_begin(NK_PROF_ELOC, st);
    if (wide)
        (k_eloc_batched<4><<<grid, warps * 32, smem, st>>>(P), nk::note_launch());
    else
        (k_eloc_batched<2><<<grid, warps * 32, smem, st>>>(P), nk::note_launch());
    const double conn = a.kind == NK_TFIM ? (double)t.N : 0.5 * (double)t.E;
    prof_end(slot, st, (double)a.Ns * conn * (double)t.M);
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_eloc(const Tables<R> &t, const ElocArgs &a, cudaStream_t st) {
    if (a.Ns <= 0) return cudaSuccess;
    if (sizeof(R) == 4 && a.theta_in && t.M >= kUnitsMappingM && (t.M % 4) == 0 &&
        eloc_batched_smem(t.N, t.M, t.M >= 4096 ? eloc_warps(4) : eloc_warps(1)) <= 227 * 1024)
        return launch_eloc_batched<R>(t, a, st);
    ElocK<R> P;
    P.t = t;
    P.a = a;
    P.units = t.M >= kUnitsMappingM ? 1 : 0;
    P.t_bytes = align16<R>(t.M * (int)sizeof(R));
    P.s_bytes = align16<R>(t.N);
    P.warp_bytes = P.t_bytes + P.s_bytes + align16<R>(4 * (a.kind == NK_HEIS ? t.E : 0));
    int wpb = 4;
    while (wpb > 1 && (size_t)wpb * P.warp_bytes > 200 * 1024) wpb >>= 1;
    size_t smem = (size_t)wpb * P.warp_bytes;
    if (smem > 227 * 1024) return cudaErrorInvalidValue;
    cudaError_t err = nk::allow_max_dynamic_smem((const void *)k_eloc<R>);
    if (err != cudaSuccess) return err;
    unsigned grid = (unsigned)((a.Ns + wpb - 1) / wpb);
    const int slot = prof_begin(NK_PROF_ELOC, st);
    (k_eloc<R><<<grid, 32 * wpb, smem, st>>>(P), nk::note_launch());
    // nominal connections per sample: N sites (Ising field) or E / 2 edges
    // (antiparallel on average at S_z = 0)
    const double conn = a.kind == NK_TFIM ? (double)t.N : 0.5 * (double)t.E;
    prof_end(slot, st, (double)a.Ns * conn * (double)t.M);
    return cudaGetLastError();
}

template cudaError_t launch_eloc<double>(const Tables<double> &, const ElocArgs &, cudaStream_t);
template cudaError_t launch_eloc<float>(const Tables<float> &, const ElocArgs &, cudaStream_t);

cudaError_t launch_theta_tanh(int N, int M, const double *b, const double *W, const int8_t *s,
                              int64_t B, double *T, cudaStream_t st) {
    if (B <= 0) return cudaSuccess;
    dim3 grid((unsigned)((B + 15) / 16), (M + 15) / 16);
    (k_theta_tanh<<<grid, 256, 0, st>>>(N, M, b, W, s, B, T), nk::note_launch());
    return cudaGetLastError();
}

}  // namespace nk
