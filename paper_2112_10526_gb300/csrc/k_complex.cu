// The complex holomorphic RBM (NetKet 3, Sec. 3.2 with complex parameters)
// and the pieces of time-dependent variational Monte Carlo (Sec. 4.3):
//     ln psi(s) = a.s + sum_j ln cosh(b_j + W_j.s),  a, b, W complex,
// sampled from |psi|^2, with local energies, log-derivatives O = [s, tanh
// theta, tanh theta s^T] (holomorphic, Eq. eq:log-derivative-O) and the
// realified Jacobian whose Gram gives the real embedding of the complex QGT.
//
// Complex numbers are double2 (x = real, y = imaginary part); results are FP64
// on CUDA cores.  One warp per chain or sample, theta in shared memory.  A
// Metropolis decision needs only the sign of a real difference, which FP32
// with an error bound settles for nearly every proposal; the local energies
// take each amplitude ratio as one product over the hidden units.

#include <cuda_runtime.h>

#include "nk_common.cuh"
#include "nk_internal.h"

namespace nk {

namespace {

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
__device__ __forceinline__ double2 cexp(double2 z) {
    const double m = exp(z.x);
    double sn, cs;
    sincos(z.y, &sn, &cs);
    return make_double2(m * cs, m * sn);
}

// ln cosh z = y + ln(1 + e^{-2y}) - ln 2 with y = z or -z, whichever has a
// non-negative real part (cosh is even), so that |e^{-2y}| <= 1.  The
// logarithm of 1 + w takes its modulus through log1p and its argument
// through atan2.
__device__ __forceinline__ double2 clncosh(double2 z) {
    const double2 y = z.x >= 0.0 ? z : make_double2(-z.x, -z.y);
    const double2 w = cexp(make_double2(-2.0 * y.x, -2.0 * y.y));
    const double re = 0.5 * log1p(2.0 * w.x + w.x * w.x + w.y * w.y);
    const double im = atan2(w.y, 1.0 + w.x);
    return make_double2(y.x + re - 0.69314718055994530942, y.y + im);
}

// tanh z = (sinh 2x + i sin 2y) / (cosh 2x + cos 2y), z = x + i y; for |x|
// > 20 it is sign(x) to within e^{-40}.
__device__ __forceinline__ double2 ctanh(double2 z) {
    if (fabs(z.x) > 20.0) return make_double2(z.x > 0.0 ? 1.0 : -1.0, 0.0);
    double s2, c2;
    sincos(2.0 * z.y, &s2, &c2);
    const double d = cosh(2.0 * z.x) + c2;
    return make_double2(sinh(2.0 * z.x) / d, s2 / d);
}

__device__ __forceinline__ double2 warp_csum(double2 v) {
    v.x = warp_sum(v.x);
    v.y = warp_sum(v.y);
    return v;
}

// parameters: interleaved complex [a (N); b (M); W (M x N)]
struct CView {
    const double2 *a, *b, *W;
};
__device__ __forceinline__ CView cview(const double *p, int N, int M) {
    const double2 *q = reinterpret_cast<const double2 *>(p);
    return CView{q, q + N, q + N + M};
}

// theta_j = b_j + sum_i W_ji s_i for this lane's units; returns sum_i a_i s_i
// (lane 0 holds it after the reduction).
__device__ __forceinline__ double2 hidden(const CView &v, int N, int M, const int8_t *sv, double2 *th, int lane) {
    for (int j = lane; j < M; j += 32) {
        double2 acc = v.b[j];
        for (int i = 0; i < N; ++i) {
            const double si = (double)sv[i];
            acc.x = fma(v.W[(size_t)j * N + i].x, si, acc.x);
            acc.y = fma(v.W[(size_t)j * N + i].y, si, acc.y);
        }
        th[j] = acc;
    }
    double2 as = make_double2(0.0, 0.0);
    for (int i = lane; i < N; i += 32) as = cadd(as, cscale(v.a[i], (double)sv[i]));
    return warp_csum(as);
}

// ln psi(s') - ln psi(s) for the n sites flipped (term by term on the moved
// activations theta_j - 2 sum W_ji s_i); warp-uniform result.
__device__ __forceinline__ double2 clog_ratio(const CView &v, int N, int M, const int8_t *sv, const double2 *th,
                                              const int *sites, int n, int lane) {
    double2 d = make_double2(0.0, 0.0);
    for (int j = lane; j < M; j += 32) {
        double2 tp = th[j];
        for (int r = 0; r < n; ++r) {
            const double s2 = 2.0 * (double)sv[sites[r]];
            const double2 w = v.W[(size_t)j * N + sites[r]];
            tp.x -= s2 * w.x;
            tp.y -= s2 * w.y;
        }
        d = cadd(d, csub(clncosh(tp), clncosh(th[j])));
    }
    d = warp_csum(d);
    for (int r = 0; r < n; ++r) d = csub(d, cscale(v.a[sites[r]], 2.0 * (double)sv[sites[r]]));
    return d;
}

// ---------------------------------------------------------------- ln psi ---

__global__ void k_crbm_logpsi(int N, int M, const double *__restrict__ p, const int8_t *__restrict__ s, int64_t B,
                              double *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t k = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    const size_t wb = ((size_t)M * sizeof(double2) + (size_t)N + 15) / 16 * 16;
    double2 *th = reinterpret_cast<double2 *>(sm + warp * wb);
    int8_t *sv = reinterpret_cast<int8_t *>(th + M);
    if (k >= B) return;
    for (int i = lane; i < N; i += 32) sv[i] = s[(size_t)k * N + i];
    __syncwarp();
    const CView v = cview(p, N, M);
    double2 lp = hidden(v, N, M, sv, th, lane);
    __syncwarp();
    double2 acc = make_double2(0.0, 0.0);
    for (int j = lane; j < M; j += 32) acc = cadd(acc, clncosh(th[j]));
    acc = warp_csum(acc);
    lp = cadd(lp, acc);
    if (lane == 0) reinterpret_cast<double2 *>(out)[k] = lp;
}

// ------------------------------------------------------------ Metropolis ---
// Chains on |psi|^2 on the Philox streams of the real RBM: proposal p of
// sweep w uses the block ((sweep0 + w) N + p, chain, stream_id, 0); site or
// edge floor(hi32(y0) n / 2^32), u = ((y1 >> 11) + 1/2) 2^-53, accept iff
// ln u < 2 Re[ln psi(s') - ln psi(s)]; an exchange on equal spins is not a
// move.  theta is rebuilt from scratch at every sweep and moved on accepted
// flips.

struct CSweepArgs {
    int N, M, E, rule, C;
    const double *p;
    const int32_t *edges;
    int8_t *s;
    int64_t sweep0;
    int n_discard, n_samples;
    unsigned long long seed;
    unsigned stream_id;
    int8_t *samples;  // [C][n_samples][N]
    unsigned long long *n_accepted;
    int warp_bytes;
};

// Re ln cosh z + ln 2 in FP32 (g.x) and a bound on its error (g.y):
// |x| + ln(w) / 2 with w = |1 + e^{-2y}|^2 = (1 - E)^2 + 4 E cos^2 Im z, E =
// e^{-2 |x|}, x = Re z.  Rounding z, the exponential, the cosine and the
// square leave w within 2^-18 (1 + |x| + |y|) (relative to w it is that over
// w, also through the poles' growth of the derivative, 2 / sqrt w), the
// logarithm and the sum within 2^-22 (1 + |x|).  No bound (infinite) below w =
// 2^-6, near the zeros of cosh, and for a NaN.
__device__ __forceinline__ float2 re_lncosh_bounded(double2 z) {
    const float x = fabsf((float)z.x), y = (float)z.y;
    const float E = expf(-2.f * x), c = cosf(y), o = 1.f - E;
    const float w = fmaf(4.f * E * c, c, o * o);
    const float e = __fdividef(3.8146973e-6f * (1.f + x + fabsf(y)), w);
    return make_float2(x + 0.5f * logf(w), w >= 0.015625f ? e : __int_as_float(0x7F800000));
}

// One warp per chain.  The move is accepted iff ln u < 2 Re[ln psi(s') - ln
// psi(s)].  Both sides are first taken in FP32 from Re ln cosh of the moved
// units (that of the present ones is kept), with the sum of the units' error
// bounds: a difference above it decides.  Otherwise (about one proposal in a
// few thousand at M = 20) the FP64 log-ratio of clog_ratio decides, which
// used to be taken for every proposal: two complex ln cosh a unit, some 150
// FP64 operations each on a pipe of 2 lanes a clock and SM.  theta stays in
// FP64.  20 sites, M = 20, 1024 chains, 24 sweeps: 11.4 ms
// with every proposal in FP64, 0.29 now.
__global__ void __launch_bounds__(128) k_crbm_sweep(CSweepArgs A) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * (blockDim.x >> 5) + warp;
    const int N = A.N, M = A.M;
    double2 *th = reinterpret_cast<double2 *>(sm + (size_t)warp * A.warp_bytes);
    float2 *g = reinterpret_cast<float2 *>(th + M);  // Re ln cosh theta + ln 2 and its error bound
    int8_t *sv = reinterpret_cast<int8_t *>(g + M);
    if (c >= A.C) return;
    for (int i = lane; i < N; i += 32) sv[i] = A.s[(size_t)c * N + i];
    __syncwarp();
    const CView v = cview(A.p, N, M);
    unsigned long long acc = 0;
    for (int w = 0; w < A.n_discard + A.n_samples; ++w) {
        hidden(v, N, M, sv, th, lane);
        for (int j = lane; j < M; j += 32) g[j] = re_lncosh_bounded(th[j]);  // the lane's own units
        __syncwarp();
        const unsigned long long qbase = (unsigned long long)(A.sweep0 + w) * (unsigned long long)N;
        int b_i = 0, b_k = 0, b_ok = 1;
        double b_u = 1.0;
        float b_h = 0.f, b_a2 = 0.f;  // ln u / 2, 2 Re(a_i - a_k)
        for (int q = 0; q < N; ++q) {
            const int src = q & 31;
            if (src == 0) {  // lane l prepares proposal q + l
                const Philox4 y = philox4x64_10(qbase + (unsigned long long)(q + lane), (unsigned long long)c,
                                                (unsigned long long)A.stream_id, 0ULL, A.seed, 0ULL);
                b_u = uniform53(y.v[1]);
                b_h = 0.5f * logf((float)b_u);
                if (A.rule == NK_RULE_LOCAL) {
                    b_i = pick_index(y.v[0], N);
                    b_a2 = (float)(2.0 * v.a[b_i].x);
                } else {
                    const int e = pick_index(y.v[0], A.E);
                    const int i0 = A.edges[2 * e], k0 = A.edges[2 * e + 1];
                    b_ok = (unsigned)i0 < (unsigned)N && (unsigned)k0 < (unsigned)N;
                    b_i = b_ok ? i0 : 0;
                    b_k = b_ok ? k0 : 0;
                    b_a2 = b_ok ? (float)(2.0 * (v.a[b_i].x - v.a[b_k].x)) : 0.f;
                }
            }
            int sites[2] = {__shfl_sync(0xffffffffu, b_i, src), __shfl_sync(0xffffffffu, b_k, src)};
            const float h = __shfl_sync(0xffffffffu, b_h, src), a2 = __shfl_sync(0xffffffffu, b_a2, src);
            const int ok = __shfl_sync(0xffffffffu, b_ok, src);
            const int n = A.rule == NK_RULE_LOCAL ? 1 : 2;
            if (n == 2 && (!ok || sv[sites[0]] == sv[sites[1]])) continue;
            const double s0 = 2.0 * (double)sv[sites[0]];
            auto moved = [&](int j) {
                double2 t = th[j];
                const double2 w0 = v.W[(size_t)j * N + sites[0]];
                t.x = fma(-s0, w0.x, t.x);
                t.y = fma(-s0, w0.y, t.y);
                if (n == 2) {  // s_k = -s_i
                    const double2 w1 = v.W[(size_t)j * N + sites[1]];
                    t.x = fma(s0, w1.x, t.x);
                    t.y = fma(s0, w1.y, t.y);
                }
                return t;
            };
            // sum_j Re[ln cosh theta' - ln cosh theta] > ln u / 2 + 2 Re(a-part) s
            const float thr = fmaf(a2, (float)sv[sites[0]], h);
            float d = 0.f, err = 0.f;
            float2 g0 = make_float2(0.f, 0.f);
            double2 t0 = make_double2(0.0, 0.0);
            for (int j = lane; j < M; j += 32) {
                t0 = moved(j);
                g0 = re_lncosh_bounded(t0);
                d += g0.x - g[j].x;
                err += g0.y + g[j].y + 4.7683716e-7f * (fabsf(g0.x) + fabsf(g[j].x));
            }
            d = warp_sum(d);
            err = warp_sum(err) + 4.7683716e-7f * (fabsf(h) + fabsf(a2)) + 1.9073486e-6f;
            bool accept;
            if (fabsf(d - thr) > err) {  // false for an infinite bound and for NaNs
                accept = d > thr;
            } else {
                const double2 d2 = clog_ratio(v, N, M, sv, th, sites, n, lane);
                accept = log(__shfl_sync(0xffffffffu, b_u, src)) < 2.0 * d2.x;
            }
            if (accept) {
                if (M <= 32) {  // the lane's only unit is still in registers
                    if (lane < M) {
                        th[lane] = t0;
                        g[lane] = g0;
                    }
                } else {
                    for (int j = lane; j < M; j += 32) {
                        const double2 t = moved(j);
                        th[j] = t;
                        g[j] = re_lncosh_bounded(t);
                    }
                }
                __syncwarp();
                if (lane == 0)
                    for (int r = 0; r < n; ++r) sv[sites[r]] = (int8_t)-sv[sites[r]];
                ++acc;
            }
            __syncwarp();
        }
        if (w >= A.n_discard) {
            const size_t row = (size_t)c * A.n_samples + (w - A.n_discard);
            for (int i = lane; i < N; i += 32) A.samples[row * N + i] = sv[i];
        }
        __syncwarp();
    }
    for (int i = lane; i < N; i += 32) A.s[(size_t)c * N + i] = sv[i];
    if (lane == 0 && A.n_accepted) A.n_accepted[c] += acc;
}

// ----------------------------------------------------------- local energy ---
// E_loc(s) = sum_s' H_ss' psi(s')/psi(s) (Eq. eq:local-estimator): diagonal
// sum_e J_e s_i s_k; TFIM: -h e^{dlnpsi} per single flip; Heisenberg: the
// element (+-2 J_e, Marshall sign on the nearest-neighbour class) per
// antiparallel edge.  out: complex [Ns].

// An amplitude ratio is a product over the hidden units: with p_j = 1 / (1 +
// e^{-2 theta_j}) and q_j = 1 - p_j = 1 / (1 + e^{2 theta_j}),
//     cosh(theta_j - d_j) / cosh theta_j = e^{-d_j} p_j + e^{d_j} q_j,
// which has no cancellation of its own (both terms are positive for real
// arguments; a small sum is a theta_j - d_j near a zero of cosh, where ln cosh
// is as sensitive).  e^{+-2 W_ji} come from a table (one exponential per weight
// instead of two complex ln cosh per weight and sample), so a term costs 12
// FP64 operations for a flip and 20 for a pair against about 300.  Lanes run
// over the connected configurations, the tables are unit-major as W is, so the
// lanes' loads coalesce and no reduction is needed per ratio.  20 sites, M =
// 20, 4096 samples: 1.7 ms with the logarithms, 0.16 now.
// The exponentials stay in range, and above the subnormal numbers, for |Re 2 W| <=
// 170 and |Re theta| <= 300 (|d| <= 340, the running product within e^{+-166}).
// Samples beyond, and those whose sum is not finite for another reason, take the
// differences of ln cosh.
constexpr double kMaxRe2W = 170.0, kMaxReTheta = 300.0;

struct CElocArgs {
    int N, M, E, E2, kind, marshall;
    double J, J2, h;
    const double *p;
    const double2 *ep, *em;  // e^{2 W}, e^{-2 W}, [M][N]; null: by logarithms
    const int32_t *edges;
    const int8_t *s;
    int64_t Ns;
    double *eloc;
    int warp_bytes, pq_bytes, s_bytes;
    int compact;  // the antiparallel edges are listed in shared memory first
};

__global__ void k_crbm_exp_tables(int64_t n, const double2 *__restrict__ W, double2 *__restrict__ ep,
                                  double2 *__restrict__ em) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double sn, cs;
    sincos(2.0 * W[i].y, &sn, &cs);
    double a = exp(2.0 * W[i].x), b = exp(-2.0 * W[i].x);
    if (!(fabs(2.0 * W[i].x) <= kMaxRe2W)) a = b = __longlong_as_double(0x7FF8000000000000LL);
    ep[i] = make_double2(a * cs, a * sn);
    em[i] = make_double2(b * cs, -b * sn);
}

// 1 / (1 + e^{-2z}) and 1 / (1 + e^{2z}), from the exponential that does not
// grow: with y = +-z, Re y >= 0, w = e^{-2y}: 1 / (1 + w) and w / (1 + w).
__device__ __forceinline__ void logistic_pair(double2 z, double2 &p, double2 &q) {
    const bool neg = z.x < 0.0;
    const double2 y = neg ? make_double2(-z.x, -z.y) : z;
    const double2 w = cexp(make_double2(-2.0 * y.x, -2.0 * y.y));
    const double2 o = make_double2(1.0 + w.x, w.y);
    const double inv = 1.0 / (o.x * o.x + o.y * o.y);
    const double2 a = make_double2(o.x * inv, -o.y * inv), b = cmul(w, a);
    p = neg ? b : a;
    q = neg ? a : b;
}

// The off-diagonal part by logarithms, one connected configuration after the other,
// the lanes over the hidden units; th: room for theta.
__device__ __noinline__ double2 log_offdiag(const CElocArgs &A, const CView &v, const int8_t *sv, double2 *th,
                                            int lane) {
    const int N = A.N, M = A.M, E1 = A.E - A.E2;
    __syncwarp();
    hidden(v, N, M, sv, th, lane);
    __syncwarp();
    double2 off = make_double2(0.0, 0.0);
    if (A.kind == NK_TFIM) {
        for (int i = 0; i < N; ++i)
            off = cadd(off, cscale(cexp(clog_ratio(v, N, M, sv, th, &i, 1, lane)), -A.h));
        return off;
    }
    for (int e = 0; e < A.E; ++e) {
        const int pair[2] = {A.edges[2 * e], A.edges[2 * e + 1]};
        if ((unsigned)pair[0] >= (unsigned)N || (unsigned)pair[1] >= (unsigned)N || sv[pair[0]] == sv[pair[1]]) continue;
        const double el = e < E1 ? (A.marshall ? -2.0 * A.J : 2.0 * A.J) : 2.0 * A.J2;
        off = cadd(off, cscale(cexp(clog_ratio(v, N, M, sv, th, pair, 2, lane)), el));
    }
    return off;
}

__global__ void __launch_bounds__(128) k_crbm_eloc(CElocArgs A) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t k = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    const int N = A.N, M = A.M, E1 = A.E - A.E2;
    unsigned char *base = sm + (size_t)warp * A.warp_bytes;
    double2 *pq = reinterpret_cast<double2 *>(base);  // [M][2]
    int8_t *sv = reinterpret_cast<int8_t *>(base + A.pq_bytes);
    int *list = reinterpret_cast<int *>(base + A.pq_bytes + A.s_bytes);
    if (k >= A.Ns) return;
    for (int i = lane; i < N; i += 32) sv[i] = A.s[(size_t)k * N + i];
    __syncwarp();
    const CView v = cview(A.p, N, M);
    hidden(v, N, M, sv, pq, lane);  // theta in pq[0 .. M - 1]
    __syncwarp();
    bool beyond = false;  // (also for a NaN)
    for (int j = lane; j < M; j += 32) beyond |= !(fabs(pq[j].x) <= kMaxReTheta);
    // (p, q) of the units from the last to the first block of 32: a block's
    // theta is read by its lanes before pairs are written over it
    for (int j0 = (M - 1) / 32 * 32; j0 >= 0; j0 -= 32) {
        const int j = j0 + lane;
        double2 p = make_double2(0.0, 0.0), q = p;
        if (j < M) logistic_pair(pq[j], p, q);
        __syncwarp();
        if (j < M) {
            pq[2 * j] = p;
            pq[2 * j + 1] = q;
        }
        __syncwarp();
    }
    double diag = 0.0;
    for (int e = lane; e < A.E; e += 32) {
        const int i = A.edges[2 * e], kk = A.edges[2 * e + 1];
        if ((unsigned)i < (unsigned)N && (unsigned)kk < (unsigned)N)
            diag += (e < E1 ? A.J : A.J2) * (double)sv[i] * (double)sv[kk];
    }
    // the connected configurations: the N sites, or the antiparallel edges
    // (all edges, the parallel ones skipped, where the list does not fit)
    int n = A.kind == NK_TFIM ? N : A.E;
    if (A.compact) {
        n = 0;
        for (int e0 = 0; e0 < A.E; e0 += 32) {
            const int e = e0 + lane;
            bool f = false;
            if (e < A.E) {
                const int i = A.edges[2 * e], kk = A.edges[2 * e + 1];
                f = (unsigned)i < (unsigned)N && (unsigned)kk < (unsigned)N && sv[i] != sv[kk];
            }
            const unsigned mask = __ballot_sync(0xffffffffu, f);
            if (f) list[n + __popc(mask & ((1u << lane) - 1u))] = e;
            n += __popc(mask);
        }
        __syncwarp();
    }
    double2 off = make_double2(0.0, 0.0);
    if (!A.ep) {
        beyond = true;
        n = 0;
    }
    for (int x = lane; x < n; x += 32) {
        int i = x, kk = -1;
        double el = -A.h;
        if (A.kind != NK_TFIM) {
            const int e = A.compact ? list[x] : x;
            i = A.edges[2 * e];
            kk = A.edges[2 * e + 1];
            if (!A.compact && ((unsigned)i >= (unsigned)N || (unsigned)kk >= (unsigned)N || sv[i] == sv[kk])) continue;
            el = e < E1 ? (A.marshall ? -2.0 * A.J : 2.0 * A.J) : 2.0 * A.J2;
        }
        // d_j = 2 s_i (W_ji - W_jk): e^{-d} is em for s_i = 1, ep for s_i = -1
        const bool up = sv[i] > 0;
        const double2 *dn = (up ? A.em : A.ep), *gr = (up ? A.ep : A.em);
        double2 r = make_double2(1.0, 0.0);
        int ex = 0;
        for (int j = 0; j < M; ++j) {
            const size_t at = (size_t)j * N;
            double2 a = dn[at + i], b = gr[at + i];
            if (kk >= 0) {
                a = cmul(a, gr[at + kk]);
                b = cmul(b, dn[at + kk]);
            }
            const double2 p = pq[2 * j], q = pq[2 * j + 1];
            const double2 f = make_double2(fma(b.x, q.x, -b.y * q.y) + fma(a.x, p.x, -a.y * p.y),
                                           fma(b.x, q.y, b.y * q.x) + fma(a.x, p.y, a.y * p.x));
            r = cmul(r, f);
            // keep the product's exponent within +-240
            const int eb = max((__double2hiint(r.x) >> 20) & 0x7FF, (__double2hiint(r.y) >> 20) & 0x7FF) - 1023;
            if ((eb > 240 && eb < 1024) || (eb < -240 && eb > -1023)) {
                r.x = ldexp(r.x, -eb);
                r.y = ldexp(r.y, -eb);
                ex += eb;
            }
        }
        // e^{-2 s_i (a_i - a_k)} 2^ex, the product brought to [1, 2) first
        const int eb = max((__double2hiint(r.x) >> 20) & 0x7FF, (__double2hiint(r.y) >> 20) & 0x7FF) - 1023;
        if (eb < 1024 && eb > -1023) {
            r.x = ldexp(r.x, -eb);
            r.y = ldexp(r.y, -eb);
            ex += eb;
        }
        double2 av = v.a[i];
        if (kk >= 0) av = csub(av, v.a[kk]);
        const double sg = up ? -2.0 : 2.0;
        double2 z = cscale(av, sg);
        z.x += (double)ex * 0.69314718055994530942;
        off = cadd(off, cscale(cmul(r, cexp(z)), el));
    }
    beyond |= !isfinite(off.x) || !isfinite(off.y);
    off = warp_csum(off);
    diag = warp_sum(diag);
    if (__any_sync(0xffffffffu, beyond)) off = log_offdiag(A, v, sv, pq, lane);
    if (lane == 0) reinterpret_cast<double2 *>(A.eloc)[k] = make_double2(diag + off.x, off.y);
}

// --------------------------------------------------------------- Jacobian ---
// O [Ns][Np] complex: O_a = s, O_b = tanh theta, O_W = tanh theta s^T.
__global__ void k_crbm_jacobian(int N, int M, const double *__restrict__ p, const int8_t *__restrict__ s,
                                int64_t Ns, double *__restrict__ O) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t k = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
    const size_t wb = ((size_t)M * sizeof(double2) + (size_t)N + 15) / 16 * 16;
    double2 *th = reinterpret_cast<double2 *>(sm + warp * wb);
    int8_t *sv = reinterpret_cast<int8_t *>(th + M);
    if (k >= Ns) return;
    for (int i = lane; i < N; i += 32) sv[i] = s[(size_t)k * N + i];
    __syncwarp();
    const CView v = cview(p, N, M);
    hidden(v, N, M, sv, th, lane);
    __syncwarp();
    for (int j = lane; j < M; j += 32) th[j] = ctanh(th[j]);
    __syncwarp();
    const int64_t Np = (int64_t)N + M + (int64_t)M * N;
    double2 *row = reinterpret_cast<double2 *>(O) + (size_t)k * Np;
    for (int i = lane; i < N; i += 32) row[i] = make_double2((double)sv[i], 0.0);
    for (int j = lane; j < M; j += 32) row[N + j] = th[j];
    for (int64_t q = lane; q < (int64_t)M * N; q += 32) {
        const int j = (int)(q / N), i = (int)(q % N);
        row[N + M + q] = cscale(th[j], (double)sv[i]);
    }
}

// Column means of a complex [rows][cols] matrix: 32 columns a block, 32 threads
// a column (one thread a column waited on its loads: 0.8 ms for 440 columns of
// 4096 rows, 0.085 now), summed in a fixed order.
__global__ void __launch_bounds__(1024) k_ccolmean(int64_t rows, int64_t cols, const double2 *__restrict__ O,
                                                   double2 *__restrict__ mean) {
    __shared__ double2 part[32][33];
    const int c = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int64_t q = (int64_t)blockIdx.x * 32 + c;
    double2 acc = make_double2(0.0, 0.0);
    if (q < cols) {
#pragma unroll 4
        for (int64_t k = y; k < rows; k += 32) acc = cadd(acc, O[(size_t)k * cols + q]);
    }
    part[c][y] = acc;
    __syncthreads();
    const double2 v = warp_csum(part[y][c]);  // warp y sums column y of the block
    const int64_t qo = (int64_t)blockIdx.x * 32 + y;
    if (c == 0 && qo < cols) mean[qo] = cscale(v, 1.0 / (double)rows);
}

// The realified centred Jacobian R [2 rows][2 cols]: with dO = X + i Y
// (centred), row 2k = [X_k, -Y_k], row 2k + 1 = [Y_k, X_k], so that
// R^T R = Ns [[Re G, -Im G], [Im G, Re G]] for G = dO^H dO / Ns.
__global__ void k_realify(int64_t rows, int64_t cols, const double2 *__restrict__ O, const double2 *__restrict__ mean,
                          double *__restrict__ R) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= rows * cols) return;
    const int64_t k = idx / cols, q = idx % cols;
    const double2 d = csub(O[idx], mean[q]);
    double *r0 = R + (size_t)(2 * k) * (2 * cols), *r1 = r0 + 2 * cols;
    r0[q] = d.x;
    r0[cols + q] = -d.y;
    r1[q] = d.y;
    r1[cols + q] = d.x;
}

// The realified right-hand side of the force: g [2 Ns] with g_2k = Re(E_k -
// Ebar) / Ns, g_2k+1 = Im(E_k - Ebar) / Ns, so that R^T g = [Re f; Im f] for
// f = dO^H (E - Ebar) / Ns.  Ebar: complex mean (emean).
__global__ void k_cforce_g(int64_t Ns, const double2 *__restrict__ e, const double2 *__restrict__ emean,
                           double *__restrict__ g) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Ns) return;
    const double2 d = csub(e[k], *emean);
    g[2 * k] = d.x / (double)Ns;
    g[2 * k + 1] = d.y / (double)Ns;
}

// Complex mean and variance of the local energies (one block; fixed order):
// out = [Re mean, Im mean, var = mean |E - Ebar|^2, error sqrt(var / Ns)].
__global__ void k_cstats(int64_t Ns, const double2 *__restrict__ e, double *__restrict__ out) {
    __shared__ double red[3][32];
    double sr = 0.0, si = 0.0;
    for (int64_t k = threadIdx.x; k < Ns; k += blockDim.x) {
        sr += e[k].x;
        si += e[k].y;
    }
    sr = warp_sum(sr);
    si = warp_sum(si);
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = sr;
        red[1][threadIdx.x >> 5] = si;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        double u = threadIdx.x < (blockDim.x >> 5) ? red[0][threadIdx.x] : 0.0;
        double v = threadIdx.x < (blockDim.x >> 5) ? red[1][threadIdx.x] : 0.0;
        u = warp_sum(u);
        v = warp_sum(v);
        if (threadIdx.x == 0) {
            red[0][0] = u / (double)Ns;
            red[1][0] = v / (double)Ns;
        }
    }
    __syncthreads();
    const double mr = red[0][0], mi = red[1][0];
    __syncthreads();
    double q = 0.0;
    for (int64_t k = threadIdx.x; k < Ns; k += blockDim.x) {
        const double dr = e[k].x - mr, di = e[k].y - mi;
        q += dr * dr + di * di;
    }
    q = warp_sum(q);
    if ((threadIdx.x & 31) == 0) red[2][threadIdx.x >> 5] = q;
    __syncthreads();
    if (threadIdx.x < 32) {
        double v = threadIdx.x < (blockDim.x >> 5) ? red[2][threadIdx.x] : 0.0;
        v = warp_sum(v);
        if (threadIdx.x == 0) {
            out[0] = mr;
            out[1] = mi;
            out[2] = v / (double)Ns;
            out[3] = sqrt(v / (double)Ns / (double)Ns);
        }
    }
}

// The TDVP right-hand side gamma f from the realified force [Re f; Im f]
// (n complex entries): gamma = -i (real time): [Im f; -Re f]; gamma = -1
// (imaginary time): [-Re f; -Im f].
__global__ void k_tdvp_rhs(int64_t n, const double *__restrict__ f, int real_time, double *__restrict__ rhs) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const double fr = f[q], fi = f[n + q];
    rhs[q] = real_time ? fi : -fr;
    rhs[n + q] = real_time ? -fr : -fi;
}

// theta (interleaved complex, n entries) <- base + h x with x realified
// [Re; Im]; base == null reads as zero.
__global__ void k_caxpy_realified(int64_t n, const double *base, double h, const double *__restrict__ x,
                                  double *out) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const double b0 = base ? base[2 * q] : 0.0, b1 = base ? base[2 * q + 1] : 0.0;
    out[2 * q] = b0 + h * x[q];
    out[2 * q + 1] = b1 + h * x[n + q];
}

size_t cwarp_bytes(int N, int M) { return ((size_t)M * sizeof(double2) + (size_t)N + 15) / 16 * 16; }

}  // namespace

size_t crbm_smem_per_warp(int N, int M) { return cwarp_bytes(N, M); }

cudaError_t launch_crbm_logpsi(int N, int M, const double *p, const int8_t *s, int64_t B, double *out,
                               cudaStream_t st) {
    if (B <= 0) return cudaSuccess;
    const size_t smem = 4 * cwarp_bytes(N, M);
    cudaError_t e = nk::allow_max_dynamic_smem((const void *)k_crbm_logpsi);
    if (e != cudaSuccess) return e;
    (k_crbm_logpsi<<<nblk(B, 4), 128, smem, st>>>(N, M, p, s, B, out), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_crbm_sweep(int N, int M, const double *p, int rule, int E, const int32_t *edges, int C, int8_t *s,
                              int64_t sweep0, int n_discard, int n_samples, uint64_t seed, uint32_t stream_id,
                              int8_t *samples, unsigned long long *n_accepted, cudaStream_t st) {
    if (C <= 0) return cudaSuccess;
    const int wb = (int)(((size_t)M * (sizeof(double2) + sizeof(float2)) + (size_t)N + 15) / 16 * 16);
    CSweepArgs a{N, M, E, rule, C, p, edges, s, sweep0, n_discard, n_samples, seed, stream_id, samples, n_accepted,
                 wb};
    int wpb = 4;
    while (wpb > 1 && (size_t)wpb * wb > 227 * 1024) wpb >>= 1;
    if ((size_t)wpb * wb > 227 * 1024) return cudaErrorInvalidValue;
    cudaError_t e = nk::allow_max_dynamic_smem((const void *)k_crbm_sweep);
    if (e != cudaSuccess) return e;
    const int slot = prof_begin(NK_PROF_SWEEP, st);
    (k_crbm_sweep<<<nblk(C, wpb), 32 * wpb, (size_t)wpb * wb, st>>>(a), nk::note_launch());
    prof_end(slot, st, (double)C * (n_discard + n_samples) * N * (double)M);
    return cudaGetLastError();
}

size_t crbm_eloc_ws_bytes(int N, int M) { return (size_t)2 * N * M * sizeof(double2); }

cudaError_t launch_crbm_eloc(int N, int M, const double *p, const nk_ham *ham, const int8_t *s, int64_t Ns,
                             double *eloc, void *ws, cudaStream_t st) {
    if (Ns <= 0) return cudaSuccess;
    const int64_t nw = (int64_t)N * M;
    double2 *ep = static_cast<double2 *>(ws), *em = ep ? ep + nw : nullptr;
    if (ep)
        (k_crbm_exp_tables<<<nblk(nw, 256), 256, 0, st>>>(nw, reinterpret_cast<const double2 *>(p) + N + M, ep, em),
         nk::note_launch());
    const bool pairs = ham->kind != NK_TFIM;
    const int pq = M * 2 * (int)sizeof(double2), sb = (N + 15) / 16 * 16;
    const size_t lb = ((size_t)ham->n_edges * 4 + 15) / 16 * 16;
    const bool compact = pairs && (size_t)pq + sb + lb <= 100 * 1024;
    const size_t wb = (size_t)pq + sb + (compact ? lb : 0);
    int wpb = 4;
    while (wpb > 1 && wpb * wb > 227 * 1024) wpb >>= 1;
    if (wpb * wb > 227 * 1024) return cudaErrorInvalidValue;
    CElocArgs a{N, M, ham->n_edges, ham->n_edges2, ham->kind, ham->marshall, ham->J, ham->J2, ham->h,
                p, ep, em, ham->edges, s, Ns, eloc, (int)wb, pq, sb, compact ? 1 : 0};
    cudaError_t e = nk::allow_max_dynamic_smem((const void *)k_crbm_eloc);
    if (e != cudaSuccess) return e;
    const int slot = prof_begin(NK_PROF_ELOC, st);
    (k_crbm_eloc<<<nblk(Ns, wpb), 32 * wpb, wpb * wb, st>>>(a), nk::note_launch());
    prof_end(slot, st, (double)Ns * (ham->kind == NK_TFIM ? N : 0.5 * ham->n_edges) * (double)M);
    return cudaGetLastError();
}

cudaError_t launch_crbm_jacobian(int N, int M, const double *p, const int8_t *s, int64_t Ns, double *O,
                                 cudaStream_t st) {
    if (Ns <= 0) return cudaSuccess;
    const size_t smem = 4 * cwarp_bytes(N, M);
    cudaError_t e = nk::allow_max_dynamic_smem((const void *)k_crbm_jacobian);
    if (e != cudaSuccess) return e;
    (k_crbm_jacobian<<<nblk(Ns, 4), 128, smem, st>>>(N, M, p, s, Ns, O), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_crealify(int64_t rows, int64_t cols, const double *O, double *mean, double *R, cudaStream_t st) {
    (k_ccolmean<<<nblk(cols, 32), 1024, 0, st>>>(rows, cols, reinterpret_cast<const double2 *>(O),
                                                 reinterpret_cast<double2 *>(mean)), nk::note_launch());
    (k_realify<<<nblk(rows * cols, 256), 256, 0, st>>>(rows, cols, reinterpret_cast<const double2 *>(O),
                                                       reinterpret_cast<const double2 *>(mean), R), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_cstats(int64_t Ns, const double *e, double *out4, cudaStream_t st) {
    (k_cstats<<<1, 1024, 0, st>>>(Ns, reinterpret_cast<const double2 *>(e), out4), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_cforce_g(int64_t Ns, const double *e, const double *stats4, double *g, cudaStream_t st) {
    (k_cforce_g<<<nblk(Ns, 256), 256, 0, st>>>(Ns, reinterpret_cast<const double2 *>(e),
                                               reinterpret_cast<const double2 *>(stats4), g), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_tdvp_rhs(int64_t n, const double *f, int real_time, double *rhs, cudaStream_t st) {
    (k_tdvp_rhs<<<nblk(n, 256), 256, 0, st>>>(n, f, real_time, rhs), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_caxpy_realified(int64_t n, const double *base, double h, const double *x, double *out,
                                   cudaStream_t st) {
    (k_caxpy_realified<<<nblk(n, 256), 256, 0, st>>>(n, base, h, x, out), nk::note_launch());
    return cudaGetLastError();
}

}  // namespace nk
