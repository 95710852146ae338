// The symmetric RBM (RBMSymm, NetKet 3 Sec. 5): a permutation group G of
// the sites acts on the configurations, and feature f at group element g has
// the activation
//     theta_{f,g}(s) = b_f + sum_j W_{f,j} s_{pi_g(j)}
// (the embedding layer, Eq. eq: equivariant: embedding), with
//     ln psi(s) = a sum_j s_j + sum_{f,g} ln cosh theta_{f,g}(s).
// Parameters [a (1); b (alpha); W (alpha x N)], Np = 1 + alpha + alpha N.
//
// The model is a plain RBM with M = alpha |G| hidden units and tied
// parameters: unit f |G| + g has bias b_f and weight W_{f,j} on site pi_g(j),
// every visible bias equals a.  The sampler and the local energies run on
// those expanded parameters; the log-derivatives in the symmetric parameters
// follow by the chain rule (a sum over the units each parameter ties):
//     O_a = sum_j s_j,  O_{b_f} = sum_g t_{f,g},
//     O_{W_{f,j}} = sum_g t_{f,g} s_{pi_g(j)},   t = tanh theta.

#include <cuda_runtime.h>

#include "nk_common.cuh"
#include "nk_internal.h"

namespace nk {

namespace {

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// err |= 1 if a row of perms is not a permutation of [0, N).  One block per
// group element; a bitmap of the sites seen in shared memory.
__global__ void k_check_perms(int N, int G, const int32_t *__restrict__ perms, int *__restrict__ err) {
    extern __shared__ unsigned int seen[];
    const int g = blockIdx.x;
    const int words = (N + 31) / 32;
    for (int w = threadIdx.x; w < words; w += blockDim.x) seen[w] = 0u;
    __syncthreads();
    bool bad = false;
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
        const int v = perms[(size_t)g * N + j];
        if ((unsigned)v >= (unsigned)N) {
            bad = true;
            continue;
        }
        const unsigned int bit = 1u << (v & 31);
        if (atomicOr(&seen[v >> 5], bit) & bit) bad = true;  // a site hit twice
    }
    if (bad) atomicOr(err, 1);
}

// Expanded plain-RBM parameters [a_i = a (N); b_{fG+g} = b_f (M); W (M x N)]
// with W[(f G + g) N + pi_g(j)] = W_{f,j}: one thread per (f, g, j); every
// entry of a row is written once because pi_g is a permutation (checked
// before), and indices are bounds-checked all the same.
__global__ void k_symm_expand(int N, int alpha, int G, const int32_t *__restrict__ perms,
                              const double *__restrict__ p, double *__restrict__ out) {
    const int64_t M = (int64_t)alpha * G;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const double a = p[0];
    if (idx < N) out[idx] = a;
    if (idx < M) out[N + idx] = p[1 + idx / G];
    if (idx >= M * N) return;
    const int64_t unit = idx / N;
    const int j = (int)(idx % N);
    const int f = (int)(unit / G), g = (int)(unit % G);
    const int site = perms[(size_t)g * N + j];
    if ((unsigned)site < (unsigned)N) out[N + M + (size_t)unit * N + site] = p[1 + alpha + (size_t)f * N + j];
}

// One row of the symmetric Jacobian in FP64, thread (f, j) summing its G terms
// in group order: for configurations that are not +-1, more than 512 group elements
// and activations near the lower end of the FP64 range.
__device__ __noinline__ void symm_row_f64(int N, int alpha, int G, const int32_t *__restrict__ perms, const int8_t *__restrict__ sv,
                             const double *__restrict__ t, double *__restrict__ row) {
    if (threadIdx.x < 32) {
        double acc = 0.0;
        for (int j = threadIdx.x; j < N; j += 32) acc += (double)sv[j];
        acc = warp_sum(acc);
        if (threadIdx.x == 0) row[0] = acc;
    }
    for (int f = threadIdx.x; f < alpha; f += blockDim.x) {
        double acc = 0.0;
        for (int g = 0; g < G; ++g) acc += t[f * G + g];
        row[1 + f] = acc;
    }
    for (int64_t q = threadIdx.x; q < (int64_t)alpha * N; q += blockDim.x) {
        const int f = (int)(q / N), j = (int)(q % N);
        double acc = 0.0;
        for (int g = 0; g < G; ++g) {
            const int site = perms[(size_t)g * N + j];
            if ((unsigned)site < (unsigned)N) acc = fma(t[f * G + g], (double)sv[site], acc);
        }
        row[1 + alpha + q] = acc;
    }
}

// Rows of the symmetric Jacobian: O [Ns][1 + alpha + alpha N] from the samples
// and t = tanh theta of the expanded units ([Ns][alpha G]).  A block takes K
// samples.
//
// A sum over the group adds +-t only, so it runs on integers: the G values of a
// (sample, feature) are scaled by a power of two to 62 - ceil(log2 G) bits of
// their largest, and thread (f, j) adds those whose spin is up, two predicated
// integer adds a term where FP64 has 2 lanes a cycle on an SM; twice that less
// the sum of all is the result (exact modulo 2^64, and |result| <= 2^62).  Each
// term is rounded once, to at most 2^-54 of the largest, and the sum not at all,
// where FP64 rounds every partial sum.  From 513 elements on a term would keep
// fewer than 53 bits of the largest: those sums stay in FP64 (f64).  K samples
// share the loads of the permutation, coalesced over j, and one byte a site holds
// their spins; the values of a (f, g) are broadcast.
// 10 x 10 lattice, 4 features, 100 translations, 4096 samples: 1290 us as one
// block per sample with FP64 sums, 129 us now.
template <int K>
__global__ void __launch_bounds__(512) k_symm_jacobian(int N, int alpha, int G, int lg, bool f64,
                                                       const int32_t *__restrict__ perms,
                                                       const int8_t *__restrict__ s, const double *__restrict__ T,
                                                       int64_t Ns, double *__restrict__ O) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int M = alpha * G;
    const int64_t Np = 1 + alpha + (int64_t)alpha * N;
    long long *ti = reinterpret_cast<long long *>(sm);             // [M][K]
    long long *tot = ti + (size_t)M * K;                           // [alpha][K]
    double *down = reinterpret_cast<double *>(tot + (size_t)alpha * K);  // [alpha][K]
    uint8_t *up = reinterpret_cast<uint8_t *>(down + (size_t)alpha * K);  // [N]: bit q = spin of sample q is +1
    const int64_t k0 = (int64_t)blockIdx.x * K;
    const int nq = Ns - k0 < K ? (int)(Ns - k0) : K;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;

    bool odd = false;
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
        unsigned b = 0;
#pragma unroll
        for (int q = 0; q < K; ++q) {
            const int v = q < nq ? s[(size_t)(k0 + q) * N + j] : 1;
            odd |= v != 1 && v != -1;
            b |= (unsigned)(v > 0) << q;
        }
        up[j] = (uint8_t)b;
    }
    auto rows_f64 = [&] {
        for (int q = 0; q < nq; ++q)
            symm_row_f64(N, alpha, G, perms, s + (size_t)(k0 + q) * N, T + (size_t)(k0 + q) * M,
                         O + (size_t)(k0 + q) * Np);
    };
    if (__syncthreads_or(odd || f64)) {
        rows_f64();
        return;
    }
    bool tiny = false;
    for (int r = warp; r < alpha * K; r += warps) {
        const int f = r / K, q = r % K;
        if (q >= nq) {
            for (int g = lane; g < G; g += 32) ti[(size_t)(f * G + g) * K + q] = 0;
            continue;
        }
        const double *tf = T + (size_t)(k0 + q) * M + (size_t)f * G;
        unsigned e = 0;
        bool some = false;
        for (int g = lane; g < G; g += 32) {
            e = max(e, ((unsigned)__double2hiint(tf[g]) >> 20) & 0x7ffu);
            some |= tf[g] != 0.0;
        }
        e = __reduce_max_sync(0xffffffffu, e);  // |t| < 2^(e - 1022)
        tiny |= some && e < 84;                 // below 2^-938: the scale has no such exponent
        const int sh = min(62 - lg + 1022 - (int)e, 1000);
        const double scale = __hiloint2double((sh + 1023) << 20, 0);
        long long sum = 0;
        for (int g = lane; g < G; g += 32) {
            const long long v = __double2ll_rn(tf[g] * scale);
            ti[(size_t)(f * G + g) * K + q] = v;
            sum += v;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) {
            // a feature with an infinity or NaN among its values is NaN throughout
            const double d = e == 0x7ffu ? __longlong_as_double(0x7ff8000000000000LL)
                                         : __hiloint2double((1023 - sh) << 20, 0);
            tot[r] = sum;
            down[r] = d;
            O[(size_t)(k0 + q) * Np + 1 + f] = (double)sum * d;
        }
    }
    for (int q = warp; q < nq; q += warps) {
        int n = 0;
        for (int j = lane; j < N; j += 32) n += (up[j] >> q) & 1;
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0) O[(size_t)(k0 + q) * Np] = (double)(2 * n - N);
    }
    if (__syncthreads_or(tiny)) {
        rows_f64();
        return;
    }
    for (int64_t x = threadIdx.x; x < (int64_t)alpha * N; x += blockDim.x) {
        const int f = (int)(x / N), j = (int)(x % N);
        const long long *tf = ti + (size_t)f * G * K;
        long long pos[K];
#pragma unroll
        for (int q = 0; q < K; ++q) pos[q] = 0;
#pragma unroll 4
        for (int g = 0; g < G; ++g) {
            const int site = perms[(size_t)g * N + j];
            const unsigned b = (unsigned)site < (unsigned)N ? up[site] : 0u;
#pragma unroll
            for (int q = 0; q < K; ++q)
                if ((b >> q) & 1u) pos[q] += tf[(size_t)g * K + q];
        }
#pragma unroll
        for (int q = 0; q < K; ++q)
            if (q < nq)
                O[(size_t)(k0 + q) * Np + 1 + alpha + x] = (double)(2 * pos[q] - tot[f * K + q]) * down[f * K + q];
    }
}

size_t symm_staged_smem(int N, int alpha, int G, int K) {
    return (size_t)K * 8 * ((size_t)alpha * G + 2 * (size_t)alpha) + (size_t)(N + 15) / 16 * 16;
}

template <int K>
cudaError_t symm_jacobian_launch(int N, int alpha, int G, const int32_t *perms, const int8_t *s, const double *T,
                                 int64_t Ns, double *O, cudaStream_t st) {
    cudaError_t e = nk::allow_max_dynamic_smem((const void *)k_symm_jacobian<K>);
    if (e != cudaSuccess) return e;
    const size_t smem = symm_staged_smem(N, alpha, G, K);
    int lg = 0;
    while (lg < 30 && (1 << lg) < G) ++lg;
    // as many threads as (f, j) outputs, at most 512, in equal passes
    const int64_t passes = ((int64_t)alpha * N + 511) / 512;
    const int threads = (int)((((int64_t)alpha * N + passes - 1) / passes + 31) / 32 * 32);
    const int64_t Np = 1 + alpha + (int64_t)alpha * N;
    for (int64_t k0 = 0; k0 < Ns; k0 += 65535 * K) {
        const int64_t kb = Ns - k0 < 65535 * K ? Ns - k0 : 65535 * K;
        (k_symm_jacobian<K><<<(unsigned)((kb + K - 1) / K), threads, smem, st>>>(
             N, alpha, G, lg, G > 512, perms, s + (size_t)k0 * N, T + (size_t)k0 * alpha * G, kb, O + (size_t)k0 * Np),
         nk::note_launch());
    }
    return cudaGetLastError();
}

// dJ[k][q] = O[k][q] - mean[q], in place.
__global__ void k_sub_colmean(int64_t rows, int64_t cols, const double *__restrict__ mean, double *__restrict__ O) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < rows * cols) O[idx] -= mean[idx % cols];
}

}  // namespace

cudaError_t launch_symm_check_perms(int N, int G, const int32_t *perms, int *err, cudaStream_t st) {
    const size_t smem = (size_t)((N + 31) / 32) * sizeof(unsigned int);
    (k_check_perms<<<G, 256, smem, st>>>(N, G, perms, err), nk::note_launch());
    return cudaGetLastError();
}

cudaError_t launch_symm_expand(int N, int alpha, int G, const int32_t *perms, const double *p, double *out,
                               cudaStream_t st) {
    const int64_t M = (int64_t)alpha * G;
    const int64_t n = M * N > M ? M * N : M;
    (k_symm_expand<<<nblk(n > N ? n : N, 256), 256, 0, st>>>(N, alpha, G, perms, p, out), nk::note_launch());
    return cudaGetLastError();
}

size_t symm_jacobian_smem(int N, int alpha, int G) {
    return (size_t)alpha * G * sizeof(double) + (size_t)(N + 15) / 16 * 16;
}

cudaError_t launch_symm_jacobian(int N, int alpha, int G, const int32_t *perms, const int8_t *s, const double *T,
                                 int64_t Ns, double *O, cudaStream_t st) {
    if (Ns <= 0) return cudaSuccess;
    if (symm_jacobian_smem(N, alpha, G) > 227 * 1024) return cudaErrorInvalidValue;
    // Four samples a block, or two, while three blocks fit an SM and there are two
    // blocks for each SM; one sample always fits (alpha G <= 8192: 201 KB).
    const auto good = [&](int K) {
        return G <= 512 && symm_staged_smem(N, alpha, G, K) <= 75 * 1024 && Ns >= 304 * K;
    };
    if (good(4)) return symm_jacobian_launch<4>(N, alpha, G, perms, s, T, Ns, O, st);
    if (good(2)) return symm_jacobian_launch<2>(N, alpha, G, perms, s, T, Ns, O, st);
    return symm_jacobian_launch<1>(N, alpha, G, perms, s, T, Ns, O, st);
}

cudaError_t launch_sub_colmean(int64_t rows, int64_t cols, const double *mean, double *O, cudaStream_t st) {
    if (rows <= 0 || cols <= 0) return cudaSuccess;
    (k_sub_colmean<<<nblk(rows * cols, 256), 256, 0, st>>>(rows, cols, mean, O), nk::note_launch());
    return cudaGetLastError();
}

}  // namespace nk
