// Symmetric rank-K products C = scale X^T X + eps I of FP64 matrices on the
// tensor cores, for K of any length (the dense S of App. B.2: NetKet 3, Sec.
// 3.5), with the integer slices of k_tc.cu.
//
// Every column of X is scaled by one power of two (its largest entry over all
// rows, so that the scale does not depend on k), rounded to 56 bits and cut into
// 7 slices of 8-bit integers, stored with k contiguous: [7][n][ldk] BF16.  A CTA
// owns one 128 x 32 tile of the lower triangle and a range of k (a split), and
// walks it in chunks of 64: the products of slices s + t = g, g = 2 .. 9, land in
// one FP32 level g in TMEM, exact over a chunk, and are added up over the chunks
// as integers in registers (two 64-bit sums an entry), so C is touched once
// however long K is.  (The 64-row passes of k_ozaki_gemm that this replaces read and wrote C
// once a chunk and took a slicing and a product launch each: 2.68 ms for the
// 405 x 405 x 8192 matrix of the symmetric RBM; FP64 on CUDA cores took 16.8
// ms for 880 x 880 x 8192.)
//
// Accuracy: with r = max |x| / rms x of a column, the rounding and the products left
// out (s + t >= 10) err by at most 2^-56 r_i + 2^-56 r_j + 2^-59 r_i r_j of
// sqrt(S_ii S_jj).  Where the scale's square is over 256 mean squares (a spin that
// flips in a few samples of a thousand), the column's products are done over in
// FP64 (k_syrk_exact), so that S is as accurate as sums in FP64 for every column.
// (Without level 9, and truncated, a column of 1 flip in 1000 lost 10 bits.)
//
// Roles: warp 0 (one thread) streams operands by TMA, the 7 B slices of a
// chunk into one of two 28 KB buffers and the A slices one by one into a ring
// of nine 16 KB slots, so that a chunk's 140 KB need not be there before its
// MMAs start; warp 1 (one thread) issues, per A slice, 4 MMAs against B slices
// 1 .. min(7, 9-s) side by side (M = 128, N up to 224, K = 16) into one of two TMEM
// accumulator sets; warps 2 - 17 drain the other set.  What bounds it: the
// drain (8 float-to-integer conversions an entry and chunk, 16 lanes a clock
// and SM, about 1.2 us a chunk) and the 34 slice products (about as long).
// Every wait is bounded; on a time-out the kernel records a code, lets its
// copies and MMAs in flight finish, frees its TMEM and returns.

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "nk_common.cuh"
#include "nk_internal.h"
#include "tc_ptx.cuh"

namespace nk {

namespace {

constexpr int kS = 7;                          // slices
constexpr int kLevels = 8;                     // s + t = 2 .. 9 (slices from 1)
constexpr int kYM = 128, kYN = 32, kYK = 64;   // tile and chunk
constexpr int kYA = kYM * kYK * 2;             // one A slice of a chunk, bytes
constexpr int kYB = kYN * kYK * 2;             // one B slice
constexpr int kYSlots = 9;                     // A slice ring
constexpr int kYEpiWarps = 16;
constexpr int kYThreads = 64 + 32 * kYEpiWarps;
constexpr int kYCols = kYN / (kYEpiWarps / 4);  // tile columns per epilogue warp: 8
constexpr uint32_t kYAcc = 256;                // TMEM columns per accumulator set
constexpr int kBadExp = 100000;                // column exponent of an infinity or NaN
// The slices of at most this many bytes are held at a time (and of at most 2^19
// rows: the integer sums of an entry stay below 2^62).
constexpr size_t kSliceBytes = (size_t)1 << 30;
constexpr int64_t kSegRows = 1 << 19;

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

size_t syrk_smem_bytes() {
    return 1024 + (size_t)kYSlots * kYA + 2 * (size_t)kS * kYB + (2 * kYSlots + 8) * sizeof(uint64_t) + 16;
}

// ---------------------------------------------------------------- slicing ---

// Exponent of every column of X [rows][n] (|x| < 2^e; -100000 for a zero
// column, kBadExp for one that holds an infinity or a NaN), by atomicMax over
// blocks of 32 columns x 256 rows; expo starts at -100000.
__global__ void __launch_bounds__(256) k_col_exponents(const double *__restrict__ X, int64_t rows, int64_t n,
                                                       int *__restrict__ expo) {
    const int c = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int64_t p = (int64_t)blockIdx.x * 32 + c, r0 = (int64_t)blockIdx.y * 256;
    int ex = -100000;
    if (p < n) {
        const int64_t r1 = r0 + 256 < rows ? r0 + 256 : rows;
#pragma unroll 4
        for (int64_t r = r0 + y; r < r1; r += 8) {
            int b;
            unsigned long long m;
            bool neg;
            split_bits(X[(size_t)r * n + p], b, m, neg);
            if (m) ex = max(ex, b == 2047 ? kBadExp : b - 1022);
        }
    }
    __shared__ int red[8][32];
    red[y][c] = ex;
    __syncthreads();
    if (y == 0 && p < n) {
        for (int q = 1; q < 8; ++q) ex = max(ex, red[q][c]);
        if (ex != -100000) atomicMax(&expo[p], ex);
    }
}

__global__ void k_exponents_init(int64_t n, int *__restrict__ expo, unsigned long long *__restrict__ sq) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        expo[i] = -100000;
        sq[i] = 0;
    }
}

// Whether a column's entries are too uneven for its slices: 2^(2 e) above 256 mean
// squares (sq: sum of the squares of floor(2^12 |x| 2^-e)), or not finite.
__device__ __forceinline__ bool uneven(int64_t rows, int e, unsigned long long sq) {
    return e != -100000 && (e == kBadExp || (sq >> 16) < (unsigned long long)rows);
}

// X [rows][n] -> slices out [7][n][ldk] (column p of X is row p; zero from
// rows to ldk): 64 rows x 32 columns per block through shared memory, BF16
// pairs along k; the squares of the columns' leading 12 bits are added to sq.
__global__ void __launch_bounds__(256) k_slice_cols_long(const double *__restrict__ X, int64_t rows, int64_t n,
                                                         int64_t ldk, const int *__restrict__ expo,
                                                         __nv_bfloat162 *__restrict__ out,
                                                         unsigned long long *__restrict__ sq) {
    __shared__ double tile[64][33];
    const int tid = threadIdx.x;
    const int64_t p0 = (int64_t)blockIdx.x * 32, r0 = (int64_t)blockIdx.y * 64;
    for (int i = tid; i < 64 * 32; i += 256) {
        const int r = i >> 5, c = i & 31;
        tile[r][c] = (r0 + r < rows && p0 + c < n) ? X[(size_t)(r0 + r) * n + p0 + c] : 0.0;
    }
    __syncthreads();
    const int64_t plane2 = n * ldk / 2;
    const int k2 = tid & 31;  // rows 2 k2, 2 k2 + 1 of the block
    for (int c = tid >> 5; c < 32; c += 8) {
        if (p0 + c >= n) break;
        const int e = expo[p0 + c];
        unsigned long long y[2];
        bool neg[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int b;
            unsigned long long m;
            split_bits(tile[2 * k2 + h][c], b, m, neg[h]);
            const int sh = b - 1075 + 8 * kS - e;
            // (only values below 2^(e - 3) are rounded: none reaches 2^e)
            y[h] = !m || sh <= -64 || e == kBadExp
                       ? 0ULL
                       : (sh >= 0 ? (m << sh) : (m >> (-sh)) + ((m >> (-sh - 1)) & 1ULL));
        }
        const unsigned q0 = (unsigned)(y[0] >> 44), q1 = (unsigned)(y[1] >> 44);
        const unsigned qq = __reduce_add_sync(0xffffffffu, q0 * q0 + q1 * q1);
        if (k2 == 0 && qq) atomicAdd(&sq[p0 + c], (unsigned long long)qq);
        __nv_bfloat162 *o = out + ((size_t)(p0 + c) * ldk + r0) / 2 + k2;
#pragma unroll
        for (int q = 0; q < kS; ++q) {
            const int d0 = (int)((y[0] >> (8 * (kS - 1 - q))) & 0xFFULL);
            const int d1 = (int)((y[1] >> (8 * (kS - 1 - q))) & 0xFFULL);
            o[(size_t)q * plane2] =
                __halves2bfloat162(__int2bfloat16_rn(neg[0] ? -d0 : d0), __int2bfloat16_rn(neg[1] ? -d1 : d1));
        }
    }
}

// ------------------------------------------------------------ the product ---

struct SyrkArgs {
    int64_t n;
    int chunks;      // of 64 along k
    int per_split;   // chunks per split (blockIdx.y)
    const int *expo; // [n]
    double *C;       // one split: the result (row stride n); else partials [split][n][n]
    double scale, eps;
    int splits;
    int add;         // C += the product (a later segment of rows; eps is in already)
    int *err;
};

// 2^e as a product of two factors, so that every intermediate is the value of
// the product or its overflow or underflow
__device__ __forceinline__ double scale_pow2(double v, int e) {
    const int e1 = e / 2, e2 = e - e1;
    auto p2 = [](int x) { return __longlong_as_double((long long)(x < -1022 ? 1 : (x > 1023 ? 2046 : x + 1023)) << 52); };
    return v * p2(e1) * p2(e2);
}

// tile index t of the lower triangle (row tiles of 128, column tiles of 32)
__device__ __forceinline__ void tile_of(int t, int64_t n, int64_t &m0, int64_t &n0) {
    int mb = 0;
    for (;; ++mb) {
        const int64_t last = ((int64_t)mb * kYM + kYM - 1) / kYN + 1, all = (n + kYN - 1) / kYN;
        const int in_row = (int)(last < all ? last : all);
        if (t < in_row) break;
        t -= in_row;
    }
    m0 = (int64_t)mb * kYM;
    n0 = (int64_t)t * kYN;
}

__global__ void __launch_bounds__(kYThreads, 1)
    k_oz_syrk(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, SyrkArgs a) {
    extern __shared__ unsigned char smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    unsigned char *sA = smem_raw + ((1024 - (base & 1023)) & 1023);  // [9][128][64] bf16
    unsigned char *sB = sA + (size_t)kYSlots * kYA;                  // [2][7][32][64] bf16
    uint64_t *bars = reinterpret_cast<uint64_t *>(sB + 2 * (size_t)kS * kYB);
    uint64_t *a_full = bars, *a_empty = bars + kYSlots, *b_full = bars + 2 * kYSlots, *b_empty = b_full + 2;
    uint64_t *acc_full = b_empty + 2, *acc_empty = acc_full + 2;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(acc_empty + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int64_t m0, n0;
    tile_of((int)blockIdx.x, a.n, m0, n0);
    const int c0 = (int)blockIdx.y * a.per_split;
    const int count = a.chunks - c0 < a.per_split ? a.chunks - c0 : a.per_split;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kYSlots; ++s) {
            mbar_init(&a_full[s], 1);
            mbar_init(&a_empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&b_full[b], 1);
            mbar_init(&b_empty[b], 1);
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kYEpiWarps);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tslot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    auto fail = [&](int code) {
        *abort_flag = 1;
        atomicExch(a.err, code);
    };

    if (warp == 0 && lane == 0) {
        // ---------------------------------------------------------- producer
        int na = 0, nb = 0;  // A slices and B buffers filled so far
        for (int i = 0; i < count && !*abort_flag; ++i) {
            const int b = i & 1, kx = (c0 + i) * kYK;
            if (i >= 2 && !mbar_wait_or_abort_sleep(&b_empty[b], (uint32_t)((i / 2 - 1) & 1), abort_flag)) {
                fail(12);
                break;
            }
            mbar_expect_tx(&b_full[b], (uint32_t)(kS * kYB));
            for (int s = 0; s < kS; ++s)
                tma_load_3d(sB + (size_t)(b * kS + s) * kYB, &mapB, &b_full[b], kx, (int)n0, s);
            ++nb;
            bool ok = true;
            for (int s = 0; s < kS; ++s, ++na) {
                const int slot = na % kYSlots;
                if (na >= kYSlots &&
                    !mbar_wait_or_abort_sleep(&a_empty[slot], (uint32_t)((na / kYSlots - 1) & 1), abort_flag)) {
                    ok = false;
                    break;
                }
                mbar_expect_tx(&a_full[slot], (uint32_t)kYA);
                tma_load_3d(sA + (size_t)slot * kYA, &mapA, &a_full[slot], kx, (int)m0, s);
            }
            if (!ok) {
                fail(13);
                break;
            }
        }
        if (*abort_flag) {
            // the copies in flight land before the CTA exits
            for (int h = na > kYSlots ? na - kYSlots : 0; h < na; ++h)
                mbar_wait(&a_full[h % kYSlots], (uint32_t)((h / kYSlots) & 1));
            for (int h = nb > 2 ? nb - 2 : 0; h < nb; ++h) mbar_wait(&b_full[h & 1], (uint32_t)((h / 2) & 1));
        }
    } else if (warp == 1 && lane == 0) {
        // ------------------------------------------------------- MMA issuer
        int na = 0, committed = -1;
        for (int i = 0; i < count && !*abort_flag; ++i) {
            const int b = i & 1;
            const uint32_t use = (uint32_t)(i >> 1);
            if (use > 0 && !mbar_wait_or_abort(&acc_empty[b], (use - 1) & 1, abort_flag)) {
                fail(15);
                break;
            }
            if (!mbar_wait_or_abort_sleep(&b_full[b], use & 1, abort_flag)) {
                fail(14);
                break;
            }
            const uint32_t d = tmem + (uint32_t)b * kYAcc;
            const uint64_t db = sw128_desc(sB + (size_t)b * kS * kYB);
            bool ok = true;
            for (int s = 0; s < kS; ++s, ++na) {
                const int slot = na % kYSlots;
                if (!mbar_wait_or_abort_sleep(&a_full[slot], (uint32_t)((na / kYSlots) & 1), abort_flag)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint64_t da = sw128_desc(sA + (size_t)slot * kYA);
                // levels s .. 7 (from 0): B slices 0 .. 7 - s, of which there are 7; slice
                // 1 opens level 7 with its product by B slice 6
                const uint32_t ds = d + (uint32_t)(s * kYN);
                const uint32_t idesc = idesc_bf16(kYM, kYN * (s == 0 ? kS : kLevels - s));
                const uint64_t db6 = sw128_desc(sB + (size_t)(b * kS + kS - 1) * kYB);
#pragma unroll
                for (int kk = 0; kk < kYK / 16; ++kk) {
                    const uint64_t dak = da + (uint64_t)(kk * 2), dbk = db + (uint64_t)(kk * 2);
                    if (s == 1 && kk == 0) {
                        umma_bf16(ds, dak, dbk, idesc_bf16(kYM, kYN * (kS - 1)), 1u);
                        umma_bf16(d + (uint32_t)((kLevels - 1) * kYN), dak, db6, idesc_bf16(kYM, kYN), 0u);
                    } else {
                        umma_bf16(ds, dak, dbk, idesc, (kk > 0 || s > 0) ? 1u : 0u);
                    }
                }
                umma_commit(&a_empty[slot]);
            }
            umma_commit(&b_empty[b]);
            umma_commit(&acc_full[b]);
            committed = i;
            if (!ok) {
                fail(14);
                break;
            }
        }
        if (*abort_flag && committed >= 0)  // the MMAs in flight finish before the TMEM is released
            mbar_wait(&acc_full[committed & 1], (uint32_t)((committed >> 1) & 1));
    } else if (warp >= 2) {
        // --------------------------------------------------------- epilogue
        // warp: tile rows 32q .. 32q + 31 (its TMEM lane quarter), 8 columns;
        // an entry's levels D_2 .. D_9 as hi = sum D_2 2^24 + D_3 2^16 + D_4 2^8 +
        // D_5 and lo = sum D_6 2^24 + D_7 2^16 + D_8 2^8 + D_9 over the chunks (both
        // below 2^49 a chunk): the product is (hi 2^32 + lo) 2^(e_i + e_j - 72)
        const int q = warp & 3, cw = ((warp - 2) >> 2) * kYCols;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        long long hi[kYCols], lo[kYCols];
#pragma unroll
        for (int j = 0; j < kYCols; ++j) hi[j] = lo[j] = 0;
        bool done = true;
        for (int i = 0; i < count; ++i) {
            const int b = i & 1;
            int ok = 1;
            if (lane == 0) ok = mbar_wait_or_abort_sleep(&acc_full[b], (uint32_t)(i >> 1) & 1, abort_flag) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) {
                if (lane == 0) fail(16);
                done = false;
                break;
            }
            tc_fence_after();
#pragma unroll
            for (int c4 = 0; c4 < kYCols; c4 += 4) {
                uint32_t r[kLevels][4];
#pragma unroll
                for (int g = 0; g < kLevels; ++g)
                    tmem_ld4(tmem + (uint32_t)b * kYAcc + lane_base + (uint32_t)(g * kYN + cw + c4), r[g]);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    int v[kLevels];
#pragma unroll
                    for (int g = 0; g < kLevels; ++g) v[g] = __float2int_rn(__uint_as_float(r[g][j]));
                    hi[c4 + j] += (long long)v[0] * 16777216 + (long long)v[1] * 65536 + (long long)v[2] * 256 + v[3];
                    lo[c4 + j] += (long long)v[4] * 16777216 + (long long)v[5] * 65536 + (long long)v[6] * 256 + v[7];
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[b]);
        }
        const int64_t row = m0 + q * 32 + lane;
        if (done && row < a.n) {
            const int ei = a.expo[row];
            double *dst = a.C + (a.splits > 1 ? (size_t)blockIdx.y * a.n * a.n : 0) + (size_t)row * a.n;
#pragma unroll
            for (int j = 0; j < kYCols; ++j) {
                const int64_t col = n0 + cw + j;
                if (col > row) continue;  // also the columns past n
                const int ej = a.expo[col];
                double v = 0.0;
                if (ei != -100000 && ej != -100000 && ei != kBadExp && ej != kBadExp)  // (bad: k_syrk_exact)
                    v = scale_pow2(fma((double)hi[j], 4294967296.0, (double)lo[j]), ei + ej - 72);
                if (a.splits == 1) v = v * a.scale + (a.add ? dst[col] : (col == row ? a.eps : 0.0));
                dst[col] = v;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// C <- scale sum_z P[z] + eps I (add: + C) on the lower triangle, in split order.
__global__ void k_syrk_finish(int64_t n, int splits, const double *__restrict__ P, double scale, double eps, int add,
                              double *__restrict__ C) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
    if (j > i || i >= n) return;
    double v = 0.0;
    for (int z = 0; z < splits; ++z) v += P[(size_t)z * n * n + (size_t)i * n + j];
    C[(size_t)i * n + j] = v * scale + (add ? C[(size_t)i * n + j] : (i == j ? eps : 0.0));
}

// The entries of C in the rows and columns of uneven columns of X, in FP64: items
// of one such column by 64 others, 4 threads a pair over the rows, 4 chains each.
// All columns so take what the FP64 pipe takes for the whole product (16 ms for 880
// x 880 x 8192); without any, 3 us for the look at sq.
__global__ void __launch_bounds__(256) k_syrk_exact(const double *__restrict__ X, int64_t rows, int64_t n,
                                                    const int *__restrict__ expo,
                                                    const unsigned long long *__restrict__ sq, double scale, double eps,
                                                    double *__restrict__ C) {
    __shared__ int list[256], count[8];
    __shared__ double part[4][64];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, c = t & 63, y = t >> 6;
    const int64_t tiles = (n + 63) / 64;
    for (int64_t base = 0; base < n; base += 256) {
        const bool f = base + t < n && uneven(rows, expo[base + t], sq[base + t]);
        const unsigned mask = __ballot_sync(0xffffffffu, f);
        if (lane == 0) count[warp] = __popc(mask);
        if (!__syncthreads_or(f)) continue;
        int before = 0, total = 0;
        for (int w = 0; w < 8; ++w) {
            if (w < warp) before += count[w];
            total += count[w];
        }
        if (f) list[before + __popc(mask & ((1u << lane) - 1u))] = t;
        __syncthreads();
        for (int64_t it = blockIdx.x; it < total * tiles; it += gridDim.x) {
            const int64_t i = base + list[it / tiles], j = it % tiles * 64 + c;
            // a pair of uneven columns is the later one's
            const bool on = j < n && !(j > i && uneven(rows, expo[j], sq[j]));
            double q[4] = {0.0, 0.0, 0.0, 0.0};
            if (on) {
                int64_t r = y;
                for (; r + 12 < rows; r += 16)
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        q[u] = fma(X[(size_t)(r + 4 * u) * n + i], X[(size_t)(r + 4 * u) * n + j], q[u]);
                for (; r < rows; r += 4) q[0] = fma(X[(size_t)r * n + i], X[(size_t)r * n + j], q[0]);
            }
            part[y][c] = (q[0] + q[1]) + (q[2] + q[3]);
            __syncthreads();
            if (y == 0 && on) {
                const double v = ((part[0][c] + part[1][c]) + (part[2][c] + part[3][c])) * scale;
                C[(size_t)(i > j ? i : j) * n + (i > j ? j : i)] = v + (i == j ? eps : 0.0);
            }
            __syncthreads();
        }
        __syncthreads();
    }
}

int64_t lower_tiles(int64_t n) {
    int64_t t = 0;
    for (int64_t m0 = 0; m0 < n; m0 += kYM) {
        const int64_t last = (m0 + kYM - 1) / kYN + 1, all = (n + kYN - 1) / kYN;
        t += last < all ? last : all;
    }
    return t;
}

// Splits of k: enough CTAs for one full wave of the 152 SMs (one CTA an SM),
// no more than 8 partial matrices, at least one chunk each.
int syrk_splits(int64_t rows, int64_t n) {
    const int64_t chunks = (rows + kYK - 1) / kYK, tiles = lower_tiles(n);
    int64_t z = tiles > 0 ? 152 / tiles : 1;
    if (z > 8) z = 8;
    if (z > chunks) z = chunks;
    return z < 1 ? 1 : (int)z;
}

// Rows sliced at a time.
int64_t seg_rows(int64_t rows, int64_t n) {
    int64_t cap = (int64_t)(kSliceBytes / ((size_t)kS * 2 * n)) / kYK * kYK;
    if (cap > kSegRows) cap = kSegRows;
    if (cap < kYK) cap = kYK;
    const int64_t all = (rows + kYK - 1) / kYK * kYK;
    return all < cap ? all : cap;
}

size_t round256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

size_t tc_syrk_ws_bytes(int64_t rows, int64_t n) {
    const int64_t ldk = seg_rows(rows, n);
    const int z = syrk_splits(ldk, n);
    return round256((size_t)kS * n * ldk * 2) + round256((size_t)n * 4) + round256((size_t)n * 8) +
           (z > 1 ? (size_t)z * n * n * 8 : 0) + 256;
}

cudaError_t launch_syrk_tc(const double *X, int64_t rows, int64_t n, double scale, double eps, double *C, int *err,
                           void *ws, cudaStream_t st) {
    if (rows <= 0 || n <= 0) return cudaSuccess;
    const int64_t ldk = seg_rows(rows, n);
    const int64_t tiles = lower_tiles(n);
    if (tiles > (1LL << 31) - 1) return cudaErrorInvalidValue;
    char *p = static_cast<char *>(ws);
    auto *sl = reinterpret_cast<__nv_bfloat16 *>(p);
    p += round256((size_t)kS * n * ldk * 2);
    int *expo = reinterpret_cast<int *>(p);
    p += round256((size_t)n * 4);
    auto *sq = reinterpret_cast<unsigned long long *>(p);
    p += round256((size_t)n * 8);
    double *partial = reinterpret_cast<double *>(p);
    const int slot = prof_begin(NK_PROF_GRAM, st);
    (k_exponents_init<<<nblk(n, 256), 256, 0, st>>>(n, expo, sq), nk::note_launch());
    constexpr int64_t kExpRows = 65535LL * 256;
    for (int64_t r0 = 0; r0 < rows; r0 += kExpRows) {
        const int64_t nr = rows - r0 < kExpRows ? rows - r0 : kExpRows;
        (k_col_exponents<<<dim3(nblk(n, 32), nblk(nr, 256)), 256, 0, st>>>(X + (size_t)r0 * n, nr, n, expo),
         nk::note_launch());
    }
    EncodeTiledFn fn = encode_fn();
    if (!fn) return cudaErrorInvalidValue;
    CUtensorMap ma, mb;
    cuuint64_t dims[3] = {(cuuint64_t)ldk, (cuuint64_t)n, (cuuint64_t)kS};
    cuuint64_t strides[2] = {(cuuint64_t)ldk * 2, (cuuint64_t)n * ldk * 2};
    cuuint32_t estr[3] = {1, 1, 1};
    for (int o = 0; o < 2; ++o) {
        cuuint32_t box[3] = {(cuuint32_t)kYK, (cuuint32_t)(o ? kYN : kYM), 1};
        if (fn(o ? &mb : &ma, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, sl, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    cudaError_t e = nk::allow_max_dynamic_smem((const void *)k_oz_syrk);
    if (e != cudaSuccess) return e;
    for (int64_t r0 = 0; r0 < rows; r0 += ldk) {
        const int64_t nr = rows - r0 < ldk ? rows - r0 : ldk;
        const int chunks = (int)((nr + kYK - 1) / kYK), add = r0 > 0 ? 1 : 0;
        (k_slice_cols_long<<<dim3(nblk(n, 32), (unsigned)chunks), 256, 0, st>>>(
            X + (size_t)r0 * n, nr, n, ldk, expo, reinterpret_cast<__nv_bfloat162 *>(sl), sq), nk::note_launch());
        int z = syrk_splits(nr, n);
        const int per = (chunks + z - 1) / z;
        z = (chunks + per - 1) / per;
        SyrkArgs a{n, chunks, per, expo, z > 1 ? partial : C, scale, eps, z, add, err};
        (k_oz_syrk<<<dim3((unsigned)tiles, (unsigned)z), kYThreads, syrk_smem_bytes(), st>>>(ma, mb, a),
         nk::note_launch());
        if (z > 1)  // (at most 76 tiles, so n fits the grid)
            (k_syrk_finish<<<dim3(nblk(n, 256), (unsigned)n), 256, 0, st>>>(n, z, partial, scale, eps, add, C),
             nk::note_launch());
    }
    (k_syrk_exact<<<304, 256, 0, st>>>(X, rows, n, expo, sq, scale, eps, C), nk::note_launch());
    prof_end(slot, st, (double)rows * n * (double)(n + 1),
             (double)tiles * (double)((rows + kYK - 1) / kYK) * 34.0 * 2.0 * kYM * kYN * kYK);
    return cudaGetLastError();
}

}  // namespace nk
