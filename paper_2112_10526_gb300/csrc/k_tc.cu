// Tensor-core (tcgen05) products for the dense contractions of the SR solve.
//
// FP64-accurate GEMM by integer splitting (the Ozaki scheme: Ozaki, Ogita,
// Oishi, Rump, Numer. Algorithms 59 (2012); Ootomo, Ozaki, Yokota,
// IJHPCA 2024).  Every row r of an FP64 operand (K <= 64 columns) is scaled
// by its own power of two 2^-e_r (max |a_rk| < 2^e_r) and cut into S slices
// of 8-bit integers alpha_s in [-255, 255]:
//     a_rk = 2^e_r sum_{s=1..S} alpha_s,rk 2^{-8s} + (remainder < 2^{e_r - 8S}).
// Integers of at most 8 bits are exact in BF16, their products exact in the
// FP32 accumulator of kind::f16 MMAs, and a sum of up to four slice products
// over K = 64 stays below 2^24, so the partial products
//     D_g = sum_{s+t=g} sum_k alpha_s,ik beta_t,jk      (g = 2 .. S+1)
// are exact integers for g <= 5 (the levels that carry the leading bits) and
// carry a relative error 2^-24 x 2^{-8g} < 2^-70 beyond.  The epilogue
// recombines C_ij = 2^{e_i + f_j} sum_g 2^{-8g} D_g in FP64.  With S = 7 the
// dropped terms are below 2^-56 of K max|a| max|b|: FP64-level accuracy.
// S = 3 gives about FP32 accuracy (24 bits per operand).
//
// Kernel shape: a CTA per strip of up to eight 128 x 32 output tiles (K =
// 64): TMA brings the S slices of the A rows (once per strip) and of the B
// rows (3-D tensor maps [S][rows][64] BF16, 128-byte swizzle), one thread
// issues S x 4 tcgen05.mma (M = 128, K = 16, A slice s against B slices
// 1 .. S+1-s side by side: N = 32 (S+1-s)) into S accumulators of 32 TMEM
// columns, double-buffered, and sixteen warps drain the other buffer and
// update C.  Every wait is bounded by the global timer; on time-out the
// kernel records an error code, lets its copies and MMAs in flight finish,
// frees its TMEM and returns.

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "nk_common.cuh"
#include "nk_internal.h"
#include "tc_ptx.cuh"

namespace nk {

namespace {

constexpr int kTileM = 128;
constexpr int kTileK = 64;
constexpr int kMaxSlices = 7;
constexpr uint32_t kTmemCols = 512;
constexpr int kABytes = kTileM * kTileK * 2;  // one slice of the A tile

// ---------------------------------------------------------------- slicing ---

// One warp per row: the first kcols (<= 64) entries of row r of A (row
// stride lda) -> S BF16 integer slices out[s][r][0..63] (zero beyond kcols)
// and the row exponent e_r (max |a_rk| < 2^e_r).  The slices are the bytes,
// from the top, of the fixed-point magnitude floor(|a| 2^(8S - e_r)), with the
// sign of a: exactly the digits of repeated multiply-by-256-and-truncate,
// taken from the FP64 bit pattern with integer shifts only.  round (NK_F64): the
// magnitude to nearest instead (only entries below 2^(e_r - 3) have bits to lose, so
// none reaches 2^e_r).
// The warp's row r, with lane l holding columns l (x0) and l + 32 (x1), as S
// slices out[q][r][0..63] (plane stride `rows` rows) and the row exponent.
__device__ __forceinline__ void slice_row_warp(double x0, double x1, int lane, int64_t rows, int64_t r, int S,
                                               bool round, __nv_bfloat16 *__restrict__ out,
                                               int *__restrict__ expo) {
    int b0, b1;
    unsigned long long m0, m1;
    bool n0, n1;
    split_bits(x0, b0, m0, n0);
    split_bits(x1, b1, m1, n1);
    // |x| < 2^(biased - 1022) for nonzero x; the row exponent is the largest
    int ex = -100000;
    if (m0) ex = b0 - 1022;
    if (m1) ex = max(ex, b1 - 1022);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, off));
    const int e = ex == -100000 ? 0 : ex;
    // fixed point Y = floor(|x| 2^(8S - e)) = mant 2^(biased - 1075 + 8S - e) < 2^(8S)
    auto fixp = [&](int biased, unsigned long long mant) -> unsigned long long {
        if (!mant) return 0ULL;
        const int sh = biased - 1075 + 8 * S - e;
        if (sh >= 0) return mant << sh;  // sh <= 3 here
        if (sh <= -64) return 0ULL;
        return (mant >> (-sh)) + (round ? (mant >> (-sh - 1)) & 1ULL : 0ULL);
    };
    const unsigned long long y0 = fixp(b0, m0), y1 = fixp(b1, m1);
    for (int q = 0; q < S; ++q) {
        const int sh = 8 * (S - 1 - q);
        const int d0 = (int)((y0 >> sh) & 0xFFULL), d1 = (int)((y1 >> sh) & 0xFFULL);
        __nv_bfloat16 *o = out + ((size_t)q * rows + r) * kTileK;
        o[lane] = __int2bfloat16_rn(n0 ? -d0 : d0);
        o[lane + 32] = __int2bfloat16_rn(n1 ? -d1 : d1);
    }
    if (lane == 0) expo[r] = e;
}

__global__ void k_slice_rows(const double *__restrict__ A, int64_t lda, int64_t rows, int kcols, int S, bool round,
                             __nv_bfloat16 *__restrict__ out, int *__restrict__ expo) {
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= rows) return;
    const double x0 = lane < kcols ? A[(size_t)r * lda + lane] : 0.0;
    const double x1 = lane + 32 < kcols ? A[(size_t)r * lda + lane + 32] : 0.0;
    slice_row_warp(x0, x1, lane, rows, r, S, round, out, expo);
}

// ------------------------------------------------------------- the GEMM ---
//
// Warp-specialised kernel over output strips: a CTA owns up to `chunk` (<= 8)
// consecutive 128 x 32 tiles of one tile row (a 128 x 256 strip at most), keeps the
// S slices of its 128 A rows resident, and pipelines the tiles:
//   warp 0 (one thread): TMA producer, A slices once, B slices per tile into
//     one of two buffers;
//   warp 1 (one thread): MMA issuer, S MMAs (one per A slice, against the
//     B slices side by side) x 4 K-steps per tile into one of two TMEM
//     accumulator sets (S x 32 columns each), so
//     that the MMAs of tile i+1 run while tile i is drained;
//   warps 2-17: epilogue; warp w owns tile rows 32 (w % 4) .. +31 (its TMEM
//     lane quarter) and 8 columns, loads its C entries a tile ahead, and
//     turns the S accumulators into FP64 by exact integer recombination
//     before writing C back.
// A tile's epilogue takes the longest (6000 cycles on 16 warps, against 1800 of
// MMAs and 2000 of FP64 additions, two lanes a cycle): whole tiles test no entry,
// C moves 16 bytes a lane where its rows allow it, and L2 is asked for a row's
// segment once, which took 170 instructions an entry to 98 and the trailing
// update of a 8064 x 8064 matrix from 228 to 194 us.
// Strips (lower triangle only when `lower`) are numbered row by row.  CTAs
// are short-lived on purpose: kernels of a higher-priority stream (the
// Cholesky look-ahead) get SMs as strips retire.  mbarriers hand buffers
// between the roles; every wait is bounded by the global timer and gives up
// when another role of the CTA has aborted.
// kWide (NK_F64, on rounded slices): the products of slices s + t = 9 as well, and the
// window of the levels to nearest: 2^-56 of the rows' largest entries an operand and
// 2^-57 a product, where the 28 slice products leave out up to 2^-51.

struct OzArgs {
    int64_t rows, cols;   // output rows (A rows) and columns (B rows)
    int S;
    const int *expA, *expB;
    double *C;
    int64_t ldc;
    int mode;             // 0: C = R, 1: C -= R, 2: C += R
    int lower;            // only entries with col <= row (tiles above are skipped)
    int *err;
    int64_t n_nb;         // tile columns
    int chunk;            // tiles per strip: 1, 2, 4 or 8
    int chunk_log2;
    int vec;              // pairs of C's entries are 16-byte aligned
};

constexpr int kPN = 32;                      // tile columns
constexpr int kMaxChunk = 8;                 // tiles per strip at most
constexpr int kPEpiWarps = 16;
constexpr int kPThreads = 64 + 32 * kPEpiWarps;        // producer, MMA issuer, epilogue warps
constexpr int kPColsPerWarp = kPN / (kPEpiWarps / 4);  // 8
constexpr int kPBBytes = kPN * kTileK * 2;   // one slice of the B tile (4 KB)
constexpr uint32_t kPAccCols = 256;          // TMEM columns per accumulator set

__host__ __device__ inline int64_t oz_row_tiles(int64_t n_nb, bool lower, int64_t mb) {
    if (!lower) return n_nb;
    const int64_t last = (mb * kTileM + kTileM - 1) / kPN + 1;
    return last < n_nb ? last : n_nb;
}

// strips of tile row mb (a power-of-two chunk: every CTA walks the rows before
// its own, so the step is a shift, not a 64-bit division)
__host__ __device__ inline int64_t oz_row_strips(int64_t n_nb, bool lower, int64_t mb, int chunk_log2) {
    return (oz_row_tiles(n_nb, lower, mb) + ((int64_t)1 << chunk_log2) - 1) >> chunk_log2;
}

// The MMAs of one tile: level g = s + t (2 .. S+1) collects the products of
// A slice s and B slice t in TMEM columns dbase + (g - 2) 32.  The B slices
// of a tile lie back to back in shared memory ([S][32][64], 128-byte rows),
// so B slices 1 .. S+1-s read as one operand of 32 (S+1-s) rows, and a single
// MMA of that width adds A slice s times all of them to the contiguous levels
// s+1 .. S+1.  S MMAs per K-step (instead of S(S+1)/2 of width 32) read each
// A slice once; the first one of a tile (s = 1, K-step 0) initialises every
// level.  SS > 0 fixes S at compile time.  kWide adds level S + 2, which A slices 2 ..
// S reach with one B slice more; slice 2 initialises it by itself (B slice S).
template <int SS, bool kWide>
__device__ __forceinline__ void issue_tile(uint32_t dbase, uint64_t da, uint64_t db,
                                           const uint32_t (&idesc)[kMaxSlices], int S_rt) {
    const int S = SS > 0 ? SS : S_rt;
    constexpr int kS = (SS > 0 ? SS : kMaxSlices);
#pragma unroll 1
    for (int kk = 0; kk < kTileK / 16; ++kk) {
#pragma unroll
        for (int sa = 1; sa <= kS; ++sa) {
            if (sa > S) continue;
            const uint32_t acc = (kk > 0 || sa > 1) ? 1u : 0u;
            // A slice sa starts (sa - 1) kABytes after slice 1 (descriptor address field in 16-byte units)
            const uint64_t das = da + (uint64_t)((sa - 1) * (kABytes >> 4) + kk * 2), dbk = db + (uint64_t)(kk * 2);
            if (kWide && sa == 2 && kk == 0) {
                umma_bf16(dbase + (uint32_t)kPN, das, dbk, idesc_bf16(kTileM, kPN * (kS - 1)), 1u);
                umma_bf16(dbase + (uint32_t)(kS * kPN), das, dbk + (uint64_t)((kS - 1) * (kPBBytes >> 4)),
                          idesc_bf16(kTileM, kPN), 0u);
                continue;
            }
            umma_bf16(dbase + (uint32_t)((sa - 1) * kPN), das, dbk, idesc[sa - 1], acc);
        }
    }
}

template <int SS, bool kWide>
__global__ void __launch_bounds__(kPThreads, 1)
    k_ozaki_gemm(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, OzArgs a) {
    extern __shared__ unsigned char smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    unsigned char *ops = smem_raw + ((1024 - (base & 1023)) & 1023);
    unsigned char *sA = ops;                                            // [S][128][64] bf16
    unsigned char *sB = ops + (size_t)kMaxSlices * kABytes;             // [2][S][32][64] bf16
    unsigned char *sE = sB + (size_t)2 * kMaxSlices * kPBBytes;         // [16 warps][32][8] fp64
    uint64_t *bars = reinterpret_cast<uint64_t *>(sE + (size_t)kPEpiWarps * 32 * kPColsPerWarp * 8);
    uint64_t *a_full = bars, *b_full = bars + 2, *b_empty = bars + 4;
    uint64_t *acc_full = bars + 6, *acc_empty = bars + 8;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + 10);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    static_assert(!kWide || SS == kMaxSlices, "level 9 of 7 slices");
    constexpr int kLevels = kMaxSlices + (kWide ? 1 : 0);
    const int S = SS > 0 ? SS : a.S;
    // strip -> tile row mb, first tile column nb0, tile count: every warp scans
    // the strips per tile row, 32 rows per round (inclusive prefix by
    // shuffles), and takes the first row whose prefix passes blockIdx.x
    int64_t mb = 0, rem = blockIdx.x;
    {
        const int64_t n_mb = (a.rows + kTileM - 1) / kTileM;
        for (int64_t base = 0; base < n_mb; base += 32) {
            const int64_t m = base + lane;
            const int64_t ns = m < n_mb ? oz_row_strips(a.n_nb, a.lower != 0, m, a.chunk_log2) : 0;
            int64_t incl = ns;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int64_t v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            const int64_t total = __shfl_sync(0xffffffffu, incl, 31);
            if (rem < total) {  // warp-uniform
                const int l = __ffs(__ballot_sync(0xffffffffu, rem < incl)) - 1;
                mb = base + l;
                rem -= __shfl_sync(0xffffffffu, incl - ns, l);
                break;
            }
            rem -= total;
            mb = base + 32;
        }
    }
    const int64_t nb0 = rem << a.chunk_log2, in_row = oz_row_tiles(a.n_nb, a.lower != 0, mb);
    const int count = (int)(in_row - nb0 < a.chunk ? in_row - nb0 : a.chunk);
    const int64_t m0 = mb * kTileM;

    if (threadIdx.x == 0) {
        mbar_init(a_full, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&b_full[b], 1);
            mbar_init(&b_empty[b], 1);
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kPEpiWarps);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(tslot, kTmemCols);
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
        uint32_t fills0 = 0, fills1 = 0;  // loads issued into B buffer 0 / 1
        mbar_expect_tx(a_full, (uint32_t)S * kABytes);
        for (int s = 0; s < S; ++s) tma_load_3d(sA + (size_t)s * kABytes, &mapA, a_full, 0, (int)m0, s);
        for (int i = 0; i < count && !*abort_flag; ++i) {
            const int b = i & 1;
            const uint32_t fills = b ? fills1 : fills0;
            if (fills > 0 && !mbar_wait_or_abort(&b_empty[b], (fills - 1) & 1, abort_flag)) {
                fail(12);
                break;
            }
            mbar_expect_tx(&b_full[b], (uint32_t)S * kPBBytes);
            for (int s = 0; s < S; ++s)
                tma_load_3d(sB + (size_t)(b * kMaxSlices + s) * kPBBytes, &mapB, &b_full[b], 0,
                            (int)((nb0 + i) * kPN), s);
            if (b)
                ++fills1;
            else
                ++fills0;
        }
        if (*abort_flag) {
            // let the copies in flight land before the CTA exits
            mbar_wait(a_full, 0);
            if (fills0 > 0) mbar_wait(&b_full[0], (fills0 - 1) & 1);
            if (fills1 > 0) mbar_wait(&b_full[1], (fills1 - 1) & 1);
        }
    } else if (warp == 1 && lane == 0) {
        // ------------------------------------------------------- MMA issuer
        int issued = 0;
        uint32_t idesc[kMaxSlices];  // A slice s + 1 meets B slices 1 .. S - s: N = 32 (S - s); kWide: one more
#pragma unroll
        for (int s = 0; s < kMaxSlices; ++s)
            idesc[s] = idesc_bf16(kTileM, kPN * (kWide && s > 0 ? S + 1 - s : (S - s > 0 ? S - s : 1)));
        const uint64_t da = sw128_desc(sA), db0 = sw128_desc(sB),
                       db1 = sw128_desc(sB + (size_t)kMaxSlices * kPBBytes);
        if (!mbar_wait_or_abort(a_full, 0, abort_flag)) fail(13);
        for (int i = 0; i < count && !*abort_flag; ++i) {
            const int b = i & 1;
            const uint32_t use = (uint32_t)(i >> 1);
            if (!mbar_wait_or_abort(&b_full[b], use & 1, abort_flag)) {
                fail(14);
                break;
            }
            if (use > 0 && !mbar_wait_or_abort(&acc_empty[b], (use - 1) & 1, abort_flag)) {
                fail(15);
                break;
            }
            tc_fence_after();
            if (b)
                issue_tile<SS, kWide>(tmem + kPAccCols, da, db1, idesc, S);
            else
                issue_tile<SS, kWide>(tmem, da, db0, idesc, S);
            umma_commit(&acc_full[b]);
            umma_commit(&b_empty[b]);
            ++issued;
        }
        if (*abort_flag && issued > 0) {
            // the MMAs in flight must finish before the TMEM is released
            const int last = issued - 1;
            mbar_wait(&acc_full[last & 1], (uint32_t)(last >> 1) & 1);
        }
    } else if (warp >= 2) {
        // --------------------------------------------------------- epilogue
        // Lane l turns TMEM lane 32q + l (tile row 32q + l) into FP64 for the
        // warp's 8 columns and parks the values in its shared block
        // [32 rows][8 columns], 16 bytes at a time (pair index XOR (row / 2) mod
        // 4: conflict-free for both access patterns); C is then read and written
        // with lane l on row 8k + l / 4, columns 2 (l mod 4) and the next (k = 0
        // .. 3), 64-byte row segments.
        const int q = warp & 3;                 // TMEM lane quarter = tile rows 32q .. 32q + 31
        const int c0 = ((warp - 2) >> 2) * kPColsPerWarp;  // the warp's 8 tile columns
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        double2 *stage = reinterpret_cast<double2 *>(sE) + (warp - 2) * 32 * (kPColsPerWarp / 2);
        const int64_t row = m0 + q * 32 + lane;
        const int ei = row < a.rows ? a.expA[row] : 0;
        const int rr = lane >> 2, cc = 2 * (lane & 3);
        const int64_t row_c = m0 + q * 32 + rr;  // + 8k: the rows this lane reads and writes in C
        const int64_t step = 8 * a.ldc;
        auto on = [&](int64_t r, int64_t col) { return r < a.rows && col < a.cols && !(a.lower && col > r); };
        // tiles that lie in C (and below its diagonal) whole need no test of their entries
        auto whole = [&](int i) {
            const int64_t end = (nb0 + i + 1) * kPN;
            return m0 + kTileM <= a.rows && end <= a.cols && !(a.lower && end > m0 + 1);
        };
        auto load_c = [&](int i, double2 (&cv)[4]) {
            const int64_t col = (nb0 + i) * kPN + c0 + cc;
            const double *p = a.C + (size_t)row_c * a.ldc + col;
            if (a.mode == 0) {
#pragma unroll
                for (int k = 0; k < 4; ++k) cv[k] = make_double2(0.0, 0.0);
            } else if (whole(i)) {
                if (a.vec) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) cv[k] = *reinterpret_cast<const double2 *>(p + k * step);
                } else {
#pragma unroll
                    for (int k = 0; k < 4; ++k) cv[k] = make_double2(p[k * step], p[k * step + 1]);
                }
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int64_t r = row_c + 8 * k;
                    cv[k] = make_double2(on(r, col) ? p[k * step] : 0.0, on(r, col + 1) ? p[k * step + 1] : 0.0);
                }
            }
        };
        // column exponents (lane & 7 holds column c0 + (lane & 7)), broadcast by shuffles
        auto load_f = [&](int i) {
            const int64_t col = (nb0 + i) * kPN + c0 + (lane & 7);
            return col < a.cols ? a.expB[col] : 0;
        };
        const int flip = a.mode == 1 ? (int)0x80000000 : 0;  // of the sign in the upper half
        if (a.mode != 0) {
            // the strip's C entries (at most 128 x 256 FP64 per CTA) into L2 up
            // front, so that the per-tile loads below wait on L2, not on HBM:
            // a lane per row of the warp's 8 columns
            for (int i = 0; i < count; ++i) {
                const int64_t col = (nb0 + i) * kPN + c0;
                if (on(row, col)) prefetch_l2(a.C + (size_t)row * a.ldc + col);
            }
        }
        for (int i = 0; i < count; ++i) {
            const int b = i & 1;
            const uint32_t use = (uint32_t)(i >> 1);
            // this tile's C entries and column exponents are in flight while
            // the accumulators fill and drain; C is needed only at the end
            double2 cv[4];
            load_c(i, cv);
            const int fj_lane = load_f(i);
            int ok = 1;
            if (lane == 0) ok = mbar_wait_or_abort(&acc_full[b], use & 1, abort_flag) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) {
                if (lane == 0) fail(16);
                break;
            }
            tc_fence_after();
#pragma unroll 1
            for (int c4 = 0; c4 < kPColsPerWarp; c4 += 2) {
                uint32_t r[kLevels][2];
#pragma unroll
                for (int gi = 0; gi < kLevels; ++gi)
                    if (kWide || gi < S)
                        tmem_ld2(tmem + (uint32_t)b * kPAccCols + lane_base + (uint32_t)(gi * kPN + c0 + c4), r[gi]);
                tmem_wait_ld();
                double v[2];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    int d[kMaxSlices];
#pragma unroll
                    for (int gi = 0; gi < kMaxSlices; ++gi)
                        d[gi] = gi < S ? __float2int_rn(__uint_as_float(r[gi][j])) : 0;
                    if constexpr (kWide)  // D_9 2^-8, and the window's last bit to nearest
                        d[kMaxSlices - 1] += ((__float2int_rn(__uint_as_float(r[kMaxSlices][j])) + 128) >> 8) + 128;
                    // V 2^sc with V = sum_g D_g 2^(8 (8 - g)); C - R as C + (-R)
                    const int sc = ei + __shfl_sync(0xffffffffu, fj_lane, c4 + j) - 56;
                    const double x = window_to_double_seldom(ozaki_window8(d), sc);
                    v[j] = __hiloint2double(__double2hiint(x) ^ flip, __double2loint(x));
                }
                stage[lane * 4 + ((c4 >> 1) ^ ((lane >> 1) & 3))] = make_double2(v[0], v[1]);
            }
            // the accumulators are drained: hand the buffer back before the C traffic
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[b]);
            const int64_t col = (nb0 + i) * kPN + c0 + cc;
            double *p = a.C + (size_t)row_c * a.ldc + col;
            const bool all = whole(i);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int rl = 8 * k + rr;
                const double2 v = stage[rl * 4 + ((lane & 3) ^ ((rl >> 1) & 3))];
                const double x = cv[k].x + v.x, y = cv[k].y + v.y;  // C reads as 0 in mode 0
                if (all && a.vec) {
                    *reinterpret_cast<double2 *>(p + k * step) = make_double2(x, y);
                } else {
                    const int64_t r = row_c + 8 * k;
                    if (on(r, col)) p[k * step] = x;
                    if (on(r, col + 1)) p[k * step + 1] = y;
                }
            }
            __syncwarp();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// ------------------------------------------------- Cholesky building blocks ---

constexpr int kNB = 64;

// Factor the kb x kb diagonal block at (k, k) in place (lower), in 64-bit fixed
// point, as L D L^T with the square roots taken at the end.  An SM does two FP64
// lanes a cycle, a warp's FP64 instruction is some 64 cycles in flight, and a
// block is 64 dependent pivots and kb^3/6 multiply-adds: integers are several
// times faster at both.
// With row and column i scaled by 2^-k_i so that a_ii is in [1/4, 1), every entry
// of a positive definite block and of what is left of it after each column lies
// in (-1, 1): entries are 2^60 a.  Column c (u = L D) is normalised by the even
// power of two that takes its pivot to M = d 2^(2 f) in [1/4, 1): |u 2^f| <=
// sqrt(M) < 1 is held to 2^-62, y = 1 / M (held below 4) and (u 2^f) y to 2^-60,
// and a product of the last two enters the block to 2^-59: sqrt(a_ii a_jj) 2^-59
// an operation, where FP64's backward error is 2^-53 of it.
// One CTA holds the block in shared memory (continued by the identity beyond
// kb).  Phase p does at the same time
//   * warp 0: d_{p+1} by columns p - 1 and p and its reciprocal, the chain that
//     all else follows;
//   * warps 1 and 2 (a row a lane): column p normalised and divided, column p +
//     1 by columns p - 1 and p;
//   * twenty warps (one of them on the chain's scheduler): column p - 1 applied
//     to the columns right of p + 1.  A thread keeps its three entries of the
//     lower triangle in registers, in order of their columns from the last, so
//     that whole warps finish as the columns do; a column goes back to shared
//     memory when it is the next in work.
// and ends with its one barrier.  A block that leaves these bounds (not positive
// definite, or a pivot below 2^-52 of its diagonal entry, which FP64 could not
// tell from zero either) is done over in FP64, column by column.
// 30 us a block of 64, 46 as a Cholesky in FP64.  What is left: loading and storing
// it 5 us; 63 phases of 700 cycles while few columns are left, which is the chain
// (a third of it the reciprocal), and 1000 at first, the multiplications of the
// bulk: a 32 x 32 -> 64-bit product holds a scheduler's pipe for some ten cycles,
// half of what the FP64 multiply-add it replaces takes.
constexpr int kPotrfThreads = 896;
constexpr int kLd = kNB + 1;
constexpr int kTriEntries = kNB * (kNB - 1) / 2 + 0;  // (r, q) with 1 <= q <= r <= 63: 2016

// 2^60 a 2^-sh to nearest; |.| >= 2^60, infinities and NaN come back as 2^62.
__device__ __forceinline__ long long to_fixed60(double a, int sh) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(a);
    const int b = (int)(bits >> 52) & 0x7ff;
    const unsigned long long m = (bits & 0xfffffffffffffULL) | (b ? 1ULL << 52 : 0ULL);
    const int s = (b ? b : 1) - 1075 + 60 - sh;  // 2^60 a 2^-sh = m 2^s
    if (b == 2047 || s > 7) return m ? 1LL << 62 : 0;
    const unsigned long long v = s >= 0 ? m << s : s < -54 ? 0ULL : ((m >> (-s - 1)) + 1) >> 1;
    return (bits >> 63) ? -(long long)v : (long long)v;
}

__host__ __device__ __forceinline__ float rcp_approx(float x) {  // to 2^-23
#ifdef __CUDA_ARCH__
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
#else
    return 1.0f / x;
#endif
}

// A number of 63 bits as hi 2^31 + lo, 0 <= lo < 2^31, and x y 2^-62 without the
// product of the low halves (from 0 to 2 below): three 32 x 32-bit products, 32
// cycles a warp.  (__mul64hi takes as long, but wants the operands' signs mended
// each time, where halves are split once: 35 us a block with it.)
__host__ __device__ __forceinline__ int2 halves(long long x) { return make_int2((int)(x >> 31), (int)x & 0x7fffffff); }

__host__ __device__ __forceinline__ long long mul62(int2 x, int2 y) {
    return (long long)x.x * y.x + (((long long)x.x * y.y + (long long)x.y * y.x) >> 31);
}

// y = 2^60 / x for x = X 2^-60 in [1/4, 1): the FP32 reciprocal y0 and one
// third-order step, y0 + y0 (e + e^2) with e = 1 - x y0 (|e| < 2^-21, so the
// rest is below 2^-63).  At x = 1/4, the pivots 4^k, y would be 2^62, one more
// than `halves` holds: it is kept at 2^62 - 1, 2^-62 of itself below.
__host__ __device__ __forceinline__ unsigned long long fixed_reciprocal(unsigned long long X) {
    const uint32_t xh = (uint32_t)(X >> 28), xl = (uint32_t)X & 0xfffffffu;
    const float yf = rcp_approx((float)xh) * 2305843009213693952.0f;  // 2^29 / x: 2^61 / xh
#ifdef __CUDA_ARCH__
    const uint32_t y0 = __float2uint_rn(yf);
#else
    const uint32_t y0 = (uint32_t)yf;  // at least 2^29: a whole number
#endif
    const long long e = (1LL << 61) - (long long)((unsigned long long)xh * y0 + (((unsigned long long)xl * y0) >> 28));
    const int e40 = (int)(e >> 21);                             // 2^40 e
    const long long h = e + ((long long)e40 * e40 >> 19);       // 2^61 (e + e^2)
    const int hh = (int)(h >> 16);
    const long long yh =  // 2^74 y0 (e + e^2)
        (long long)hh * (long long)y0 + (long long)(((unsigned long long)((uint32_t)h & 0xffffu) * y0) >> 16);
    const unsigned long long y = ((unsigned long long)y0 << 31) + (unsigned long long)(yh >> 14);
    return y < 0x3fffffffffffffffULL ? y : 0x3fffffffffffffffULL;
}

__host__ __device__ constexpr int tri_from(int x) {  // packed entries with column q >= x (1 <= x <= 64)
    return (64 - x) * (65 - x) / 2;
}

__device__ __forceinline__ bool positive_finite(double x) {  // integer compares, off the FP64 pipe
    const long long bits = __double_as_longlong(x);
    return bits > 0 && bits < 0x7FF0000000000000LL;
}

// The block in FP64 (shared memory L, lower triangle), column by column.
__device__ __noinline__ void potrf64_f64(double *L, int64_t k, int kb, int *info) {
    for (int c = 0; c < kNB; ++c) {
        double d = L[c * kLd + c];
        if (!positive_finite(d)) {
            if (threadIdx.x == 0 && info && c < kb) atomicCAS(info, 0, (int)(k + c + 1));  // the first failure
            d = 1e-300;
        }
        const double rs = rsqrt(d);
        __syncthreads();
        for (int r = c + threadIdx.x; r < kNB; r += blockDim.x) L[r * kLd + c] = (r == c ? d : L[r * kLd + c]) * rs;
        __syncthreads();
        for (int e = threadIdx.x; e < kNB * kNB; e += blockDim.x) {
            const int r = e >> 6, q = e & 63;
            if (q > c && r >= q) L[r * kLd + q] = fma(-L[r * kLd + c], L[q * kLd + c], L[r * kLd + q]);
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kPotrfThreads) k_potrf64(double *__restrict__ A, int64_t n, int64_t k, int kb,
                                                           int *__restrict__ info) {
    __shared__ long long L[kNB * kLd];  // 2^60 u below the diagonal, 2^60 a right of the columns in work
    __shared__ int2 un[2][kNB];         // u 2^f of the last two columns (2^62 of it)
    __shared__ int2 ln[2][kNB];         // and that divided by M (2^60)
    __shared__ int2 ybuf[2];
    __shared__ long long dd[kNB];
    __shared__ double rs[kNB];
    __shared__ int fbuf[2], ke[kNB];
    __shared__ uint16_t tab[kTriEntries];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    constexpr int kEach = (kNB * kNB + kPotrfThreads - 1) / kPotrfThreads;
    double a[kEach];
#pragma unroll
    for (int i = 0; i < kEach; ++i) {
        const int e = t + i * kPotrfThreads, r = e >> 6, c = e & 63;
        a[i] = e < kNB * kNB && r < kb && c <= r ? A[(size_t)(k + r) * n + k + c] : r == c ? 0.5 : 0.0;
    }
#pragma unroll
    for (int i = 0; i < kEach; ++i) {
        const int e = t + i * kPotrfThreads, r = e >> 6, c = e & 63;
        if (e >= kNB * kNB) break;
        if (r == c) {
            int x = (__double2hiint(a[i]) >> 20) - 1022;  // a < 2^x
            if (x < -800 || x > 800) x = 0;               // (also what is not positive: such a block ends in FP64)
            ke[r] = r < kb ? (x + 1) >> 1 : 0;            // 2 k_i is x or x + 1
        }
        // column q (1 .. 63) owns entries [(63 - q)(64 - q)/2, +64 - q): rows q .. 63
        if (c >= 1 && r >= c) tab[(63 - c) * (64 - c) / 2 + r - c] = (uint16_t)((r << 8) | c);
    }
    __syncthreads();
    bool out = false;
#pragma unroll
    for (int i = 0; i < kEach; ++i) {
        const int e = t + i * kPotrfThreads, r = e >> 6, c = e & 63;
        if (e >= kNB * kNB) break;
        const long long v = to_fixed60(a[i], ke[r] + ke[c]);
        out |= v >= 1LL << 60 || v <= -(1LL << 60) || (r == c && v < 1LL << 58);
        L[r * kLd + c] = v;
    }
    // warp 0: the pivot of column c, its reciprocal and its power of two
    int2 y = make_int2(0, 0);
    int f = 0;
    auto pivot = [&](int c, long long d) {
        if (d < 256) {
            out = true;
            d = 1LL << 59;
        }
        f = (__clzll(d) - 4) >> 1;  // d 2^(2 f) in [2^58, 2^60)
        y = halves((long long)fixed_reciprocal((unsigned long long)d << (2 * f)));
        if (lane == 0) {
            ybuf[c & 1] = y;
            fbuf[c & 1] = f;
            dd[c] = d;
        }
    };
    // bulk warps: 3, and 5 up without the chain's scheduler (8, 12, ...); 4 last
    constexpr int kBulk = 20 * 32, kOwn = 3;
    static_assert(kBulk * kOwn >= tri_from(3), "a thread has three entries");
    const bool bulk = warp >= 3 && ((warp & 3) || warp == 4);
    const int rank = warp == 4 ? 19 : warp - 3 - (warp >> 2);  // 3, 5, 6, 7, 9 ..: 0 ..
    __syncthreads();
    long long own[kOwn] = {};
    int at[kOwn] = {};
    long long u0 = 0;  // columns: the row's entry of column p
    int2 un0 = make_int2(0, 0);  // and its normalised one of column p - 1
    if (warp == 0) {
        pivot(0, L[0]);
    } else if (warp <= 2) {
        u0 = L[(t - 32) * kLd];
    } else if (bulk) {
#pragma unroll
        for (int i = 0; i < kOwn; ++i) {
            const int e = i * kBulk + rank * 32 + lane;
            at[i] = e < tri_from(3) ? tab[e] : 0;  // (0: column 0, never written back)
            own[i] = L[(at[i] >> 8) * kLd + (at[i] & 255)];
        }
    }
    __syncthreads();
    for (int p = 0; p + 1 < kNB; ++p) {
        const int2 *uprev = un[(p + 1) & 1], *lprev = ln[(p + 1) & 1];
        const int c1 = p + 1;
        if (warp == 0) {
            const int2 u = halves(L[c1 * kLd + p] << (f + 2));
            long long a = L[c1 * kLd + c1];
            if (p > 0) a -= mul62(uprev[c1], lprev[c1]);
            const long long u2 = (long long)u.x * u.x + (((long long)u.x * u.y) >> 30);
            pivot(c1, a - mul62(halves(u2), y));
        } else if (warp <= 2) {
            if (32 * warp > c1) {  // rows of this warp are left
                const int r = t - 32, fp = fbuf[p & 1] + 2;
                const int2 yp = ybuf[p & 1];
                const int2 lq = halves(mul62(halves(L[c1 * kLd + p] << fp), yp));
                const long long ul = (long long)((unsigned long long)u0 << fp);
                const int2 u = halves(ul);
                long long v = L[r * kLd + c1];
                if (p > 0) v -= mul62(un0, lprev[c1]);
                out |= r > p && ((ul >> fp) != u0 || ul >= 1LL << 62 || ul <= -(1LL << 62));
                un[p & 1][r] = u;
                ln[p & 1][r] = halves(mul62(u, yp));
                un0 = u;
                u0 = v - mul62(u, lq);
                // (the pivot's row is warp 0's: it reads the entry meanwhile)
                if (r > c1) L[r * kLd + c1] = u0;
            }
        } else if (bulk && p > 0) {
            const int ne = tri_from(p + 2);
#pragma unroll
            for (int i = 0; i < kOwn; ++i) {
                if (i * kBulk + rank * 32 >= ne) break;  // warp-uniform
                own[i] -= mul62(uprev[at[i] >> 8], lprev[at[i] & 255]);
                if ((at[i] & 255) == p + 2) L[(at[i] >> 8) * kLd + p + 2] = own[i];
            }
        }
        __syncthreads();
    }
    if (t < kNB) rs[t] = rsqrt((double)dd[t]);
    if (__syncthreads_or(out)) {
        double *Lf = reinterpret_cast<double *>(L);
        for (int e = t; e < kNB * kNB; e += kPotrfThreads) {
            const int r = e >> 6, c = e & 63;
            Lf[r * kLd + c] = (r < kb && c <= r) ? A[(size_t)(k + r) * n + k + c] : (r == c ? 1.0 : 0.0);
        }
        __syncthreads();
        potrf64_f64(Lf, k, kb, info);
        for (int e = t; e < kNB * kNB; e += kPotrfThreads) {
            const int r = e >> 6, c = e & 63;
            if (r < kb && c <= r) A[(size_t)(k + r) * n + k + c] = Lf[r * kLd + c];
        }
        return;
    }
    // l = u / sqrt(d): 2^60 u 2^-60 2^(k_r + k_c) / sqrt(2^60 d 2^-60 2^(2 k_c))
    for (int e = t; e < kNB * kNB; e += kPotrfThreads) {
        const int r = e >> 6, c = e & 63;
        if (r < kb && c <= r) {
            const double l = (double)(r == c ? dd[c] : L[r * kLd + c]) * rs[c];
            // (times 2^(k_r - 30) on the exponent: |l| is 0 or above 2^-31)
            A[(size_t)(k + r) * n + k + c] =
                l == 0.0 ? 0.0 : __hiloint2double(__double2hiint(l) + ((ke[r] - 30) << 20), __double2loint(l));
        }
    }
}

// Linv = L^-1 for the factored kb x kb diagonal block at (k, k): a lower-
// triangular 64 x 64 block, zero above the diagonal and beyond kb, written
// row by row together with its S slices (out [S][kb][64], exponents expo[kb];
// the B operand of the panel solve).  Row i of L^-1 solves x^T L = e_i^T;
// with U'_rc = l_rc / l_cc (columns divided by their diagonal on load) it is
// x_i = 1 / l_ii and x_c = -sum_{r > c} x_r U'_rc, taken by backward
// substitution: one warp per row (16 CTAs of 4 warps, one per SM
// sub-partition, each staging only the rows its rows read), lanes holding
// columns lane and lane + 32, one shuffle and one FMA per step.  A dependent
// FP64 operation costs about as much as a shuffle on this part, so the unit
// diagonal keeps the division off the chain.  The warp then slices its row
// as k_slice_rows would.
constexpr int kTrtriWarps = 4;

__global__ void __launch_bounds__(32 * kTrtriWarps) k_trtri64(const double *__restrict__ A, int64_t n, int64_t k,
                                                              int kb, double *__restrict__ Linv, int S,
                                                              __nv_bfloat16 *__restrict__ out, int *__restrict__ expo) {
    __shared__ double U[kNB * kLd];
    __shared__ double rd[kNB];
    const int t = threadIdx.x, lane = t & 31;
    const int i = blockIdx.x * kTrtriWarps + (t >> 5);
    // row i of the inverse reads only rows 0 .. i of L
    const int rows = blockIdx.x * kTrtriWarps + kTrtriWarps;  // rows staged: 0 .. rows - 1
    for (int c = t; c < kNB; c += 32 * kTrtriWarps) rd[c] = c < kb ? 1.0 / A[(size_t)(k + c) * n + k + c] : 1.0;
    __syncthreads();
    for (int e = t; e < rows * kNB; e += 32 * kTrtriWarps) {
        const int r = e / kNB, c = e % kNB;
        U[r * kLd + c] = (r < kb && c < r) ? A[(size_t)(k + r) * n + k + c] * rd[c] : 0.0;
    }
    __syncthreads();
    double x0 = 0.0, x1 = 0.0;  // columns lane, lane + 32 of row i
    if (i < kb) {
        // acc holds -sum_{r > c} x_r U'_rc over the rows finished so far; x_c is
        // final once row c + 1 has been applied
        double acc0 = lane == i ? rd[i] : 0.0, acc1 = lane + 32 == i ? rd[i] : 0.0;
        for (int r = i; r >= 1; --r) {  // warp-uniform bounds
            const double xr = r < 32 ? __shfl_sync(0xffffffffu, acc0, r) : __shfl_sync(0xffffffffu, acc1, r - 32);
            // columns c < r take -x_r U'_rc (U' is zero on and above the diagonal)
            acc0 = fma(-xr, U[r * kLd + lane], acc0);
            if (r > 32) acc1 = fma(-xr, U[r * kLd + lane + 32], acc1);
        }
        x0 = acc0;
        x1 = acc1;
        slice_row_warp(x0, x1, lane, kb, i, S, false, out, expo);
    }
    Linv[(size_t)i * kNB + lane] = x0;
    Linv[(size_t)i * kNB + lane + 32] = x1;
}

// Rows below the diagonal block: X = A L_kk^-T by substitution in FP64, the
// result written back and, in the same pass, as S slices (out [S][rows][64],
// exponents expo[rows]) for the updates to come.  With y_c = x_c l_cc and V_cj
// = l_cj / l_jj the substitution is y_c = a_c - sum_{j < c} y_j V_cj: one
// shuffle and one FMA a step on the chain, the scaling by 1 / l_cc at the end.
// One warp per row, lanes holding columns lane and lane + 32, 8 rows a CTA at
// a time.
// Against the product with the inverted block (k_trtri64 + k_slice_rows +
// k_ozaki_gemm + k_slice_rows: about 28 us on the panel chain): substitution
// is backward stable whatever the block's condition, takes one launch, and
// 17 to 22 us up to 3072 rows (FP64 latencies, whatever the number of rows), 50
// us at 8192.  kTrsmRows is where the two meet; NK_F64 takes the
// substitution at every size.
constexpr int64_t kTrsmRows = 3072;

__global__ void __launch_bounds__(256) k_trsm_rows(double *__restrict__ A, int64_t n, int64_t k, int64_t rows, int S,
                                                   bool round, __nv_bfloat16 *__restrict__ out,
                                                   int *__restrict__ expo) {
    __shared__ double V[kNB * kLd];
    __shared__ double rd[kNB];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (t < kNB) rd[t] = 1.0 / A[(size_t)(k + t) * n + k + t];
    __syncthreads();
    for (int e = t; e < kNB * kNB; e += 256) {
        const int c = e >> 6, j = e & 63;
        V[c * kLd + j] = j < c ? A[(size_t)(k + c) * n + k + j] * rd[j] : 0.0;
    }
    __syncthreads();
    for (int64_t r = (int64_t)blockIdx.x * 8 + warp; r < rows; r += (int64_t)gridDim.x * 8) {
        double *row = A + (size_t)(k + kNB + r) * n + k;
        double y0 = row[lane], y1 = row[lane + 32];
#pragma unroll 8
        for (int c = 0; c < 32; ++c) {
            const double yc = __shfl_sync(0xffffffffu, y0, c);
            y0 = fma(-yc, V[lane * kLd + c], y0);
            y1 = fma(-yc, V[(lane + 32) * kLd + c], y1);
        }
#pragma unroll 8
        for (int c = 32; c < 64; ++c)
            y1 = fma(-__shfl_sync(0xffffffffu, y1, c - 32), V[(lane + 32) * kLd + c], y1);
        const double x0 = y0 * rd[lane], x1 = y1 * rd[lane + 32];
        row[lane] = x0;
        row[lane + 32] = x1;
        slice_row_warp(x0, x1, lane, rows, r, S, round, out, expo);
    }
}

// ---------------------------------------------- triangular solves with L ---
//
// One cooperative launch per direction.  CTA b owns block rows b, b + G, ...
// (64 rows each) in solve order.  For its block row i it streams the blocks
// L_ij of the rows already solved, accumulating L_ij y_j with coalesced row
// loads, then applies the inverted diagonal block and writes y_i.  There are
// no flags: the solved vector starts filled with a NaN sentinel (all bytes
// 0xFF, a pattern FP64 arithmetic does not produce), and each warp waits on
// the values themselves, so that the wait and the load of y_j are one L2
// access on the chain of dependent block rows.  Every block row waits only on
// rows that come earlier in solve order, and a CTA takes its rows in that
// order, so with all CTAs resident (cooperative launch) every wait ends; each
// wait is still bounded by the global timer and records error 6 (forward) or
// 7 (backward), after which the CTA finishes its row without waiting again.
// (A right-hand side holding a NaN with exactly the sentinel's payload would
// read as unsolved and end in that time-out error rather than in a NaN.)
constexpr int kTrsvThreads = 256;
constexpr unsigned long long kSolveSentinel = 0xFFFFFFFFFFFFFFFFULL;

__device__ __forceinline__ double ld_relaxed_f64(const double *p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return __longlong_as_double((long long)v);
}

// The warp waits until both y[lane] and y[lane + 32] hold solved values
// (lanes past `valid` read nothing and give 0); false on time-out.
__device__ bool wait_solved(const double *y, int lane, int valid, double &a, double &b, int *err, int code) {
    const unsigned long long t0 = global_ns();
    for (long long it = 0;; ++it) {
        a = lane < valid ? ld_relaxed_f64(y + lane) : 0.0;
        b = lane + 32 < valid ? ld_relaxed_f64(y + lane + 32) : 0.0;
        const bool ok = (unsigned long long)__double_as_longlong(a) != kSolveSentinel &&
                        (unsigned long long)__double_as_longlong(b) != kSolveSentinel;
        if (__all_sync(0xffffffffu, ok)) return true;
        if ((it & 63) == 63 && global_ns() - t0 > kWaitNs) {
            if (lane == 0) atomicExch(err, code);
            return false;
        }
    }
}

// One step of refinement of z = M acc, M = L_ii^-1 (or its transpose) as
// computed: z += M (acc - L z), so that the block solve is as accurate as
// substitution with L_ii whatever its condition (NK_F64).  Thread (r, q) holds
// 16 entries of row r of M (m) and of L (l); v: its row's entry of z, summed
// over the four threads of the row.  zs, rs: 64 doubles of shared memory each.
__device__ __forceinline__ double refine_block(const double (&m)[16], const double (&l)[16], double v, int r, int q,
                                               const double *acc, double *zs, double *rs) {
    if (q == 0) zs[r] = v;
    __syncthreads();
    double a = 0.0, b = 0.0;
#pragma unroll
    for (int u = 0; u < 16; u += 2) {
        a = fma(l[u], zs[q * 16 + u], a);
        b = fma(l[u + 1], zs[q * 16 + u + 1], b);
    }
    double lz = a + b;
    lz += __shfl_xor_sync(0xffffffffu, lz, 1);
    lz += __shfl_xor_sync(0xffffffffu, lz, 2);
    if (q == 0) rs[r] = acc[r] - lz;
    __syncthreads();
    a = b = 0.0;
#pragma unroll
    for (int u = 0; u < 16; u += 2) {
        a = fma(m[u], rs[q * 16 + u], a);
        b = fma(m[u + 1], rs[q * 16 + u + 1], b);
    }
    double dz = a + b;
    dz += __shfl_xor_sync(0xffffffffu, dz, 1);
    dz += __shfl_xor_sync(0xffffffffu, dz, 2);
    return v + dz;
}

// L y = b: y (sentinel-filled) receives the solution; b is read and refilled
// with the sentinel for the backward solve.
// Row stride of the inverse in shared memory: the rows and columns that a half
// warp reads at a time fall on different banks.
// What bounds a block row is the FP64 pipe of its SM, 19 cycles a warp
// instruction: 128 for the last block's product, and the sums over the lanes and
// the product with the inverse, which take 72 each (320 and 128, and 32-way bank
// conflicts, as sums row by row and a square product: 6.8 us a block row forward
// and 3.8 back, 3.2 and 2.9 now, n = 8192).
constexpr int kInvLd = kNB + 4;

template <bool kRefine>
__global__ void __launch_bounds__(kTrsvThreads) k_trsv_fwd(const double *__restrict__ L, int64_t n,
                                                           const double *__restrict__ Linv, double *b, double *y,
                                                           int *err) {
    __shared__ double inv[kNB * kInvLd];
    __shared__ double acc[kNB];
    const int nb = (int)((n + kNB - 1) / kNB);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int i = blockIdx.x; i < nb; i += gridDim.x) {
        const int64_t r0 = (int64_t)i * kNB;
        const int kb = (int)(n - r0 < kNB ? n - r0 : kNB);
        for (int e = t; e < kNB * kNB; e += kTrsvThreads)
            inv[(e >> 6) * kInvLd + (e & 63)] = Linv[(size_t)i * kNB * kNB + e];
        // warp w: rows 8w .. 8w + 7 of the block; lanes: columns lane, lane + 32
        // (the right-hand side of row lane / 4 read early)
        // Sums over groups of blocks (16 terms a lane) are added up: one chain of n / 32
        // terms errs several times as much, also systematically where rows are alike
        // (n = 8000, samples most of which agree: residual 6.0e-15, 1.1e-15 by columns).
        // The last block goes on from the total, so that nothing waits for it.
        double part[8] = {}, total[8] = {};
        const double bi = warp * 8 + (lane >> 2) < kb ? b[r0 + warp * 8 + (lane >> 2)] : 0.0;
        bool live = true;
        for (int j = 0; j < i && live; ++j) {
            const int64_t c0 = (int64_t)j * kNB;  // j < i: a full block
            // the block's L entries are in flight while the warp waits for y_j
            double p0[8], p1[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int r = warp * 8 + u;
                const double *row = L + (size_t)(r0 + (r < kb ? r : 0)) * n + c0;
                p0[u] = row[lane];
                p1[u] = row[lane + 32];
            }
            if ((j & 7) == 0 || j + 1 == i) {  // (before the wait: nothing is late by it)
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    total[u] += part[u];
                    part[u] = j + 1 == i ? total[u] : 0.0;
                }
            }
            double y0, y1;
            live = wait_solved(y + c0, lane, kNB, y0, y1, err, 6);
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (warp * 8 + u < kb) part[u] = fma(p0[u], y0, fma(p1[u], y1, part[u]));
        }
        // sums over the lanes, eight at a time: each exchange halves the values a
        // lane holds, 9 additions in place of 40; lane 4 u ends with row u's
#pragma unroll
        for (int h = 4; h >= 1; h >>= 1) {
            const bool hi = lane & (4 * h);
#pragma unroll
            for (int u = 0; u < h; ++u) {
                const double give = hi ? part[u] : part[u + h], keep = hi ? part[u + h] : part[u];
                part[u] = keep + __shfl_xor_sync(0xffffffffu, give, 4 * h);
            }
        }
        part[0] += __shfl_xor_sync(0xffffffffu, part[0], 2);
        part[0] += __shfl_xor_sync(0xffffffffu, part[0], 1);
        if ((lane & 3) == 0) {
            const int r = warp * 8 + (lane >> 2);
            acc[r] = r < kb ? bi - part[0] : 0.0;
            if (r < kb) b[r0 + r] = __longlong_as_double((long long)kSolveSentinel);
        }
        __syncthreads();
        // y_i = Linv_i acc: four threads per row, every fourth column each up to
        // the last row of the warp, in two independent FMA chains
        {
            const int r = t >> 2, q = t & 3;
            double ya = 0.0, yb = 0.0;
#pragma unroll 2
            for (int c = q; c < 8 * warp + 8; c += 8) {
                ya = fma(inv[r * kInvLd + c], acc[c], ya);
                yb = fma(inv[r * kInvLd + c + 4], acc[c + 4], yb);
            }
            double v = ya + yb;
            v += __shfl_xor_sync(0xffffffffu, v, 1);
            v += __shfl_xor_sync(0xffffffffu, v, 2);
            if (kRefine) {
                __shared__ double zs[kNB], rs[kNB];
                double m[16], l[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    const int c = q * 16 + u;
                    m[u] = inv[r * kInvLd + c];
                    l[u] = (r < kb && c <= r) ? L[(size_t)(r0 + r) * n + r0 + c] : 0.0;
                }
                v = refine_block(m, l, v, r, q, acc, zs, rs);
            }
            if (q == 0 && r < kb) __stcg(y + r0 + r, v);
        }
        __syncthreads();  // inv and acc are reused by the CTA's next row
    }
}

// L^T x = y: y holds the forward solution; x goes to b (sentinel-filled by
// the forward solve).  Block rows are solved from the last to the first.
template <bool kRefine>
__global__ void __launch_bounds__(kTrsvThreads) k_trsv_bwd(const double *__restrict__ L, int64_t n,
                                                           const double *__restrict__ Linv, double *b,
                                                           const double *y, int *err) {
    __shared__ double inv[kNB * kInvLd];
    __shared__ double part_s[kTrsvThreads / 32][kNB];
    __shared__ double acc[kNB];
    const int nb = (int)((n + kNB - 1) / kNB);
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int ii = blockIdx.x; ii < nb; ii += gridDim.x) {
        const int i = nb - 1 - ii;
        const int64_t c0 = (int64_t)i * kNB;
        const int kb = (int)(n - c0 < kNB ? n - c0 : kNB);
        for (int e = t; e < kNB * kNB; e += kTrsvThreads)
            inv[(e >> 6) * kInvLd + (e & 63)] = Linv[(size_t)i * kNB * kNB + e];
        // lanes: columns lane, lane + 32 of block column i; warp w: rows w, w + 8, ... of block row j
        // (in groups of four blocks, as the forward sums)
        double p0 = 0.0, p1 = 0.0, t0 = 0.0, t1 = 0.0;
        const bool v0 = lane < kb, v1 = lane + 32 < kb;
        const double yi = t < kb ? y[c0 + t] : 0.0;  // the right-hand side, read early (threads < 64 use it)
        bool live = true;
        for (int j = nb - 1; j > i && live; --j) {
            const int64_t r0 = (int64_t)j * kNB;
            const int kr = (int)(n - r0 < kNB ? n - r0 : kNB);
            // the block's L entries are in flight while the warp waits for x_j
            double q0[8], q1[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int r = warp + 8 * u;
                const double *row = L + (size_t)(r0 + (r < kr ? r : 0)) * n + c0;
                q0[u] = v0 ? row[lane] : 0.0;
                q1[u] = v1 ? row[lane + 32] : 0.0;
            }
            if ((j & 3) == 0 || j == i + 1) {
                t0 += p0;
                t1 += p1;
                p0 = j == i + 1 ? t0 : 0.0;
                p1 = j == i + 1 ? t1 : 0.0;
            }
            double xa, xb;  // x_j: lane holds rows lane, lane + 32 of block j
            live = wait_solved(b + r0, lane, kr, xa, xb, err, 7);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int r = warp + 8 * u;  // < 64: its x is in lane r (xa) or r - 32 (xb)
                const double xr = r < 32 ? __shfl_sync(0xffffffffu, xa, r) : __shfl_sync(0xffffffffu, xb, r - 32);
                if (r < kr) {
                    p0 = fma(q0[u], xr, p0);
                    p1 = fma(q1[u], xr, p1);
                }
            }
        }
        part_s[warp][lane] = p0;
        part_s[warp][lane + 32] = p1;
        __syncthreads();
        if (t < kNB) {
            double sum = 0.0;
#pragma unroll
            for (int w = 0; w < kTrsvThreads / 32; ++w) sum += part_s[w][t];
            acc[t] = t < kb ? yi - sum : 0.0;
        }
        __syncthreads();
        // x_i = Linv_i^T acc: four threads per column, every fourth row each from
        // the first column of the warp on, in two independent FMA chains
        {
            const int c = t >> 2, q = t & 3;
            double xa = 0.0, xb = 0.0;
#pragma unroll 2
            for (int r = 8 * warp + q; r < kNB; r += 8) {
                xa = fma(inv[r * kInvLd + c], acc[r], xa);
                xb = fma(inv[(r + 4) * kInvLd + c], acc[r + 4], xb);
            }
            double x = xa + xb;
            x += __shfl_xor_sync(0xffffffffu, x, 1);
            x += __shfl_xor_sync(0xffffffffu, x, 2);
            if (kRefine) {
                __shared__ double zs[kNB], rs[kNB];
                double m[16], l[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) {
                    const int r = q * 16 + u;
                    m[u] = inv[r * kInvLd + c];
                    l[u] = (r < kb && r >= c) ? L[(size_t)(c0 + r) * n + c0 + c] : 0.0;
                }
                x = refine_block(m, l, x, c, q, acc, zs, rs);
            }
            if (q == 0 && c < kb) __stcg(b + c0 + c, x);
        }
        __syncthreads();  // inv, part_s and acc are reused by the CTA's next row
    }
}

// Lower triangle of K holds g_t = t_k . t_l; replace it (both triangles) by
// the Gram of the Jacobian rows g_s + g_t + g_t g_s with g_s = s_k . s_l
// (exact integer dot products of the +-1 configurations).  The tile passes
// through shared memory, so that both triangles are read and written in rows
// (entry by entry from the registers of the products, 8 bytes at a stride of a
// row: 434 us for 8192 rows, 285 so).
__global__ void __launch_bounds__(256) k_gram_combine(int N, int64_t Ns, const int8_t *__restrict__ s,
                                                      double *__restrict__ K) {
    __shared__ __align__(16) unsigned char raw[64 * 65 * 8];
    int8_t(*sa)[132] = reinterpret_cast<int8_t(*)[132]>(raw);
    int8_t(*sb)[132] = reinterpret_cast<int8_t(*)[132]>(raw + 64 * 132);
    double(*tile)[65] = reinterpret_cast<double(*)[65]>(raw);  // once the configurations are done with
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t m0 = (int64_t)blockIdx.y * 64, n0 = (int64_t)blockIdx.x * 64;
    if (n0 > m0 + 63) return;
    int gs[4][4] = {};
    for (int i0 = 0; i0 < N; i0 += 128) {
        for (int e = threadIdx.x; e < 64 * 128; e += 256) {
            const int r = e >> 7, c = e & 127;
            const int i = i0 + c;
            sa[r][c] = (m0 + r < Ns && i < N) ? s[(size_t)(m0 + r) * N + i] : (int8_t)0;
            sb[r][c] = (n0 + r < Ns && i < N) ? s[(size_t)(n0 + r) * N + i] : (int8_t)0;
        }
        __syncthreads();
        for (int c = 0; c < 128; c += 4) {
            int av[4], bv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                av[u] = *reinterpret_cast<const int *>(&sa[ty * 4 + u][c]);
                bv[u] = *reinterpret_cast<const int *>(&sb[tx * 4 + u][c]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) gs[u][v] = __dp4a(av[u], bv[v], gs[u][v]);
        }
        __syncthreads();
    }
    auto in_lower = [&](int r, int c) { return m0 + r < Ns && n0 + c <= m0 + r; };  // then n0 + c < Ns too
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int e = threadIdx.x + 256 * i, r = e >> 6, c = e & 63;
        tile[r][c] = in_lower(r, c) ? K[(size_t)(m0 + r) * Ns + n0 + c] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            double &x = tile[ty * 4 + u][tx * 4 + v];
            const double gt = x;
            x = (double)gs[u][v] + gt + gt * (double)gs[u][v];
        }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int e = threadIdx.x + 256 * i, r = e >> 6, c = e & 63;
        if (in_lower(r, c)) K[(size_t)(m0 + r) * Ns + n0 + c] = tile[r][c];
        if (in_lower(c, r)) K[(size_t)(n0 + r) * Ns + m0 + c] = tile[c][r];
    }
}

size_t ozaki_smem_bytes() {
    return 1024 + (size_t)kMaxSlices * kABytes + (size_t)2 * kMaxSlices * kPBBytes +
           (size_t)kPEpiWarps * 32 * kPColsPerWarp * sizeof(double) + 10 * sizeof(uint64_t) + 16;
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// ============================================================ launchers ====

size_t slice_elems(int64_t rows, int S) { return (size_t)S * (size_t)rows * kTileK; }

cudaError_t launch_slice_rows(const double *A, int64_t lda, int64_t rows, int kcols, int S,
                              __nv_bfloat16 *out, int *expo, cudaStream_t st, bool round) {
    if (rows <= 0) return cudaSuccess;
    if (kcols < 1 || kcols > kTileK || S < 1 || S > kMaxSlices) return cudaErrorInvalidValue;
    (k_slice_rows<<<nblk(rows, 8), 256, 0, st>>>(A, lda, rows, kcols, S, round, out, expo), nk::note_launch());
    return cudaGetLastError();
}

// R = A B^T (FP64-accurate to the slice count), applied to C by mode.
// A and B are given by their slices (rows x 64, as written by
// launch_slice_rows) and row exponents.  wide: 7 slices, level 9 kept (NK_F64).
cudaError_t launch_ozaki_gemm_strided(const __nv_bfloat16 *Asl, const int *expA, int64_t rows, int64_t a_stride,
                                      const __nv_bfloat16 *Bsl, const int *expB, int64_t cols, int64_t b_stride,
                                      int S, double *C, int64_t ldc, int mode, bool lower, int *err,
                                      cudaStream_t st, bool wide) {
    if (rows <= 0 || cols <= 0) return cudaSuccess;
    if (S < 1 || S > kMaxSlices || (wide && S != kMaxSlices)) return cudaErrorInvalidValue;
    if (rows > (1LL << 31) - kTileM || cols > (1LL << 31) - kPN) return cudaErrorInvalidValue;
    CUtensorMap ma, mb;
    if (!make_slice_map(&ma, Asl, rows, S, kTileM, a_stride) || !make_slice_map(&mb, Bsl, cols, S, kPN, b_stride))
        return cudaErrorInvalidValue;
    const auto kern = wide ? k_ozaki_gemm<kMaxSlices, true>
                           : (S == kMaxSlices ? k_ozaki_gemm<kMaxSlices, false> : k_ozaki_gemm<0, false>);
    cudaError_t e = nk::allow_max_dynamic_smem((const void *)kern);
    if (e != cudaSuccess) return e;
    OzArgs a{rows, cols, S, expA, expB, C, ldc, mode, lower ? 1 : 0, err, (cols + kPN - 1) / kPN, 1, 0,
             ldc % 2 == 0 && reinterpret_cast<uintptr_t>(C) % 16 == 0};
    const int64_t n_mb = (rows + kTileM - 1) / kTileM;
    // strips of up to 8 tiles amortise a CTA's A slices over its tiles; a
    // product with few tiles per SM (the panel solve and the narrow update of
    // the Cholesky, on its critical path) takes one tile per CTA instead
    int64_t tiles = 0;
    for (int64_t m = 0; m < n_mb; ++m) tiles += oz_row_tiles(a.n_nb, lower, m);
    int dev = 0, sms = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int64_t per_sm = sms > 0 ? tiles / sms : kMaxChunk;
    while (a.chunk < kMaxChunk && 2 * a.chunk <= per_sm) {
        a.chunk *= 2;
        ++a.chunk_log2;
    }
    int64_t strips = 0;
    for (int64_t m = 0; m < n_mb; ++m) strips += oz_row_strips(a.n_nb, lower, m, a.chunk_log2);
    if (strips > (1LL << 31) - 1) return cudaErrorInvalidValue;
    (kern<<<(unsigned)strips, kPThreads, ozaki_smem_bytes(), st>>>(ma, mb, a), nk::note_launch());
    return cudaGetLastError();
}

// BF16 MMA flops a launch executes: active tiles x S(S+1)/2 slice products (wide: S -
// 1 more) x 2 x 128 x 32 x 64.
double ozaki_mma_flops(int64_t rows, int64_t cols, int S, bool lower, bool wide = false) {
    const int64_t tm = (rows + kTileM - 1) / kTileM, tn = (cols + kPN - 1) / kPN;
    int64_t tiles = 0;
    for (int64_t i = 0; i < tm; ++i) tiles += oz_row_tiles(tn, lower, i);
    return (double)tiles * (S * (S + 1) / 2 + (wide ? S - 1 : 0)) * 2.0 * kTileM * kPN * kTileK;
}

cudaError_t launch_ozaki_gemm(const __nv_bfloat16 *Asl, const int *expA, int64_t rows,
                              const __nv_bfloat16 *Bsl, const int *expB, int64_t cols, int S, double *C,
                              int64_t ldc, int mode, bool lower, int *err, cudaStream_t st, bool wide) {
    return launch_ozaki_gemm_strided(Asl, expA, rows, rows, Bsl, expB, cols, cols, S, C, ldc, mode, lower, err, st,
                                     wide);
}

size_t tc_chol_ws_bytes(int64_t n) {
    const int64_t nb = (n + kNB - 1) / kNB;
    return 2 * slice_elems(n, kMaxSlices) * 2 + slice_elems(kNB, kMaxSlices) * 2 + (size_t)(2 * n + kNB) * 4 +
           (size_t)nb * kNB * kNB * 8 + (size_t)n * 8 + 9 * 256;
}

namespace {
struct TcWs {
    __nv_bfloat16 *Asl, *Bsl, *Asl2;
    int *expA, *expB, *expA2;
    double *Linv;
    double *y;   // [n] forward-solve vector of the triangular solves
};
TcWs carve_tc(void *ws, int64_t n) {
    char *p = static_cast<char *>(ws);
    auto take = [&](size_t bytes) {
        char *q = p;
        p += (bytes + 255) & ~size_t(255);
        return q;
    };
    TcWs w;
    w.Asl = reinterpret_cast<__nv_bfloat16 *>(take(slice_elems(n, kMaxSlices) * 2));
    w.Bsl = reinterpret_cast<__nv_bfloat16 *>(take(slice_elems(kNB, kMaxSlices) * 2));
    w.expA = reinterpret_cast<int *>(take((size_t)n * 4));
    w.expB = reinterpret_cast<int *>(take((size_t)kNB * 4));
    w.Linv = reinterpret_cast<double *>(take((size_t)((n + kNB - 1) / kNB) * kNB * kNB * 8));
    w.Asl2 = reinterpret_cast<__nv_bfloat16 *>(take(slice_elems(n, kMaxSlices) * 2));
    w.expA2 = reinterpret_cast<int *>(take((size_t)n * 4));
    w.y = reinterpret_cast<double *>(take((size_t)n * 8));
    return w;
}
}  // namespace

// Blocked right-looking Cholesky with tensor-core (Ozaki, 7 slices) panel
// solves and trailing updates, and a look-ahead of one panel: after panel k
// the side stream updates block column k + 1 alone (the "narrow" update) and
// factors panel k + 1 (diagonal block, its inverse, the panel product and its
// slices), while the main stream applies panel k to the rest of the trailing
// matrix (the "wide" update).  Panel slices alternate between two buffers.
// The inverted diagonal blocks stay in the workspace for
// launch_cholesky_solve_tc.
namespace {

// Factor panel k (columns k0 .. k0 + kb - 1) whose block column is up to date:
// diagonal block, L_panel = A_panel L_kk^-T, slices of L_panel, and the inverse
// of the diagonal block for the triangular solves.
// By substitution (k_trsm_rows; `exact`, or few rows) the inverse is off the
// chain: with an aux stream (cs non-null) it runs there, and `joined` says that
// the aux stream must be joined before the inverses are read.  As a product
// with the inverse, the rows below the diagonal block are sliced on the aux
// stream beside the diagonal block's factorisation: the slicing depends only
// on the narrow update that precedes the panel.
cudaError_t panel_step(double *A, int64_t n, int64_t k0, int *info, int *err, TcWs &w, __nv_bfloat16 *Lsl,
                       int *Lexp, cudaStream_t st, const CholStreams *cs, bool exact, bool &joined) {
    const int S = kMaxSlices;
    const int kb = (int)(n - k0 < kNB ? n - k0 : kNB);
    const int64_t rest = n - k0 - kb;
    double *Linv = w.Linv + (size_t)(k0 / kNB) * kNB * kNB;
    double *panel = A + (size_t)(k0 + kb) * n + k0;
    cudaError_t e = cudaSuccess;
    const bool aux = cs != nullptr && cs->aux != nullptr;
    if (exact || rest <= kTrsmRows) {
        int slot = prof_begin(NK_PROF_CHOL_PANEL, st);
        (k_potrf64<<<1, kPotrfThreads, 0, st>>>(A, n, k0, kb, info), nk::note_launch());
        cudaStream_t is = st;
        if (aux && rest > 0) {
            e = cudaEventRecord(cs->ev_fork, st);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(cs->aux, cs->ev_fork, 0);
            if (e != cudaSuccess) return e;
            is = cs->aux;
            joined = false;
        }
        // (the slices of the inverse that the kernel also writes are not used here)
        (k_trtri64<<<kNB / kTrtriWarps, 32 * kTrtriWarps, 0, is>>>(A, n, k0, kb, Linv, S, w.Bsl, w.expB),
         nk::note_launch());
        if (rest > 0) {
            const unsigned grid = nblk(rest, 8) < 304 ? nblk(rest, 8) : 304;
            (k_trsm_rows<<<grid, 256, 0, st>>>(A, n, k0, rest, S, exact, Lsl, Lexp), nk::note_launch());
        }
        prof_end(slot, st, 2.0 * (double)kb * kb * kb / 3.0 + (double)rest * kb * kb);
        return cudaGetLastError();
    }
    if (aux) {
        e = cudaEventRecord(cs->ev_fork, st);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(cs->aux, cs->ev_fork, 0);
        if (e != cudaSuccess) return e;
        const int aslot = prof_begin(NK_PROF_CHOL_PANEL, cs->aux);
        e = launch_slice_rows(panel, n, rest, kb, S, Lsl, Lexp, cs->aux, false);
        prof_end(aslot, cs->aux, 0.0);
        if (e == cudaSuccess) e = cudaEventRecord(cs->ev_join, cs->aux);
        if (e != cudaSuccess) return e;
        joined = true;
    }
    // timing classes: the FP64 diagonal-block kernels and the slicing count
    // as the panel, the tensor-core panel product with the trailing updates
    int slot = prof_begin(NK_PROF_CHOL_PANEL, st);
    (k_potrf64<<<1, kPotrfThreads, 0, st>>>(A, n, k0, kb, info), nk::note_launch());
    // the inverse and its slices (the B operand of the panel solve)
    (k_trtri64<<<kNB / kTrtriWarps, 32 * kTrtriWarps, 0, st>>>(A, n, k0, kb, Linv, S, w.Bsl, w.expB),
     nk::note_launch());
    e = aux ? cudaStreamWaitEvent(st, cs->ev_join, 0) : launch_slice_rows(panel, n, rest, kb, S, Lsl, Lexp, st, false);
    prof_end(slot, st, 2.0 * (double)kb * kb * kb / 3.0);
    if (e == cudaSuccess) {
        slot = prof_begin(NK_PROF_CHOL_UPDATE, st);
        e = launch_ozaki_gemm(Lsl, Lexp, rest, w.Bsl, w.expB, kb, S, panel, n, 0, false, err, st, false);
        // the triangular solve L21 = A21 L11^-T: rest kb^2 flops in FP64
        prof_end(slot, st, (double)rest * kb * kb, ozaki_mma_flops(rest, kb, S, false));
        slot = prof_begin(NK_PROF_CHOL_PANEL, st);
        if (e == cudaSuccess) e = launch_slice_rows(panel, n, rest, kb, S, Lsl, Lexp, st, false);
        prof_end(slot, st, 0.0);
    }
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t launch_cholesky_tc(double *A, int64_t n, int *info, int *err, void *ws, cudaStream_t st,
                               const CholStreams *cs, bool exact) {
    // Step k, with panel k factored and sliced:
    //   side stream: the narrow update (block column k+1 by panel k), then
    //     panel k+1 (factor, invert, solve, slice);
    //   main stream: the wide update (everything right of block column k+1).
    // The side stream waits for the previous wide update (block column k+1
    // must have received it, and panel k+1's slice buffer is the one that
    // update read); the main stream waits for panel k+1 before the next wide
    // update.  A step then takes max(wide, narrow + panel).
    TcWs w = carve_tc(ws, n);
    const int S = kMaxSlices;
    cudaError_t e = cudaSuccess;
    __nv_bfloat16 *buf[2] = {w.Asl, w.Asl2};
    int *bexp[2] = {w.expA, w.expA2};
    const int64_t nb = (n + kNB - 1) / kNB;
    const bool two = cs != nullptr && cs->side != nullptr;
    cudaStream_t side = two ? cs->side : nullptr, ps = two ? cs->side : st;
    cudaEvent_t ev_wide = two ? cs->ev_wide : nullptr, ev_panel = two ? cs->ev_panel : nullptr;
    bool joined = true;
    e = panel_step(A, n, 0, info, err, w, buf[0], bexp[0], st, cs, exact, joined);
    if (e != cudaSuccess) return e;
    for (int64_t k = 0; k + 1 < nb; ++k) {
        const int64_t k0 = k * kNB;
        const int64_t rest = n - k0 - kNB;         // rows of panel k below its diagonal block
        const int kb1 = (int)(rest < kNB ? rest : kNB);  // width of block column k + 1
        __nv_bfloat16 *Lk = buf[k & 1];
        int *Le = bexp[k & 1];
        double *C1 = A + (size_t)(k0 + kNB) * n + (k0 + kNB);
        if (two) {
            e = cudaEventRecord(ev_wide, st);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(side, ev_wide, 0);
            if (e != cudaSuccess) return e;
        }
        // narrow: block column k + 1 (all rows below panel k)
        int slot = prof_begin(NK_PROF_CHOL_UPDATE, ps);
        e = launch_ozaki_gemm_strided(Lk, Le, rest, rest, Lk, Le, kb1, rest, S, C1, n, 1, true, err, ps, exact);
        // FP64 flops of the lower part of the rest x kb1 block column, K = kNB
        prof_end(slot, ps, 2.0 * kNB * ((double)rest * kb1 - 0.5 * (double)kb1 * (kb1 - 1)),
                 ozaki_mma_flops(rest, kb1, S, true, exact));
        if (e != cudaSuccess) return e;
        e = panel_step(A, n, k0 + kNB, info, err, w, buf[(k + 1) & 1], bexp[(k + 1) & 1], ps, cs, exact,
                       joined);
        if (e != cudaSuccess) return e;
        if (two) {
            e = cudaEventRecord(ev_panel, side);
            if (e != cudaSuccess) return e;
        }
        // wide: everything right of block column k + 1
        const int64_t rest2 = rest - kb1;
        if (rest2 > 0) {
            slot = prof_begin(NK_PROF_CHOL_UPDATE, st);
            e = launch_ozaki_gemm_strided(Lk + (size_t)kb1 * kTileK, Le + kb1, rest2, rest, Lk + (size_t)kb1 * kTileK,
                                          Le + kb1, rest2, rest, S, C1 + (size_t)kb1 * n + kb1, n, 1, true, err, st,
                                          exact);
            // FP64 flops of the lower rest2 x rest2 trailing update, K = kNB
            prof_end(slot, st, (double)kNB * rest2 * (double)(rest2 + 1),
                     ozaki_mma_flops(rest2, rest2, S, true, exact));
            if (e != cudaSuccess) return e;
        }
        if (two) {
            e = cudaStreamWaitEvent(st, ev_panel, 0);
            if (e != cudaSuccess) return e;
        }
    }
    if (!joined) {  // the inverted diagonal blocks
        e = cudaEventRecord(cs->ev_join, cs->aux);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(st, cs->ev_join, 0);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

cudaError_t launch_cholesky_solve_tc(const double *L, int64_t n, const void *ws, double *b, int *err,
                                     cudaStream_t st, bool exact) {
    if (n <= 0) return cudaSuccess;
    TcWs w = carve_tc(const_cast<void *>(ws), n);
    const int nb = (int)((n + kNB - 1) / kNB);
    int dev = 0, sms = 0, per_sm_f = 0, per_sm_b = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const void *fwd = exact ? (const void *)k_trsv_fwd<true> : (const void *)k_trsv_fwd<false>;
    const void *bwd = exact ? (const void *)k_trsv_bwd<true> : (const void *)k_trsv_bwd<false>;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_f, fwd, kTrsvThreads, 0);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_b, bwd, kTrsvThreads, 0);
    if (e != cudaSuccess) return e;
    // at most one CTA per SM: the resident grid needs no more, and blocks
    // rows then spread over the SMs' load bandwidth
    const int gf = std::min(nb, sms * std::min(per_sm_f, 1)), gb = std::min(nb, sms * std::min(per_sm_b, 1));
    if (gf < 1 || gb < 1) return cudaErrorLaunchOutOfResources;
    const int slot = prof_begin(NK_PROF_TRSV, st);
    e = cudaMemsetAsync(w.y, 0xFF, (size_t)n * 8, st);  // the sentinel of unsolved entries
    if (e != cudaSuccess) return e;
    const double *Linv = w.Linv;
    double *y = w.y;
    void *args[] = {(void *)&L, (void *)&n, (void *)&Linv, (void *)&b, (void *)&y, (void *)&err};
    e = cudaLaunchCooperativeKernel(fwd, dim3(gf), dim3(kTrsvThreads), args, 0, st);
    nk::note_launch();
    if (e != cudaSuccess) return e;
    e = cudaLaunchCooperativeKernel(bwd, dim3(gb), dim3(kTrsvThreads), args, 0, st);
    nk::note_launch();
    prof_end(slot, st, 2.0 * (double)n * (double)n);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Lower triangle of K = T T^T by tensor cores with S slices per 64-column
// chunk of T [Ns][M], then the Jacobian-row Gram s.s + t.t + (t.t)(s.s)
// written to both triangles.
cudaError_t launch_gram_tc(int N, int M, int64_t Ns, const int8_t *s, const double *T, int S, double *K,
                           int *err, void *ws, cudaStream_t st, bool wide) {
    TcWs w = carve_tc(ws, Ns);
    const int slot = prof_begin(NK_PROF_GRAM, st);
    for (int c = 0; c < M; c += kTileK) {
        const int kc = M - c < kTileK ? M - c : kTileK;
        cudaError_t e = launch_slice_rows(T + c, M, Ns, kc, S, w.Asl, w.expA, st, wide);
        if (e == cudaSuccess)
            e = launch_ozaki_gemm(w.Asl, w.expA, Ns, w.Asl, w.expA, Ns, S, K, Ns, c == 0 ? 0 : 2, true, err, st,
                                  wide);
        if (e != cudaSuccess) return e;
    }
    dim3 grid(nblk(Ns, 64), nblk(Ns, 64));
    (k_gram_combine<<<grid, 256, 0, st>>>(N, Ns, s, K), nk::note_launch());
    // the lower triangle of the Jacobian-row Gram through s.s + t.t + (t.t)(s.s):
    // (N + M) flops per entry, the count of the FP64 path
    prof_end(slot, st, (double)Ns * (Ns + 1) * (double)(N + M),
             (double)((M + kTileK - 1) / kTileK) * ozaki_mma_flops(Ns, Ns, S, true, wide));
    return cudaGetLastError();
}

}  // namespace nk
