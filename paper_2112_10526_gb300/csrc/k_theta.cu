// Batched hidden activations theta = S W^T + b on the tensor cores (NetKet 3,
// Sec. 3.2): +-1 configurations [B][N] against W [M][N] cut row by row into 5
// FP16 slices of digits in base 4096, [-2048, 2048], of an integer of up to 59
// bits and a sign times a power of two per row (k_slice_rows_h5).  FP16 holds
// every integer up to 2048, so the sums over N <= 4096 are exact in FP32.  The
// five slices of 32 units lie side by side as one operand of 160 rows, so that
// one tcgen05.mma per 16 of K (M = 128, N = 160) fills the five FP32 levels of a
// 128 x 32 tile.  (The 7 BF16 slices of 8 bits of the other products hold 56
// bits in 7/5 of the tensor work and operand bytes.)
//
// A persistent kernel: each CTA walks a contiguous range of (row tile of 128
// configurations, unit tile) pairs, units fastest.  Up to 9 chunks of K (N <= 576)
// it keeps its configurations in shared memory for all its unit tiles and only the
// slices stream through a TMA ring; beyond, configurations stream along.  Warp 0 loads, warp 1 issues the MMAs into
// one of two accumulator sets, sixteen warps turn the other set into FP64 and
// store it by rows.
// What bounds it: for theta the slices in flight (20 KB a chunk, three to six
// stages, against about 1 us of L2 latency); with tanh and pairs the epilogue's
// integer instructions (8192 x 4608: ALU pipe 60 %, issue 54 %, tensor pipe 12 %).
// The tile kernel this replaces (k_sgemm: one 128 x 64 tile a CTA, nothing
// overlapping its drain) took 19 us for 1024 x 200 x 100 and 4.70 ms for 65536 x
// 4608 x 576.
// The epilogue writes theta in FP64, or (for the products of NK_MIXED that read
// tanh(theta) as FP32 pairs) t' = [tanh(theta), 1] straight into the tile order
// of k_tc4, with the exponents of its columns: the 24 x 24 lattice's 302 M
// activations then cross HBM once instead of six times (theta, tanh, exponents
// and two passes of pairs: 11 ms).
// Every wait is bounded; a time-out records a code, drains the copies and MMAs
// in flight and returns.

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "nk_common.cuh"
#include "nk_internal.h"
#include "tanh64.cuh"
#include "tc_ptx.cuh"

namespace nk {

namespace {

constexpr int kHS = 5;                          // slices
constexpr int kHM = 128, kHN = 32, kHK = 64;
constexpr int kHA = kHM * kHK * 2;              // a chunk of the configurations: 16 KB
constexpr int kHB = kHN * kHK * 2;              // one slice of a chunk: 4 KB
constexpr int kHResident = 9;                   // chunks of K kept in shared memory at most
constexpr int kHMaxStages = 6;
constexpr int kHEpiWarps = 16;
constexpr int kHThreads = 64 + 32 * kHEpiWarps;
constexpr uint32_t kHAcc = 256;                 // TMEM columns per accumulator set (160 used)
constexpr size_t kHStageOut = (size_t)kHEpiWarps * 32 * 4 * 8;  // 4 columns of 32 rows per warp
constexpr size_t kHSmem = 227 * 1024;

struct ThetaArgs {
    int64_t rows;
    int units, N;
    int kchunks, resident, nstages;
    int n_nt;            // unit tiles
    int64_t tiles;       // row tiles x n_nt
    int64_t per;         // tiles per CTA
    int bits, drop;      // V 2^(expW - bits), its lowest `drop` bits left out
    const int *expW;     // [units]
    const double *bias;  // [units]
    double *out;         // [rows][ld], or null:
    float4 *pairs;       // t' as FP32 pairs, tile-major (launch_split_t)
    int *colexp;         // [units + 1], -100000 before: exponents of the columns of t'
    int64_t ld;
    const int8_t *s;     // [rows][N] and W [units][N]: the units whose exponent is flagged
    const double *W;
    int *err;
};

__device__ __noinline__ double raw_theta(const ThetaArgs &a, int64_t row, int unit) {
    double acc = 0.0;
    for (int i = 0; i < a.N; ++i) acc = fma((double)a.s[(size_t)row * a.N + i], a.W[(size_t)unit * a.N + i], acc);
    return acc;
}

// floor(V / 2^drop) of the exact levels D_1 .. D_5, V = sum D_t 2^(12 (5 - t));
// |D_t| <= 2048 N.
__device__ __forceinline__ long long window_of(const uint32_t (&r)[kHS], int drop) {
    int d[kHS];
#pragma unroll
    for (int t = 0; t < kHS; ++t) d[t] = __float2int_rn(__uint_as_float(r[t]));
    const long long hi = (long long)d[0] * 16777216 + (long long)d[1] * 4096 + d[2];  // V = hi 2^24 + lo
    const long long lo = (long long)d[3] * 4096 + d[4];
    return (long long)((unsigned long long)hi << (24 - drop)) + (lo >> drop);
}

template <bool kPairs>
__global__ void __launch_bounds__(kHThreads, 1)
    k_theta(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, ThetaArgs a) {
    extern __shared__ unsigned char smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    unsigned char *ops = smem_raw + ((1024 - (base & 1023)) & 1023);
    const int NS = a.nstages;
    const int stage_bytes = kHS * kHB + (a.resident ? 0 : kHA);
    unsigned char *sA = ops;  // resident: [kchunks][128][64]
    unsigned char *sS = ops + (a.resident ? (size_t)a.kchunks * kHA : 0);
    unsigned char *sO = sS + (size_t)NS * stage_bytes;
    uint64_t *bars = reinterpret_cast<uint64_t *>(sO + kHStageOut);
    uint64_t *full = bars, *empty = bars + kHMaxStages, *a_full = bars + 2 * kHMaxStages, *a_empty = a_full + 1;
    uint64_t *acc_full = a_full + 2, *acc_empty = acc_full + 2;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(acc_empty + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t t0 = blockIdx.x * a.per;
    const int64_t t1 = t0 + a.per < a.tiles ? t0 + a.per : a.tiles;

    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(a_full, 1);
        mbar_init(a_empty, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kHEpiWarps);
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
        int64_t g = 0, row_loads = 0, mt_held = -1;
        for (int64_t t = t0; t < t1 && !*abort_flag; ++t) {
            const int64_t mt = t / a.n_nt;
            const int m0 = (int)(mt * kHM), n0 = (int)(t % a.n_nt) * kHN;
            if (a.resident && mt != mt_held) {
                if (row_loads > 0 &&
                    !mbar_wait_or_abort_sleep(a_empty, (uint32_t)((row_loads - 1) & 1), abort_flag)) {
                    fail(3);
                    break;
                }
                mbar_expect_tx(a_full, (uint32_t)(a.kchunks * kHA));
                for (int kc = 0; kc < a.kchunks; ++kc) tma_load_2d(sA + (size_t)kc * kHA, &mapA, a_full, kc * kHK, m0);
                mt_held = mt;
                ++row_loads;
            }
            for (int kc = 0; kc < a.kchunks; ++kc, ++g) {
                const int s = (int)(g % NS);
                if (g >= NS && !mbar_wait_or_abort_sleep(&empty[s], (uint32_t)((g / NS - 1) & 1), abort_flag)) {
                    fail(3);
                    break;
                }
                unsigned char *sp = sS + (size_t)s * stage_bytes;
                mbar_expect_tx(&full[s], (uint32_t)stage_bytes);
                for (int q = 0; q < kHS; ++q) tma_load_3d(sp + q * kHB, &mapB, &full[s], kc * kHK, n0, q);
                if (!a.resident) tma_load_2d(sp + kHS * kHB, &mapA, &full[s], kc * kHK, m0);
            }
        }
        if (*abort_flag) {
            // the copies in flight land before the CTA exits
            if (row_loads > 0) mbar_wait(a_full, (uint32_t)((row_loads - 1) & 1));
            for (int64_t h = g > NS ? g - NS : 0; h < g; ++h) mbar_wait(&full[h % NS], (uint32_t)((h / NS) & 1));
        }
    } else if (warp == 1 && lane == 0) {
        // ------------------------------------------------------- MMA issuer
        const uint32_t idesc = idesc_f16(kHM, kHN * kHS);
        int64_t g = 0, rows_used = 0, mt_held = -1, committed = -1;
        for (int64_t t = t0; t < t1 && !*abort_flag; ++t) {
            const int64_t li = t - t0, mt = t / a.n_nt;
            const int b = (int)(li & 1);
            const uint32_t use = (uint32_t)(li >> 1);
            if (use > 0 && !mbar_wait_or_abort_sleep(&acc_empty[b], (use - 1) & 1, abort_flag)) {
                fail(4);
                break;
            }
            if (a.resident && mt != mt_held) {
                if (!mbar_wait_or_abort_sleep(a_full, (uint32_t)(rows_used & 1), abort_flag)) {
                    fail(4);
                    break;
                }
                mt_held = mt;
                ++rows_used;
            }
            bool ok = true;
            for (int kc = 0; kc < a.kchunks; ++kc, ++g) {
                const int s = (int)(g % NS);
                if (!mbar_wait_or_abort_sleep(&full[s], (uint32_t)((g / NS) & 1), abort_flag)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                unsigned char *sp = sS + (size_t)s * stage_bytes;
                const uint64_t da = sw128_desc(a.resident ? sA + (size_t)kc * kHA : sp + kHS * kHB);
                const uint64_t db = sw128_desc(sp);
#pragma unroll
                for (int kk = 0; kk < kHK / 16; ++kk)
                    umma_bf16(tmem + (uint32_t)b * kHAcc, da + (uint64_t)(kk * 2), db + (uint64_t)(kk * 2), idesc,
                              (kc > 0 || kk > 0) ? 1u : 0u);
                umma_commit(&empty[s]);
            }
            if (a.resident && (t + 1 == t1 || (t + 1) / a.n_nt != mt)) umma_commit(a_empty);
            umma_commit(&acc_full[b]);
            committed = li;
            if (!ok) {
                fail(4);
                break;
            }
        }
        if (*abort_flag && committed >= 0)  // the MMAs in flight finish before the TMEM is released
            mbar_wait(&acc_full[committed & 1], (uint32_t)((committed >> 1) & 1));
    } else if (warp >= 2) {
        // --------------------------------------------------------- epilogue
        // warp: tile rows 32q .. 32q + 31 (its TMEM lane quarter), 8 units in two
        // passes of 4; values are parked in shared memory ([32 rows][4], unit
        // XOR row / 4 mod 4) and stored with 4 lanes on a row's 32 bytes
        const int q = warp & 3, c0 = ((warp - 2) >> 2) * 8;
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        double *stage = reinterpret_cast<double *>(sO) + (warp - 2) * 32 * 4;
        const int rr = lane >> 2, cc = lane & 3;
        for (int64_t t = t0; t < t1; ++t) {
            const int64_t li = t - t0;
            const int64_t m0 = t / a.n_nt * kHM + q * 32;
            const int n0 = (int)(t % a.n_nt) * kHN + c0;
            const int b = (int)(li & 1);
            int e_lane = 0;
            {
                const int u = n0 + (lane & 7);
                e_lane = u < a.units ? __ldg(a.expW + u) : 0;
            }
            double bv[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) bv[h] = n0 + 4 * h + cc < a.units ? __ldg(a.bias + n0 + 4 * h + cc) : 0.0;
            int ok = 1;
            if (lane == 0) ok = mbar_wait_or_abort_sleep(&acc_full[b], (uint32_t)(li >> 1) & 1, abort_flag) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) {
                if (lane == 0) fail(5);
                break;
            }
            tc_fence_after();
            // columns of t' that this warp's tile holds; the column of ones is `units`
            int held = -100000;
            if (kPairs) held = n0 + (lane & 7) <= a.units ? __ldcg(a.colexp + n0 + (lane & 7)) : 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t r[kHS][4];
#pragma unroll
                for (int g = 0; g < kHS; ++g)
                    tmem_ld4(tmem + (uint32_t)b * kHAcc + lane_base + (uint32_t)(g * kHN + c0 + 4 * h), r[g]);
                tmem_wait_ld();
                if (h == 1) {  // drained: the next tile but one may overwrite it
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[b]);
                }
                float2 pr[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t d[kHS];
#pragma unroll
                    for (int g = 0; g < kHS; ++g) d[g] = r[g][j];
                    const int e = __shfl_sync(0xffffffffu, e_lane, 4 * h + j);
                    double v = window_to_double(window_of(d, a.drop), e - a.bits + a.drop);
                    const int unit = n0 + 4 * h + j;
                    if (flagged_exp(e) && m0 + lane < a.rows && unit < a.units) v = raw_theta(a, m0 + lane, unit);
                    if (kPairs) {
                        // t', 0 past the last row and past the column of ones
                        const double b = __shfl_sync(0xffffffffu, bv[h], j);  // lane j holds unit 4 h + j
                        double t = unit < a.units ? tanh64(v + b) : (unit == a.units ? 1.0 : 0.0);
                        if (m0 + lane >= a.rows) t = 0.0;
                        pr[j] = fp32_pair(t);
                        const int be = (__double2hiint(t) >> 20) & 0x7FF;
                        int ex = be == 0 ? -100000 : (be == 2047 ? 100000 : be - 1022);
                        ex = __reduce_max_sync(0xffffffffu, ex);
                        if (lane == 4 * h + j && unit <= a.units && ex > held) atomicMax(a.colexp + unit, ex);
                    } else {
                        stage[lane * 4 + (j ^ ((lane >> 2) & 3))] = v;
                    }
                }
                if (kPairs) {
                    // 64-unit tiles of 32 column pairs x 128 rows
                    const int u0 = n0 + 4 * h;
                    const int64_t mt = t / a.n_nt;
                    float4 *dst = a.pairs + ((size_t)(mt * (a.n_nt / 2) + (u0 >> 6)) * 32 + ((u0 & 63) >> 1)) * kHM +
                                  q * 32 + lane;
                    __stcs(dst, make_float4(pr[0].x, pr[0].y, pr[1].x, pr[1].y));
                    __stcs(dst + kHM, make_float4(pr[2].x, pr[2].y, pr[3].x, pr[3].y));
                    continue;
                }
                __syncwarp();
                const int u = n0 + 4 * h + cc;
                if (u < a.units) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int rl = 8 * k + rr;
                        if (m0 + rl < a.rows)
                            a.out[(size_t)(m0 + rl) * a.ld + u] = stage[rl * 4 + (cc ^ ((rl >> 2) & 3))] + bv[h];
                    }
                }
                __syncwarp();
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

}  // namespace

cudaError_t launch_theta_product(const __half *A, int64_t rows, int64_t ldA, const __half *Wsl,
                                 const int *expW, int units, int N, const double *bias, double *out, int64_t ld,
                                 int bits, const int8_t *s, const double *W, int *err, cudaStream_t st,
                                 void *pairs, int *colexp) {
    if (rows <= 0 || units <= 0) return cudaSuccess;
    if (N > 4096 || rows > (1LL << 31) - 2 * kHM) return cudaErrorInvalidValue;
    EncodeTiledFn fn = encode_fn();
    if (!fn) return cudaErrorInvalidValue;
    CUtensorMap ma, mb;
    {
        cuuint64_t dims[2] = {(cuuint64_t)N, (cuuint64_t)rows}, str[1] = {(cuuint64_t)ldA * 2};
        cuuint32_t box[2] = {(cuuint32_t)kHK, (cuuint32_t)kHM}, es[2] = {1, 1};
        if (fn(&ma, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half *>(A), dims, str, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
        cuuint64_t dimb[3] = {(cuuint64_t)N, (cuuint64_t)units, (cuuint64_t)kHS};
        cuuint64_t strb[2] = {(cuuint64_t)ldA * 2, (cuuint64_t)units * ldA * 2};
        cuuint32_t boxb[3] = {(cuuint32_t)kHK, (cuuint32_t)kHN, 1}, esb[3] = {1, 1, 1};
        if (fn(&mb, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half *>(Wsl), dimb, strb, boxb, esb,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    const void *kern = pairs ? (const void *)k_theta<true> : (const void *)k_theta<false>;
    cudaError_t e = nk::allow_max_dynamic_smem(kern);
    int dev = 0, sms = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    ThetaArgs a{};
    a.rows = rows;
    a.units = units;
    a.N = N;
    a.kchunks = (N + kHK - 1) / kHK;
    a.resident = a.kchunks <= kHResident ? 1 : 0;
    // pairs: whole 64-unit tiles with the column of ones
    a.n_nt = pairs ? (units + 1 + 63) / 64 * 2 : (units + kHN - 1) / kHN;
    a.pairs = static_cast<float4 *>(pairs);
    a.colexp = colexp;
    // |V| <= N 2^bits in 63 bits; 56-bit integers drop ten bits whatever N is
    a.bits = bits;
    a.drop = bits == 56 ? 10 : window_drop(8 * (int64_t)N);
    a.expW = expW;
    a.bias = bias;
    a.out = out;
    a.ld = ld;
    a.s = s;
    a.W = W;
    a.err = err;
    const size_t fixed = 1024 + kHStageOut + (2 * kHMaxStages + 6) * sizeof(uint64_t) + 16 +
                         (a.resident ? (size_t)a.kchunks * kHA : 0);
    const size_t stage = (size_t)kHS * kHB + (a.resident ? 0 : kHA);
    a.nstages = (int)((kHSmem - fixed) / stage);
    if (a.nstages > kHMaxStages) a.nstages = kHMaxStages;
    const size_t smem = fixed + a.nstages * stage;
    const int64_t n_mt = (rows + kHM - 1) / kHM;
    a.tiles = n_mt * a.n_nt;
    const int64_t ctas = sms < a.tiles ? sms : a.tiles;
    a.per = (a.tiles + ctas - 1) / ctas;
    const unsigned grid = (unsigned)((a.tiles + a.per - 1) / a.per);
    if (pairs)
        (k_theta<true><<<grid, kHThreads, smem, st>>>(ma, mb, a), nk::note_launch());
    else
        (k_theta<false><<<grid, kHThreads, smem, st>>>(ma, mb, a), nk::note_launch());
    return cudaGetLastError();
}

}  // namespace nk
