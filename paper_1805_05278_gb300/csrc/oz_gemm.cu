// FP64 products on the BF16 tensor cores by exact digit splitting (the Ozaki
// scheme: Ozaki, Ogita, Oishi, Rump 2012), for the update, T-assembly and
// Q-application products of QR-EG once they are large:
//
//   C (FP64, M x N) = alpha * op(A) * B + beta * C.
//
// Why: this part runs FP64 at 1/64 of its FP32 rate and has no FP64 tensor
// pipe worth using (1.26 TFLOP/s either way), while BF16 tensor cores run
// at 1.9 PFLOP/s: 34 exact digit products cost far less than one FP64 one.
//
// Digits.  Every row of op(A) and every column of B is scaled by a power of
// two to magnitude < 1 and written as a 55-bit fixed-point number, cut into
// 7 balanced base-256 digits d_1 ... d_7, |d| <= 128, each exact in BF16 and
// stored with its weight 256^-(i-1).  A digit product is an integer of at
// most 2^14 times its weight, so the tensor cores' FP32 accumulators hold a
// sum of products of equal weight exactly while fewer than 2^24 / 2^14 =
// 1024 of them meet.  The weights i + j = 2 ... 7 (1 to 6 products per k)
// have an accumulator each, i + j = 8 and 9 share one; i + j >= 10 (below
// 2^-62 of the row and column maxima) is left out.  Every 256 k the
// accumulators are drained into a 64-bit integer per output (unit 2^-40 of a
// leading digit product), and the integer is rounded to FP64 once.  Sums over
// more than 512 k are integer partials, so neither the split nor the order
// changes a bit of the result.
//
// Error.  Entries within a factor 4 of the row (column) maximum are exact,
// the others lose what lies below 2^-56 of it; the sums are exact but for
// the FP32 rounding of the shared accumulator (2^-24 of a weight 2^-48).
// Measured on whole factorizations, backward error and orthogonality are at
// or below the FMA kernel's, which rounds at every k (graded 8192^2: backward
// error 6.6e-16, FMA 8.4e-16; Gaussian 4096^2: 1.8e-15, 2.3e-15).  Sharing
// one accumulator among i + j = 6, 7, 8 instead cost a digit and a half: the
// tensor cores' accumulation truncates, and its bias grows with K.
//
// Kernels of one product:
//   oz_slice_kernel   digits of both operands, K-major (HBM: 8 B read, 14
//                     written per entry), one launch
//   oz_mma_kernel     TMA -> shared memory -> tcgen05.mma -> TMEM -> C, or
//                     integer partials where K is split
//   oz_reduce_kernel  sums the partials and rounds (only where K is split)
//
// Measured (one factorization with the FMA kernel against this one): graded
// 8192^2 687 -> 157 ms, 32768 x 2048 256 -> 65 ms; the thin Q of 16001 x 1000
// 31.3 -> 3.3 ms.
#include "common.cuh"
#include "tc_ptx.cuh"

#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cmath>

namespace gbqr {
namespace {

constexpr int OZ_D = 7;              // digits per operand
constexpr int OZ_ACC = 7;            // accumulators: weights 2 .. 7, and 8 and 9 together
constexpr int OZ_BM = 128;
constexpr int OZ_BN = 64;            // 7 x 64 FP32 columns: 448 of the 512 of TMEM
constexpr int OZ_TOP = 9;            // largest i + j of the digit products taken
constexpr int OZ_BK = 32;            // one 64-byte swizzle row of BF16
constexpr int OZ_CHUNK = 8;          // K tiles per drain (256 k: the accumulators stay exact)
constexpr int OZ_MAX_KT = 16;        // K tiles per CTA (512 k: the 64-bit sum stays exact)
constexpr int OZ_STAGES = 2;
constexpr int OZ_EPI_WARPS = 8;
constexpr int OZ_THREADS = 64 + 32 * OZ_EPI_WARPS;
constexpr int OZ_COLS = OZ_BN / (OZ_EPI_WARPS / 4);   // columns per epilogue thread
static_assert(OZ_COLS % 8 == 0, "the epilogue works in groups of 8 columns");
constexpr uint32_t OZ_A_TILE = OZ_BM * OZ_BK * 2, OZ_B_TILE = OZ_BN * OZ_BK * 2;
constexpr uint32_t OZ_A_STAGE = OZ_D * OZ_A_TILE, OZ_B_STAGE = OZ_D * OZ_B_TILE;
constexpr size_t OZ_SMEM = 1024 + OZ_STAGES * (size_t)(OZ_A_STAGE + OZ_B_STAGE) + 256;
constexpr int kExpNan = 1 << 20;     // exponent of a row with a NaN or an infinity

// ------------------------------------------------------------- digits

// x 2^(55 - e) rounded to an integer, e = exmax - 1022 (exmax: the largest
// biased exponent of the row, so |x| < 2^e).
__device__ __forceinline__ long long fixed55(double x, int exmax) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7ff);
    unsigned long long mant = b & 0xfffffffffffffull;
    if (ex) mant |= 0x10000000000000ull;
    const int d = exmax - max(ex, 1);          // >= 0
    unsigned long long f;
    if (d <= 2) f = mant << (2 - d);
    else if (d < 58) f = (mant + (1ull << (d - 3))) >> (d - 2);
    else f = 0;
    return (long long)b < 0 ? -(long long)f : (long long)f;
}

// Digit i (0-based) of the biased fixed-point number u, with its weight.
__device__ __forceinline__ float digit_of(unsigned long long u, int i) {
    constexpr float w[OZ_D] = {1.0f, 0x1p-8f, 0x1p-16f, 0x1p-24f, 0x1p-32f, 0x1p-40f, 0x1p-48f};
    const uint32_t v = (uint32_t)(u >> (8 * (OZ_D - 1 - i))) & (i == 0 ? 0x1ffu : 0xffu);
    return (__uint_as_float(0x4b000000u | v) - 8388736.0f) * w[i];   // (2^23 + v) - (2^23 + 128)
}
constexpr unsigned long long kDigitBias = 0x80808080808080ull;

struct OzOperand {
    const double *X; int64_t ld;
    int64_t R, K;              // operand rows and their length
    int mask;                  // MASK_UNIT_LOWER: the strict lower part only (the diagonal is added apart)
    int by_row;                // 0: operand row r is column r of X; 1: row r of X
    __nv_bfloat16 *dst;        // [digit][r][ldk]
    int64_t ldk;
    int *exps;                 // per operand row
    unsigned blocks;           // CTAs working on it
    const int *skip;           // non-null: nothing to do while *skip != 0
    const int *kexp; int ksign;   // entries of index k scaled by 2^(ksign kexp[k]) first
};

// x 2^e, exact unless it leaves the normal range.
__device__ __forceinline__ double mul_pow2(double x, int e) {
    const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
    if (ex == 0 && x == 0.0) return x;
    if (ex == 0x7ff) return x;
    if (ex > 0 && ex + e > 0 && ex + e < 0x7ff && e > -4096 && e < 4096)
        return __hiloint2double(hi + (e << 20), __double2loint(x));
    return scalbn(x, e);
}

__device__ __forceinline__ double oz_load(const OzOperand &o, int64_t r, int64_t k) {
    const int64_t i = o.by_row ? r : k, j = o.by_row ? k : r;
    if (k >= o.K || r >= o.R) return 0.0;
    if (o.mask == MASK_UNIT_LOWER && i <= j) return 0.0;
    if (o.mask == MASK_UPPER && i > j) return 0.0;
    const double x = o.X[i + j * o.ld];
    return o.kexp ? mul_pow2(x, o.ksign * __ldcg(o.kexp + k)) : x;
}

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// n consecutive digits of every weight for the values v (n = 4 or 16).
template <int NV>
__device__ __forceinline__ void store_digits(const OzOperand &o, int64_t r, int64_t k0, const double (&v)[NV], int exmax) {
    unsigned long long u[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) u[q] = (unsigned long long)(fixed55(v[q], exmax) + (long long)kDigitBias);
    const size_t slice = (size_t)o.R * o.ldk;
    __nv_bfloat16 *p = o.dst + (size_t)r * o.ldk + k0;
#pragma unroll
    for (int i = 0; i < OZ_D; ++i) {
        uint32_t w[NV / 2];
#pragma unroll
        for (int q = 0; q < NV / 2; ++q) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(digit_of(u[2 * q], i), digit_of(u[2 * q + 1], i));
            w[q] = *reinterpret_cast<const uint32_t *>(&h);
        }
        if constexpr (NV == 4) {
            *reinterpret_cast<uint2 *>(p + i * slice) = make_uint2(w[0], w[1]);
        } else {
#pragma unroll
            for (int q = 0; q < NV / 8; ++q)
                reinterpret_cast<uint4 *>(p + i * slice)[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
        }
    }
}

// Four consecutive entries of operand row r (a column of X) from k0 on.
__device__ __forceinline__ void load_quad(const OzOperand &o, bool plain, int64_t r, int64_t k0, double (&v)[4]) {
    if (plain && k0 + 4 <= o.K) {
        const double *x = o.X + k0 + r * o.ld;
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = x[q];
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = oz_load(o, r, k0 + q);
    }
}

// Digits of both operands of a product: the first a.blocks CTAs work on A.
// Bound by HBM (8 bytes read, 14 written per entry) and, for few rows, by
// latency, so every entry is read once where registers hold the row between
// the search for its maximum and the split: NT threads keep NQ quads each
// (256 x 8: rows of 8192; 1024 x 4: 16384; what lies beyond is read again).
//   by column: a warp per operand row (K <= 1024) or a CTA per row; a thread
//              takes 4 consecutive k (8-byte stores, a warp 256 bytes).
//   by row:    a CTA takes 32 rows, lane = row, a warp 16 consecutive k (reads
//              are coalesced along the rows, a store is one 32-byte sector).
template <int NT, int NQ>
__global__ void __launch_bounds__(NT) oz_slice_kernel(const OzOperand a, const OzOperand b) {
    __shared__ int red[NT / 32][32];
    constexpr int NW = NT / 32;
    const bool isB = blockIdx.x >= a.blocks;
    const OzOperand &o = isB ? b : a;
    if (o.skip && *(volatile const int *)o.skip) return;
    const int64_t blk = isB ? blockIdx.x - a.blocks : blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int ex = 0;
    if (o.by_row) {
        const int64_t r = blk * 32 + lane;
        double v[16];
        for (int64_t k0 = warp * 16; k0 < o.K; k0 += 16 * NW) {
#pragma unroll
            for (int q = 0; q < 16; ++q) v[q] = oz_load(o, r, k0 + q);
#pragma unroll
            for (int q = 0; q < 16; ++q) ex = max(ex, exp_field(v[q]));
        }
        red[warp][lane] = ex;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < NW; ++w) ex = max(ex, red[w][lane]);
        ex = max(ex, 1);
        if (r >= o.R) return;
        if (warp == 0) o.exps[r] = ex == 0x7ff ? kExpNan : ex - 1022;
        const bool kept = o.K <= 16 * NW;                       // v holds this warp's only 16 k
        for (int64_t k0 = warp * 16; k0 < o.ldk; k0 += 16 * NW) {
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                if (ex == 0x7ff || (kept && k0 >= o.K)) v[q] = 0.0;
                else if (!kept) v[q] = oz_load(o, r, k0 + q);
            }
            store_digits(o, r, k0, v, ex);
        }
        return;
    }
    const bool wide = o.K > 1024;
    const int64_t r = wide ? blk : blk * NW + warp;
    const int t = wide ? (int)threadIdx.x : lane, nt = wide ? NT : 32;
    const bool plain = o.mask == MASK_NONE && !o.kexp;
    double v[NQ][4];
    if (r < o.R) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) load_quad(o, plain, r, (int64_t)(t + q * nt) * 4, v[q]);
#pragma unroll
        for (int q = 0; q < NQ; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) ex = max(ex, exp_field(v[q][i]));
        for (int64_t k0 = (int64_t)(t + NQ * nt) * 4; k0 < o.K; k0 += nt * 4) {
            double x[4];
            load_quad(o, plain, r, k0, x);
#pragma unroll
            for (int i = 0; i < 4; ++i) ex = max(ex, exp_field(x[i]));
        }
    }
    ex = __reduce_max_sync(0xffffffffu, ex);
    if (wide) {
        if (lane == 0) red[0][warp] = ex;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < NW; ++w) ex = max(ex, red[0][w]);
    }
    if (r >= o.R) return;
    ex = max(ex, 1);
    if (t == 0) o.exps[r] = ex == 0x7ff ? kExpNan : ex - 1022;
    if (ex == 0x7ff) {
#pragma unroll
        for (int q = 0; q < NQ; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) v[q][i] = 0.0;
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q)
        if ((int64_t)(t + q * nt) * 4 < o.ldk) store_digits(o, r, (int64_t)(t + q * nt) * 4, v[q], ex);
    for (int64_t k0 = (int64_t)(t + NQ * nt) * 4; k0 < o.ldk; k0 += nt * 4) {
        double x[4];
        load_quad(o, plain, r, k0, x);
        if (ex == 0x7ff)
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = 0.0;
        store_digits(o, r, k0, x, ex);
    }
}

// ------------------------------------------------------------ conversion

// X 2^e rounded to FP64 with integer instructions (an FP64 instruction takes
// a warp 64 cycles here, and a conversion by FP64 adds needs two).
__device__ __forceinline__ double fixed_to_double(long long X, int e) {
    if (X == 0) return 0.0;
    unsigned long long m = (unsigned long long)(X < 0 ? -X : X);
    const int lz = __clzll((long long)m);
    m <<= lz;
    unsigned long long r = (m >> 11) + ((m >> 10) & 1);       // 53 bits, round half up
    const int ex = 1022 + 63 - lz + e;                         // + 1 from the leading bit of r
    if (ex <= 0 || ex >= 0x7fe) {
        const double d = scalbn((double)r, 11 - lz + e);
        return X < 0 ? -d : d;
    }
    r += (unsigned long long)(uint32_t)ex << 52;
    if (X < 0) r |= 0x8000000000000000ull;
    return __longlong_as_double((long long)r);
}

__device__ __forceinline__ double nan_value() { return __longlong_as_double(0x7ff8000000000000ll); }

struct OzParams {
    int M, N, K;
    int ktiles, kt_per;        // K tiles in all and per CTA
    int clipA;                 // op(A) strict lower: 1 K x M stored (k > i), 2 M x K stored (k < i); 0 dense
    const int *ea, *eb;
    long long *partial;        // K split: [z][M x N] column-major
    double *C; int64_t ldc;
    double alpha, beta;
    const double *add; int64_t ldadd; int add_rows;   // unit diagonal of op(A): + alpha * B(i, j), i < add_rows
    const int *skip;           // non-null: nothing to do while *skip != 0
    int *err;
};

// Shared-memory descriptor of a K-major BF16 tile written by TMA with 64-byte
// swizzle: rows of 64 bytes, 8-row atoms 512 bytes apart.
__device__ __forceinline__ uint64_t sw64_desc(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;
    return d;
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&r)[8]) {
    uint32_t v[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 8; ++i) r[i] = __uint_as_float(v[i]);
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// One CTA per 128 x 64 tile and K range, 10 warps: TMA producer (a box brings
// all 7 digits of a 32-k step: 56 KB of A, 28 KB of B, two stages), MMA issuer
// (34 products x 2 instructions per stage), 8 epilogue warps (warp w reads
// TMEM lanes 32 (w % 4) .. + 31 and half of the columns).  Waits are bounded
// as in the mixed-precision kernel.
__global__ void __launch_bounds__(OZ_THREADS, 1)
    oz_mma_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const OzParams p) {
    extern __shared__ uint8_t smem_raw[];
    if (p.skip && *(volatile const int *)p.skip) return;
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sA = smem, *sB = sA + OZ_STAGES * OZ_A_STAGE;
    uint64_t *bars = (uint64_t *)(sB + OZ_STAGES * OZ_B_STAGE);
    uint32_t *tmem_slot = (uint32_t *)(bars + 2 * OZ_STAGES + 2);
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + OZ_STAGES);
    const uint32_t acc_full = smem_u32(bars + 2 * OZ_STAGES), acc_empty = smem_u32(bars + 2 * OZ_STAGES + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * OZ_BM, n0 = blockIdx.y * OZ_BN, z = blockIdx.z;
    int kt0 = z * p.kt_per, kt1 = min(p.ktiles, kt0 + p.kt_per);
    if (p.clipA == 1) kt0 = max(kt0, m0 / OZ_BK);
    else if (p.clipA == 2) kt1 = min(kt1, (m0 + OZ_BM + OZ_BK - 1) / OZ_BK);
    const int total = max(0, kt1 - kt0);
    const int nchunk = (total + OZ_CHUNK - 1) / OZ_CHUNK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < OZ_STAGES; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, OZ_EPI_WARPS);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int issued = 0;
            for (int it = 0; it < total; ++it) {
                const int s = it % OZ_STAGES, r = it / OZ_STAGES;
                if (!mbar_wait(empty0 + 8 * s, (uint32_t)((r & 1) ^ 1), p.err)) break;
                mbar_expect_tx(full0 + 8 * s, OZ_A_STAGE + OZ_B_STAGE);
                tma_load_3d(smem_u32(sA + s * OZ_A_STAGE), &tmA, (kt0 + it) * OZ_BK, m0, 0, full0 + 8 * s);
                tma_load_3d(smem_u32(sB + s * OZ_B_STAGE), &tmB, (kt0 + it) * OZ_BK, n0, 0, full0 + 8 * s);
                issued = it + 1;
            }
            // after an abort, let the loads already issued land before the CTA exits
            if (issued < total)
                for (int it = max(0, issued - OZ_STAGES); it < issued; ++it)
                    mbar_wait(full0 + 8 * (it % OZ_STAGES), (uint32_t)((it / OZ_STAGES) & 1), p.err);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16(OZ_BM, OZ_BN);
            bool ok = true;
            for (int c = 0, it = 0; c < nchunk && ok; ++c) {
                if (c > 0) {
                    ok = mbar_wait(acc_empty, (uint32_t)((c - 1) & 1), p.err);
                    if (!ok) break;
                    tc_fence_after();
                }
                const int end = min(total, it + OZ_CHUNK);
                for (bool first = true; it < end; ++it, first = false) {
                    const int s = it % OZ_STAGES, r = it / OZ_STAGES;
                    ok = mbar_wait(full0 + 8 * s, (uint32_t)(r & 1), p.err);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t ad = sw64_desc(smem_u32(sA + s * OZ_A_STAGE));
                    const uint64_t bd = sw64_desc(smem_u32(sB + s * OZ_B_STAGE));
                    // lowest weight first: i + j = 8 down to 2 (1-based digits)
#pragma unroll
                    for (int w = OZ_TOP - 2; w >= 0; --w) {
                        const uint32_t acc = tmem + (uint32_t)((w < OZ_ACC - 1 ? w : OZ_ACC - 1) * OZ_BN);
                        const int i0 = w < OZ_D ? 0 : w - OZ_D + 1;
#pragma unroll
                        for (int i = i0; i <= w - i0; ++i) {
                            const int j = w - i;
                            const bool fresh = first && i == i0 && (w < OZ_ACC - 1 || w == OZ_TOP - 2);
#pragma unroll
                            for (int kk = 0; kk < OZ_BK / 16; ++kk)
                                mma_bf16(acc, ad + (uint64_t)(i * (OZ_A_TILE >> 4) + 2 * kk),
                                         bd + (uint64_t)(j * (OZ_B_TILE >> 4) + 2 * kk), idesc,
                                         (fresh && kk == 0) ? 0u : 1u);
                        }
                    }
                    mma_commit(empty0 + 8 * s);
                }
                mma_commit(acc_full);
            }
        }
    } else {
        const int q = warp & 3, half = (warp - 2) >> 2;
        const int row = q * 32 + lane, m = m0 + row;
        const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * OZ_COLS);
        long long X[OZ_COLS];
#pragma unroll
        for (int c = 0; c < OZ_COLS; ++c) X[c] = 0;
        bool ok = true;
        for (int ch = 0; ch < nchunk; ++ch) {
            ok = mbar_wait(acc_full, (uint32_t)(ch & 1), p.err);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
#pragma unroll
            for (int g = 0; g < OZ_COLS / 8; ++g) {
                float a[OZ_ACC][8];
#pragma unroll
                for (int s = 0; s < OZ_ACC; ++s) tmem_ld8(tbase + (uint32_t)(s * OZ_BN + g * 8), a[s]);
                tmem_wait_ld();
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    // the weights 2 .. 7 in units of their own; the last rounded to the unit 2^-40
                    const long long hi = ((long long)__float2int_rn(a[0][c]) << 24) +
                                         ((long long)__float2int_rn(a[1][c] * 0x1p8f) << 16) +
                                         ((long long)__float2int_rn(a[2][c] * 0x1p16f) << 8) +
                                         (long long)__float2int_rn(a[3][c] * 0x1p24f);
                    const int lo = __float2int_rn(a[5][c] * 0x1p40f) + __float2int_rn(a[6][c] * 0x1p40f);
                    X[g * 8 + c] += (hi << 16) + ((long long)__float2int_rn(a[4][c] * 0x1p32f) << 8) + (long long)lo;
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acc_empty) : "memory");
        }
        const int nb = n0 + half * OZ_COLS;
        if (ok && m < p.M) {
            if (p.partial) {
                long long *pp = p.partial + (size_t)z * p.M * p.N + m;
#pragma unroll
                for (int c = 0; c < OZ_COLS; ++c)
                    if (nb + c < p.N) pp[(size_t)(nb + c) * p.M] = X[c];
            } else {
                const int ea = p.ea[m];
                const bool sub = p.beta == 1.0 && p.alpha == -1.0;
                double *cp = p.C + m + (int64_t)nb * p.ldc;
                const double *ap = (m < p.add_rows) ? p.add + m + (int64_t)nb * p.ldadd : nullptr;
#pragma unroll
                for (int g = 0; g < OZ_COLS / 8; ++g) {
                    double cv[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        cv[c] = (p.beta != 0.0 && nb + g * 8 + c < p.N) ? cp[(int64_t)(g * 8 + c) * p.ldc] : 0.0;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const int n = nb + g * 8 + c;
                        if (n < p.N) {
                            const int eb = p.eb[n];
                            double d = (ea == kExpNan || eb == kExpNan) ? nan_value()
                                                                        : fixed_to_double(X[g * 8 + c], ea + eb - 54);
                            if (ap) {
                                const double u = ap[(int64_t)(g * 8 + c) * p.ldadd];
                                if (sub) cv[c] -= u;
                                else d += u;
                            }
                            double out;
                            if (sub) out = cv[c] - d;
                            else if (p.beta == 0.0) out = p.alpha == 1.0 ? d : p.alpha * d;
                            else out = fma(p.beta, cv[c], p.alpha * d);
                            cp[(int64_t)(g * 8 + c) * p.ldc] = out;
                        }
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
    }
}

// C = beta C + alpha (2^(ea + eb - 54) sum_z P[z] + unit-diagonal term): the
// sum is exact (high and low halves in 64 bits each), one rounding.
__global__ void __launch_bounds__(kThreads) oz_reduce_kernel(const OzParams p, int S) {
    if (p.skip && *(volatile const int *)p.skip) return;
    const size_t total = (size_t)p.M * p.N;
    for (size_t e = blockIdx.x * (size_t)kThreads + threadIdx.x; e < total; e += (size_t)gridDim.x * kThreads) {
        const int i = (int)(e % (unsigned)p.M), j = (int)(e / (unsigned)p.M);
        long long H = 0;
        unsigned long long L = 0;
        const long long *P = p.partial + e;
#pragma unroll 8
        for (int z = 0; z < S; ++z) {
            const long long v = P[(size_t)z * total];
            H += v >> 32;
            L += (unsigned long long)v & 0xffffffffull;
        }
        const int ea = p.ea[i], eb = p.eb[j];
        double d = (ea == kExpNan || eb == kExpNan)
                       ? nan_value()
                       : mul_pow2(fma((double)H, 4294967296.0, (double)L), ea + eb - 54);
        double *cp = p.C + i + (int64_t)j * p.ldc;
        if (i < p.add_rows) d += p.add[i + (int64_t)j * p.ldadd];
        double out;
        if (p.beta == 0.0) out = p.alpha == 1.0 ? d : p.alpha * d;
        else if (p.beta == 1.0 && p.alpha == -1.0) out = *cp - d;
        else out = fma(p.beta, *cp, p.alpha * d);
        *cp = out;
    }
}

bool oz_map(CUtensorMap *map, const void *base, int64_t rows, int64_t ldk, int box_rows) {
    auto enc = (PFN_cuTensorMapEncodeTiled_v12000)tensor_map_encoder();
    if (!enc) return false;
    cuuint64_t dims[3] = {(cuuint64_t)ldk, (cuuint64_t)rows, (cuuint64_t)OZ_D};
    cuuint64_t strides[2] = {(cuuint64_t)ldk * 2, (cuuint64_t)ldk * (cuuint64_t)rows * 2};
    cuuint32_t box[3] = {(cuuint32_t)OZ_BK, (cuuint32_t)box_rows, (cuuint32_t)OZ_D};
    cuuint32_t estr[3] = {1, 1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

size_t a256(size_t x) { return (x + 255) / 256 * 256; }
int64_t pad_k(int64_t K) { return (K + 15) / 16 * 16; }

// Scratch layout of one product.
struct OzLayout { int64_t ldk; size_t a, b, ea, eb, part, total; };
OzLayout oz_layout(int64_t M, int64_t N, int64_t K, int64_t S) {
    OzLayout L;
    L.ldk = pad_k(K);
    L.a = 0;                       // A first: its place does not depend on N
    L.ea = L.a + a256((size_t)OZ_D * M * L.ldk * 2);
    L.b = L.ea + a256((size_t)M * 4);
    L.eb = L.b + a256((size_t)OZ_D * N * L.ldk * 2);
    L.part = L.eb + a256((size_t)N * 4);
    L.total = L.part + (S > 1 ? a256((size_t)S * M * N * 8) : 0);
    return L;
}

// Split of a product: K tiles per CTA, splits and the estimated time (us).
// Per-CTA cycles are those of the kernel's parts: about 2900 per 32-k step (68
// MMAs of 128 x 64 x 16), 3500 per drain, 9000 for an FP64 epilogue.
struct OzSplit { int kt_per, S; double us; };
OzSplit oz_split(int64_t M, int64_t N, int64_t K, int num_sms, size_t part_cap_elems) {
    const int64_t tiles = ((M + OZ_BM - 1) / OZ_BM) * ((N + OZ_BN - 1) / OZ_BN);
    const int kt = (int)((K + OZ_BK - 1) / OZ_BK);
    OzSplit best{0, 0, 1e30};
    for (int per = 1; per <= std::min(kt, OZ_MAX_KT); ++per) {
        const int S = (kt + per - 1) / per;
        if (S > 1 && ((size_t)S * M * N > part_cap_elems || S > 65535)) continue;
        const double cta = 3000.0 + 2900.0 * per + 3500.0 * ((per + OZ_CHUNK - 1) / OZ_CHUNK) + (S == 1 ? 9000.0 : 2500.0);
        double clk = std::ceil((double)tiles * S / num_sms) * cta;
        if (S > 1) clk += 6000.0 + (double)S * M * N * 16.0 / 2500.0;
        if (clk / 1900.0 < best.us) best = {per, S, clk / 1900.0};
    }
    return best;
}

}  // namespace

// Digits of op(A) and of up to N columns of B, and the partials of a split
// that gives every CTA at most 512 k and a small output two CTAs per SM.
size_t oz_gemm_scratch_bytes(int64_t M, int64_t N, int64_t K) {
    const int64_t tiles = std::max<int64_t>(1, ((M + OZ_BM - 1) / OZ_BM) * ((N + OZ_BN - 1) / OZ_BN));
    const int64_t S = std::max((K + OZ_MAX_KT * OZ_BK - 1) / (OZ_MAX_KT * OZ_BK),
                               std::min<int64_t>({(K + OZ_BK - 1) / OZ_BK, (304 + tiles - 1) / tiles, 64}));
    return oz_layout(M, N, K, S).total;
}

// How C = alpha op(A) B + beta C is done here, if at all: the columns of B in
// chunks whose digits fit the scratch, where the estimated time beats the
// FMA kernel's (1.15 TFLOP/s on large products).
struct OzPlan { int64_t nc; OzSplit split; };
static bool oz_plan(const GemmOp &op, const OzScratch &sc, int num_sms, OzPlan *plan, double *gain_us) {
    if (!sc.base || op.M < 8 || op.N < 8 || op.K < 8) return false;
    if (op.M > (1 << 30) || op.N > (1 << 30) || op.K > (1 << 30)) return false;
    if (op.maskB == MASK_UNIT_LOWER) return false;
    int64_t nc = std::min<int64_t>(op.N, (int64_t)OZ_BN * 65535);
    const size_t room = sc.bytes - sc.bytes / 8;                 // an eighth for partials
    if (oz_layout(op.M, nc, op.K, 1).total > room) {
        const size_t fixed = oz_layout(op.M, 0, op.K, 1).total + 1024, col = (size_t)OZ_D * pad_k(op.K) * 2 + 4;
        const int64_t most = fixed < room ? (int64_t)((room - fixed) / col) / OZ_BN * OZ_BN : 0;
        if (most >= OZ_BN) {                                     // equal chunks of whole tiles
            const int64_t chunks = (nc + most - 1) / most;
            nc = ((nc + chunks - 1) / chunks + OZ_BN - 1) / OZ_BN * OZ_BN;
        }
    }
    const OzLayout L = oz_layout(op.M, nc, op.K, 1);
    if (L.total > sc.bytes) return false;
    if ((size_t)op.M * nc >= ((size_t)1 << 32)) return false;
    plan->nc = nc;
    plan->split = oz_split(op.M, nc, op.K, num_sms, (sc.bytes - L.total) / 8);
    if (plan->split.S == 0) return false;
    const double chunks = std::ceil((double)op.N / nc);
    const double slice_us = 22.0 * ((double)op.M + nc) * op.K / 4.0e6;
    *gain_us = gemm_algorithmic_flops(op) / 1.15e6 - chunks * (plan->split.us + slice_us + 10.0);
    return true;
}

bool oz_gemm_wanted(const GemmOp &op, const OzScratch &sc, int num_sms) {
    OzPlan p;
    double gain = 0.0;
    return sc.base && gemm_algorithmic_flops(op) > 1.4e7 && oz_plan(op, sc, num_sms, &p, &gain) && gain > 0.0;
}

// One chunk of columns; slice_a: op(A)'s digits are not in the scratch yet.
static gbqr_status oz_chunk(const Exec &ex, const GemmOp &op, const OzScratch &sc, bool slice_a) {
    OzLayout L = oz_layout(op.M, op.N, op.K, 1);
    if (L.total > sc.bytes) return GBQR_ENOMEM;
    const OzSplit sp = oz_split(op.M, op.N, op.K, ex.num_sms, (sc.bytes - L.total) / 8);
    if (sp.S == 0) return GBQR_ENOMEM;
    char *base = (char *)sc.base;
    OzOperand a{}, b{};
    a.X = op.A; a.ld = op.lda; a.R = op.M; a.K = op.K; a.mask = op.maskA; a.by_row = op.ta ? 0 : 1;
    a.dst = (__nv_bfloat16 *)(base + L.a); a.ldk = L.ldk; a.exps = (int *)(base + L.ea);
    b.X = op.B; b.ld = op.ldb; b.R = op.N; b.K = op.K; b.mask = op.maskB; b.by_row = 0;
    b.dst = (__nv_bfloat16 *)(base + L.b); b.ldk = L.ldk; b.exps = (int *)(base + L.eb);
    const bool tall = op.K > 8192;                               // 1024 threads per row, else 256
    const int warps = tall ? 32 : 8;
    auto blocks = [&](const OzOperand &o) {
        return (unsigned)(o.by_row ? (o.R + 31) / 32 : (o.K > 1024 ? o.R : (o.R + warps - 1) / warps));
    };
    a.blocks = slice_a ? blocks(a) : 0;
    b.blocks = blocks(b);
    if (op.ta && op.A == op.B && op.lda == op.ldb && op.M == op.N && op.maskA == op.maskB) {
        b = a;                         // X^T X: one set of digits
        b.blocks = 0;
    }
    a.skip = b.skip = op.skip;
    a.kexp = b.kexp = op.kexp;
    a.ksign = -1;
    b.ksign = 1;
    trace_begin(ex, FAM_OTHER);
    const unsigned nblk = a.blocks + b.blocks;
    if (nblk && tall) oz_slice_kernel<1024, 4><<<nblk, 1024, 0, ex.stream>>>(a, b);
    else if (nblk) oz_slice_kernel<kThreads, 8><<<nblk, kThreads, 0, ex.stream>>>(a, b);
    TRY_ST(trace_end(ex, FAM_OTHER, 0.0, 22.0 * ((double)op.M + op.N) * op.K));

    OzParams p{};
    p.M = (int)op.M; p.N = (int)op.N; p.K = (int)op.K;
    p.ktiles = (int)((op.K + OZ_BK - 1) / OZ_BK);
    p.kt_per = sp.kt_per;
    // a strict lower op(A) is zero for k <= i (stored K x M) or k >= i (stored M x K)
    p.clipA = op.maskA == MASK_UNIT_LOWER ? (op.ta ? 1 : 2) : 0;
    p.ea = a.exps; p.eb = b.exps;
    p.partial = sp.S > 1 ? (long long *)(base + L.part) : nullptr;
    p.C = op.C; p.ldc = op.ldc; p.alpha = op.alpha; p.beta = op.beta;
    p.add = op.B; p.ldadd = op.ldb;
    p.add_rows = op.maskA == MASK_UNIT_LOWER ? (int)std::min(op.M, op.K) : 0;
    p.skip = op.skip;
    p.err = sc.err;
    CUtensorMap mA, mB;
    if (!oz_map(&mA, a.dst, op.M, L.ldk, OZ_BM) || !oz_map(&mB, b.dst, op.N, L.ldk, OZ_BN)) return GBQR_ECUDA;
    static std::atomic<bool> attr[64];
    const bool cached = ex.device >= 0 && ex.device < 64;
    if (!cached || !attr[ex.device].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(oz_mma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_SMEM) != cudaSuccess)
            return GBQR_ECUDA;
        if (cached) attr[ex.device].store(true, std::memory_order_release);
    }
    const dim3 grid((unsigned)((op.M + OZ_BM - 1) / OZ_BM), (unsigned)((op.N + OZ_BN - 1) / OZ_BN), (unsigned)sp.S);
    trace_begin(ex, FAM_TC_GEMM);
    oz_mma_kernel<<<grid, OZ_THREADS, OZ_SMEM, ex.stream>>>(mA, mB, p);
    TRY_ST(trace_end(ex, FAM_TC_GEMM, 2.0 * 34.0 * (double)op.M * op.N * op.K, 14.0 * ((double)op.M + op.N) * op.K));
    if (sp.S > 1) {
        trace_begin(ex, FAM_OTHER);
        const size_t total = (size_t)op.M * op.N;
        const unsigned g = (unsigned)std::min<size_t>((total + kThreads - 1) / kThreads, (size_t)ex.num_sms * 16);
        oz_reduce_kernel<<<g, kThreads, 0, ex.stream>>>(p, sp.S);
        TRY_ST(trace_end(ex, FAM_OTHER, (double)sp.S * total, 8.0 * sp.S * total + 16.0 * total));
    }
    return GBQR_OK;
}

gbqr_status oz_gemm(const Exec &ex, const GemmOp &op, const OzScratch &sc) {
    OzPlan pl;
    double gain = 0.0;
    if (!oz_plan(op, sc, ex.num_sms, &pl, &gain)) return GBQR_ENOMEM;
    for (int64_t j = 0; j < op.N; j += pl.nc) {
        GemmOp c = op;
        c.N = std::min(pl.nc, op.N - j);
        c.B = op.B + j * op.ldb;
        c.C = op.C + j * op.ldc;
        TRY_ST(oz_chunk(ex, c, sc, j == 0));
    }
    return GBQR_OK;
}

}  // namespace gbqr
