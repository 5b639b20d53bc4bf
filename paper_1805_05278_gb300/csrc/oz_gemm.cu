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
// most 2^14 times its weight, so an FP32 accumulator of the tensor cores holds
// a sum of products of equal weight exactly while it stays below 2^24 of them.
// The weights i + j = 2 ... 7 (1 to 6 products per k) have an accumulator
// each, i + j = 8 and 9 share one; i + j >= 10 (below 2^-62 of the row and
// column maxima) is left out.  Every 256 k the accumulators are drained into a
// 64-bit integer per output (unit 2^-40 of a leading digit product), and the
// integer is rounded to FP64 once.  Sums over more than 512 k are integer
// partials, which add without rounding in any order.
//
// Error.  Entries within a factor 4 of the row (column) maximum are exact, the
// others lose what lies below 2^-56 of it.  A drain's 256 k are 1280 products
// of weight 6 and 1536 of weight 7: these sums leave the exact range only where
// the products of their digits average more than 114^2 or 104^2 of 128^2, all
// of one sign; the steps past 2^24 then truncate, at worst (every digit 127)
// 32 units of 2^-32 and 64 of 2^-40, 2^-48.6 of sum |a_ik b_kj| (the FMA
// kernel's bound over 256 k is 2^-45).  The shared accumulator truncates at
// 2^-59 of it.  Where none of this happens a result does not depend on the
// split.  Measured on whole factorizations, backward error and orthogonality
// are at or below the FMA kernel's, which rounds at every k (graded 8192^2:
// backward error 6.6e-16, FMA 8.4e-16; Gaussian 4096^2: 1.8e-15, 2.3e-15).
// Sharing one accumulator among i + j = 6, 7, 8 instead cost a digit and a
// half: the tensor cores' accumulation truncates, and its bias grows with K.
//
// Kernels of one product:
//   oz_slice_kernel   digits of the operands (HBM: 8 B read, 14 written per
//                     entry), one launch
//   oz_mma_kernel     bulk copies -> shared memory -> tcgen05.mma -> TMEM ->
//                     C, or integer partials where K is split
//   oz_reduce_kernel  sums the partials and rounds (only where K is split), or
//                     oz_requant_kernel, which writes them as the digits of
//                     the next product's operand
//
// FP32 (the FP32 factorizations) is the same with four digits (31 bits), ten
// digit products and an accumulator for each of the weights 2 to 5.
//
// Digits lie in memory as the shared-memory images of their tiles: 128 (the M
// side) or 64 rows x 32 k of every digit, rows of 64 bytes with the 64-byte
// swizzle the MMA descriptors name, so a stage is filled by one bulk copy an
// operand and a product needs no tensor map.
//
// Measured with the FMA kernel against this one, all else as it was then (TSQR
// panels): graded 8192^2 687 -> 157 ms, 32768 x 2048 256 -> 65 ms; the thin Q
// of 16001 x 1000 31.3 -> 3.2 ms.
#include "oz.cuh"
#include "tc_ptx.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cmath>

namespace gbqr {
namespace {

constexpr int OZ_BM = 128;
constexpr int OZ_BN = 64;
constexpr int OZ_BK = 32;            // one 64-byte row of BF16
constexpr uint32_t OZ_PIECE = 4096;  // bytes per bulk copy
constexpr int OZ_CHUNK = 8;          // K tiles per drain (256 k; see the error above)
constexpr int OZ_EPI_WARPS = 16;
constexpr int OZ_THREADS = 64 + 32 * OZ_EPI_WARPS;
constexpr int OZ_COLS = OZ_BN / (OZ_EPI_WARPS / 4);   // columns per epilogue thread
constexpr int kExpNan = 1 << 20;     // exponent of a row with a NaN or an infinity
constexpr uint32_t OZ_A_TILE = OZ_BM * OZ_BK * 2, OZ_B_TILE = OZ_BN * OZ_BK * 2;   // one digit
static_assert(OZ_COLS <= 32 && OZ_COLS % 8 == 0, "a lane per column's exponent, groups of 8 columns");
static_assert(OZ_BM == kOzTileA && OZ_BN == kOzTileB, "digit tiles");

// Digits, the largest i + j of the digit products taken, accumulators (one per
// weight from 2 on, the last shared by the rest: 7 x 64 of TMEM's 512
// columns), the unit 2^-UNIT of the integer sums and the K tiles per CTA that
// keep them in 64 bits.
template <class Real> struct OzTraits;
template <> struct OzTraits<double> {
    static constexpr int D = 7, TOP = 9, ACC = 7, UNIT = 40, STAGES = 2, MAX_KT = 16;
};
template <> struct OzTraits<float> {
    static constexpr int D = 4, TOP = 5, ACC = 4, UNIT = 24, STAGES = 4, MAX_KT = 64;
};
constexpr int kD64 = OzTraits<double>::D, kD32 = OzTraits<float>::D;
template <class Real> constexpr uint32_t oz_stage_bytes() { return OzTraits<Real>::D * (OZ_A_TILE + OZ_B_TILE); }
template <class Real> constexpr size_t oz_smem() { return 1024 + OzTraits<Real>::STAGES * (size_t)oz_stage_bytes<Real>() + 256; }
template <class Real> constexpr int oz_products() {
    int n = 0;
    for (int i = 1; i <= OzTraits<Real>::D; ++i)
        for (int j = 1; j <= OzTraits<Real>::D; ++j) n += i + j <= OzTraits<Real>::TOP;
    return n;
}
static_assert(OzTraits<double>::MAX_KT == oz_max_ktiles<double>() && OzTraits<float>::MAX_KT == oz_max_ktiles<float>(), "item sizes");
static_assert(kD64 == kOzDigits64 && kD32 == kOzDigits32, "digits");
static_assert(oz_products<double>() == 34 && oz_products<float>() == 10, "digit products");

// ------------------------------------------------------------- digits

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ int exp_field(float x) { return (__float_as_int(x) >> 23) & 0xff; }
template <class Real> struct ExpOf;
template <> struct ExpOf<double> { static constexpr int INF = 0x7ff, BIAS = 1022; };
template <> struct ExpOf<float> { static constexpr int INF = 0xff, BIAS = 126; };

// x 2^(8 D - 1 - e) rounded to an integer, e = exmax - BIAS (exmax: the
// largest biased exponent of the row, so |x| < 2^e).
template <int D>
__device__ __forceinline__ long long fixed_of(double x, int exmax) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7ff);
    unsigned long long mant = b & 0xfffffffffffffull;
    if (ex) mant |= 0x10000000000000ull;
    const int d = exmax - max(ex, 1);          // >= 0
    unsigned long long f;
    if (d <= 2) f = mant << (2 - d);
    else if (d < 58) f = (mant + (1ull << (d - 3))) >> (d - 2);
    else f = 0;
    if (D == kD32) f = (f + (1ull << 23)) >> 24;   // 31 bits
    return (long long)b < 0 ? -(long long)f : (long long)f;
}
template <int D>
__device__ __forceinline__ long long fixed_of(float x, int exmax) {
    const uint32_t b = (uint32_t)__float_as_int(x);
    const int ex = (int)((b >> 23) & 0xff);
    uint32_t mant = b & 0x7fffffu;
    if (ex) mant |= 0x800000u;
    const int d = exmax - max(ex, 1);
    uint32_t f;
    if (d <= 7) f = mant << (7 - d);
    else if (d < 33) f = (mant + (1u << (d - 8))) >> (d - 7);
    else f = 0;
    return (int)b < 0 ? -(long long)f : (long long)f;
}

// Digit i (0-based) of the biased fixed-point number u, with its weight.
template <int D>
__device__ __forceinline__ float digit_of(unsigned long long u, int i) {
    constexpr float w[7] = {1.0f, 0x1p-8f, 0x1p-16f, 0x1p-24f, 0x1p-32f, 0x1p-40f, 0x1p-48f};
    const uint32_t v = (uint32_t)(u >> (8 * (D - 1 - i))) & (i == 0 ? 0x1ffu : 0xffu);
    return (__uint_as_float(0x4b000000u | v) - 8388736.0f) * w[i];   // (2^23 + v) - (2^23 + 128)
}
template <int D> constexpr unsigned long long digit_bias() {
    unsigned long long b = 0;
    for (int i = 0; i < D; ++i) b = (b << 8) | 0x80;
    return b;
}

// x 2^e, exact unless it leaves the normal range.
__device__ __forceinline__ double mul_pow2(double x, int e) {
    const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff;
    if (ex == 0 && x == 0.0) return x;
    if (ex == 0x7ff) return x;
    if (ex > 0 && ex + e > 0 && ex + e < 0x7ff && e > -4096 && e < 4096)
        return __hiloint2double(hi + (e << 20), __double2loint(x));
    return scalbn(x, e);
}
__device__ __forceinline__ float mul_pow2(float x, int e) {
    const int b = __float_as_int(x), ex = (b >> 23) & 0xff;
    if (ex == 0xff || x == 0.0f) return x;
    if (ex > 0 && ex + e > 0 && ex + e < 0xff && e > -512 && e < 512) return __int_as_float(b + (e << 23));
    return scalbnf(x, e);
}

// Entry k of operand row r.
template <class Real>
__device__ __forceinline__ Real oz_load(const OzOperand<Real> &o, int64_t r, int64_t k) {
    const int64_t i = o.by_row ? r : k, j = o.by_row ? k : r;
    if (k >= o.K || r >= o.R) return Real(0);
    if (o.mask == MASK_UNIT_LOWER && i <= j) return i == j && o.unit ? Real(1) : Real(0);
    if (o.mask == MASK_UPPER && i > j) return Real(0);
    const Real x = o.X[i + j * o.ld];
    return o.kexp ? mul_pow2(x, o.ksign * o.kexp[k]) : x;
}

// Digits of the NV = 4 or 8 consecutive entries v of operand row r from k0.
template <int D, class Real, int NV>
__device__ __forceinline__ void store_digits(uint8_t *dst, int KT, int rt, int64_t r, int64_t k0, const Real (&v)[NV],
                                             int exmax) {
    unsigned long long u[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) u[q] = (unsigned long long)(fixed_of<D>(v[q], exmax) + (long long)digit_bias<D>());
    const int rr = (int)(r & (rt - 1)), swz = (rr >> 1) & 3;          // rt: rows per tile, 64 or 128
    const uint32_t dig = (uint32_t)rt * 64;
    uint8_t *p = dst + ((size_t)(r >> (rt == OZ_BM ? 7 : 6)) * KT + (size_t)(k0 >> 5)) * (D * dig) + rr * 64;
    const int ch = (int)(k0 >> 3) & 3;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        uint32_t w[NV / 2];
#pragma unroll
        for (int q = 0; q < NV / 2; ++q) {
            const __nv_bfloat162 h = __floats2bfloat162_rn(digit_of<D>(u[2 * q], i), digit_of<D>(u[2 * q + 1], i));
            w[q] = *reinterpret_cast<const uint32_t *>(&h);
        }
        if constexpr (NV == 4) {
            *reinterpret_cast<uint2 *>(p + i * dig + ((ch ^ swz) << 4) + (k0 & 4) * 2) = make_uint2(w[0], w[1]);
        } else {
#pragma unroll
            for (int q = 0; q < NV / 8; ++q)
                *reinterpret_cast<uint4 *>(p + i * dig + (((ch + q) ^ swz) << 4)) =
                    make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
        }
    }
}

// Four consecutive entries of operand row r (a column of X) from k0 on.
template <class Real>
__device__ __forceinline__ void load_quad(const OzOperand<Real> &o, bool plain, int64_t r, int64_t k0, Real (&v)[4]) {
    if (plain && k0 + 4 <= o.K) {
        const Real *x = o.X + k0 + r * o.ld;
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = x[q];
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = oz_load(o, r, k0 + q);
    }
}

template <class Real>
__device__ __forceinline__ void store_exp(const OzOperand<Real> &o, int64_t r, int ex) {
    o.exps[r] = ex == ExpOf<Real>::INF ? kExpNan : ex - ExpOf<Real>::BIAS;
}

// Digits of up to kOzOps operands (or of a list of them): operand i works on
// CTAs [first[i], first[i + 1]).  Bound by HBM (8 bytes read, 14 written per
// entry) and, for few rows, by latency, so every entry is read once where
// registers hold the row between the search for its maximum and the split:
// NT threads keep NQ quads each (256 x 8: rows of 8192; 512 x 8: 16384; what
// lies beyond is read again).
//   by column: a warp per operand row (K <= 1024) or a CTA per row; a thread
//              takes 4 consecutive k (8-byte stores, 64 bytes a row tile).
//   by row:    eight warps take 32 rows, lane = row, a warp 16 consecutive k
//              (reads are coalesced along the rows, stores are 16 bytes).
template <class Real, int D, int NT, int NQ>
__global__ void __launch_bounds__(NT, 512 / NT) oz_slice_kernel(const __grid_constant__ OzSliceArgs<Real> args) {
    __shared__ int red[NT / 32][32];
    constexpr int NW = NT / 32, INF = ExpOf<Real>::INF;
    int which = 0;
    if (args.list) {
        int lo = 0, hi = args.n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(&args.list[mid].first) <= blockIdx.x) lo = mid;
            else hi = mid - 1;
        }
        which = lo;
    } else {
        while (which + 1 < args.n && blockIdx.x >= args.op[which + 1].first) ++which;
    }
    const OzOperand<Real> o = args.list ? args.list[which] : args.op[which];
    if (o.skip && *(volatile const int *)o.skip) return;
    const int64_t blk = blockIdx.x - o.first;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t kpad = (int64_t)o.KT * OZ_BK;
    int ex = 0;
    if (o.by_row) {
        const int sub = warp >> 3, w8 = warp & 7;
        const int64_t r0 = blk * (4 * NW) + sub * 32, r = r0 + lane;
        // rows that no mask touches (a V basis below its triangle) are read directly
        const bool direct = o.mask == MASK_NONE || (o.mask == MASK_UNIT_LOWER && r0 >= o.K);
        auto load16 = [&](int64_t k0, Real (&v)[16]) {
            if (direct && k0 + 16 <= o.K) {
                const Real *x = o.X + r + k0 * o.ld;
#pragma unroll
                for (int q = 0; q < 16; ++q) v[q] = r < o.R ? x[q * o.ld] : Real(0);
                if (o.kexp) {
                    const int ke = o.ksign * o.kexp[k0 + (lane & 15)];
#pragma unroll
                    for (int q = 0; q < 16; ++q) v[q] = mul_pow2(v[q], __shfl_sync(0xffffffffu, ke, q));
                }
            } else {
#pragma unroll
                for (int q = 0; q < 16; ++q) v[q] = oz_load(o, r, k0 + q);
            }
        };
        Real v[16];
        for (int64_t k0 = w8 * 16; k0 < o.K; k0 += 128) {
            load16(k0, v);
#pragma unroll
            for (int q = 0; q < 16; ++q) ex = max(ex, exp_field(v[q]));
        }
        red[warp][lane] = ex;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < 8; ++w) ex = max(ex, red[sub * 8 + w][lane]);
        ex = max(ex, 1);
        if (w8 == 0 && r < o.R) store_exp(o, r, ex);
        const bool kept = o.K <= 128;                           // v holds this warp's only 16 k
        for (int64_t k0 = w8 * 16; k0 < kpad; k0 += 128) {
            if (!kept) load16(k0, v);
            if (ex == INF || (kept && k0 >= o.K)) {
#pragma unroll
                for (int q = 0; q < 16; ++q) v[q] = Real(0);
            }
            if (r < o.R) {
                Real h[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) h[q] = v[q];
                store_digits<D>(o.dst, o.KT, o.rt, r, k0, h, ex);
#pragma unroll
                for (int q = 0; q < 8; ++q) h[q] = v[8 + q];
                store_digits<D>(o.dst, o.KT, o.rt, r, k0 + 8, h, ex);
            }
        }
        return;
    }
    const bool wide = o.K > 1024;
    const int64_t r = wide ? blk : blk * NW + warp;
    const int t = wide ? (int)threadIdx.x : lane, nt = wide ? NT : 32;
    const bool plain = o.mask == MASK_NONE && !o.kexp;
    Real v[NQ][4];
    if (r < o.R) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) load_quad(o, plain, r, (int64_t)(t + q * nt) * 4, v[q]);
#pragma unroll
        for (int q = 0; q < NQ; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) ex = max(ex, exp_field(v[q][i]));
        for (int64_t k0 = (int64_t)(t + NQ * nt) * 4; k0 < o.K; k0 += nt * 4) {
            Real x[4];
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
    if (t == 0) store_exp(o, r, ex);
    if (ex == INF) {
#pragma unroll
        for (int q = 0; q < NQ; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) v[q][i] = Real(0);
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q)
        if ((int64_t)(t + q * nt) * 4 < kpad) store_digits<D>(o.dst, o.KT, o.rt, r, (int64_t)(t + q * nt) * 4, v[q], ex);
    for (int64_t k0 = (int64_t)(t + NQ * nt) * 4; k0 < kpad; k0 += nt * 4) {
        Real x[4];
        load_quad(o, plain, r, k0, x);
        if (ex == INF)
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = Real(0);
        store_digits<D>(o.dst, o.KT, o.rt, r, k0, x, ex);
    }
}

// ------------------------------------------------------------ conversion

// X 2^e, X rounded to Real once.  To FP64 by integer instructions alone: an
// FP64 instruction takes a warp 64 cycles here, and the conversion of a 64-bit
// integer is several of them (it took a tile's epilogue 20 us).  e comes from
// exponents of operand rows; outside the everyday range, and for rows with a
// NaN or an infinity (exponent kExpNan), scalbn.
__device__ __noinline__ double scaled_far(long long X, int e) {
    return e > kExpNan / 2 ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(__ll2double_rn(X), e);
}
__device__ __forceinline__ double scaled(long long X, int e, double) {
    if ((unsigned)(e + 900) > 1800u) return scaled_far(X, e);
    const int sign = (int)(X >> 63);
    const unsigned long long m = (unsigned long long)((X ^ (long long)sign) - (long long)sign);
    const uint32_t hi = (uint32_t)(m >> 32), lo = (uint32_t)m;
    const bool small = hi == 0;
    const int lz = __clz(small ? lo : hi);                     // 32 if X == 0
    const uint32_t th = __funnelshift_l(small ? 0u : lo, small ? lo : hi, lz);   // leading one at bit 31
    const uint32_t tl = small ? 0u : lo << lz;
    unsigned long long r = ((unsigned long long)(th >> 11) << 32) | __funnelshift_r(tl, th, 11);
    r += (tl >> 10) & 1u;                                      // 53 bits, round half up
    // biased exponent, less the one that the leading bit of r adds
    const uint32_t ex = (uint32_t)(1022 + (small ? 31 : 63) - lz + e) << 20;
    const uint32_t rh = m == 0 ? 0u : ((uint32_t)(r >> 32) + ex) | ((uint32_t)sign & 0x80000000u);
    return __hiloint2double((int)rh, (int)(uint32_t)r);
}
__device__ __forceinline__ float scaled(long long X, int e, float) {
    const float f = __ll2float_rn(X);
    if ((unsigned)(e + 60) > 120u) return (float)scaled_far(X, e);
    return __int_as_float(__float_as_int(f) + (X == 0 ? 0 : e << 23));
}

template <class Real> __device__ __forceinline__ Real nan_value();
template <> __device__ __forceinline__ double nan_value<double>() { return __longlong_as_double(0x7ff8000000000000ll); }
template <> __device__ __forceinline__ float nan_value<float>() { return __int_as_float(0x7fc00000); }

// Shared-memory descriptor of a K-major BF16 tile with 64-byte swizzle: rows
// of 64 bytes, 8-row atoms 512 bytes apart.
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

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(mbar)
                 : "memory");
}

__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}

// The accumulators of one output as an integer in units of 2^-UNIT: weight i
// (0-based) counts 2^-8i; FP64's last two share a[6], rounded to 2^-40.
template <int ACC>
__device__ __forceinline__ long long collect(const float (&a)[ACC]) {
    // the two leading ones fit 32 bits together: K = 256 gives 2^22 and 2^23
    const int top = __float2int_rn(a[0]) * 256 + __float2int_rn(a[1] * 0x1p8f);
    const int r2 = __float2int_rn(a[2] * 0x1p16f), r3 = __float2int_rn(a[3] * 0x1p24f);
    if constexpr (ACC == 7) {
        long long x = (long long)((unsigned long long)(uint32_t)top << 32);
        x = mad_wide(r2, 1 << 24, x);
        x = mad_wide(r3, 1 << 16, x);
        x = mad_wide(__float2int_rn(a[4] * 0x1p32f), 1 << 8, x);
        return x + (long long)(__float2int_rn(a[5] * 0x1p40f) + __float2int_rn(a[6] * 0x1p40f));
    } else {
        return mad_wide(top, 1 << 16, mad_wide(r2, 1 << 8, (long long)r3));
    }
}

// One work item: a 128 x 64 tile of a problem's output and a K range.
struct OzItem { int prob, m0, n0, z, kt0, kt1; };

template <class Real>
__device__ __forceinline__ OzItem oz_item(const OzMmaArgs<Real> &args, int item, OzProblem<Real> &p) {
    OzItem t;
    int which = 0;
    if (args.list) {
        int lo = 0, hi = args.n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(&args.list[mid].first) <= item) lo = mid;
            else hi = mid - 1;
        }
        which = lo;
        p = args.list[which];
    } else {
        while (which + 1 < args.n && item >= args.prob[which + 1].first) ++which;
        p = args.prob[which];
    }
    t.prob = which;
    int e = item - p.first;
    const int tm = (p.M + OZ_BM - 1) / OZ_BM, tn = (p.N + OZ_BN - 1) / OZ_BN;
    t.m0 = (e % tm) * OZ_BM;
    e /= tm;
    t.n0 = (e % tn) * OZ_BN;
    t.z = e / tn;
    t.kt0 = t.z * p.kt_per;
    t.kt1 = min(p.KT, t.kt0 + p.kt_per);
    if (p.clip == 1) t.kt0 = max(t.kt0, t.m0 / OZ_BK);
    else if (p.clip == 2) t.kt1 = min(t.kt1, (t.m0 + OZ_BM + OZ_BK - 1) / OZ_BK);
    if (p.clipB == 2) t.kt1 = min(t.kt1, (t.n0 + OZ_BN + OZ_BK - 1) / OZ_BK);
    if (p.skip && *(volatile const int *)p.skip) t.kt1 = -1;        // nothing at all
    return t;
}

// 18 warps per CTA: bulk-copy producer (per 32-k step all digits of a tile of
// A, 56 KB in FP64, and of one of B, 28 KB), MMA issuer (two instructions
// per digit product and stage), 16 epilogue warps (warp w reads TMEM lanes 32
// (w % 4) .. + 31 and a quarter of the columns; with 8 warps the epilogue, a
// chain of dependent integer instructions an output, took 48000 cycles an
// item where the MMAs take 13000).  A CTA takes items blockIdx.x,
// + gridDim.x, ...: once an item's accumulators are in the epilogue's
// registers, the MMAs of the next one run while C is updated.  Waits are
// bounded as in the mixed-precision kernel.
template <class Real>
__global__ void __launch_bounds__(OZ_THREADS, 1) oz_mma_kernel(const __grid_constant__ OzMmaArgs<Real> args) {
    using Tr = OzTraits<Real>;
    constexpr int D = Tr::D, STAGES = Tr::STAGES;
    constexpr uint32_t A_STAGE = D * OZ_A_TILE, B_STAGE = D * OZ_B_TILE;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sA = smem, *sB = sA + STAGES * A_STAGE;
    uint64_t *bars = (uint64_t *)(sB + STAGES * B_STAGE);
    uint32_t *tmem_slot = (uint32_t *)(bars + 2 * STAGES + 2);
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES);
    const uint32_t acc_full = smem_u32(bars + 2 * STAGES), acc_empty = smem_u32(bars + 2 * STAGES + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(acc_full, 1);
        mbar_init(acc_empty, OZ_EPI_WARPS);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    constexpr uint32_t TCOLS = Tr::ACC * OZ_BN <= 256 ? 256 : 512;
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < args.items && ok; item += gridDim.x) {
                OzProblem<Real> p;
                const OzItem t = oz_item(args, item, p);
                // A in tiles of 128 rows; B in tiles of 64, or (X^T X) half a tile of 128
                const uint8_t *a = p.a + (size_t)(t.m0 / OZ_BM) * p.KT * A_STAGE;
                const uint8_t *b = p.b128 ? p.b + (size_t)(t.n0 / OZ_BM) * p.KT * A_STAGE + (t.n0 & OZ_BN ? OZ_B_TILE : 0)
                                          : p.b + (size_t)(t.n0 / OZ_BN) * p.KT * B_STAGE;
                for (int kt = t.kt0; kt < t.kt1; ++kt, ++it) {
                    const int s = it % STAGES, r = it / STAGES;
                    ok = mbar_wait(empty0 + 8 * s, (uint32_t)((r & 1) ^ 1), args.err);
                    if (!ok) break;
                    const uint32_t fb = full0 + 8 * s, db = smem_u32(sB + s * B_STAGE);
                    mbar_expect_tx(fb, A_STAGE + B_STAGE);
#pragma unroll
                    for (uint32_t o = 0; o < A_STAGE; o += OZ_PIECE)
                        bulk_load(smem_u32(sA + s * A_STAGE) + o, a + (size_t)kt * A_STAGE + o, OZ_PIECE, fb);
                    if (p.b128) {
#pragma unroll
                        for (int i = 0; i < D; ++i)
                            bulk_load(db + i * OZ_B_TILE, b + (size_t)kt * A_STAGE + i * OZ_A_TILE, OZ_B_TILE, fb);
                    } else {
#pragma unroll
                        for (uint32_t o = 0; o < B_STAGE; o += OZ_PIECE)
                            bulk_load(db + o, b + (size_t)kt * B_STAGE + o, OZ_PIECE, fb);
                    }
                }
            }
            // after an abort, let the loads already issued land before the CTA exits
            if (!ok)
                for (int q = max(0, it - STAGES); q < it; ++q)
                    mbar_wait(full0 + 8 * (q % STAGES), (uint32_t)((q / STAGES) & 1), args.err);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16(OZ_BM, OZ_BN);
            bool ok = true;
            int it = 0, ch = 0;
            for (int item = blockIdx.x; item < args.items && ok; item += gridDim.x) {
                OzProblem<Real> p;
                const OzItem t = oz_item(args, item, p);
                for (int kt = t.kt0; kt < t.kt1 && ok; ++ch) {
                    if (ch > 0) {
                        ok = mbar_wait(acc_empty, (uint32_t)((ch - 1) & 1), args.err);
                        if (!ok) break;
                        tc_fence_after();
                    }
                    const int end = min(t.kt1, kt + OZ_CHUNK);
                    for (bool first = true; kt < end; ++kt, ++it, first = false) {
                        const int s = it % STAGES, r = it / STAGES;
                        ok = mbar_wait(full0 + 8 * s, (uint32_t)(r & 1), args.err);
                        if (!ok) break;
                        tc_fence_after();
                        const uint64_t ad = sw64_desc(smem_u32(sA + s * A_STAGE));
                        const uint64_t bd = sw64_desc(smem_u32(sB + s * B_STAGE));
                        // lowest weight first: i + j = TOP down to 2 (1-based digits)
#pragma unroll
                        for (int w = Tr::TOP - 2; w >= 0; --w) {
                            const uint32_t acc = tmem + (uint32_t)((w < Tr::ACC - 1 ? w : Tr::ACC - 1) * OZ_BN);
                            const int i0 = w < D ? 0 : w - D + 1;
#pragma unroll
                            for (int i = i0; i <= w - i0; ++i) {
                                const int j = w - i;
                                const bool fresh = first && i == i0 && (w < Tr::ACC - 1 || w == Tr::TOP - 2);
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
        }
    } else {
        const int q = warp & 3, part = (warp - 2) >> 2;     // lane quadrant, column quarter
        const int row = q * 32 + lane;
        const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(part * OZ_COLS);
        bool ok = true;
        int ch = 0;
        for (int item = blockIdx.x; item < args.items && ok; item += gridDim.x) {
            OzProblem<Real> p;
            const OzItem t = oz_item(args, item, p);
            if (t.kt1 < 0) continue;
            // exponents (column nb + lane's in this lane) and C on its way to
            // L2 while the MMAs run
            const int nb = t.n0 + part * OZ_COLS, m = t.m0 + row;
            const int ea = m < p.M ? __ldcg(p.ea + m) : 0, eb = nb + lane < p.N ? __ldcg(p.eb + nb + lane) : 0;
            if (!p.partial && p.beta != Real(0) && nb + lane < p.N) {
                const Real *c = p.C + (int64_t)(nb + lane) * p.ldc + t.m0 + q * 32;
                const int rows = min(32, p.M - (t.m0 + q * 32));
                for (int r = 0; r < rows; r += 128 / (int)sizeof(Real)) asm volatile("prefetch.global.L2 [%0];" ::"l"(c + r));
                if (rows > 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(c + rows - 1));
            }
            long long X[OZ_COLS];
#pragma unroll
            for (int c = 0; c < OZ_COLS; ++c) X[c] = 0;
            for (int kt = t.kt0; kt < t.kt1; kt += OZ_CHUNK, ++ch) {
                ok = mbar_wait_warp(acc_full, (uint32_t)(ch & 1), args.err);
                if (!ok) break;
                tc_fence_after();
#pragma unroll
                for (int g = 0; g < OZ_COLS / 8; ++g) {
                    float a[Tr::ACC][8];
#pragma unroll
                    for (int s = 0; s < Tr::ACC; ++s) tmem_ld8(tbase + (uint32_t)(s * OZ_BN + g * 8), a[s]);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        float f[Tr::ACC];
#pragma unroll
                        for (int i = 0; i < Tr::ACC; ++i) f[i] = a[i][c];
                        X[g * 8 + c] += collect<Tr::ACC>(f);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acc_empty) : "memory");
            }
            // (every lane takes the same branch: the loops below shuffle)
            if (ok && p.partial) {
                if (m < p.M) {
                    long long *pp = p.partial + (size_t)t.z * p.M * p.N + m;
#pragma unroll
                    for (int c = 0; c < OZ_COLS; ++c)
                        if (nb + c < p.N) pp[(size_t)(nb + c) * p.M] = X[c];
                }
            } else if (ok) {
                // compared once: an FP64 comparison costs as much as an addition
                const bool minus = p.beta == Real(1) && p.alpha == Real(-1), read = p.beta != Real(0), plain = p.alpha == Real(1);
                const bool whole = t.m0 >= p.add_rows && t.m0 + OZ_BM <= p.M && nb + OZ_COLS <= p.N;
                if (whole && minus) {
                    // a whole tile of C -= V W
                    Real *cp = p.C + m + (int64_t)nb * p.ldc;
#pragma unroll
                    for (int g = 0; g < OZ_COLS; g += 8) {
                        Real cv[8], *cg = cp;
#pragma unroll
                        for (int c = 0; c < 8; ++c, cg += p.ldc) cv[c] = __ldcg(cg);
#pragma unroll
                        for (int c = 0; c < 8; ++c, cp += p.ldc)
                            *cp = cv[c] - scaled(X[g + c], ea + __shfl_sync(0xffffffffu, eb, g + c) - 14 - Tr::UNIT, Real(0));
                    }
                } else if (whole && !read && plain) {
                    // a whole tile of C = A X
                    Real *cp = p.C + m + (int64_t)nb * p.ldc;
#pragma unroll
                    for (int c = 0; c < OZ_COLS; ++c, cp += p.ldc)
                        *cp = scaled(X[c], ea + __shfl_sync(0xffffffffu, eb, c) - 14 - Tr::UNIT, Real(0));
                } else {
                    Real *cp = p.C + m + (int64_t)nb * p.ldc;
                    const Real *ap = m < min(p.add_rows, p.M) ? p.add + m + (int64_t)nb * p.ldadd : nullptr;
#pragma unroll
                    for (int c = 0; c < OZ_COLS; ++c) {
                        Real d = scaled(X[c], ea + __shfl_sync(0xffffffffu, eb, c) - 14 - Tr::UNIT, Real(0));
                        if (nb + c < p.N && m < p.M) {
                            const Real old = read ? __ldcg(cp + (int64_t)c * p.ldc) : Real(0);
                            Real out;
                            if (minus) {
                                out = (ap ? old - __ldcg(ap + (int64_t)c * p.ldadd) : old) - d;
                            } else {
                                if (ap) d += __ldcg(ap + (int64_t)c * p.ldadd);
                                if (!read) out = plain ? d : p.alpha * d;
                                else out = p.beta * old + p.alpha * d;
                            }
                            cp[(int64_t)c * p.ldc] = out;
                        }
                    }
                }
            }
            __syncwarp();
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCOLS));
    }
}

// sum_z P[z][e]: exact, high and low halves in 64 bits each, then FP64.
__device__ __forceinline__ double sum_partials(const long long *P, size_t stride, int S) {
    long long H = 0;
    unsigned long long L = 0;
#pragma unroll 8
    for (int z = 0; z < S; ++z) {
        const long long v = __ldcg(P + (size_t)z * stride);
        H += v >> 32;
        L += (unsigned long long)v & 0xffffffffull;
    }
    return fma((double)H, 4294967296.0, (double)L);
}

template <class Real>
__device__ __forceinline__ const OzProblem<Real> &nth_problem(const OzMmaArgs<Real> &args, int which) {
    return args.list ? args.list[which] : args.prob[which];
}

// C = beta C + alpha 2^(ea + eb - 14 - UNIT) sum_z P[z], one rounding to FP64
// (FP32: and one to FP32).  blockIdx.y: the problem.
template <class Real>
__global__ void __launch_bounds__(kThreads) oz_reduce_kernel(const __grid_constant__ OzMmaArgs<Real> args) {
    const OzProblem<Real> p = nth_problem(args, blockIdx.y);
    if (p.skip && *(volatile const int *)p.skip) return;
    const size_t total = (size_t)p.M * p.N;
    for (size_t e = blockIdx.x * (size_t)kThreads + threadIdx.x; e < total; e += (size_t)gridDim.x * kThreads) {
        const int i = (int)(e % (unsigned)p.M), j = (int)(e / (unsigned)p.M);
        const double s = sum_partials(p.partial + e, total, p.S);
        const int ea = __ldcg(p.ea + i), eb = __ldcg(p.eb + j);
        double d = (ea == kExpNan || eb == kExpNan) ? nan_value<double>()
                                                    : mul_pow2(s, ea + eb - 14 - OzTraits<Real>::UNIT);
        if (i < p.add_rows) d += (double)p.add[i + (int64_t)j * p.ldadd];
        if (p.Cd) {                                        // FP64 result of an FP32 product
            p.Cd[i + (int64_t)j * p.ldc] = d;
            continue;
        }
        Real *cp = p.C + i + (int64_t)j * p.ldc;
        Real out;
        if (p.beta == Real(0)) out = p.alpha == Real(1) ? (Real)d : p.alpha * (Real)d;
        else if (p.beta == Real(1) && p.alpha == Real(-1)) out = *cp - (Real)d;
        else out = p.beta * *cp + p.alpha * (Real)d;
        *cp = out;
    }
}

// The M x N sums (M <= 128) as the digits of the next product's B operand:
// column j becomes operand row j with M entries, and (for the unit diagonal
// of a V basis, which no digits carry) the rounded sums.  A warp per column, 4
// consecutive rows per lane.
template <class Real>
__global__ void __launch_bounds__(kThreads) oz_requant_kernel(const __grid_constant__ OzMmaArgs<Real> args) {
    const OzProblem<Real> p = nth_problem(args, blockIdx.y);
    const int lane = threadIdx.x & 31, KT = (p.M + OZ_BK - 1) / OZ_BK;
    const size_t total = (size_t)p.M * p.N;
    for (int j = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5); j < p.N; j += gridDim.x * (kThreads / 32)) {
        const int eb = __ldcg(p.eb + j);
        Real v[4];
        int ex = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = lane * 4 + q;
            v[q] = Real(0);
            if (i < p.M) {
                const double s = sum_partials(p.partial + i + (size_t)j * p.M, total, p.S);
                const int ea = __ldcg(p.ea + i);
                v[q] = (ea == kExpNan || eb == kExpNan) ? nan_value<Real>()
                                                        : (Real)mul_pow2(s, ea + eb - 14 - OzTraits<Real>::UNIT);
            }
            ex = max(ex, exp_field(v[q]));
            if (p.C && i < p.M) p.C[i + (int64_t)j * p.ldc] = v[q];
        }
        ex = max(__reduce_max_sync(0xffffffffu, ex), 1);
        if (lane == 0) p.qexp[j] = ex == ExpOf<Real>::INF ? kExpNan : ex - ExpOf<Real>::BIAS;
        if (ex == ExpOf<Real>::INF)
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = Real(0);
        if (lane * 4 < KT * OZ_BK) store_digits<OzTraits<Real>::D>(p.qdst, KT, OZ_BN, j, lane * 4, v, ex);
    }
}

size_t a256(size_t x) { return (x + 255) / 256 * 256; }

// Split of a product: K tiles per item, splits and the estimated time (us).
// Cycles per item are those of the kernel's parts: about 2900 (FP32: 900) per
// 32-k step, 3500 per drain; the FP64 epilogue, 9000, runs beside the next
// item's MMAs where a CTA has one.
struct OzSplit { int kt_per, S; double us; };
template <class Real>
OzSplit oz_split(int64_t M, int64_t N, int64_t K, int num_sms, size_t part_cap_elems, bool force_partial) {
    const int64_t tiles = ((M + OZ_BM - 1) / OZ_BM) * ((N + OZ_BN - 1) / OZ_BN);
    const int kt = (int)((K + OZ_BK - 1) / OZ_BK);
    const double step = std::is_same<Real, double>::value ? 2900.0 : 900.0;
    OzSplit best{0, 0, 1e30};
    for (int per = 1; per <= std::min(kt, OzTraits<Real>::MAX_KT); ++per) {
        const int S = (kt + per - 1) / per;
        if ((S > 1 || force_partial) && ((size_t)S * M * N > part_cap_elems || S > kOzMaxSplits)) continue;
        const double item = 1000.0 + step * per + 3500.0 * ((per + OZ_CHUNK - 1) / OZ_CHUNK) + (S == 1 && !force_partial ? 3000.0 : 1500.0);
        double clk = 4000.0 + std::ceil((double)tiles * S / num_sms) * item;
        if (S > 1) clk += 6000.0 + (double)S * M * N * 16.0 / 2500.0;
        if (clk / 1900.0 < best.us) best = {per, S, clk / 1900.0};
    }
    return best;
}

}  // namespace

int oz_ktiles(int64_t K) { return (int)((K + OZ_BK - 1) / OZ_BK); }

size_t oz_digit_bytes(int D, int64_t R, int64_t K, int rt) {
    return a256((size_t)((R + rt - 1) / rt) * oz_ktiles(K) * D * rt * 64) + a256((size_t)R * 4);
}

template <class Src>
OzOperand<Src> oz_operand(int D, const Src *X, int64_t ld, int64_t R, int64_t K, bool by_row, int mask, int rt,
                          void *mem) {
    OzOperand<Src> o{};
    o.X = X; o.ld = ld; o.R = R; o.K = K; o.by_row = by_row ? 1 : 0; o.mask = mask;
    o.KT = oz_ktiles(K);
    o.rt = rt;
    o.dst = (uint8_t *)mem;
    o.exps = (int *)((char *)mem + oz_digit_bytes(D, R, K, rt) - a256((size_t)R * 4));
    return o;
}
template OzOperand<double> oz_operand(int, const double *, int64_t, int64_t, int64_t, bool, int, int, void *);
template OzOperand<float> oz_operand(int, const float *, int64_t, int64_t, int64_t, bool, int, int, void *);

template <class Real>
unsigned oz_slice_blocks(const OzOperand<Real> &o, bool tall) {
    const int warps = tall ? 16 : 8;
    return (unsigned)(o.by_row ? (o.R + 4 * warps - 1) / (4 * warps) : (o.K > 1024 ? o.R : (o.R + warps - 1) / warps));
}
template unsigned oz_slice_blocks(const OzOperand<double> &, bool);
template unsigned oz_slice_blocks(const OzOperand<float> &, bool);

template <class Src>
gbqr_status oz_slice_launch(const Exec &ex, int D, const OzSliceArgs<Src> &args, unsigned blocks, bool tall, double elems) {
    if (!blocks) return GBQR_OK;
    if (D != kD32 && (D != kD64 || std::is_same<Src, float>::value)) return GBQR_EINVAL;
    trace_begin(ex, FAM_OTHER);
    if (D == kD32) {
        if (tall) oz_slice_kernel<Src, kD32, 512, 8><<<blocks, 512, 0, ex.stream>>>(args);
        else oz_slice_kernel<Src, kD32, kThreads, 8><<<blocks, kThreads, 0, ex.stream>>>(args);
    } else if constexpr (std::is_same<Src, double>::value) {
        if (tall) oz_slice_kernel<Src, kD64, 512, 8><<<blocks, 512, 0, ex.stream>>>(args);
        else oz_slice_kernel<Src, kD64, kThreads, 8><<<blocks, kThreads, 0, ex.stream>>>(args);
    }
    return trace_end(ex, FAM_OTHER, 0.0, ((double)sizeof(Src) + 2.0 * D) * elems);
}
template gbqr_status oz_slice_launch(const Exec &, int, const OzSliceArgs<double> &, unsigned, bool, double);
template gbqr_status oz_slice_launch(const Exec &, int, const OzSliceArgs<float> &, unsigned, bool, double);

template <class Src>
gbqr_status oz_slice(const Exec &ex, int D, OzOperand<Src> *ops, int n) {
    OzSliceArgs<Src> args{};
    unsigned blocks = 0;
    bool tall = false;
    double elems = 0.0;
    if (n > kOzOps) return GBQR_EINVAL;
    for (int i = 0; i < n; ++i) tall = tall || (!ops[i].by_row && ops[i].K > 8192);
    for (int i = 0; i < n; ++i) {
        ops[i].first = blocks;
        blocks += oz_slice_blocks(ops[i], tall);
        elems += (double)ops[i].R * ops[i].K;
        args.op[i] = ops[i];
    }
    args.n = n;
    return oz_slice_launch(ex, D, args, blocks, tall, elems);
}
template gbqr_status oz_slice(const Exec &, int, OzOperand<double> *, int);
template gbqr_status oz_slice(const Exec &, int, OzOperand<float> *, int);

template <class Real, class SA, class SB>
OzProblem<Real> oz_problem(const OzOperand<SA> &a, const OzOperand<SB> &b) {
    OzProblem<Real> p{};
    p.a = a.dst; p.b = b.dst; p.ea = a.exps; p.eb = b.exps;
    p.M = (int)a.R; p.N = (int)b.R; p.KT = a.KT;
    p.kt_per = p.KT; p.S = 1;
    p.alpha = Real(1);
    p.skip = a.skip;
    p.b128 = b.rt == OZ_BM;
    // op(A) lower: zero for k < i (stored K x M) or k > i; B upper: zero for k > j
    if (a.mask == MASK_UNIT_LOWER) p.clip = a.by_row ? 2 : 1;
    if (b.mask == MASK_UPPER && !b.by_row) p.clipB = 2;
    return p;
}
template OzProblem<double> oz_problem<double>(const OzOperand<double> &, const OzOperand<double> &);
template OzProblem<float> oz_problem<float>(const OzOperand<float> &, const OzOperand<float> &);
template OzProblem<float> oz_problem<float>(const OzOperand<float> &, const OzOperand<double> &);

int oz_items(int M, int N, int S) { return ((M + OZ_BM - 1) / OZ_BM) * ((N + OZ_BN - 1) / OZ_BN) * S; }

// Chooses the split of a product whose partials fit part_bytes.
template <class Real>
bool oz_choose_split(OzProblem<Real> &p, int num_sms, size_t part_bytes, bool force_partial) {
    const OzSplit s = oz_split<Real>(p.M, p.N, (int64_t)p.KT * OZ_BK, num_sms, part_bytes / 8, force_partial);
    p.kt_per = s.kt_per;
    p.S = s.S;
    return s.S > 0;
}
template bool oz_choose_split(OzProblem<double> &, int, size_t, bool);
template bool oz_choose_split(OzProblem<float> &, int, size_t, bool);

template <class Real>
gbqr_status oz_mma_launch(const Exec &ex, const OzMmaArgs<Real> &args, double elems) {
    if (args.items <= 0) return GBQR_OK;
    static std::atomic<bool> attr[64];
    const bool cached = ex.device >= 0 && ex.device < 64;
    if (!cached || !attr[ex.device].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(oz_mma_kernel<Real>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)oz_smem<Real>()) != cudaSuccess)
            return GBQR_ECUDA;
        if (cached) attr[ex.device].store(true, std::memory_order_release);
    }
    // a few items per CTA, so that epilogues overlap MMAs; no more, so that a
    // look-ahead panel's launches on another stream find free SMs soon
    const int grid = std::min(args.items, std::max(ex.num_sms, (args.items + kOzItemsPerCta - 1) / kOzItemsPerCta));
    trace_begin(ex, FAM_TC_GEMM);
    oz_mma_kernel<Real><<<grid, OZ_THREADS, oz_smem<Real>(), ex.stream>>>(args);
    return trace_end(ex, FAM_TC_GEMM, 2.0 * oz_products<Real>() * elems, 0.0);
}
template gbqr_status oz_mma_launch(const Exec &, const OzMmaArgs<double> &, double);
template gbqr_status oz_mma_launch(const Exec &, const OzMmaArgs<float> &, double);

template <class Real>
gbqr_status oz_reduce_launch(const Exec &ex, const OzMmaArgs<Real> &args, size_t largest) {
    trace_begin(ex, FAM_OTHER);
    const unsigned g = (unsigned)std::min<size_t>((largest + kThreads - 1) / kThreads, (size_t)ex.num_sms * 16);
    oz_reduce_kernel<Real><<<dim3(g, (unsigned)args.n), kThreads, 0, ex.stream>>>(args);
    return trace_end(ex, FAM_OTHER, 0.0, 0.0);
}
template gbqr_status oz_reduce_launch(const Exec &, const OzMmaArgs<double> &, size_t);
template gbqr_status oz_reduce_launch(const Exec &, const OzMmaArgs<float> &, size_t);

template <class Real>
gbqr_status oz_requant_launch(const Exec &ex, const OzMmaArgs<Real> &args, int widest) {
    trace_begin(ex, FAM_OTHER);
    const unsigned g = (unsigned)std::min((widest + 7) / 8, ex.num_sms * 16);
    oz_requant_kernel<Real><<<dim3(g, (unsigned)args.n), kThreads, 0, ex.stream>>>(args);
    return trace_end(ex, FAM_OTHER, 0.0, 0.0);
}
template gbqr_status oz_requant_launch(const Exec &, const OzMmaArgs<double> &, int);
template gbqr_status oz_requant_launch(const Exec &, const OzMmaArgs<float> &, int);

// Digits of op(A) and of up to N columns of B, and the partials of a split
// that gives every item at most 512 k and a small output two CTAs per SM.
template <class Real>
size_t oz_gemm_scratch_bytes(int64_t M, int64_t N, int64_t K) {
    const int64_t tiles = std::max<int64_t>(1, ((M + OZ_BM - 1) / OZ_BM) * ((N + OZ_BN - 1) / OZ_BN));
    const int64_t S = std::max((K + 16 * OZ_BK - 1) / (16 * OZ_BK),
                               std::min<int64_t>({(K + OZ_BK - 1) / OZ_BK, (304 + tiles - 1) / tiles, 64}));
    return oz_digit_bytes(OzTraits<Real>::D, M, K, OZ_BM) + oz_digit_bytes(OzTraits<Real>::D, N, K, OZ_BN) + (S > 1 ? a256((size_t)S * M * N * 8) : 0);
}
template size_t oz_gemm_scratch_bytes<double>(int64_t, int64_t, int64_t);
template size_t oz_gemm_scratch_bytes<float>(int64_t, int64_t, int64_t);

// How C = alpha op(A) B + beta C is done here, if at all: the columns of B in
// chunks whose digits fit the scratch, where the estimated time beats the
// FMA kernel's (1.15 TFLOP/s on large products; FP32 about 9).
struct OzPlan { int64_t nc; OzSplit split; };
template <class Real>
static bool oz_plan(const GemmOpT<Real> &op, const OzScratch &sc, int num_sms, OzPlan *plan, double *gain_us) {
    if (!sc.base || op.M < 8 || op.N < 8 || op.K < 8) return false;
    if (op.M > (1 << 30) || op.N > (1 << 30) || op.K > (1 << 30)) return false;
    int64_t nc = op.N;
    const size_t room = sc.bytes - sc.bytes / 8;                 // an eighth for partials
    const size_t fixed = oz_digit_bytes(OzTraits<Real>::D, op.M, op.K, OZ_BM) + 512;
    if (fixed + oz_digit_bytes(OzTraits<Real>::D, nc, op.K, OZ_BN) > room) {
        const size_t col = oz_digit_bytes(OzTraits<Real>::D, OZ_BN, op.K, OZ_BN);
        const int64_t most = fixed < room ? (int64_t)((room - fixed) / col) * OZ_BN : 0;
        if (most >= OZ_BN) {                                     // equal chunks of whole tiles
            const int64_t chunks = (nc + most - 1) / most;
            nc = ((nc + chunks - 1) / chunks + OZ_BN - 1) / OZ_BN * OZ_BN;
        }
    }
    const size_t digits = oz_digit_bytes(OzTraits<Real>::D, op.M, op.K, OZ_BM) + oz_digit_bytes(OzTraits<Real>::D, nc, op.K, OZ_BN);
    if (digits > sc.bytes) return false;
    // a chunk of a masked B starts off B's diagonal: below it a unit lower
    // trapezoid is one again (oz_gemm), the others are not cut
    if (nc < op.N && op.maskB != MASK_NONE &&
        !(op.maskB == MASK_UNIT_LOWER && op.maskA == MASK_NONE && op.K >= op.N + 64)) return false;
    if ((size_t)op.M * nc >= ((size_t)1 << 32) || oz_items((int)op.M, (int)nc, 1) < 0) return false;
    plan->nc = nc;
    plan->split = oz_split<Real>(op.M, nc, op.K, num_sms, (sc.bytes - digits) / 8, false);
    if (plan->split.S == 0) return false;
    const double chunks = std::ceil((double)op.N / nc);
    const double slice_us = (sizeof(Real) + 2.0 * OzTraits<Real>::D) * ((double)op.M + nc) * op.K / 4.0e6;
    const double rate = std::is_same<Real, double>::value ? 1.15e6 : 9.0e6;
    *gain_us = gemm_algorithmic_flops(op) / rate - chunks * (plan->split.us + slice_us + 10.0);
    return true;
}

template <class Real>
bool oz_gemm_wanted(const GemmOpT<Real> &op, const OzScratch &sc, int num_sms) {
    OzPlan p;
    double gain = 0.0;
    return sc.base && gemm_algorithmic_flops(op) > 1.4e7 && oz_plan(op, sc, num_sms, &p, &gain) && gain > 0.0;
}
template bool oz_gemm_wanted(const GemmOpT<double> &, const OzScratch &, int);
template bool oz_gemm_wanted(const GemmOpT<float> &, const OzScratch &, int);

// One chunk of columns; slice_a: op(A)'s digits are not in the scratch yet.
template <class Real>
static gbqr_status oz_chunk(const Exec &ex, const GemmOpT<Real> &op, const OzScratch &sc, bool slice_a) {
    char *base = (char *)sc.base;
    const size_t na = oz_digit_bytes(OzTraits<Real>::D, op.M, op.K, OZ_BM), nb = oz_digit_bytes(OzTraits<Real>::D, op.N, op.K, OZ_BN);
    if (na + nb > sc.bytes) return GBQR_ENOMEM;
    OzOperand<Real> a = oz_operand(OzTraits<Real>::D, op.A, op.lda, op.M, op.K, !op.ta, op.maskA, OZ_BM, base);
    OzOperand<Real> b = oz_operand(OzTraits<Real>::D, op.B, op.ldb, op.N, op.K, false, op.maskB, OZ_BN, base + na);
    b.unit = 1;
    OzOperand<Real> ops[2];
    int n = 0;
    if (slice_a) ops[n++] = a;
    if (op.ta && op.A == op.B && op.lda == op.ldb && op.M == op.N && op.maskA == MASK_NONE && op.maskB == MASK_NONE) b = a;   // X^T X
    else ops[n++] = b;
    TRY_ST(oz_slice(ex, OzTraits<Real>::D, ops, n));
    OzMmaArgs<Real> args{};
    OzProblem<Real> &p = args.prob[0];
    p = oz_problem<Real>(a, b);
    p.C = op.C; p.ldc = op.ldc; p.alpha = op.alpha; p.beta = op.beta;
    if (op.maskA == MASK_UNIT_LOWER) {
        // + B(i, j) for the unit diagonal; the strict part is split without it,
        // whose entries it would outweigh by orders of magnitude
        p.add = op.B; p.ldadd = op.ldb;
        p.add_rows = (int)std::min(op.M, op.K);
    }
    if (!oz_choose_split(p, ex.num_sms, sc.bytes - na - nb, false)) return GBQR_ENOMEM;
    p.partial = p.S > 1 ? (long long *)(base + na + nb) : nullptr;
    args.n = 1;
    args.items = oz_items(p.M, p.N, p.S);
    args.err = sc.err;
    TRY_ST(oz_mma_launch(ex, args, (double)op.M * op.N * op.K));
    return p.S > 1 ? oz_reduce_launch(ex, args, (size_t)op.M * op.N) : GBQR_OK;
}

template <class Real>
gbqr_status oz_gemm(const Exec &ex, const GemmOpT<Real> &op, const OzScratch &sc) {
    OzPlan pl;
    double gain = 0.0;
    if (!oz_plan(op, sc, ex.num_sms, &pl, &gain)) return GBQR_ENOMEM;
    for (int64_t j = 0; j < op.N; j += pl.nc) {
        GemmOpT<Real> c = op;
        c.N = std::min(pl.nc, op.N - j);
        c.B = op.B + j * op.ldb;
        c.C = op.C + j * op.ldc;
        const bool below = j > 0 && op.maskB == MASK_UNIT_LOWER;   // the rows above the chunk's diagonal are zero
        if (below) {
            c.K = op.K - j;
            c.A = op.ta ? op.A + j : op.A + j * op.lda;
            c.B += j;
        }
        TRY_ST(oz_chunk(ex, c, sc, j == 0 || below));
    }
    return GBQR_OK;
}
template gbqr_status oz_gemm(const Exec &, const GemmOpT<double> &, const OzScratch &);
template gbqr_status oz_gemm(const Exec &, const GemmOpT<float> &, const OzScratch &);

}  // namespace gbqr
