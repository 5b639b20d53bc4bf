// Householder QR of a well-conditioned m x w panel (w <= 128, m >= 4 w) from
// its Gram matrix, the fast base case of QR-EG in FP64.
//
// The TSQR base case (tsqr.cu) is a serial chain of w Householder steps per
// tree level, about 12 us a column, whatever the number of rows.  A panel
// whose columns are far from dependent needs no tree:
//
//   G = P^T P                     one tall product (digit-split: exact sums)
//   R+^T R+ = G                   Cholesky
//   A1 - S R+ = V1 U              LU without pivoting of the top w x w block,
//                                 S_jj = -sgn(pivot before the subtraction)
//   Z = -R+^{-1} S V1^{-T},  T = U Z
//   V2 = A2 U^{-1}                the rows below, one tall product,
//   Y2 = A2 Z                     and where the caller asks, Y = V T beside it
//
// R = S R+.  Why this is the Householder QR: with Q = I - V T V^T and Q^T A =
// [R; 0], A - [R; 0] = -V (T V1^T R), a unit lower trapezoidal matrix times
// an upper triangular one; that factorization is unique, and its pivots
// before the subtraction are the entries alpha_j that fix the Householder
// signs.  It is the reconstruction of Appendix C.2 with A R^{-1} for W
// (Ballard, Demmel, Grigori, Jacquelin, Nguyen, Solomonik 2014, who note
// that it is the less stable variant: errors grow with the panel's
// condition).  So it is taken only where the condition allows: every entry
// of R+^{-1}, its rows scaled by the column norms, has to stay at or below 4
// in magnitude (1 on the diagonal and 0 off it for orthogonal columns).  Then
// the Cholesky's few u are amplified by a small factor, and V, T and R agree
// with the TSQR's to rounding.  Otherwise a device flag is raised, the panel
// is left untouched, and the caller's TSQR launches, which return at once
// while the flag is zero, factor it.
//
// The w x w work runs in 32-wide blocks, three launches a block:
//   diag   one CTA: Cholesky and LU of the diagonal block
//   row    triangular solves with it: block row k of R and U, block column k
//          of L, the diagonal blocks of R^{-1}, U^{-1} and V1^{-1}, ...
//   trail  the trailing blocks of G and A1; R^{-1}, U^{-1} and V1^{-1} grow by
//          one block column or row.
// FP64 issues one instruction per warp per 64 cycles and per SM sub-partition
// per 76 on this part, so diag is bound by its 64 dependent pivots (a
// reciprocal, a multiply-add and a barrier each) and does nothing else: with
// the block's inverses formed in it by augmented columns, it took 75 us, the
// columns' FP64 issue delaying the chain; without them 20 us.  A 32^3 product
// on one SM would take 9 us, so row and trail spread every block over 8 CTAs;
// a triangular solve with a unit diagonal is 32 shuffles and multiply-adds,
// no longer than a product with the inverse.
#include "oz.cuh"
#include "tsqr_dev.cuh"

#include <algorithm>
#include <cmath>
#include <type_traits>

namespace gbqr {
namespace {

constexpr int GB = 32;               // block width
constexpr int GLD = kGramMaxW;       // leading dimension of every w x w array
constexpr int GT = 128;              // threads of the row / trail kernels: 32 x 4 outputs
constexpr double kGramBound2 = 16.0; // largest accepted (R^-1)_ij^2 g_ii

template <class Real>
struct GramArgs {
    Real *A; int64_t lda;            // panel
    Real *Tout; int64_t ldt;
    Real *Y; int64_t ldy;            // V T (null: not wanted)
    int w, nblk;
    double *G, *R, *RI, *A1, *L, *U, *LI, *X, *YX, *YR, *YL, *B1, *Z, *sgn, *gd;
    double *M;                       // the block's unit triangular factors, M[t][lane]: see UnitFactor
    double *sc;                      // ... and the reciprocals of R's and U's diagonal
    int *flag, *kexp;                // kexp: exponents of the column norms
};

template <class Real>
__device__ __forceinline__ double g_at(const GramArgs<Real> &p, int i, int j, int k) {
    if (k > 0) return __ldcg(p.G + i + j * GLD);
    return (i < p.w && j < p.w) ? __ldcg(p.G + i + j * GLD) : (i == j ? 1.0 : 0.0);
}
template <class Real>
__device__ __forceinline__ double a1_at(const GramArgs<Real> &p, int i, int j, int k) {
    if (k > 0) return __ldcg(p.A1 + i + j * GLD);
    return (i < p.w && j < p.w) ? (double)p.A[i + (int64_t)j * p.lda] : (i == j ? 1.0 : 0.0);
}

// 1/d by the reciprocal approximation and one third-order Newton step
// (r + r (e + e^2), e = 1 - d r): three dependent FP64 instructions, where
// the correctly rounded reciprocal takes about twice as long.
__device__ __forceinline__ double quick_rcp(double d) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    const double e = rfma(-d, r, 1.0);
    return rfma(r, rfma(e, e, e), r);
}

// Unit triangular factors of the diagonal block, row t holding the
// coefficients of step t of a substitution: Cholesky's L (M[t][i] = L(i, t),
// i > t), V1's diagonal block the same way, and U scaled to a unit diagonal
// (M[t][j] = U(t, j) / U(t, t), j > t).
enum UnitFactor { UF_CHOL = 0, UF_L = 1, UF_U = 2 };

// Diagonal block k: S = D^{1/2}-free Cholesky G_kk = Lc D Lc^T, then the LU of
// A1_kk - S R_kk.  Warp 0 carries the chain: it brings the next column up to
// date, takes its pivot's reciprocal and publishes both, while the other
// warps apply the current column to the ones behind; in the LU warp 1 carries
// the next row of U the same way.  One barrier a step.  Warp 4, which shares
// warp 0's sub-partition, stays idle, so that the chain's instructions do not
// queue behind it.
template <class Real>
__global__ void __launch_bounds__(kThreads) gram_diag_kernel(const GramArgs<Real> p, int k) {
    __shared__ double S[GB][GB + 1], Rb[GB][GB + 1];     // [column][row]; Rb: R(row, column)
    __shared__ double cb[2][GB], ub[2][GB], rb[2], rd[GB], sg[GB];
    __shared__ int bad;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, b0 = k * GB;
    if (k > 0 && *(volatile int *)p.flag) return;
    double a1[GB / 8];                                   // the LU's block, loaded behind the Cholesky's
#pragma unroll
    for (int q = 0; q < GB / 8; ++q) {
        const int c = warp + 8 * q;
        S[c][lane] = lane <= c ? g_at(p, b0 + lane, b0 + c, k) : g_at(p, b0 + c, b0 + lane, k);
        a1[q] = a1_at(p, b0 + lane, b0 + c, k);
    }
    if (k == 0)
        for (int i = tid; i < p.nblk * GB; i += kThreads) {
            const double g = i < p.w ? __ldcg(p.G + i + i * GLD) : 1.0;
            p.gd[i] = g;
            p.kexp[i] = (((__double2hiint(g) >> 20) & 0x7ff) - 1023) >> 1;
        }
    if (tid == 0) bad = 0;
    __syncthreads();
    // ---- Cholesky
    double v = 0.0, r = 0.0;                             // warp 0: column t below (and at) its pivot, 1 / pivot
    if (warp == 0) {
        v = S[0][lane];
        r = quick_rcp(__shfl_sync(kFull, v, 0));
        cb[0][lane] = v;
        if (lane == 0) rb[0] = rd[0] = r;
    }
    __syncthreads();
    for (int t = 0; t + 1 < GB; ++t) {
        if (warp == 0) {
            v = rfma(-r, v * __shfl_sync(kFull, v, t + 1), S[t + 1][lane]);
            r = quick_rcp(__shfl_sync(kFull, v, t + 1));
            S[t + 1][lane] = v;
            cb[(t + 1) & 1][lane] = v;
            if (lane == 0) rb[(t + 1) & 1] = rd[t + 1] = r;
        } else if (warp != 4) {
            const double *c = cb[t & 1];
            const int first = t + 2 + (warp > 4 ? warp - 2 : warp - 1);      // six warps share the columns
            if (first < GB) {
                const double li = lane > t ? c[lane] * rb[t & 1] : 0.0;
                for (int j = first; j < GB; j += 6) S[j][lane] = rfma(-li, c[j], S[j][lane]);
            }
        }
        __syncthreads();
    }
    // R = D^{1/2} Lc^T; column t of S holds d_t Lc(:, t)
    if (warp == 0) {
        const double d = S[lane][lane];
        if (!(d > 0.0 && d < 1e300)) bad = 1;
        const double s = sqrt(d);
        sg[lane] = s;
        p.sc[lane] = s * rd[lane];                       // 1 / r_tt
    }
    __syncthreads();
    if (bad) {
        if (tid == 0) *p.flag = 1;
        return;
    }
    if (k == 0 && tid == 0) *p.flag = 0;
#pragma unroll
    for (int q = 0; q < GB / 8; ++q) {
        // row t = c of the factor, lane = i
        const int c = warp + 8 * q;
        const double lc = S[c][lane] * rd[c];
        p.M[c * GB + lane] = lane > c ? lc : 0.0;
        const double rv = lane > c ? lc * sg[c] : (lane == c ? sg[c] : 0.0);
        Rb[lane][c] = rv;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < GB / 8; ++q) {
        const int c = warp + 8 * q;
        p.R[(b0 + lane) + (b0 + c) * GLD] = Rb[c][lane];
        S[c][lane] = a1[q];
    }
    __syncthreads();
    // ---- LU of A1 - S R.  v: column t; ub: row t of U
    if (warp == 0) {
        v = S[0][lane];
        const double al = __shfl_sync(kFull, v, 0), rr = Rb[0][0];
        r = quick_rcp(al - (al < 0.0 ? rr : -rr));
        cb[0][lane] = v;
        if (lane == 0) rb[0] = rd[0] = r;
    } else if (warp == 1) {
        const double x = S[lane][0], s = __shfl_sync(kFull, x, 0) < 0.0 ? 1.0 : -1.0;
        if (lane == 0) sg[0] = s;
        const double u = x - s * Rb[lane][0];
        ub[0][lane] = u;
        p.U[b0 + (b0 + lane) * GLD] = u;
    }
    __syncthreads();
    for (int t = 0; t + 1 < GB; ++t) {
        const double *u = ub[t & 1];
        if (warp == 0) {
            // (the product first: the same bits as in warp 1, so that both see one pivot)
            v = rfma(-r, v * u[t + 1], S[t + 1][lane]);
            const double al = __shfl_sync(kFull, v, t + 1), rr = Rb[t + 1][t + 1];
            r = quick_rcp(al - (al < 0.0 ? rr : -rr));
            if (lane > t + 1) S[t + 1][lane] = v;           // (warp 1 reads the pivot entry)
            cb[(t + 1) & 1][lane] = v;
            if (lane == 0) rb[(t + 1) & 1] = rd[t + 1] = r;
        } else if (warp == 1) {
            const double x = rfma(-rb[t & 1], cb[t & 1][t + 1] * u[lane], S[lane][t + 1]);
            const double s = __shfl_sync(kFull, x, t + 1) < 0.0 ? 1.0 : -1.0;
            if (lane == 0) sg[t + 1] = s;
            const double un = lane > t ? x - s * Rb[lane][t + 1] : 0.0;
            ub[(t + 1) & 1][lane] = un;
            p.U[(b0 + t + 1) + (b0 + lane) * GLD] = un;
        } else if (warp != 4) {
            const int first = t + 2 + (warp > 4 ? warp - 3 : warp - 2);      // five warps
            if (first < GB) {
                const double li = cb[t & 1][lane] * rb[t & 1];
                if (lane > t + 1)
                    for (int j = first; j < GB; j += 5) S[j][lane] = rfma(-li, u[j], S[j][lane]);
            }
        }
        __syncthreads();
    }
    // L(i, t) = column t times 1 / u_tt
#pragma unroll
    for (int q = 0; q < GB / 8; ++q) {
        const int c = warp + 8 * q;
        const double l = S[c][lane] * rd[c];
        p.L[(b0 + lane) + (b0 + c) * GLD] = lane > c ? l : (lane == c ? 1.0 : 0.0);
        p.M[(UF_L * GB + c) * GB + lane] = lane > c ? l : 0.0;
        p.M[(UF_U * GB + c) * GB + lane] = lane > c ? __ldcg(p.U + (b0 + c) + (b0 + lane) * GLD) * rd[c] : 0.0;
    }
    if (tid < GB) {
        p.sgn[b0 + tid] = sg[tid];
        p.sc[GB + tid] = rd[tid];
    }
}

// acc += sum_kk A(i, kk) B(kk, c) over one 32-wide step; A staged in sA
// ([kk][i]), B in sB ([c][kk]).
struct Tile {
    double (*sA)[GB + 1];
    double (*sB)[GB];
    int warp, lane;
    __device__ __forceinline__ void load_a(const double *A, bool trans) {
#pragma unroll
        for (int kk = warp; kk < GB; kk += 4) {
            if (!trans) sA[kk][lane] = __ldcg(A + lane + kk * GLD);
            else sA[lane][kk] = __ldcg(A + lane + kk * GLD);
        }
    }
    __device__ __forceinline__ void load_b(const double *B, bool trans = false) {
        sB[warp][lane] = trans ? __ldcg(B + warp + lane * GLD) : __ldcg(B + lane + warp * GLD);
    }
    __device__ __forceinline__ double dot(double acc) const {
        double a0 = acc, a1 = 0.0;
#pragma unroll
        for (int kk = 0; kk < GB; kk += 2) {
            a0 = rfma(sA[kk][lane], sB[warp][kk], a0);
            a1 = rfma(sA[kk + 1][lane], sB[warp][kk + 1], a1);
        }
        return a0 + a1;
    }
};

__device__ __forceinline__ const double *blk(const double *M, int i, int j) { return M + i * GB + j * GB * GLD; }
__device__ __forceinline__ double *blk(double *M, int i, int j) { return M + i * GB + j * GB * GLD; }

// y <- the solution of a unit triangular system by substitution, one warp,
// lane = unknown: y_i -= M[t][i] y_t for t = 0, 1, ...
__device__ __forceinline__ double unit_solve(const double (*M)[GB + 1], double y) {
    const int lane = threadIdx.x & 31;
#pragma unroll 8
    for (int t = 0; t + 1 < GB; ++t) y = rfma(-M[t][lane], __shfl_sync(kFull, y, t), y);
    return y;
}
__device__ __forceinline__ void load_unit(double (*M)[GB + 1], const double *src, int which) {
    for (int t = threadIdx.x >> 5; t < GB; t += GT / 32)
        M[t][threadIdx.x & 31] = __ldcg(src + (which * GB + t) * GB + (threadIdx.x & 31));
}

// Solves with diagonal block k, a warp per column or row: block row k of R and
// U (tasks 0 .. n-k-2), block column k of L (the next n-k-1), the diagonal
// blocks of U^{-1}, R^{-1} and V1^{-1} (3 tasks); then for l < k: YX_l = U_lk
// U_kk^{-1}, YR_l = R_lk R_kk^{-1} and YL_l = sum_j L_kj LI_jl.
// blockIdx.x = task * 8 + column (row) group.
template <class Real>
__global__ void __launch_bounds__(GT) gram_row_kernel(const GramArgs<Real> p, int k) {
    __shared__ double sA[GB][GB + 1], sB[4][GB];
    if (*(volatile int *)p.flag) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int task = blockIdx.x >> 3;
    const int c0 = (blockIdx.x & 7) * 4, rest = p.nblk - k - 1, c = c0 + warp;
    const double rinv = __ldcg(p.sc + lane), uinv = __ldcg(p.sc + GB + lane);
    if (task < rest) {
        const int j = k + 1 + task;
        const double g = g_at(p, k * GB + lane, j * GB + c, k), a = a1_at(p, k * GB + lane, j * GB + c, k);
        load_unit(sA, p.M, UF_CHOL);                           // R_kk^T R_kj = G_kj
        __syncthreads();
        const double r = unit_solve(sA, g) * rinv;
        blk(p.R, k, j)[lane + c * GLD] = r;
        __syncthreads();
        load_unit(sA, p.M, UF_L);                              // V1_kk U_kj = A1_kj - S R_kj
        __syncthreads();
        blk(p.U, k, j)[lane + c * GLD] = unit_solve(sA, rfma(-__ldcg(p.sgn + k * GB + lane), r, a));
        return;
    }
    task -= rest;
    if (task < rest) {
        const int i = k + 1 + task;                            // L_ik U_kk = A1_ik, row c
        const double a = a1_at(p, i * GB + c, k * GB + lane, k);
        load_unit(sA, p.M, UF_U);
        __syncthreads();
        blk(p.L, i, k)[c + lane * GLD] = unit_solve(sA, a) * uinv;
        return;
    }
    task -= rest;
    if (task < 3) {
        load_unit(sA, p.M, task == 0 ? UF_U : (task == 1 ? UF_CHOL : UF_L));
        __syncthreads();
        double y = unit_solve(sA, lane == c ? 1.0 : 0.0);      // row c of U^{-1}, R^{-1}; column c of V1^{-1}
        if (task == 0) {
            blk(p.X, k, k)[c + lane * GLD] = y * uinv;
        } else if (task == 1) {
            y *= rinv;
            blk(p.RI, k, k)[c + lane * GLD] = y;
            // the row is scaled by the norm of column b0 + c of the panel
            if (!(y * y * __ldcg(p.gd + k * GB + c) <= kGramBound2)) *(volatile int *)p.flag = 1;
        } else {
            blk(p.LI, k, k)[lane + c * GLD] = y;
        }
        return;
    }
    const int e = task - 3, l = e / 3, what = e % 3;
    if (what < 2) {
        const double a = __ldcg(blk(what == 0 ? p.U : p.R, l, k) + c + lane * GLD);   // row c
        load_unit(sA, p.M, what == 0 ? UF_U : UF_CHOL);
        __syncthreads();
        (what == 0 ? p.YX : p.YR)[l * GB + c + lane * GLD] = unit_solve(sA, a) * (what == 0 ? uinv : rinv);
        return;
    }
    Tile tl{sA, sB, warp, lane};
    double acc = 0.0;
    for (int j = l; j < k; ++j) {
        __syncthreads();
        tl.load_a(blk(p.L, k, j), false);
        tl.load_b(blk(p.LI, j, l) + c0 * GLD);
        __syncthreads();
        acc = tl.dot(acc);
    }
    p.YL[l * GB + lane + c * GLD] = acc;                       // Y_l: block row l of a w x 32 array
}

// Trailing blocks of G (upper) and A1, then for l < k: X_lk = -sum X_lj YX_j,
// RI_lk = -sum RI_lj YR_j, LI_kl = -LI_kk YL_l.
template <class Real>
__global__ void __launch_bounds__(GT) gram_trail_kernel(const GramArgs<Real> p, int k) {
    __shared__ double sA[GB][GB + 1], sB[4][GB];
    if (*(volatile int *)p.flag) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Tile tl{sA, sB, warp, lane};
    const int c0 = (blockIdx.x & 7) * 4, rest = p.nblk - k - 1, c = c0 + warp;
    int task = blockIdx.x >> 3;
    if (task < 2 * rest * rest) {
        const bool lu = task >= rest * rest;
        if (lu) task -= rest * rest;
        const int i = k + 1 + task % rest, j = k + 1 + task / rest;
        if (!lu && i > j) return;
        tl.load_a(lu ? blk(p.L, i, k) : blk(p.R, k, i), !lu);
        tl.load_b(blk(lu ? p.U : p.R, k, j) + c0 * GLD);
        const double old = lu ? a1_at(p, i * GB + lane, j * GB + c, k) : g_at(p, i * GB + lane, j * GB + c, k);
        __syncthreads();
        blk(lu ? p.A1 : p.G, i, j)[lane + c * GLD] = old - tl.dot(0.0);
        return;
    }
    const int e = task - 2 * rest * rest, l = e / 3, what = e % 3;
    double acc = 0.0;
    if (what == 2) {
        tl.load_a(blk(p.LI, k, k), false);
        tl.load_b(p.YL + l * GB + c0 * GLD);
        __syncthreads();
        blk(p.LI, k, l)[lane + c * GLD] = -tl.dot(0.0);
        return;
    }
    const double *M = what == 0 ? p.X : p.RI, *Y = what == 0 ? p.YX : p.YR;
    for (int j = l; j < k; ++j) {
        __syncthreads();
        tl.load_a(blk(M, l, j), false);
        tl.load_b(Y + j * GB + c0 * GLD);
        __syncthreads();
        acc = tl.dot(acc);
    }
    blk(what == 0 ? p.X : p.RI, l, k)[lane + c * GLD] = -acc;
    if (what == 1 && !(acc * acc * __ldcg(p.gd + l * GB + lane) <= kGramBound2)) *(volatile int *)p.flag = 1;
}

// Z = X T = -R+^{-1} S V1^{-T} (step 0), then T = U Z, the top block of Y = V T
// = (A - [R; 0]) Z and V1 \\ R over the panel's top block (step 1).  A CTA
// takes 32 x 2 outputs of block (i, j), a warp one column and the even or odd
// 32-wide steps; all operands are staged at once.  blockIdx.x = block * 16 +
// column pair, blockIdx.y = 1: Y.
template <class Real>
__global__ void __launch_bounds__(GT) gram_t_kernel(const GramArgs<Real> p, int step) {
    __shared__ double sA[4][GB][GB + 1], sB[2][4 * GB], part[2][GB];
    if (*(volatile int *)p.flag) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, col = warp & 1, half = warp >> 1;
    const int c0 = (blockIdx.x & 15) * 2, c = c0 + col, task = blockIdx.x >> 4;
    const bool top = blockIdx.y == 1;
    const int i = task % p.nblk, j = task / p.nblk, l0 = top ? 0 : i;
    const int gi = i * GB + lane, gj = j * GB + c;
    double acc = 0.0;
    if (l0 <= j) {
        const double *A = step == 0 ? p.RI : (top ? p.B1 : p.U);
        for (int l = l0; l <= j; ++l) {
#pragma unroll
            for (int q = 0; q < GB / 4; ++q) sA[l - l0][warp + 4 * q][lane] = __ldcg(blk(A, i, l) + lane + (warp + 4 * q) * GLD);
            // step 0: (S V1^{-T})(l, j) = S_l LI(j, l)^T; step 1: Z block (l, j)
            if (half == ((l - l0) & 1))
                sB[col][(l - l0) * GB + lane] =
                    step == 0 ? __ldcg(p.sgn + l * GB + lane) * __ldcg(blk(p.LI, j, l) + c + lane * GLD)
                              : __ldcg(blk(p.Z, l, j) + lane + c * GLD);
        }
        __syncthreads();
        double a0 = 0.0, a1 = 0.0;
        for (int l = half; l <= j - l0; l += 2)
#pragma unroll
            for (int kk = 0; kk < GB; kk += 2) {
                a0 = rfma(sA[l][kk][lane], sB[col][l * GB + kk], a0);
                a1 = rfma(sA[l][kk + 1][lane], sB[col][l * GB + kk + 1], a1);
            }
        acc = a0 + a1;
        if (half) part[col][lane] = acc;
        __syncthreads();
        if (half) return;
        acc += part[col][lane];
    } else if (half) {
        return;
    }
    if (step == 0) {
        blk(p.Z, i, j)[lane + c * GLD] = i <= j ? -acc : 0.0;
        if (p.Y) {
            const double a = a1_at(p, gi, gj, 0);
            blk(p.B1, i, j)[lane + c * GLD] = gi <= gj ? rfma(-__ldcg(p.sgn + gi), __ldcg(p.R + gi + gj * GLD), a) : a;
        }
        return;
    }
    if (gi >= p.w || gj >= p.w) return;
    if (top) {
        p.Y[gi + (int64_t)gj * p.ldy] = (Real)acc;
        return;
    }
    p.Tout[gi + (int64_t)gj * p.ldt] = gi <= gj ? (Real)acc : Real(0);
    p.A[gi + (int64_t)gj * p.lda] =
        (Real)(gi <= gj ? __ldcg(p.sgn + gi) * __ldcg(p.R + gi + gj * GLD) : __ldcg(p.L + gi + gj * GLD));
}

}  // namespace

size_t gram_work_elems() { return (size_t)13 * GLD * GLD + 3 * GB * GB + 2 * GB + 4 * GLD; }

namespace {

// Scratch of one panel: the digits of P (later of A2), of X and Z, and the
// partials of the Gram matrix's split.
struct GramScratch { size_t p, xz, total; };
GramScratch gram_scratch(int D, int64_t m, int64_t w, bool with_y) {
    GramScratch s;
    s.p = std::max(oz_digit_bytes(D, w, m, kOzTileA), oz_digit_bytes(D, m, w, kOzTileA));
    s.xz = oz_digit_bytes(D, w, w, kOzTileB) * (with_y ? 2 : 1);
    const size_t splits = std::min<size_t>(oz_ktiles(m), 128);
    s.total = s.p + std::max(s.xz, splits * w * w * 8);
    return s;
}

}  // namespace

template <class Real>
size_t gram_scratch_bytes(int64_t m, int64_t w) { return gram_scratch(oz_digits<Real>(), m, w, true).total; }
template size_t gram_scratch_bytes<double>(int64_t, int64_t);
template size_t gram_scratch_bytes<float>(int64_t, int64_t);

template <class Real>
bool gram_qr_fits(const OzScratch &oz, int64_t m, int64_t w) {
    return w >= kGramMinW && w <= kGramMaxW && m >= 4 * w && m <= (1 << 30) && oz.base &&
           gram_scratch(oz_digits<Real>(), m, w, true).total <= oz.bytes;
}
template bool gram_qr_fits<double>(const OzScratch &, int64_t, int64_t);
template bool gram_qr_fits<float>(const OzScratch &, int64_t, int64_t);

template <class Real>
gbqr_status gram_qr(const Exec &ex, int64_t m, int64_t w, Real *A, int64_t lda, Real *T, int64_t ldt, Real *Y, int64_t ldy,
                    double *work, int *flag, const OzScratch &oz) {
    constexpr int D = oz_digits<Real>();
    GramArgs<Real> p{};
    p.A = A; p.lda = lda; p.Tout = T; p.ldt = ldt; p.Y = Y; p.ldy = ldy;
    p.w = (int)w; p.nblk = (int)((w + GB - 1) / GB);
    double **slots[] = {&p.G, &p.R, &p.RI, &p.A1, &p.L, &p.U, &p.LI, &p.X, &p.YX, &p.YR, &p.YL, &p.B1, &p.Z};
    double *at = work;
    for (double **s : slots) { *s = at; at += (size_t)GLD * GLD; }
    p.M = at;
    p.sc = p.M + 3 * GB * GB;
    p.sgn = p.sc + 2 * GB;
    p.gd = p.sgn + GLD;
    p.flag = flag;
    p.kexp = (int *)(p.gd + GLD);
    const GramScratch sc = gram_scratch(D, m, w, Y != nullptr);
    if (sc.total > oz.bytes) return GBQR_ENOMEM;
    char *base = (char *)oz.base;
    // G = P^T P
    OzOperand<Real> pc = oz_operand(D, (const Real *)A, lda, w, m, false, MASK_NONE, kOzTileA, base);
    TRY_ST(oz_slice(ex, D, &pc, 1));
    OzMmaArgs<Real> g{};
    g.prob[0] = oz_problem<Real>(pc, pc);
    g.prob[0].partial = (long long *)(base + sc.p);
    g.prob[0].Cd = p.G;
    g.prob[0].ldc = GLD;
    if (!oz_choose_split(g.prob[0], ex.num_sms, sc.total - sc.p, true)) return GBQR_ENOMEM;
    g.n = 1;
    g.items = oz_items((int)w, (int)w, g.prob[0].S);
    g.err = oz.err;
    TRY_ST(oz_mma_launch(ex, g, (double)w * w * m));
    TRY_ST(oz_reduce_launch(ex, g, (size_t)w * w));
    auto mark = [&](double flops) { return trace_end(ex, FAM_OTHER, flops, 0.0); };
    const double f3 = 2.0 * GB * GB * GB;
    for (int k = 0; k < p.nblk; ++k) {
        trace_begin(ex, FAM_OTHER);
        gram_diag_kernel<Real><<<1, kThreads, 0, ex.stream>>>(p, k);
        TRY_ST(mark(f3));
        const int rest = p.nblk - k - 1, row = 2 * rest + 3 + 3 * k, trail = 2 * rest * rest + 3 * k;
        trace_begin(ex, FAM_OTHER);
        gram_row_kernel<Real><<<row * 8, GT, 0, ex.stream>>>(p, k);
        TRY_ST(mark(row * f3));
        if (trail) {
            trace_begin(ex, FAM_OTHER);
            gram_trail_kernel<Real><<<trail * 8, GT, 0, ex.stream>>>(p, k);
            TRY_ST(mark(trail * f3));
        }
    }
    for (int step = 0; step < 2; ++step) {
        trace_begin(ex, FAM_OTHER);
        gram_t_kernel<Real><<<dim3(p.nblk * p.nblk * 16, step == 1 && Y ? 2 : 1), GT, 0, ex.stream>>>(p, step);
        TRY_ST(mark(p.nblk * p.nblk * f3));
    }
    if (m > w) {
        // V2 = A2 X in place (the digits of A2 are taken before C is written)
        // and Y2 = A2 Z; columns of A2 may differ by any scale, so may the
        // rows of X and Z: kexp
        OzOperand<Real> a2 = oz_operand(D, (const Real *)(A + w), lda, m - w, w, true, MASK_NONE, kOzTileA, base);
        OzOperand<double> xz[2];
        const size_t xb = oz_digit_bytes(D, w, w, kOzTileB);
        xz[0] = oz_operand(D, (const double *)p.X, GLD, w, w, false, MASK_UPPER, kOzTileB, base + sc.p);
        xz[1] = oz_operand(D, (const double *)p.Z, GLD, w, w, false, MASK_UPPER, kOzTileB, base + sc.p + xb);
        a2.skip = xz[0].skip = xz[1].skip = flag;
        a2.kexp = xz[0].kexp = xz[1].kexp = p.kexp;
        a2.ksign = -1;
        xz[0].ksign = xz[1].ksign = 1;
        const int nb = Y ? 2 : 1;
        if constexpr (std::is_same<Real, double>::value) {
            OzOperand<double> ops[3] = {a2, xz[0], xz[1]};
            TRY_ST(oz_slice(ex, D, ops, 1 + nb));
        } else {
            TRY_ST(oz_slice(ex, D, &a2, 1));
            TRY_ST(oz_slice(ex, D, xz, nb));
        }
        OzMmaArgs<Real> v{};
        for (int q = 0; q < nb; ++q) {
            v.prob[q] = oz_problem<Real>(a2, xz[q]);
            v.prob[q].C = q == 0 ? A + w : Y + w;
            v.prob[q].ldc = q == 0 ? lda : ldy;
            v.prob[q].first = v.items;
            v.items += oz_items((int)(m - w), (int)w, 1);
        }
        v.n = nb;
        v.err = oz.err;
        TRY_ST(oz_mma_launch(ex, v, (double)nb * w * w * (m - w)));
    }
    return GBQR_OK;
}
template gbqr_status gram_qr(const Exec &, int64_t, int64_t, double *, int64_t, double *, int64_t, double *, int64_t,
                             double *, int *, const OzScratch &);
template gbqr_status gram_qr(const Exec &, int64_t, int64_t, float *, int64_t, float *, int64_t, float *, int64_t,
                             double *, int *, const OzScratch &);

}  // namespace gbqr
