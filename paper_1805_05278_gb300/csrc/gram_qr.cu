// Householder QR of a well-conditioned m x w panel (w <= 128, m >= 4 w) from
// its Gram matrix, the fast base case of QR-EG in FP64 and FP32.
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
// condition).  So it is taken only where the condition allows: no column may
// be nearly a combination of the others (gram_bound).  Then orthogonality and
// backward error are at or below the TSQR's, and V, T and R agree with its to
// rounding.  Otherwise a device flag is raised, the panel is left untouched,
// and the launch that the caller puts behind (panel_chain.cu), which returns at
// once while the flag is zero, factors it.
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
// columns' FP64 issue delaying the chain; without them 33 us.  A 32^3 product
// on one SM would take 9 us, so row and trail spread every block over 8 CTAs;
// a triangular solve with a unit diagonal is 32 shuffles and multiply-adds,
// no longer than a product with the inverse.
#include "oz.cuh"
#include "tsqr_dev.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <new>
#include <type_traits>
#include <vector>

namespace gbqr {
namespace {

constexpr int GB = 32;               // block width
constexpr int GLD = kGramMaxW;       // leading dimension of every w x w array
constexpr int GT = 128;              // threads of the row / trail kernels: 32 x 4 outputs

// Largest accepted g_ii (G^-1)_ii = sum_j (R^-1)_ij^2 g_ii of a panel of w
// columns: how far column i's part orthogonal to all the others is below its
// length, squared (1 for orthogonal columns).  The loss of orthogonality grows
// with it and with the number of columns that share a direction.  FP64: at
// sqrt(360 / w) - 1.7 for 128 columns, 2.4 for 64, 4.7 for 16 - it is below
// Householder's for every kind of columns tried (a common mean, a common
// factor, chains and pairs of correlated ones; at 2 and 128 columns with a
// mean it is 1.3 times Householder's, at 16 thirty times), and no panel of
// Gaussian columns with 4 rows a column is refused (1.55 the largest of 100
// at 128, 2.2 of 300 at 16).  FP32: the same in FP64 costs no accuracy up to 16.
template <class Real>
double gram_bound(int w) { return sizeof(Real) == 8 ? std::sqrt(360.0 / w) : 16.0; }

// Squared column norms a panel may have.  The factorizations multiply two
// entries of the Gram matrix (fourth powers of the norms), and what such a
// product loses to underflow has to lie below the rounding of the smallest:
// at 2^-250 the norms 2^-75 of it do.  FP32: R's entries stay finite.
constexpr double kGramLeast = 0x1p-500;
template <class Real> __device__ constexpr double gram_most() { return sizeof(Real) == 8 ? 0x1p500 : 0x1p250; }

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
    int raise;                       // what an ill-conditioned panel writes to *flag
    int keep;                        // batch: *flag is the matrix's, clear at the start; a raised one skips the rest
    int tb;                          // batch: T's blocks of width tb alone (0: the whole T)
    double bound;                    // gram_bound()
};

// The panels of one launch: by value, or (blockIdx.y: which) a list in device memory.
template <class Real>
struct GramList {
    GramArgs<Real> one;
    const GramArgs<Real> *list;
};
template <class Real>
__device__ __forceinline__ const GramArgs<Real> &nth_panel(const GramList<Real> &g) {
    return g.list ? g.list[blockIdx.y] : g.one;
}

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

// Whether the panel was given up: read once for the whole CTA, since another
// CTA of the same launch (of gram_t's first step) may raise the flag meanwhile,
// and threads of one CTA that saw different values would part ahead of a barrier.
template <class Real>
__device__ __forceinline__ bool given_up(const GramArgs<Real> &p) {
    return __syncthreads_or(threadIdx.x == 0 && *(volatile int *)p.flag);
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
__global__ void __launch_bounds__(kThreads) gram_diag_kernel(const __grid_constant__ GramList<Real> args, int k) {
    __shared__ double S[GB][GB + 1], Rb[GB][GB + 1];     // [column][row]; Rb: R(row, column)
    __shared__ double cb[2][GB], ub[2][GB], rb[2], rd[GB], sg[GB];
    __shared__ int bad;
    const GramArgs<Real> p = nth_panel(args);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, b0 = k * GB;
    if (k >= p.nblk || ((k > 0 || p.keep) && *(volatile int *)p.flag)) return;
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
        // (the pivot's own share of the sum that gram_t bounds: most panels that
        // will not do stop here)
        const double d = S[lane][lane];
        if (!(d > kGramLeast && d < gram_most<Real>() && d * p.bound >= __ldcg(p.gd + b0 + lane))) bad = 1;
        const double s = sqrt(d);
        sg[lane] = s;
        p.sc[lane] = s * rd[lane];                       // 1 / r_tt
    }
    __syncthreads();
    if (bad) {
        if (tid == 0) *p.flag = p.raise;
        return;
    }
    if (k == 0 && tid == 0 && !p.keep) *p.flag = 0;
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
__global__ void __launch_bounds__(GT) gram_row_kernel(const __grid_constant__ GramList<Real> args, int k) {
    __shared__ double sA[GB][GB + 1], sB[4][GB];
    const GramArgs<Real> p = nth_panel(args);
    if (k >= p.nblk || *(volatile int *)p.flag) return;
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
            blk(p.RI, k, k)[c + lane * GLD] = y * rinv;
        } else {
            blk(p.LI, k, k)[lane + c * GLD] = y;
        }
        return;
    }
    const int e = task - 3, l = e / 3, what = e % 3;
    if (l >= k) return;
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
__global__ void __launch_bounds__(GT) gram_trail_kernel(const __grid_constant__ GramList<Real> args, int k) {
    __shared__ double sA[GB][GB + 1], sB[4][GB];
    const GramArgs<Real> p = nth_panel(args);
    if (k >= p.nblk || *(volatile int *)p.flag) return;
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
    if (l >= k) return;
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
}

// Z = X T = -R+^{-1} S V1^{-T} and the condition check (step 0), then T = U Z, the top block of Y = V T
// = (A - [R; 0]) Z and V1 \\ R over the panel's top block (step 1).  A CTA
// takes 32 x 2 outputs of block (i, j), a warp one column and the even or odd
// 32-wide steps; all operands are staged at once.  blockIdx.x = block * 16 +
// column pair, blockIdx.z = 1: Y.
template <class Real>
__global__ void __launch_bounds__(GT) gram_t_kernel(const __grid_constant__ GramList<Real> args, int step) {
    __shared__ double sA[4][GB][GB + 1], sB[2][4 * GB], part[4][GB];
    const GramArgs<Real> p = nth_panel(args);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, col = warp & 1, half = warp >> 1;
    const int c0 = (blockIdx.x & 15) * 2, c = c0 + col, task = blockIdx.x >> 4;
    const bool top = blockIdx.z == 1;
    if (task >= p.nblk * p.nblk || (top && !p.Y) || given_up(p)) return;
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
        if (step == 0 && j == p.nblk - 1 && c0 == 0) {
            // block row i of R^{-1} is here whole: rows' sums of squares, times g_ii
            double q = 0.0;
            for (int l = 0; l <= j - i; ++l)
#pragma unroll
                for (int kk = 0; kk < GB; kk += 4) q = rfma(sA[l][kk + warp][lane], sA[l][kk + warp][lane], q);
            part[warp][lane] = q;
            __syncthreads();
            q = part[0][lane] + part[1][lane] + part[2][lane] + part[3][lane];
            if (warp == 0 && !(q * __ldcg(p.gd + gi) <= p.bound)) *(volatile int *)p.flag = p.raise;
            __syncthreads();
        }
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
    if (gj >= p.w) return;
    if (p.tb && !top && gi / p.tb == gj / p.tb)        // rows past the last block's width are zeroed too
        p.Tout[gi % p.tb + (int64_t)gj * p.ldt] = gi <= gj && gi < p.w ? (Real)acc : Real(0);
    if (gi >= p.w) return;
    if (top) {
        p.Y[gi + (int64_t)gj * p.ldy] = (Real)acc;
        return;
    }
    if (!p.tb) p.Tout[gi + (int64_t)gj * p.ldt] = gi <= gj ? (Real)acc : Real(0);
    p.A[gi + (int64_t)gj * p.lda] =
        (Real)(gi <= gj ? __ldcg(p.sgn + gi) * __ldcg(p.R + gi + gj * GLD) : __ldcg(p.L + gi + gj * GLD));
}

}  // namespace

namespace {

// Points p's arrays into `work` (gram_work_elems() doubles).
template <class Real>
void gram_carve(GramArgs<Real> &p, double *work) {
    double **slots[] = {&p.G, &p.R, &p.RI, &p.A1, &p.L, &p.U, &p.LI, &p.X, &p.YX, &p.YR, &p.YL, &p.B1, &p.Z};
    double *at = work;
    for (double **s : slots) { *s = at; at += (size_t)GLD * GLD; }
    p.M = at;
    p.sc = p.M + 3 * GB * GB;
    p.sgn = p.sc + 2 * GB;
    p.gd = p.sgn + GLD;
    p.kexp = (int *)(p.gd + GLD);
}

int gram_row_blocks(int nblk, int k) { return (2 * (nblk - k - 1) + 3 + 3 * k) * 8; }
int gram_trail_blocks(int nblk, int k) { return (2 * (nblk - k - 1) * (nblk - k - 1) + 3 * k) * 8; }

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
    // a split has at most 16 K tiles (512 rows), and up to 128 splits fill the GPU
    const size_t kt = oz_ktiles(m), splits = std::max<size_t>(std::min<size_t>(kt, 128), (kt + 15) / 16);
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
    return w >= kGramMinW && w <= kGramMaxW && m >= 4 * w && m <= kOzMaxRows && oz.base &&
           gram_scratch(oz_digits<Real>(), m, w, true).total <= oz.bytes;
}
template bool gram_qr_fits<double>(const OzScratch &, int64_t, int64_t);
template bool gram_qr_fits<float>(const OzScratch &, int64_t, int64_t);

template <class Real>
gbqr_status gram_qr(const Exec &ex, int64_t m, int64_t w, Real *A, int64_t lda, Real *T, int64_t ldt, Real *Y, int64_t ldy,
                    double *work, int *flag, const OzScratch &oz) {
    constexpr int D = oz_digits<Real>();
    GramList<Real> gl{};
    GramArgs<Real> &p = gl.one;
    p.A = A; p.lda = lda; p.Tout = T; p.ldt = ldt; p.Y = Y; p.ldy = ldy;
    p.w = (int)w; p.nblk = (int)((w + GB - 1) / GB);
    gram_carve(p, work);
    p.flag = flag;
    p.raise = 1;
    p.bound = gram_bound<Real>((int)w);
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
        gram_diag_kernel<Real><<<1, kThreads, 0, ex.stream>>>(gl, k);
        TRY_ST(mark(f3));
        const int row = gram_row_blocks(p.nblk, k), trail = gram_trail_blocks(p.nblk, k);
        trace_begin(ex, FAM_OTHER);
        gram_row_kernel<Real><<<row, GT, 0, ex.stream>>>(gl, k);
        TRY_ST(mark(row / 8 * f3));
        if (trail) {
            trace_begin(ex, FAM_OTHER);
            gram_trail_kernel<Real><<<trail, GT, 0, ex.stream>>>(gl, k);
            TRY_ST(mark(trail / 8 * f3));
        }
    }
    for (int step = 0; step < 2; ++step) {
        trace_begin(ex, FAM_OTHER);
        gram_t_kernel<Real><<<dim3(p.nblk * p.nblk * 16, 1, step == 1 && Y ? 2 : 1), GT, 0, ex.stream>>>(gl, step);
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


// ------------------------------------------------------------------ batches
// The panels of many matrices in lockstep: every launch above over a list of
// panels.  A plan holds the lists of all launches as one blob whose pointers
// are offsets (into the workspace, or into a matrix's A or T); a call copies
// the blob into the workspace and relocates it there, so a plan serves any
// buffers.  Matrices go in groups whose scratch fits kGroupBytes.
namespace {

constexpr size_t kGroupBytes = (size_t)6 << 30;
constexpr int kBatchTb = 16;                     // width of a batch's T blocks
constexpr int kGroupPanels = 4;

enum RelocBase { RB_WS = 0, RB_A = 1, RB_T = 2 };
struct Reloc { uint64_t off; uint32_t word; int mat; int base; int pad; };

enum StepKind { ST_SLICE, ST_MMA, ST_REDUCE, ST_REQUANT, ST_DIAG, ST_ROW, ST_TRAIL, ST_T };
struct GroupStep {
    StepKind kind;
    size_t list = 0;          // the list's place in the blob
    int n = 0;                // its length
    int grid = 0;             // CTAs (slice), items (MMA), blocks per panel, columns (requant)
    int k = 0;                // block (diag, row, trail) or step (T)
    int z = 1;                // T: 2 where Y is wanted
    bool tall = false;
    double elems = 0.0;
};

__global__ void __launch_bounds__(256) reloc_kernel(const Reloc *r, int n, uint64_t *blob, char *ws, const char *mats,
                                                    int stride) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const Reloc x = r[i];
    uint64_t base = (uint64_t)ws;
    if (x.base != RB_WS) {
        // the matrix table starts with its pointers A and T
        double *const *p = reinterpret_cast<double *const *>(mats + (size_t)x.mat * stride);
        base = (uint64_t)p[x.base == RB_A ? 0 : 1];
    }
    blob[x.word] = base + x.off;
}

}  // namespace

// Device copies of a plan's blob and relocations.  A captured graph reads them
// at every launch, so it shares them with the plan: whichever goes last frees
// them.
struct GroupLists {
    uint8_t *blob = nullptr;
    Reloc *relocs = nullptr;
    ~GroupLists() {
        cudaFree(blob);
        cudaFree(relocs);
    }
};

struct GroupPlan {
    size_t blob_off = 0, status_off = 0, total = 0;      // workspace layout, from its start
    std::vector<uint8_t> blob;
    std::vector<Reloc> relocs;
    std::vector<GroupStep> steps;
    std::vector<int> width;                              // per matrix: its panels' width, 0 = not grouped
    double est_ms = 0.0;
    std::shared_ptr<GroupLists> lists;                   // device copies (group_plan_upload)
};

void group_plan_free(GroupPlan *g) { delete g; }
size_t group_plan_bytes(const GroupPlan *g) { return g ? g->total : 0; }
const int *group_widths(const GroupPlan *g) { return g->width.data(); }
size_t group_status_offset(const GroupPlan *g) { return g->status_off; }
double group_plan_ms(const GroupPlan *g) { return g->est_ms; }

namespace {

// The panel width of an m x n matrix: equal panels of at most 128 columns, a
// multiple of T's block width, each with 4 rows a column.  Shorter matrices
// take narrower panels, up to kGroupPanels of them; 0 beyond that.
int group_width(int64_t m, int64_t n) {
    if (n < kGramMinW || m > (1 << 28)) return 0;
    const int64_t np0 = (n + kGramMaxW - 1) / kGramMaxW;
    for (int64_t np = np0; np <= std::max<int64_t>(np0, kGroupPanels); ++np) {
        const int64_t w = ((n + np - 1) / np + kBatchTb - 1) / kBatchTb * kBatchTb;
        if (w > kGramMaxW) continue;
        bool fits = true;
        for (int64_t j = 0; j < n; j += w) fits = fits && m - j >= 4 * std::min(w, n - j);
        if (fits) return (int)w;
    }
    return 0;
}

struct GroupBuilder {
    GroupPlan *g;
    size_t arena = 0, peak = 0;
    static constexpr int D = kOzDigits64;

    static size_t al(size_t x) { return (x + 255) / 256 * 256; }
    size_t take(size_t bytes) {
        const size_t o = arena;
        arena += al(std::max<size_t>(bytes, 16));
        peak = std::max(peak, arena);
        return o;
    }
    // appends a list to the blob; fix(entry, place of the entry) adds relocations
    template <class E>
    size_t put(const std::vector<E> &v) {
        size_t at = (g->blob.size() + 255) / 256 * 256;
        g->blob.resize(at + v.size() * sizeof(E), 0);
        memcpy(g->blob.data() + at, v.data(), v.size() * sizeof(E));
        return at;
    }
    template <class F>
    void rel(size_t at, const void *entry, const F *field, int base, int mat, uint64_t off) {
        const size_t byte = at + (size_t)((const char *)field - (const char *)entry);
        g->relocs.push_back({off, (uint32_t)(byte / 8), mat, base, 0});
    }
    template <class F>
    void rel_flag(size_t at, const void *entry, const F *field, size_t flag) {
        rel(at, entry, field, RB_WS, 0, flag);
        g->relocs.back().pad = 1;                  // a place outside the arena
    }
    void places(size_t at, const OzOperand<double> &o, int base, int mat, uint64_t x, size_t digits, int64_t R, int64_t K,
                size_t flag, size_t kexp) {
        rel(at, &o, &o.X, base, mat, x);
        rel(at, &o, &o.dst, RB_WS, 0, digits);
        rel(at, &o, &o.exps, RB_WS, 0, exps_of(digits, R, K, o.rt));
        rel_flag(at, &o, &o.skip, flag);
        if (kexp) rel(at, &o, &o.kexp, RB_WS, 0, kexp);
    }
    size_t exps_of(size_t digits, int64_t R, int64_t K, int rt) const {
        return digits + oz_digit_bytes(D, R, K, rt) - al((size_t)R * 4);
    }
};

// Arena of one panel of one matrix, in bytes from the workspace's start.
struct PanelPlaces { size_t work, p, x, z, part, y, vd, yd, c, wd, wf; };

}  // namespace

GroupPlan *group_plan_build(int count, const int64_t *m, const int64_t *n, const int64_t *lda, const int64_t *ldt,
                            int num_sms, size_t ws_off) {
    std::vector<int> mats;
    std::vector<int> width(count, 0);
    constexpr int D = kOzDigits64;
    const size_t work_bytes = gram_work_elems() * 8;
    // scratch of matrix i (its first panel is its largest)
    auto need = [&](int i) {
        const int64_t w = std::min<int64_t>(width[i], n[i]), nc = n[i] - w;
        const size_t splits = oz_ktiles(m[i]);
        size_t s = work_bytes + std::max(oz_digit_bytes(D, w, m[i], kOzTileA), oz_digit_bytes(D, m[i], w, kOzTileA)) +
                   2 * oz_digit_bytes(D, w, w, kOzTileB) + std::max(std::min<size_t>(splits, 40), splits / 16 + 1) * w * w * 8;
        if (nc > 0)
            s += (size_t)m[i] * w * 8 + oz_digit_bytes(D, m[i], w, kOzTileA) + oz_digit_bytes(D, w, m[i], kOzTileA) +
                 oz_digit_bytes(D, nc, m[i], kOzTileB) + oz_digit_bytes(D, nc, w, kOzTileB) + (size_t)w * nc * 8 +
                 (splits / 16 + 1) * w * nc * 8;
        return s + 16 * 256;
    };
    for (int i = 0; i < count; ++i) {
        width[i] = group_width(m[i], n[i]);
        if (width[i] && need(i) > kGroupBytes) width[i] = 0;       // a group of its own would not hold it
        if (width[i]) mats.push_back(i);
    }
    if (mats.empty()) return nullptr;
    GroupPlan *g = new (std::nothrow) GroupPlan();
    if (!g) return nullptr;
    g->width = width;
    GroupBuilder b{g};
    g->status_off = GroupBuilder::al(ws_off);
    // the arena's place depends on the blob's size: offsets are relative to
    // the arena while building, and shifted at the end
    auto flag_of = [&](int i) { return g->status_off + (size_t)i * 4; };
    size_t at = 0;
    while (at < mats.size()) {
        size_t end = at, bytes = 0;
        while (end < mats.size() && bytes + need(mats[end]) <= kGroupBytes && end - at < 60000) bytes += need(mats[end++]);
        int64_t panels = 0;
        for (size_t q = at; q < end; ++q) panels = std::max<int64_t>(panels, (n[mats[q]] + width[mats[q]] - 1) / width[mats[q]]);
        // a panel's chain, and 4 TFLOP/s: 200 of 2000 x 128 take 4.5 ms, the
        // 2000 benchmark matrices (351 GFLOP) 109
        g->est_ms += 0.4 * panels;
        for (size_t q = at; q < end; ++q) {
            const double mm = (double)m[mats[q]], nn = (double)n[mats[q]];
            g->est_ms += (2.0 * mm * nn * nn - 2.0 / 3.0 * nn * nn * nn) / 4e9;
        }
        for (int64_t pn = 0; pn < panels; ++pn) {
            b.arena = 0;
            std::vector<int> act;
            for (size_t q = at; q < end; ++q)
                if ((int64_t)width[mats[q]] * pn < n[mats[q]]) act.push_back(mats[q]);
            const int na = (int)act.size();
            std::vector<PanelPlaces> pl(na);
            std::vector<OzOperand<double>> sp(na), sa, sv, sx;
            std::vector<OzProblem<double>> pg(na), pv, p1, p2;
            std::vector<GramArgs<double>> ga(na);
            std::vector<int> trailing;
            auto W = [&](int i) { return std::min<int64_t>(width[i], n[i] - width[i] * pn); };
            auto J = [&](int i) { return (int64_t)width[i] * pn; };
            auto M = [&](int i) { return m[i] - J(i); };
            auto NC = [&](int i) { return n[i] - J(i) - W(i); };
            auto Aoff = [&](int i, int64_t r, int64_t c) { return (uint64_t)((r + c * lda[i]) * 8); };
            for (int q = 0; q < na; ++q) {
                const int i = act[q];
                PanelPlaces &s = pl[q];
                s.work = b.take(work_bytes);
                s.p = b.take(std::max(oz_digit_bytes(D, W(i), M(i), kOzTileA), oz_digit_bytes(D, M(i), W(i), kOzTileA)));
                s.x = b.take(oz_digit_bytes(D, W(i), W(i), kOzTileB));
                s.z = b.take(oz_digit_bytes(D, W(i), W(i), kOzTileB));
                if (NC(i) > 0) {
                    trailing.push_back(q);
                    s.y = b.take((size_t)M(i) * W(i) * 8);
                    s.vd = b.take(oz_digit_bytes(D, M(i), W(i), kOzTileA));
                    s.yd = b.take(oz_digit_bytes(D, W(i), M(i), kOzTileA));
                    s.c = b.take(oz_digit_bytes(D, NC(i), M(i), kOzTileB));
                    s.wd = b.take(oz_digit_bytes(D, NC(i), W(i), kOzTileB));
                    s.wf = b.take((size_t)W(i) * NC(i) * 8);
                }
            }
            // ---- digits of P, G = P^T P
            bool tall = false;
            unsigned blocks = 0;
            int items = 0;
            size_t largest = 0;
            double elems = 0.0, prods = 0.0;
            for (int i : act) tall = tall || M(i) > 8192;
            for (int q = 0; q < na; ++q) {
                const int i = act[q];
                sp[q] = oz_operand(D, (const double *)nullptr, lda[i], W(i), M(i), false, MASK_NONE, kOzTileA, nullptr);
                sp[q].first = blocks;
                blocks += oz_slice_blocks(sp[q], tall);
                elems += (double)W(i) * M(i);
                pg[q] = oz_problem<double>(sp[q], sp[q]);
                // a full GPU of matrices needs no fine splits: 512 k an item
                pg[q].kt_per = std::max(1, std::min(pg[q].KT, 16));
                if (na < num_sms) pg[q].kt_per = std::max(1, std::min(pg[q].kt_per, (pg[q].KT * na + num_sms - 1) / num_sms));
                pg[q].kt_per = std::max(pg[q].kt_per, std::min((pg[q].KT + 39) / 40, oz_max_ktiles<double>()));
                pg[q].S = (pg[q].KT + pg[q].kt_per - 1) / pg[q].kt_per;
                pg[q].ldc = GLD;
                pg[q].first = items;
                items += oz_items((int)W(i), (int)W(i), pg[q].S);
                largest = std::max(largest, (size_t)W(i) * W(i));
                prods += (double)W(i) * W(i) * M(i);
                pl[q].part = b.take((size_t)pg[q].S * W(i) * W(i) * 8);
                GramArgs<double> &p = ga[q];
                p = GramArgs<double>{};
                p.lda = lda[i]; p.ldt = ldt[i]; p.ldy = M(i);
                p.w = (int)W(i); p.nblk = (int)((W(i) + GB - 1) / GB);
                p.raise = 1 + (int)pn; p.keep = 1; p.tb = kBatchTb;
                p.bound = gram_bound<double>(p.w);
            }
            size_t L = b.put(sp);
            for (int q = 0; q < na; ++q) {
                const int i = act[q];
                const size_t e = L + q * sizeof(sp[0]);
                b.places(e, sp[q], RB_A, i, Aoff(i, J(i), J(i)), pl[q].p, W(i), M(i), flag_of(i), 0);
            }
            g->steps.push_back({ST_SLICE, L, na, (int)blocks, 0, 1, tall, elems});
            L = b.put(pg);
            const size_t gram_list = b.put(ga);
            for (int q = 0; q < na; ++q) {
                const int i = act[q];
                const size_t e = L + q * sizeof(pg[0]);
                const OzProblem<double> &p = pg[q];
                b.rel(e, &p, &p.a, RB_WS, 0, pl[q].p);
                b.rel(e, &p, &p.b, RB_WS, 0, pl[q].p);
                b.rel(e, &p, &p.ea, RB_WS, 0, b.exps_of(pl[q].p, W(i), M(i), kOzTileA));
                b.rel(e, &p, &p.eb, RB_WS, 0, b.exps_of(pl[q].p, W(i), M(i), kOzTileA));
                b.rel(e, &p, &p.partial, RB_WS, 0, pl[q].part);
                b.rel_flag(e, &p, &p.skip, flag_of(i));
                // the panel's arrays: carved from a null base, so that the fields hold their offsets
                GramArgs<double> c = ga[q];
                gram_carve(c, (double *)nullptr);
                b.rel(e, &p, &p.Cd, RB_WS, 0, pl[q].work + (size_t)(char *)c.G);
                const size_t ge = gram_list + q * sizeof(ga[0]);
                const GramArgs<double> &a = ga[q];
                double *GramArgs<double>::*const f[] = {&GramArgs<double>::G, &GramArgs<double>::R, &GramArgs<double>::RI, &GramArgs<double>::A1,
                    &GramArgs<double>::L, &GramArgs<double>::U, &GramArgs<double>::LI, &GramArgs<double>::X, &GramArgs<double>::YX, &GramArgs<double>::YR,
                    &GramArgs<double>::YL, &GramArgs<double>::B1, &GramArgs<double>::Z, &GramArgs<double>::sgn, &GramArgs<double>::gd,
                    &GramArgs<double>::M, &GramArgs<double>::sc};
                for (auto fp : f) b.rel(ge, &a, &(a.*fp), RB_WS, 0, pl[q].work + (size_t)(char *)(c.*fp));
                b.rel(ge, &a, &a.kexp, RB_WS, 0, pl[q].work + (size_t)(char *)c.kexp);
                b.rel_flag(ge, &a, &a.flag, flag_of(i));
                b.rel(ge, &a, &a.A, RB_A, i, Aoff(i, J(i), J(i)));
                b.rel(ge, &a, &a.Tout, RB_T, i, (uint64_t)(J(i) * ldt[i] * 8));
                if (NC(i) > 0) b.rel(ge, &a, &a.Y, RB_WS, 0, pl[q].y);
            }
            g->steps.push_back({ST_MMA, L, na, items, 0, 1, false, prods});
            g->steps.push_back({ST_REDUCE, L, na, (int)((largest + kThreads - 1) / kThreads), 0, 1, false, 0.0});
            int nblk = 1;
            for (auto &p : ga) nblk = std::max(nblk, p.nblk);
            for (int k = 0; k < nblk; ++k) {
                int row = 0, trail = 0;
                for (auto &p : ga)
                    if (k < p.nblk) {
                        row = std::max(row, gram_row_blocks(p.nblk, k));
                        trail = std::max(trail, gram_trail_blocks(p.nblk, k));
                    }
                g->steps.push_back({ST_DIAG, gram_list, na, 1, k, 1, false, 0.0});
                g->steps.push_back({ST_ROW, gram_list, na, row, k, 1, false, 0.0});
                if (trail) g->steps.push_back({ST_TRAIL, gram_list, na, trail, k, 1, false, 0.0});
            }
            for (int k = 0; k < 2; ++k)
                g->steps.push_back({ST_T, gram_list, na, nblk * nblk * 16, k, k == 1 && !trailing.empty() ? 2 : 1, false, 0.0});
            // ---- digits of A2, X, Z; V2 = A2 X, Y2 = A2 Z
            blocks = 0;
            unsigned xblocks = 0;
            items = 0;
            elems = prods = 0.0;
            double xelems = 0.0;
            struct Fix { int q; int what; };   // what: 0 A2, 1 X, 2 Z
            std::vector<Fix> fa, fx, fv;
            auto place_of = [&](int q, int what) { return what == 0 ? pl[q].p : (what == 1 ? pl[q].x : pl[q].z); };
            for (int q = 0; q < na; ++q) {
                const int i = act[q];
                if (M(i) <= W(i)) continue;
                OzOperand<double> a2 = oz_operand(D, (const double *)nullptr, lda[i], M(i) - W(i), W(i), true, MASK_NONE, kOzTileA, nullptr);
                a2.ksign = -1;
                a2.first = blocks;
                blocks += oz_slice_blocks(a2, false);
                elems += (double)(M(i) - W(i)) * W(i);
                sa.push_back(a2);
                fa.push_back({q, 0});
                for (int y = 0; y < (NC(i) > 0 ? 2 : 1); ++y) {
                    OzOperand<double> x = oz_operand(D, (const double *)nullptr, GLD, W(i), W(i), false, MASK_UPPER, kOzTileB, nullptr);
                    x.ksign = 1;
                    x.first = xblocks;
                    xblocks += oz_slice_blocks(x, false);
                    xelems += (double)W(i) * W(i);
                    sx.push_back(x);
                    fx.push_back({q, 1 + y});
                    OzProblem<double> p = oz_problem<double>(a2, x);
                    p.ldc = y == 0 ? lda[i] : M(i);
                    p.first = items;
                    items += oz_items((int)(M(i) - W(i)), (int)W(i), 1);
                    prods += (double)(M(i) - W(i)) * W(i) * W(i);
                    pv.push_back(p);
                    fv.push_back({q, 1 + y});
                }
            }
            if (!sa.empty()) {
                GramArgs<double> c{};
                gram_carve(c, (double *)nullptr);
                L = b.put(sa);
                for (size_t e = 0; e < sa.size(); ++e) {
                    const int q = fa[e].q, i = act[q];
                    b.places(L + e * sizeof(sa[0]), sa[e], RB_A, i, Aoff(i, J(i) + W(i), J(i)), pl[q].p, M(i) - W(i), W(i), flag_of(i),
                             pl[q].work + (size_t)(char *)c.kexp);
                }
                g->steps.push_back({ST_SLICE, L, (int)sa.size(), (int)blocks, 0, 1, false, elems});
                L = b.put(sx);
                for (size_t e = 0; e < sx.size(); ++e) {
                    const int q = fx[e].q, i = act[q];
                    b.places(L + e * sizeof(sx[0]), sx[e], RB_WS, 0, pl[q].work + (size_t)(char *)(fx[e].what == 1 ? c.X : c.Z),
                             place_of(q, fx[e].what), W(i), W(i), flag_of(i), pl[q].work + (size_t)(char *)c.kexp);
                }
                g->steps.push_back({ST_SLICE, L, (int)sx.size(), (int)xblocks, 0, 1, false, xelems});
                L = b.put(pv);
                for (size_t e = 0; e < pv.size(); ++e) {
                    const int q = fv[e].q, i = act[q];
                    const size_t pe = L + e * sizeof(pv[0]), xp = place_of(q, fv[e].what);
                    const OzProblem<double> &p = pv[e];
                    b.rel(pe, &p, &p.a, RB_WS, 0, pl[q].p);
                    b.rel(pe, &p, &p.ea, RB_WS, 0, b.exps_of(pl[q].p, M(i) - W(i), W(i), kOzTileA));
                    b.rel(pe, &p, &p.b, RB_WS, 0, xp);
                    b.rel(pe, &p, &p.eb, RB_WS, 0, b.exps_of(xp, W(i), W(i), kOzTileB));
                    b.rel_flag(pe, &p, &p.skip, flag_of(i));
                    if (fv[e].what == 1) b.rel(pe, &p, &p.C, RB_A, i, Aoff(i, J(i) + W(i), J(i)));
                    else b.rel(pe, &p, &p.C, RB_WS, 0, pl[q].y + (size_t)W(i) * 8);
                }
                g->steps.push_back({ST_MMA, L, (int)pv.size(), items, 0, 1, false, prods});
            }
            if (!trailing.empty()) {
                // ---- C -= V (Y^T C)
                blocks = 0;
                elems = prods = 0.0;
                items = 0;
                int items2 = 0, widest = 0;
                for (int q : trailing) {
                    const int i = act[q];
                    OzOperand<double> v = oz_operand(D, (const double *)nullptr, lda[i], M(i), W(i), true, MASK_UNIT_LOWER, kOzTileA, nullptr);
                    OzOperand<double> y = oz_operand(D, (const double *)nullptr, M(i), W(i), M(i), false, MASK_NONE, kOzTileA, nullptr);
                    OzOperand<double> c = oz_operand(D, (const double *)nullptr, lda[i], NC(i), M(i), false, MASK_NONE, kOzTileB, nullptr);
                    const OzOperand<double> wq = oz_operand(D, (const double *)nullptr, 1, NC(i), W(i), false, MASK_NONE, kOzTileB, nullptr);
                    for (OzOperand<double> *o : {&v, &y, &c}) {
                        o->first = blocks;
                        blocks += oz_slice_blocks(*o, tall);
                        elems += (double)o->R * o->K;
                        sv.push_back(*o);
                    }
                    OzProblem<double> p = oz_problem<double>(y, c);
                    p.kt_per = std::max(1, std::min(p.KT, 16));
                    if ((int)trailing.size() < num_sms)
                        p.kt_per = std::max(1, std::min(p.kt_per, (int)((p.KT * trailing.size() + num_sms - 1) / num_sms)));
                    p.kt_per = std::max(p.kt_per, std::min((p.KT + 39) / 40, oz_max_ktiles<double>()));
                    p.S = (p.KT + p.kt_per - 1) / p.kt_per;
                    p.ldc = W(i);
                    p.first = items;
                    items += oz_items((int)W(i), (int)NC(i), p.S);
                    pl[q].part = b.take((size_t)p.S * W(i) * NC(i) * 8);
                    p1.push_back(p);
                    widest = std::max(widest, (int)NC(i));
                    prods += (double)W(i) * NC(i) * M(i);
                    OzProblem<double> u = oz_problem<double>(v, wq);
                    u.ldc = lda[i];
                    u.alpha = -1.0;
                    u.beta = 1.0;
                    u.ldadd = W(i);
                    u.add_rows = (int)W(i);
                    u.first = items2;
                    items2 += oz_items((int)M(i), (int)NC(i), 1);
                    p2.push_back(u);
                }
                L = b.put(sv);
                const size_t L1 = b.put(p1), L2 = b.put(p2);
                for (size_t t = 0; t < trailing.size(); ++t) {
                    const int q = trailing[t], i = act[q];
                    const uint64_t ctop = Aoff(i, J(i), J(i) + W(i));
                    const size_t e = L + 3 * t * sizeof(sv[0]);
                    b.places(e, sv[3 * t], RB_A, i, Aoff(i, J(i), J(i)), pl[q].vd, M(i), W(i), flag_of(i), 0);
                    b.places(e + sizeof(sv[0]), sv[3 * t + 1], RB_WS, 0, pl[q].y, pl[q].yd, W(i), M(i), flag_of(i), 0);
                    b.places(e + 2 * sizeof(sv[0]), sv[3 * t + 2], RB_A, i, ctop, pl[q].c, NC(i), M(i), flag_of(i), 0);
                    const size_t e1 = L1 + t * sizeof(p1[0]), e2 = L2 + t * sizeof(p2[0]);
                    const OzProblem<double> &p = p1[t], &u = p2[t];
                    b.rel(e1, &p, &p.a, RB_WS, 0, pl[q].yd);
                    b.rel(e1, &p, &p.ea, RB_WS, 0, b.exps_of(pl[q].yd, W(i), M(i), kOzTileA));
                    b.rel(e1, &p, &p.b, RB_WS, 0, pl[q].c);
                    b.rel(e1, &p, &p.eb, RB_WS, 0, b.exps_of(pl[q].c, NC(i), M(i), kOzTileB));
                    b.rel(e1, &p, &p.partial, RB_WS, 0, pl[q].part);
                    b.rel_flag(e1, &p, &p.skip, flag_of(i));
                    b.rel(e1, &p, &p.C, RB_WS, 0, pl[q].wf);
                    b.rel(e1, &p, &p.qdst, RB_WS, 0, pl[q].wd);
                    b.rel(e1, &p, &p.qexp, RB_WS, 0, b.exps_of(pl[q].wd, NC(i), W(i), kOzTileB));
                    b.rel(e2, &u, &u.a, RB_WS, 0, pl[q].vd);
                    b.rel(e2, &u, &u.ea, RB_WS, 0, b.exps_of(pl[q].vd, M(i), W(i), kOzTileA));
                    b.rel(e2, &u, &u.b, RB_WS, 0, pl[q].wd);
                    b.rel(e2, &u, &u.eb, RB_WS, 0, b.exps_of(pl[q].wd, NC(i), W(i), kOzTileB));
                    b.rel_flag(e2, &u, &u.skip, flag_of(i));
                    b.rel(e2, &u, &u.add, RB_WS, 0, pl[q].wf);
                    b.rel(e2, &u, &u.C, RB_A, i, ctop);
                }
                g->steps.push_back({ST_SLICE, L, (int)sv.size(), (int)blocks, 0, 1, tall, elems});
                g->steps.push_back({ST_MMA, L1, (int)p1.size(), items, 0, 1, false, prods});
                g->steps.push_back({ST_REQUANT, L1, (int)p1.size(), widest, 0, 1, false, 0.0});
                g->steps.push_back({ST_MMA, L2, (int)p2.size(), items2, 0, 1, false, prods});
            }
        }
        at = end;
    }
    // workspace: [... | status | blob | arena]; arena offsets are shifted to
    // their place (status places are absolute already)
    g->blob_off = GroupBuilder::al(g->status_off + (size_t)count * 4);
    const size_t arena0 = GroupBuilder::al(g->blob_off + g->blob.size());
    for (Reloc &r : g->relocs)
        if (r.base == RB_WS && !r.pad) r.off += arena0;
    g->total = arena0 + b.peak;
    return g;
}

// Device copies of the plan's blob and relocations (not during a capture).
// Waits for them: the calls that read them may be on another stream.
gbqr_status group_plan_upload(GroupPlan *g, cudaStream_t stream) {
    if (!g || g->lists) return GBQR_OK;
    std::shared_ptr<GroupLists> l(new (std::nothrow) GroupLists());
    if (!l) return GBQR_ENOMEM;
    const size_t nb = g->blob.size(), nr = g->relocs.size() * sizeof(Reloc);
    if (cudaMalloc((void **)&l->blob, nb) != cudaSuccess || cudaMalloc((void **)&l->relocs, nr) != cudaSuccess) {
        cudaGetLastError();
        return GBQR_ENOMEM;
    }
    if (cudaMemcpyAsync(l->blob, g->blob.data(), nb, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
        cudaMemcpyAsync(l->relocs, g->relocs.data(), nr, cudaMemcpyHostToDevice, stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess)
        return GBQR_ECUDA;
    g->lists = std::move(l);
    return GBQR_OK;
}
std::shared_ptr<void> group_plan_lists(const GroupPlan *g) { return g->lists; }

// Enqueues the grouped factorizations; mats: the matrix table in device
// memory (A and T first).  status[i] stays 0 for a grouped matrix that is
// done, else 1 + the panel it stopped at.
gbqr_status group_enqueue(const Exec &ex, const GroupPlan *g, char *ws, const void *mats, int stride, int count, int *err) {
    if (!g->lists) return GBQR_EINVAL;
    uint8_t *blob = (uint8_t *)ws + g->blob_off;
    if (cudaMemsetAsync(ws + g->status_off, 0, (size_t)count * 4, ex.stream) != cudaSuccess ||
        cudaMemcpyAsync(blob, g->lists->blob, g->blob.size(), cudaMemcpyDeviceToDevice, ex.stream) != cudaSuccess)
        return GBQR_ECUDA;
    const int nr = (int)g->relocs.size();
    trace_begin(ex, FAM_OTHER);
    reloc_kernel<<<(nr + 255) / 256, 256, 0, ex.stream>>>(g->lists->relocs, nr, (uint64_t *)blob, ws, (const char *)mats, stride);
    TRY_ST(trace_end(ex, FAM_OTHER, 0.0, 0.0));
    for (const GroupStep &s : g->steps) {
        switch (s.kind) {
            case ST_SLICE: {
                OzSliceArgs<double> a{};
                a.list = reinterpret_cast<const OzOperand<double> *>(blob + s.list);
                a.n = s.n;
                TRY_ST(oz_slice_launch(ex, kOzDigits64, a, (unsigned)s.grid, s.tall, s.elems));
                break;
            }
            case ST_MMA:
            case ST_REDUCE:
            case ST_REQUANT: {
                OzMmaArgs<double> a{};
                a.list = reinterpret_cast<const OzProblem<double> *>(blob + s.list);
                a.n = s.n;
                a.items = s.grid;
                a.err = err;
                if (s.kind == ST_MMA) TRY_ST(oz_mma_launch(ex, a, s.elems));
                else if (s.kind == ST_REDUCE) TRY_ST(oz_reduce_launch(ex, a, (size_t)s.grid * kThreads));
                else TRY_ST(oz_requant_launch(ex, a, s.grid));
                break;
            }
            default: {
                GramList<double> gl{};
                gl.list = reinterpret_cast<const GramArgs<double> *>(blob + s.list);
                trace_begin(ex, FAM_OTHER);
                const dim3 grid((unsigned)s.grid, (unsigned)s.n, (unsigned)s.z);
                if (s.kind == ST_DIAG) gram_diag_kernel<double><<<grid, kThreads, 0, ex.stream>>>(gl, s.k);
                else if (s.kind == ST_ROW) gram_row_kernel<double><<<grid, GT, 0, ex.stream>>>(gl, s.k);
                else if (s.kind == ST_TRAIL) gram_trail_kernel<double><<<grid, GT, 0, ex.stream>>>(gl, s.k);
                else gram_t_kernel<double><<<grid, GT, 0, ex.stream>>>(gl, s.k);
                TRY_ST(trace_end(ex, FAM_OTHER, 0.0, 0.0));
            }
        }
    }
    return GBQR_OK;
}

}  // namespace gbqr
