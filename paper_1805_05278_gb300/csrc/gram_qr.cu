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
//   V2 = A2 U^{-1}                the rows below, one tall product
//   T = -U R+^{-1} S V1^{-T}
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
//   diag   one CTA: Cholesky and LU of the diagonal block with their inverses
//          (Gauss-Jordan: the inverses cost columns, not steps),
//   row    block row k of R and U, block column k of L, ...
//   trail  the trailing blocks of G and A1; R^{-1}, U^{-1} and V1^{-1} grow by
//          one block column or row.
// FP64 issues one instruction per warp per 64 cycles on this part, so a 32^3
// product on one SM takes 9 us: row and trail spread every block over 8 CTAs.
#include "tsqr_dev.cuh"

#include <algorithm>
#include <cmath>

namespace gbqr {
namespace {

constexpr int GB = 32;               // block width
constexpr int GLD = kGramMaxW;       // leading dimension of every w x w array
constexpr int GT = 128;              // threads of the row / trail kernels: 32 x 4 outputs
constexpr double kGramBound2 = 16.0; // largest accepted (R^-1)_ij^2 g_ii

struct GramArgs {
    double *A; int64_t lda;          // panel
    double *Tout; int64_t ldt;
    int w, nblk;
    double *G, *R, *RI, *A1, *L, *U, *LI, *X, *YX, *YR, *YL, *K, *sgn, *gd;
    int *flag, *kexp;                // kexp: exponents of the column norms
};

__device__ __forceinline__ double g_at(const GramArgs &p, int i, int j, int k) {
    if (k > 0) return __ldcg(p.G + i + j * GLD);
    return (i < p.w && j < p.w) ? __ldcg(p.G + i + j * GLD) : (i == j ? 1.0 : 0.0);
}
__device__ __forceinline__ double a1_at(const GramArgs &p, int i, int j, int k) {
    if (k > 0) return __ldcg(p.A1 + i + j * GLD);
    return (i < p.w && j < p.w) ? p.A[i + (int64_t)j * p.lda] : (i == j ? 1.0 : 0.0);
}

// Diagonal block k.  In both eliminations warp 0 carries the chain (update of
// the next column, pivot, reciprocal, multipliers) one step ahead of the
// other warps, which update the remaining columns and the augmented identity;
// in the LU warp 1 carries the next row of U the same way.
__global__ void __launch_bounds__(kThreads) gram_diag_kernel(const GramArgs p, int k) {
    __shared__ double S[GB][GB + 1], E[GB][GB + 1], Rb[GB][GB + 1];   // [column][row]
    __shared__ double cb[2][GB], lb[2][GB], rd[GB], sg[GB];
    __shared__ int bad;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, b0 = k * GB;
    if (k > 0 && *(volatile int *)p.flag) return;
    for (int c = warp; c < GB; c += 8) {
        S[c][lane] = lane <= c ? g_at(p, b0 + lane, b0 + c, k) : g_at(p, b0 + c, b0 + lane, k);
        E[c][lane] = lane == c ? 1.0 : 0.0;
    }
    if (k == 0) {
        for (int i = tid; i < p.nblk * GB; i += kThreads) {
            const double g = i < p.w ? __ldcg(p.G + i + i * GLD) : 1.0;
            p.gd[i] = g;
            p.kexp[i] = (((__double2hiint(g) >> 20) & 0x7ff) - 1023) >> 1;
        }
        if (tid == 0) *p.flag = 0;
    }
    if (tid == 0) bad = 0;
    __syncthreads();
    // ---- Cholesky: S = L D L^T, E -> L^{-1}
    if (warp == 0) {
        const double v = S[0][lane];
        const double r = real_rcp(__shfl_sync(kFull, v, 0));
        cb[0][lane] = v;
        lb[0][lane] = v * r;
    }
    __syncthreads();
    for (int t = 0; t < GB; ++t) {
        const double *c = cb[t & 1], *l = lb[t & 1];
        const double li = lane > t ? l[lane] : 0.0;
        if (warp == 0) {
            if (t + 1 < GB) {
                const double v = rfma(-li, c[t + 1], S[t + 1][lane]);
                const double r = real_rcp(__shfl_sync(kFull, v, t + 1));
                S[t + 1][lane] = v;
                cb[(t + 1) & 1][lane] = v;
                lb[(t + 1) & 1][lane] = v * r;
            }
        } else {
            for (int q = warp - 1; q < GB - 1; q += 7) {
                // columns 0..t of E, then t+2.. of S
                if (q <= t) E[q][lane] = rfma(-li, E[q][t], E[q][lane]);
                else S[q + 1][lane] = rfma(-li, c[q + 1], S[q + 1][lane]);
            }
            if (t == GB - 1 && warp == 1) E[GB - 1][lane] = rfma(-li, E[GB - 1][t], E[GB - 1][lane]);
        }
        __syncthreads();
    }
    // R = D^{1/2} L^T, R^{-1} = L^{-T} D^{-1/2}; S[t][i] = d_t L(i, t)
    if (warp == 0) {
        const double d = S[lane][lane];
        const double s = sqrt(d);
        rd[lane] = real_rcp(s);
        if (!(d > 0.0)) bad = 1;
    }
    __syncthreads();
    for (int c = warp; c < GB; c += 8) {
        // column c: R(lane, c) = S[lane][c] rd[lane], RI(lane, c) = E[lane][c] rd[c]
        const double rv = lane <= c ? S[lane][c] * rd[lane] : 0.0;
        const double ri = lane <= c ? E[lane][c] * rd[c] : 0.0;
        Rb[c][lane] = rv;
        p.R[(b0 + lane) + (b0 + c) * GLD] = rv;
        p.RI[(b0 + lane) + (b0 + c) * GLD] = ri;
        const double g = k == 0 ? (b0 + lane < p.w ? __ldcg(p.G + (b0 + lane) * (GLD + 1)) : 1.0) : __ldcg(p.gd + b0 + lane);
        if (!(ri * ri * g <= kGramBound2)) bad = 1;
    }
    __syncthreads();
    if (bad) {
        if (tid == 0) *p.flag = 1;
        return;
    }
    // ---- LU of A1 - S R: E -> V1^{-1} (diagonal block)
    for (int c = warp; c < GB; c += 8) {
        S[c][lane] = a1_at(p, b0 + lane, b0 + c, k);
        E[c][lane] = lane == c ? 1.0 : 0.0;
    }
    __syncthreads();
    // cb: row t of U (entry j at [j]); lb: multipliers
    if (warp == 0) {
        const double v = S[0][lane], al = __shfl_sync(kFull, v, 0);
        const double u = al - (al < 0.0 ? Rb[0][0] : -Rb[0][0]);
        const double r = real_rcp(u);
        if (lane == 0) rd[0] = r;
        lb[0][lane] = v * r;
    } else if (warp == 1) {
        const double x = S[lane][0], al = __shfl_sync(kFull, x, 0);
        const double s = al < 0.0 ? 1.0 : -1.0;
        if (lane == 0) sg[0] = s;
        cb[0][lane] = x - s * Rb[lane][0];
    }
    __syncthreads();
    for (int t = 0; t < GB; ++t) {
        const double *u = cb[t & 1], *l = lb[t & 1];
        const double li = lane > t ? l[lane] : 0.0;
        if (warp == 0) {
            double v = 0.0;
            if (t + 1 < GB) {
                v = rfma(-li, u[t + 1], S[t + 1][lane]);
                const double al = __shfl_sync(kFull, v, t + 1), rr = Rb[t + 1][t + 1];
                const double r = real_rcp(al - (al < 0.0 ? rr : -rr));
                if (lane == 0) rd[t + 1] = r;
                lb[(t + 1) & 1][lane] = v * r;
            }
            S[t][lane] = lane > t ? li : S[t][lane];                    // L below the diagonal
        } else if (warp == 1) {
            if (t + 1 < GB) {
                const double x = rfma(-l[t + 1], u[lane], S[lane][t + 1]);
                const double al = __shfl_sync(kFull, x, t + 1);
                const double s = al < 0.0 ? 1.0 : -1.0;
                if (lane == 0) sg[t + 1] = s;
                cb[(t + 1) & 1][lane] = lane > t ? x - s * Rb[lane][t + 1] : 0.0;
            }
            if (lane >= t) p.U[(b0 + t) + (b0 + lane) * GLD] = u[lane];  // row t of U
        } else {
            for (int q = warp - 2; q < GB - 1; q += 6) {
                if (q <= t) E[q][lane] = rfma(-li, E[q][t], E[q][lane]);
                else if (lane != t + 1) S[q + 1][lane] = rfma(-li, u[q + 1], S[q + 1][lane]);
            }
            if (t == GB - 1 && warp == 2) E[GB - 1][lane] = rfma(-li, E[GB - 1][t], E[GB - 1][lane]);
        }
        __syncthreads();
    }
    for (int c = warp; c < GB; c += 8) {
        p.L[(b0 + lane) + (b0 + c) * GLD] = lane > c ? S[c][lane] : (lane == c ? 1.0 : 0.0);
        p.LI[(b0 + lane) + (b0 + c) * GLD] = E[c][lane];
        if (lane > c) p.U[(b0 + lane) + (b0 + c) * GLD] = 0.0;
    }
    if (tid < GB) p.sgn[b0 + tid] = sg[tid];
    __syncthreads();
    // X = U^{-1}: upper triangular inverse, diagonal 1 / u_tt in rd
    double *Gs = &E[0][0], *Ts = &S[0][0], *Ms = &Rb[0][0];
    for (int idx = tid; idx < GB * GB; idx += kThreads)
        Gs[idx] = __ldcg(p.U + (b0 + idx % GB) + (b0 + idx / GB) * GLD);
    __syncthreads();
    build_t(Ts, Gs, rd, Ms, GB);
    for (int idx = tid; idx < GB * GB; idx += kThreads) p.X[(b0 + idx % GB) + (b0 + idx / GB) * GLD] = Ts[idx];
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

// Block row k of R and U (tasks 0 .. n-k-2), block column k of L (the next
// n-k-1), then for l < k: YX_l = U_lk X_kk, YR_l = R_lk RI_kk and YL_l =
// sum_j L_kj LI_jl.  blockIdx.x = task * 8 + column group.
__global__ void __launch_bounds__(GT) gram_row_kernel(const GramArgs p, int k) {
    __shared__ double sA[GB][GB + 1], sB[4][GB];
    if (*(volatile int *)p.flag) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Tile tl{sA, sB, warp, lane};
    const int task = blockIdx.x >> 3, c0 = (blockIdx.x & 7) * 4, rest = p.nblk - k - 1;
    const int c = c0 + warp;
    if (task < rest) {
        const int j = k + 1 + task;
        tl.load_a(blk(p.RI, k, k), true);                      // R_kj = RI_kk^T G_kj
        sB[warp][lane] = g_at(p, k * GB + lane, j * GB + c, k);
        const double a = a1_at(p, k * GB + lane, j * GB + c, k);
        __syncthreads();
        const double r = tl.dot(0.0);
        __syncthreads();
        blk(p.R, k, j)[lane + c * GLD] = r;
        tl.load_a(blk(p.LI, k, k), false);                     // U_kj = V1_kk^{-1} (A1_kj - S R_kj)
        sB[warp][lane] = rfma(-__ldcg(p.sgn + k * GB + lane), r, a);
        __syncthreads();
        blk(p.U, k, j)[lane + c * GLD] = tl.dot(0.0);
        return;
    }
    if (task < 2 * rest) {
        const int i = k + 1 + task - rest;                     // L_ik = A1_ik X_kk
        for (int kk = warp; kk < GB; kk += 4) sA[kk][lane] = a1_at(p, i * GB + lane, k * GB + kk, k);
        tl.load_b(blk(p.X, k, k) + c0 * GLD);
        __syncthreads();
        blk(p.L, i, k)[lane + c * GLD] = tl.dot(0.0);
        return;
    }
    const int e = task - 2 * rest, l = e / 3, what = e % 3;
    double *out = what == 0 ? p.YX : (what == 1 ? p.YR : p.YL);
    double acc = 0.0;
    if (what < 2) {
        tl.load_a(blk(what == 0 ? p.U : p.R, l, k), false);
        tl.load_b(blk(what == 0 ? p.X : p.RI, k, k) + c0 * GLD);
        __syncthreads();
        acc = tl.dot(0.0);
    } else {
        for (int j = l; j < k; ++j) {
            __syncthreads();
            tl.load_a(blk(p.L, k, j), false);
            tl.load_b(blk(p.LI, j, l) + c0 * GLD);
            __syncthreads();
            acc = tl.dot(acc);
        }
    }
    out[l * GB + lane + c * GLD] = acc;                        // Y_l: block row l of a w x 32 array
}

// Trailing blocks of G (upper) and A1, then for l < k: X_lk = -sum X_lj YX_j,
// RI_lk = -sum RI_lj YR_j, LI_kl = -LI_kk YL_l.
__global__ void __launch_bounds__(GT) gram_trail_kernel(const GramArgs p, int k) {
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

// K = U R^{-1} (step 0), then T = -K S' ... (step 1): T = -U (S R)^{-1} V1^{-T}
// = -U R^{-1} S V1^{-T}.  Step 1 also writes V1 \ R over the panel's top block.
__global__ void __launch_bounds__(GT) gram_t_kernel(const GramArgs p, int step) {
    __shared__ double sA[GB][GB + 1], sB[4][GB];
    if (*(volatile int *)p.flag) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Tile tl{sA, sB, warp, lane};
    const int c0 = (blockIdx.x & 7) * 4, c = c0 + warp, task = blockIdx.x >> 3;
    const int i = task % p.nblk, j = task / p.nblk;
    const int gi = i * GB + lane, gj = j * GB + c;
    double acc = 0.0;
    if (i <= j)
        for (int l = i; l <= j; ++l) {
            __syncthreads();
            if (step == 0) {
                tl.load_a(blk(p.U, i, l), false);
                tl.load_b(blk(p.RI, l, j) + c0 * GLD);
            } else {
                tl.load_a(blk(p.K, i, l), false);
                tl.load_b(blk(p.LI, j, l) + c0, true);         // (V1^{-T})(l, j) = LI(j, l)^T
            }
            __syncthreads();
            acc = tl.dot(acc);
        }
    if (step == 0) {
        if (i <= j) blk(p.K, i, j)[lane + c * GLD] = acc * __ldcg(p.sgn + gj);   // (U R^{-1}) S
        return;
    }
    if (gi >= p.w || gj >= p.w) return;
    p.Tout[gi + (int64_t)gj * p.ldt] = gi <= gj ? -acc : 0.0;
    p.A[gi + (int64_t)gj * p.lda] =
        gi <= gj ? __ldcg(p.sgn + gi) * __ldcg(p.R + gi + gj * GLD) : __ldcg(p.L + gi + gj * GLD);
}

}  // namespace

size_t gram_work_elems() { return (size_t)13 * GLD * GLD + 4 * GLD; }

bool gram_qr_fits(const OzScratch &oz, int64_t m, int64_t w) {
    return w >= kGramMinW && w <= kGramMaxW && m >= 4 * w && oz.base &&
           std::max(oz_gemm_scratch_bytes(w, w, m), oz_gemm_scratch_bytes(m - w, w, w)) <= oz.bytes;
}

gbqr_status gram_qr(const Exec &ex, int64_t m, int64_t w, double *A, int64_t lda, double *T, int64_t ldt,
                    double *work, int *flag, const OzScratch &oz) {
    GramArgs p{};
    p.A = A; p.lda = lda; p.Tout = T; p.ldt = ldt;
    p.w = (int)w; p.nblk = (int)((w + GB - 1) / GB);
    double **slots[] = {&p.G, &p.R, &p.RI, &p.A1, &p.L, &p.U, &p.LI, &p.X, &p.YX, &p.YR, &p.YL, &p.K};
    double *at = work;
    for (double **s : slots) { *s = at; at += (size_t)GLD * GLD; }
    p.sgn = at;
    p.gd = p.sgn + GLD;
    p.flag = flag;
    p.kexp = (int *)(p.gd + GLD);
    GemmOp g;
    g.M = w; g.N = w; g.K = m;
    g.A = A; g.lda = lda; g.ta = true; g.B = A; g.ldb = lda; g.C = p.G; g.ldc = GLD;
    TRY_ST(oz_gemm(ex, g, oz));
    auto mark = [&](double flops) { return trace_end(ex, FAM_OTHER, flops, 0.0); };
    const double f3 = 2.0 * GB * GB * GB;
    for (int k = 0; k < p.nblk; ++k) {
        trace_begin(ex, FAM_OTHER);
        gram_diag_kernel<<<1, kThreads, 0, ex.stream>>>(p, k);
        TRY_ST(mark(3.0 * f3));
        const int rest = p.nblk - k - 1, row = 2 * rest + 3 * k, trail = 2 * rest * rest + 3 * k;
        if (row) {
            trace_begin(ex, FAM_OTHER);
            gram_row_kernel<<<row * 8, GT, 0, ex.stream>>>(p, k);
            TRY_ST(mark(row * f3));
            trace_begin(ex, FAM_OTHER);
            gram_trail_kernel<<<trail * 8, GT, 0, ex.stream>>>(p, k);
            TRY_ST(mark(trail * f3));
        }
    }
    for (int step = 0; step < 2; ++step) {
        trace_begin(ex, FAM_OTHER);
        gram_t_kernel<<<p.nblk * p.nblk * 8, GT, 0, ex.stream>>>(p, step);
        TRY_ST(mark(p.nblk * p.nblk * f3));
    }
    if (m > w) {
        // V2 = A2 X, in place: the digits of A2 are taken before C is written
        GemmOp v;
        v.M = m - w; v.N = w; v.K = w;
        v.A = A + w; v.lda = lda; v.ta = false; v.B = p.X; v.ldb = GLD; v.maskB = MASK_UPPER;
        v.C = A + w; v.ldc = lda;
        v.skip = flag;
        v.kexp = p.kexp;                 // columns of A2 may differ by any scale, so may X's rows
        TRY_ST(oz_gemm(ex, v, oz));
    }
    return GBQR_OK;
}

}  // namespace gbqr
