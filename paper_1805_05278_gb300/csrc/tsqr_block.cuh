// The TSQR of a panel as the work of its CTAs, one a leaf: the upsweep, and the
// downsweep with the reconstruction.  tsqr.cu launches each for all leaves;
// panel_chain.cu runs them as steps of a whole panel's factorization.
#pragma once

#include "panel_chain.cuh"
#include "tsqr_dev.cuh"

namespace gbqr {
namespace {

// The cnt consecutive w x w slots at src (slot i, entry (row, col) at
// i w^2 + row + col w) stacked into S: slot i's entry goes to S(i w + row,
// col).  Up to 8 loads in flight per thread, as in load_block.
template <class Real>
__device__ __forceinline__ void load_stack(Real *S, int64_t ldS, const Real *src, int cnt, int w) {
    constexpr int kBatch = 8;
    const int tid = threadIdx.x, nthr = blockDim.x, ww = w * w, total = cnt * ww;
    for (int base = tid; base < total; base += kBatch * nthr) {
        Real v[kBatch];
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int e = base + k * nthr;
            if (e < total) v[k] = __ldcg(src + e);
        }
#pragma unroll
        for (int k = 0; k < kBatch; ++k) {
            const int e = base + k * nthr;
            if (e < total) {
                const int i = e / ww, rem = e - i * ww, col = rem / w, row = rem - col * w;
                S[(i * w + row) + (int64_t)col * ldS] = v[k];
            }
        }
    }
}

__device__ __forceinline__ int64_t leaf_begin(int64_t mp, int P, int p) { return (int64_t)p * mp / P; }

// Upsweep of leaf `leaf` (one CTA).  Shared memory: S (ldS x w), then T, G (w x w each), then the
// per-column reflector data (Refl: tau, d, beta*d, q, 1/d, norm; w each).
template <class Real>
__device__ __forceinline__ void tsqr_up(const TsqrParamsT<Real> &p, int leaf, Real *smem) {
    const int w = p.w, ldS = p.ldS, tid = threadIdx.x, nthr = blockDim.x;
    Real *S = smem;
    Real *T = S + (size_t)ldS * w;
    Real *G = T + w * w;
    Real *aux = G + w * w;
    const Refl<Real> rf{aux, aux + w, aux + 2 * w, aux + 3 * w, aux + 4 * w, aux + 5 * w};
    __shared__ int s_last;

    const int64_t r0 = leaf_begin(p.mp, p.P, leaf), r1 = leaf_begin(p.mp, p.P, leaf + 1);
    const int h = (int)(r1 - r0);
    const size_t ww = (size_t)w * w;

    load_block(S, ldS, p.A + r0, p.lda, h, w);
    __syncthreads();
    householder_block(S, ldS, w, LeafRows{h}, rf, G);
    finish_block(S, ldS, w, rf, G);

    // V_p (strict lower, normalised here) and R_p (upper) back to the panel
    // rows, R_p to the tree; then T_p, with the leaf block's shared memory as
    // scratch.  Leaf 0 also keeps a copy of its top w x w block of V: every
    // CTA of the downsweep reads it to form X while CTA 0 overwrites those
    // rows of the panel.
    for (int c = 0; c < w; ++c) {
        const Real sc = rf.sc[c];
        for (int r = tid; r < h; r += nthr) {
            const Real x = S[(size_t)c * ldS + r];
            p.A[(r0 + r) + c * p.lda] = (r > c) ? x * sc : x;
        }
    }
    if (leaf == 0)
        for (int idx = tid; idx < w * w; idx += nthr) {
            const int i = idx % w, c = idx / w;
            p.wsX[idx] = (i > c) ? S[(size_t)c * ldS + i] * rf.sc[c] : Real(0);
        }
    {
        Real *Rn = p.wsR + (size_t)leaf * ww;
        for (int idx = tid; idx < w * w; idx += nthr) {
            const int i = idx % w, c = idx / w;
            Rn[idx] = (i <= c) ? S[(size_t)c * ldS + i] : Real(0);
        }
    }
    __syncthreads();
    build_t(T, G, rf.tau, S, w);
    {
        Real *Tn = p.wsT + (size_t)leaf * ww;
        for (int idx = tid; idx < w * w; idx += nthr) Tn[idx] = T[idx];
    }

    // Climb: the last of a node's children to arrive merges them.
    int node = leaf, Nl = p.P;
    int64_t off = 0, off_next = p.P;
    while (Nl > 1) {
        const int parent = node / p.k, first = parent * p.k;
        const int cnt = min(p.k, Nl - first);
        const int Nnext = (Nl + p.k - 1) / p.k;
        const int64_t pidx = off_next + parent;
        __threadfence();
        __syncthreads();
        if (cnt > 1) {
            if (tid == 0) {
                const unsigned prev = atomicAdd(&p.counters[pidx - p.P], 1u);
                s_last = (prev == (unsigned)(cnt - 1));
            }
            __syncthreads();
            if (!s_last) return;
            __threadfence();
            if (tid == 0) p.counters[pidx - p.P] = 0u;
            load_stack(S, ldS, p.wsR + (size_t)(off + first) * ww, cnt, w);   // the children's R, stacked
            __syncthreads();
            householder_block(S, ldS, w, MergeRows{w, cnt}, rf, G);
            finish_block(S, ldS, w, rf, G);
            Real *Rn = p.wsR + (size_t)pidx * ww, *Tn = p.wsT + (size_t)pidx * ww;
            Real *Yn = p.wsY + (size_t)(pidx - p.P) * (p.k - 1) * ww;
            for (int idx = tid; idx < w * w; idx += nthr) {
                const int i = idx % w, c = idx / w;
                Rn[idx] = (i <= c) ? S[(size_t)c * ldS + i] : Real(0);
            }
            for (int b = 1; b < cnt; ++b)
                for (int idx = tid; idx < w * w; idx += nthr) {
                    const int i = idx % w, c = idx / w;
                    Yn[(size_t)(b - 1) * ww + idx] = (i <= c) ? S[(size_t)c * ldS + b * w + i] * rf.sc[c] : Real(0);
                }
            __syncthreads();
            build_t(T, G, rf.tau, S, w);
            for (int idx = tid; idx < w * w; idx += nthr) Tn[idx] = T[idx];
        } else {
            // single child: the node is the identity, its R passes through
            const Real *Rc = p.wsR + (size_t)(off + node) * ww;
            Real *Rn = p.wsR + (size_t)pidx * ww;
            for (int idx = tid; idx < w * w; idx += nthr) Rn[idx] = Rc[idx];
        }
        node = parent;
        off = off_next;
        off_next += Nnext;
        Nl = Nnext;
    }
}

// B <- (the node Q-factors along the root-to-`target` path) applied to
// B = I at the root, or to the upper triangular Binit (Appendix C.2,
// downsweep): each node on the path gives its child [B_0; B_1; ...] =
// (I - V T V^T)[B; 0] = [B - T B; -Y_1 T B; ...].  T, Y and B are upper
// triangular, so B stays upper triangular and each product costs about
// w^3/6 multiply-adds.  C, M: w x w scratch.
template <int MaxW, class Real>
__device__ void walk_path(const TsqrParamsT<Real> &p, int target, Real *B, Real *C, Real *M, Real *Yb,
                          const Real *Binit = nullptr) {
    const int w = p.w, tid = threadIdx.x, nthr = blockDim.x;
    const int ww = w * w;
    constexpr int kPer = (MaxW * MaxW + kThreads - 1) / kThreads;   // entries per thread
    int anc[41], Nlev[41];
    int64_t offl[41];
    anc[0] = target; Nlev[0] = p.P; offl[0] = 0;
    for (int lv = 0; lv < p.L; ++lv) {
        anc[lv + 1] = anc[lv] / p.k;
        Nlev[lv + 1] = (Nlev[lv] + p.k - 1) / p.k;
        offl[lv + 1] = offl[lv] + Nlev[lv];
    }
    // the node above level lv merges cnt children; a single child passes through
    auto count = [&](int lv) { return min(p.k, Nlev[lv] - anc[lv + 1] * p.k); };
    auto next_merge = [&](int lv) {
        while (lv >= 0 && count(lv) == 1) --lv;
        return lv;
    };
    // the node's T and (for a child after the first) its Y block, staged in
    // registers so that the next level's loads overlap this level's products
    Real tn[kPer], yn[kPer];
    auto fetch = [&](int lv) {
        const int parent = anc[lv + 1], pos = anc[lv] - parent * p.k;
        const int64_t pidx = offl[lv + 1] + parent;
        const Real *Tn = p.wsT + (size_t)pidx * ww;
        const Real *Yn = p.wsY + ((size_t)(pidx - p.P) * (p.k - 1) + (pos > 0 ? pos - 1 : 0)) * ww;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int idx = tid + q * nthr;
            if (idx < ww) {
                tn[q] = __ldcg(Tn + idx);
                if (pos > 0) yn[q] = __ldcg(Yn + idx);
            }
        }
    };
    for (int idx = tid; idx < ww; idx += nthr) B[idx] = Binit ? Binit[idx] : ((idx % w == idx / w) ? Real(1) : Real(0));
    int cur = next_merge(p.L - 1);
    if (cur >= 0) fetch(cur);
    __syncthreads();
    while (cur >= 0) {
        const int pos = anc[cur] - anc[cur + 1] * p.k;
#pragma unroll
        for (int q = 0; q < kPer; ++q) {
            const int idx = tid + q * nthr;
            if (idx < ww) {
                M[idx] = tn[q];
                if (pos > 0) Yb[idx] = yn[q];
            }
        }
        __syncthreads();
        const int nxt = next_merge(cur - 1);
        if (nxt >= 0) fetch(nxt);
        upper_upper(M, B, C, w, Real(1));          // C = T_node B
        __syncthreads();
        if (pos == 0) {
            for (int idx = tid; idx < ww; idx += nthr) B[idx] -= C[idx];
        } else {
            upper_upper(Yb, C, B, w, -Real(1));    // B = -Y_pos C
        }
        __syncthreads();
        cur = nxt;
    }
}

// Downsweep and reconstruction for leaf `leaf` (one CTA; Appendix C.2).  W = Q [I; 0]
// row block p is W_p = (I - V_p T_p V_p^T)[B_p; 0] with B_p from the path
// root -> leaf p.  The top block X of W (leaf 0's top rows) is formed by every
// CTA from leaf 0's path and the copy of leaf 0's top V block that the
// upsweep kept, so no CTA waits for another; then, in every CTA:
//   X + S = L U with S_jj = sgn(X^_jj) added before column j is eliminated;
//   V rows = W rows U^{-1} for this leaf's rows below the top w;
// and CTA 0 writes T = U S L^{-T}, V_top = L and R = -S R^(L) (R^(L) at the root).
// MaxW: the widest panel (registers that stage a node's blocks).
template <int MaxW, class Real>
__device__ __forceinline__ void tsqr_down(const TsqrParamsT<Real> &p, int leaf, Real *smem) {
    const int w = p.w, ldS = p.ldW, tid = threadIdx.x, nthr = blockDim.x;
    const size_t ww = (size_t)w * w;
    Real *B = smem;          // w x w: B of the path walked
    Real *C = B + ww;        // w x w scratch
    Real *M = C + ww;        // w x w: T, then Z, then U^{-1}, then T_p and Z_p
    Real *X = M + ww;        // w x w: X, then L (strict lower) and U
    Real *Li = X + ww;       // w x w: leaf 0's top V block, then L^{-1}
    Real *Sg = Li + ww;      // w signs
    Real *rU = Sg + w;       // w reciprocals of diag(U)
    Real *Vs = rU + w;       // ldS x w: this leaf's rows of V, then of W and V
    // X = [B_0; 0] top rows - V0 Z0, V0 = leaf 0's unit lower top block
    walk_path<MaxW>(p, 0, B, C, M, X);                          // X is free until formed below
    for (int idx = tid; idx < w * w; idx += nthr) {
        Li[idx] = __ldcg(p.wsX + idx);
        M[idx] = __ldcg(p.wsT + idx);                        // T of leaf 0
    }
    __syncthreads();
    leaf_z<MaxW>(Li, w, B, C, M, w);
    for (int idx = tid; idx < w * w; idx += nthr) {
        const int r = idx % w, c = idx / w;
        Real s = (r <= c) ? M[r + c * w] : Real(0);
        for (int i = 0; i < min(r, c + 1); ++i) s = rfma(Li[i * w + r], M[i + c * w], s);
        X[idx] = B[idx] - s;
    }
    __syncthreads();
    // X + S = L U.  Per step one thread adds the sign to the pivot and takes
    // its reciprocal; then every entry of the trailing block forms its own
    // multiplier l_i = X(i, j) / pivot and is updated in the same pass, the
    // multipliers going to C, so X's column j and row j are only read during
    // the step (two barriers per step).  C is free here.
    for (int j = 0; j < w; ++j) {
        if (tid == 0) {
            const Real sg = X[j + j * w] < Real(0) ? -Real(1) : Real(1);
            Sg[j] = sg;
            const Real piv = X[j + j * w] + sg;
            X[j + j * w] = piv;
            rU[j] = real_rcp(piv);
        }
        __syncthreads();
        const Real rp = rU[j];
        const int rem = w - j - 1;
        for (int idx = tid; idx < rem * (rem + 1); idx += nthr) {
            const int i = j + 1 + idx % rem, c = j + idx / rem;
            const Real l = X[i + j * w] * rp;
            if (c == j) C[i + j * w] = l;
            else X[i + c * w] = rfma(-l, X[j + c * w], X[i + c * w]);
        }
        __syncthreads();
    }
    for (int idx = tid; idx < w * w; idx += nthr) {
        const int i = idx % w, c = idx / w;
        if (i > c) X[idx] = C[idx];                           // L below the diagonal
    }
    __syncthreads();
    // U^{-1} into M (Z of leaf 0 is no longer needed): the inverse of the
    // upper triangular matrix with strict upper part U and diagonal 1/rU,
    // which is what build_t computes from (G, tau)
    Real *Ui = M;
    build_t(Ui, X, rU, C, w);
    if (leaf == 0) {
        // T = U S L^{-T}: T(i, c) = sum_{l=i}^{c} U(i, l) S_l Li(c, l)
        unit_lower_inverse(X, Li, C, w);
        for (int idx = tid; idx < w * w; idx += nthr) {
            const int i = idx % w, c = idx / w;
            Real t = Real(0);
            for (int l = i; l <= c; ++l) t = rfma(X[i + l * w] * Sg[l], (l == c) ? Real(1) : Li[c + l * w], t);
            p.Tout[i + c * p.ldt] = t;
        }
        __syncthreads();
        upper_upper(B, Ui, C, w, Real(1));                    // leaf 0: B_0 U^{-1}
        __syncthreads();
        for (int idx = tid; idx < w * w; idx += nthr) B[idx] = C[idx];
    } else {
        // from B^(L) = U^{-1}: the walk copies Ui into B before it first
        // stages a node's T in M; Li is free here
        walk_path<MaxW>(p, leaf, B, C, M, Li, Ui);
    }
    __syncthreads();

    // this leaf: V_p = (I - V_p T_p V_p^T)[B_p; 0] with B_p from B^(L) = U^{-1}
    const int64_t r0 = leaf_begin(p.mp, p.P, leaf), r1 = leaf_begin(p.mp, p.P, leaf + 1);
    const int h = (int)(r1 - r0);
    load_block(Vs, ldS, p.A + r0, p.lda, h, w);
    {
        const Real *Tp = p.wsT + (size_t)leaf * ww;
        for (int idx = tid; idx < w * w; idx += nthr) M[idx] = Tp[idx];
    }
    __syncthreads();
    leaf_z<MaxW>(Vs, ldS, B, C, M, w);
    for (int r = tid; r < h; r += nthr) {
        if (r0 + r < w) continue;                           // leaf 0's top block: L \ R below
        // V(r, c) = [B; 0](r, c) - sum_{i <= min(r, c)} Vhat(r, i) Z(i, c), in place, c descending
        for (int c = w - 1; c >= 0; --c) {
            Real s = (r <= c) ? M[r + c * w] : Real(0);
            const int iend = min(r, c + 1);
            for (int i = 0; i < iend; ++i) s = rfma(Vs[(size_t)i * ldS + r], M[i + c * w], s);
            Vs[(size_t)c * ldS + r] = ((r < w) ? B[r + c * w] : Real(0)) - s;
        }
    }
    __syncthreads();
    for (int c = 0; c < w; ++c)
        for (int r = tid; r < h; r += nthr)
            if (r0 + r >= w) p.A[(r0 + r) + c * p.lda] = Vs[(size_t)c * ldS + r];
    if (leaf == 0) {
        // top block: L strictly below the diagonal, R = -S R^(L) on and above;
        // R^(L) sits in the last node slot (the root)
        int64_t nodes = p.P, Nl = p.P;
        while (Nl > 1) { Nl = (Nl + p.k - 1) / p.k; nodes += Nl; }
        const Real *RL = p.wsR + (size_t)(nodes - 1) * ww;
        for (int idx = tid; idx < w * w; idx += nthr) {
            const int i = idx % w, c = idx / w;
            p.A[i + c * p.lda] = (i <= c) ? -Sg[i] * __ldcg(RL + idx) : X[i + c * w];
        }
    }
}

}  // namespace
}  // namespace gbqr
