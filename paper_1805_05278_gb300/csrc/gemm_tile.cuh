// One output tile of a masked product by CUDA-core FMA, as the work of a CTA:
// gemm.cu launches it for all tiles, panel_chain.cu runs it as part of a whole
// panel's factorization.
#pragma once

#include "panel_chain.cuh"
#include "tsqr_dev.cuh"

#include <algorithm>

namespace gbqr {
namespace {

constexpr int BK = 16;
constexpr int kGroup = 8;   // fan-in of the split-K reduction tree

template <class Real>
__device__ __forceinline__ Real masked(const Real *X, int64_t ld, int64_t r, int64_t c, int mask) {
    if (mask == MASK_UNIT_LOWER) {
        if (r < c) return Real(0);
        if (r == c) return Real(1);
    } else if (mask == MASK_UPPER) {
        if (r > c) return Real(0);
    }
    return X[r + c * ld];
}

// K range [kb, ke) outside which op(A)(i, k) or op(B)(k, j) is structurally
// zero for every i in [m0, m0+BM) and j in [n0, n0+BN).
template <class P>
__device__ __forceinline__ void k_range(const P &p, bool ta, int64_t m0, int64_t n0,
                                        int BM, int BN, int64_t &kb, int64_t &ke) {
    kb = 0; ke = p.K;
    if (p.maskA == MASK_UNIT_LOWER) {
        if (!ta) ke = min(ke, m0 + BM);   // A(i,k) != 0 needs k <= i
        else kb = max(kb, m0);            // A(k,i) != 0 needs k >= i
    } else if (p.maskA == MASK_UPPER) {
        if (!ta) kb = max(kb, m0);        // A(i,k) != 0 needs k >= i
        else ke = min(ke, m0 + BM);       // A(k,i) != 0 needs k <= i
    }
    if (p.maskB == MASK_UNIT_LOWER) kb = max(kb, n0);       // B(k,j) != 0 needs k >= j
    else if (p.maskB == MASK_UPPER) ke = min(ke, n0 + BN);  // B(k,j) != 0 needs k <= j
}

// Tile (bx, by) and split z of S of C, one CTA; gx: tiles along M.  Prefetch:
// the next K tile's loads run under the current one's FMAs, for an SM that
// holds one CTA; where several share it they cover for one another.
template <class Real, int BM, int BN, bool TA, bool Prefetch>
__device__ __forceinline__ void gemm_tile(const GemmParamsT<Real> &p, int bx, int by, int z, int gx, int S,
                                          Real (*As)[BM + 1], Real (*Bs)[BN + 1]) {
    constexpr int RM = BM / 16, RN = BN / 16;
    __shared__ int s_last;

    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t m0 = (int64_t)bx * BM, n0 = (int64_t)by * BN;

    int64_t kb, ke;
    k_range(p, TA, m0, n0, BM, BN, kb, ke);
    int64_t k_lo = kb, k_hi = kb;
    if (ke > kb) {
        int64_t chunk = (ke - kb + S - 1) / S;
        chunk = (chunk + BK - 1) / BK * BK;
        k_lo = kb + (int64_t)z * chunk;
        k_hi = min(ke, k_lo + chunk);
    }

    Real acc[RM][RN];
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int c = 0; c < RN; ++c) acc[r][c] = Real(0);

    // a K tile of the operands, in registers on its way to shared memory
    constexpr int NA = BM * BK / kThreads, NB = BK * BN / kThreads;
    Real va[NA], vb[NB];
    auto load = [&](int64_t k0) {
        // op(A) tile: rows m0.., k0..
#pragma unroll
        for (int q = 0; q < NA; ++q) {
            const int idx = tid + q * kThreads;
            int i, kk;
            if (!TA) { i = idx % BM; kk = idx / BM; }   // coalesced along rows of stored A
            else     { kk = idx % BK; i = idx / BK; }   // coalesced along rows of stored A (= k)
            const int64_t gi = m0 + i, gk = k0 + kk;
            va[q] = Real(0);
            if (gi < p.M && gk < k_hi) va[q] = TA ? masked(p.A, p.lda, gk, gi, p.maskA)
                                                  : masked(p.A, p.lda, gi, gk, p.maskA);
        }
        // B tile: stored K x N, coalesced along k
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int idx = tid + q * kThreads;
            const int kk = idx % BK, j = idx / BK;
            const int64_t gk = k0 + kk, gj = n0 + j;
            vb[q] = Real(0);
            if (gj < p.N && gk < k_hi) vb[q] = masked(p.B, p.ldb, gk, gj, p.maskB);
        }
    };
    if (Prefetch && k_lo < k_hi) load(k_lo);
    for (int64_t k0 = k_lo; k0 < k_hi; k0 += BK) {
        if (!Prefetch) load(k0);
#pragma unroll
        for (int q = 0; q < NA; ++q) {
            const int idx = tid + q * kThreads;
            if (!TA) As[idx / BM][idx % BM] = va[q];
            else As[idx % BK][idx / BK] = va[q];
        }
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            const int idx = tid + q * kThreads;
            Bs[idx % BK][idx / BK] = vb[q];
        }
        __syncthreads();
        if (Prefetch && k0 + BK < k_hi) load(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            Real a[RM], b[RN];
#pragma unroll
            for (int r = 0; r < RM; ++r) a[r] = As[kk][tx + 16 * r];
#pragma unroll
            for (int c = 0; c < RN; ++c) b[c] = Bs[kk][ty + 16 * c];
#pragma unroll
            for (int r = 0; r < RM; ++r)
#pragma unroll
                for (int c = 0; c < RN; ++c) acc[r][c] = rfma(a[r], b[c], acc[r][c]);
        }
        __syncthreads();
    }

    if (S > 1) {
        // Split-K: deterministic tree of last-arriver reductions.
        const int64_t tile = bx + (int64_t)by * gx;
        Real *tp = p.partial + (size_t)tile * p.slots_per_tile * (BM * BN);
        unsigned *tc = p.counters + (size_t)tile * p.counters_per_tile;
        int slot = z, Sl = S, base = 0, cbase = 0;
        for (;;) {
            Real *dst = tp + (size_t)(base + slot) * (BM * BN);
#pragma unroll
            for (int r = 0; r < RM; ++r)
#pragma unroll
                for (int c = 0; c < RN; ++c) dst[(tx + 16 * r) + (ty + 16 * c) * BM] = acc[r][c];
            const int group = slot / kGroup, first = group * kGroup;
            const int cnt = min(kGroup, Sl - first);
            const int Snext = (Sl + kGroup - 1) / kGroup;
            __threadfence();
            __syncthreads();
            if (tid == 0) {
                unsigned prev = atomicAdd(&tc[cbase + group], 1u);
                s_last = (prev == (unsigned)(cnt - 1));
            }
            __syncthreads();
            if (!s_last) return;
            __threadfence();
            if (tid == 0) tc[cbase + group] = 0u;   // leave the counter zero for the next launch
#pragma unroll
            for (int r = 0; r < RM; ++r)
#pragma unroll
                for (int c = 0; c < RN; ++c) {
                    Real s = Real(0);
                    for (int q = 0; q < cnt; ++q)
                        s += __ldcg(tp + (size_t)(base + first + q) * (BM * BN) + (tx + 16 * r) + (ty + 16 * c) * BM);
                    acc[r][c] = s;
                }
            if (Snext == 1) break;
            base += Sl;
            cbase += Snext;
            slot = group;
            Sl = Snext;
        }
    }

#pragma unroll
    for (int c = 0; c < RN; ++c) {
        const int64_t gj = n0 + ty + 16 * c;
        if (gj >= p.N) continue;
#pragma unroll
        for (int r = 0; r < RM; ++r) {
            const int64_t gi = m0 + tx + 16 * r;
            if (gi >= p.M) continue;
            Real *cp = p.C + gi + gj * p.ldc;
            Real v = p.alpha * acc[r][c];
            if (p.beta != Real(0)) v = rfma(p.beta, *cp, v);
            *cp = v;
        }
    }
}

// Slots and counters per tile of the reduction tree for S splits.
inline void tree_shape(int S, int *slots, int *counters) {
    int s = 0, c = 0, Sl = S;
    while (Sl > 1) {
        s += Sl;
        Sl = (Sl + kGroup - 1) / kGroup;
        c += Sl;
    }
    *slots = std::max(s, 1);
    *counters = std::max(c, 1);
}

}  // namespace
}  // namespace gbqr
