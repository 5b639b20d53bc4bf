// A panel's QR-EG recursion as the steps of ONE launch (panel_chain.cu).
#pragma once

#include "common.cuh"

namespace gbqr {

// A TSQR (tsqr_block.cuh) and a product (gemm_tile.cuh).
template <class Real>
struct TsqrParamsT {
    Real *A; int64_t lda;     // panel top-left, mp x w
    int64_t mp; int w;
    int P, k, L, ldS, ldW;
    Real *wsR, *wsT, *wsY, *wsX;
    unsigned *counters;
    Real *Tout; int64_t ldt;
};
template <class Real>
struct GemmParamsT {
    int64_t M, N, K;
    const Real *A; int64_t lda; int maskA;
    const Real *B; int64_t ldb; int maskB;
    Real *C; int64_t ldc;
    Real alpha, beta;
    Real *partial;            // per tile: slots_per_tile * BM*BN elements
    unsigned *counters;       // per tile: counters_per_tile
    int slots_per_tile, counters_per_tile;
};

enum ChainKind { CH_UP, CH_DOWN, CH_TA, CH_N16, CH_N64 };   // TSQR up / down; products: A^T B, A B (16- and 64-row tiles)

// One launch's worth of work: nblk CTAs' worth of `kind`.
template <class Real>
struct ChainStep {
    int kind, nblk;
    int gx, gy;                  // products: tiles along M and N (splits: nblk / (gx gy))
    union {
        TsqrParamsT<Real> tsqr;
        GemmParamsT<Real> gemm;
    };
};

constexpr int kChainMaxW = 24;   // widest TSQR (16 and 24 measure the same; 64 columns take 37 us each, these 13)
constexpr int kChainSteps = 64;  // 8 TSQRs, 7 updates and T merges of three products each, Y

template <class Real>
struct ChainArgs {
    ChainStep<Real> step[kChainSteps];
    int nsteps = 0, total = 0;   // total: all steps' CTAs
    const int *flag;             // nothing to do while it is zero
    unsigned *ctr;               // ticket, tasks done, CTAs gone, abort: zero before and after
    int *timeout;                // raised when a wait runs out
};

// Where gemm() and tsqr_run() put their work instead of launching it.
struct ChainRecorder {
    ChainArgs<double> f64;
    ChainArgs<float> f32;
    size_t smem = 0;
    int widest = 0;
    template <class Real> ChainArgs<Real> &args();
};
template <> inline ChainArgs<double> &ChainRecorder::args<double>() { return f64; }
template <> inline ChainArgs<float> &ChainRecorder::args<float>() { return f32; }

template <class Real> gbqr_status chain_tsqr(const Exec &ex, const TsqrParamsT<Real> &p, const TsqrPlan &pl);
template <class Real> gbqr_status chain_gemm(const Exec &ex, const GemmOpT<Real> &op, const GemmScratchT<Real> &sc);
// Launches what was recorded; ctr: 4 counters, zero.
template <class Real>
gbqr_status chain_launch(const Exec &ex, ChainRecorder &rec, const int *flag, unsigned *ctr, int *timeout);

}  // namespace gbqr
