// The QR-EG recursion of a panel in ONE launch, for the panels that the
// Gram-matrix base case gives up (gram_qr.cu): a device flag says so, and the
// kernel returns at once while it is zero.
//
// Why one launch: the recursion on TSQRs of 16 columns is about 58 launches,
// and a launch with nothing to do still takes its 3 us of the stream: 1024 x
// 128, when its Gram matrix will do, took 548 us with them behind it and 393
// with nine launches of TSQRs 64 wide - which take 37 us a column where those
// of 16 take 13.  So the recursion's launches are recorded as steps, and
// persistent CTAs take the steps' CTAs in order from a ticket: a CTA waits
// until all earlier steps are done.  It waits only for tasks taken before its
// own, by CTAs that are running, so however few CTAs are resident, every wait
// ends (and is bounded).  One CTA per SM in FP64: the leaves' chains slow each
// other down on a shared one (1024 x 128 1934 us with two CTAs, 1780 with
// one); the products then load a K tile ahead (32768 x 128 4447 -> 3888).
//
// A panel given up, by launches and no Gram matrix, by TSQRs 64 wide behind
// one, and now (us): 1024 x 128 1692, 4757, 1741; 32768 x 128 3592, 15568,
// 3888; 65536 x 32 738, 1181, 971.  What the attempt costs is in the last.
// One not given up, 1024 x 128: 393 -> 353.
#include "gemm_tile.cuh"
#include "tsqr_block.cuh"

#include <algorithm>
#include <atomic>

namespace gbqr {
namespace {

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

constexpr unsigned long long kChainWaitNs = 5000000000ull;   // far beyond any step

// One thread: until n tasks are done.  False, with the abort flag up, when the
// wait runs out here or elsewhere.
__device__ bool wait_done(unsigned *ctr, unsigned n, int *timeout) {
    const unsigned long long t0 = global_ns();
    while (ld_acquire(ctr + 1) < n) {
        if (*(volatile unsigned *)(ctr + 3)) return false;
        if (global_ns() - t0 > kChainWaitNs) {
            atomicExch(ctr + 3, 1u);
            atomicExch(timeout, 1);
            return false;
        }
        __nanosleep(20);
    }
    __threadfence();
    return true;
}

// (not inlined: each alone needs about 110 registers, all in one kernel 255)
template <class Real>
__device__ __noinline__ void chain_up(const ChainStep<Real> &st, int b, Real *smem) {
    const TsqrParamsT<Real> p = st.tsqr;
    tsqr_up(p, b, smem);
}
template <class Real>
__device__ __noinline__ void chain_down(const ChainStep<Real> &st, int b, Real *smem) {
    const TsqrParamsT<Real> p = st.tsqr;
    tsqr_down<kChainMaxW>(p, b, smem);
}
template <class Real, int BM, bool TA>
__device__ __noinline__ void chain_tile(const ChainStep<Real> &st, int b, Real *smem) {
    const int tiles = st.gx * st.gy, z = b / tiles, r = b - z * tiles;
    Real (*As)[BM + 1] = reinterpret_cast<Real (*)[BM + 1]>(smem);
    Real (*Bs)[17] = reinterpret_cast<Real (*)[17]>(smem + BK * (BM + 1));
    const GemmParamsT<Real> p = st.gemm;
    gemm_tile<Real, BM, 16, TA, true>(p, r % st.gx, r / st.gx, z, st.gx, st.nblk / tiles, As, Bs);
}

template <class Real>
__global__ void __launch_bounds__(kThreads) panel_chain_kernel(const __grid_constant__ ChainArgs<Real> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Real *smem = reinterpret_cast<Real *>(smem_raw);
    __shared__ int s_ticket, s_go;
    if (*(volatile const int *)a.flag == 0) return;
    int step = 0, first = 0;                     // first: the step's first task
    for (;;) {
        __syncthreads();                         // the last task is done with shared memory
        if (threadIdx.x == 0) s_ticket = (int)atomicAdd(a.ctr, 1u);
        __syncthreads();
        const int t = s_ticket;
        if (t >= a.total) break;
        bool moved = false;
        for (; t - first >= a.step[step].nblk; ++step) {
            first += a.step[step].nblk;
            moved = true;
        }
        if (moved) {
            if (threadIdx.x == 0) s_go = wait_done(a.ctr, (unsigned)first, a.timeout);
            __syncthreads();
            if (!s_go) break;
        }
        const ChainStep<Real> &st = a.step[step];
        switch (st.kind) {
            case CH_UP: chain_up(st, t - first, smem); break;
            case CH_DOWN: chain_down(st, t - first, smem); break;
            case CH_TA: chain_tile<Real, 16, true>(st, t - first, smem); break;
            case CH_N16: chain_tile<Real, 16, false>(st, t - first, smem); break;
            default: chain_tile<Real, 64, false>(st, t - first, smem); break;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(a.ctr + 1, 1u);
        }
    }
    // the last CTA to go leaves the counters zero
    if (threadIdx.x == 0 && atomicAdd(a.ctr + 2, 1u) == gridDim.x - 1)
        for (int i = 0; i < 4; ++i) a.ctr[i] = 0u;
}

// Persistent CTAs per SM: FP64 chains slow each other down on a shared SM, FP32
// ones hide each other's latencies (32768 x 128 of close pairs 2098 -> 1910 us).
template <class Real> constexpr int chain_per_sm() { return sizeof(Real) == 8 ? 1 : 2; }

constexpr size_t kChainSmemCap = 200 * 1024;     // as the TSQR's plans

template <class Real>
ChainStep<Real> *next_step(ChainRecorder &rec, int kind, int64_t nblk) {
    ChainArgs<Real> &a = rec.args<Real>();
    if (a.nsteps >= kChainSteps || nblk < 1 || nblk > INT32_MAX / 2 - a.total) return nullptr;
    ChainStep<Real> *st = &a.step[a.nsteps++];
    st->kind = kind;
    st->nblk = (int)nblk;
    st->gx = st->gy = 1;
    a.total += (int)nblk;
    rec.widest = std::max(rec.widest, (int)nblk);
    return st;
}

}  // namespace

template <class Real>
gbqr_status chain_tsqr(const Exec &ex, const TsqrParamsT<Real> &p, const TsqrPlan &pl) {
    if (pl.w > kChainMaxW) return GBQR_EINVAL;
    for (int kind : {CH_UP, CH_DOWN}) {
        ChainStep<Real> *st = next_step<Real>(*ex.chain, kind, pl.P);
        if (!st) return GBQR_EINVAL;
        st->tsqr = p;
    }
    ex.chain->smem = std::max({ex.chain->smem, pl.smem_up, pl.smem_down});
    return GBQR_OK;
}
template gbqr_status chain_tsqr(const Exec &, const TsqrParamsT<double> &, const TsqrPlan &);
template gbqr_status chain_tsqr(const Exec &, const TsqrParamsT<float> &, const TsqrPlan &);

// Tiles of 16 columns, 16 rows high and, for tall results, 64: FP64 products
// are bound by the FMAs whatever the tile.  K is split until every CTA of the
// launch has a tile, at least 4 K-tiles a split where K allows.
template <class Real>
gbqr_status chain_gemm(const Exec &ex, const GemmOpT<Real> &op, const GemmScratchT<Real> &sc) {
    const int BM = !op.ta && op.M >= (int64_t)64 * ex.num_sms ? 64 : 16;
    const int64_t tm = (op.M + BM - 1) / BM, tn = (op.N + 15) / 16, tiles = tm * tn, kt = (op.K + BK - 1) / BK;
    const int64_t ctas = (int64_t)chain_per_sm<Real>() * ex.num_sms;
    int64_t S = std::max<int64_t>(1, std::min<int64_t>({kt / (kt >= 32 ? 4 : 1), ctas / tiles, 512}));
    int slots = 1, counters = 1;
    for (; S > 1; --S) {
        tree_shape((int)S, &slots, &counters);
        if (sc.partial && sc.counters && (size_t)(tiles * slots) * BM * 16 <= sc.partial_elems && (size_t)(tiles * counters) <= sc.ncounters) break;
    }
    if (tm > INT32_MAX / 2 || tn > INT32_MAX / 2) return GBQR_EUNSUPPORTED;
    ChainStep<Real> *st = next_step<Real>(*ex.chain, op.ta ? CH_TA : (BM == 16 ? CH_N16 : CH_N64), tiles * S);
    if (!st) return GBQR_EINVAL;
    st->gx = (int)tm;
    st->gy = (int)tn;
    GemmParamsT<Real> p;
    p.M = op.M; p.N = op.N; p.K = op.K;
    p.A = op.A; p.lda = op.lda; p.maskA = op.maskA;
    p.B = op.B; p.ldb = op.ldb; p.maskB = op.maskB;
    p.C = op.C; p.ldc = op.ldc; p.alpha = op.alpha; p.beta = op.beta;
    p.partial = sc.partial; p.counters = sc.counters;
    p.slots_per_tile = S > 1 ? slots : 1;
    p.counters_per_tile = S > 1 ? counters : 1;
    st->gemm = p;
    ex.chain->smem = std::max(ex.chain->smem, sizeof(Real) * BK * (BM + 1 + 17));
    return GBQR_OK;
}
template gbqr_status chain_gemm(const Exec &, const GemmOpT<double> &, const GemmScratchT<double> &);
template gbqr_status chain_gemm(const Exec &, const GemmOpT<float> &, const GemmScratchT<float> &);

// Launches what `rec` holds; ctr: 4 counters, zero.
template <class Real>
gbqr_status chain_launch(const Exec &ex, ChainRecorder &rec, const int *flag, unsigned *ctr, int *timeout) {
    ChainArgs<Real> &a = rec.args<Real>();
    if (!a.nsteps) return GBQR_OK;
    if (rec.smem > kChainSmemCap) return GBQR_EINVAL;
    static std::atomic<bool> attr[64];           // per device and scalar type, once
    const bool cached = ex.device >= 0 && ex.device < 64;
    if (!cached || !attr[ex.device].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(panel_chain_kernel<Real>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kChainSmemCap) != cudaSuccess)
            return GBQR_ECUDA;
        if (cached) attr[ex.device].store(true, std::memory_order_release);
    }
    a.flag = flag;
    a.ctr = ctr;
    a.timeout = timeout;
    trace_begin(ex, FAM_OTHER);
    panel_chain_kernel<Real><<<std::min(rec.widest, chain_per_sm<Real>() * ex.num_sms), kThreads, rec.smem, ex.stream>>>(a);
    return trace_end(ex, FAM_OTHER, 0.0, 0.0);
}
template gbqr_status chain_launch<double>(const Exec &, ChainRecorder &, const int *, unsigned *, int *);
template gbqr_status chain_launch<float>(const Exec &, ChainRecorder &, const int *, unsigned *, int *);

}  // namespace gbqr
