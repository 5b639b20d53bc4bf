// TSQR base case of QR-EG (Algorithm 2, base case), restated for the SMs of
// one GPU (Section 5 and Appendix C).  Each CTA plays one of the paper's
// processors: it owns a contiguous block of the panel's rows.
//
//   tsqr_up_kernel     (Appendix C.1, upsweep): every CTA factors its m_p x w
//                      row block with Householder reflectors in shared memory
//                      (local-QR), keeps (V_p, T_p) and passes R_p up a
//                      fan-out-k tree.  The tree "Reduce" is fused into the
//                      same launch: the last CTA to arrive at a node (atomic
//                      arrival counter) factors the stacked upper triangles
//                      of its children; no CTA ever waits on another.
//   tsqr_down_kernel   (Appendix C.2, downsweep and reconstruction, one
//                      launch): every CTA walks from the root to leaf 0 and
//                      forms the top w x w block X of W = Q [I; 0] (from the
//                      copy of leaf 0's top V block the upsweep kept), factors
//                      X + S = LU with S_jj = sgn(X^_jj) added before
//                      eliminating column j, and inverts U.  It then walks to
//                      its own leaf applying the node Q-factors to
//                      B^(L) = U^{-1} instead of I - the shortcut noted at the
//                      end of Appendix C - so its rows of Q [U^{-1}; 0] are
//                      V_p = W_p U^{-1} directly, with no per-row triangular
//                      solve.  CTA 0 writes T = U S L^{-T}, V_top = L and
//                      R = -S R^(L).  The small LU and the walk to leaf 0 are
//                      repeated by every CTA instead of being broadcast, so
//                      the launch needs no inter-CTA waiting.
//
// Merged nodes exploit the structure of stacked triangles: the Householder
// vector of column j has a 1 in row j of the first triangle and non-zeros
// only in rows 0..j of the others, so V = [I; Y_1; ...] with each Y_i upper
// triangular and V^T [B; 0] = B in the downsweep.
#include "tsqr_block.cuh"

#include <algorithm>
#include <atomic>

namespace gbqr {
namespace {

template <class Real>
__global__ void __launch_bounds__(kThreads) tsqr_up_kernel(TsqrParamsT<Real> p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    tsqr_up(p, blockIdx.x, reinterpret_cast<Real *>(smem_raw));
}
template <class Real>
__global__ void __launch_bounds__(kThreads) tsqr_down_kernel(TsqrParamsT<Real> p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    tsqr_down<kMaxPanel>(p, blockIdx.x, reinterpret_cast<Real *>(smem_raw));
}

size_t up_smem(int ldS, int w) { return sizeof(double) * ((size_t)ldS * w + 2 * (size_t)w * w + 6 * (size_t)w); }
size_t down_smem(int ldS, int w) { return sizeof(double) * ((size_t)ldS * w + 5 * (size_t)w * w + 2 * w); }

constexpr size_t kSmemCap = 200 * 1024;
constexpr int kDefaultFanout = 8;
constexpr int kMaxFanout = 16;

}  // namespace

bool tsqr_plan(int64_t mp, int w, int leaf_rows, int fanout, int num_sms, TsqrPlan *plan) {
    if (w < 1 || w > kMaxPanel || mp < w) return false;
    TsqrPlan pl;
    pl.mp = mp; pl.w = w;
    // tallest leaf that every kernel's shared memory can hold
    const size_t cap_el = kSmemCap / sizeof(double);
    int64_t hcap = (int64_t)((cap_el - (2 * (size_t)w * w + 6 * (size_t)w)) / w);          // up
    hcap = std::min<int64_t>(hcap, (int64_t)((cap_el - 5 * (size_t)w * w - 2 * w) / w));   // down + recon
    if (hcap < w) return false;
    // default: about one leaf per SM (the leaf phase is the only one that
    // uses the whole GPU), but at least 128 rows - shorter panels then get
    // fewer leaves and one merge level less, which measured faster - and
    // never shorter than the panel is wide
    const int sms = num_sms > 0 ? num_sms : 152;
    int64_t target = leaf_rows > 0 ? leaf_rows : std::max<int64_t>({(int64_t)w, (int64_t)128, (mp + sms - 1) / sms});
    // ... and up to 256 rows where that saves a whole merge level (17 to 32
    // leaves of 128 rows become 16 of at most 256: one merge instead of two)
    if (leaf_rows <= 0 && target == 128 && (mp + 127) / 128 > kMaxFanout && (mp + kMaxFanout - 1) / kMaxFanout <= 256)
        target = (mp + kMaxFanout - 1) / kMaxFanout;
    target = std::max<int64_t>(target, w);
    int64_t P = (mp + target - 1) / target;
    P = std::max<int64_t>(P, (mp + hcap - 1) / hcap);   // leaves no taller than hcap
    P = std::min<int64_t>(P, mp / w);                    // every leaf keeps >= w rows
    P = std::max<int64_t>(P, 1);
    if (P > (1 << 24)) return false;
    pl.P = (int)P;
    pl.hmax = (int)((mp + P - 1) / P);
    if (pl.hmax > hcap) return false;
    // fan-out: as requested (2 .. 16), else the fewest serial merge levels a
    // fan-out of at most 16 gives, with the smallest such k >= 8: a level
    // costs a fixed chain of w Householder steps, while a merge grows only
    // with the k - 1 stacked triangles below its pivots.  The merge of k
    // stacked triangles (k*w rows) must fit the up kernel's shared memory.
    auto levels = [&](int kk) { int64_t n = P; int l = 0; while (n > 1) { n = (n + kk - 1) / kk; ++l; } return l; };
    int k = kDefaultFanout;
    if (fanout > 0) {
        k = std::min(kMaxFanout, std::max(2, fanout));
    } else {
        for (int c = kDefaultFanout + 1; c <= kMaxFanout; ++c)
            if (levels(c) < levels(k)) k = c;
    }
    while (k > 2 && up_smem(k * w, w) > kSmemCap) --k;
    pl.k = k;
    pl.ldS = std::max(pl.hmax, pl.k * w);   // up kernel (leaf block or k stacked triangles)
    pl.ldW = pl.hmax;                        // down kernel (leaf block only)
    int64_t nodes = P, Nl = P, L = 0, internal = 0;
    while (Nl > 1) { Nl = (Nl + pl.k - 1) / pl.k; nodes += Nl; internal += Nl; ++L; }
    if (L > 40) return false;
    pl.L = (int)L;
    pl.nodes = nodes;
    const size_t ww = (size_t)w * w;
    pl.nR = (size_t)nodes * ww;
    pl.nT = (size_t)nodes * ww;
    pl.nY = (size_t)std::max<int64_t>(internal, 1) * (pl.k - 1) * ww;
    pl.nX = ww;
    pl.ncount = (size_t)std::max<int64_t>(internal, 1);
    pl.smem_up = up_smem(pl.ldS, w);
    pl.smem_down = down_smem(pl.ldW, w);
    if (pl.smem_up > kSmemCap || pl.smem_down > kSmemCap) return false;
    *plan = pl;
    return true;
}

TsqrPlan tsqr_plan_bound(int64_t mp, int w, int leaf_rows, int fanout, int num_sms) {
    // Workspace grows with the number of leaves P.  For panels of height
    // <= mp and width ww <= w: with an explicit leaf height P grows with the
    // height; with the default (about one leaf per SM) a shorter panel can
    // round to more leaves, but never to more than the SM count.  Take the
    // larger of the two counts, then the node counts of a tree that size.
    TsqrPlan best;
    const int sms = num_sms > 0 ? num_sms : 152;
    for (int ww = 1; ww <= w; ++ww) {
        TsqrPlan pl;
        if (mp < ww || !tsqr_plan(mp, ww, leaf_rows, fanout, num_sms, &pl)) continue;
        int64_t P = pl.P;
        if (leaf_rows <= 0) P = std::max<int64_t>(P, std::min<int64_t>(sms, mp / ww));
        // a shorter panel may get another fan-out: bound over all of them
        const size_t w2 = (size_t)ww * ww;
        for (int k = 2; k <= kMaxFanout; ++k) {
            int64_t nodes = P, Nl = P, internal = 0;
            while (Nl > 1) { Nl = (Nl + k - 1) / k; nodes += Nl; internal += Nl; }
            best.nR = std::max(best.nR, (size_t)nodes * w2);
            best.nT = std::max(best.nT, (size_t)nodes * w2);
            best.nY = std::max(best.nY, (size_t)std::max<int64_t>(internal, 1) * (k - 1) * w2);
            best.ncount = std::max(best.ncount, (size_t)std::max<int64_t>(internal, 1));
        }
        best.nX = std::max(best.nX, w2);
    }
    return best;
}

template <class Real>
gbqr_status tsqr_run(const Exec &ex, const TsqrPlan &pl, Real *A, int64_t lda,
                     Real *Tout, int64_t ldt, const TsqrWorkT<Real> &work) {
    TsqrParamsT<Real> p;
    p.A = A; p.lda = lda; p.mp = pl.mp; p.w = pl.w;
    p.P = pl.P; p.k = pl.k; p.L = pl.L; p.ldS = pl.ldS; p.ldW = pl.ldW;
    p.wsR = work.R; p.wsT = work.T; p.wsY = work.Y; p.wsX = work.X;
    p.counters = work.counters;
    p.Tout = Tout; p.ldt = ldt;
    if (ex.chain) return chain_tsqr(ex, p, pl);

    // per device and scalar type, once (server workers launch from several threads)
    static std::atomic<bool> attr_done[64];
    if (!(ex.device >= 0 && ex.device < 64) || !attr_done[ex.device].load(std::memory_order_acquire)) {
        const int cap = (int)kSmemCap;
        if (cudaFuncSetAttribute(tsqr_up_kernel<Real>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap) != cudaSuccess ||
            cudaFuncSetAttribute(tsqr_down_kernel<Real>, cudaFuncAttributeMaxDynamicSharedMemorySize, cap) != cudaSuccess)
            return GBQR_ECUDA;
        if (ex.device >= 0 && ex.device < 64) attr_done[ex.device].store(true, std::memory_order_release);
    }
    const double w = pl.w, mp = (double)pl.mp;
    const double ww = w * w;
    gbqr_status st;

    trace_begin(ex, FAM_TSQR_UP);
    tsqr_up_kernel<Real><<<pl.P, kThreads, pl.smem_up, ex.stream>>>(p);
    // leaf Householder ~2 m w^2 + T ~ m w^2; merges ~ (nodes) * w^3
    st = trace_end(ex, FAM_TSQR_UP, 3.0 * mp * ww + (double)(pl.nodes - pl.P) * 1.5 * ww * w,
                   (double)sizeof(Real) * (2.0 * mp * w + 3.0 * (double)pl.nodes * ww));
    if (st != GBQR_OK) return st;

    trace_begin(ex, FAM_TSQR_DOWN);
    tsqr_down_kernel<Real><<<pl.P, kThreads, pl.smem_down, ex.stream>>>(p);
    // per leaf: two path walks (~2 L products of w^3/6 each), X, its LU and
    // U^{-1} (~2 w^3/3), and the leaf's rows of Q [U^{-1}; 0] (~m_p w^2)
    st = trace_end(ex, FAM_TSQR_DOWN,
                   2.0 * mp * ww + (double)pl.P * ((4.0 * pl.L + 4.0) * ww * w / 3.0),
                   (double)sizeof(Real) * (2.0 * mp * w + 2.0 * (double)pl.nodes * ww));
    return st;
}

template gbqr_status tsqr_run<double>(const Exec &, const TsqrPlan &, double *, int64_t, double *, int64_t,
                                     const TsqrWorkT<double> &);
template gbqr_status tsqr_run<float>(const Exec &, const TsqrPlan &, float *, int64_t, float *, int64_t,
                                    const TsqrWorkT<float> &);

}  // namespace gbqr
