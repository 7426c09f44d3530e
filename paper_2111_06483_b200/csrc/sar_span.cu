// Launches of the span kernels (see sar_span_kernels.cuh).
#include "sar_dispatch.cuh"
#include "sar_rows.cuh"
#include "sar_span.cuh"
#include "sar_span_kernels.cuh"

namespace sar {

// ---- span kernels ---------------------------------------------------------------------------------
constexpr int kCapFwd = 256, kCapDst = 256, kCapSrc = 192, kCapSum = 256;
// Resident blocks per SM the register budget is cut for.  The backward passes hold two accumulators of V vectors; over rows of
// more than 1 KB (V > 2) they spilled a hundred bytes and more at 20 blocks, twice that with the bodies for spans and segments
// in one kernel, where shared memory leaves room for 18 blocks (V = 4) or fewer.  Forward + backward, a kernel per body at 20
// blocks / one kernel at 20 / one at 16: 250,000 nodes, 3 million edges, 8 heads of 64, float32 3.33 / 3.54 / 2.68 ms, 4 heads
// of 128 2.19 / 2.32 / 2.07, 6 heads of 128, bf16 5.33 / 5.97 / 4.07; 600,000 nodes, 8 heads of 64 5.52 / 6.32 / 4.25.
constexpr int kMinBlocksFwd = 24;
template <int V> constexpr int kMinBlocksBwd = V <= 2 ? 20 : V == 4 ? 16 : 12;
constexpr size_t kStageBytes = 16 * 1024;              // shared memory a partition step may spend on the rows' own data

static int rows_per_span(long long n_rows, long long nnz, int cap) {
    const double avg = n_rows > 0 ? (double)nnz / (double)n_rows : 0.0;
    int R = avg > 0.5 ? (int)(1.0 * cap / avg + 0.5) : kMaxSpanRows;  // about cap edges per span (the long rows counted in avg are skipped)
    const long long fill = n_rows / (148 * 24);                       // no more than leaves every SM 24 spans
    if (R > fill) R = (int)fill;
    if (R < 1) R = 1;
    if (R > kMaxSpanRows) R = kMaxSpanRows;
    return R;
}

// Launches span_kernel<MODE> over the segments of the long rows and the spans of the others.  The merge launch is the caller's.
template <typename T, int G, int V, int S, int MODE, int CAP, int MINB>
static sar_status launch_span(SpanArgs a, long long nnz, const char *name, cudaStream_t st) {
    constexpr bool kIsSum = MODE == kSum || MODE == kSumW;
    constexpr int kGeo = (kIsSum || G * V >= 4) ? 1 : 0;
    const bool geo = kGeo && a.g.n_vec == G * V && (kIsSum ? a.g.H == 1 : (a.g.H == 4 && a.g.Hp == 4 && a.hvec));
    a.R = rows_per_span(a.n_rows, nnz, CAP);
    const bool whole = (a.flags & SAR_FIRST) && (a.flags & SAR_LAST);
    // A partition step of the destination-major pass stages the rows' output-gradient rows per chunk when that fits
    // kStageBytes of shared memory, with fewer rows per span if need be.
    size_t stage_bytes = 0;
    a.stage_rows = 0;
    if (!whole && (MODE == kBwdDst || MODE == kBwdDstGivenD)) {
        const size_t rsb = (size_t)a.g.n_vec * 16;
        if (rsb <= kStageBytes) {
            if ((size_t)a.R * rsb > kStageBytes) a.R = (int)(kStageBytes / rsb);
            a.stage_rows = a.R;
            stage_bytes = (size_t)a.R * rsb;
        }
    }
    const long long blocks = a.sp.n_seg + (a.n_rows + a.R - 1) / a.R;
    if (blocks <= 0) return SAR_OK;
    // the epilogue's flag tests are decided at compile time where the call holds the whole graph (a sum reads its flags)
    const bool fixed = kIsSum || (whole && !(a.flags & (SAR_KEEP_NUMERATOR | SAR_RELU_OUT)));
    auto kern = span_kernel<T, G, V, S, MODE, CAP, MINB, kIsSum ? 1 : 0, 0>;
    if (fixed) kern = geo ? span_kernel<T, G, V, S, MODE, CAP, MINB, 1, kGeo> : span_kernel<T, G, V, S, MODE, CAP, MINB, 1, 0>;
    const size_t smem = span_layout<MODE>(a.g.Hp, V, CAP, S, 32 / G, stage_bytes).total;
    SAR_TRY(ensure_smem(kern, smem));
    SAR_LAUNCH(name, st, launch(kern, (unsigned)blocks, kSpanThreads, smem, st, a));
    return sar_after_launch();
}

// stages of the gather ring: 8 x 512 bytes in flight per warp for one-vector rows
template <int V> struct UFwd { static constexpr int u = V == 1 ? 8 : (V == 2 ? 4 : 2); };
template <int V> struct UBwd { static constexpr int u = V == 1 ? 8 : (V == 2 ? 4 : 2); };

static SpanArgs span_args(const Shape &s, const RowArgs &r) {
    SpanArgs a{};
    a.n_rows = r.n_rows;
    a.indptr = r.indptr;
    a.indices = r.indices;
    a.gather = r.gather;
    a.rowvec = r.rowvec;
    a.el = r.el;
    a.er = r.er;
    a.m = r.m;
    a.d = r.d;
    a.rec_in = r.rec;
    a.rec_out = r.rec;
    a.acc_state = r.acc;
    a.m_state = r.m_io;
    a.d_state = r.d_io;
    a.out = r.out;
    a.del = r.dscal;
    a.der = r.dscal;
    a.deg_total = r.deg;
    a.src_scale = r.src_scale;
    a.dst_scale = r.dst_scale;
    a.mix = r.mix;
    a.slope = r.slope;
    a.flags = r.flags;
    a.g = s.geom;
    a.sp = r.sp;
    a.hvec = s.geom.H % 4 == 0 && sar_aligned(r.er, 16);
    return a;
}

sar_status span_fwd(const Shape &s, const RowArgs &r, long long nnz, cudaStream_t st) {
    const SpanArgs a = span_args(s, r);
    return dispatch(s, [&](auto cfg) -> sar_status {
        using C = decltype(cfg);
        return launch_span<typename C::type, C::g, C::v, UFwd<C::v>::u, kFwd, kCapFwd, kMinBlocksFwd>(a, nnz, "gat_fwd_span", st);
    });
}
sar_status span_dst(const Shape &s, const RowArgs &r, long long nnz, bool part, cudaStream_t st) {
    const SpanArgs a = span_args(s, r);
    return dispatch(s, [&](auto cfg) -> sar_status {
        using C = decltype(cfg);
        if (part) return launch_span<typename C::type, C::g, C::v, UBwd<C::v>::u, kBwdDstGivenD, kCapDst, kMinBlocksBwd<C::v>>(a, nnz, "gat_bwd_dst_span", st);
        return launch_span<typename C::type, C::g, C::v, UBwd<C::v>::u, kBwdDst, kCapDst, kMinBlocksBwd<C::v>>(a, nnz, "gat_bwd_dst_span", st);
    });
}
sar_status span_src(const Shape &s, const RowArgs &r, long long nnz, cudaStream_t st) {
    SpanArgs a = span_args(s, r);
    a.hvec = s.geom.H % 4 == 0;
    return dispatch(s, [&](auto cfg) -> sar_status {
        using C = decltype(cfg);
        return launch_span<typename C::type, C::g, C::v, UBwd<C::v>::u, kBwdSrc, kCapSrc, kMinBlocksBwd<C::v>>(a, nnz, "gat_bwd_src_span", st);
    });
}
sar_status span_sum(const Shape &s, const RowArgs &r, long long nnz, bool weighted, cudaStream_t st) {
    const SpanArgs a = span_args(s, r);
    return dispatch(s, [&](auto cfg) -> sar_status {
        using C = decltype(cfg);
        if (weighted) return launch_span<typename C::type, C::g, C::v, UFwd<C::v>::u, kSumW, kCapSum, kMinBlocksFwd>(a, nnz, "spmm_span", st);
        return launch_span<typename C::type, C::g, C::v, UFwd<C::v>::u, kSum, kCapSum, kMinBlocksFwd>(a, nnz, "spmm_span", st);
    });
}

}  // namespace sar
