// C-ABI entry points of the fused GAT aggregation and of the sum aggregation: argument checks,
// kernel selection and launches.  Declarations and contracts are in include/sar.h.
#include "sar_dispatch.cuh"
#include "sar_gat_kernels.cuh"
#include "sar_generic_kernels.cuh"
#include "sar_lean.cuh"
#include "sar_rows.cuh"
#include "sar_span.cuh"

namespace sar {

sar_launch_hook_fn g_launch_hook = nullptr;
void *g_launch_hook_user = nullptr;

sar_status make_shape(int32_t H, int32_t F, sar_dtype t, bool ptrs_16B_aligned, Shape *out) {
    if (H < 1 || F < 1) return SAR_ERR_INVALID_ARG;
    if (t != SAR_F32 && t != SAR_BF16) return SAR_ERR_INVALID_ARG;
    if ((long long)H * F > (1 << 20)) return SAR_ERR_UNSUPPORTED;
    Shape s;
    s.H = H;
    s.F = F;
    s.t = t;
    const size_t es = sar_elem_size(t);
    s.row_bytes = (size_t)H * F * es;
    const size_t head_bytes = (size_t)F * es;
    s.fast = ptrs_16B_aligned && (head_bytes % 16 == 0) && H <= SAR_MAX_HEADS && s.row_bytes <= SAR_MAX_ROW_BYTES;
    s.G = s.V = 0;
    s.geom = RowGeom{H, 1, 0, 1, 1};
    if (s.fast) {
        const int n_vec = (int)(s.row_bytes / 16);
        const int Hp = sar_pow2_ceil(H);
        int G = sar_pow2_ceil(n_vec);
        if (G > 32) G = 32;
        if (G < 4) G = 4;
        if (G < Hp) G = Hp;
        int V = sar_pow2_ceil((n_vec + G - 1) / G);
        s.G = G;
        s.V = V;
        s.geom = RowGeom{H, Hp, sar_log2(Hp), (int)(head_bytes / 16), n_vec};
    }
    *out = s;
    return SAR_OK;
}

// ---- what the row kernels work on -------------------------------------------------------------------------------
// Heads are made of whole 16-byte vectors.  Where F elements are no multiple of 16 bytes (as wide as there are classes,
// say) the rows that are gathered are copied into a padded array in the workspace first: the copy is one pass over
// [n,H,F] against a gather of every edge's row, and an aligned row touches fewer sectors than one that starts anywhere.
struct RowShape {
    bool ok;           // H and F within what the kernels cover
    bool ragged;       // F elements are no whole number of vectors
    int vph;           // vectors per head
    unsigned row_bytes;
    RowGeo geo;
};

static int pow2_at_least(int x, int lo) {
    const int p = sar_pow2_ceil(x);
    return p < lo ? lo : p;
}

static RowShape row_shape(int H, int F, sar_dtype t) {
    RowShape r{};
    const int epv = t == SAR_BF16 ? 8 : 4;
    r.ragged = F % epv != 0;
    r.vph = (F + epv - 1) / epv;
    r.row_bytes = (unsigned)H * (unsigned)r.vph * 16u;
    r.ok = H <= SAR_MAX_HEADS && (long long)H * r.vph * 16 <= (1LL << 24) && sar_pow2_ceil(r.vph) <= 256;
    const int vphp = sar_pow2_ceil(r.vph);
    int HP = sar_pow2_ceil(H) < 8 ? sar_pow2_ceil(H) : 8;
    while (HP > 1 && HP * vphp > 64) HP /= 2;
    r.geo = RowGeo{pow2_at_least(HP * vphp, HP == 8 ? 8 : 4), HP, (H + HP - 1) / HP};
    return r;
}

static RowShape sum_shape(int F, sar_dtype t) {
    RowShape r{};
    const int epv = t == SAR_BF16 ? 8 : 4;
    r.ragged = F % epv != 0;
    r.vph = (F + epv - 1) / epv;
    r.row_bytes = (unsigned)r.vph * 16u;
    r.ok = true;
    const int NV = pow2_at_least(r.vph, 4) < 64 ? pow2_at_least(r.vph, 4) : 64;
    r.geo = RowGeo{NV, 1, (r.vph + NV - 1) / NV};
    return r;
}

// [n,H,F] -> [n,H,vph*EPV], zeros behind the F elements of a head, of one array or of two (n2 > 0); one 16-byte vector per thread
template <typename T>
__global__ void __launch_bounds__(256) pad_rows_kernel(long long vecs, long long vecs2, int F, int vph, const T *__restrict__ in, uint4 *__restrict__ out,
                                                       const T *__restrict__ in2, uint4 *__restrict__ out2) {
    after_predecessor();
    constexpr int EPV = Elem<T>::EPV;
    long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    if (i >= vecs) {
        i -= vecs;
        if (i >= vecs2) return;
        in = in2;
        out = out2;
    }
    const long long nh = i / vph;
    const int f0 = (int)(i - nh * vph) * EPV;
    const T *p = in + nh * F + f0;
    float x[EPV];
#pragma unroll
    for (int k = 0; k < EPV; ++k) x[k] = f0 + k < F ? Elem<T>::load1(p + k) : 0.f;
    out[i] = Elem<T>::pack(x);
}

static sar_status pad_rows(int H, int F, const RowShape &r, sar_dtype t, long long n, const void *in, void *out, long long n2, const void *in2, void *out2,
                           cudaStream_t st) {
    const long long vecs = n * H * r.vph, vecs2 = n2 * H * r.vph;
    if (vecs + vecs2 == 0) return SAR_OK;
    const unsigned blocks = (unsigned)((vecs + vecs2 + 255) / 256);
    uint4 *o = static_cast<uint4 *>(out), *o2 = static_cast<uint4 *>(out2);
    if (t == SAR_F32)
        SAR_LAUNCH("pad_rows", st, launch(pad_rows_kernel<float>, blocks, 256, 0, st, vecs, vecs2, F, r.vph, static_cast<const float *>(in), o, static_cast<const float *>(in2), o2));
    else
        SAR_LAUNCH("pad_rows", st, launch(pad_rows_kernel<__nv_bfloat16>, blocks, 256, 0, st, vecs, vecs2, F, r.vph, static_cast<const __nv_bfloat16 *>(in), o, static_cast<const __nv_bfloat16 *>(in2), o2));
    return sar_after_launch();
}

// The start of a propagation: x0 with padded rows and / or scaled row by row (either may be null); one 16-byte vector per thread
template <typename T>
__global__ void __launch_bounds__(256) propagate_start_kernel(long long vecs, int F, int vph, const T *__restrict__ in, const float *__restrict__ scale,
                                                              uint4 *__restrict__ padded, uint4 *__restrict__ scaled) {
    after_predecessor();
    constexpr int EPV = Elem<T>::EPV;
    const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
    if (i >= vecs) return;
    const long long row = i / vph;
    const int f0 = (int)(i - row * vph) * EPV;
    const T *p = in + row * F + f0;
    float x[EPV];
#pragma unroll
    for (int k = 0; k < EPV; ++k) x[k] = f0 + k < F ? Elem<T>::load1(p + k) : 0.f;
    if (padded) padded[i] = Elem<T>::pack(x);
    if (scaled) {
        const float s = __ldg(scale + row);
#pragma unroll
        for (int k = 0; k < EPV; ++k) x[k] *= s;
        scaled[i] = Elem<T>::pack(x);
    }
}
static sar_status propagate_start(long long n, int F, const RowShape &r, sar_dtype t, const void *in, const float *scale, void *padded, void *scaled,
                                  cudaStream_t st) {
    const long long vecs = n * r.vph;
    const unsigned blocks = (unsigned)((vecs + 255) / 256);
    uint4 *p = static_cast<uint4 *>(padded), *s = static_cast<uint4 *>(scaled);
    if (t == SAR_F32)
        SAR_LAUNCH("propagate_start", st, launch(propagate_start_kernel<float>, blocks, 256, 0, st, vecs, F, r.vph, static_cast<const float *>(in), scale, p, s));
    else
        SAR_LAUNCH("propagate_start", st, launch(propagate_start_kernel<__nv_bfloat16>, blocks, 256, 0, st, vecs, F, r.vph, static_cast<const __nv_bfloat16 *>(in), scale, p, s));
    return sar_after_launch();
}
// padded rows -> rows of F elements.  Sixteen bytes of the result per thread where it is aligned, else an element; the index of
// the row by a 32-bit division where there are no more than 2^32 elements.  Bound by that index arithmetic, not by the bytes, with
// an element per thread and 64 bits: 500,000 rows of 47 float32 100 us, now 34 (each with some 6 us of its launch; the bytes 29).
template <typename T, typename I, int N>
__global__ void __launch_bounds__(256) strip_rows_kernel(long long elems, int F, int pitch, const T *__restrict__ in, T *__restrict__ out) {
    after_predecessor();
    const long long i = ((long long)blockIdx.x * 256 + threadIdx.x) * N;
    if (i >= elems) return;
    long long row = (I)i / (I)F;
    int at = (int)((I)i - (I)row * (I)F);
    alignas(16) T x[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
        if (i + k < elems) x[k] = in[row * pitch + at];
        if (++at == F) {
            at = 0;
            ++row;
        }
    }
    if (N > 1 && i + N <= elems) {
        *reinterpret_cast<uint4 *>(out + i) = *reinterpret_cast<const uint4 *>(x);
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (i + k < elems) out[i + k] = x[k];
    }
}
template <typename T>
static sar_status strip_rows_as(long long elems, int F, int pitch, const void *in, void *out, cudaStream_t st) {
    constexpr int N = 16 / sizeof(T);
    const T *p = static_cast<const T *>(in);
    T *o = static_cast<T *>(out);
    const unsigned blocks = (unsigned)((elems + 255) / 256), blocks_n = (unsigned)((elems + 256 * N - 1) / (256 * N));
    if (elems + N > 0xffffffffLL)
        SAR_LAUNCH("strip_rows", st, launch(strip_rows_kernel<T, unsigned long long, 1>, blocks, 256, 0, st, elems, F, pitch, p, o));
    else if (sar_aligned(out, 16))
        SAR_LAUNCH("strip_rows", st, launch(strip_rows_kernel<T, unsigned, N>, blocks_n, 256, 0, st, elems, F, pitch, p, o));
    else
        SAR_LAUNCH("strip_rows", st, launch(strip_rows_kernel<T, unsigned, 1>, blocks, 256, 0, st, elems, F, pitch, p, o));
    return sar_after_launch();
}
static sar_status strip_rows(long long n, int F, const RowShape &r, sar_dtype t, const void *in, void *out, cudaStream_t st) {
    const int pitch = (int)(r.row_bytes / sar_elem_size(t));
    return t == SAR_F32 ? strip_rows_as<float>(n * F, F, pitch, in, out, st) : strip_rows_as<__nv_bfloat16>(n * F, F, pitch, in, out, st);
}

// ---- workspace layout ---------------------------------------------------------------------------
// [ destination records: n_dst*H float4 ][ padded gout ][ segments of the CSR ][ segments of the CSC ][ padded feat ]
// (the padded arrays for ragged shapes only).  The records are what sar_gat_bwd_prepare leaves for a step.  Everything else
// is written by the call that reads it, but for the copy of gout with SAR_SAME_WORKSPACE: its place, like that of the
// records, does not depend on the partition.
static size_t rec_bytes(long long n_dst, int H) { return sar_round_up((size_t)n_dst * H * 16, 256); }
static long long part_stride(int H, const RowShape &r, sar_dtype t) {  // floats per segment, a multiple of 4 (float4 rows)
    return ((long long)H * r.vph * (t == SAR_BF16 ? 8 : 4) + 3LL * H + 3) & ~3LL;
}
static size_t part_bytes(const sar_split *sp, int H, const RowShape &r, sar_dtype t) {
    return sp ? sar_round_up((size_t)sp->n_seg * part_stride(H, r, t) * 4, 256) : 0;
}
static size_t pad_bytes(long long n, const RowShape &r) { return r.ragged ? sar_round_up((size_t)n * r.row_bytes, 256) : 0; }

static SplitArgs split_args(const sar_split *sp, float *part, int H, const RowShape &r, sar_dtype t) {
    SplitArgs a;
    a.threshold = 0;
    a.n_long = 0;
    a.n_seg = 0;
    a.long_row = nullptr;
    a.long_seg = nullptr;
    a.part = part;
    a.pstride = part_stride(H, r, t);
    if (sp && sp->n_long > 0 && sp->threshold > 0) {
        a.threshold = sp->threshold;
        a.n_long = sp->n_long;
        a.n_seg = sp->n_seg;
        a.long_row = sp->long_row;
        a.long_seg = sp->long_seg;
    }
    return a;
}

static sar_status check_split(const sar_split *sp) {
    if (!sp) return SAR_OK;
    if (sp->threshold < 1 || sp->n_long < 0 || sp->n_seg < 0) return SAR_ERR_INVALID_ARG;
    if (sp->n_long > 0 && (!sp->long_row || !sp->long_seg)) return SAR_ERR_INVALID_ARG;
    return SAR_OK;
}

static sar_status check_part(const sar_part *g, bool need_csc) {
    if (!g) return SAR_ERR_INVALID_ARG;
    if (g->n_dst < 0 || g->n_src < 0 || g->nnz < 0) return SAR_ERR_INVALID_ARG;
    if (g->n_src > INT32_MAX) return SAR_ERR_UNSUPPORTED;
    if (!g->indptr || (g->nnz > 0 && !g->indices)) return SAR_ERR_INVALID_ARG;
    if (!sar_aligned(g->indptr, 8) || !sar_aligned(g->indices, 4)) return SAR_ERR_ALIGNMENT;
    if (need_csc) {
        if (!g->t_indptr || (g->nnz > 0 && !g->t_indices)) return SAR_ERR_INVALID_ARG;
        if (!sar_aligned(g->t_indptr, 8) || !sar_aligned(g->t_indices, 4)) return SAR_ERR_ALIGNMENT;
    }
    SAR_TRY(check_split(g->split));
    SAR_TRY(check_split(g->t_split));
    return SAR_OK;
}


// The row kernels, or the span kernels (for the shapes that the lean kernels do not cover)?  Times of the span kernels over
// those of the row kernels, on 8,000 to a million nodes with 2 to 32 edges per node, endpoints uniform and with hubs of
// n^0.65 edges, plans of 256:
//  * Arrays that do not fit the L2 (126 MB): the span kernels, whose ring keeps more bytes in flight.  Forward + backward
//    400,000 nodes of 256 bytes 1.55 against 1.43 ms, 1 million of 576 bytes 10.3 against 12.0.
//  * Heads: the row kernel holds the scalars of a tile's heads in registers (four or eight heads spill, see there).  One or
//    two heads: backward 1.0 to 1.5.  Tiles of eight heads: backward 0.42 to 1.05, steps 0.55 to 1.15.  Tiles of four: backward
//    0.6 to 0.95 with up to 16 edges per row from 20,000 rows on, 1.0 to 1.24 else.
//  * Rows of 512 bytes to 1 KB in tiles of four or eight heads: backward 0.42 to 0.9, forward steps 0.5 to 1.0 (8,000
//    uniform rows: up to 1.1), forward 0.55 to 0.98 with up to 12 edges per row.
//  * Short rows: a row kernel's warp spends its time on the starts and ends of rows, a span kernel's gathers across them.
//    Forward, from 60,000 rows on: 0.56 to 1.05 with up to 6 edges per row (in a step up to 4), 1.0 to 1.8 with more; with
//    20,000 rows 0.9 to 1.5.  Rows below 128 bytes: 0.95 to 1.6 throughout.
//  * Rows of more than 1 KB, backward, where they fit the L2: steps 0.85 to 1.45 (4 heads of 256, float32: 1.3 to 2.1); whole 0.52 to
//    1.05 with four heads or more, from 20,000 rows on with up to 16 edges per row (6 heads of 128, bf16: 1.1 to 1.25), 0.86
//    to 1.5 else.
// With these lines the choice costs 1.1 % over the better kernel of each call in the mean, over shapes of up to 1 KB; with lines drawn
// by the number of heads alone it was 2.8 %.
constexpr unsigned long long kSpanBytes = 128ull << 20;
static bool takes_span(const Shape &s, const RowGeo &geo, long long n_gathered, long long n_rows, long long nnz, bool backward, bool part) {
    if (!s.fast) return false;
    if ((unsigned long long)n_gathered * s.row_bytes > kSpanBytes) return true;
    if (s.row_bytes < 128) return false;
    const bool over_1k = s.row_bytes > 1024, wide = geo.HP >= 4 && geo.NV >= 64 && !over_1k;
    const bool short_rows = n_rows >= 20000 && nnz <= 16 * n_rows;
    if (backward && over_1k) return !part && s.geom.H >= 4 && short_rows;
    if (backward) return wide || geo.HP == 8 || (geo.HP == 4 && short_rows);
    if (wide) return part || nnz <= 12 * n_rows;
    return n_rows >= 60000 && nnz <= (part ? 4 : 6) * n_rows;
}

// The kernel for short rows (a row per group of lanes, sar_short_kernel.cuh) instead of either?  It wins where a row's start and
// end cost the others more than its edges: few edges per row, narrow rows, many heads in a tile.  Times of the kernel that
// takes the call otherwise over those of the kernel for short rows, 1,000 to 3 million nodes, 1 to 60 edges per node, endpoints
// uniform / with hubs of n^0.65 edges, tiles of NV vectors and HP heads:
//  * NV <= 8, HP <= 2.  From 16,000 rows on forward 1.2 to 5.2 / 1.1 to 3.2 with up to 12 edges per row, NV = 4 0.9 to 1.3 / 1.0 to
//    1.4 and NV = 8 0.8 to 1.0 / 0.9 to 1.1 with 20, 0.7 to 0.9 / 0.8 to 1.3 with 30.  Backward 1.1 to 5 / 1.1 to 3.8, NV = 4 up to 28
//    edges, NV = 8 0.85 to 1.1 with 20.
//  * NV <= 8, HP = 4: forward 0.9 to 3.2 / 1.1 to 2.0 with up to 24; backward 1.1 to 4.4 / 1.2 to 2.7 with up to 60.
//  * HP = 8: backward 1.3 to 5.7 / 1.1 to 4.0; forward 0.96 to 3.5 / 1.0 to 2.6 with up to 30 (NV = 32, in arrays of up to 32 MB:
//    0.96 to 1.5 / 0.9 to 1.2 with up to 14; else 0.73 to 1.2).
//    In launches of up to 10,000 rows with some of 60 and more edges among them, HP >= 4, backward: 1.0 to 2.1, and in 20 of 600 calls 0.78 to
//    0.95, NV = 4 with rows of 100 to 160 edges (0.81 to 0.92) and NV = 32 with ones of 60 to 100 in 1,200 to 1,600 rows (0.78 to 0.93).
//  * NV = 16, HP = 4: forward 1.0 to 1.75 / 0.95 to 1.07 with up to 10, backward 1.1 to 2.2 / 0.95 to 1.4 with up to 16.
// The rest is decided by rows of up to 100 or 240 edges, too short for segments, among ones of 2 to 20: a group waits for the longest
// row of its warp, and the plan doesn't tell such graphs from uniform ones.
//  * NV = 16, HP = 2: backward 1.0 to 1.24 with up to 6 (uniform up to 1.9); forward 0.84 to 1.13 and HP = 1 0.82 to 1.13 (uniform 1.0
//    to 1.67): not taken.
//  * NV = 32, HP = 4, backward: in arrays of up to 8 MB 1.0 to 1.23 with up to 10; of 12 MB 0.87 to 0.99, of 50 to 77 MB 0.74 to 0.89.
//  * Few rows do not fill the chip with groups.  HP >= 4, backward: 8,000 rows as above with half of these edges (1.05 to 1.9).  Else
//    16,000 rows with half (1.0 to 1.9; with as many 0.8 to 1.1), 8,000 with a quarter (1.0 to 1.24), with NV >= 8, HP = 1 or
//    NV = 16, HP = 2 not (0.89 to 1.07).
// `filled`: rows with which the limit holds in full
static bool few_edges(double limit, long long filled, long long n_rows, long long nnz) {
    const double fill = n_rows < filled ? (double)n_rows / (double)filled : 1.0;
    return limit > 0 && nnz < (1LL << 30) && (double)nnz <= limit * fill * (double)n_rows;
}
static bool takes_short(const RowGeo &geo, long long n_gathered, unsigned row_bytes, long long n_rows, long long nnz, bool backward) {
    if (n_rows < 12000 && ((geo.HP == 1 && geo.NV >= 8) || (geo.HP == 2 && geo.NV >= 16))) return false;
    return few_edges(short_edges(geo.NV, geo.HP, backward, (unsigned long long)n_gathered * row_bytes), geo.HP >= 4 && backward ? 16000 : 32000, n_rows, nnz);
}
// Sums, likewise, from 12,000 rows on (8,000: 0.83 to 1.06): rows of 64 bytes 1.0 to 4.1 / 1.0 to 2.4 with up to 20 edges per row; of 128
// bytes, in arrays of up to 12 MB 1.1 to 2.4 / 1.0 to 1.4 with up to 14, up to 64 MB 1.1 to 1.9 / 1.0 to 1.3 with up to 8, beyond 1.1 to
// 1.6 / 1.0 to 1.2 with up to 3; of 256 bytes 0.91 to 1.2 (uniform up to 1.5): not taken.
static bool sum_takes_short(const RowGeo &geo, long long n_gathered, unsigned row_bytes, long long n_rows, long long nnz) {
    const unsigned long long bytes = (unsigned long long)n_gathered * row_bytes;
    const double limit = geo.tiles > 1 || n_rows < 12000 ? 0 : sum_short_edges(geo.NV, bytes);
    return few_edges(limit, 32000, n_rows, nnz);
}
// A sum has nothing between its ids and its rows.  Where the L2 doesn't hold the array the span kernels' ring keeps more loads in
// flight (2.45 million rows of 1 KB 12.5 against 15.0 ms, 500,000 of 192 bytes with 20 edges each and hubs 0.67 against 0.72); where it does,
// and a row has a dozen edges or more to spread the start of a row over, the row kernels issue less per edge.  They lose by
// less than that the more edges a row has, so the line is a number of MB per edge of the mean row (up to 32 edges, 100 MB in all).  Over
// 782 sizes of array, rows and graph, span / row on the row kernels' side of the line:
//  * float32, rows of 144 to 512 bytes other than 256 (the span kernels leave lanes idle): plain 0.98 to 1.90, 1.35 in the median,
//    weighted 1.05 to 1.83 / 1.46, with the propagation's mix 1.04 to 1.70 / 1.31; with long rows, whose hubs make the row kernels
//    wait, 1.00 to 1.59 / 1.2 to 1.3; bf16 0.97 to 1.54 / 1.1 to 1.23.
//  * rows of 528 to 768 bytes, no long rows, in up to 40 MB: float32 1.12 to 1.70 / 1.4, bf16 weighted 1.08 to 1.30.
//  * rows of 128 and 256 bytes, full lanes in either: half the MB, from 20 edges on, 0.97 to 1.41 / 1.1 to 1.25, no mix (12 edges 0.87 to 1.0).
// Beyond the line 0.55 to 1.1.
// The numbers are where the measured curves cross and no model's.  What moves them, as far as the counters show: the ring costs a span kernel
// its instructions for every slot (82 % of the issue slots busy at 42 an edge of 512 bytes), while a row kernel waits for memory once in four slots, which
// costs the more the fewer gathers the L2 answers and the more a row reads besides (the mix: x0's row and a factor).
static bool sum_takes_rows(const RowArgs &a, sar_dtype t, long long n_gathered, long long nnz, bool weighted) {
    const int vecs = (int)(a.row_bytes / 16);
    const bool hubs = a.sp.n_long > 0, mix = a.mix.x0 != nullptr, f32 = t == SAR_F32;
    if (vecs < 8 || vecs > 48 || nnz < (hubs || vecs == 8 || vecs == 16 ? 20 : 12) * a.n_rows) return false;
    double mb = f32 ? (mix ? (hubs ? 1.25 : 1.8) : weighted ? (hubs ? 3.2 : 5.0) : hubs ? 2.5 : 3.2)
                    : (mix ? (hubs ? 0.0 : 0.9) : weighted ? (hubs ? 1.5 : 2.4) : hubs ? 1.0 : 1.9);
    if (vecs == 8 || vecs == 16) mb = mix || (!f32 && (!weighted || hubs)) ? 0.0 : 0.5 * mb;
    else if (vecs > 32 && (hubs || (!f32 && (!weighted || mix)))) mb = 0.0;
    else if (vecs < 16 && hubs && !f32 && !weighted) mb = 0.0;
    const double mean = (double)nnz / (double)a.n_rows, most = vecs > 32 ? 40.0 : 100.0, line = mb * (mean < 32.0 ? mean : 32.0);
    return (double)n_gathered * a.row_bytes <= (line < most ? line : most) * 1e6;
}
static bool sum_takes_span(const Shape &s, const RowArgs &a, sar_dtype t, long long n_gathered, long long nnz, bool weighted) {
    return s.fast && (unsigned long long)n_gathered * s.row_bytes > kSpanSumBytes && !sum_takes_rows(a, t, n_gathered, nnz, weighted);
}

static sar_status check_shape(int32_t H, int32_t F, sar_dtype t) {
    Shape s;
    return make_shape(H, F, t, false, &s);
}

// the per-head scalars of a tile's row can be read as one or two float4 (float2 for two heads)
static int heads_aligned(int H, int HP, std::initializer_list<const void *> ps) {
    if (H % HP != 0) return 0;
    for (const void *p : ps)
        if (p && !sar_aligned(p, HP >= 4 ? 16 : (size_t)HP * 4)) return 0;
    return 1;
}

}  // namespace sar

using namespace sar;

extern "C" {

const char *sar_status_string(sar_status s) {
    switch (s) {
        case SAR_OK: return "ok";
        case SAR_ERR_INVALID_ARG: return "invalid argument";
        case SAR_ERR_UNSUPPORTED: return "unsupported shape";
        case SAR_ERR_ALIGNMENT: return "misaligned pointer";
        case SAR_ERR_WORKSPACE: return "workspace missing or too small";
        case SAR_ERR_CUDA: return "CUDA error";
        case SAR_ERR_BAD_GRAPH: return "inconsistent graph";
    }
    return "unknown status";
}

void sar_set_launch_hook(sar_launch_hook_fn hook, void *user) {
    g_launch_hook = hook;
    g_launch_hook_user = user;
}

int32_t sar_built_for_sm(void) {
#ifdef SAR_BUILT_FOR_SM
    return SAR_BUILT_FOR_SM;
#else
    return 0;
#endif
}

// Offsets of the workspace's parts, and what a call that needs all of them (`full`) or no padded copies asks for.
struct WsLayout {
    size_t gout, csr, csc, feat, full, plain;
};
static WsLayout ws_layout(const sar_part *g, int H, const RowShape &r, sar_dtype t) {
    WsLayout w;
    w.gout = rec_bytes(g->n_dst, H);
    w.csr = w.gout + pad_bytes(g->n_dst, r);
    w.csc = w.csr + part_bytes(g->split, H, r, t);
    w.feat = w.csc + part_bytes(g->t_split, H, r, t);
    w.full = w.feat + pad_bytes(g->n_src, r);
    w.plain = w.gout;
    return w;
}

size_t sar_gat_workspace_bytes(const sar_part *g, int32_t H, int32_t F, sar_dtype t) {
    if (!g || H < 1 || F < 1) return 0;
    return ws_layout(g, H, row_shape(H, F, t), t).full + 256;
}

size_t sar_spmm_workspace_bytes(const sar_part *g, int32_t F, sar_dtype t) {
    if (!g || F < 1) return 0;
    const RowShape r = sum_shape(F, t);
    return part_bytes(g->split, 1, r, t) + pad_bytes(g->n_src, r) + 256;
}

// ---------------------------------------------------------------------------------------------
sar_status sar_gat_fwd(const sar_part *g, const void *feat_q, const float *el, const float *er_q, int32_t H,
                       int32_t F, sar_dtype t, float slope, uint32_t flags, float *acc, float *m, float *d,
                       void *out, void *workspace, size_t workspace_bytes, void *stream) {
    SAR_TRY(check_part(g, false));
    if (flags & ~(SAR_FIRST | SAR_LAST | SAR_KEEP_NUMERATOR | SAR_RELU_OUT)) return SAR_ERR_INVALID_ARG;
    const bool first = flags & SAR_FIRST, last = flags & SAR_LAST;
    if ((flags & (SAR_KEEP_NUMERATOR | SAR_RELU_OUT)) && !last) return SAR_ERR_INVALID_ARG;
    if (!el || !m || !d) return SAR_ERR_INVALID_ARG;
    if (g->n_src > 0 && (!feat_q || !er_q)) return SAR_ERR_INVALID_ARG;
    if (last && !out) return SAR_ERR_INVALID_ARG;
    const bool part = !(first && last) || (flags & SAR_KEEP_NUMERATOR);
    if (part && !acc) return SAR_ERR_INVALID_ARG;
    SAR_TRY(check_elem_align({el, er_q, m, d, acc}, 4));
    SAR_TRY(check_elem_align({feat_q, out}, sar_elem_size(t)));
    SAR_TRY(check_shape(H, F, t));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (g->n_dst == 0) return SAR_OK;

    const RowShape r = row_shape(H, F, t);
    const WsLayout w = ws_layout(g, H, r, t);
    const bool use_split = g->split && g->split->n_long > 0;
    const bool have_ws = workspace && sar_aligned(workspace, 16);
    char *wsb = static_cast<char *>(workspace);
    const bool rows = r.ok && (r.ragged ? have_ws && workspace_bytes >= w.full : all16({feat_q, out, acc}));
    if (!rows) {
        GenericArgs a{};
        a.n_dst = g->n_dst;
        a.indptr = g->indptr;
        a.indices = g->indices;
        a.feat = feat_q;
        a.el = el;
        a.er = er_q;
        a.acc = acc;
        a.m = m;
        a.d = d;
        a.out = out;
        a.H = H;
        a.F = F;
        a.slope = slope;
        a.flags = flags;
        const long long n = g->n_dst * H;
        const unsigned blocks = (unsigned)((n + 255) / 256);
        if (t == SAR_F32)
            SAR_LAUNCH("gat_fwd_generic", st, gat_fwd_generic<float><<<blocks, 256, 0, st>>>(a));
        else
            SAR_LAUNCH("gat_fwd_generic", st, gat_fwd_generic<__nv_bfloat16><<<blocks, 256, 0, st>>>(a));
        return sar_after_launch();
    }

    if (use_split && (!have_ws || workspace_bytes < w.csc)) return SAR_ERR_WORKSPACE;
    RowArgs a{};
    a.n_rows = g->n_dst;
    a.indptr = g->indptr;
    a.indices = g->indices;
    a.last_col = (unsigned)(g->n_src > 0 ? g->n_src - 1 : 0);
    a.gather = feat_q;
    a.row_bytes = r.row_bytes;
    a.el = el;
    a.er = er_q;
    a.acc = acc;
    a.m_io = m;
    a.d_io = d;
    a.out = out;
    a.slope = slope;
    a.flags = flags;
    a.H = H;
    a.F = F;
    a.vph = r.vph;
    a.ragged = r.ragged;
    a.hvec = heads_aligned(H, r.geo.HP, {el, er_q});
    a.sp = split_args(g->split, use_split ? reinterpret_cast<float *>(wsb + w.csr) : nullptr, H, r, t);
    if (r.ragged) {
        SAR_TRY(pad_rows(H, F, r, t, g->n_src, feat_q, wsb + w.feat, 0, nullptr, nullptr, st));
        a.gather = wsb + w.feat;
    }
    Shape s;
    SAR_TRY(make_shape(H, F, t, !r.ragged, &s));
    const bool lean_shape = lean_shape_applies(s, slope, g->split, g->n_src) && sar_aligned(er_q, 16);
    const bool lean = lean_shape && !part;
    const bool lean_part = lean_shape && part && !(first && last);
    if (lean || lean_part) {
        LeanArgs la{};
        la.n_rows = g->n_dst;
        la.indptr = g->indptr;
        la.indices = g->indices;
        la.gather = feat_q;
        la.el = el;
        la.er = er_q;
        la.m_out = m;
        la.d_out = d;
        la.acc_state = acc;
        la.first = first ? 1 : 0;
        la.out = out;
        la.relu = (flags & SAR_RELU_OUT) ? 1 : 0;
        la.slope = slope;
        la.sp = a.sp;
        la.sp.threshold = g->split->threshold;
        if (lean) {
            SAR_TRY(t == SAR_F32 ? lean_fwd_f32(s, la, g->nnz, st) : lean_fwd_bf16(s, la, g->nnz, st));
            return use_split ? rows_fwd_merge(a, t, st) : SAR_OK;
        }
        SAR_TRY(t == SAR_F32 ? lean_fwd_part_f32(s, la, g->nnz, st) : lean_fwd_part_bf16(s, la, g->nnz, st));
        // The last step folds like the others; a launch of its own divides all rows (most have no edge in a given partition).
        if (last) a.flags = first ? SAR_FIRST : 0;
        if (use_split) SAR_TRY(rows_fwd_merge(a, t, st));
        if (last) {
            a.flags = flags;
            SAR_TRY(rows_fwd_finalize(a, t, st));
        }
        return SAR_OK;
    }
    a.lone = takes_short(r.geo, g->n_src, r.row_bytes, g->n_dst, g->nnz, false);
    if (!a.lone && takes_span(s, r.geo, g->n_src, g->n_dst, g->nnz, false, part))
        SAR_TRY(span_fwd(s, a, g->nnz, st));
    else if (part)
        SAR_TRY(t == SAR_F32 ? rows_fwd_part_f32(a, r.geo, g->nnz, st) : rows_fwd_part_bf16(a, r.geo, g->nnz, st));
    else
        SAR_TRY(t == SAR_F32 ? rows_fwd_f32(a, r.geo, g->nnz, st) : rows_fwd_bf16(a, r.geo, g->nnz, st));
    return use_split ? rows_fwd_merge(a, t, st) : SAR_OK;
}

static sar_status check_fused(const sar_part *g, int32_t k, const int64_t *bounds) {
    if (!g || !bounds || k < 1) return SAR_ERR_INVALID_ARG;
    if (k > SAR_MAX_PARTS) return SAR_ERR_UNSUPPORTED;
    if (bounds[0] != 0 || bounds[k] != g->n_src) return SAR_ERR_INVALID_ARG;
    for (int32_t q = 0; q < k; ++q)
        if (bounds[q + 1] < bounds[q]) return SAR_ERR_INVALID_ARG;
    return SAR_OK;
}

sar_status sar_gat_fwd_fused(const sar_part *g, int32_t k, const int64_t *bounds, const void *feat, const float *el,
                             const float *er, int32_t H, int32_t F, sar_dtype t, float slope, float *m, float *d,
                             void *out, void *workspace, size_t workspace_bytes, void *stream) {
    SAR_TRY(check_fused(g, k, bounds));
    // Sources ascend within a row, so walking a row once IS the partition-after-partition visit.
    return sar_gat_fwd(g, feat, el, er, H, F, t, slope, SAR_FIRST | SAR_LAST, nullptr, m, d, out, workspace,
                       workspace_bytes, stream);
}

// ---------------------------------------------------------------------------------------------
sar_status sar_gat_bwd_prepare(int64_t n_dst, int32_t H, int32_t F, sar_dtype t, const void *out_or_acc,
                               int32_t acc_is_numerator, const void *gout, const float *el, const float *m,
                               const float *d, float *D, void *workspace, size_t workspace_bytes, void *stream) {
    if (n_dst < 0 || !out_or_acc || !gout || !el || !m || !d) return SAR_ERR_INVALID_ARG;
    if (!workspace || !sar_aligned(workspace, 16) || workspace_bytes < (size_t)n_dst * H * 16) return SAR_ERR_WORKSPACE;
    SAR_TRY(check_elem_align({el, m, d, D}, 4));
    SAR_TRY(check_elem_align({gout}, sar_elem_size(t)));
    SAR_TRY(check_elem_align({out_or_acc}, acc_is_numerator ? 4 : sar_elem_size(t)));
    Shape s;
    SAR_TRY(make_shape(H, F, t, all16({out_or_acc, gout}), &s));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (n_dst == 0) return SAR_OK;
    if (!s.fast) {
        GenericArgs a{};
        a.n_dst = n_dst;
        a.out_in = out_or_acc;
        a.gout = gout;
        a.el = el;
        a.m_in = m;
        a.d_in = d;
        a.D = D;
        a.rec = static_cast<float4 *>(workspace);
        a.H = H;
        a.F = F;
        a.acc_is_numerator = acc_is_numerator;
        const unsigned blocks = (unsigned)((n_dst * H + 255) / 256);
        if (t == SAR_F32)
            SAR_LAUNCH("gat_bwd_prepare_generic", st, gat_bwd_prepare_generic<float><<<blocks, 256, 0, st>>>(a));
        else
            SAR_LAUNCH("gat_bwd_prepare_generic", st, gat_bwd_prepare_generic<__nv_bfloat16><<<blocks, 256, 0, st>>>(a));
        return sar_after_launch();
    }
    PrepArgs a;
    a.n_dst = n_dst;
    a.out = out_or_acc;
    a.gout = gout;
    a.el = el;
    a.m = m;
    a.d = d;
    a.D = D;
    a.rec = static_cast<float4 *>(workspace);
    a.acc_is_numerator = acc_is_numerator;
    a.g = s.geom;
    return dispatch(s, [&](auto cfg) -> sar_status {
        using C = decltype(cfg);
        using T = typename C::type;
        const size_t smem = (size_t)kWarpsPerBlock * 32 * C::v * 4;
        const unsigned blocks = blocks_for((n_dst + PrepRows<C::v>::n - 1) / PrepRows<C::v>::n, C::g);
        if (acc_is_numerator)
            SAR_LAUNCH("gat_bwd_prepare", st, (launch(gat_bwd_prepare_kernel<T, C::g, C::v, true>, blocks, kThreads, smem, st, a)));
        else
            SAR_LAUNCH("gat_bwd_prepare", st, (launch(gat_bwd_prepare_kernel<T, C::g, C::v, false>, blocks, kThreads, smem, st, a)));
        return sar_after_launch();
    });
}

sar_status sar_gat_bwd(const sar_part *g, const void *feat_q, const float *el, const float *er_q, const float *m,
                       const float *d, const void *gout, int32_t H, int32_t F, sar_dtype t, float slope,
                       uint32_t flags, void *dfeat_q, float *del, float *der_q, void *workspace,
                       size_t workspace_bytes, void *stream) {
    SAR_TRY(check_part(g, true));
    if (flags & ~(SAR_FIRST | SAR_LAST | SAR_SAME_WORKSPACE)) return SAR_ERR_INVALID_ARG;
    if ((flags & SAR_FIRST) && (flags & SAR_SAME_WORKSPACE)) return SAR_ERR_INVALID_ARG;
    if (!el || !m || !d || !gout || !del) return SAR_ERR_INVALID_ARG;
    if (g->n_src > 0 && (!feat_q || !er_q || !dfeat_q || !der_q)) return SAR_ERR_INVALID_ARG;
    SAR_TRY(check_elem_align({el, er_q, m, d, del, der_q}, 4));
    SAR_TRY(check_elem_align({feat_q, gout, dfeat_q}, sar_elem_size(t)));
    SAR_TRY(check_shape(H, F, t));
    const RowShape r = row_shape(H, F, t);
    const WsLayout w = ws_layout(g, H, r, t);
    const bool rows = r.ok && (r.ragged ? workspace_bytes >= w.full : all16({feat_q, gout, dfeat_q}));
    if (!workspace || !sar_aligned(workspace, 16) || workspace_bytes < (rows ? w.feat : w.plain)) return SAR_ERR_WORKSPACE;
    const bool whole = (flags & SAR_FIRST) && (flags & SAR_LAST);  // D rebuilt from the edges
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char *wsb = static_cast<char *>(workspace);
    float4 *rec = reinterpret_cast<float4 *>(wsb);
    if (!rows) {
        GenericArgs a{};
        a.n_dst = g->n_dst;
        a.n_src = g->n_src;
        a.indptr = g->indptr;
        a.indices = g->indices;
        a.t_indptr = g->t_indptr;
        a.t_indices = g->t_indices;
        a.feat = feat_q;
        a.gout = gout;
        a.el = el;
        a.er = er_q;
        a.m_in = m;
        a.d_in = d;
        a.dfeat = dfeat_q;
        a.del = del;
        a.der = der_q;
        a.rec = rec;
        a.H = H;
        a.F = F;
        a.slope = slope;
        a.flags = flags;
        a.given_d = whole ? 0 : 1;
        if (g->n_dst > 0) {
            const unsigned blocks = (unsigned)((g->n_dst * H + 255) / 256);
            if (t == SAR_F32)
                SAR_LAUNCH("gat_bwd_dst_generic", st, gat_bwd_dst_generic<float><<<blocks, 256, 0, st>>>(a));
            else
                SAR_LAUNCH("gat_bwd_dst_generic", st, gat_bwd_dst_generic<__nv_bfloat16><<<blocks, 256, 0, st>>>(a));
            SAR_TRY(sar_after_launch());
        }
        if (g->n_src > 0) {
            const unsigned blocks = (unsigned)((g->n_src * H + 255) / 256);
            if (t == SAR_F32)
                SAR_LAUNCH("gat_bwd_src_generic", st, gat_bwd_src_generic<float><<<blocks, 256, 0, st>>>(a));
            else
                SAR_LAUNCH("gat_bwd_src_generic", st, gat_bwd_src_generic<__nv_bfloat16><<<blocks, 256, 0, st>>>(a));
            SAR_TRY(sar_after_launch());
        }
        return SAR_OK;
    }
    const void *feat_g = feat_q, *gout_g = gout;
    if (r.ragged) {
        // What a step finds in the workspace is the records alone (the caller may have prepared one for each step), unless
        // it is told that an earlier step has made its copy of gout there: 8 steps on 170,000 nodes of 47 bf16, 2.5 million
        // edges, forward and backward 1297 us, 1335 us with a copy in every step.
        const long long n_gout = flags & SAR_SAME_WORKSPACE ? 0 : g->n_dst;
        SAR_TRY(pad_rows(H, F, r, t, g->n_src, feat_q, wsb + w.feat, n_gout, gout, wsb + w.gout, st));
        feat_g = wsb + w.feat;
        gout_g = wsb + w.gout;
    }
    RowArgs a{};
    a.row_bytes = r.row_bytes;
    a.el = el;
    a.er = er_q;
    a.m = m;
    a.d = d;
    a.rec = rec;
    a.slope = slope;
    a.flags = flags & ~SAR_SAME_WORKSPACE;
    a.H = H;
    a.F = F;
    a.vph = r.vph;
    a.ragged = r.ragged;
    a.hvec = heads_aligned(H, r.geo.HP, {el, er_q, m, d});
    Shape s;
    SAR_TRY(make_shape(H, F, t, !r.ragged, &s));
    if (g->n_dst > 0) {   // destination-major pass over the CSR
        a.n_rows = g->n_dst;
        a.indptr = g->indptr;
        a.indices = g->indices;
        a.last_col = (unsigned)(g->n_src > 0 ? g->n_src - 1 : 0);
        a.gather = feat_g;
        a.rowvec = gout_g;
        a.dscal = del;
        a.sp = split_args(g->split, reinterpret_cast<float *>(wsb + w.csr), H, r, t);
        a.lone = takes_short(r.geo, g->n_src, r.row_bytes, g->n_dst, g->nnz, true);
        if (lean_shape_applies(s, slope, g->split, g->n_src) && sar_aligned(er_q, 16)) {
            LeanArgs la{};
            la.n_rows = g->n_dst;
            la.indptr = g->indptr;
            la.indices = g->indices;
            la.gather = feat_q;
            la.rowvec = gout;
            la.el = el;
            la.er = er_q;
            la.m = m;
            la.d = d;
            la.rec_out = rec;
            la.rec_in = rec;
            la.first = (flags & SAR_FIRST) ? 1 : 0;
            la.del = del;
            la.slope = slope;
            la.sp = a.sp;
            la.sp.threshold = g->split->threshold;
            if (whole)
                SAR_TRY(t == SAR_F32 ? lean_bwd_dst_f32(s, la, g->nnz, st) : lean_bwd_dst_bf16(s, la, g->nnz, st));
            else
                SAR_TRY(t == SAR_F32 ? lean_bwd_dst_part_f32(s, la, g->nnz, st) : lean_bwd_dst_part_bf16(s, la, g->nnz, st));
        } else if (!a.lone && takes_span(s, r.geo, g->n_src, g->n_dst, g->nnz, true, !whole))
            SAR_TRY(span_dst(s, a, g->nnz, !whole, st));
        else if (whole)
            SAR_TRY(t == SAR_F32 ? rows_dst_f32(a, r.geo, g->nnz, st) : rows_dst_bf16(a, r.geo, g->nnz, st));
        else
            SAR_TRY(t == SAR_F32 ? rows_dst_part_f32(a, r.geo, g->nnz, st) : rows_dst_part_bf16(a, r.geo, g->nnz, st));
        if (a.sp.n_long > 0) SAR_TRY(rows_dst_merge(a, !whole, st));
    }
    if (g->n_src > 0) {   // source-major pass over the CSC
        a.n_rows = g->n_src;
        a.indptr = g->t_indptr;
        a.indices = g->t_indices;
        a.last_col = (unsigned)(g->n_dst - 1);
        a.gather = gout_g;
        a.rowvec = feat_g;
        a.out = dfeat_q;
        a.dscal = der_q;
        a.sp = split_args(g->t_split, reinterpret_cast<float *>(wsb + w.csc), H, r, t);
        a.lone = takes_short(r.geo, g->n_dst, r.row_bytes, g->n_src, g->nnz, true);
        if (lean_shape_applies(s, slope, g->t_split, g->n_dst)) {
            LeanSrcArgs la{};
            la.n_rows = g->n_src;
            la.indptr = g->t_indptr;
            la.indices = g->t_indices;
            la.gather = gout;
            la.rowvec = feat_q;
            la.er = er_q;
            la.rec_in = rec;
            la.out = dfeat_q;
            la.der = der_q;
            la.slope = slope;
            la.sp = a.sp;
            la.sp.threshold = g->t_split->threshold;
            SAR_TRY(t == SAR_F32 ? lean_bwd_src_f32(s, la, g->nnz, st) : lean_bwd_src_bf16(s, la, g->nnz, st));
        } else if (!a.lone && takes_span(s, r.geo, g->n_dst, g->n_src, g->nnz, true, !whole))
            SAR_TRY(span_src(s, a, g->nnz, st));
        else
            SAR_TRY(t == SAR_F32 ? rows_src_f32(a, r.geo, g->nnz, st) : rows_src_bf16(a, r.geo, g->nnz, st));
        if (a.sp.n_long > 0) SAR_TRY(rows_src_merge(a, t, st));
    }
    return SAR_OK;
}

sar_status sar_gat_bwd_fused(const sar_part *g, int32_t k, const int64_t *bounds, const void *feat, const float *el,
                             const float *er, const float *m, const float *d, const void *gout, int32_t H, int32_t F,
                             sar_dtype t, float slope, void *dfeat, float *del, float *der, void *workspace,
                             size_t workspace_bytes, void *stream) {
    SAR_TRY(check_fused(g, k, bounds));
    return sar_gat_bwd(g, feat, el, er, m, d, gout, H, F, t, slope, SAR_FIRST | SAR_LAST, dfeat, del, der, workspace,
                       workspace_bytes, stream);
}

// ---------------------------------------------------------------------------------------------
// The sum on rows of whole vectors: gather and, unless r.ragged, out; part = room for the segments of the long rows
static sar_status sum_rows(const sar_part *g, const RowShape &r, int32_t F, sar_dtype t, uint32_t flags, const void *gather, const int64_t *deg_total,
                           const float *src_scale, const float *dst_scale, const SumMix &mix, void *out, float *part, cudaStream_t st) {
    RowArgs a{};
    a.n_rows = g->n_dst;
    a.indptr = g->indptr;
    a.indices = g->indices;
    a.last_col = (unsigned)(g->n_src > 0 ? g->n_src - 1 : 0);
    a.gather = gather;
    a.row_bytes = r.row_bytes;
    a.out = out;
    a.deg = deg_total;
    a.src_scale = src_scale;
    a.dst_scale = dst_scale;
    a.mix = mix;
    a.flags = flags;
    a.H = 1;
    a.F = F;
    a.vph = r.vph;
    a.ragged = r.ragged;
    a.sp = split_args(g->split, part, 1, r, t);
    const bool weighted = src_scale != nullptr;
    Shape s;
    SAR_TRY(make_shape(1, F, t, !r.ragged, &s));
    a.lone = sum_takes_short(r.geo, g->n_src, r.row_bytes, g->n_dst, g->nnz);
    if (!a.lone && sum_takes_span(s, a, t, g->n_src, g->nnz, weighted))
        SAR_TRY(span_sum(s, a, g->nnz, weighted, st));
    else
        SAR_TRY(t == SAR_F32 ? rows_sum_f32(a, r.geo, g->nnz, weighted, st) : rows_sum_bf16(a, r.geo, g->nnz, weighted, st));
    return a.sp.n_long > 0 ? rows_sum_merge(a, t, st) : SAR_OK;
}

static sar_status spmm_impl(const sar_part *g, const void *feat_q, int32_t F, sar_dtype t, uint32_t flags,
                            const int64_t *deg_total, const float *src_scale, const float *dst_scale, void *out,
                            void *workspace, size_t workspace_bytes, void *stream) {
    SAR_TRY(check_part(g, false));
    if (flags & ~(SAR_FIRST | SAR_LAST | SAR_MEAN)) return SAR_ERR_INVALID_ARG;
    if (!out || (g->n_src > 0 && !feat_q)) return SAR_ERR_INVALID_ARG;
    if ((flags & SAR_MEAN) && (flags & SAR_LAST) && !deg_total) return SAR_ERR_INVALID_ARG;
    SAR_TRY(check_elem_align({feat_q, out}, sar_elem_size(t)));
    SAR_TRY(check_elem_align({deg_total}, 8));
    SAR_TRY(check_elem_align({src_scale, dst_scale}, 4));
    SAR_TRY(check_shape(1, F, t));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (g->n_dst == 0) return SAR_OK;
    const RowShape r = sum_shape(F, t);
    const size_t parts = part_bytes(g->split, 1, r, t);
    const bool have_ws = workspace && sar_aligned(workspace, 16);
    const bool rows = r.ragged ? have_ws && workspace_bytes >= parts + pad_bytes(g->n_src, r) : all16({feat_q, out});
    if (!rows) {
        GenericArgs a{};
        a.n_dst = g->n_dst;
        a.indptr = g->indptr;
        a.indices = g->indices;
        a.feat = feat_q;
        a.out = out;
        a.deg_total = deg_total;
        a.src_scale = src_scale;
        a.dst_scale = dst_scale;
        a.H = 1;
        a.F = F;
        a.flags = flags;
        const unsigned blocks = (unsigned)((g->n_dst * F + 255) / 256);
        if (t == SAR_F32)
            SAR_LAUNCH("spmm_generic", st, spmm_generic<float><<<blocks, 256, 0, st>>>(a));
        else
            SAR_LAUNCH("spmm_generic", st, spmm_generic<__nv_bfloat16><<<blocks, 256, 0, st>>>(a));
        return sar_after_launch();
    }
    const bool use_split = g->split && g->split->n_long > 0;
    if (use_split && (!have_ws || workspace_bytes < parts)) return SAR_ERR_WORKSPACE;
    if (r.ragged) {
        SAR_TRY(pad_rows(1, F, r, t, g->n_src, feat_q, static_cast<char *>(workspace) + parts, 0, nullptr, nullptr, st));
        feat_q = static_cast<char *>(workspace) + parts;
    }
    return sum_rows(g, r, F, t, flags, feat_q, deg_total, src_scale, dst_scale, SumMix{}, out, static_cast<float *>(workspace), st);
}

sar_status sar_spmm_agg(const sar_part *g, const void *feat_q, int32_t F, sar_dtype t, uint32_t flags,
                        const int64_t *deg_total, void *out, void *workspace, size_t workspace_bytes,
                        void *stream) {
    return spmm_impl(g, feat_q, F, t, flags, deg_total, nullptr, nullptr, out, workspace, workspace_bytes, stream);
}

sar_status sar_spmm_agg_scaled(const sar_part *g, const void *feat_q, int32_t F, sar_dtype t, uint32_t flags,
                               const float *src_scale, const float *dst_scale, void *out, void *workspace,
                               size_t workspace_bytes, void *stream) {
    if (flags & SAR_MEAN) return SAR_ERR_INVALID_ARG;
    return spmm_impl(g, feat_q, F, t, flags, nullptr, src_scale, dst_scale, out, workspace, workspace_bytes, stream);
}

// Workspace of a propagation: [ segments of the long rows ][ the array a step reads while the next one is written ], and
// where rows are ragged or arrays misaligned [ the latter, in place of out ][ x0 with padded rows ].
static bool propagate_reads_x0(const RowShape &r, const void *x0) { return !r.ragged && all16({x0}); }
static bool propagate_writes_out(const RowShape &r, const void *out) { return !r.ragged && all16({out}); }
static int propagate_arrays(const RowShape &r, const void *x0, const void *out) {
    return 1 + (propagate_writes_out(r, out) ? 0 : 1) + (propagate_reads_x0(r, x0) ? 0 : 1);
}
static size_t propagate_parts(int32_t k, const sar_part *const *parts, const RowShape &r, sar_dtype t) {
    size_t b = 0;
    for (int32_t q = 0; q < k; ++q) {
        const size_t p = part_bytes(parts[q]->split, 1, r, t);
        b = p > b ? p : b;
    }
    return b;
}
static size_t propagate_bytes(int32_t k, const sar_part *const *parts, int32_t F, sar_dtype t, bool any, const void *x0, const void *out) {
    if (k < 1 || !parts || F < 1) return 0;
    for (int32_t q = 0; q < k; ++q)
        if (!parts[q]) return 0;
    const RowShape r = sum_shape(F, t);
    return propagate_parts(k, parts, r, t) + (any ? 3 : propagate_arrays(r, x0, out)) * sar_round_up((size_t)parts[0]->n_dst * r.row_bytes, 256) + 256;
}
size_t sar_propagate_workspace_bytes(int32_t k, const sar_part *const *parts, int32_t F, sar_dtype t) {
    return propagate_bytes(k, parts, F, t, true, nullptr, nullptr);
}
size_t sar_propagate_workspace_bytes_at(int32_t k, const sar_part *const *parts, const void *x0, int32_t F, sar_dtype t, const void *out) {
    return propagate_bytes(k, parts, F, t, false, x0, out);
}

sar_status sar_propagate(int32_t k, const sar_part *const *parts, const int64_t *bounds, const void *x0, int32_t F, sar_dtype t, float alpha,
                         int64_t iters, const float *src_scale, const float *dst_scale, void *out, void *workspace, size_t workspace_bytes,
                         void *stream) {
    if (k < 1 || !parts || !bounds || iters < 1) return SAR_ERR_INVALID_ARG;
    if (k > SAR_MAX_PARTS) return SAR_ERR_UNSUPPORTED;
    for (int32_t q = 0; q < k; ++q) {
        SAR_TRY(check_part(parts[q], false));
        if (parts[q]->n_dst != parts[0]->n_dst || bounds[q] < 0 || bounds[q + 1] - bounds[q] != parts[q]->n_src) return SAR_ERR_INVALID_ARG;
    }
    const int64_t n = parts[0]->n_dst;
    if (bounds[0] != 0 || bounds[k] != n || (n > 0 && (!x0 || !out)) || x0 == out) return SAR_ERR_INVALID_ARG;
    SAR_TRY(check_elem_align({x0, out}, sar_elem_size(t)));
    SAR_TRY(check_elem_align({src_scale, dst_scale}, 4));
    SAR_TRY(check_shape(1, F, t));
    if (n == 0) return SAR_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const RowShape ragged = sum_shape(F, t);
    const int32_t Fp = (int32_t)(ragged.row_bytes / sar_elem_size(t));
    const RowShape r = sum_shape(Fp, t);   // the same rows, every vector of them whole
    const size_t array = sar_round_up((size_t)n * r.row_bytes, 256), seg = propagate_parts(k, parts, r, t);
    const int arrays = propagate_arrays(ragged, x0, out);
    if (!workspace || !sar_aligned(workspace, 256) || workspace_bytes < seg + arrays * array) return SAR_ERR_WORKSPACE;
    const bool in_place = propagate_reads_x0(ragged, x0), out_direct = propagate_writes_out(ragged, out);
    char *ws = static_cast<char *>(workspace);
    void *y[2] = {out_direct ? out : ws + seg + array, ws + seg};         // written in turn; the last step writes y[0]
    char *padded = in_place ? nullptr : ws + seg + (arrays - 1) * array;
    const void *x0p = in_place ? x0 : padded;
    const void *cur = x0p;
    if (!in_place || src_scale) {
        void *scaled = src_scale ? y[iters & 1] : nullptr;
        if (src_scale) cur = scaled;
        SAR_TRY(propagate_start(n, F, r, t, x0, src_scale, padded, scaled, st));
    }
    for (int64_t i = 0; i < iters; ++i) {
        const bool end = i + 1 == iters;
        void *nxt = y[(iters - 1 - i) & 1];
        const SumMix mix{x0p, 1.f - alpha, alpha, end ? nullptr : src_scale};
        for (int32_t q = 0; q < k; ++q)
            SAR_TRY(sum_rows(parts[q], r, Fp, t, (q == 0 ? SAR_FIRST : 0u) | (q + 1 == k ? SAR_LAST : 0u),
                             static_cast<const char *>(cur) + (size_t)bounds[q] * r.row_bytes, nullptr, nullptr, dst_scale, mix, nxt,
                             reinterpret_cast<float *>(ws), st));
        cur = nxt;
    }
    return out_direct ? SAR_OK : strip_rows(n, F, r, t, cur, out, st);
}

}  // extern "C"
