// Host-side interface of the row kernels (internal): arguments, geometry and the launchers, which are compiled in
// translation units of their own (sar_rows_*.cu), one per pass and storage type.
#pragma once

#include "sar_rowkernels.cuh"

namespace sar {

enum RowMode {
    kRowFwd = 0,       // forward, the call holds the whole graph
    kRowFwdPart = 1,   // forward partition step: folds into the running state (acc, m, d)
    kRowDst = 2,       // destination-major backward, whole graph: D rebuilt from the edges, record written
    kRowDstPart = 3,   // destination-major backward partition step: D read from the record, del accumulated
    kRowSrc = 4,       // source-major backward (whole graph or partition step: a source lies in one partition)
    kRowSum = 5,       // sum aggregation
    kRowSumW = 6       // sum aggregation with a factor per source
};

struct RowArgs {
    long long n_rows, nnz;
    unsigned last_col;       // rows of gather - 1
    const int64_t *indptr;
    const int32_t *indices;
    const void *gather;      // rows fetched per edge, row_bytes apart, 16-byte aligned heads
    const void *rowvec;      // backward: row-stationary vector (gout / feat), same layout
    unsigned row_bytes;
    const float *el, *er;    // forward and destination-major: el[row], er[col]; source-major: er[row]
    const float *m, *d;      // destination-major: final statistics
    float4 *rec;             // {el, m, 1/d, D}: written (kRowDst), read at the row (kRowDstPart) or at the column (kRowSrc)
    float *acc;              // forward partition step: running numerator [n_rows, H*F]
    float *m_io, *d_io;      // forward: statistics out (in and out in a partition step)
    void *out;               // out / dfeat / sum, [n_rows, H*F] in the storage type
    float *dscal;            // del / der
    const int64_t *deg;      // sum: total in-degree for the mean
    const float *src_scale, *dst_scale;
    SumMix mix;              // sum
    float slope;
    unsigned flags;
    int H, F;                // heads and features per head as stored in out (F may be ragged)
    int vph;                 // 16-byte vectors per head in gather and rowvec
    int ragged;              // out / acc rows are not made of aligned 16-byte vectors: element stores
    int hvec;                // the per-head scalars of a row can be loaded as float4 / float2
    int R;                   // rows per warp (<= 32); sar_short_kernel.cuh: the most edges of a row that is one warp's
    int lone;                // a row per group of lanes (sar_short_kernel.cuh)
    int wide;                // ... and a segment per block
    SplitArgs sp;
};

// Geometry of a launch: NV lanes (times vectors) cover HP heads of vphp = NV/HP vectors each, both powers of two;
// `tiles` launches along the grid's second dimension cover the heads (for a sum: the columns).
struct RowGeo {
    int NV, HP, tiles;
};

// The most edges per row with which the kernel for short rows (sar_short_kernel.cuh) takes a call, by its tile and the bytes of the gathered
// array; 0: it doesn't, and the kernel of that tile isn't compiled.  What the lines were drawn from is with takes_short in sar_gat.cu.
constexpr double short_edges(int NV, int HP, bool backward, unsigned long long bytes) {
    if (NV > 32) return 0;
    if (HP == 8) return backward ? 100 : NV <= 16 ? 40 : bytes <= (32ull << 20) ? 14 : 0;
    if (NV == 32) return HP == 4 && backward && bytes <= (8ull << 20) ? 10 : 0;
    if (NV == 16) return HP == 4 ? (backward ? 16 : 10) : HP == 2 && backward ? 6 : 0;
    if (HP == 4) return backward ? 100 : 24;
    return NV == 4 ? (backward ? 28 : 20) : backward ? 16 : 14;
}
constexpr unsigned long long kSpanSumBytes = 12ull << 20;   // sums over larger arrays are the span kernels' where the short-row kernel does not take them
constexpr double sum_short_edges(int NV, unsigned long long bytes) {
    return NV == 4 ? 20 : NV == 8 ? (bytes <= kSpanSumBytes ? 14 : bytes <= (64ull << 20) ? 8 : 3) : 0;
}

// One launch over the segments of the long rows and the other rows.
#define SAR_ROWS_DECL(PASS) \
    sar_status rows_##PASS##_f32(const RowArgs &a, RowGeo g, long long nnz, cudaStream_t st); \
    sar_status rows_##PASS##_bf16(const RowArgs &a, RowGeo g, long long nnz, cudaStream_t st);
SAR_ROWS_DECL(fwd)
SAR_ROWS_DECL(fwd_part)
SAR_ROWS_DECL(dst)
SAR_ROWS_DECL(dst_part)
SAR_ROWS_DECL(src)
#undef SAR_ROWS_DECL
sar_status rows_sum_f32(const RowArgs &a, RowGeo g, long long nnz, bool weighted, cudaStream_t st);
sar_status rows_sum_bf16(const RowArgs &a, RowGeo g, long long nnz, bool weighted, cudaStream_t st);

// The long rows, from their segments' records.
sar_status rows_fwd_merge(const RowArgs &a, sar_dtype t, cudaStream_t st);
// The end of Algorithm 1 on its own: out = numerator / d for every row.
sar_status rows_fwd_finalize(const RowArgs &a, sar_dtype t, cudaStream_t st);
sar_status rows_dst_merge(const RowArgs &a, bool part, cudaStream_t st);
sar_status rows_src_merge(const RowArgs &a, sar_dtype t, cudaStream_t st);
sar_status rows_sum_merge(const RowArgs &a, sar_dtype t, cudaStream_t st);

}  // namespace sar
