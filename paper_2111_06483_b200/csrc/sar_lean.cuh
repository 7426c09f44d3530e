// Host-side interface of the lean span kernels (internal): arguments, applicability test and the launchers,
// which are compiled in translation units of their own (sar_lean_*.cu), one per pass and storage type.
// They cover the forward pass and both backward passes, of a call that holds the whole graph and as partition steps.
#pragma once

#include "sar_rowkernels.cuh"

namespace sar {

struct LeanArgs {
    long long n_rows;
    const int64_t *indptr;
    const int32_t *indices;
    const void *gather;      // rows fetched per edge: feat
    const void *rowvec;      // row-stationary vector of the backward pass: gout
    const float *el, *er;    // el[row], er[col]
    const float *m, *d;      // bwd-dst: final statistics of the row
    float4 *rec_out;         // bwd-dst: record {el, m, 1/d, D} written per (row, head)
    const float4 *rec_in;    // bwd-dst, partition step: the record written beforehand (D is read from it)
    int first;               // partition step: the state (forward) / del (bwd-dst) starts here, nothing is read
    float *m_out, *d_out;    // forward (a partition step reads the state there and writes it back)
    float *acc_state;        // forward, partition step: running numerator [n_rows, H*F], float32
    void *out;               // forward: out
    float *del;              // bwd-dst
    float slope;
    SplitArgs sp;
    int R;                   // rows per span (<= kMaxSpanRows)
    int relu;                // forward: out = max(out, 0)
};

struct LeanSrcArgs {
    long long n_rows;        // sources
    const int64_t *indptr;   // CSC
    const int32_t *indices;  // destinations
    const void *gather;      // gout
    const void *rowvec;      // feat
    const float *er;         // [n_rows,H]
    const float4 *rec_in;    // [n_dst,H] {el, m, 1/d, D}
    void *out;               // dfeat
    float *der;
    float slope;
    SplitArgs sp;
    int R;
};

constexpr int kLeanCap = 256;   // edges a chunk stages; rows and segments must not exceed it
// Where the lean kernels cover a shape they take every pass of it; the row kernels (sar_rows_kernel.cuh) take the others.
// Both cover these shapes; measured on them, lean against row kernels, bf16, 4 heads of 32, forward / destination-major /
// source-major: large workload 15.2 / 15.2 / 16.8 against 20.2 / 20.1 / 32.7 ms, 100,000 nodes and 2 million edges
// 117 / 116 / 120 against 115 / 111 / 181 us; a partition step of the large workload 3.0 / 2.2 / 1.0 against
// 3.9 / 2.8 / 2.1 ms.  (The short-row kernel, sar_short_kernel.cuh, has not been compared with them on these shapes.)

// Do the lean kernels cover this shape?  Slope >= 0, heads in groups of four, rows of
// exactly G*V vectors with V <= 2, the vectors of a head a power of two within one lane group, and a long-row
// plan whose threshold fits a chunk (so that no span's row and no segment exceeds it), and a gathered
// array of n_gathered rows whose 16-byte vectors can be counted in 32 bits (the staged row offsets are 32-bit).
static inline bool lean_shape_applies(const Shape &s, float slope, const sar_split *sp, long long n_gathered) {
    if (!s.fast) return false;
    if (!(slope >= 0.f) || !sp || sp->threshold < 1 || sp->threshold > kLeanCap) return false;
    const int H = s.geom.H, nv = s.geom.n_vec;
    if (H % 4 != 0 || nv != s.G * s.V || s.V > 2 || nv % H != 0) return false;
    const int vph = nv / H;
    if (vph > s.G || (vph & (vph - 1)) != 0) return false;
    if ((unsigned long long)nv * (unsigned long long)(n_gathered > 0 ? n_gathered : 0) > 0xffffffffull) return false;
    return (s.G == 16 && s.V == 1 && H == 4) || (s.G == 32 && s.V == 1 && (H == 4 || H == 8)) ||
           (s.G == 32 && s.V == 2 && H == 4);
}
// Segments of the long rows and spans of the other rows, of one pass.
sar_status lean_fwd_f32(const Shape &s, const LeanArgs &a, long long nnz, cudaStream_t st);
sar_status lean_fwd_bf16(const Shape &s, const LeanArgs &a, long long nnz, cudaStream_t st);
sar_status lean_fwd_part_f32(const Shape &s, const LeanArgs &a, long long nnz, cudaStream_t st);
sar_status lean_fwd_part_bf16(const Shape &s, const LeanArgs &a, long long nnz, cudaStream_t st);
sar_status lean_bwd_dst_f32(const Shape &s, const LeanArgs &a, long long nnz, cudaStream_t st);
sar_status lean_bwd_dst_bf16(const Shape &s, const LeanArgs &a, long long nnz, cudaStream_t st);
sar_status lean_bwd_dst_part_f32(const Shape &s, const LeanArgs &a, long long nnz, cudaStream_t st);
sar_status lean_bwd_dst_part_bf16(const Shape &s, const LeanArgs &a, long long nnz, cudaStream_t st);
sar_status lean_bwd_src_f32(const Shape &s, const LeanSrcArgs &a, long long nnz, cudaStream_t st);
sar_status lean_bwd_src_bf16(const Shape &s, const LeanSrcArgs &a, long long nnz, cudaStream_t st);

}  // namespace sar
