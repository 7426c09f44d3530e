// Host-side interface of the span kernels (internal): sar_span.cu.
#pragma once

#include "sar_rows.cuh"

namespace sar {

// One launch over the segments of the long rows and the spans of the other rows.
sar_status span_fwd(const Shape &s, const RowArgs &r, long long nnz, cudaStream_t st);
sar_status span_dst(const Shape &s, const RowArgs &r, long long nnz, bool part, cudaStream_t st);
sar_status span_src(const Shape &s, const RowArgs &r, long long nnz, cudaStream_t st);
sar_status span_sum(const Shape &s, const RowArgs &r, long long nnz, bool weighted, cudaStream_t st);

}  // namespace sar
