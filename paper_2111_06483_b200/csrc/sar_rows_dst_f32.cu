// Row kernels of one pass (dst), f32 storage (see sar_rows_kernel.cuh).
#include "sar_rows_launch.cuh"

namespace sar {
sar_status rows_dst_f32(const RowArgs &a, RowGeo g, long long nnz, cudaStream_t st) {
    return dispatch_rows<float, kRowDst>(a, g, nnz, "gat_bwd_dst", st);
}
}  // namespace sar
