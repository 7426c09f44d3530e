// Row kernels of one pass (dst part), bf16 storage (see sar_rows_kernel.cuh).
#include "sar_rows_launch.cuh"

namespace sar {
sar_status rows_dst_part_bf16(const RowArgs &a, RowGeo g, long long nnz, cudaStream_t st) {
    return dispatch_rows<__nv_bfloat16, kRowDstPart>(a, g, nnz, "gat_bwd_dst", st);
}
}  // namespace sar
