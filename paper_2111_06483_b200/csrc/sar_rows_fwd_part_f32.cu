// Row kernels of one pass (fwd part), f32 storage (see sar_rows_kernel.cuh).
#include "sar_rows_launch.cuh"

namespace sar {
sar_status rows_fwd_part_f32(const RowArgs &a, RowGeo g, long long nnz, cudaStream_t st) {
    return dispatch_rows<float, kRowFwdPart>(a, g, nnz, "gat_fwd", st);
}
}  // namespace sar
