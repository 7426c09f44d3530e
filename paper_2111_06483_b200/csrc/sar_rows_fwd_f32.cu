// Row kernels of one pass (fwd), f32 storage (see sar_rows_kernel.cuh).
#include "sar_rows_launch.cuh"

namespace sar {
sar_status rows_fwd_f32(const RowArgs &a, RowGeo g, long long nnz, cudaStream_t st) {
    return dispatch_rows<float, kRowFwd>(a, g, nnz, "gat_fwd", st);
}
}  // namespace sar
