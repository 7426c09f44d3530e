// Row kernels of the sum aggregation, f32 storage (see sar_rows_kernel.cuh).
#include "sar_rows_launch.cuh"

namespace sar {
sar_status rows_sum_f32(const RowArgs &a, RowGeo g, long long nnz, bool weighted, cudaStream_t st) {
    return weighted ? dispatch_rows<float, kRowSumW>(a, g, nnz, "spmm", st) : dispatch_rows<float, kRowSum>(a, g, nnz, "spmm", st);
}
}  // namespace sar
