// Row kernels of the sum aggregation, bf16 storage (see sar_rows_kernel.cuh).
#include "sar_rows_launch.cuh"

namespace sar {
sar_status rows_sum_bf16(const RowArgs &a, RowGeo g, long long nnz, bool weighted, cudaStream_t st) {
    return weighted ? dispatch_rows<__nv_bfloat16, kRowSumW>(a, g, nnz, "spmm", st) : dispatch_rows<__nv_bfloat16, kRowSum>(a, g, nnz, "spmm", st);
}
}  // namespace sar
