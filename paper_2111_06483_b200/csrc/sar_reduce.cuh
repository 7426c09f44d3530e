// Per-block partial sums -> totals (internal), the second launch of the column reductions of sar_norm.cu and sar_glue.cu.
#pragma once

#include "sar_common.cuh"
#include "sar_launch.cuh"

namespace sar {

// partial [blocks][cols] -> out0 [split] and out1 [cols - split] (either may be null), times scale, in float64.  A block
// owns 32 columns and 16 threads share each of them: a thread per column alone walked the blocks' records one after the
// other, 53 us for 1184 records of 256 columns (now 4 us).  The order of the additions is fixed.
constexpr int kReduceSlices = 16;
static __global__ void __launch_bounds__(32 * kReduceSlices) reduce_partials_kernel(int blocks, int cols, int split, const float *__restrict__ partial,
                                                                                    double scale, float *__restrict__ out0, float *__restrict__ out1) {
    after_predecessor();
    __shared__ double red[kReduceSlices][32];
    const int x = blockIdx.x * 32 + threadIdx.x;
    double acc = 0.0;
    if (x < cols) {
#pragma unroll 4
        for (int b = threadIdx.y; b < blocks; b += kReduceSlices) acc += (double)partial[(size_t)b * cols + x];
    }
    red[threadIdx.y][threadIdx.x] = acc;
    __syncthreads();
    if (threadIdx.y != 0 || x >= cols) return;
#pragma unroll
    for (int k = 1; k < kReduceSlices; ++k) acc += red[k][threadIdx.x];
    acc *= scale;
    if (x < split) {
        if (out0) out0[x] = (float)acc;
    } else if (out1) {
        out1[x - split] = (float)acc;
    }
}

static inline sar_status reduce_partials(const char *name, int blocks, int cols, int split, const float *partial, double scale, float *out0, float *out1,
                                         cudaStream_t st) {
    SAR_LAUNCH(name, st, launch(reduce_partials_kernel, (cols + 31) / 32, dim3(32, kReduceSlices), 0, st, blocks, cols, split, partial, scale, out0, out1));
    return sar_after_launch();
}

}  // namespace sar
