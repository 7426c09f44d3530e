// Launches that overlap the end of the launch before them (internal).
//
// A pass over a small graph is a chain of kernels of 3 to 5 us, and between two of them lies 1.5 us in which the second is
// only being set up.  So every kernel of the aggregation and of the streaming steps around it is launched with programmatic
// stream serialisation and begins with after_predecessor(): its blocks may be placed as soon as all blocks of the launch
// before run, wait there until that launch has ended and its writes are visible, and then let the next launch be placed in
// turn.  Every block waits, and nothing is read or written before: that is what makes the writes of a launch visible to
// the next one and, since that one ends only after its own wait, to all that follow.  So the order of the stream holds
// for every pair of launches, whoever issued them; a launch that follows another kind of work, or carries the attribute
// without need, simply does not overlap.  2,000 nodes, 22,000 edges, forward and backward (three launches): 18.6 -> 14.2 us.
#pragma once

#include "sar_common.cuh"

namespace sar {

__device__ __forceinline__ void after_predecessor() {
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

// One grid that strides over its array: its blocks have to be spread evenly, and placed into what the launch before leaves
// free they are not (layer of a million nodes, 256 MB arrays: 3.02 ms in stream order, 3.14 ms overlapped), so these
// overlap on arrays of a few million elements only, where the gap between the launches counts (16,485 nodes of 128: 157
// against 141 us a step).
constexpr long long kOverlapElems = 8LL << 20;

template <typename... K, typename... A>
static inline void launch_if(bool overlap, void (*kernel)(K...), dim3 grid, dim3 threads, size_t smem, cudaStream_t st, const A &...args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = threads;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = overlap ? 1 : 0;
    (void)cudaLaunchKernelEx(&c, kernel, static_cast<K>(args)...);   // reported by sar_after_launch
}

template <typename... K, typename... A>
static inline void launch(void (*kernel)(K...), dim3 grid, dim3 threads, size_t smem, cudaStream_t st, const A &...args) {
    launch_if(true, kernel, grid, threads, smem, st, args...);
}

}  // namespace sar
