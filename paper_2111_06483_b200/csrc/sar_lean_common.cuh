// Lean span kernels of libsar (internal), shared part: the whole-graph forward pass (sar_lean_fwd_kernels.cuh), the
// destination-major (sar_lean_dst_kernels.cuh) and the source-major (sar_lean_src_kernels.cuh) whole-graph backward
// pass for the common shapes (heads in groups of four, rows of exactly G*V 16-byte vectors), written for the fewest
// issued instructions per edge.
//
// The plan: a warp owns a span of consecutive rows, stages a chunk of whole
// rows in shared memory slot-major and streams the gathered rows through a cp.async ring:
//   * The ring works in STAGES of 2 or 4 KB (SPS slots): one commit group and one wait per stage, the slots of a
//     stage walked with compile-time offsets (fully unrolled), the stage refilled as a whole.  The staged column ids
//     are pre-scaled row offsets in 16-byte units, stored per stage with the slot index fastest, so that one
//     16-byte shared load brings the offsets of four consecutive slots; the weights likewise.
//   * The inputs of a stage's scores (16 bytes of er per position and head group, or the 64-byte record of the
//     destination in the source-major pass) are copied into a small ring with the stage's rows, and the weights of a
//     stage are computed just before the stage is consumed, one (position, head) pair per lane: no score phase over
//     the whole chunk, no weight array of the chunk's size, and the gather of the score inputs hides behind the rows.
//   * A row's padding position repeats the row's last column with weight zero, and a chunk's last stage is filled
//     up with repeats: every copy is a real copy of a real row, no predicates, no zero fill.
//   * Everything the control flow depends on (slot counts, row-end masks) is produced by warp votes and reductions,
//     so that the branches around the row epilogues are uniform branches.
//   * Exponentials are one FFMA + EX2; the forward row max uses max_j LeakyReLU(el + er_j) = LeakyReLU(el + max_j er_j)
//     (slope >= 0) and runs online, stage by stage.
//   * Dot products of the backward epilogues are taken on the un-folded accumulators and reduced with three shuffles
//     per quantity; per-(row, head) scalars leave through shared memory, coalesced, once per chunk.
// Preconditions (checked by the host, which otherwise launches the row or span kernels): slope >= 0, every row that is no
// long one at most CAP edges (a long-row plan with threshold <= CAP), segments of at most CAP edges, fewer
// than 2^32 16-byte vectors in the gathered array.
#pragma once

#include "sar_device.cuh"
#include "sar_lean.cuh"
#include "sar_dispatch.cuh"

namespace sar {

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void sts_f32(unsigned addr, float v) {
    asm volatile("st.shared.f32 [%0], %1;\n" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void sts_u32(unsigned addr, unsigned v) {
    asm volatile("st.shared.u32 [%0], %1;\n" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned lds_u32(unsigned addr) {
    unsigned v;
    asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ unsigned lds_u8(unsigned addr) {
    unsigned v;
    asm volatile("ld.shared.u8 %0, [%1];\n" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_u8(unsigned addr, unsigned v) {
    asm volatile("st.shared.u8 [%0], %1;\n" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ float4 lds_f4(unsigned addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
    return v;
}
// shared-memory max without a return value: nobody waits for it
__device__ __forceinline__ void red_max_u32(unsigned addr, unsigned v) {
    asm volatile("red.shared.max.u32 [%0], %1;\n" ::"r"(addr), "r"(v) : "memory");
}
// plain 16-byte asynchronous copy (every copy of the lean kernels is a whole, valid vector)
__device__ __forceinline__ void cp_async16_full(unsigned smem_addr, const void *gsrc) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr), "l"(gsrc) : "memory");
}

constexpr float kLog2e = 1.4426950408889634f;

// ---- launch parameters shared by the three passes --------------------------------------------------------------
// One configuration: chunks of kLeanCap edges, ring of two stages of 2 KB (4 KB for rows of 512 bytes and more), measured
// best on the large workload among stages of 2 / 4 KB, two to four stages, chunks of 128 / 192 / 256 edges.
constexpr int kLeanMinBlocks = 8;
// The rows of the two backward passes are compiled for 24 resident blocks per SM (64-80 registers instead of 88; no
// spills but for bf16 rows of 1 KB source-major, 40 bytes): step of the large workload 153.1 -> 147.2 ms.  The same bound
// on the forward rows and on launches over segments alone changes nothing (147.3 ms).
constexpr int kLeanMinBlocksBwdRows = 24;

// Resident blocks per SM the rows of a partition step are compiled for.
constexpr int kLeanMinBlocksPart = 16;

constexpr int kMaxSpanRows = 16;   // rows a span holds at most

// Rows per span: about `cap` edges (the long rows counted in the average are skipped), but no more than leaves every SM
// kLeanFill spans: a graph with fewer is done when its longest span is.
constexpr int kLeanSMs = 148, kLeanFill = 24;
static inline int lean_rows_per_span(long long n_rows, long long nnz, int cap, int max_rows = kMaxSpanRows) {
    const double avg = n_rows > 0 ? (double)nnz / (double)n_rows : 0.0;
    long long R = avg > 0.5 ? (long long)(1.0 * cap / avg + 0.5) : max_rows;
    const long long fill = n_rows / (kLeanSMs * kLeanFill);
    if (R > fill) R = fill;
    if (R < 1) R = 1;
    if (R > max_rows) R = max_rows;
    return (int)R;
}

// What the blocks of a launch work on: a segment of a long row each, a span of the other rows each, or both, the segments
// first.  A segment is the longest chain of work in a pass: where there are few, the spans fill what they leave free (a
// partition step's pass over 100,000 rows and 250,000 edges: 60 us, and 80 with the segments in a launch of their own).
// Where the segments alone fill every SM several times over, one launch after the other costs their tail and no more, and
// the segments run with the shared memory that they need themselves, more of them at a time.  Forward + backward, one launch
// against two: 4,666 segments (300,000 nodes, 8 heads of 32, bf16) 0.92 against 1.00 ms; 12,000 (500,000 nodes, 4 heads of
// 32) 1.09 against 1.11; 23,000 (a million nodes) 1.984 against 1.976; 30,000 (2 million, 4 heads of 16, float32) 2.57
// against 2.60; 47,000 (200,000 nodes, 20 million edges, 8 heads of 32) 3.82 against 3.78; 130,000 (a million nodes, 4 heads
// of 64) 11.5 against 11.0; 575,000 (200 edges per node, 8 heads of 32) 42.7 against 41.6 ms.
enum { kLeanBoth = 0, kLeanSegments = 1, kLeanRows = 2 };
constexpr long long kLeanSegmentsAlone = 148 * 256;
template <typename LR, typename LS, typename K, typename A>
static sar_status launch_lean(const char *name, const char *seg_name, K both, K segments, K rows, const A &a, cudaStream_t st) {
    const long long spans = (a.n_rows + a.R - 1) / a.R, n_seg = a.sp.n_seg;
    auto go = [&](const char *what, K kern, size_t smem, long long blocks) -> sar_status {
        if (blocks <= 0) return SAR_OK;
        SAR_TRY(ensure_smem(kern, smem));
        SAR_LAUNCH(what, st, launch(kern, (unsigned)blocks, 32, smem, st, a));
        return sar_after_launch();
    };
    if (n_seg > 0 && n_seg < kLeanSegmentsAlone) return go(name, both, LR::total > LS::total ? LR::total : LS::total, n_seg + spans);
    SAR_TRY(go(seg_name, segments, LS::total, n_seg));
    return go(name, rows, LR::total, spans);
}

}  // namespace sar
