// Stable counting passes over (key, value) pairs of 32-bit ids (internal): the sort behind graph preparation.
//
// One pass orders the pairs by up to 8 bits of the key; node ids need ceil(log2 n) bits, so a graph of up to 16 million
// nodes is sorted by one endpoint in three passes over 8-byte pairs.
//
//   counts   every block counts its tile's digits in shared memory -> counts[digit][block]
//   offsets  exclusive prefix sum over (digit, block)
//   move     a warp takes consecutive elements 32 at a time; eight ballots tell every lane which lanes have its digit, and
//            they take consecutive ranks from the warp's own counter of that digit, so equal digits keep their order.  The
//            warps' counts are summed up per digit, the tile is put in digit order in shared memory and written out from
//            there, so that a digit's elements leave as one run.
// No block waits for another one.
//
// What bounds a pass: 20 bytes of traffic an element would take 0.19 ms for 62 million pairs, the move takes 0.30 ms and
// the counts 0.05.  The move issues 94 instructions per 32 elements, most of them on the half-rate integer pipe (67 to 77 % busy);
// matching by shared-memory atomics or match_any instead of ballots, writing without the detour through shared memory,
// and 11-bit digits (two passes of 0.7 ms: 2048 counters a tile, runs of 4) all measured the same or slower, and so did
// 512 threads or 8 to 12 elements a thread.  Before, eight-bit passes over 8-byte keys of both endpoints took seven times
// 0.59 ms for each of the two orientations.
#pragma once

#include <cub/device/device_scan.cuh>

#include "sar_common.cuh"

namespace sar {

constexpr int kRadixMaxBits = 8, kRadixMaxBins = 1 << kRadixMaxBits;
constexpr int kRadixThreads = 256, kRadixWarps = kRadixThreads / 32, kRadixItems = 16;
constexpr int kRadixTile = kRadixThreads * kRadixItems;
constexpr long long kRadixSmallScan = 16 * 1024;   // counters up to which one block does the prefix sum

static inline long long radix_blocks(long long n) { return (n + kRadixTile - 1) / kRadixTile; }

__global__ void __launch_bounds__(kRadixThreads) radix_count_kernel(long long n, const unsigned *__restrict__ keys, int shift, int bits,
                                                                    unsigned *__restrict__ counts, unsigned blocks) {
    __shared__ unsigned bin[kRadixMaxBins];
    const unsigned mask = (1u << bits) - 1u;
    bin[threadIdx.x] = 0;
    const long long base = (long long)blockIdx.x * kRadixTile;
    const int left = (int)min((long long)kRadixTile, n - base) - (int)threadIdx.x;
    keys += base + threadIdx.x;
    unsigned key[kRadixItems];
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i) key[i] = i * kRadixThreads < left ? keys[i * kRadixThreads] : 0u;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i)
        if (i * kRadixThreads < left) atomicAdd(&bin[(key[i] >> shift) & mask], 1u);
    __syncthreads();
    if (threadIdx.x <= mask) counts[(size_t)threadIdx.x * blocks + blockIdx.x] = bin[threadIdx.x];
}
static_assert(kRadixThreads == kRadixMaxBins, "a thread per digit");

// exclusive prefix sum of `n` counters in place, one block
__global__ void __launch_bounds__(1024) radix_scan_kernel(int n, unsigned *__restrict__ counts) {
    __shared__ unsigned warp_sum[32], carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < n; base += 4096) {
        unsigned v[4], s = 0;
        const int at = base + threadIdx.x * 4;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = at + k < n ? counts[at + k] : 0u;
            s += v[k];
        }
        unsigned inc = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) warp_sum[warp] = inc;
        __syncthreads();
        if (warp == 0) {
            unsigned w = warp_sum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned t = __shfl_up_sync(0xffffffffu, w, o);
                if (lane >= o) w += t;
            }
            warp_sum[lane] = w;
        }
        __syncthreads();
        unsigned run = carry + (warp ? warp_sum[warp - 1] : 0u) + inc - s;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (at + k < n) counts[at + k] = run;
            run += v[k];
        }
        __syncthreads();
        if (threadIdx.x == 0) carry += warp_sum[31];
        __syncthreads();
    }
}

struct RadixShared {
    unsigned delta[kRadixMaxBins];   // where the block's elements of a digit go, less their place in the tile
    unsigned first[kRadixMaxBins];   // place in the tile of a digit's first element
    unsigned warp_sum[kRadixWarps];
    union {
        unsigned short count[kRadixWarps][kRadixMaxBins];
        struct {
            unsigned key[kRadixTile], val[kRadixTile];
        } tile;
    };
};

// FULL: the block's tile lies in the array as a whole
template <bool FULL>
__device__ __forceinline__ void radix_move(RadixShared &sm, long long n, const unsigned *__restrict__ keys, const unsigned *__restrict__ vals, int shift, int bits,
                                           const unsigned *__restrict__ offsets, unsigned blocks, unsigned *__restrict__ keys_out,
                                           unsigned *__restrict__ vals_out) {
    const unsigned mask = (1u << bits) - 1u;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x <= mask) sm.delta[threadIdx.x] = offsets[(size_t)threadIdx.x * blocks + blockIdx.x];
#pragma unroll
    for (int w = 0; w < kRadixWarps; ++w) sm.count[w][threadIdx.x] = 0;
    const long long tile0 = (long long)blockIdx.x * kRadixTile;
    const int size = (int)min((long long)kRadixTile, n - tile0);
    const int at0 = warp * (32 * kRadixItems) + lane, left = size - at0;   // element i of this thread exists if i * 32 < left
    keys += tile0 + at0;
    vals += tile0 + at0;
    unsigned key[kRadixItems], rank[kRadixItems / 2];   // two 16-bit ranks in a word
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i) key[i] = FULL || i * 32 < left ? keys[i * 32] : 0u;
    __syncthreads();
    unsigned short *mine = sm.count[warp];
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i) {
        const bool in = FULL || i * 32 < left;
        const unsigned d = (key[i] >> shift) & mask;
        unsigned same = FULL ? 0xffffffffu : __ballot_sync(0xffffffffu, in);
#pragma unroll
        for (int b = 0; b < kRadixMaxBits; ++b) {
            const bool set = (d >> b) & 1u;
            const unsigned m = __ballot_sync(0xffffffffu, set);
            same &= set ? m : ~m;
        }
        const unsigned before = mine[d], r = before + __popc(same & lt);
        rank[i / 2] = i % 2 ? rank[i / 2] | r << 16 : r;
        __syncwarp();
        if (in && (same & lt) == 0u) mine[d] = (unsigned short)(before + __popc(same));   // the group's first lane
        __syncwarp();
    }
    __syncthreads();
    {   // the warps' counts -> those of the warps before; the digits' totals -> places in the tile
        unsigned total = 0;
#pragma unroll
        for (int w = 0; w < kRadixWarps; ++w) {
            const unsigned c = sm.count[w][threadIdx.x];
            sm.count[w][threadIdx.x] = (unsigned short)total;
            total += c;
        }
        unsigned inc = total;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        if (lane == 31) sm.warp_sum[warp] = inc;
        __syncthreads();
        unsigned first = inc - total;
#pragma unroll
        for (int w = 0; w < kRadixWarps; ++w) first += w < warp ? sm.warp_sum[w] : 0u;
        sm.first[threadIdx.x] = first;
        if (threadIdx.x <= mask) sm.delta[threadIdx.x] -= first;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i) {
        const unsigned d = (key[i] >> shift) & mask, place = (unsigned)mine[d] + sm.first[d];
        rank[i / 2] += i % 2 ? place << 16 : place;   // a place in the tile fits 16 bits
    }
    __syncthreads();   // the counters give way to the tile
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i)
        if (FULL || i * 32 < left) sm.tile.key[i % 2 ? rank[i / 2] >> 16 : rank[i / 2] & 0xffffu] = key[i];
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i) key[i] = FULL || i * 32 < left ? vals[i * 32] : 0u;
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i)
        if (FULL || i * 32 < left) sm.tile.val[i % 2 ? rank[i / 2] >> 16 : rank[i / 2] & 0xffffu] = key[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kRadixItems; ++i) {
        const int p = i * kRadixThreads + threadIdx.x;
        if (FULL || p < size) {
            const unsigned k = sm.tile.key[p], to = sm.delta[(k >> shift) & mask] + p;
            keys_out[to] = k;
            vals_out[to] = sm.tile.val[p];
        }
    }
}

__global__ void __launch_bounds__(kRadixThreads, 5)
    radix_move_kernel(long long n, const unsigned *__restrict__ keys, const unsigned *__restrict__ vals, int shift, int bits,
                      const unsigned *__restrict__ offsets, unsigned blocks, unsigned *__restrict__ keys_out, unsigned *__restrict__ vals_out) {
    __shared__ RadixShared sm;
    if ((long long)(blockIdx.x + 1) * kRadixTile <= n)
        radix_move<true>(sm, n, keys, vals, shift, bits, offsets, blocks, keys_out, vals_out);
    else
        radix_move<false>(sm, n, keys, vals, shift, bits, offsets, blocks, keys_out, vals_out);
}

// ---- host ------------------------------------------------------------------------------------------------------------------
static inline int radix_passes(int bits) { return (bits + kRadixMaxBits - 1) / kRadixMaxBits; }
static inline long long radix_counters(long long n) { return radix_blocks(n) << kRadixMaxBits; }

static size_t radix_scan_bytes(long long n) {
    if (radix_counters(n) <= kRadixSmallScan) return 0;
    size_t bytes = 0;
    unsigned *p = nullptr;
    if (cub::DeviceScan::ExclusiveSum(nullptr, bytes, p, p, (long long)radix_counters(n)) != cudaSuccess) {
        (void)cudaGetLastError();
        bytes = (size_t)(radix_counters(n) / 256 + 4096) * 64;   // no device to ask: generous guess
    }
    return bytes;
}
// bytes behind the pair buffers: the counters and the prefix sum's scratch
static size_t radix_scratch_bytes(long long n) {
    return sar_round_up((size_t)radix_counters(n) * 4, 256) + sar_round_up(radix_scan_bytes(n), 256);
}

// One stable sort by the low `bits` bits of the keys, pairs (k0, v0) -> (k_out, v_out); (kt, vt) holds intermediate pairs.
// k0 / v0 may be kt / vt only when the number of passes is even.
static sar_status radix_sort_pairs(long long n, int bits, const unsigned *k0, const unsigned *v0, unsigned *kt, unsigned *vt, unsigned *k_out,
                                   unsigned *v_out, void *scratch, cudaStream_t st) {
    const int passes = radix_passes(bits);
    const unsigned blocks = (unsigned)radix_blocks(n);
    unsigned *counts = static_cast<unsigned *>(scratch);
    void *scan_ws = static_cast<char *>(scratch) + sar_round_up((size_t)radix_counters(n) * 4, 256);
    int shift = 0;
    for (int p = 0; p < passes; ++p) {
        const int b = (bits - shift + passes - p - 1) / (passes - p), bins = 1 << b;
        const bool to_out = (passes - 1 - p) % 2 == 0;
        unsigned *ko = to_out ? k_out : kt, *vo = to_out ? v_out : vt;
        radix_count_kernel<<<blocks, kRadixThreads, 0, st>>>(n, k0, shift, b, counts, blocks);
        SAR_TRY(sar_after_launch());
        const long long counters = (long long)bins * blocks;
        if (counters <= kRadixSmallScan) {
            radix_scan_kernel<<<1, 1024, 0, st>>>((int)counters, counts);
            SAR_TRY(sar_after_launch());
        } else {
            size_t need = 0;
            SAR_CUDA_TRY(cub::DeviceScan::ExclusiveSum(nullptr, need, counts, counts, counters, st));
            SAR_CUDA_TRY(cub::DeviceScan::ExclusiveSum(scan_ws, need, counts, counts, counters, st));
        }
        radix_move_kernel<<<blocks, kRadixThreads, 0, st>>>(n, k0, v0, shift, b, counts, blocks, ko, vo);
        SAR_TRY(sar_after_launch());
        k0 = ko;
        v0 = vo;
        shift += b;
    }
    return SAR_OK;
}

}  // namespace sar
