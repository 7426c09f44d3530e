// Long rows, from their segments' records (see sar_rows_kernel.cuh).  Most long rows have a handful of segments, and what their
// merge costs is a chain of loads (which row, its records' statistics, its records), not the bytes: so where there are more long
// rows than a couple of blocks per SM, a row of up to kMergeFew segments is one warp's, four of them to a block, and its loads go out
// together.  With a block of 128 threads per
// row, whatever its length, and a warp per row and head for the destination-major records, the three merges of 8 heads of 32
// (1 million nodes, 200 edges per node, 575,000 segments) took 0.48, 0.50 and 0.29 ms, now 0.30, 0.08 and 0.19; the forward merge of 2 heads of
// 64 (233,000 nodes, 11.6 million edges) 17 us, now 10.5.  Hubs (8 heads of 32, bf16, us each, by the block per row and head / by
// four neighbouring rows and one warp / now): four of 100,000 edges beside 400 of 600, forward 45 / 167 / 48, destination-major 19 / 52 / 13;
// one of a million, destination-major 212 / 487 / 79.
// The records of a hub row (hundreds) are read by all threads of the block, by several streams at once - a thread holds one
// float4 column of every kStreams-th record - and the streams are added up in shared memory in a fixed order, so a result does
// not depend on the schedule.
#include "sar_dispatch.cuh"
#include "sar_rows.cuh"

namespace sar {

constexpr int kMergeThreads = 128;

__device__ __forceinline__ void add4(float4 &a, const float4 &b, float f) {
    a.x = fmaf(b.x, f, a.x);
    a.y = fmaf(b.y, f, a.y);
    a.z = fmaf(b.z, f, a.z);
    a.w = fmaf(b.w, f, a.w);
}

// Elements of a finished row.  `c` = first float of the column in the padded row (heads of vph*EPV floats).
template <typename T, typename Fn>
__device__ __forceinline__ void merge_store(const RowArgs &a, long long row, int c, const float4 &x, Fn &&finish) {
    const int fp = a.vph * Elem<T>::EPV;
    const float v[4] = {x.x, x.y, x.z, x.w};
    const int head = c / fp, f0 = c - head * fp;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (f0 + k < a.F) finish(row * (long long)a.H * a.F + (long long)head * a.F + f0 + k, head, v[k]);
}

// Sum over a row's records of (column of the record) x (factor of (record, head)); valid in the threads of stream 0.
template <typename Fn>
__device__ __forceinline__ float4 merge_columns(const RowArgs &a, long long s0, long long s1, int c, int stream, int streams,
                                                float4 *red, int cols_pad, int col, Fn &&factor) {
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    long long s = s0 + stream;
    for (; s + 3LL * streams < s1; s += 4LL * streams) {
        float4 r[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) r[u] = *reinterpret_cast<const float4 *>(a.sp.part + (s + (long long)u * streams) * a.sp.pstride + c);
#pragma unroll
        for (int u = 0; u < 4; ++u) add4(x, r[u], factor(s + (long long)u * streams));
    }
    for (; s < s1; s += streams) add4(x, *reinterpret_cast<const float4 *>(a.sp.part + s * a.sp.pstride + c), factor(s));
    if (streams > 1) {
        if (stream < streams) red[stream * cols_pad + col] = x;
        __syncthreads();
        if (stream == 0)
            for (int k = 1; k < streams; ++k) add4(x, red[k * cols_pad + col], 1.f);
        __syncthreads();
    }
    return x;
}

// What a row's records are scaled against: its maximum, or the lowest finite number where that is -inf, so that a record of masked
// scores alone (maximum -inf) weighs nothing.
__device__ __forceinline__ float merge_shift(float m) { return fmaxf(m, -3.402823466e38f); }

// One column (float4 x, its first float c of the padded row) of a finished row; what a forward row needs besides: its
// denominator d and the factor `old` of the state's numerator.
template <typename T, int MODE>
__device__ __forceinline__ void merge_finish(const RowArgs &a, long long row, int c, const float4 &x, float d, float old) {
    const bool first = a.flags & SAR_FIRST, last = a.flags & SAR_LAST;
    T *out = reinterpret_cast<T *>(a.out);
    if constexpr (MODE == kRowFwd) {
        merge_store<T>(a, row, c, x, [&](long long o, int, float y) {
            if (!first) y += a.acc[o] * old;
            if (!last || (a.flags & SAR_KEEP_NUMERATOR)) a.acc[o] = y;
            if (last) {
                y *= d > 0.f ? 1.f / d : 0.f;
                Elem<T>::store1(out + o, (a.flags & SAR_RELU_OUT) ? fmaxf(y, 0.f) : y);
            }
        });
    } else if constexpr (MODE == kRowSrc) {
        merge_store<T>(a, row, c, x, [&](long long o, int, float y) { Elem<T>::store1(out + o, y); });
    } else {
        const float ds = a.dst_scale ? a.dst_scale[row] : 1.f;
        float inv = 1.f;
        if ((a.flags & SAR_MEAN) && last) inv = a.deg[row] > 0 ? 1.f / (float)a.deg[row] : 0.f;
        merge_store<T>(a, row, c, x, [&](long long o, int, float y) {
            y *= ds;
            if (!first) {
                if constexpr (sizeof(T) == 4) y += out[o];
                else y += __bfloat162float(out[o]);
            }
            y *= inv;
            if (a.mix.x0 && last)
                y = (a.mix.keep * Elem<T>::load1(reinterpret_cast<const T *>(a.mix.x0) + o) + a.mix.scale * y) * (a.mix.post ? a.mix.post[row] : 1.f);
            Elem<T>::store1(out + o, y);
        });
    }
}

// A row of up to kMergeFew records and (forward, source-major) kMergeHeads heads, by one warp: a lane is a record for the
// statistics and a float4 column, or several, for the sums.
constexpr int kMergeFew = 32, kMergeHeads = 16;
// With up to two blocks per SM a block per row is as fast or faster: 128 rows of 6 segments, 8 heads of 48 bf16, source-major 8.6
// against 10.6 us; 592 rows 12.6 against 10.7, 9600 rows 56 against 50 and forward 85 against 55.
constexpr int kMergeMany = 296;
// the most long rows of a block; a sum has no statistics to wait for, and there a block per row is faster (2.45 million rows of 1 KB 55 us against 57 to 80)
template <int MODE>
struct MergeRows {
    static constexpr int n = MODE == kRowSum ? 1 : kMergeThreads / 32;
};
template <typename T, int MODE>
__device__ __forceinline__ void merge_few(const RowArgs &a, long long row, long long s0, int n, float (*fac)[kMergeHeads], float *sM, float *sD, float *sOld) {
    constexpr int EPV = Elem<T>::EPV;
    constexpr bool kF = MODE == kRowFwd;
    const int lane = threadIdx.x & 31;
    const int rowf = a.H * a.vph * EPV;
    const bool first = a.flags & SAR_FIRST;
    // two columns of four records at a time; the first ones are asked for before the statistics are there
    float4 r[2][4];
    auto ask = [&](int c, int s) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (c + j * 128 < rowf && s + u < n) r[j][u] = *reinterpret_cast<const float4 *>(a.sp.part + (s0 + s + u) * a.sp.pstride + c + j * 128);
    };
    ask(lane * 4, 0);
    const float *rec = a.sp.part + (s0 + (lane < n ? lane : n - 1)) * a.sp.pstride + rowf;
    if constexpr (kF) {
        for (int h0 = 0; h0 < a.H; h0 += 4) {
            float m[4], d[4], mo[4], dold[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int h = h0 + k < a.H ? h0 + k : a.H - 1;
                m[k] = rec[h];
                d[k] = lane < n ? rec[a.H + h] : 0.f;
                mo[k] = first ? SAR_NEG_INF : a.m_io[row * a.H + h];
                dold[k] = first ? 0.f : a.d_io[row * a.H + h];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float M = m[k];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
                const float mn = fmaxf(M, mo[k]), f = fast_exp(m[k] - merge_shift(mn));
                float s = d[k] * f;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                const float fo = mo[k] == mn ? 1.f : fast_exp(mo[k] - mn);
                if (h0 + k < a.H) {
                    if (lane < n) fac[lane][h0 + k] = f;
                    if (lane == 0) {
                        sM[h0 + k] = mn;
                        sD[h0 + k] = s + dold[k] * fo;
                        sOld[h0 + k] = fo;
                    }
                }
            }
        }
        __syncwarp();
        if (lane < a.H) {
            a.m_io[row * a.H + lane] = sM[lane];
            a.d_io[row * a.H + lane] = sD[lane];
        }
    }
    if constexpr (MODE == kRowSrc) {
        for (int h = 0; h < a.H; ++h) {
            float d = lane < n ? rec[h] : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            if (lane == 0) a.dscal[row * a.H + h] = d;
        }
    }
    for (int c = lane * 4; c < rowf; c += 256) {
        const int head[2] = {c / (a.vph * EPV), (c + 128) / (a.vph * EPV)};
        float4 x[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
        for (int s = 0; s < n; s += 4) {
            if (c != lane * 4 || s > 0) ask(c, s);
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (c + j * 128 < rowf && s + u < n) add4(x[j], r[j][u], kF ? fac[s + u][head[j]] : 1.f);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if (c + j * 128 < rowf) merge_finish<T, MODE>(a, row, c + j * 128, x[j], kF ? sD[head[j]] : 0.f, kF ? sOld[head[j]] : 0.f);
    }
}

// The w-th long row of a block: the rows of a block are far apart, for the heaviest often follow one another (nodes in the order of
// their degrees), and a block takes its heavy rows one after the other.
__device__ __forceinline__ int merge_row_of(unsigned block, int w) { return (int)(block + (unsigned)w * gridDim.x); }

// MODE: kRowFwd, kRowSrc, kRowSum.  A block has ROWS long rows, a warp each; then those of more records together.
template <typename T, int MODE, int ROWS>
__global__ void __launch_bounds__(kMergeThreads) rows_merge_kernel(const RowArgs a) {
    constexpr int EPV = Elem<T>::EPV;
    constexpr bool kF = MODE == kRowFwd;
    after_predecessor();
    __shared__ float4 red[kMergeThreads];
    __shared__ float sM[SAR_MAX_HEADS], sD[SAR_MAX_HEADS], sOld[SAR_MAX_HEADS];
    __shared__ float fac[ROWS][kF && ROWS > 1 ? kMergeFew : 1][kMergeHeads], stat[ROWS][3][kMergeHeads];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rowf = a.H * a.vph * EPV;
    const bool first = a.flags & SAR_FIRST;
    auto few = [&](int lr, long long &s0, long long &s1) {
        s0 = a.sp.long_seg[lr];
        s1 = a.sp.long_seg[lr + 1];
        return ROWS > 1 && s1 - s0 <= kMergeFew && a.H <= kMergeHeads;
    };
    if constexpr (ROWS > 1) {
        const int lr = merge_row_of(blockIdx.x, warp);
        long long s0, s1;
        if (lr < a.sp.n_long && few(lr, s0, s1))
            merge_few<T, MODE>(a, a.sp.long_row[lr], s0, (int)(s1 - s0), fac[warp], stat[warp][0], stat[warp][1], stat[warp][2]);
    }
    for (int w = 0; w < ROWS; ++w) {
        const int lr = merge_row_of(blockIdx.x, w);
        long long s0, s1;
        if (lr >= a.sp.n_long || few(lr, s0, s1)) continue;
        const long long row = a.sp.long_row[lr];
        __syncthreads();

        if constexpr (kF) {   // statistics of the row: a warp per head
            for (int h = warp; h < a.H; h += kMergeThreads / 32) {
                float M = SAR_NEG_INF;
                for (long long s = s0 + lane; s < s1; s += 32) M = fmaxf(M, a.sp.part[s * a.sp.pstride + rowf + h]);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
                const float m_old = first ? SAR_NEG_INF : a.m_io[row * a.H + h], d_old = first ? 0.f : a.d_io[row * a.H + h];
                const float mn = fmaxf(M, m_old);
                float d = 0.f;
                for (long long s = s0 + lane; s < s1; s += 32) {
                    const float *rec = a.sp.part + s * a.sp.pstride + rowf;
                    d += rec[a.H + h] * fast_exp(rec[h] - merge_shift(mn));
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
                const float fo = m_old == mn ? 1.f : fast_exp(m_old - mn);
                d += d_old * fo;
                if (lane == 0) {
                    sM[h] = mn;
                    sD[h] = d;
                    sOld[h] = fo;
                }
            }
            __syncthreads();
            if (tid < a.H) {
                a.m_io[row * a.H + tid] = sM[tid];
                a.d_io[row * a.H + tid] = sD[tid];
            }
        }
        if constexpr (MODE == kRowSrc) {
            for (int h = warp; h < a.H; h += kMergeThreads / 32) {
                float d = 0.f;
                for (long long s = s0 + lane; s < s1; s += 32) d += a.sp.part[s * a.sp.pstride + rowf + h];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
                if (lane == 0) a.dscal[row * a.H + h] = d;
            }
        }

        const int cols = rowf / 4;
        const int cols_pad = cols < kMergeThreads ? cols : kMergeThreads;
        const int streams = (kMergeThreads / cols_pad) < (int)(s1 - s0) ? kMergeThreads / cols_pad : (int)(s1 - s0);
        const int col = tid % cols_pad, stream = tid / cols_pad;
        for (int c0 = 0; c0 < cols; c0 += cols_pad) {
            const bool in = c0 + col < cols && stream < streams;
            const int c = in ? (c0 + col) * 4 : 0;
            const int head = c / (a.vph * EPV);
            const float shift = kF ? merge_shift(sM[head]) : 0.f;
            const float4 x = merge_columns(a, in ? s0 : s1, s1, c, stream, streams, red, cols_pad, col, [&](long long s) {
                if constexpr (kF) return fast_exp(a.sp.part[s * a.sp.pstride + rowf + head] - shift);
                else return 1.f;
            });
            if (!in || stream != 0) continue;
            merge_finish<T, MODE>(a, row, c, x, kF ? sD[head] : 0.f, kF ? sOld[head] : 0.f);
        }
    }
}

// Destination-major: D, B and S of the segments are numbers, 3 H of them one after the other in a record; a lane per number (of the
// heads h0 .. h0 + 9, so that they fit a warp), half a warp per record where 15 lanes do.  A row of up to kMergeAlone records is one
// warp's; one of more is summed by the warps of the block together, every fourth step's records a warp's, and added up in shared
// memory in a fixed order.
constexpr int kMergeAlone = 64;
// the sum of number p over the records s, s + step, .., eight loads in flight
__device__ __forceinline__ float merge_numbers(const float *p, long long pstride, long long s, long long s1, int step) {
    constexpr int U = 8;
    float part[U];
#pragma unroll
    for (int u = 0; u < U; ++u) part[u] = 0.f;
    p += s * pstride;
    pstride *= step;
    int n = s < s1 ? (int)((s1 - s + step - 1) / step) : 0;
    for (; n >= U; n -= U, p += U * pstride) {
        float r[U];
#pragma unroll
        for (int u = 0; u < U; ++u) r[u] = __ldg(p + u * pstride);
#pragma unroll
        for (int u = 0; u < U; ++u) part[u] += r[u];
    }
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
        if (u < n) part[u] += __ldg(p + u * pstride);
    return ((part[0] + part[1]) + (part[2] + part[3])) + ((part[4] + part[5]) + (part[6] + part[7]));
}
template <bool PART>
__global__ void __launch_bounds__(kMergeThreads) rows_dst_merge_kernel(const RowArgs a) {
    after_predecessor();
    constexpr int W = kMergeThreads / 32;
    __shared__ float red[W][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto merge_row = [&](int lr, bool alone) {   // by this warp, or by all of the block
        const long long row = a.sp.long_row[lr], s0 = a.sp.long_seg[lr], s1 = a.sp.long_seg[lr + 1];
        for (int h0 = 0; h0 < a.H; h0 += 10) {
            const int H = min(a.H - h0, 10), lanes = H <= 5 ? 16 : 32, at = lane & (lanes - 1), step = 32 / lanes;
            const int q = at / H, h = at - q * H;   // number q (D, B, S) of head h0 + h
            float x = 0.f;
            if (q < 3 && !(PART && q == 0)) {
                const float *p = a.sp.part + q * a.H + h0 + h;
                x = merge_numbers(p, a.sp.pstride, s0 + (alone ? 0 : warp * step) + lane / lanes, s1, alone ? step : W * step);
            }
            if (!alone) {
                red[warp][lane] = x;
                __syncthreads();
                x = (red[0][lane] + red[1][lane]) + (red[2][lane] + red[3][lane]);
                __syncthreads();
            }
            if (lanes == 16) x += __shfl_xor_sync(0xffffffffu, x, 16);
            const float D = x, Bs = __shfl_sync(0xffffffffu, x, (lane + H) & 31), S = __shfl_sync(0xffffffffu, x, (lane + 2 * H) & 31);
            if (lane < H && (alone || warp == 0)) {
                const long long o = row * a.H + h0 + lane;
                if (PART) {
                    const float y = Bs - a.rec[o].w * S;
                    a.dscal[o] = (a.flags & SAR_FIRST) ? y : a.dscal[o] + y;
                } else {
                    const float dd = a.d[o];
                    a.dscal[o] = Bs - D * S;
                    a.rec[o] = make_float4(a.el[o], a.m[o], dd > 0.f ? __fdividef(1.f, dd) : 0.f, D);
                }
            }
        }
    };
    static_assert(W == 4, "four shares");
    auto is_few = [&](int lr) { return a.sp.long_seg[lr + 1] - a.sp.long_seg[lr] <= kMergeAlone; };
    const int mine = merge_row_of(blockIdx.x, warp);
    const bool there = mine < a.sp.n_long, few = there && is_few(mine);
    if (few) merge_row(mine, true);
    if (!__syncthreads_or(there && !few)) return;
    for (int w = 0; w < W; ++w) {
        const int lr = merge_row_of(blockIdx.x, w);
        if (lr < a.sp.n_long && !is_few(lr)) merge_row(lr, false);
    }
}

// The end of Algorithm 1: out = numerator / d for every row (0 where d = 0), one thread per 16-byte vector of `out`.
// Follows a last partition step that left the complete state behind (aligned shapes).
template <typename T>
__global__ void __launch_bounds__(256) rows_finalize_kernel(const RowArgs a) {
    after_predecessor();
    constexpr int EPV = Elem<T>::EPV;
    const long long vi = (long long)blockIdx.x * 256 + threadIdx.x;
    const int n_vec = a.H * a.vph;
    if (vi >= a.n_rows * n_vec) return;
    const long long row = vi / n_vec;
    const float dd = a.d_io[row * a.H + (int)(vi - row * n_vec) / a.vph];
    const float inv = dd > 0.f ? __fdividef(1.f, dd) : 0.f;
    const float4 *src = reinterpret_cast<const float4 *>(a.acc) + vi * (EPV / 4);
    float x[EPV];
#pragma unroll
    for (int q = 0; q < EPV / 4; ++q) {
        const float4 t = src[q];
        x[4 * q] = t.x * inv;
        x[4 * q + 1] = t.y * inv;
        x[4 * q + 2] = t.z * inv;
        x[4 * q + 3] = t.w * inv;
    }
    if (a.flags & SAR_RELU_OUT) {
#pragma unroll
        for (int e = 0; e < EPV; ++e) x[e] = fmaxf(x[e], 0.f);
    }
    reinterpret_cast<uint4 *>(a.out)[vi] = Elem<T>::pack(x);
}

template <typename T, int MODE, int ROWS>
static sar_status launch_merge_rows(const RowArgs &a, const char *name, cudaStream_t st) {
    SAR_LAUNCH(name, st, launch(rows_merge_kernel<T, MODE, ROWS>, (unsigned)((a.sp.n_long + ROWS - 1) / ROWS), kMergeThreads, 0, st, a));
    return sar_after_launch();
}
template <int MODE>
static sar_status launch_merge(const RowArgs &a, sar_dtype t, const char *name, cudaStream_t st) {
    constexpr int R = MergeRows<MODE>::n;
    if (R > 1 && a.sp.n_long > kMergeMany)
        return t == SAR_F32 ? launch_merge_rows<float, MODE, R>(a, name, st) : launch_merge_rows<__nv_bfloat16, MODE, R>(a, name, st);
    return t == SAR_F32 ? launch_merge_rows<float, MODE, 1>(a, name, st) : launch_merge_rows<__nv_bfloat16, MODE, 1>(a, name, st);
}

sar_status rows_fwd_merge(const RowArgs &a, sar_dtype t, cudaStream_t st) { return launch_merge<kRowFwd>(a, t, "gat_fwd_merge", st); }
sar_status rows_src_merge(const RowArgs &a, sar_dtype t, cudaStream_t st) { return launch_merge<kRowSrc>(a, t, "gat_bwd_src_merge", st); }
sar_status rows_sum_merge(const RowArgs &a, sar_dtype t, cudaStream_t st) { return launch_merge<kRowSum>(a, t, "spmm_merge", st); }

sar_status rows_fwd_finalize(const RowArgs &a, sar_dtype t, cudaStream_t st) {
    const unsigned blocks = (unsigned)((a.n_rows * a.H * a.vph + 255) / 256);
    if (t == SAR_F32)
        SAR_LAUNCH("gat_fwd_finalize", st, launch(rows_finalize_kernel<float>, blocks, 256, 0, st, a));
    else
        SAR_LAUNCH("gat_fwd_finalize", st, launch(rows_finalize_kernel<__nv_bfloat16>, blocks, 256, 0, st, a));
    return sar_after_launch();
}

sar_status rows_dst_merge(const RowArgs &a, bool part, cudaStream_t st) {
    constexpr int W = kMergeThreads / 32;
    const unsigned blocks = (unsigned)(a.sp.n_long > kMergeMany ? (a.sp.n_long + W - 1) / W : a.sp.n_long);
    if (part)
        SAR_LAUNCH("gat_bwd_dst_merge", st, launch(rows_dst_merge_kernel<true>, blocks, kMergeThreads, 0, st, a));
    else
        SAR_LAUNCH("gat_bwd_dst_merge", st, launch(rows_dst_merge_kernel<false>, blocks, kMergeThreads, 0, st, a));
    return sar_after_launch();
}

}  // namespace sar
