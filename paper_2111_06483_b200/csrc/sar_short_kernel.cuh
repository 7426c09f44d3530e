// Kernel for short rows (internal): the gather passes - forward, destination-major and source-major backward, sum - of narrow
// rows (up to 32 vectors of 16 bytes), a row per group of lanes and nothing else.
//
// G lanes x 16 bytes cover a gathered row, and a group of G lanes owns one row: it reads the row's column ids, asks for the score
// terms and the rows of four edges at a time and adds them up; every lane forms the weight of its own head itself.  No shared
// memory, nothing staged, nothing folded over lanes but the dot products of a head.  That repeats an exponential in the lanes of
// a head, and the longest of a warp's 32/G rows sets its pace; but a row costs next to nothing besides its edges, where the row
// kernel spends 500 and more instructions of a whole warp on the start and the end of each.  So rows of more than kShortEdges
// edges are left for last and shared by all groups of the warp (four edges to each at a time), and a segment of a long row has a
// warp to itself from the start: without that a segment of 256 edges was a chain of 64 loads, 50 us, whatever the rest did.
// Where a row fills the warp there are no groups to share it, and in a launch of few rows a segment or a row of a hundred edges and more is
// taken by the four warps of a block (rest_of_block): 8 heads of 24, bf16, 3,200 nodes with 2 edges and hubs of 400, backward 70 -> 32 us
// (span kernels 57), 5 heads of 24, 8,600 nodes, likewise 73 -> 35 (51).
//
// What bounds it: the chain row pointers -> column ids -> rows of a warp, which 32 warps an SM hide, then the issue slots of groups that
// wait for longer ones.  Measured against the kernels that took these rows before (kShortEdges 12 and 48 within 5 %, but for
// long uniform rows, where 48 is better by up to 25 %, and hubs, where it is worse by as much): 200,000 nodes, 3 edges each,
// 1 head of 32, bf16, forward 77 -> 21 us, backward 180 -> 45; 8 heads of 8, backward 446 -> 104; a sum of 64-byte rows over 1.5 million
// edges 58 -> 36; the same head over 445,858 nodes in 16 steps, forward and backward, 2.74 -> 1.74 ms.
//
// Sums of four edges are formed first and added to the row's: chains of 4 + deg/4 additions, fewer with the groups' shares.
// The softmax is taken against the running maximum of the row's scores: the sums so far times exp(m_before - m) in the
// multiply-add that adds the next four edges, so that it costs one exponential per lane and step, and no weight exceeds 1 whatever the
// scores and features.  The maximum starts at the lowest finite number: a score of -inf (a masked source) weighs nothing against it, and
// a row without any other has m = -inf and d = 0, like one without edges.  A row's arithmetic does not depend on the rows around it, but for
// those that a block may share.
#pragma once

#include "sar_rows_kernel.cuh"

namespace sar {

constexpr int kShortThreads = 128, kShortWarps = kShortThreads / 32;
constexpr int kShortEdges = 24;   // rows of more are shared by the groups of the warp

// A row, or a segment of one
struct ShortItem {
    long long row, p;   // row, first edge
    int n, seg;         // edges (< 0: nothing to do); segment (< 0: a row)
};
// The rows of a block (or the segment, where it has one): one row per group of NG to a warp, or a segment per warp.  A row has no more edges
// than there are (fewer than 2^30, see few_edges), whatever its pointers say, so that no position and no step beyond it overflows.
template <int NG, bool SHARE>
__device__ __forceinline__ ShortItem short_item(const RowArgs &a, unsigned block) {
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const long long item = SHARE && a.wide ? (block < a.sp.n_seg ? block : a.sp.n_seg + (block - a.sp.n_seg) * kShortWarps + wid) : (long long)block * kShortWarps + wid;
    ShortItem x{0, 0, -1, -1};
    if (item < a.sp.n_seg) {
        x.seg = (int)item;
        int lo = 0, hi = a.sp.n_long;   // last lo with long_seg[lo] <= item, 32 probes at a time
        while (hi - lo > 1) {
            const int step = (hi - lo + 31) >> 5;
            const int at = lo + lane * step;
            const bool ok = at < hi && __ldg(a.sp.long_seg + at) <= item;
            lo += (__popc(__ballot_sync(kAll, ok)) - 1) * step;
            hi = min(hi, lo + step);
        }
        x.row = __ldg(a.sp.long_row + lo);
        x.p = __ldg(a.indptr + x.row) + (item - __ldg(a.sp.long_seg + lo)) * a.sp.threshold;
        const long long rest = __ldg(a.indptr + x.row + 1) - x.p;
        x.n = (int)(rest < a.sp.threshold ? rest : a.sp.threshold);
    } else {
        x.row = (item - a.sp.n_seg) * NG + lane / (32 / NG);
        if (x.row < a.n_rows) {
            x.p = __ldg(a.indptr + x.row);
            const long long len = __ldg(a.indptr + x.row + 1) - x.p;
            if (a.sp.threshold <= 0 || len <= a.sp.threshold) x.n = (int)min(len, a.nnz);   // else its segments are items of their own
        }
    }
    return x;
}

// One row (or segment) of n edges from position p on, every `step`-th four of them from the e0-th on.  FOLD: the groups of the warp share
// it, group 0 writes; with `share` the warps of the block too, warp 0 writes.
template <typename T, int NV, int HP, int MODE>
struct ShortRow {
    static constexpr int EPV = Elem<T>::EPV, NP = EPV / 2, U = 4;
    static constexpr int G = NV, NG = 32 / G, VPHP = NV / HP;
    static constexpr bool kF = MODE == kRowFwd || MODE == kRowFwdPart, kD = MODE == kRowDst || MODE == kRowDstPart;
    static constexpr bool kS = MODE == kRowSrc, kAgg = MODE == kRowSum || MODE == kRowSumW;
    static constexpr bool kAcc = kF || kS || kAgg, kDot = kD || kS;
    // Floats per lane that warps hand over: up to EPV + 2.  The same for every pass, for between two launches that need different shares of the
    // L1 as shared memory an SM has to run empty (backward passes of 1,500 rows 13.6 -> 15.8 us).
    static constexpr int kShare = 10;
    static_assert(NV <= 32, "one vector per lane");

    template <bool FOLD>
    static __device__ __forceinline__ void process(const RowArgs &a, const ShortItem &item, int e0, int step, bool live, float (*share)[G][kShare]) {
        constexpr unsigned kAll = 0xffffffffu;
        constexpr float kLowest = -3.402823466e38f;
        const int lane = threadIdx.x & 31, gl = lane & (G - 1), grp = lane / G;
        const int h0 = kAgg ? 0 : (int)blockIdx.y * HP, have = a.H - h0;
        const int hv = gl / VPHP, vec = gl % VPHP + (kAgg ? (int)blockIdx.y * NV : 0);
        const bool okv = hv < have && vec < a.vph;
        const int hc = h0 + (hv < have ? hv : have - 1), vc = vec < a.vph ? vec : a.vph - 1;   // a lane without a vector repeats the last one
        const bool first = a.flags & SAR_FIRST, last = a.flags & SAR_LAST;
        const unsigned HF = (unsigned)(a.H * a.F);
        const int oel = hc * a.F + vec * EPV, left = okv ? a.F - vec * EPV : 0;
        const bool head_lane = okv && gl % VPHP == 0;
        const unsigned gofs = (unsigned)(hc * a.vph + vc) * 16u;
        const char *gsrc = reinterpret_cast<const char *>(a.gather) + gofs;
        const long long row = item.row, p = item.p;
        const int n = item.n;
        const bool seg = FOLD && item.seg >= 0;
        const long long so = row * a.H + hc;
        // an inconsistent graph gives wrong sums, not a wrong address
        auto column = [&](int e) {
            const long long q = p + min(e, n - 1);
            return min((unsigned)ld_stream_i32(a.indices + (q < a.nnz ? q : a.nnz - 1)), a.last_col);
        };
        float rs = 0.f, rm = 0.f, ri = 0.f, pm = kF ? SAR_NEG_INF : 0.f, pd = 0.f;
        uint4 rv = make_uint4(0u, 0u, 0u, 0u);
        unsigned col[U];
        if (live && n > 0) {
#pragma unroll
            for (int u = 0; u < U; ++u) col[u] = column(e0 + u);
            if constexpr (!kAgg) rs = __ldg((kS ? a.er : a.el) + so);
            if constexpr (kD) {
                rm = __ldg(a.m + so);
                ri = __ldg(a.d + so);
            }
            if constexpr (kDot) {
                if (okv) rv = __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const char *>(a.rowvec) + (unsigned long long)row * a.row_bytes + gofs));
            }
            if constexpr (MODE == kRowDstPart) {
                if (!seg && okv) {
                    pd = a.rec[so].w;
                    if (!first) pm = a.dscal[so];
                }
            }
        }
        if constexpr (MODE == kRowFwdPart) {
            if (live && !seg && !first && okv && (n > 0 || last)) {
                pm = a.m_io[so];
                pd = a.d_io[so];
            }
        }
        if constexpr (MODE == kRowFwdPart || MODE == kRowDstPart) __syncwarp();   // every lane of a head has read the state before one writes it
        f32x2 acc[NP], go[NP];
        float l = 0.f, m = kLowest, dD = 0.f, dB = 0.f;
#pragma unroll
        for (int k = 0; k < NP; ++k) acc[k] = zero2();
        if constexpr (kDot) Pairs<T>::get(rv, go);
        if constexpr (kD) ri = ri > 0.f ? __fdividef(1.f, ri) : 0.f;

        // four edges at a time; positions past the end repeat the last edge's loads and add nothing: not zero times its row, which may hold
        // an infinity, but in a sum no product, in the other passes zero times zeros (the cheaper of the two for each)
        for (int e = e0; e < n; e += step) {
            float t[U], g4[U], ag[U], keep = 1.f;
            float4 rc[kS ? U : 1];
            uint4 x[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if constexpr (kF || kD) t[u] = __ldg(a.er + (long long)col[u] * a.H + hc);
                if constexpr (kS) rc[u] = __ldg(a.rec + (long long)col[u] * a.H + hc);
                if constexpr (MODE == kRowSumW) t[u] = __ldg(a.src_scale + col[u]);
                if constexpr (MODE == kRowSum) t[u] = 1.f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) x[u] = __ldg(reinterpret_cast<const uint4 *>(gsrc + (unsigned long long)col[u] * a.row_bytes));
            if (e + step < n) {
#pragma unroll
                for (int u = 0; u < U; ++u) col[u] = column(e + step + u);
            }
            if constexpr (kF) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    float gr;
                    t[u] = leaky(rs + t[u], a.slope, gr);
                }
                const float top = fmaxf(fmaxf(fmaxf(t[0], t[1]), fmaxf(t[2], t[3])), m);
                keep = row_ex2((m - top) * kRowLog2e);   // the sums so far follow the maximum (Sec. 3.4)
                m = top;
#pragma unroll
                for (int u = 0; u < U; ++u) t[u] = row_ex2((t[u] - top) * kRowLog2e);
            } else if constexpr (kD) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const float s = leaky(rs + t[u], a.slope, g4[u]);
                    t[u] = row_ex2((s - rm) * kRowLog2e) * ri;
                }
            } else if constexpr (kS) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const float s = leaky(rc[u].x + rs, a.slope, g4[u]);
                    t[u] = row_ex2((s - rc[u].y) * kRowLog2e) * rc[u].z;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (!kAgg && u > 0 && e + u >= n) t[u] = 0.f;
                if constexpr (kDot) ag[u] = t[u] * g4[u];
            }
            if constexpr (kF) l = fmaf(l, keep, (t[0] + t[1]) + (t[2] + t[3]));
            if constexpr (kD) l += (ag[0] + ag[1]) + (ag[2] + ag[3]);
            if constexpr (kS) l += (ag[0] * rc[0].w + ag[1] * rc[1].w) + (ag[2] * rc[2].w + ag[3] * rc[3].w);
            if (!kAgg && e + U > n) {
#pragma unroll
                for (int u = 1; u < U; ++u)
                    if (e + u >= n) x[u] = make_uint4(0u, 0u, 0u, 0u);
            }
            f32x2 part[NP];
            float b = 0.f, d = 0.f;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                f32x2 y[NP];
                Pairs<T>::get(x[u], y);
                if (kAgg && u > 0 && e + u >= n) continue;
                if constexpr (kAcc) {
#pragma unroll
                    for (int k = 0; k < NP; ++k) part[k] = fma2(y[k], pack2(t[u], t[u]), u == 0 ? zero2() : part[k]);
                }
                if constexpr (kDot) {
                    f32x2 dot = fma2(y[0], go[0], zero2());
#pragma unroll
                    for (int k = 1; k < NP; ++k) dot = fma2(y[k], go[k], dot);
                    const float s = dot.x + dot.y;
                    b = fmaf(s, ag[u], b);
                    if constexpr (MODE == kRowDst) d = fmaf(s, t[u], d);
                }
            }
            if constexpr (kAcc) {
#pragma unroll
                for (int k = 0; k < NP; ++k) acc[k] = fma2(acc[k], pack2(keep, keep), part[k]);
            }
            dB += b;
            dD += d;
        }

        // ---- the row's end ----------------------------------------------------------------------------------------------------
        float y[EPV];
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            y[2 * k] = acc[k].x;
            y[2 * k + 1] = acc[k].y;
        }
        if constexpr (FOLD) {
            if constexpr (kF) {   // the groups' sums against one shift, the maximum
                float mm = m;
#pragma unroll
                for (int off = G; off < 32; off <<= 1) mm = fmaxf(mm, __shfl_xor_sync(kAll, mm, off));
                const float f = row_ex2((m - mm) * kRowLog2e);
                l *= f;
#pragma unroll
                for (int k = 0; k < EPV; ++k) y[k] *= f;
                m = mm;
            }
#pragma unroll
            for (int off = G; off < 32; off <<= 1) {
                if constexpr (!kAgg) l += __shfl_xor_sync(kAll, l, off);
                if constexpr (kAcc) {
#pragma unroll
                    for (int k = 0; k < EPV; ++k) y[k] += __shfl_xor_sync(kAll, y[k], off);
                }
            }
        }
        if constexpr (kDot) {
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                if (off < VPHP || (FOLD && off >= G)) {
                    if constexpr (MODE == kRowDst) dD += __shfl_xor_sync(kAll, dD, off);
                    dB += __shfl_xor_sync(kAll, dB, off);
                }
            }
        }
        if (FOLD && share) {
            const int wid = threadIdx.x >> 5;
            if (grp == 0) {
                float *mine = share[wid][gl];
                if constexpr (kAcc) {
#pragma unroll
                    for (int k = 0; k < EPV; ++k) mine[k] = y[k];
                }
                if constexpr (!kAgg) mine[kAcc ? EPV : 0] = l;
                if constexpr (kF) mine[EPV + 1] = m;
                if constexpr (kDot) mine[kAcc ? EPV + 1 : 1] = dB;
                if constexpr (kD) mine[2] = dD;
            }
            __syncthreads();
            if (wid == 0) {
                float mm = m;
                if constexpr (kF) {
#pragma unroll
                    for (int w = 1; w < kShortWarps; ++w) mm = fmaxf(mm, share[w][gl][EPV + 1]);
                    const float f = row_ex2((m - mm) * kRowLog2e);
                    l *= f;
#pragma unroll
                    for (int k = 0; k < EPV; ++k) y[k] *= f;
                }
#pragma unroll
                for (int w = 1; w < kShortWarps; ++w) {
                    const float *x = share[w][gl];
                    const float f = kF ? row_ex2((x[kF ? EPV + 1 : 0] - mm) * kRowLog2e) : 1.f;
                    if constexpr (kAcc) {
#pragma unroll
                        for (int k = 0; k < EPV; ++k) y[k] = fmaf(x[k], f, y[k]);
                    }
                    if constexpr (!kAgg) l = fmaf(x[kAcc ? EPV : 0], f, l);
                    if constexpr (kDot) dB += x[kAcc ? EPV + 1 : 1];
                    if constexpr (kD) dD += x[2];
                }
                m = mm;
            }
            __syncthreads();
            live = wid == 0;
        }
        if constexpr (kF) m = l == 0.f ? SAR_NEG_INF : m;
        if (!live || (FOLD && grp != 0)) return;
        if (seg) {
            float *part = a.sp.part + item.seg * a.sp.pstride;
            const long long rowf = (long long)a.H * a.vph * EPV;
            if constexpr (kAcc) {
                if (okv) store_elems<float, EPV>(part + (hc * a.vph + vc) * EPV, y, EPV, false);
            }
            if (head_lane) {
                if constexpr (kF) {
                    part[rowf + hc] = m;
                    part[rowf + a.H + hc] = l;
                } else if constexpr (kD) {
                    part[hc] = dD;
                    part[a.H + hc] = dB;
                    part[2 * a.H + hc] = l;
                } else if constexpr (kS) {
                    part[rowf + hc] = dB - l;
                }
            }
            return;
        }
        T *outp = reinterpret_cast<T *>(a.out) + row * (long long)HF + oel;
        if constexpr (MODE == kRowFwd) {
            const float inv = l > 0.f ? __fdividef(1.f, l) : 0.f;
#pragma unroll
            for (int k = 0; k < EPV; ++k) {
                y[k] *= inv;
                if (a.flags & SAR_RELU_OUT) y[k] = fmaxf(y[k], 0.f);
            }
            if (left > 0) store_elems<T, EPV>(outp, y, left, a.ragged);
            if (head_lane) {
                a.m_io[so] = m;
                a.d_io[so] = l;
            }
        } else if constexpr (MODE == kRowFwdPart) {
            if (n == 0 && !first && !last) return;   // nothing to add, nothing to write
            float *ap = a.acc + row * (long long)HF + oel;
            const float mn = fmaxf(pm, m);
            float pa[EPV];
#pragma unroll
            for (int k = 0; k < EPV; ++k) pa[k] = 0.f;
            if (!first && left > 0) load_elems<float, EPV>(ap, pa, left, a.ragged);
            const float fo = pm == mn ? 1.f : row_ex2((pm - mn) * kRowLog2e), fn = m == mn ? 1.f : row_ex2((m - mn) * kRowLog2e);
            const float dn = pd * fo + l * fn;
#pragma unroll
            for (int k = 0; k < EPV; ++k) y[k] = pa[k] * fo + y[k] * fn;
            if (left > 0 && (n > 0 || first) && (!last || (a.flags & SAR_KEEP_NUMERATOR))) store_elems<float, EPV>(ap, y, left, a.ragged);
            if (last) {
                const float inv = dn > 0.f ? __fdividef(1.f, dn) : 0.f;
#pragma unroll
                for (int k = 0; k < EPV; ++k) {
                    y[k] *= inv;
                    if (a.flags & SAR_RELU_OUT) y[k] = fmaxf(y[k], 0.f);
                }
                if (left > 0) store_elems<T, EPV>(outp, y, left, a.ragged);
            }
            if (head_lane && (n > 0 || first)) {
                a.m_io[so] = mn;
                a.d_io[so] = dn;
            }
        } else if constexpr (MODE == kRowDst) {
            if (head_lane) {
                a.dscal[so] = dB - dD * l;
                a.rec[so] = n > 0 ? make_float4(rs, rm, ri, dD) : make_float4(__ldg(a.el + so), __ldg(a.m + so), 0.f, 0.f);
            }
        } else if constexpr (MODE == kRowDstPart) {
            if (head_lane && (n > 0 || first)) a.dscal[so] = n > 0 ? pm + (dB - pd * l) : 0.f;
        } else if constexpr (kS) {
            if (left > 0) store_elems<T, EPV>(outp, y, left, a.ragged);
            if (head_lane) a.dscal[so] = dB - l;
        } else {
            const bool mean = (a.flags & SAR_MEAN) && last, mix = a.mix.x0 && last;
            if ((n == 0 && !first && !mean && !mix) || left <= 0) return;
            const float ds = a.dst_scale ? __ldg(a.dst_scale + row) : 1.f;
            float old[EPV];
#pragma unroll
            for (int k = 0; k < EPV; ++k) old[k] = 0.f;
            if (!first) load_elems<T, EPV>(outp, old, left, a.ragged);
            float inv = 1.f;
            if (mean) {
                const long long dg = a.deg[row];
                inv = dg > 0 ? 1.f / (float)dg : 0.f;
            }
#pragma unroll
            for (int k = 0; k < EPV; ++k) y[k] = (y[k] * ds + old[k]) * inv;
            if (mix) {
                load_elems<T, EPV>(reinterpret_cast<const T *>(a.mix.x0) + row * (long long)HF + oel, old, left, a.ragged);
                const float post = a.mix.post ? __ldg(a.mix.post + row) : 1.f;
#pragma unroll
                for (int k = 0; k < EPV; ++k) y[k] = (a.mix.keep * old[k] + a.mix.scale * y[k]) * post;
            }
            store_elems<T, EPV>(outp, y, left, a.ragged);
        }
    }

    // Where a row fills the warp: rows of more than a.R edges are taken by the warps of the block together, one after the other, unless that
    // takes longer than each warp with its own (a step per four edges, two to end a shared row); or the block's segment (a.wide).  A
    // function of its own that looks its rows up again: compiled into the kernel it took registers from the short rows and cost them up to 25 %.
    static __device__ __noinline__ void rest_of_block(const RowArgs &a) {
        __shared__ float share[kShortWarps][G][kShare];
        __shared__ ShortItem items[kShortWarps];
        const int wid = threadIdx.x >> 5;
        const ShortItem x = short_item<1, true>(a, blockIdx.x);
        if ((threadIdx.x & 31) == 0) items[wid] = x;
        __syncthreads();
        auto shared = [&](const ShortItem &y) { return y.seg < 0 && y.n > a.R; };
        bool own = false;
        int entries = a.wide && x.seg >= 0 ? 1 : kShortWarps;
        if (entries > 1) {
            int block_steps = 0, warp_steps = 0;
            for (int w = 0; w < kShortWarps; ++w) {
                const int steps = shared(items[w]) ? (items[w].n + U - 1) / U : 0;
                if (steps > 0) block_steps += (steps + kShortWarps - 1) / kShortWarps + 2;
                warp_steps = max(warp_steps, steps);
            }
            if (block_steps >= warp_steps) {
                own = shared(x);
                entries = 0;
            }
        }
        for (int at = own ? -1 : 0; at < entries; ++at) {
            const bool block = at >= 0;
            const ShortItem y = block ? items[at] : x;
            if (entries > 1 && !shared(y)) continue;
            process<true>(a, y, block ? wid * U : 0, (block ? kShortWarps : 1) * U, true, block ? share : nullptr);
        }
    }
};

// SHARE (where a row fills the warp): what the warps of a block share is left to rest_of_block.
template <typename T, int NV, int HP, int MODE, int MINB, bool SHARE>
__global__ void __launch_bounds__(kShortThreads, MINB) short_kernel(const __grid_constant__ RowArgs a) {
    after_predecessor();
    using Row = ShortRow<T, NV, HP, MODE>;
    const ShortItem x = short_item<Row::NG, SHARE>(a, blockIdx.x);
    const int most = SHARE ? a.R : Row::NG > 1 ? kShortEdges : 0x7fffffff;   // edges of a row that is one group's
    const bool alone = x.n >= 0 && x.n <= most;
    if (x.seg < 0) Row::template process<false>(a, alone ? x : ShortItem{x.row, x.p, 0, -1}, 0, Row::U, alone, nullptr);
    if constexpr (SHARE) {
        const bool wide = a.wide && x.seg >= 0;
        if (x.seg >= 0 && !wide) Row::template process<true>(a, x, 0, Row::U, true, nullptr);
        if (__syncthreads_or(wide || (x.seg < 0 && x.n > most))) Row::rest_of_block(a);
    } else {
        // segments, and rows of more edges, one after the other, the groups of the warp together
        const int lane = threadIdx.x & 31;
        unsigned rest = x.seg >= 0 ? 1u : Row::NG > 1 ? __ballot_sync(0xffffffffu, x.n > most && (lane & (Row::G - 1)) == 0) : 0u;
        while (rest) {
            const int from = __ffs(rest) - 1;
            rest &= rest - 1;
            const ShortItem y{__shfl_sync(0xffffffffu, x.row, from), __shfl_sync(0xffffffffu, x.p, from), __shfl_sync(0xffffffffu, x.n, from), x.seg};
            Row::template process<true>(a, y, lane / Row::G * Row::U, Row::NG * Row::U, true, nullptr);
        }
    }
}

}  // namespace sar
