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
// a row without any other has m = -inf and d = 0, like one without edges.  A row's arithmetic does not depend on the rows around it.
#pragma once

#include "sar_rows_kernel.cuh"

namespace sar {

constexpr int kShortThreads = 128;
constexpr int kShortEdges = 24;   // rows of more are shared by the groups of the warp

template <typename T, int NV, int HP, int MODE, int MINB>
__global__ void __launch_bounds__(kShortThreads, MINB) short_kernel(const RowArgs a) {
    after_predecessor();
    constexpr int EPV = Elem<T>::EPV, NP = EPV / 2, U = 4;
    constexpr int G = NV, NG = 32 / G, VPHP = NV / HP;
    constexpr bool kF = MODE == kRowFwd || MODE == kRowFwdPart, kD = MODE == kRowDst || MODE == kRowDstPart;
    constexpr bool kS = MODE == kRowSrc, kAgg = MODE == kRowSum || MODE == kRowSumW;
    constexpr bool kAcc = kF || kS || kAgg, kDot = kD || kS;
    constexpr unsigned kAll = 0xffffffffu;
    constexpr float kLowest = -3.402823466e38f;
    static_assert(NV <= 32, "one vector per lane");
    const int lane = threadIdx.x & 31, gl = lane & (G - 1), grp = lane / G;
    const long long warp = (long long)blockIdx.x * (kShortThreads / 32) + (threadIdx.x >> 5);
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

    // ---- which rows: one segment of a long row per warp, or one row per group ---------------------------------------------
    const bool seg = warp < a.sp.n_seg;
    long long row, p = 0;
    int n = -1;                         // edges; < 0: nothing to do
    if (seg) {
        int lo = 0, hi = a.sp.n_long;   // last lo with long_seg[lo] <= warp, 32 probes at a time
        while (hi - lo > 1) {
            const int step = (hi - lo + 31) >> 5;
            const int at = lo + lane * step;
            const bool ok = at < hi && __ldg(a.sp.long_seg + at) <= warp;
            lo += (__popc(__ballot_sync(kAll, ok)) - 1) * step;
            hi = min(hi, lo + step);
        }
        row = __ldg(a.sp.long_row + lo);
        p = __ldg(a.indptr + row) + (warp - __ldg(a.sp.long_seg + lo)) * a.sp.threshold;
        const long long rest = __ldg(a.indptr + row + 1) - p;
        n = (int)(rest < a.sp.threshold ? rest : a.sp.threshold);
    } else {
        row = (warp - a.sp.n_seg) * NG + grp;
        if (row < a.n_rows) {
            p = __ldg(a.indptr + row);
            const long long len = __ldg(a.indptr + row + 1) - p;
            if (a.sp.threshold <= 0 || len <= a.sp.threshold) n = (int)min(len, 0x7fffffffLL);   // else its segments are items of their own
        }
    }

    // One row (or segment) of n edges from position p on, every `step`-th four of them from the e0-th on.  fold: the groups of the warp share
    // it, group 0 writes.
    auto process = [&](long long row, long long p, int n, int e0, int step, bool fold, bool live) {
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
        if (fold) {
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
                if (off < VPHP || (fold && off >= G)) {
                    if constexpr (MODE == kRowDst) dD += __shfl_xor_sync(kAll, dD, off);
                    dB += __shfl_xor_sync(kAll, dB, off);
                }
            }
        }
        if constexpr (kF) m = l == 0.f ? SAR_NEG_INF : m;
        if (!live || (fold && grp != 0)) return;
        if (seg) {
            float *part = a.sp.part + warp * a.sp.pstride;
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
    };

    // short rows, one per group; then the others and segments, one after the other, the groups of the warp together
    const bool mine = !seg && n >= 0 && (NG == 1 || n <= kShortEdges);
    if (!seg) process(row, p, mine ? n : 0, 0, U, false, mine);
    if constexpr (NG > 1) {
        unsigned rest = seg ? 1u : __ballot_sync(kAll, n > kShortEdges && gl == 0);
        while (rest) {
            const int from = __ffs(rest) - 1;
            rest &= rest - 1;
            process(__shfl_sync(kAll, row, from), __shfl_sync(kAll, p, from), __shfl_sync(kAll, n, from), grp * U, NG * U, true, true);
        }
    } else if (seg) {
        process(row, p, n, 0, U, true, true);
    }
}

}  // namespace sar
