// Lean span kernel of the source-major whole-graph backward pass (internal): dfeat_j = sum_i alpha * gout_i and
// der_j = <feat_j, sum_i alpha g' gout_i> - sum_i alpha g' D_i over the CSC, alpha rebuilt from the destination
// records {el, m, 1/d, D} the destination-major pass left in the workspace.
//
// The plan is the one sar_lean_common.cuh describes (span of rows -> chunk -> stage-granular cp.async ring of the
// gathered gout rows, uniform control flow, padding by repetition, weights of a stage computed JUST BEFORE the stage
// is consumed): the 64-byte destination record of every position of a stage travels with the stage's rows (one
// 16-byte cp.async per lane and stage into a small record ring), and when the stage has landed each lane scores one
// (position, head) pair into a 256-byte weight block.  Nothing per chunk is staged except the row offsets, so a warp
// needs 7.5 KB of shared memory, no record is ever loaded into a register ahead of its use, and no lane waits for a
// gather inside a sweep.
// Preconditions (checked by the host): SAR_FIRST|SAR_LAST, slope >= 0, a long-row plan of the CSC with threshold <= CAP,
// fewer than 2^32 16-byte vectors in gout.
#pragma once

#include "sar_lean_common.cuh"

namespace sar {


template <int G, int V, int H, bool SEG, int CAP, int P, int NS>
struct LeanSrcLayout {
    static constexpr int EPW = 32 / G;
    static constexpr int ROWB = G * V * 16;
    static constexpr int STAGE = P * ROWB;
    static constexpr int MAXR = SEG ? 1 : kMaxSpanRows;
    static constexpr int POSMAX = ((CAP + MAXR * (EPW - 1) + 31) / 32) * 32;
    static constexpr int RCN = ((MAXR * H * 4 + 15) / 16) * 16;
    static constexpr int MASKW = POSMAX / EPW / 32 + 1;
    static constexpr int RECB = P * H * 16;                       // records of one stage
    static constexpr int WB = P * H * 4;                          // one weight plane of one stage
    static constexpr int ring = 0;
    static constexpr int rec = ring + NS * STAGE;
    static constexpr int w = rec + NS * RECB;                     // two planes
    static constexpr int offs = w + 2 * WB;
    static constexpr int prow = offs + POSMAX * 4;
    static constexpr int rc = prow + POSMAX;                      // er of the chunk's rows
    static constexpr int sout = rc + RCN;                         // der
    static constexpr int srb = sout + RCN;
    static constexpr int sso = srb + ((MAXR + 1) * 4 + 15) / 16 * 16;
    static constexpr int endm = sso + ((MAXR + 1) * 4 + 15) / 16 * 16;
    static constexpr int total = endm + ((MASKW * 4 + 15) / 16) * 16;
};

template <typename T, int G, int V, int H, bool SEG, int CAP, int P, int NS>
__device__ __forceinline__ void lean_src_warp(const LeanSrcArgs a, long long item) {
    using L = LeanSrcLayout<G, V, H, SEG, CAP, P, NS>;
    constexpr int EPV = Elem<T>::EPV, NP = EPV / 2;
    constexpr int EPW = L::EPW, ROWB = L::ROWB, STAGE = L::STAGE;
    constexpr int NVEC = G * V, VPH = NVEC / H;
    constexpr int LGNVEC = NVEC == 16 ? 4 : (NVEC == 32 ? 5 : 6);
    constexpr int SPS = P / EPW;                   // slots per stage
    constexpr int ITEMS = P * H;                   // (position, head) pairs of a stage
    static_assert(H % 4 == 0 && NVEC % H == 0 && VPH <= G && (VPH & (VPH - 1)) == 0, "head geometry");
    static_assert((1 << LGNVEC) == NVEC, "row geometry");
    static_assert(P <= 32 && 32 % P == 0 && (SPS == 4 || SPS == 8), "stage geometry: four or eight slots per stage");
    static_assert(ITEMS <= 64, "at most two (position, head) pairs per lane");
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const unsigned sbase = (unsigned)__cvta_generic_to_shared(smem_raw);
    const unsigned ring_s = sbase + L::ring, rec_s = sbase + L::rec, w_s = sbase + L::w, offs_s = sbase + L::offs;
    const unsigned prow_s = sbase + L::prow, rc_s = sbase + L::rc, sout_s = sbase + L::sout, endm_s = sbase + L::endm;
    int *srb = reinterpret_cast<int *>(smem_raw + L::srb);
    int *sso = reinterpret_cast<int *>(smem_raw + L::sso);

    const int lane = threadIdx.x;
    const int gl = lane & (G - 1), half = lane / G;
    auto perm = [](int q) { return (q / P) * P + ((q % P) % EPW) * SPS + (q % P) / EPW; };

    // ---- which rows ---------------------------------------------------------------------------
    long long row0, eb = 0, ee = 0;
    int nrows;
    bool excluded = false;
    long long seg = -1;
    if constexpr (!SEG) {
        row0 = item * a.R;
        if (row0 >= a.n_rows) return;
        nrows = (int)((a.n_rows - row0) < a.R ? (a.n_rows - row0) : a.R);
        long long p = 0;
        if (lane <= nrows) p = __ldg(a.indptr + row0 + lane);
        const long long pn = __shfl_down_sync(0xffffffffu, p, 1);
        if (lane < nrows) {
            eb = p;
            ee = pn;
            excluded = ee - eb > a.sp.threshold;
        }
    } else {
        int lo = 0, hi = a.sp.n_long;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (__ldg(a.sp.long_seg + mid) <= item) lo = mid; else hi = mid;
        }
        row0 = __ldg(a.sp.long_row + lo);
        nrows = 1;
        seg = item;
        if (lane == 0) {
            const long long c = item - __ldg(a.sp.long_seg + lo);
            const long long rb_ = __ldg(a.indptr + row0), re_ = __ldg(a.indptr + row0 + 1);
            eb = rb_ + c * a.sp.threshold;
            ee = eb + a.sp.threshold < re_ ? eb + a.sp.threshold : re_;
        }
    }

    // ---- lane geometry ------------------------------------------------------------------------
    int hv[V];
#pragma unroll
    for (int v = 0; v < V; ++v) hv[v] = (v * G + gl) / VPH;
    unsigned long long gbase_v[V];
#pragma unroll
    for (int v = 0; v < V; ++v) gbase_v[v] = reinterpret_cast<unsigned long long>(reinterpret_cast<const uint4 *>(a.gather) + gl + v * G);
    const unsigned ring_l = ring_s + (unsigned)(half * ROWB + gl * 16);
    // the (position, head) pairs this lane copies the record of and scores: it = lane (+ 32)
    constexpr int NIT = (ITEMS + 31) / 32;

    f32x2 pacc0[V][NP], pacc1[V][NP];
    float sv[V];
    uint4 rvq[V], rvq_next[V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
        sv[v] = 0.f;
#pragma unroll
        for (int k = 0; k < NP; ++k) pacc0[v][k] = pacc1[v][k] = zero2();
        rvq[v] = rvq_next[v] = make_uint4(0u, 0u, 0u, 0u);
    }
    auto request_rowvec = [&](long long row_, uint4 (&dst)[V]) {
        const uint4 *rp = reinterpret_cast<const uint4 *>(a.rowvec) + row_ * NVEC + gl;
#pragma unroll
        for (int v = 0; v < V; ++v) dst[v] = __ldg(rp + v * G);
    };

    const int deg_l = (lane < nrows && !excluded) ? (int)(ee - eb) : 0;
    const unsigned excl_all = __ballot_sync(0xffffffffu, excluded);

    int r = 0;
    while (r < nrows) {
        if ((excl_all >> r) & 1u) {
            ++r;
            continue;
        }
        // ---- choose the chunk: rows [r, r2), none excluded, at most CAP edges in all ----------------
        int r2, ne;
        const long long cb = __shfl_sync(0xffffffffu, eb, r);
        if constexpr (SEG) {
            r2 = 1;
            ne = __shfl_sync(0xffffffffu, deg_l, 0);
        } else {
            int pre = (lane >= r && lane < nrows) ? deg_l : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, pre, o);
                if (lane >= o) pre += t;
            }
            const unsigned later = excl_all & ~((1u << r) - 1u);
            const int stop = later ? __ffs(later) - 1 : nrows;
            const unsigned fits = __ballot_sync(0xffffffffu, lane >= r && lane < stop && pre <= CAP);
            r2 = r + __popc(fits);
            ne = __shfl_sync(0xffffffffu, pre, r2 - 1);
        }
        const int nr = r2 - r;

        // ---- stage A: row tables, row-end mask, non-empty rows -----------------------------------------
        unsigned nemask;
        int nslots;
        {
            const int i = lane - r;
            const bool mine = i >= 0 && i < nr;
            int ns = 0;
            if (mine) {
                srb[i] = (int)(eb - cb);
                if (i == nr - 1) srb[nr] = ne;
                ns = (deg_l + EPW - 1) / EPW;
            }
            int inc = ns;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += t;
            }
            if (mine) sso[i] = inc - ns;
            if (i == nr - 1) sso[nr] = inc;
            nslots = (int)__reduce_add_sync(0xffffffffu, (unsigned)ns);
            nemask = __ballot_sync(0xffffffffu, mine && ns > 0) >> r;
            if constexpr (!SEG) {
                if (lane < L::MASKW) sts_u32(endm_s + 4 * lane, 0u);
                __syncwarp();
                if (mine && ns > 0) atomicOr(reinterpret_cast<unsigned *>(smem_raw + L::endm) + ((inc - 1) >> 5), 1u << ((inc - 1) & 31));
            }
        }
        __syncwarp();
        const int npos = nslots * EPW;
        const int nstages = (npos + P - 1) / P;

        // ---- stage B: row offsets of the columns (padding and the fill of the last stage repeat a real column and
        // are marked so that they weigh nothing), position -> row, the rows' own score terms ------------------------
        {
            int i = 0;
            for (int q0 = 0; q0 < nstages * P; q0 += 64) {
                int c[2] = {0, 0}, pr[2] = {0x80, 0x80};
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int q = q0 + 32 * u + lane;
                    if (q < npos) {
                        if constexpr (!SEG) {
                            while (q >= sso[i + 1] * EPW) ++i;
                        }
                        const int t = srb[i] + (q - sso[i] * EPW);
                        const int last = srb[i + 1] - 1;
                        const bool pad = t > last;
                        c[u] = ld_stream_i32(a.indices + cb + (pad ? last : t));
                        pr[u] = i | (pad ? 0x80 : 0);
                    } else if (q < nstages * P) {
                        c[u] = ld_stream_i32(a.indices + cb + (ne - 1));
                    }
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int q = q0 + 32 * u + lane;
                    if (q < nstages * P) {
                        sts_u32(offs_s + 4 * (unsigned)perm(q), (unsigned)c[u] << LGNVEC);
                        sts_u8(prow_s + q, (unsigned)pr[u]);
                    }
                }
            }
            for (int x = lane; x < nr * H; x += 32) {
                sts_f32(rc_s + 4 * x, __ldg(a.er + (row0 + r) * H + x));
                sts_f32(sout_s + 4 * x, 0.f);
            }
        }
        __syncwarp();

        // ---- the ring: the gathered rows of a stage and the destination records of its positions, one commit group
        // per stage ------------------------------------------------------------------------------------------------
        auto issue_stage = [&](int j) {
            const unsigned dst = ring_l + (unsigned)((j % NS) * STAGE);
            const unsigned ob = offs_s + (unsigned)((j * P + half * SPS) * 4);
#pragma unroll
            for (int kq = 0; kq < SPS; kq += 4) {
                const uint4 o4 = lds128(ob + kq * 4);
                const unsigned ov[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
                for (int t = 0; t < 4; ++t)
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        unsigned long long src;
                        asm("mad.wide.u32 %0, %1, 16, %2;\n" : "=l"(src) : "r"(ov[t]), "l"(gbase_v[v]));
                        cp_async16_full(dst + (unsigned)((kq + t) * EPW * ROWB + v * G * 16), reinterpret_cast<const void *>(src));
                    }
            }
#pragma unroll
            for (int n = 0; n < NIT; ++n) {
                const int it = lane + 32 * n;
                if (ITEMS % 32 == 0 || it < ITEMS) {
                    const int p = it / H, h = it % H;
                    const unsigned col = lds_u32(offs_s + 4 * (unsigned)perm(j * P + p)) >> LGNVEC;
                    cp_async16_full(rec_s + (unsigned)((j % NS) * L::RECB + it * 16), a.rec_in + (size_t)col * H + h);
                }
            }
        };
#pragma unroll
        for (int j = 0; j < NS; ++j) {
            if (j < nstages) issue_stage(j);
            cp_async_commit();
        }

        // rows without edges: dfeat = 0 (der leaves with the others at the chunk's end)
        if constexpr (!SEG) {
            unsigned em = ~nemask & ((1u << nr) - 1u);
            while (em) {
                const int i = __ffs(em) - 1;
                em &= em - 1;
                uint4 *rp = reinterpret_cast<uint4 *>(a.out) + (row0 + r + i) * NVEC;
                for (int x = lane; x < NVEC; x += 32) rp[x] = make_uint4(0u, 0u, 0u, 0u);
            }
        }
        if (nslots > 0) request_rowvec(row0 + r + (SEG ? 0 : __ffs(nemask) - 1), rvq_next);

        // ---- the stages ------------------------------------------------------------------------------------------
        {
            int s = 0;
            int ri = SEG ? 0 : (__ffs(nemask) - 1);
            for (int j = 0; j < nstages; ++j) {
                cp_async_wait<NS - 1>();
                __syncwarp();   // the records of this stage were copied by other lanes; the previous weights are consumed
                // -- weights of this stage: one (position, head) pair per lane --
#pragma unroll
                for (int n = 0; n < NIT; ++n) {
                    const int it = lane + 32 * n;
                    if (ITEMS % 32 == 0 || it < ITEMS) {
                        const int p = it / H, h = it % H;
                        const unsigned pr = lds_u8(prow_s + (unsigned)(j * P + p));
                        const int i = SEG ? 0 : (int)(pr & 0x7f);
                        const float4 rec = lds_f4(rec_s + (unsigned)((j % NS) * L::RECB + it * 16));
                        const float s_ = rec.x + lds_f32(rc_s + (unsigned)((i * H + h) * 4));
                        float gr;
                        const float e = leaky(s_, a.slope, gr);
                        const float al = ex2_approx((e - rec.y) * kLog2e) * rec.z;
                        float w0 = s_ > 0.f ? al : -al;   // the sign bit carries LeakyReLU' = slope
                        float w1 = al * gr * rec.w;
                        if (pr & 0x80) w0 = w1 = 0.f;
                        const unsigned wi = (unsigned)((((p % EPW) * H + h) * SPS + p / EPW) * 4);
                        sts_f32(w_s + wi, w0);
                        sts_f32(w_s + L::WB + wi, w1);
                    }
                }
                __syncwarp();
                const unsigned ring_a = ring_l + (unsigned)((j % NS) * STAGE);
                const int cnt = nslots - s;
                unsigned ends;
                if constexpr (SEG) {
                    ends = cnt <= SPS ? (1u << (cnt - 1)) : 0u;
                } else {
                    unsigned bit = 0;
                    if (lane < SPS) {
                        const int sl = s + lane;
                        bit = (lds_u32(endm_s + 4 * (unsigned)(sl >> 5)) >> (sl & 31)) & 1u;
                    }
                    ends = __ballot_sync(0xffffffffu, bit != 0);
                }
                float4 w4[V], u4[V];
#pragma unroll
                for (int k = 0; k < SPS; ++k) {
                    if (k % 4 == 0) {
#pragma unroll
                        for (int v = 0; v < V; ++v) {
                            w4[v] = lds_f4(w_s + (unsigned)(((half * H + hv[v]) * SPS + k) * 4));
                            u4[v] = lds_f4(w_s + L::WB + (unsigned)(((half * H + hv[v]) * SPS + k) * 4));
                        }
                    }
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        const float wk = k % 4 == 0 ? w4[v].x : k % 4 == 1 ? w4[v].y : k % 4 == 2 ? w4[v].z : w4[v].w;
                        const float uk = k % 4 == 0 ? u4[v].x : k % 4 == 1 ? u4[v].y : k % 4 == 2 ? u4[v].z : u4[v].w;
                        f32x2 x[NP];
                        Pairs<T>::get(lds128(ring_a + (unsigned)(k * EPW * ROWB + v * G * 16)), x);
                        const float al = fabsf(wk);
                        const float wg = wk < 0.f ? al * a.slope : al;   // alpha * LeakyReLU'
                        sv[v] += uk;
                        const f32x2 a2 = pack2(al, al), g2 = pack2(wg, wg);
#pragma unroll
                        for (int t = 0; t < NP; ++t) {
                            pacc0[v][t] = fma2(a2, x[t], pacc0[v][t]);
                            pacc1[v][t] = fma2(g2, x[t], pacc1[v][t]);
                        }
                    }
                    if (ends & (1u << k)) {
                        // ---- the row is complete -------------------------------------------------------------
                        const long long row = row0 + r + ri;
#pragma unroll
                        for (int v = 0; v < V; ++v) rvq[v] = rvq_next[v];
                        if constexpr (!SEG) {
                            const unsigned rest = nemask & ~((2u << ri) - 1u);
                            if (rest) request_rowvec(row0 + r + (__ffs(rest) - 1), rvq_next);
                        }
                        float acc0[V][EPV];
#pragma unroll
                        for (int v = 0; v < V; ++v)
#pragma unroll
                            for (int t = 0; t < NP; ++t) unpack2(pacc0[v][t], acc0[v][2 * t], acc0[v][2 * t + 1]);
                        {
                            // <feat_j, C> on the un-folded accumulator, reduced over the lanes of each head and the edge lanes
                            float pC[V];
#pragma unroll
                            for (int v = 0; v < V; ++v) {
                                f32x2 rv[NP];
                                Pairs<T>::get(rvq[v], rv);
                                f32x2 qc = zero2();
#pragma unroll
                                for (int t = 0; t < NP; ++t) qc = fma2(rv[t], pacc1[v][t], qc);
                                pC[v] = qc.x + qc.y;
                            }
#pragma unroll
                            for (int off = 1; off < 32; off <<= 1) {
                                if (off < VPH || off >= G) {
#pragma unroll
                                    for (int v = 0; v < V; ++v) {
                                        pC[v] += __shfl_xor_sync(0xffffffffu, pC[v], off);
                                        if (off >= G) sv[v] += __shfl_xor_sync(0xffffffffu, sv[v], off);
                                    }
                                }
                            }
#pragma unroll
                            for (int off = G; off < 32; off <<= 1)
#pragma unroll
                                for (int v = 0; v < V; ++v)
#pragma unroll
                                    for (int e = 0; e < EPV; ++e) acc0[v][e] += __shfl_xor_sync(0xffffffffu, acc0[v][e], off);
                            if constexpr (SEG) {   // the segment's share of dfeat (float32) and of der, for the merge launch
                                if (half == 0) {
                                    constexpr long long rowf = (long long)NVEC * EPV;
                                    float *rec = a.sp.part + seg * a.sp.pstride;
                                    bool vok[V];
#pragma unroll
                                    for (int v = 0; v < V; ++v) vok[v] = true;
                                    store_acc_row<G, V, EPV>(rec, gl, vok, acc0);
#pragma unroll
                                    for (int v = 0; v < V; ++v)
                                        if ((gl % VPH) == 0) rec[rowf + hv[v]] = pC[v] - sv[v];
                                }
                            } else
                            if (half == 0) {
                                uint4 *rp = reinterpret_cast<uint4 *>(a.out) + row * NVEC + gl;
#pragma unroll
                                for (int v = 0; v < V; ++v) {
                                    rp[v * G] = Elem<T>::pack(acc0[v]);
                                    if ((gl % VPH) == 0) sts_f32(sout_s + (unsigned)((ri * H + hv[v]) * 4), pC[v] - sv[v]);   // der
                                }
                            }
                        }
#pragma unroll
                        for (int v = 0; v < V; ++v) {
                            sv[v] = 0.f;
#pragma unroll
                            for (int t = 0; t < NP; ++t) pacc0[v][t] = pacc1[v][t] = zero2();
                        }
                        if constexpr (!SEG) {
                            const unsigned rest = nemask & ~((2u << ri) - 1u);
                            ri = rest ? __ffs(rest) - 1 : nr;
                        }
                        if (k + 1 >= cnt) goto chunk_done;
                    }
                }
                s += SPS;
                if (j + NS < nstages) issue_stage(j + NS);
                cp_async_commit();
            }
        chunk_done:
            cp_async_wait<0>();
        }

        // ---- the chunk's der, coalesced ----------------------------------------------------------------------------
        if constexpr (!SEG) {
            __syncwarp();
            for (int x = lane; x < nr * H; x += 32) a.der[(row0 + r) * H + x] = lds_f32(sout_s + 4 * x);
            __syncwarp();
        }
        r = r2;
    }
}

template <typename T, int G, int V, int H, int CAP, int P, int NS, int MINB, int ITEMS>
__global__ void __launch_bounds__(32, MINB) lean_src_kernel(const LeanSrcArgs a) {
    after_predecessor();
    const long long item = blockIdx.x;
    if (ITEMS == kLeanSegments || (ITEMS == kLeanBoth && item < a.sp.n_seg)) lean_src_warp<T, G, V, H, true, CAP, P, NS>(a, item);
    else lean_src_warp<T, G, V, H, false, CAP, P, NS>(a, ITEMS == kLeanBoth ? item - a.sp.n_seg : item);
}

// ---- launcher ------------------------------------------------------------------------------------------------------
template <typename T, int G, int V, int H>
static sar_status launch_lean_src(LeanSrcArgs a, long long nnz, cudaStream_t st) {
    constexpr int NS = 2;
    constexpr int P = (G == 32 && V == 1) ? 8 : 4 * (32 / G);   // stages of 2 KB (4 KB for rows of 512 bytes and more)
    using LR = LeanSrcLayout<G, V, H, false, kLeanCap, P, NS>;
    using LS = LeanSrcLayout<G, V, H, true, kLeanCap, P, NS>;
    a.R = lean_rows_per_span(a.n_rows, nnz, kLeanCap);
    return launch_lean<LR, LS>("gat_bwd_src", "gat_bwd_src_seg", lean_src_kernel<T, G, V, H, kLeanCap, P, NS, kLeanMinBlocksBwdRows, kLeanBoth>,
                               lean_src_kernel<T, G, V, H, kLeanCap, P, NS, kLeanMinBlocks, kLeanSegments>,
                               lean_src_kernel<T, G, V, H, kLeanCap, P, NS, kLeanMinBlocksBwdRows, kLeanRows>, a, st);
}

template <typename T>
static sar_status dispatch_lean_src(const Shape &s, const LeanSrcArgs &a, long long nnz, cudaStream_t st) {
    if (s.G == 16 && s.V == 1 && s.geom.H == 4) return launch_lean_src<T, 16, 1, 4>(a, nnz, st);
    if (s.G == 32 && s.V == 1 && s.geom.H == 4) return launch_lean_src<T, 32, 1, 4>(a, nnz, st);
    if (s.G == 32 && s.V == 1 && s.geom.H == 8) return launch_lean_src<T, 32, 1, 8>(a, nnz, st);
    if (s.G == 32 && s.V == 2 && s.geom.H == 4) return launch_lean_src<T, 32, 2, 4>(a, nnz, st);
    return SAR_ERR_UNSUPPORTED;
}

}  // namespace sar

#define SAR_LEAN_SRC_TU(SUFFIX, TYPE)                                                                        \
    namespace sar {                                                                                          \
    sar_status lean_bwd_src_##SUFFIX(const Shape &s, const LeanSrcArgs &a, long long nnz, cudaStream_t st) { \
        return dispatch_lean_src<TYPE>(s, a, nnz, st);                                                       \
    }                                                                                                        \
    }
