// Row kernel (internal): the aggregation's gather passes - forward, destination-major and source-major backward, sum -
// for every shape whose heads (for a sum: columns) fit tiles of at most 256 16-byte vectors.
//
// A warp takes one row after the other (R consecutive ones, or one segment of a long row) and a row 32 edges at a time.
// Lanes play two parts:
//   * edge lanes: one edge each.  A lane loads the score terms of its edge's column and forms the weights of all heads;
//     the weights go to shared memory (and nothing else does).
//   * gather lanes: G lanes x 16 bytes cover a gathered row, 32/G edges per SLOT.  U slots are loaded straight into
//     registers before the first is accumulated.  What a lane holds per row is one vector of float32 sums (forward,
//     source-major) or three numbers (destination-major).
//
// What bounds it: latency, then issue slots.  The L2 is not what a gather out of it waits for (36 % of its throughput in the
// two-head case below), but a short row is a chain of dependent loads: row pointers, column ids, rows.  So a warp keeps
// no stage and no ring, and 32 of them fit an SM with 64 registers a thread (25 are there on average); the
// row pointers of a warp's rows are one load, the column ids of the next 32 edges are asked for before the present ones
// are used, and the score terms, the row's own data and the first U slots are all in flight together.  A row of up to
// U slots costs one memory latency, which the other warps hide.  Measured, before (a warp staging 256 edges in shared
// memory) and now: 233,000 nodes, 11.6 million edges, 2 heads of 64, bf16, forward 554 -> 408 us (7.3 TB/s of gathered
// rows, 23 instructions per edge, issue slots 68 % busy); 20,000 nodes, 400,000 edges, 1 head of 64, float32, 4 partition
// steps forward and backward 497 -> 274 us; 2,000 nodes, 22,000 edges, 4 heads of 16, one pass 15 -> 5 us.
// 64 registers are not enough for every pass.  The sums and the forward pass of one head in float32 spill nothing; the other
// passes of one or two heads 8 to 150 bytes a thread (0.3 to 6 % of the instructions they issue), tiles of four heads 60
// to 200 (64 vectors of bf16: 116 to 372), of eight heads 90 to 560, and there the span kernels take over (takes_span in
// sar_gat.cu).
//
// Forward: the softmax is taken against the exact maximum of the row's scores among 32 edges (one `redux` per head); a
// row of more carries the running-max correction of Sec. 3.4.
// Destination-major: D = sum alpha <gout, feat_j> and sum alpha g' <gout, feat_j> are linear in the dot products, so a
// lane adds up alpha times its own 16 bytes' share of <gout, feat_j> and the lanes of a head are reduced once per row.
// Source-major: dfeat = sum alpha gout_i; der = sum alpha g' (<feat_j, gout_i> - D_i), the dot product likewise.
#pragma once

#include "sar_device.cuh"
#include "sar_launch.cuh"
#include "sar_rows.cuh"

namespace sar {

constexpr int kRowWarps = 4;   // independent warps per block (no block-wide step)

__device__ __forceinline__ float row_ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float redux_max(float x) {
    float y;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;\n" : "=f"(y) : "f"(x));
    return y;
}
constexpr float kRowLog2e = 1.4426950408889634f;

// Floats of shared memory per (edge, head): forward alpha; destination-major alpha, alpha g'; source-major also alpha g' D.
template <int MODE>
struct RowW {
    static constexpr int n = MODE == kRowSrc ? 4 : (MODE == kRowDst || MODE == kRowDstPart) ? 2 : 1;
};
template <int HP, int MODE>
struct RowSmem {
    static constexpr int total = (MODE == kRowSum || MODE == kRowSumW) ? 0 : 32 * HP * RowW<MODE>::n;   // floats per warp
};

__device__ __forceinline__ uint4 row_lds128(unsigned addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ float2 row_lds64(unsigned addr) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ unsigned row_lds32(unsigned addr) {
    unsigned v;
    asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(v) : "r"(addr));
    return v;
}

// HP per-head scalars of one row / column starting at head 0 of the tile; heads beyond `have` repeat the last one
template <int HP>
__device__ __forceinline__ void load_heads(const float *p, int have, int hvec, float (&x)[HP]) {
    if (HP % 4 == 0 && hvec) {
#pragma unroll
        for (int q = 0; q < HP / 4; ++q) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(p) + q);
            x[4 * q] = v.x;
            x[(4 * q + 1) % HP] = v.y;
            x[(4 * q + 2) % HP] = v.z;
            x[(4 * q + 3) % HP] = v.w;
        }
    } else if (HP == 2 && hvec) {
        const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
        x[0] = v.x;
        x[HP - 1] = v.y;
    } else {
#pragma unroll
        for (int h = 0; h < HP; ++h) x[h] = __ldg(p + (h < have ? h : have - 1));
    }
}

// n consecutive elements of type T held as floats -> memory (aligned to n elements, or element by element)
template <typename T, int N>
__device__ __forceinline__ void store_elems(T *p, const float (&x)[N], int n, bool ragged) {
    if (!ragged) {
        if constexpr (sizeof(T) == 4) {
            if constexpr (N % 4 == 0) {
#pragma unroll
                for (int q = 0; q < N / 4; ++q)
                    reinterpret_cast<float4 *>(p)[q] = make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
            } else if constexpr (N == 2) *reinterpret_cast<float2 *>(p) = make_float2(x[0], x[1]);
            else *reinterpret_cast<float *>(p) = x[0];
        } else {
            if constexpr (N == 8) *reinterpret_cast<uint4 *>(p) = Elem<__nv_bfloat16>::pack(x);
            else if constexpr (N == 4) *reinterpret_cast<uint2 *>(p) = make_uint2(Elem<__nv_bfloat16>::pack2(x[0], x[1]), Elem<__nv_bfloat16>::pack2(x[2], x[3]));
            else if constexpr (N == 2) *reinterpret_cast<uint32_t *>(p) = Elem<__nv_bfloat16>::pack2(x[0], x[1]);
            else *p = __float2bfloat16_rn(x[0]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (k < n) Elem<T>::store1(p + k, x[k]);
    }
}
// the inverse, plain loads (arrays the launch also writes)
template <typename T, int N>
__device__ __forceinline__ void load_elems(const T *p, float (&x)[N], int n, bool ragged) {
    if (!ragged && sizeof(T) == 4 && N % 4 == 0) {
#pragma unroll
        for (int q = 0; q < N / 4; ++q) {
            const float4 v = reinterpret_cast<const float4 *>(p)[q];
            x[4 * q] = v.x;
            x[(4 * q + 1) % N] = v.y;
            x[(4 * q + 2) % N] = v.z;
            x[(4 * q + 3) % N] = v.w;
        }
    } else if (!ragged && sizeof(T) == 2 && N == 8) {
        float y[8];
        Elem<__nv_bfloat16>::unpack(*reinterpret_cast<const uint4 *>(p), y);
#pragma unroll
        for (int k = 0; k < N; ++k) x[k] = y[k % 8];
    } else {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            x[k] = 0.f;
            if (!ragged || k < n) {
                if constexpr (sizeof(T) == 4) x[k] = p[k];
                else x[k] = __bfloat162float(p[k]);
            }
        }
    }
}

// Sum over the 32/G edge groups of the lanes' vectors, by halving: at each step a lane hands over the half of its
// elements that it will not keep (4 + 2 + ... shuffles instead of EPV per step).  Leaves N elements, in x[0 .. N).
template <int G, int EPV, int N>
__device__ __forceinline__ void fold_groups(float (&x)[EPV], float (&y)[N], int lane) {
#pragma unroll
    for (int off = 16, n = EPV; off >= G; off >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = lane & off;
#pragma unroll
            for (int k = 0; k < n; ++k) {
                const float send = up ? x[k] : x[k + n], keep = up ? x[k + n] : x[k];
                x[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
            }
        } else {
            x[0] += __shfl_xor_sync(0xffffffffu, x[0], off);
        }
    }
#pragma unroll
    for (int k = 0; k < N; ++k) y[k] = x[k];
}

// x[h] for a head that is known per lane only
template <int HP>
__device__ __forceinline__ float pick_head(const float (&x)[HP], int h) {
    float r = x[0];
#pragma unroll
    for (int k = 1; k < HP; ++k) r = h == k ? x[k] : r;
    return r;
}

template <typename T, int NV, int HP, int MODE, int MINB>
__global__ void __launch_bounds__(kRowWarps * 32, MINB) row_kernel(const RowArgs a) {
    constexpr int EPV = Elem<T>::EPV, NP = EPV / 2;
    constexpr int G = NV < 32 ? NV : 32, V = NV / G, E = 32 / G;   // lanes per row, vectors per lane, edges per slot
    constexpr int VPHP = NV / HP;                                  // lanes (x vectors) per head
    constexpr int U = V == 1 ? 4 : V == 2 ? 2 : 1;   // slots in flight (8 and 4: 5-20 % slower for the warps they cost)
    constexpr int NE = EPV / E > 0 ? EPV / E : 1;                  // elements a lane holds after the fold over the edge groups
    constexpr bool kF = MODE == kRowFwd || MODE == kRowFwdPart, kD = MODE == kRowDst || MODE == kRowDstPart;
    constexpr bool kS = MODE == kRowSrc, kAgg = MODE == kRowSum || MODE == kRowSumW;
    constexpr bool kPart = MODE == kRowFwdPart || MODE == kRowDstPart;
    constexpr bool kAcc = kF || kS || kAgg;                        // a vector is accumulated
    constexpr bool kDot = kD || kS;                                // dot products with the row-stationary vector
    constexpr int WN = RowW<MODE>::n;
    after_predecessor();
    extern __shared__ __align__(16) float smem_f[];
    const int lane = threadIdx.x & 31;
    float *sw = smem_f + (threadIdx.x >> 5) * RowSmem<HP, MODE>::total;
    const long long item = (long long)blockIdx.x * kRowWarps + (threadIdx.x >> 5);
    const int h0 = kAgg ? 0 : (int)blockIdx.y * HP;
    const int have = a.H - h0;                                     // heads from h0 on
    const int tvec = kAgg ? (int)blockIdx.y * NV : 0;              // first vector of a sum's column tile

    // ---- which rows: one segment of a long row, or R consecutive rows -----------------------------------------------
    long long row0, p0 = 0;    // first row; where its edges begin
    unsigned ptr = 0;          // lane r: where row r's edges begin, counted from p0
    int nrows;
    const bool seg = item < a.sp.n_seg;
    if (seg) {
        int lo = 0, hi = a.sp.n_long;   // last lo with long_seg[lo] <= item, 32 probes at a time
        while (hi - lo > 1) {
            const int step = (hi - lo + 31) >> 5;
            const int at = lo + lane * step;
            const bool ok = at < hi && __ldg(a.sp.long_seg + at) <= item;
            lo += (__popc(__ballot_sync(0xffffffffu, ok)) - 1) * step;
            hi = min(hi, lo + step);
        }
        row0 = __ldg(a.sp.long_row + lo);
        nrows = 1;
        const long long rb = __ldg(a.indptr + row0), re = __ldg(a.indptr + row0 + 1);
        p0 = rb + (item - __ldg(a.sp.long_seg + lo)) * a.sp.threshold;
        ptr = lane == 0 ? 0u : (unsigned)(re - p0 < a.sp.threshold ? re - p0 : a.sp.threshold);
    } else {
        row0 = (item - a.sp.n_seg) * a.R;
        if (row0 >= a.n_rows) return;
        nrows = (int)(a.n_rows - row0 < a.R ? a.n_rows - row0 : a.R);
        const long long p = __ldg(a.indptr + row0 + (lane < nrows ? lane : nrows));
        p0 = __shfl_sync(0xffffffffu, p, 0);
        ptr = (unsigned)(p - p0);
    }
    const int32_t *idx = a.indices + p0;
    const unsigned avail = (unsigned)(a.nnz - p0 < 0xffffffffLL ? a.nnz - p0 : 0xffffffffLL);
    // an inconsistent graph gives wrong sums, not a wrong address
    auto column = [&](unsigned at) { return min((unsigned)ld_stream_i32(idx + min(at, avail - 1u)), a.last_col); };

    // ---- lane geometry --------------------------------------------------------------------------------------------
    const int gl = lane & (G - 1), half = lane / G;
    int hv[V], oel[V], orem[V];                 // head within the tile, first element in a row of `out`, elements left
    unsigned long long gb[V];                   // address of the lane's vector in row 0 of the gathered array
    bool okv[V];
    int eo = 0;                                 // element within the vector that the fold leaves to this lane
    bool mine = true;                           // ... unless another lane holds the same one
#pragma unroll
    for (int off = 16, n = EPV; off >= G; off >>= 1) {
        if (n > 1) {
            n >>= 1;
            if (lane & off) eo += n;
        } else if (lane & off) {
            mine = false;
        }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int idx = v * G + gl, head = idx / VPHP, vec = idx % VPHP + tvec;
        const int hc = head < have ? head : have - 1, vc = vec < a.vph ? vec : a.vph - 1;
        hv[v] = head;
        okv[v] = head < have && vec < a.vph;
        gb[v] = reinterpret_cast<unsigned long long>(a.gather) + ((unsigned long long)(h0 + hc) * a.vph + vc) * 16u;
        oel[v] = (h0 + hc) * a.F + vec * EPV + eo;
        orem[v] = (okv[v] && mine) ? a.F - (vec * EPV + eo) : 0;
    }
    auto gofs = [&](int v) { return gb[v] - reinterpret_cast<unsigned long long>(a.gather); };   // ... within a row
    const unsigned HF = (unsigned)(a.H * a.F);
    T *outp = reinterpret_cast<T *>(a.out);
    const unsigned w_l = (unsigned)__cvta_generic_to_shared(sw) + half * HP * WN * 4;
    const bool first = a.flags & SAR_FIRST, last = a.flags & SAR_LAST;
    const unsigned limit = seg || a.sp.threshold <= 0 ? 0xffffffffu : (unsigned)a.sp.threshold;

    unsigned colN = 0, atN = 0xffffffffu;   // column ids asked for ahead: those of the 32 edges from atN on
    for (int r = 0; r < nrows; ++r) {
        const unsigned beg = __shfl_sync(0xffffffffu, ptr, r), end = __shfl_sync(0xffffffffu, ptr, r + 1);
        if (end - beg > limit) continue;    // a long row: its segments are items of their own
        if (beg == end) {                   // nothing to add: only what a flag forces to be written
            if (MODE == kRowFwdPart && !first && !last) continue;
            if (MODE == kRowDstPart && !first) continue;
            if (kAgg && !first && !(((a.flags & SAR_MEAN) || a.mix.x0) && last)) continue;
        }
        const long long row = row0 + r;

        f32x2 acc[V][NP];      // kAcc: float32 sums of the lane's vector
        f32x2 pin[V][NP];      // sum: the sum of up to eight slots, added to acc after them (shorter chains of additions)
        f32x2 go[V][NP];       // kDot: row-stationary vector
        f32x2 d2[V], b2[V];    // kDot: this lane's share of sum alpha <.,.> and of sum alpha g' <.,.>
        float sv[V];           // forward: sum alpha; backward: sum alpha g' (D)
        float mc[HP];          // forward: the row's maximum so far
#pragma unroll
        for (int v = 0; v < V; ++v) {
            sv[v] = 0.f;
            d2[v] = b2[v] = zero2();
#pragma unroll
            for (int k = 0; k < NP; ++k) acc[v][k] = pin[v][k] = zero2();
        }
#pragma unroll
        for (int h = 0; h < HP; ++h) mc[h] = SAR_NEG_INF;
        auto flush = [&]() {
            if constexpr (kAgg) {
#pragma unroll
                for (int v = 0; v < V; ++v)
#pragma unroll
                    for (int k = 0; k < NP; ++k) {
                        acc[v][k] = fma2(pin[v][k], pack2(1.f, 1.f), acc[v][k]);
                        pin[v][k] = zero2();
                    }
            }
        };

        // the row's own data: in flight with everything else
        uint4 rv[V];
        float rs[HP], rm[HP], ri[HP];   // el (er); destination-major: m, 1/d
        if constexpr (kDot) {
#pragma unroll
            for (int v = 0; v < V; ++v) rv[v] = __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<unsigned long long>(a.rowvec) + (unsigned long long)row * a.row_bytes + gofs(v)));
        }
        if constexpr (!kAgg) load_heads<HP>((kS ? a.er : a.el) + row * a.H + h0, have, a.hvec, rs);
        if constexpr (kD) {
            load_heads<HP>(a.m + row * a.H + h0, have, a.hvec, rm);
            load_heads<HP>(a.d + row * a.H + h0, have, a.hvec, ri);
        }
        float pm[V], pd[V], pa[V][NE];
        if constexpr (MODE == kRowFwdPart) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                pm[v] = SAR_NEG_INF;
                pd[v] = 0.f;
#pragma unroll
                for (int k = 0; k < NE; ++k) pa[v][k] = 0.f;
                if (!seg && !first && orem[v] > 0) {
                    pm[v] = a.m_io[row * a.H + h0 + hv[v]];
                    pd[v] = a.d_io[row * a.H + h0 + hv[v]];
                    load_elems<float, NE>(a.acc + row * (long long)HF + oel[v], pa[v], orem[v], a.ragged);
                }
            }
        }
        if constexpr (MODE == kRowDstPart) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                pm[v] = pd[v] = 0.f;
                if (!seg && okv[v]) {
                    const long long o = row * a.H + h0 + hv[v];
                    pd[v] = a.rec[o].w;
                    if (!first) pm[v] = a.dscal[o];
                }
            }
        }

        for (unsigned base = beg; base < end; base += 32) {
            const int nb = (int)min(32u, end - base);
            const unsigned col = atN == base ? colN : column(min(base + lane, end - 1u));   // lanes past the row repeat its last edge
            const int slots = (nb + E - 1) / E;
            // -- edge lanes ask for their score terms, gather lanes for the first U slots --
            float x[HP];
            float4 rc[kS ? HP : 1];
            float wcol = 1.f;
            if constexpr (kF || kD) load_heads<HP>(a.er + (long long)col * a.H + h0, have, a.hvec, x);
            if constexpr (kS) {
#pragma unroll
                for (int h = 0; h < HP; ++h) rc[h] = __ldg(a.rec + (long long)col * a.H + h0 + (h < have ? h : have - 1));
            }
            if constexpr (MODE == kRowSumW) wcol = __ldg(a.src_scale + col);
            uint4 xv[U][V];
            auto load_slots = [&](int s, bool all) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (all || s + u < slots) {
                        const unsigned c = __shfl_sync(0xffffffffu, col, (s + u) * E + half);
#pragma unroll
                        for (int v = 0; v < V; ++v) xv[u][v] = __ldg(reinterpret_cast<const uint4 *>(gb[v] + (unsigned long long)c * a.row_bytes));
                    }
                }
            };
            load_slots(0, false);
            // the column ids of the next 32 edges: this row's, or the next row's
            atN = base + 32 < end ? base + 32 : end;
            {
                const unsigned stop = base + 32 < end ? end : __shfl_sync(0xffffffffu, ptr, r + 2 <= nrows ? r + 2 : nrows);
                if (atN < stop) colN = column(min(atN + lane, stop - 1u));
                else atN = 0xffffffffu;
            }

            // -- edge lanes: the weights of all heads --
            if constexpr (kF) {
                float f[HP];   // how far the sums so far move with the maximum
#pragma unroll
                for (int h = 0; h < HP; ++h) {
                    float gr;
                    x[h] = leaky(rs[h] + x[h], a.slope, gr);
                    const float mx = fmaxf(redux_max(x[h]), mc[h]);
                    f[h] = mc[h];
                    mc[h] = mx;
                    x[h] = lane < nb ? row_ex2((x[h] - mx) * kRowLog2e) : 0.f;
                }
                if (base != beg) {
#pragma unroll
                    for (int h = 0; h < HP; ++h) f[h] = f[h] == mc[h] ? 1.f : row_ex2((f[h] - mc[h]) * kRowLog2e);
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        const float fv = pick_head<HP>(f, hv[v]);
                        sv[v] *= fv;
#pragma unroll
                        for (int k = 0; k < NP; ++k) acc[v][k] = fma2(acc[v][k], pack2(fv, fv), zero2());
                    }
                }
                if constexpr (HP % 4 == 0) {
#pragma unroll
                    for (int q = 0; q < HP / 4; ++q)
                        reinterpret_cast<float4 *>(sw + lane * HP)[q] = make_float4(x[4 * q], x[(4 * q + 1) % HP], x[(4 * q + 2) % HP], x[(4 * q + 3) % HP]);
                } else if constexpr (HP == 2) {
                    *reinterpret_cast<float2 *>(sw + lane * HP) = make_float2(x[0], x[HP - 1]);
                } else {
                    sw[lane] = x[0];
                }
            } else if constexpr (kD) {
#pragma unroll
                for (int h = 0; h < HP; ++h) {
                    if (base == beg) ri[h] = ri[h] > 0.f ? __fdividef(1.f, ri[h]) : 0.f;
                    float gr;
                    const float s = leaky(rs[h] + x[h], a.slope, gr);
                    const float al = lane < nb ? row_ex2((s - rm[h]) * kRowLog2e) * ri[h] : 0.f;
                    *reinterpret_cast<float2 *>(sw + (lane * HP + h) * 2) = make_float2(al, al * gr);
                }
            } else if constexpr (kS) {
#pragma unroll
                for (int h = 0; h < HP; ++h) {
                    float gr;
                    const float s = leaky(rc[h].x + rs[h], a.slope, gr);
                    const float al = lane < nb ? row_ex2((s - rc[h].y) * kRowLog2e) * rc[h].z : 0.f;
                    *reinterpret_cast<float4 *>(sw + (lane * HP + h) * 4) = make_float4(al, al * gr, al * gr * rc[h].w, 0.f);
                }
            }
            if constexpr (!kAgg) __syncwarp();
            if constexpr (kDot) {
                if (base == beg) {
#pragma unroll
                    for (int v = 0; v < V; ++v) Pairs<T>::get(okv[v] ? rv[v] : make_uint4(0u, 0u, 0u, 0u), go[v]);   // a lane beyond the head repeats its last vector
                }
            }

            // -- gather lanes --
            unsigned wa = w_l;
            auto add_slots = [&](int s, bool all) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (all || s + u < slots) {
                        float wsum = 1.f;
                        if (MODE == kRowSumW) wsum = __shfl_sync(0xffffffffu, wcol, (s + u) * E + half);
                        // a sum's last slot may be short of edges: nothing is added for them (zero times the last edge's row is no zero if
                        // that holds an infinity)
                        const bool there = !kAgg || E == 1 || (s + u) * E + half < nb;
#pragma unroll
                        for (int v = 0; v < V; ++v) {
                            f32x2 y[NP];
                            Pairs<T>::get(xv[u][v], y);
                            const unsigned wv = wa + hv[v] * WN * 4 + u * E * HP * WN * 4;
                            if constexpr (kF || kAgg) {
                                float w = wsum;
                                if constexpr (kF) w = __uint_as_float(row_lds32(wv));
                                const f32x2 w2 = pack2(w, w);
                                if constexpr (kF) {
                                    sv[v] += w;
#pragma unroll
                                    for (int k = 0; k < NP; ++k) acc[v][k] = fma2(y[k], w2, acc[v][k]);
                                } else {
#pragma unroll
                                    for (int k = 0; k < NP; ++k)
                                        if (there) pin[v][k] = fma2(y[k], w2, pin[v][k]);
                                }
                            } else {
                                float al, ag, agd = 0.f;
                                if constexpr (kD) {
                                    const float2 w = row_lds64(wv);
                                    al = w.x;
                                    ag = w.y;
                                } else {
                                    const uint4 w = row_lds128(wv);
                                    al = __uint_as_float(w.x);
                                    ag = __uint_as_float(w.y);
                                    agd = __uint_as_float(w.z);
                                }
                                f32x2 dot = fma2(y[0], go[v][0], zero2());
#pragma unroll
                                for (int k = 1; k < NP; ++k) dot = fma2(y[k], go[v][k], dot);
                                b2[v] = fma2(dot, pack2(ag, ag), b2[v]);
                                if constexpr (kD) {
                                    if constexpr (MODE == kRowDst) d2[v] = fma2(dot, pack2(al, al), d2[v]);
                                    sv[v] += ag;
                                } else {
                                    sv[v] += agd;
                                    const f32x2 a2 = pack2(al, al);
#pragma unroll
                                    for (int k = 0; k < NP; ++k) acc[v][k] = fma2(y[k], a2, acc[v][k]);
                                }
                            }
                        }
                    }
                }
                wa += U * E * HP * WN * 4;
            };
            int s = 0;
            while (s + U <= slots) {
                add_slots(s, true);
                s += U;
                if (kAgg && (s & 7) == 0) flush();
                if (s + U <= slots) load_slots(s, true);
                else load_slots(s, false);
            }
            if (s < slots) add_slots(s, false);
            flush();
            if constexpr (!kAgg) __syncwarp();   // the weights are consumed
        }

        {   // ---- the row (or segment) is complete ----------------------------------------------------------------------
        float *part = a.sp.part + item * a.sp.pstride;
        const long long rowf = (long long)a.H * a.vph * EPV;   // floats of a segment's vector part
        float y[V][NE];
        if constexpr (kAcc) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                float xx[EPV];
#pragma unroll
                for (int k = 0; k < NP; ++k) {
                    xx[2 * k] = acc[v][k].x;
                    xx[2 * k + 1] = acc[v][k].y;
                }
                fold_groups<G, EPV, NE>(xx, y[v], lane);
            }
        }
        if constexpr (!kAgg) {
#pragma unroll
            for (int off = 16; off >= G; off >>= 1)
#pragma unroll
                for (int v = 0; v < V; ++v) sv[v] += __shfl_xor_sync(0xffffffffu, sv[v], off);
        }
        float dD[V], dB[V];   // dot products of the lane's head
        if constexpr (kDot) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                dD[v] = d2[v].x + d2[v].y;
                dB[v] = b2[v].x + b2[v].y;
            }
            if constexpr (VPHP > 32) {   // one head over several vectors of a lane
#pragma unroll
                for (int v = 1; v < V; ++v) {
                    dD[0] += dD[v];
                    dB[0] += dB[v];
                }
            }
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                if (off < VPHP || off >= G) {
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        if constexpr (MODE == kRowDst) dD[v] += __shfl_xor_sync(0xffffffffu, dD[v], off);
                        dB[v] += __shfl_xor_sync(0xffffffffu, dB[v], off);
                    }
                }
            }
        }
        if (seg) {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                if constexpr (kAcc) {
                    if (okv[v] && mine) store_elems<float, NE>(part + gofs(v) / 16 * EPV + eo, y[v], NE, false);
                }
                if (half == 0 && okv[v] && (v * G + gl) % VPHP == 0) {
                    if constexpr (kF) {
                        part[rowf + h0 + hv[v]] = pick_head<HP>(mc, hv[v]);
                        part[rowf + a.H + h0 + hv[v]] = sv[v];
                    }
                    if constexpr (kD) {
                        part[h0 + hv[v]] = dD[v];
                        part[a.H + h0 + hv[v]] = dB[v];
                        part[2 * a.H + h0 + hv[v]] = sv[v];
                    }
                    if constexpr (kS) part[rowf + h0 + hv[v]] = dB[v] - sv[v];
                }
            }
        } else {
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const bool head_lane = half == 0 && okv[v] && (v * G + gl) % VPHP == 0;
                const long long o = row * a.H + h0 + hv[v];
                if constexpr (MODE == kRowFwd) {
                    const float inv = sv[v] > 0.f ? __fdividef(1.f, sv[v]) : 0.f;
#pragma unroll
                    for (int k = 0; k < NE; ++k) {
                        y[v][k] *= inv;
                        if (a.flags & SAR_RELU_OUT) y[v][k] = fmaxf(y[v][k], 0.f);
                    }
                    if (orem[v] > 0) store_elems<T, NE>(outp + row * (long long)HF + oel[v], y[v], orem[v], a.ragged);
                    if (head_lane) {
                            a.m_io[o] = pick_head<HP>(mc, hv[v]);
                            a.d_io[o] = sv[v];
                        }
                } else if constexpr (MODE == kRowFwdPart) {
                    const float mk = pick_head<HP>(mc, hv[v]);
                    const float mn = fmaxf(pm[v], mk);
                    const float fo = pm[v] == mn ? 1.f : row_ex2((pm[v] - mn) * kRowLog2e);
                    const float fn = mk == mn ? 1.f : row_ex2((mk - mn) * kRowLog2e);
                    const float dn = pd[v] * fo + sv[v] * fn;
#pragma unroll
                    for (int k = 0; k < NE; ++k) y[v][k] = pa[v][k] * fo + y[v][k] * fn;
                    const bool last = a.flags & SAR_LAST;
                    if (orem[v] > 0 && (!last || (a.flags & SAR_KEEP_NUMERATOR)))
                        store_elems<float, NE>(a.acc + row * (long long)HF + oel[v], y[v], orem[v], a.ragged);
                    if (last) {
                        const float inv = dn > 0.f ? __fdividef(1.f, dn) : 0.f;
#pragma unroll
                        for (int k = 0; k < NE; ++k) {
                            y[v][k] *= inv;
                            if (a.flags & SAR_RELU_OUT) y[v][k] = fmaxf(y[v][k], 0.f);
                        }
                        if (orem[v] > 0) store_elems<T, NE>(outp + row * (long long)HF + oel[v], y[v], orem[v], a.ragged);
                    }
                    __syncwarp();   // every lane has read the state's m and d
                    if (head_lane) {
                        a.m_io[o] = mn;
                        a.d_io[o] = dn;
                    }
                } else if constexpr (MODE == kRowDst) {
                    if (head_lane) {
                        a.dscal[o] = dB[v] - dD[v] * sv[v];
                        const float iv = pick_head<HP>(ri, hv[v]);   // (without edges: still d)
                        a.rec[o] = make_float4(pick_head<HP>(rs, hv[v]), pick_head<HP>(rm, hv[v]), beg == end ? 0.f : iv, dD[v]);
                    }
                } else if constexpr (MODE == kRowDstPart) {
                    if (head_lane) a.dscal[o] = pm[v] + (dB[v] - pd[v] * sv[v]);
                } else if constexpr (kS) {
                    if (orem[v] > 0) store_elems<T, NE>(outp + row * (long long)HF + oel[v], y[v], orem[v], a.ragged);
                    if (head_lane) a.dscal[o] = dB[v] - sv[v];
                } else {
                    if (orem[v] > 0) {
                        const float ds = a.dst_scale ? __ldg(a.dst_scale + row) : 1.f;
                        float old[NE];
#pragma unroll
                        for (int k = 0; k < NE; ++k) old[k] = 0.f;
                        if (!(a.flags & SAR_FIRST)) load_elems<T, NE>(outp + row * (long long)HF + oel[v], old, orem[v], a.ragged);
                        float inv = 1.f;
                        if ((a.flags & SAR_MEAN) && (a.flags & SAR_LAST)) {
                            const long long dg = a.deg[row];
                            inv = dg > 0 ? 1.f / (float)dg : 0.f;
                        }
#pragma unroll
                        for (int k = 0; k < NE; ++k) y[v][k] = (y[v][k] * ds + old[k]) * inv;
                        if (a.mix.x0 && last) {
                            load_elems<T, NE>(reinterpret_cast<const T *>(a.mix.x0) + row * (long long)HF + oel[v], old, orem[v], a.ragged);
                            const float post = a.mix.post ? __ldg(a.mix.post + row) : 1.f;
#pragma unroll
                            for (int k = 0; k < NE; ++k) y[v][k] = (a.mix.keep * old[k] + a.mix.scale * y[v][k]) * post;
                        }
                        store_elems<T, NE>(outp + row * (long long)HF + oel[v], y[v], orem[v], a.ragged);
                    }
                }
            }
        }
        }
    }
}

}  // namespace sar
