// Launch of the row kernels (internal): grid, rows per warp, and the instantiation that fits a geometry.
#pragma once

#include "sar_dispatch.cuh"
#include "sar_rows_kernel.cuh"
#include "sar_short_kernel.cuh"

namespace sar {

constexpr int kRowSMs = 148;

// Rows a warp takes: several, so that their row pointers are one load and the next row's column ids can be asked for a
// row ahead, but no more than leaves every SM kRowFill warps.
constexpr int kRowMax = 8, kRowFill = 64;
static inline int rows_per_warp(long long n_rows) {
    const long long R = n_rows / (kRowSMs * kRowFill);
    return R < 1 ? 1 : R > kRowMax ? kRowMax : (int)R;
}

template <typename T, int NV, int HP, int MODE>
static sar_status launch_row_kernel(RowArgs a, RowGeo g, long long nnz, const char *name, cudaStream_t st) {
    constexpr int MINB = NV >= 256 ? 2 : NV == 128 ? 4 : (NV == 64 || HP == 8) ? 7 : 8;
    // 32 warps per SM at 64 registers (28 at 72 for 64 vectors or eight heads).  7 and 10 blocks were 2 and 10 % slower for two
    // heads of 64, bf16, forward, where 8 spill 16 bytes; passes that spill more were not tried apart.
    a.nnz = nnz;
    a.R = rows_per_warp(a.n_rows);
    const long long items = a.sp.n_seg + (a.n_rows + a.R - 1) / a.R;
    if (items <= 0) return SAR_OK;
    constexpr size_t smem = (size_t)kRowWarps * RowSmem<HP, MODE>::total * 4;
    auto kern = row_kernel<T, NV, HP, MODE, MINB>;
    SAR_TRY(ensure_smem(kern, smem));
    const dim3 grid((unsigned)((items + kRowWarps - 1) / kRowWarps), (unsigned)g.tiles);
    SAR_LAUNCH(name, st, launch(kern, grid, kRowWarps * 32, smem, st, a));
    return sar_after_launch();
}

constexpr long long kShortBlock = 96, kShortFew = 4 * 32 * kRowSMs;   // edges (64: 0.79 to 1.0 of the speed with rows of 60); rows: four waves
template <typename T, int NV, int HP, int MODE>
static sar_status launch_short_kernel(RowArgs a, RowGeo g, long long nnz, cudaStream_t st) {
    constexpr int NG = 32 / NV;
    if (a.n_rows <= 0) return SAR_OK;   // a partition without sources
    // 32 warps an SM at 64 registers; the backward passes over bf16 rows need 70 and more (24 warps at 80)
    constexpr int MINB = sizeof(T) == 2 && (MODE == kRowSrc || MODE == kRowDst || MODE == kRowDstPart) ? 6 : 8;
    a.nnz = nnz;
    constexpr const char *name = MODE == kRowFwd || MODE == kRowFwdPart ? "gat_fwd_short" : MODE == kRowDst || MODE == kRowDstPart ? "gat_bwd_dst_short"
                                 : MODE == kRowSrc ? "gat_bwd_src_short" : "spmm_short";
    auto go = [&](auto kernel) {
        const long long warps = (a.wide ? a.sp.n_seg * kShortWarps : a.sp.n_seg) + (a.n_rows + NG - 1) / NG;
        SAR_LAUNCH(name, st, launch(kernel, dim3((unsigned)((warps + kShortWarps - 1) / kShortWarps), (unsigned)g.tiles), kShortThreads, 0, st, a));
        return sar_after_launch();
    };
    if constexpr (NG == 1) {
        // A long row is a chain of steps, and where a row fills the warp that chain decides how long a launch of few rows takes: there
        // rows much longer than the others are shared by the warps of a block, and so are segments where a block for each fits the chip
        // at once.  Times without over with it, backward, rows of 240 to 256 edges among ones of 2 to 20: 1.1 to 1.8; without such rows
        // 0.91 to 1.0, and with ones of 40 to 100 0.88 to 1.05, so that launches of more rows, which hide the chain, go without.
        a.wide = a.sp.n_seg > 0 && a.sp.n_seg * g.tiles <= kRowSMs * MINB;
        if (a.n_rows * g.tiles <= (a.wide ? 2 : 1) * kShortFew) {
            a.R = (int)(3 * nnz < kShortBlock * a.n_rows ? kShortBlock : 3 * nnz / a.n_rows);
            return go(short_kernel<T, NV, HP, MODE, MINB, true>);
        }
    }
    a.wide = 0;
    return go(short_kernel<T, NV, HP, MODE, MINB, false>);
}

template <int MODE>
constexpr bool has_short(int NV, int HP) {
    return MODE == kRowSum || MODE == kRowSumW ? sum_short_edges(NV, 0) > 0 : short_edges(NV, HP, MODE != kRowFwd && MODE != kRowFwdPart, 0) > 0;
}

template <typename T, int MODE>
static sar_status dispatch_rows(const RowArgs &a, RowGeo g, long long nnz, const char *name, cudaStream_t st) {
#define SAR_ROW_CASE(NV_, HP_) \
    if (g.NV == NV_ && g.HP == HP_) { \
        if constexpr (has_short<MODE>(NV_, HP_)) \
            if (a.lone) return launch_short_kernel<T, NV_, HP_, MODE>(a, g, nnz, st); \
        return launch_row_kernel<T, NV_, HP_, MODE>(a, g, nnz, name, st); \
    }
    SAR_ROW_CASE(4, 1) SAR_ROW_CASE(8, 1) SAR_ROW_CASE(16, 1) SAR_ROW_CASE(32, 1) SAR_ROW_CASE(64, 1)
    SAR_ROW_CASE(128, 1) SAR_ROW_CASE(256, 1)
    if constexpr (MODE != kRowSum && MODE != kRowSumW) {
        SAR_ROW_CASE(4, 2) SAR_ROW_CASE(8, 2) SAR_ROW_CASE(16, 2) SAR_ROW_CASE(32, 2) SAR_ROW_CASE(64, 2)
        SAR_ROW_CASE(4, 4) SAR_ROW_CASE(8, 4) SAR_ROW_CASE(16, 4) SAR_ROW_CASE(32, 4) SAR_ROW_CASE(64, 4)
        SAR_ROW_CASE(8, 8) SAR_ROW_CASE(16, 8) SAR_ROW_CASE(32, 8) SAR_ROW_CASE(64, 8)
    }
#undef SAR_ROW_CASE
    return SAR_ERR_UNSUPPORTED;
}

}  // namespace sar
