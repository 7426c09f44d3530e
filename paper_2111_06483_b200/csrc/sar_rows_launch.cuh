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

template <typename T, int NV, int HP, int MODE>
static sar_status launch_short_kernel(RowArgs a, RowGeo g, long long nnz, cudaStream_t st) {
    constexpr int NG = 32 / NV;
    // 32 warps an SM at 64 registers; the backward passes over bf16 rows need 70 to 80 (24 warps, no spills)
    constexpr int MINB = sizeof(T) == 2 && (MODE == kRowSrc || MODE == kRowDst || MODE == kRowDstPart) ? 6 : 8;
    a.nnz = nnz;
    const long long warps = a.sp.n_seg + (a.n_rows + NG - 1) / NG;
    if (warps <= 0) return SAR_OK;
    const dim3 grid((unsigned)((warps * 32 + kShortThreads - 1) / kShortThreads), (unsigned)g.tiles);
    constexpr const char *name = MODE == kRowFwd || MODE == kRowFwdPart ? "gat_fwd_short" : MODE == kRowDst || MODE == kRowDstPart ? "gat_bwd_dst_short"
                                 : MODE == kRowSrc ? "gat_bwd_src_short" : "spmm_short";
    SAR_LAUNCH(name, st, launch(short_kernel<T, NV, HP, MODE, MINB>, grid, kShortThreads, 0, st, a));
    return sar_after_launch();
}

template <typename T, int MODE>
static sar_status dispatch_rows(const RowArgs &a, RowGeo g, long long nnz, const char *name, cudaStream_t st) {
#define SAR_ROW_CASE(NV_, HP_) \
    if (g.NV == NV_ && g.HP == HP_) { \
        if constexpr (NV_ <= 32) \
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
