// Diagonal-block solve of many rows in one launch (internal header; panel_kernel.cuh).
#pragma once
#include "common.cuh"

namespace gb {

// Largest block: X of a CTA's right-hand sides stays in shared memory.
template <typename T>
constexpr int kPanelRows = sizeof(T) == 8 ? 512 : 1024;

// FP32: the right-hand sides from which a lane holds one of them (512 rows:
// 2048 right-hand sides 93 us with eight per CTA, 115 with one per lane; 8192 265
// with sixteen per CTA and 138, now 104).
constexpr int64_t kWideColumns = 2432;

// Solve Mv[r0:r0+nr, r0:r0+nr] X = alpha Bv[r0:r0+nr, :] in place, nr <=
// kPanelRows<T>, each CTA with CW right-hand sides.
template <typename T, int CW>
int launch_panel_cw(const Canon<T> &c, int64_t r0, int nr, T alpha);

// The same with 32 right-hand sides per CTA, one per lane (panel_wide.cu).
int launch_panel_wide(const Canon<float> &c, int64_t r0, int nr, float alpha);

template <typename T>
int launch_panel_solve(const Canon<T> &c, int64_t r0, int nr, T alpha)
{
    if (nr <= 0 || c.ncols <= 0) return 0;
    if (nr > kPanelRows<T>) return GB_STATUS_CUDA_ERROR;
    if constexpr (sizeof(T) == 8) {
        // as few right-hand sides per CTA as fill two CTAs of every SM
        if (c.ncols <= 304) return launch_panel_cw<T, 1>(c, r0, nr, alpha);
        if (c.ncols <= 608) return launch_panel_cw<T, 2>(c, r0, nr, alpha);
        if (c.ncols <= 1216) return launch_panel_cw<T, 4>(c, r0, nr, alpha);
        return launch_panel_cw<T, 8>(c, r0, nr, alpha);
    } else {
        // (not below four: every CTA streams the whole triangle from L2)
        if (c.ncols <= 1216) return launch_panel_cw<T, 4>(c, r0, nr, alpha);
        if (c.ncols <= kWideColumns) return launch_panel_cw<T, 8>(c, r0, nr, alpha);
        return launch_panel_wide(c, r0, nr, alpha);
    }
}

}  // namespace gb
