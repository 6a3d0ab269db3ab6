// vgr_tiletest.cuh -- tile-level preemptive alpha test (paper Sec. 4.2,
// Eq. 4, moved to binning), in explicitly rounded operations.
#pragma once

#include "vgr_internal.cuh"

namespace vgr {

// rho = -1/2 (a dx^2 + c dy^2) - b dx dy
__device__ __forceinline__ float rho_rn(float a, float b, float c, float dx, float dy) {
    const float t1 = __fmul_rn(__fmul_rn(a, dx), dx);
    const float t2 = __fmul_rn(__fmul_rn(c, dy), dy);
    const float t3 = __fmul_rn(__fmul_rn(b, dx), dy);
    return __fsub_rn(__fmul_rn(-0.5f, __fadd_rn(t1, t2)), t3);
}

__device__ __forceinline__ float clampf(float x, float lo, float hi) { return fminf(fmaxf(x, lo), hi); }

// Keep the pair when the maximum of rho over the rectangle spanned by the
// tile's pixel centres reaches thre (= ln alpha* - ln theta - slack).  The
// maximum is 0 when the mean lies inside; otherwise it is on an edge that faces
// the mean (rho rises on the way from any point towards the mean, which leaves
// the rectangle through one), where rho is a concave quadratic in the free
// coordinate: on x = x0 or x1 its optimum is dy* = (-b/c) dx = ry dx, on y = y0 or
// y1 it is dx* = (-b/a) dy = rx dy, each clamped to the edge.  At most one edge
// of each pair faces the mean.
// T is the tile side in pixels (8, 16 or 32): every coordinate below is exact in FP32.
__device__ __forceinline__ bool tile_keep(float u, float v, float a, float b, float c, float rx, float ry, float thre,
                                          int tx, int ty, float W, float H, int T) {
    const float x0 = (float)(tx * T) + 0.5f;
    const float x1 = fminf((float)(tx * T) + ((float)T - 0.5f), W - 0.5f);
    const float y0 = (float)(ty * T) + 0.5f;
    const float y1 = fminf((float)(ty * T) + ((float)T - 0.5f), H - 0.5f);
    if (u >= x0 && u <= x1 && v >= y0 && v <= y1) return thre <= 0.f;
    const float dy_lo = __fsub_rn(y0, v), dy_hi = __fsub_rn(y1, v);
    const float dx_lo = __fsub_rn(x0, u), dx_hi = __fsub_rn(x1, u);
    const float dx = u < x0 ? dx_lo : dx_hi, dy = v < y0 ? dy_lo : dy_hi;
    const float rx_best = rho_rn(a, b, c, dx, clampf(__fmul_rn(ry, dx), dy_lo, dy_hi));
    const float ry_best = rho_rn(a, b, c, clampf(__fmul_rn(rx, dy), dx_lo, dx_hi), dy);
    return ((u < x0 || u > x1) && rx_best >= thre) || ((v < y0 || v > y1) && ry_best >= thre);
}

}  // namespace vgr
