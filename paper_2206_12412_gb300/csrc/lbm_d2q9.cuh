// lbm_d2q9.cuh -- the arithmetic that every D2Q9 update shares.
#pragma once

#include "lbm_internal.cuh"

namespace lbm {

// The rate and integration of one D2Q9 site, with every rounding fixed:
// wdot' = wdot + (g_a axis + g_d diag) as fma(g_a, axis, g_d diag) and
// w' = fma(dt, wdot', w).  The sum of two products could otherwise be
// contracted into an FMA either way round, and a compiler may choose
// differently in different code paths (the bare, interior and edge-row
// updates); fixed here, every path -- and so every band partition and every
// row-slab split -- gives the same bits.
__device__ __forceinline__ float d9_rate(float wd, float axis, float diag, float ga, float gd)
{
    return __fadd_rn(wd, __fmaf_rn(ga, axis, __fmul_rn(gd, diag)));
}
__device__ __forceinline__ double d9_rate(double wd, double axis, double diag, double ga, double gd)
{
    return __dadd_rn(wd, __fma_rn(ga, axis, __dmul_rn(gd, diag)));
}
__device__ __forceinline__ float d9_integrate(float w, float wd, float dt) { return __fmaf_rn(dt, wd, w); }
__device__ __forceinline__ double d9_integrate(double w, double wd, double dt) { return __fma_rn(dt, wd, w); }

// Twice the Dirichlet value of each edge, selected without indexing (so that
// it stays in registers).
template <typename T>
struct TwoWs {
    T l, r, b, t;
    __device__ __forceinline__ T operator[](int e) const { return e == LEFT ? l : (e == RIGHT ? r : (e == BOTTOM ? b : t)); }
};

// The value a link streams back when it leaves the body (ox: across the
// left / right edge, oy: across the bottom / top edge; dx, dy its direction):
// anti-bounce-back 2 w* - w on a Dirichlet edge, bounce-back w otherwise; a
// link through a corner follows the Dirichlet edge if just one of the two is
// Dirichlet, else the bottom / top edge.
template <typename T>
__device__ __forceinline__ T leaving(const int32_t *edge, const TwoWs<T> &two_ws, bool ox, bool oy, int dx, int dy, T w0)
{
    const int ex = dx < 0 ? LEFT : RIGHT, ey = dy < 0 ? BOTTOM : TOP;
    int e = ox ? ex : ey;
    if (ox && oy) e = (edge[ex] == EDGE_DIRICHLET && edge[ey] != EDGE_DIRICHLET) ? ex : ey;
    return edge[e] == EDGE_DIRICHLET ? two_ws[e] - w0 : w0;
}

}  // namespace lbm
