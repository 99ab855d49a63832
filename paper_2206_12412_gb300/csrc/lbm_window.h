// lbm_window.h -- the near end of the K window (eq. r(v)) in FP32, and how far
// it may lie from r0 / (1 - v).  Plain C++, so that the bound can be compared
// with FP64 on the host.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define LBM_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define LBM_HOST_DEVICE inline
#endif

namespace lbm {

// r0 / (1 - v) in FP32 (r0 rounded already).
LBM_HOST_DEVICE float window_start(float r0, double v) { return r0 / (1.0f - (float)v); }

// Bound on its distance from r0 / (1 - v) where it lies below lo_max <= kWindowLo, r0
// >= kWindowR0 (the crack step's exact form elsewhere), in units of 2^-32 (grid
// spacings where dh = 1).  v is off by 2^-25 after its rounding, which 1 / (1 - v) =
// lo / r0 magnifies; r0, 1 - v and the division add 2^-24 each, relative.  The
// bound doubles the sum: 32-bit numbers, 4.4e4 at r0 = 2, speeds up to 0.85.
constexpr float kWindowR0 = 1e-3f, kWindowLo = 24.0f;
LBM_HOST_DEVICE int32_t window_slack(float r0, float lo_max)
{
    return (int32_t)(lo_max * (lo_max * (256.0f / r0) + 1536.0f)) + 4;
}

}  // namespace lbm
