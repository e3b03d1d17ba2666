// Device helpers shared by the TMA-staged 3D kernels (kernels3d_tma.cu,
// kernels3d_x2.cu): the central-difference weights as compile-time constants.
//
// The weights are the unscaled Taylor weights of orders 8 (R = 4) and 10
// (R = 5), second derivative w2[1..R] and first derivative w1[1..R]; with a
// compile-time j they fold into immediate operands of the multiply-adds, so
// the per-axis sums need no constant loads.  The 1/h^2 (1/h) factor of an
// axis is applied once to that axis's sum.
#pragma once

namespace fwi {

template <int R>
__device__ __forceinline__ constexpr float w2c(int j) {
  return R == 4 ? (j == 1 ? 8.0f / 5.0f : j == 2 ? -1.0f / 5.0f : j == 3 ? 8.0f / 315.0f
                                                                         : -1.0f / 560.0f)
                : (j == 1 ? 5.0f / 3.0f : j == 2 ? -5.0f / 21.0f : j == 3 ? 5.0f / 126.0f
                   : j == 4 ? -5.0f / 1008.0f : 1.0f / 3150.0f);
}

// w2c with the third weight one unit in the last place further (order 10; order 8: nearer
// zero): the rounding errors of the weights then cancel in sum j^2 w2[j] = 1, and the
// second derivative of a smooth wave is off by under 6e-9 for k h <= 0.5 where the nearest
// weights are off by 3.3e-8 (order 8: 1.5e-8), which a run of many steps adds up as phase.
template <int R>
__device__ __forceinline__ constexpr float w2s(int j) {
  return j == 3 ? (R == 4 ? 0x1.a01ap-6f : 0x1.451454p-5f) : w2c<R>(j);
}

template <int R>
__device__ __forceinline__ constexpr float w1c(int j) {
  return R == 4 ? (j == 1 ? 4.0f / 5.0f : j == 2 ? -1.0f / 5.0f : j == 3 ? 4.0f / 105.0f
                                                                         : -1.0f / 280.0f)
                : (j == 1 ? 5.0f / 6.0f : j == 2 ? -5.0f / 21.0f : j == 3 ? 5.0f / 84.0f
                   : j == 4 ? -5.0f / 504.0f : 1.0f / 1260.0f);
}

}  // namespace fwi
