// What an apply / sweep launch writes at a point with (A u) = au:
//   MODE_APPLY:    y = A u
//   MODE_JACOBI:   y = u + omega dinv (b - A u)   (one weighted Jacobi sweep)
//   MODE_RESIDUAL: y = b - A u
// (u = x at the point; b and dinv in the slot layout, copies equal).
//   MODE_PARTIAL:  y = A u inside the macros; at interface points every copy
//                  receives its own macro's partial row instead of the sum
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace hyteg {

constexpr int MODE_APPLY = 0, MODE_JACOBI = 1, MODE_RESIDUAL = 2, MODE_PARTIAL = 3;

struct ModeArgs {
  const void* b;
  const void* dinv;
  double omega;
};

#ifdef __CUDACC__
// u, b and dinv of the point already in registers
template <int MODE, class T>
__device__ __forceinline__ T mode_out_staged(T au, T u, T b, T d, double omega) {
  if (MODE != MODE_JACOBI && MODE != MODE_RESIDUAL) return au;
  if (MODE == MODE_RESIDUAL) return b - au;
  return u + (T)omega * d * (b - au);
}

template <int MODE, class T>
__device__ __forceinline__ T mode_out(T au, const T* __restrict__ x, const ModeArgs& md, int64_t i) {
  if (MODE != MODE_JACOBI && MODE != MODE_RESIDUAL) return au;
  const T bi = __ldg(static_cast<const T*>(md.b) + i);
  if (MODE == MODE_RESIDUAL) return bi - au;
  const T ui = __ldg(x + i), di = __ldg(static_cast<const T*>(md.dinv) + i);
  return ui + (T)md.omega * di * (bi - au);
}
#endif

}  // namespace hyteg
