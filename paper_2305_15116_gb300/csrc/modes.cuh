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
// A load of a vector's value: a plain one, or (CG) from L2, where values
// written by other blocks of the same launch are seen after a barrier between
// them.  Not the read-only path: a kernel may start before the one that writes
// the vector has finished (group.cuh), and the code generator may move a
// read-only load, which it takes for invariant, above the wait.  For the same
// reason no vector of such a kernel is a __restrict__ pointer: that promises
// that nothing else, the wait included, changes what it points to.
template <bool CG, class T>
__device__ __forceinline__ T ld(const T* p) {
  if constexpr (CG)
    return __ldcg(p);
  else
    return *p;
}

__device__ __forceinline__ float jacobi_out(float au, float u, float b, float d, float omega) {
  return __fmaf_rn(__fmul_rn(omega, d), __fsub_rn(b, au), u);
}
__device__ __forceinline__ double jacobi_out(double au, double u, double b, double d, double omega) {
  return __fma_rn(__dmul_rn(omega, d), __dsub_rn(b, au), u);
}
// u, b and dinv of the point already in registers
template <int MODE, class T>
__device__ __forceinline__ T mode_out_staged(T au, T u, T b, T d, double omega) {
  if (MODE != MODE_JACOBI && MODE != MODE_RESIDUAL) return au;
  if (MODE == MODE_RESIDUAL) return b - au;
  return jacobi_out(au, u, b, d, (T)omega);
}

// CG: loads from L2 (vectors written earlier in the same launch)
template <int MODE, bool CG, class T>
__device__ __forceinline__ T mode_out(T au, const T* x, const ModeArgs& md, int64_t i) {
  if (MODE != MODE_JACOBI && MODE != MODE_RESIDUAL) return au;
  const T* const bp = static_cast<const T*>(md.b) + i;
  const T bi = ld<CG>(bp);
  if (MODE == MODE_RESIDUAL) return bi - au;
  const T ui = ld<CG>(x + i), di = __ldg(static_cast<const T*>(md.dinv) + i);
  return jacobi_out(au, ui, bi, di, (T)md.omega);
}
#endif

}  // namespace hyteg
