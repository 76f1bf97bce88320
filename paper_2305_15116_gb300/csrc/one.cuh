// Single-point forms of the arithmetic policies (arith.cuh).
#pragma once

#include "arith.cuh"

namespace hyteg {

// Single-point forms of the policies' pair operations, in the same order of
// roundings, so that a point's value does not depend on the kernel that
// computes it.
template <class P>
struct One;
template <>
struct One<ArF32> {
  using Acc = float;
  static __device__ __forceinline__ void first(Acc& a, const float& w, float v) { a = __fmul_rn(w, v); }
  static __device__ __forceinline__ void sym(Acc& a, const float& w, float u, float v) {
    a = __fmaf_rn(w, __fadd_rn(u, v), a);
  }
  static __device__ __forceinline__ float finish(Acc a) { return a; }
  static __device__ __forceinline__ bool bad(Acc) { return false; }
};
template <>
struct One<ArF64Native> {
  using Acc = double;
  static __device__ __forceinline__ void first(Acc& a, const double& w, double v) { a = __dmul_rn(w, v); }
  static __device__ __forceinline__ void sym(Acc& a, const double& w, double u, double v) {
    a = __fma_rn(w, __dadd_rn(u, v), a);
  }
  static __device__ __forceinline__ double finish(Acc a) { return a; }
  static __device__ __forceinline__ bool bad(Acc) { return false; }
};
template <>
struct One<ArF64FF> {
  struct Acc {
    float s, e;
  };
  static __device__ __forceinline__ void first(Acc& a, const ArF64FF::W& w, FF v) {
    const float pm = __fmul_rn(-w.h1, v.h);
    a.s = __fsub_rn(0.0f, pm);
    float e = __fmaf_rn(w.h1, v.h, pm);
    e = __fmaf_rn(w.h1, v.l, e);
    a.e = __fmaf_rn(w.l1, v.h, e);
  }
  static __device__ __forceinline__ void sym(Acc& a, const ArF64FF::W& w, FF u, FF v) {
    const float sh = __fadd_rn(u.h, v.h);
    const float bb = __fsub_rn(sh, u.h);
    const float er = __fadd_rn(__fsub_rn(u.h, __fsub_rn(sh, bb)), __fsub_rn(v.h, bb));
    const float sl = __fadd_rn(__fadd_rn(u.l, v.l), er);
    float e = __fmaf_rn(w.h1, sl, a.e);
    const float pm = __fmul_rn(-w.h1, sh);
    e = __fmaf_rn(w.l1, sh, e);
    const float sn = __fsub_rn(a.s, pm);
    const float nbp = __fsub_rn(a.s, sn);
    const float t2 = __fsub_rn(a.s, __fadd_rn(sn, nbp));
    a.s = sn;
    e = __fadd_rn(e, __fmaf_rn(w.h1, sh, nbp));
    a.e = __fadd_rn(e, t2);
  }
  static __device__ __forceinline__ double finish(const Acc& a) { return ff_join(a.s, a.e); }
  static __device__ __forceinline__ bool bad(const Acc& a) { return a.s != a.s; }
};

}  // namespace hyteg
