// The multigrid transfers point by point.
#pragma once

#include "lattice.cuh"

namespace hyteg {

// Half of a positive normal number; in float64 with an integer subtraction, beside
// the fp64 pipe that bounds the restriction.
__device__ __forceinline__ float half_of(float v) { return 0.5f * v; }
__device__ __forceinline__ double half_of(double v) {
  return __hiloint2double(__double2hiint(v) - (1 << 20), __double2loint(v));
}

// One macro's partial of (P^T r) at its coarse point p (local coordinates on
// the coarse level): the fine value at the coincident point plus half the
// values at the midpoints of the coarse micro-edges around it (6 in 2D, 14 in
// 3D), each divided by the number of macros holding a copy of it (mi: the
// macro's table by boundary class; r: the macro's fine vector, nf = 2 n).  A
// midpoint lies on those of the point's faces that its edge runs along.  INNER:
// a macro-interior point, around which every such number is 1.
template <int DIM, bool CG, bool INNER, class T>
__device__ __forceinline__ T restrict_row(const T* r, const T* __restrict__ mi, const Pt<DIM>& p, int nf) {
  using L = Lat<DIM>;
  Pt<DIM> f;
#pragma unroll
  for (int i = 0; i < 3; ++i) f.q[i] = DIM == 2 && i == 2 ? 0 : 2 * p.q[i];
  f.set(nf);
  const int cls = INNER ? 0 : L::cls(nf, f.q);
  const unsigned out = L::out(cls);
  const typename L::Off off(f.M, f.A);
  const T* const rp = r + f.slot;
  T v[2 * L::ND], m[L::ND];  // m: half the divisor
  const T c = ld<CG>(rp), mc = INNER ? T(1) : __ldg(mi + cls);
#pragma unroll
  for (int d = 0; d < L::ND; ++d) {
    int a, b, along;
    L::dir(d, a, b, along);
    m[d] = INNER ? T(0.5) : half_of(__ldg(mi + (cls & along)));
    v[2 * d] = (out >> a) & 1u ? T(0) : ld<CG>(rp + off[a]);
    v[2 * d + 1] = (out >> b) & 1u ? T(0) : ld<CG>(rp + off[b]);
  }
  T acc = INNER ? c : i3_mul(c, mc);  // every rounding written out: the same in every kernel
#pragma unroll
  for (int d = 0; d < L::ND; ++d) {
    acc = i3_fma(v[2 * d], m[d], acc);
    acc = i3_fma(v[2 * d + 1], m[d], acc);
  }
  return acc;
}

// Interpolation of the coarse vector e (one macro's) at the fine point q:
// coincident points copy, micro-edge midpoints take the mean of the two coarse
// end points.
template <int DIM, bool CG, class T>
__device__ __forceinline__ T prolong_value(const T* e, const int q[3], int nc) {
  const int px = q[0] & 1, py = q[1] & 1, pz = DIM == 3 ? q[2] & 1 : 0;
  int d[3] = {px, py, pz};
  if (DIM == 2) {
    if (px && py) d[1] = -1;  // the diagonal (1,-1)
  } else {
    if (px && py && !pz) d[1] = -1;        // (1,-1,0)
    else if (px && pz && !py) d[2] = -1;   // (1,0,-1)
    else if (py && pz && !px) d[2] = -1;   // (0,1,-1)
    else if (px && py && pz) d[1] = -1;    // (1,-1,1)
  }
  Pt<DIM> c1, c2;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    c1.q[i] = DIM == 2 && i == 2 ? 0 : (q[i] - d[i]) >> 1;
    c2.q[i] = DIM == 2 && i == 2 ? 0 : (q[i] + d[i]) >> 1;
  }
  c1.set(nc);
  c2.set(nc);
  const T a = ld<CG>(e + c1.slot);
  if (!(px | py | pz)) return a;
  return T(0.5) * (a + ld<CG>(e + c2.slot));
}

}  // namespace hyteg
