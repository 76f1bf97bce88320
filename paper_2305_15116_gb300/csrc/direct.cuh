// One macro-interior point in the direct form: the neighbours straight from
// memory.
#pragma once

#include "lattice.cuh"
#include "one.cuh"

namespace hyteg {

// Interior weights of a macro, the centre's and one per pair of opposite
// neighbours (the interior stencil is symmetric).
template <int DIM, class P>
struct InnerW {
  static constexpr int N = DIM == 2 ? 4 : 8;
  typename P::W w[N];
  __device__ __forceinline__ void load(const StencilPtr& st, int64_t wb) {
    if constexpr (DIM == 2) {  // C, E, N, SE
      w[0] = P::weight(st, wb + 3), w[1] = P::weight(st, wb + 4);
      w[2] = P::weight(st, wb + 6), w[3] = P::weight(st, wb + 1);
    } else {
      w[0] = P::weight(st, wb), w[1] = P::weight(st, wb + 1), w[2] = P::weight(st, wb + 3);
      w[3] = P::weight(st, wb + 5), w[4] = P::weight(st, wb + 7), w[5] = P::weight(st, wb + 8);
      w[6] = P::weight(st, wb + 9), w[7] = P::weight(st, wb + 10);
    }
  }
};

// (A x) at the point with value pointer xp and neighbour offsets o, in the
// order of roundings of the row walkers; uc: the centre value.
template <int DIM, class P, bool CG>
__device__ __forceinline__ typename P::T inner_row(const typename P::T* xp, const typename Lat<DIM>::Off& o,
                                                   const InnerW<DIM, P>& W, const StencilPtr& st, int64_t wb,
                                                   typename P::T& uc) {
  using T = typename P::T;
  using O = One<P>;
  constexpr int NW = Lat<DIM>::NW;
  T v[NW];
#pragma unroll
  for (int k = 0; k < NW; ++k) v[k] = ld<CG>(xp + o[k]);
  typename O::Acc a;
  if constexpr (DIM == 2) {
    uc = v[3];
    O::first(a, W.w[0], P::conv(v[3]));
    O::sym(a, W.w[1], P::conv(v[4]), P::conv(v[2]));
    O::sym(a, W.w[2], P::conv(v[6]), P::conv(v[0]));
    O::sym(a, W.w[3], P::conv(v[1]), P::conv(v[5]));
  } else {
    uc = v[0];
    O::first(a, W.w[0], P::conv(v[0]));
    O::sym(a, W.w[1], P::conv(v[1]), P::conv(v[2]));
    O::sym(a, W.w[2], P::conv(v[3]), P::conv(v[4]));
    O::sym(a, W.w[3], P::conv(v[5]), P::conv(v[6]));
    O::sym(a, W.w[4], P::conv(v[7]), P::conv(v[11]));
    O::sym(a, W.w[5], P::conv(v[8]), P::conv(v[12]));
    O::sym(a, W.w[6], P::conv(v[9]), P::conv(v[13]));
    O::sym(a, W.w[7], P::conv(v[10]), P::conv(v[14]));
  }
  T r = O::finish(a);
  if constexpr (P::kPoison) {  // an input outside the float-float range: native fp64, as fallback.cuh
    if (O::bad(a)) {
      const double* __restrict__ wd = st.d + wb;
      if constexpr (DIM == 2) {
        r = __dmul_rn(__ldg(wd + 3), v[3]);
        r = __fma_rn(__ldg(wd + 4), v[4], r);
        r = __fma_rn(__ldg(wd + 2), v[2], r);
        r = __fma_rn(__ldg(wd + 6), v[6], r);
        r = __fma_rn(__ldg(wd + 5), v[5], r);
        r = __fma_rn(__ldg(wd + 0), v[0], r);
        r = __fma_rn(__ldg(wd + 1), v[1], r);
      } else {
        r = 0.0;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
          const double wk = __ldg(wd + k);
          if (wk != 0.0) r = __fma_rn(wk, v[k], r);
        }
      }
    }
  }
  return r;
}

// Interior point t of a macro in 2D: rows y = 1 .. n-2 of n-1-y points.
__device__ __forceinline__ void inner_point2(int t, int n, int& slot, int& A) {
  const int K = n - 2;
  const int j = tri_row(t, K), y = j + 1;
  const int x = 1 + t - (j * K - (j * (j - 1)) / 2);
  A = n + 1 - y;
  slot = y * (n + 2) - ((y * (y + 1)) >> 1) + x;
}

}  // namespace hyteg
