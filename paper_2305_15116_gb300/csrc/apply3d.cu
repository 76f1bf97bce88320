// 3D apply and sweeps of small vectors: one thread per macro-interior point,
// neighbours straight from memory, and the interface points in the same
// launch (iface3d.cuh).
//
// The 15-point Kuhn stencil in the direct form reads every value 15 times,
// through L1 and L2; on a level whose vector stays in L2 what counts is the
// length of the chain of dependent loads, and here it is one table entry
// (read before the previous kernel has finished) and one round of loads.
#include <vector>

#include "fallback.cuh"
#include "group.cuh"
#include "iface3d.cuh"

namespace hyteg {

namespace {

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

template <class P, int MODE>
struct Direct3 {
  using T = typename P::T;
  static constexpr int kThreads = 256;
  static constexpr bool kLateWait = true;  // the tables first
  struct Prm {
    const T* x;
    T* y;
    const int2* pts;  // interior points of a macro: (slot, A | M << 16)
    int n_pts, bpm;   // per macro: points, blocks
    const int4* items;
    int n_items, n_if_blocks;
    const Prim* prims;
    const Inc* incs;
    StencilPtr st;
    ModeArgs md;
    int n;
    int64_t S;
  };
  static __device__ __forceinline__ void run(const Prm& p, int block, int) {
    if (block < p.n_if_blocks) {
      const int item = 2 * block + (int)(threadIdx.x >> 7);
      if (item >= p.n_items) return;
      const int4 it = p.items[item];
      const Prim pr = p.prims[it.x];
      pdl_wait();
      iface3d_item<MODE, P::kPoison, T>(p.x, p.y, it, (int)(threadIdx.x & 127), pr, p.incs, p.n, p.S, p.st, p.md);
      return;
    }
    const int b = block - p.n_if_blocks;
    const int m = b / p.bpm;
    const int t = (b - m * p.bpm) * kThreads + (int)threadIdx.x;
    if (t >= p.n_pts) return;
    const int2 e = p.pts[t];
    const int64_t wb = (int64_t)m * (NCLS3 * NW3);
    const typename P::W w0 = P::weight(p.st, wb), w1 = P::weight(p.st, wb + 1), w3 = P::weight(p.st, wb + 3),
                        w5 = P::weight(p.st, wb + 5), w7 = P::weight(p.st, wb + 7), w8 = P::weight(p.st, wb + 8),
                        w9 = P::weight(p.st, wb + 9), w10 = P::weight(p.st, wb + 10);
    const Off15 o(e.y >> 16, e.y & 0xFFFF);
    const int64_t i = (int64_t)m * p.S + e.x;
    const T* __restrict__ xp = p.x + i;
    pdl_wait();
    T v[NW3];
#pragma unroll
    for (int k = 0; k < NW3; ++k) v[k] = __ldg(xp + o[k]);
    T bi = T(0), di = T(0);
    if (MODE == MODE_JACOBI || MODE == MODE_RESIDUAL) bi = __ldg(static_cast<const T*>(p.md.b) + i);
    if (MODE == MODE_JACOBI) di = __ldg(static_cast<const T*>(p.md.dinv) + i);
    using O = One<P>;
    typename O::Acc a;
    O::first(a, w0, P::conv(v[0]));
    O::sym(a, w1, P::conv(v[1]), P::conv(v[2]));
    O::sym(a, w3, P::conv(v[3]), P::conv(v[4]));
    O::sym(a, w5, P::conv(v[5]), P::conv(v[6]));
    O::sym(a, w7, P::conv(v[7]), P::conv(v[11]));
    O::sym(a, w8, P::conv(v[8]), P::conv(v[12]));
    O::sym(a, w9, P::conv(v[9]), P::conv(v[13]));
    O::sym(a, w10, P::conv(v[10]), P::conv(v[14]));
    T r = O::finish(a);
    if constexpr (P::kPoison) {  // an input outside the float-float range: native fp64 row
      if (O::bad(a)) {
        const double* __restrict__ wd = p.st.d + wb;
        r = 0.0;
#pragma unroll
        for (int k = 0; k < NW3; ++k) {
          const double wk = __ldg(wd + k);
          if (wk != 0.0) r = __fma_rn(wk, v[k], r);
        }
      }
    }
    p.y[i] = mode_out_staged<MODE, T>(r, v[0], bi, di, p.md.omega);
  }
};

template <class P, int MODE>
cudaError_t launch_direct(const Mesh* const* ms, const int* levels, const void* const* xs, void* const* ys,
                          const ModeArgs* md, int count, cudaStream_t s) {
  using B = Direct3<P, MODE>;
  using T = typename P::T;
  std::vector<typename B::Prm> prm;
  std::vector<int> blocks;
  prm.reserve(count);
  blocks.reserve(count);
  for (int i = 0; i < count; ++i) {
    const Mesh& m = *ms[i];
    const LevelDev& L = m.levels[levels[i]];
    typename B::Prm p;
    p.x = static_cast<const T*>(xs[i]);
    p.y = static_cast<T*>(ys[i]);
    p.pts = L.pts3;
    p.n_pts = L.n_pts3;
    p.bpm = (L.n_pts3 + B::kThreads - 1) / B::kThreads;
    p.items = L.if3;
    p.n_items = L.n_if3;
    p.n_if_blocks = (L.n_if3 + 1) / 2;
    p.prims = m.d_prims;
    p.incs = m.d_incs;
    p.st = StencilPtr{L.st64, L.st32, L.st_hi, L.st_lo};
    p.md = md ? md[i] : ModeArgs{nullptr, nullptr, 0.0};
    p.n = L.n;
    p.S = L.slots_per_macro;
    prm.push_back(p);
    blocks.push_back(p.n_if_blocks + p.bpm * int(m.n_cells));
  }
  return launch_group<B>(prm.data(), blocks.data(), count, s);
}

template <int MODE>
cudaError_t launch_direct_dt(int dtype, const Mesh* const* ms, const int* levels, const void* const* xs,
                             void* const* ys, int count, cudaStream_t s) {
  switch (dtype) {
    case 1: return launch_direct<ArF64FF, MODE>(ms, levels, xs, ys, nullptr, count, s);
    case 2: return launch_direct<ArF32, MODE>(ms, levels, xs, ys, nullptr, count, s);
    case 3: return launch_direct<ArF64Native, MODE>(ms, levels, xs, ys, nullptr, count, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_direct3d_group(int dtype, bool partial, const Mesh* const* ms, const int* levels,
                                  const void* const* xs, void* const* ys, int count, cudaStream_t s) {
  return partial ? launch_direct_dt<MODE_PARTIAL>(dtype, ms, levels, xs, ys, count, s)
                 : launch_direct_dt<MODE_APPLY>(dtype, ms, levels, xs, ys, count, s);
}

}  // namespace hyteg
