// Geometry of a refined macro for kernels that take points one by one, in 2D
// and 3D: slots, boundary classes, neighbour offsets, and the interface work
// items.  Vectors are read with ld (modes.cuh), tables with __ldg.
#pragma once

#include "arith.cuh"
#include "group.cuh"
#include "hyteg_internal.h"
#include "modes.cuh"

namespace hyteg {


// Row y of the points q = 0.. of a triangle whose row j (j = 0..) holds K - j
// points: the largest y with y K - y(y-1)/2 <= q.
__device__ __forceinline__ int tri_row(int q, int K) {
  const float b = 2.0f * K + 1.0f;
  int y = (int)((b - sqrtf(fmaxf(b * b - 8.0f * q, 0.0f))) * 0.5f);
  y = max(y, 0);
  while (y > 0 && y * K - (y * (y - 1)) / 2 > q) --y;
  while ((y + 1) * K - ((y + 1) * y) / 2 <= q) ++y;
  return y;
}

// First slot of the slice of side M: T3(n+1) - T3(M), T3(k) = k(k+1)(k+2)/6
// (in 32 bits up to n = 1024).
__device__ __forceinline__ int slice_begin(int n, int M) {
  if (n <= 1024) {
    const unsigned N = n + 1, B = M;
    return (int)((N * (N + 1) * (N + 2) - B * (B + 1) * (B + 2)) / 6u);
  }
  const int64_t N = n + 1, B = M;
  return (int)((N * (N + 1) * (N + 2) - B * (B + 1) * (B + 2)) / 6);
}

// Slot offsets of the 15 stencil points of (x, y, z) from its own slot, from
// the slice side M = n+1-z and the row length A = M - y (slot order of
// NW3's weights).
struct Off15 {
  int A, U, D;
  __device__ __forceinline__ Off15(int M, int A_) : A(A_), U(M * (M - 1) / 2 + A_), D((M + 1) * (M + 2) / 2 - M + A_) {}
  __device__ __forceinline__ int operator[](int k) const {
    switch (k) {
      case 0: return 0;
      case 1: return 1;
      case 2: return -1;
      case 3: return A;
      case 4: return -A - 1;
      case 5: return -A;
      case 6: return A - 1;
      case 7: return U;
      case 8: return U - 1;
      case 9: return U - A;
      case 10: return U - A + 1;
      case 11: return -D;
      case 12: return 1 - D;
      case 13: return A + 1 - D;
      default: return A - D;
    }
  }
};
// The 7 of (x, y) in 2D, from the row length A = n+1-y (slot order of NW2's
// weights).
struct Off7 {
  int A;
  __device__ __forceinline__ Off7(int, int A_) : A(A_) {}
  __device__ __forceinline__ int operator[](int k) const {
    switch (k) {
      case 0: return -A - 1;
      case 1: return -A;
      case 2: return -1;
      case 3: return 0;
      case 4: return 1;
      case 5: return A - 1;
      default: return A;
    }
  }
};

// 3D: neighbours (bits) that lie outside the macro, by face of the point's class
constexpr unsigned OUT_X0 = 1u << 2 | 1u << 6 | 1u << 8 | 1u << 14;   // x = 0: dx < 0
constexpr unsigned OUT_Y0 = 1u << 4 | 1u << 5 | 1u << 9 | 1u << 10;   // y = 0: dy < 0
constexpr unsigned OUT_Z0 = 1u << 11 | 1u << 12 | 1u << 13 | 1u << 14;  // z = 0: dz < 0
constexpr unsigned OUT_N = 1u << 1 | 1u << 3 | 1u << 7 | 1u << 10;    // x+y+z = n: dx+dy+dz > 0

template <int DIM>
struct Lat;
template <>
struct Lat<2> {
  static constexpr int NW = NW2, NCLS = NCLS2;
  using Off = Off7;
  static __device__ __forceinline__ int side(int n, const int q[3]) { return n + 1; }
  static __device__ __forceinline__ int slot(int n, int, int, const int q[3]) {
    return q[1] * (n + 2) - ((q[1] * (q[1] + 1)) >> 1) + q[0];
  }
  static __device__ __forceinline__ int cls(int n, const int q[3]) {
    return (q[0] == 0 ? 1 : 0) | (q[1] == 0 ? 2 : 0) | (q[0] + q[1] == n ? 4 : 0);
  }
  static __device__ __forceinline__ unsigned out(int c) {
    return (c & 1 ? 1u << 2 | 1u << 5 : 0u) | (c & 2 ? 1u << 0 | 1u << 1 : 0u) | (c & 4 ? 1u << 4 | 1u << 6 : 0u);
  }
  // micro-edge directions of the refinement: weight slots of -d and +d, and the
  // faces of the macro that d runs along (class bits)
  static constexpr int ND = 3;
  static __device__ __forceinline__ void dir(int i, int& minus, int& plus, int& along) {
    switch (i) {
      case 0: minus = 2, plus = 4, along = 2; break;   // (1,0)
      case 1: minus = 0, plus = 6, along = 1; break;   // (0,1)
      default: minus = 5, plus = 1, along = 4; break;  // (1,-1)
    }
  }
};
template <>
struct Lat<3> {
  static constexpr int NW = NW3, NCLS = NCLS3;
  using Off = Off15;
  static __device__ __forceinline__ int side(int n, const int q[3]) { return n + 1 - q[2]; }
  static __device__ __forceinline__ int slot(int n, int M, int, const int q[3]) {
    return slice_begin(n, M) + q[1] * M - ((q[1] * (q[1] - 1)) >> 1) + q[0];
  }
  static __device__ __forceinline__ int cls(int n, const int q[3]) {
    return (q[0] == 0 ? 1 : 0) | (q[1] == 0 ? 2 : 0) | (q[2] == 0 ? 4 : 0) | (q[0] + q[1] + q[2] == n ? 8 : 0);
  }
  static __device__ __forceinline__ unsigned out(int c) {
    return (c & 1 ? OUT_X0 : 0u) | (c & 2 ? OUT_Y0 : 0u) | (c & 4 ? OUT_Z0 : 0u) | (c & 8 ? OUT_N : 0u);
  }
  static constexpr int ND = 7;
  static __device__ __forceinline__ void dir(int i, int& minus, int& plus, int& along) {
    switch (i) {
      case 0: minus = 2, plus = 1, along = 2 | 4; break;        // (1,0,0)
      case 1: minus = 4, plus = 3, along = 1 | 4; break;        // (0,1,0)
      case 2: minus = 11, plus = 7, along = 1 | 2; break;       // (0,0,1)
      case 3: minus = 6, plus = 5, along = 4 | 8; break;        // (1,-1,0)
      case 4: minus = 8, plus = 12, along = 2 | 8; break;       // (1,0,-1)
      case 5: minus = 9, plus = 13, along = 1 | 8; break;       // (0,1,-1)
      default: minus = 14, plus = 10, along = 0; break;         // (1,-1,1)
    }
  }
};

// A point of a macro: local coordinates, slice side, row length, slot.
template <int DIM>
struct Pt {
  int q[3], M, A, slot;
  __device__ __forceinline__ void set(int n) {
    M = Lat<DIM>::side(n, q);
    A = M - q[1];
    slot = Lat<DIM>::slot(n, M, A, q);
  }
};

__device__ __forceinline__ double i3_w(const StencilPtr& st, int64_t i, double) { return __ldg(st.d + i); }
__device__ __forceinline__ float i3_w(const StencilPtr& st, int64_t i, float) { return __ldg(st.f + i); }
__device__ __forceinline__ double i3_fma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float i3_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double i3_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float i3_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ bool i3_zero(double w) {
  return ((unsigned)__double2hiint(w) | (unsigned)__double2loint(w)) == 0u;
}
__device__ __forceinline__ bool i3_zero(float w) { return w == 0.0f; }

// The partial row of macro `cell` (vector xm) at its point p: the class
// stencil, neighbours outside the macro left out.  SKIP0 (float-float apply,
// 3D): a zero weight does not read its neighbour into the sum, so that an
// infinity or NaN beyond it leaves the row alone, as in the native
// recomputation of the macro-interior rows (fallback.cuh).
template <int DIM, bool SKIP0, bool CG, class T>
__device__ __forceinline__ T partial_row(const T* xm, const Pt<DIM>& p, int cell, int n, const StencilPtr& st) {
  using L = Lat<DIM>;
  constexpr int NW = L::NW;
  const int cls = L::cls(n, p.q);
  const unsigned out = L::out(cls);
  const int64_t wb = ((int64_t)cell * L::NCLS + cls) * NW;
  const typename L::Off off(p.M, p.A);
  T v[NW], w[NW];
#pragma unroll
  for (int k = 0; k < NW; ++k) {
    w[k] = i3_w(st, wb + k, T(0));
    v[k] = (out >> k) & 1u ? T(0) : ld<CG>(xm + p.slot + off[k]);
  }
  // a neighbour outside the macro adds 0 * 0 (its weight is zero)
  T a = i3_mul(w[0], v[0]);
#pragma unroll
  for (int k = 1; k < NW; ++k) {
    const T t = i3_fma(w[k], v[k], a);
    a = SKIP0 && i3_zero(w[k]) ? a : t;
  }
  return a;
}

// ---- interface work items ---------------------------------------------------------
// Work is taken by warps, lane t of item `it` (LevelDev::ifi): (-, first point,
// points, lanes per point).  A point of at most two copies, or a Dirichlet
// point, takes one lane (two independent partials in flight); one with more
// copies a lane per copy, the partials added in ascending copy order through
// shuffles (walked one after another, the copies' dependent loads were the
// latency floor of small levels).
//   part(cell, point)      the copy's partial value
//   dirichlet(slot)        the value of a Dirichlet point (slot of a copy)
//   finish(sum, slot)      the value written, from the sum (slot: first copy's)
//   store(slot, value)
// KEEP: every copy is written its own partial value, without a sum.
template <int DIM, bool KEEP, class T, class Part, class Dir, class Fin, class Put>
__device__ __forceinline__ void run_item(const int4 it, int t, const Prim& p, const Inc* __restrict__ incs, int n,
                                         int64_t S, Part part, Dir dirichlet, Fin finish, Put store) {
  const int G = it.w;
  const int pt = t / G;
  const bool live = pt < it.z;
  const int i = it.y + (live ? pt : 0);
  int wv[3];  // weights on the primitive's canonical vertices
  if (p.type == 0) {
    wv[0] = n, wv[1] = 0, wv[2] = 0;
  } else if (DIM == 2 || p.type == 1) {
    wv[0] = n - 1 - i, wv[1] = i + 1, wv[2] = 0;
  } else {  // rows b = 1.. of the face's interior points, a = 1 .. n-1-b
    const int K = n - 2;
    const int j = tri_row(i, K);
    const int a = 1 + i - (j * K - (j * (j - 1)) / 2);
    wv[0] = n - a - (j + 1), wv[1] = a, wv[2] = j + 1;
  }
  const Inc* __restrict__ ic = incs + p.inc_begin;
  auto place = [&](const Inc& inc, Pt<DIM>& o) -> int64_t {
    o.q[0] = o.q[1] = o.q[2] = 0;
#pragma unroll
    for (int j = 0; j < DIM; ++j) {
      if (j > p.type) continue;
      const int c = inc.corner[j];
      o.q[0] += c == 1 ? wv[j] : 0;
      o.q[1] += c == 2 ? wv[j] : 0;
      if (DIM == 3) o.q[2] += c == 3 ? wv[j] : 0;
    }
    o.set(n);
    return (int64_t)inc.cell * S + o.slot;
  };
  if (G > 1) {  // one lane per copy
    const int lane = t & (G - 1), base = t & ~(G - 1);
    const bool mine = live && lane < p.inc_count;
    int64_t slot = 0;
    T v = T(0);
    if (mine) {
      const Inc inc = ic[lane];
      Pt<DIM> o;
      slot = place(inc, o);
      v = part(inc.cell, o);
    }
    if (KEEP) {
      if (mine) store(slot, v);
      return;
    }
    T acc = T(0);
    for (int k = 0; k < p.inc_count; ++k) acc += __shfl_sync(0xFFFFFFFFu, v, base + k);
    const int64_t s0 = __shfl_sync(0xFFFFFFFFu, slot, base);  // copies hold equal values: the first one's
    if (mine) store(slot, finish(acc, s0));
    return;
  }
  if (!live) return;
  if (!KEEP && p.boundary) {
    Pt<DIM> o;
    const int64_t s0 = place(ic[0], o);
    const T v = finish(dirichlet(s0), s0);
    store(s0, v);
    for (int k = 1; k < p.inc_count; ++k) store(place(ic[k], o), v);
    return;
  }
  if (p.inc_count <= 2) {
    const bool two = p.inc_count == 2;
    const Inc i0 = ic[0], i1 = ic[two ? 1 : 0];
    Pt<DIM> o0, o1;
    const int64_t s0 = place(i0, o0), s1 = place(i1, o1);
    const T p0 = part(i0.cell, o0), p1 = part(i1.cell, o1);
    if (KEEP) {
      store(s0, p0);
      if (two) store(s1, p1);
      return;
    }
    T acc = T(0) + p0;
    if (two) acc += p1;
    const T v = finish(acc, s0);
    store(s0, v);
    if (two) store(s1, v);
    return;
  }
  // more copies than a warp has lanes
  T acc = T(0);
  int64_t s0 = 0;
  for (int k = 0; k < p.inc_count; ++k) {
    const Inc inc = ic[k];
    Pt<DIM> o;
    const int64_t s = place(inc, o);
    if (k == 0) s0 = s;
    const T v = part(inc.cell, o);
    if (KEEP) store(s, v);
    acc += v;
  }
  if (KEEP) return;
  const T v = finish(acc, s0);
  for (int k = 0; k < p.inc_count; ++k) {
    Pt<DIM> o;
    store(place(ic[k], o), v);
  }
}

// The apply's and the sweeps' item.
template <int DIM, int MODE, bool SKIP0, bool CG, class T>
__device__ __forceinline__ void apply_item(const T* x, T* y, const IfItem& it, int t, const Inc* __restrict__ incs,
                                           int n, int64_t S, const StencilPtr& st, const ModeArgs& md) {
  run_item<DIM, MODE == MODE_PARTIAL, T>(
      it.work, t, it.prim, incs, n, S,
      [&](int cell, const Pt<DIM>& p) { return partial_row<DIM, SKIP0, CG>(x + (int64_t)cell * S, p, cell, n, st); },
      [&](int64_t s) { return ld<CG>(x + s); }, [&](T a, int64_t s) { return mode_out<MODE, CG>(a, x, md, s); },
      [&](int64_t s, T v) { y[s] = v; });
}

}  // namespace hyteg
