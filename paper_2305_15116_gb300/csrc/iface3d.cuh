// The interface step of the 3D apply and sweeps: points on macro faces, edges
// and vertices, completed in the launch that sweeps the macros (the paper's
// interface primitives, Sec. 5.1).
//
// A copy of such a point contributes its macro's PARTIAL row, the class
// stencil restricted to the micro-elements of that macro, evaluated straight
// from x; the partials are summed in ascending macro order and the sum goes
// to every copy.  Dirichlet points get y = x.  Arithmetic in the element type
// (float64 for the float-float apply).
//
// Why the partial rows are formed here from x and not left in y by the macro
// kernel and summed by a second launch: the second launch read a table of
// slots as large as the vector's interface part (16 B per point) and both
// copies, and took a launch of its own (36 us of 285 at level 6 with 384
// macro-tets, 6 to 8 us on a small level, as long as the apply itself).
//
// Work is taken by warps.  Work list (LevelDev::if3): int4 (-, first point,
// points, lanes per point), 32 lanes per item, edges and vertices; and units of
// a face's points.  A face point (two copies) or a
// Dirichlet point takes one thread; a point on an edge or vertex inside the
// domain one lane per copy, the partials added in ascending copy order
// through shuffles (walked one after another, the copies' dependent loads
// were the latency floor of small levels).
//
// SKIP0 (float-float apply): a zero weight does not read its neighbour into
// the sum, so that an infinity or NaN beyond it leaves the row alone, as in
// the native recomputation of the macro-interior rows (fallback.cuh).
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

// neighbours (bits) that lie outside the macro, by face of the point's class
constexpr unsigned OUT_X0 = 1u << 2 | 1u << 6 | 1u << 8 | 1u << 14;   // x = 0: dx < 0
constexpr unsigned OUT_Y0 = 1u << 4 | 1u << 5 | 1u << 9 | 1u << 10;   // y = 0: dy < 0
constexpr unsigned OUT_Z0 = 1u << 11 | 1u << 12 | 1u << 13 | 1u << 14;  // z = 0: dz < 0
constexpr unsigned OUT_N = 1u << 1 | 1u << 3 | 1u << 7 | 1u << 10;    // x+y+z = n: dx+dy+dz > 0

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

// A copy of an interface point: its slot and its macro's partial row there.
template <class T>
struct Copy3 {
  int64_t slot;
  T part;
};

template <bool PART, bool SKIP0, class T>
__device__ __forceinline__ Copy3<T> iface3d_copy(const T* __restrict__ x, const Inc& inc, const int wv[3], int type,
                                                 int n, int64_t S, const StencilPtr& st) {
  int q[3] = {0, 0, 0};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    if (j > type) continue;
    const int c = inc.corner[j];
    q[0] += c == 1 ? wv[j] : 0;
    q[1] += c == 2 ? wv[j] : 0;
    q[2] += c == 3 ? wv[j] : 0;
  }
  const int M = n + 1 - q[2], A = M - q[1];
  Copy3<T> r;
  r.slot = (int64_t)inc.cell * S + (slice_begin(n, M) + q[1] * M - ((q[1] * (q[1] - 1)) >> 1) + q[0]);
  r.part = T(0);
  if (PART) {
    const int cls = (q[0] == 0 ? 1 : 0) | (q[1] == 0 ? 2 : 0) | (q[2] == 0 ? 4 : 0) |
                    (q[0] + q[1] + q[2] == n ? 8 : 0);
    const unsigned out = (cls & 1 ? OUT_X0 : 0u) | (cls & 2 ? OUT_Y0 : 0u) | (cls & 4 ? OUT_Z0 : 0u) |
                         (cls & 8 ? OUT_N : 0u);
    const int64_t wb = ((int64_t)inc.cell * NCLS3 + cls) * NW3;
    const T* __restrict__ xp = x + r.slot;
    const Off15 off(M, A);
    T v[NW3], w[NW3];
#pragma unroll
    for (int k = 0; k < NW3; ++k) {
      w[k] = i3_w(st, wb + k, T(0));
      v[k] = (out >> k) & 1u ? T(0) : __ldg(xp + off[k]);
    }
    // a neighbour outside the macro adds 0 * 0 (its weight is zero)
    T a = i3_mul(w[0], v[0]);
#pragma unroll
    for (int k = 1; k < NW3; ++k) {
      const T t = i3_fma(w[k], v[k], a);
      a = SKIP0 && i3_zero(w[k]) ? a : t;
    }
    r.part = a;
  }
  return r;
}

// Face points.  Inside one item both copies' macros, the face of each macro
// (x = 0, y = 0, z = 0 or x+y+z = n) and the local axes are the same for every
// lane, a face cuts off 4 of the 14 neighbours, and the 11 terms left take
// their weights, in the order of NW3's slots, from a table of 12 per (cell,
// face) read as vectors: about 55 instructions per copy where testing 15
// neighbours one by one took about 500, more than the macros' interiors.
constexpr int NFW = 12;
template <unsigned OUT, class T>
__device__ __forceinline__ void face_load(const T* __restrict__ xp, const Off15& o, T v[11]) {
  const T *pa = xp + o.A, *ps = xp - o.A, *pu = xp + o.U, *pua = pu - o.A, *pd = xp - o.D, *pda = pd + o.A;
  int t = 0;
#define HY_TERM(k, e) \
  if (!((OUT >> k) & 1)) v[t++] = __ldg(e);
  HY_TERM(0, xp)
  HY_TERM(1, xp + 1)
  HY_TERM(2, xp - 1)
  HY_TERM(3, pa)
  HY_TERM(4, ps - 1)
  HY_TERM(5, ps)
  HY_TERM(6, pa - 1)
  HY_TERM(7, pu)
  HY_TERM(8, pu - 1)
  HY_TERM(9, pua)
  HY_TERM(10, pua + 1)
  HY_TERM(11, pd)
  HY_TERM(12, pd + 1)
  HY_TERM(13, pda + 1)
  HY_TERM(14, pda)
#undef HY_TERM
}
__device__ __forceinline__ void face_weights(const double* __restrict__ p, double w[NFW]) {
#pragma unroll
  for (int i = 0; i < NFW / 2; ++i) {
    const double2 t = __ldg(reinterpret_cast<const double2*>(p) + i);
    w[2 * i] = t.x;
    w[2 * i + 1] = t.y;
  }
}
__device__ __forceinline__ void face_weights(const float* __restrict__ p, float w[NFW]) {
#pragma unroll
  for (int i = 0; i < NFW / 4; ++i) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(p) + i);
    w[4 * i] = t.x;
    w[4 * i + 1] = t.y;
    w[4 * i + 2] = t.z;
    w[4 * i + 3] = t.w;
  }
}

// One copy of a face point: its slot and the 11 values of its partial row.
template <class T>
struct Face3 {
  int64_t slot;
  T v[11];
  static __device__ __forceinline__ int coef(unsigned m, int i) { return (int)(m << (30 - 2 * i)) >> 30; }
  // where the point lies in the macro `cell`
  __device__ __forceinline__ Off15 place(int cell, unsigned map, int a, int b, int n, int64_t S) {
    const int q0 = n * (int)(map & 1u) + coef(map, 1) * a + coef(map, 2) * b;
    const int q1 = n * (int)((map >> 6) & 1u) + coef(map, 4) * a + coef(map, 5) * b;
    const int q2 = n * (int)((map >> 12) & 1u) + coef(map, 7) * a + coef(map, 8) * b;
    const int M = n + 1 - q2;
    slot = (int64_t)cell * S + (slice_begin(n, M) + q1 * M - ((q1 * (q1 - 1)) >> 1) + q0);
    return Off15(M, M - q1);
  }
  __device__ __forceinline__ void load(const T* __restrict__ x, unsigned map, const Off15& o) {
    const T* __restrict__ xp = x + slot;
    switch ((int)(map >> 18)) {  // the corner that the face does not hold
      case 0: face_load<OUT_N>(xp, o, v); break;
      case 1: face_load<OUT_X0>(xp, o, v); break;
      case 2: face_load<OUT_Y0>(xp, o, v); break;
      default: face_load<OUT_Z0>(xp, o, v); break;
    }
  }
  template <bool SKIP0>
  __device__ __forceinline__ T row(const T* __restrict__ wf) const {
    T w[NFW];
    face_weights(wf, w);
    T a = i3_mul(w[0], v[0]);
#pragma unroll
    for (int k = 1; k < 11; ++k) a = i3_fma(w[k], v[k], a);
    if (SKIP0 && a != a) {  // perhaps a zero weight met an infinity
      a = i3_mul(w[0], v[0]);
#pragma unroll
      for (int k = 1; k < 11; ++k)
        if (!i3_zero(w[k])) a = i3_fma(w[k], v[k], a);
    }
    return a;
  }
};

// Lane t of work item `it` (one warp).  MODE_SUM: the copies of y hold their macros' partial rows already.
constexpr int MODE_SUM = 4;

template <int MODE, bool SKIP0, class T>
__device__ __forceinline__ void iface3d_item(const T* __restrict__ x, T* __restrict__ y, const int4 it, int t,
                                             const Prim& p, const Inc* __restrict__ incs, int n, int64_t S,
                                             const StencilPtr& st, const ModeArgs& md) {
  const int G = it.w;
  const int pt = t / G;
  const bool live = pt < it.z;
  const int i = it.y + (live ? pt : 0);
  int wv[3];
  if (p.type == 0) {
    wv[0] = n, wv[1] = 0, wv[2] = 0;
  } else if (p.type == 1) {
    wv[0] = n - 1 - i, wv[1] = i + 1, wv[2] = 0;
  } else {  // rows b = 1.. of the face's interior points, a = 1 .. n-1-b
    const int K = n - 2;
    const int j = tri_row(i, K);
    const int a = 1 + i - (j * K - (j * (j - 1)) / 2);
    wv[0] = n - a - (j + 1), wv[1] = a, wv[2] = j + 1;
  }
  const Inc* __restrict__ ic = incs + p.inc_begin;
  auto copy_of = [&](int k) -> Copy3<T> {
    Copy3<T> c = iface3d_copy<MODE != MODE_SUM, SKIP0, T>(x, ic[k], wv, p.type, n, S, st);
    if (MODE == MODE_SUM) c.part = y[c.slot];
    return c;
  };
  if (G > 1) {  // one lane per copy
    const int lane = t & (G - 1), base = (t & 31) & ~(G - 1);
    const bool mine = live && lane < p.inc_count;
    Copy3<T> c{0, T(0)};
    if (mine) c = copy_of(lane);
    if (MODE == MODE_PARTIAL) {
      if (mine) y[c.slot] = c.part;
      return;
    }
    T acc = T(0);
    for (int k = 0; k < p.inc_count; ++k) acc += __shfl_sync(0xFFFFFFFFu, c.part, base + k);
    // copies hold equal u, b and dinv: the first one's
    const int64_t s0 = __shfl_sync(0xFFFFFFFFu, c.slot, base);
    if (mine) y[c.slot] = mode_out<MODE>(acc, x, md, s0);
    return;
  }
  if (!live) return;
  if (MODE != MODE_PARTIAL && p.boundary) {
    Copy3<T> c = iface3d_copy<false, SKIP0, T>(x, ic[0], wv, p.type, n, S, st);
    const T v = mode_out<MODE>(__ldg(x + c.slot), x, md, c.slot);
    y[c.slot] = v;
    for (int k = 1; k < p.inc_count; ++k) y[iface3d_copy<false, SKIP0, T>(x, ic[k], wv, p.type, n, S, st).slot] = v;
    return;
  }
  if (p.inc_count <= 2) {
    const bool two = p.inc_count == 2;
    const Copy3<T> c0 = copy_of(0);
    const Copy3<T> c1 = copy_of(two ? 1 : 0);
    if (MODE == MODE_PARTIAL) {
      y[c0.slot] = c0.part;
      if (two) y[c1.slot] = c1.part;
      return;
    }
    T acc = T(0) + c0.part;
    if (two) acc += c1.part;
    const T v = mode_out<MODE>(acc, x, md, c0.slot);
    y[c0.slot] = v;
    if (two) y[c1.slot] = v;
    return;
  }
  // more copies than a warp has lanes
  T acc = T(0);
  int64_t s0 = 0;
  for (int k = 0; k < p.inc_count; ++k) {
    const Copy3<T> c = copy_of(k);
    if (k == 0) s0 = c.slot;
    if (MODE == MODE_PARTIAL) y[c.slot] = c.part;
    acc += c.part;
  }
  if (MODE == MODE_PARTIAL) return;
  const T v = mode_out<MODE>(acc, x, md, s0);
  for (int k = 0; k < p.inc_count; ++k) y[iface3d_copy<false, SKIP0, T>(x, ic[k], wv, p.type, n, S, st).slot] = v;
}

// Face units: a warp takes 32 points of one face, 22 loads in flight per lane
// (two points per lane need too many registers beside the march: level 6, 384
// macro-tets 272 against 233 us in float-float, 87 against 84 us in fp32).
// ab: the face points' (a | b << 16) in order, the same for every face.
template <int MODE, bool SKIP0, class T>
__device__ __forceinline__ void face3d_unit(const T* __restrict__ x, T* __restrict__ y, const Face3Rec* __restrict__ rec,
                                            int run, int n_pts, const unsigned* __restrict__ ab,
                                            const T* __restrict__ wf, int n, int64_t S, const ModeArgs& md) {
  const int t = run * 32 + (int)(threadIdx.x & 31);
  const bool live = t < n_pts;
  const unsigned pt = __ldg(ab + (live ? t : 0));
  const int a = (int)(pt & 0xFFFFu), b = (int)(pt >> 16);
  const Face3Rec r = *rec;
  const bool two = r.cell1 >= 0;
  Face3<T> f0, f1;
  const Off15 o0 = f0.place(r.cell0, r.map0, a, b, n, S);
  if (MODE != MODE_PARTIAL && r.dirichlet) {
    pdl_wait();
    if (live) y[f0.slot] = mode_out<MODE>(__ldg(x + f0.slot), x, md, f0.slot);
    return;
  }
  const Off15 o1 = f1.place(two ? r.cell1 : r.cell0, two ? r.map1 : r.map0, a, b, n, S);
  pdl_wait();  // the vectors after the previous kernel in the stream
  f0.load(x, r.map0, o0);
  if (two) f1.load(x, r.map1, o1);
  const T p0 = f0.template row<SKIP0>(wf + ((int64_t)r.cell0 * 4 + (int)(r.map0 >> 18)) * NFW);
  T p1 = T(0);
  if (two) p1 = f1.template row<SKIP0>(wf + ((int64_t)r.cell1 * 4 + (int)(r.map1 >> 18)) * NFW);
  if (!live) return;
  if (MODE == MODE_PARTIAL) {
    y[f0.slot] = p0;
    if (two) y[f1.slot] = p1;
    return;
  }
  T acc = T(0) + p0;
  if (two) acc += p1;
  const T v = mode_out<MODE>(acc, x, md, f0.slot);
  y[f0.slot] = v;
  if (two) y[f1.slot] = v;
}

// Everything that the interface step of a launch reads.
template <class T>
struct Iface3 {
  const If3Item* items;  // edges and vertices
  int n_items, n_faces, per_face, n_pts, n_units;  // items, faces, units and points per face, units in all
  const Face3Rec* faces;
  const unsigned* ab;
  const Inc* incs;
  const T* wf;
};

__device__ __forceinline__ void cp_async_one(float* smem, const float* g) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(g));
}
__device__ __forceinline__ void cp_async_one(double* smem, const double* g) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(g));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;"); }
// waits until all but the newest LEFT committed groups have landed
template <int LEFT>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// Unit `u` of a mesh's interface step, by one warp: an item (the first ones)
// or a unit of a face.
template <int MODE, bool SKIP0, class T>
__device__ __forceinline__ void iface3d_unit(const T* __restrict__ x, T* __restrict__ y, const Iface3<T>& f, int u,
                                             int n, int64_t S, const StencilPtr& st, const ModeArgs& md) {
  if (u >= f.n_items) {
    const int v = u - f.n_items, face = v / f.per_face;
    face3d_unit<MODE, SKIP0, T>(x, y, f.faces + face, v - face * f.per_face, f.n_pts, f.ab, f.wf, n, S, md);
    return;
  }
  const If3Item it = f.items[u];
  pdl_wait();
  iface3d_item<MODE, SKIP0, T>(x, y, it.work, (int)(threadIdx.x & 31), it.prim, f.incs, n, S, st, md);
}

}  // namespace hyteg
