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
// Work is taken by warps: the items of lattice.cuh for edges and vertices, and
// units of 32 points of a face.
#pragma once

#include "lattice.cuh"

namespace hyteg {

// Face points.  Inside one item both copies' macros, the face of each macro
// (x = 0, y = 0, z = 0 or x+y+z = n) and the local axes are the same for every
// lane, a face cuts off 4 of the 14 neighbours, and the 11 terms left take
// their weights, in the order of NW3's slots, from a table of 12 per (cell,
// face) read as vectors: about 55 instructions per copy where testing 15
// neighbours one by one took about 500, more than the macros' interiors.
constexpr int NFW = 12;
template <unsigned OUT, class T>
__device__ __forceinline__ void face_load(const T* xp, const Off15& o, T v[11]) {
  const T *pa = xp + o.A, *ps = xp - o.A, *pu = xp + o.U, *pua = pu - o.A, *pd = xp - o.D, *pda = pd + o.A;
  int t = 0;
#define HY_TERM(k, e) \
  if (!((OUT >> k) & 1)) v[t++] = ld<false>(e);
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
  __device__ __forceinline__ void load(const T* x, unsigned map, const Off15& o) {
    const T* xp = x + slot;
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

// Face units: a warp takes 32 points of one face, 22 loads in flight per lane
// (two points per lane need too many registers beside the march: level 6, 384
// macro-tets 272 against 233 us in float-float, 87 against 84 us in fp32).
// ab: the face points' (a | b << 16) in order, the same for every face.
template <int MODE, bool SKIP0, class T>
__device__ __forceinline__ void face3d_unit(const T* x, T* y, const Face3Rec* __restrict__ rec,
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
    if (live) y[f0.slot] = mode_out<MODE, false>(ld<false>(x + f0.slot), x, md, f0.slot);
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
  const T v = mode_out<MODE, false>(acc, x, md, f0.slot);
  y[f0.slot] = v;
  if (two) y[f1.slot] = v;
}

// Everything that the interface step of a launch reads.
template <class T>
struct Iface3 {
  const IfItem* items;  // edges and vertices
  int n_items, per_face, n_pts, n_units;  // items, units and points per face, units in all
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
__device__ __forceinline__ void iface3d_unit(const T* x, T* y, const Iface3<T>& f, int u,
                                             int n, int64_t S, const StencilPtr& st, const ModeArgs& md) {
  if (u >= f.n_items) {
    const int v = u - f.n_items, face = v / f.per_face;
    face3d_unit<MODE, SKIP0, T>(x, y, f.faces + face, v - face * f.per_face, f.n_pts, f.ab, f.wf, n, S, md);
    return;
  }
  const IfItem it = f.items[u];
  pdl_wait();
  apply_item<3, MODE, SKIP0, false>(x, y, it, (int)(threadIdx.x & 31), f.incs, n, S, st, md);
}

}  // namespace hyteg
