// The launch sequence of one apply, and the sum of partial rows that a
// vector's interface copies hold (float64 difference form of the solver).
//
// The paper hands the points on the macro boundary to separate "interface
// primitives" (Sec. 5.1).  The applies complete them inside their own launch
// (interior2d.cu, iface3d.cuh); the solver's difference-form residual leaves
// every copy its macro's partial row, and the kernels here sum the partials of
// all incident macros in ascending macro order — a fixed order, so the result
// is deterministic — and write the sum to every copy.  Points on the domain
// boundary get the Dirichlet identity row: y = x.
#include <algorithm>
#include <vector>

#include "group.cuh"
#include "hyteg_internal.h"
#include "modes.cuh"

namespace hyteg {

namespace {

__device__ __forceinline__ int64_t tri_slot(int n, int x, int y) {
  return (int64_t)y * (n + 2) - ((int64_t)y * (y + 1)) / 2 + x;
}

// 2D: one block per item (primitive, -, points a0..a1-1) of at most 128
// points; a vertex item has one point.  A point with a single copy is already
// complete.
struct SumItems2 {
  static constexpr int kThreads = 128;
  static constexpr bool kLateWait = true;  // the items' tables first
  struct Prm {
    const double* x;
    double* y;
    const int4* items;
    const Prim* prims;
    const Inc* incs;
    int n;
    int64_t S;
  };
  static __device__ __forceinline__ void run(const Prm& p, int block, int) {
    const int4 it = p.items[block];
    const Prim pr = p.prims[it.x];
    if (!pr.boundary && pr.inc_count == 1) return;
    const int n = p.n;
    const int a = it.z + (pr.type == 0 ? 0 : threadIdx.x);
    const int wv0 = pr.type == 0 ? n : n - a, wv1 = pr.type == 0 ? 0 : a;
    auto slot_of = [&](int i) -> int64_t {
      const Inc inc = p.incs[pr.inc_begin + i];
      int q[2] = {0, 0};
      if (inc.corner[0] >= 1) q[inc.corner[0] - 1] += wv0;
      if (pr.type == 1 && inc.corner[1] >= 1) q[inc.corner[1] - 1] += wv1;
      return (int64_t)inc.cell * p.S + tri_slot(n, q[0], q[1]);
    };
    pdl_wait();
    if (pr.type == 0 && !pr.boundary && pr.inc_count <= 32) {
      // a coarse vertex inside the domain: lane i of the first warp takes
      // copy i, added in ascending copy order through shuffles
      if (threadIdx.x >= 32) return;
      const bool mine = (int)threadIdx.x < pr.inc_count;
      const int64_t s = mine ? slot_of(threadIdx.x) : 0;
      const double v = mine ? p.y[s] : 0.0;
      double acc = 0.0;
      for (int i = 0; i < pr.inc_count; ++i) acc += __shfl_sync(0xFFFFFFFFu, v, i);
      if (mine) p.y[s] = acc;
      return;
    }
    if (it.z + (int)threadIdx.x >= it.w) return;
    double acc = 0.0;
    if (pr.boundary) {
      acc = ld<false>(p.x + slot_of(0));
    } else {
      for (int i = 0; i < pr.inc_count; ++i) acc += p.y[slot_of(i)];
    }
    for (int i = 0; i < pr.inc_count; ++i) p.y[slot_of(i)] = acc;
  }
};

}  // namespace

cudaError_t launch_sum_copies(const Mesh* const* ms, const int* levels, const double* const* x, double* const* y,
                              int cnt, cudaStream_t s) {
  if (cnt <= 0) return cudaSuccess;
  if (ms[0]->dim == 3) return launch_sum_copies3d(ms, levels, x, y, cnt, s);
  std::vector<SumItems2::Prm> p;
  std::vector<int> blocks;
  for (int i = 0; i < cnt; ++i) {
    const LevelDev& L = ms[i]->levels[levels[i]];
    p.push_back({x[i], y[i], L.items, ms[i]->d_prims, ms[i]->d_incs, L.n, L.slots_per_macro});
    blocks.push_back(L.n_items);
  }
  return launch_group<SumItems2>(p.data(), blocks.data(), cnt, s);
}

cudaError_t launch_apply(const Mesh& m, int level, int dtype, const void* x, void* y, cudaStream_t s,
                         cudaEvent_t ev_mid, const char** what) {
  const LevelDev& L = m.levels[level];
  if (dtype == 1 && !L.ff_ok) dtype = 3;  // weights outside the float-float range: native fp64
  cudaError_t e;
  if (m.dim == 2) {
    // one launch: macro-interior tiles and interface points side by side
    *what = "2D apply kernel";
    e = launch_apply2d(dtype, m, L, x, y, s);
    if (e != cudaSuccess) return e;
    if (ev_mid) {
      *what = "cudaEventRecord";
      e = cudaEventRecord(ev_mid, s);
    }
    return e;
  }
  *what = "3D apply kernel";
  const Mesh* mp = &m;
  e = launch_apply3d_group(dtype, false, &mp, &level, &x, &y, 1, s);
  if (e != cudaSuccess) return e;
  if (ev_mid) {
    *what = "cudaEventRecord";
    e = cudaEventRecord(ev_mid, s);
  }
  return e;
}

cudaError_t launch_apply_partial(const Mesh& m, int level, int dtype, const void* x, void* y, cudaStream_t s,
                                 const char** what) {
  const LevelDev& L = m.levels[level];
  if (dtype == 1 && !L.ff_ok) dtype = 3;  // weights outside the float-float range: native fp64
  if (m.dim == 2) {
    *what = "2D apply kernel (partial rows)";
    return launch_apply2d_partial(dtype, m, L, x, y, s);
  }
  *what = "3D apply kernel (partial rows)";
  const Mesh* mp = &m;
  return launch_apply3d_group(dtype, true, &mp, &level, &x, &y, 1, s);
}

}  // namespace hyteg
