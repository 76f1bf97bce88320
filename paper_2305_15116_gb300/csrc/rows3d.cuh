// 3D apply and sweeps of very fine macros: warps walk along rows.
//
// The march (march3d.cuh) stages a column range with its neighbour rows, 256 +
// 2n elements per slice for 256 columns: from n = 512 on mostly neighbour rows,
// and its ring leaves a block or two on an SM.  Here a warp takes 32 columns (30
// written) and up to 32 rows of one slice and walks up the rows: cp.async stages
// the next rows of slices z-1, z and z+1, a column per lane; three rows of each
// stay in registers, the x-1 / x+1 neighbours come by warp shuffles.  Every
// slice is read three times, mostly from L2, but nothing grows with n.
//
// What bounds it: the issue of its instructions (66 % at 13 warps per SM with 120
// registers in float-float, 65 % at 25 warps in fp32, L1 68 %), DRAM at 15 and 21 %.
// us per apply against the march: 6 macros level 8 228 / 264 and 69 / 113, level 9
// 1532 / 2061 and 471 / 863; further sizes at takes_rows3 (apply3d.cu).
//
// Macro-interior points only (x, y, z >= 1, x + y + z < n), whose neighbours all
// lie inside the macro: what a lane holds beyond a row's end reaches no written
// point.  Further blocks of the launch take the interface step (iface3d.cuh).
#pragma once

#include <type_traits>

#include "fallback.cuh"
#include "group.cuh"
#include "iface3d.cuh"
#include "one.cuh"

namespace hyteg {

constexpr int ROWS3_WIDTH = 30;  // written columns of a tile

// Offset of row r inside its slice's macro array, and its length.
struct RowCur {
  int off, len;
  __device__ __forceinline__ void init(int n, int z, int r) {
    const int M = n + 1 - z;
    off = slice_begin(n, M) + r * M - (r * (r - 1)) / 2;
    len = M - r;
  }
  __device__ __forceinline__ void next() {
    off += len;
    len -= 1;
  }
};

template <class P, int MODE>
struct Rows3 {
  using T = typename P::T;
  using V = typename P::V;
  using O = One<P>;
  static constexpr int kThreads = 256;
  static constexpr bool kLateWait = true;  // the tables first
  static constexpr bool kSweep = MODE == MODE_JACOBI || MODE == MODE_RESIDUAL;
  static constexpr int kRing = sizeof(T) == 4 ? 8 : 4;  // rows in flight per warp
  static constexpr int kArrays = kSweep ? 4 : 3;        // slices z, z+1, z-1; b
  struct Prm {
    const T* x;
    T* y;
    const int4* tiles;  // (x0, y0, y1, z) of a macro
    int n_tiles, n_if_blocks;
    int64_t n_warps;
    Iface3<T> f;
    StencilPtr st;
    ModeArgs md;
    int n;
    int64_t S;
  };
  struct Trip {
    V c, e, w;  // own column, x+1, x-1
  };
  struct Rec {
    Trip z, u, d;  // a row of slice z, z+1, z-1
    T x, b;        // sweeps: the value and b of slice z
  };

  static __device__ __forceinline__ void run(const Prm& p, int block, int) {
    if (block < p.n_if_blocks) {
      const int u = (kThreads / 32) * block + (int)(threadIdx.x >> 5);
      if (u < p.f.n_units) iface3d_unit<MODE, P::kPoison, T>(p.x, p.y, p.f, u, p.n, p.S, p.st, p.md);
      return;
    }
    __shared__ T ring_all[kThreads / 32][kRing][kArrays][32];
    const int64_t warp = ((int64_t)(block - p.n_if_blocks) * kThreads + threadIdx.x) >> 5;
    if (warp >= p.n_warps) return;  // whole warps leave together
    const int lane = threadIdx.x & 31, n = p.n;
    T(*ring)[kArrays][32] = ring_all[threadIdx.x >> 5];
    const int64_t m = warp / p.n_tiles;
    const int4 t = p.tiles[warp - m * p.n_tiles];
    const int z = t.w, c = t.x - 1 + lane;
    const T* const xm = p.x + m * p.S + c;
    const T* const bm = kSweep ? static_cast<const T*>(p.md.b) + m * p.S + c : nullptr;
    T* const ym = p.y + m * p.S + c;
    const int64_t wb = m * (int64_t)(NCLS3 * NW3);
    InnerW<3, P> W;
    W.load(p.st, wb);
    // inside a macro the inverse diagonal is one value
    const T di = MODE == MODE_JACOBI
                     ? __ldg(static_cast<const T*>(p.md.dinv) + m * p.S + slice_begin(n, n) + n + 1)  // (1, 1, 1)
                     : T(0);

    // rows t.y-1 .. t.z of the three slices are read; rows t.y .. t.z-1 of
    // slice z written
    const int steps = t.z - t.y + 2;
    RowCur sz, su, sd;  // the rows to stage
    sz.init(n, z, t.y - 1);
    su.init(n, z + 1, t.y - 1);
    sd.init(n, z - 1, t.y - 1);
    RowCur co = sz;  // the row to write
    co.next();
    pdl_wait();
    auto stage = [&](int slot) {
      if (c < sz.len) {
        cp_async_one(&ring[slot][0][lane], xm + sz.off);
        if constexpr (kSweep) cp_async_one(&ring[slot][3][lane], bm + sz.off);
      }
      if (c < su.len) cp_async_one(&ring[slot][1][lane], xm + su.off);
      if (c < sd.len) cp_async_one(&ring[slot][2][lane], xm + sd.off);
      sz.next();
      su.next();
      sd.next();
    };
#pragma unroll
    for (int k = 0; k < kRing; ++k) {
      if (k < steps) stage(k);
      cp_async_commit();
    }
    auto trip = [](V v) { return Trip{v, P::down(v), P::up(v)}; };
    auto take = [&](int k) -> Rec {
      cp_async_wait<kRing - 1>();
      const int slot = k & (kRing - 1);
      const T vz = ring[slot][0][lane], vu = ring[slot][1][lane], vd = ring[slot][2][lane];
      Rec r;
      if constexpr (kSweep) {
        r.x = vz;
        r.b = ring[slot][3][lane];
      }
      if (k + kRing < steps) stage(slot);
      cp_async_commit();
      r.z = trip(P::conv(vz));
      r.u = trip(P::conv(vu));
      r.d = trip(P::conv(vd));
      return r;
    };
    const bool writer = lane >= 1 && lane <= ROWS3_WIDTH;
    auto step = [&](const Rec& lo, const Rec& ce, const Rec& hi) {
      if (writer && c < co.len - 1) {
        typename O::Acc a;  // the order of roundings of the march and the direct kernel
        O::first(a, W.w[0], ce.z.c);
        O::sym(a, W.w[1], ce.z.e, ce.z.w);  // (1,0,0) + (-1,0,0)
        O::sym(a, W.w[2], hi.z.c, lo.z.c);  // (0,1,0) + (0,-1,0)
        O::sym(a, W.w[3], lo.z.e, hi.z.w);  // (1,-1,0) + (-1,1,0)
        O::sym(a, W.w[4], ce.u.c, ce.d.c);  // (0,0,1) + (0,0,-1)
        O::sym(a, W.w[5], ce.u.w, ce.d.e);  // (-1,0,1) + (1,0,-1)
        O::sym(a, W.w[6], lo.u.c, hi.d.c);  // (0,-1,1) + (0,1,-1)
        O::sym(a, W.w[7], lo.u.e, hi.d.w);  // (1,-1,1) + (-1,1,-1)
        T r = O::finish(a);
        if constexpr (P::kPoison) {  // an input outside the float-float range: native fp64 row
          if (O::bad(a)) r = native_row3d(xm - c, n, c, n + 1 - z - co.len, z, p.st.d + wb);
        }
        if constexpr (kSweep) r = mode_out_staged<MODE, T>(r, ce.x, ce.b, di, p.md.omega);
        ym[co.off] = r;
      }
      co.next();
    };
    // three records whose roles rotate
    Rec r0 = take(0), r1 = take(1), r2;
    for (int k = 2; k < steps; k += 3) {
      r2 = take(k);
      step(r0, r1, r2);
      if (k + 1 >= steps) break;
      r0 = take(k + 1);
      step(r1, r2, r0);
      if (k + 2 >= steps) break;
      r1 = take(k + 2);
      step(r2, r0, r1);
    }
    cp_async_wait<0>();
  }
};

}  // namespace hyteg
