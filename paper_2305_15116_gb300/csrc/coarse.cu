// The coarse levels of a 2D fp32 V-cycle in one kernel: a thread-block cluster
// per mesh runs every phase of the cycle from level `top` down to the direct
// solve on level 0 and back up, a cluster barrier between the phases.
//
// On these levels a phase is a launch, table loads and one round of gathers for well
// under a microsecond of work, and a cycle has eight phases per level.  In the
// cluster a phase costs its gathers and one hardware barrier.
//
// The vectors stay in global memory (L2): every load of a vector goes to L2
// (ld.cg), since other blocks of the cluster write it between barriers, whose
// release / acquire orders the writes.  The arithmetic is that of the separate
// launches, point by point (direct.cuh, lattice.cuh, transfer.cuh), so a cycle
// gives the same bits.
//
// Which levels (solver_setup): those that give every warp of the cluster at most
// one task of a phase, an interface item or 32 interior points, from level 1 up,
// and level 0 with at most a slot per thread.  A second round of tasks costs a
// phase's chain of loads again, while a launch spreads them over the device.  A
// cycle in us, all levels in launches / this rule / one task more per warp and so
// on up to 32768 slots: 2 macros level 4 68 / 52 / 52, level 7 109 / 98 / 106; 18
// macros level 4 67 / 63 / 63, level 5 81 / 79 / 85; 50 macros level 5 85 / 84 / 106;
// 128 macros level 4 72 / 73 / 122; 512 macros level 3 69 / 69 / 203; 2048 macros
// level 0 52 / 45 / 45 and level 2 104 / 95 / 437.
//
// 384 threads per block (1024 spilled: 156 us for a cycle of 128; 256: 131, 128:
// 150), 16 blocks (8: 142 us).  In 3D the launches stay: the gathers are twice as
// long and need the whole device (a level-5 solve 5.44 against 6.21 ms).
#include <vector>

#include "direct.cuh"
#include "per_device.h"
#include "transfer.cuh"

namespace hyteg {

namespace {

constexpr int CTHREADS = 384;

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ int cluster_rank() {
  int r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

struct CoarsePrm {
  const CoarseLev* lv;
  const float* b;  // of the top level
  float* u;
  const Inc* incs;
  const float* a0inv;
  const int *v_of_slot, *slot_of_v;
  int V, n_cells, top, nu1, nu2, first_done;
  float omega;
};
struct CoarseArgs {
  CoarsePrm p[kGroupMax];
};

struct Cycle {
  const CoarsePrm& p;
  int gw, nw, lane;  // this warp in the cluster, warps, lane

  __device__ __forceinline__ StencilPtr st(const CoarseLev& L) const {
    return StencilPtr{nullptr, L.st, nullptr, nullptr};
  }
  // y = sweep (MODE) of x with right-hand side b
  template <int MODE>
  __device__ __forceinline__ void sweep(const CoarseLev& L, const float* x, const float* b, float* y) const {
    const ModeArgs md{b, L.dinv, (double)p.omega};
    const int ch = (L.n_inner + 31) >> 5, tasks = L.n_ifi + p.n_cells * ch;
    for (int t = gw; t < tasks; t += nw) {
      if (t < L.n_ifi) {
        apply_item<2, MODE, false, true>(x, y, L.ifi[t], lane, p.incs, L.n, L.S, st(L), md);
        continue;
      }
      const int c = t - L.n_ifi, m = c / ch, i = (c - m * ch) * 32 + lane;
      if (i >= L.n_inner) continue;
      int slot, A;
      inner_point2(i, L.n, slot, A);
      const int64_t wb = (int64_t)m * (NCLS2 * NW2);
      InnerW<2, ArF32> W;
      W.load(st(L), wb);
      const int64_t s = (int64_t)m * L.S + slot;
      const float bi = __ldcg(b + s), di = MODE == MODE_JACOBI ? __ldg(L.dinv + s) : 0.0f;
      float uc;
      const float au = inner_row<2, ArF32, true>(x + s, Off7(0, A), W, st(L), wb, uc);
      y[s] = mode_out_staged<MODE, float>(au, uc, bi, di, (double)p.omega);
    }
  }
  // bc = P^T r; first: the coarse level's first sweep from zero, into uc
  __device__ __forceinline__ void restrict_to(const CoarseLev& F, const CoarseLev& C, bool first) const {
    float* const uc = first ? C.y : nullptr;
    auto row = [&](int cell, const Pt<2>& q) {
      return restrict_row<2, true, false>(F.r + (int64_t)cell * F.S, C.multinv + cell * NCLS2, q, F.n);
    };
    auto put = [&](int64_t s, float v) {
      C.b[s] = v;
      if (uc) uc[s] = __fmul_rn(__fmul_rn(p.omega, __ldg(C.dinv + s)), v);
    };
    const int ch = (C.n_inner + 31) >> 5, tasks = C.n_ifi + p.n_cells * ch;
    for (int t = gw; t < tasks; t += nw) {
      if (t < C.n_ifi) {
        const IfItem it = C.ifi[t];
        run_item<2, false, float>(
            it.work, lane, it.prim, p.incs, C.n, C.S, row, [](int64_t) { return 0.0f; },
            [](float a, int64_t) { return a; }, put);
        continue;
      }
      const int c = t - C.n_ifi, m = c / ch, i = (c - m * ch) * 32 + lane;
      if (i >= C.n_inner) continue;
      Pt<2> q;
      inner_point2(i, C.n, q.slot, q.A);
      q.q[1] = C.n + 1 - q.A;
      q.q[0] = q.slot - (q.q[1] * (C.n + 2) - ((q.q[1] * (q.q[1] + 1)) >> 1));
      q.q[2] = 0;
      q.M = C.n + 1;
      put((int64_t)m * C.S + q.slot, restrict_row<2, true, true>(F.r + (int64_t)m * F.S, C.multinv, q, F.n));
    }
  }
  __device__ __forceinline__ void prolong(const CoarseLev& C, const CoarseLev& F, float* uf) const {
    const int total = F.S * p.n_cells;
    for (int i = gw * 32 + lane; i < total; i += nw * 32) {
      const int cell = i / F.S;
      const unsigned v = __ldg(F.lpts + (i - cell * F.S));
      const int q[3] = {int(v & 0xFFFFu), int(v >> 16), 0};
      uf[i] = __ldcg(uf + i) + prolong_value<2, true>(C.u + (int64_t)cell * C.S, q, C.n);
    }
  }
  __device__ __forceinline__ void copy(float* dst, const float* src, int total) const {
    for (int i = gw * 32 + lane; i < total; i += nw * 32) dst[i] = src ? __ldcg(src + i) : 0.0f;
  }
  // level 0: u = A0^{-1} b on the coarse vertices, written to every copy, a thread
  // per slot; the right-hand side staged by every block, the sum over the vertices
  // in order
  __device__ __forceinline__ void level0(const float* b, float* u, float* sh) const {
    const int s = gw * 32 + lane;
    const bool live = s < p.n_cells * 3;
    const float* __restrict__ row = p.a0inv + (int64_t)(live ? __ldg(p.v_of_slot + s) : 0) * p.V;
    float acc = 0.0f;
    for (int j0 = 0; j0 < p.V; j0 += CTHREADS) {
      const int cnt = min(CTHREADS, p.V - j0);
      __syncthreads();
      if ((int)threadIdx.x < cnt) sh[threadIdx.x] = __ldcg(b + __ldg(p.slot_of_v + j0 + threadIdx.x));
      __syncthreads();
      if (live) {
#pragma unroll 8
        for (int j = 0; j < cnt; ++j) acc = __fmaf_rn(__ldg(row + j0 + j), sh[j], acc);
      }
    }
    if (live) u[s] = acc;
  }
};

__global__ void __launch_bounds__(CTHREADS, 1) k_coarse(const __grid_constant__ CoarseArgs g, int cluster) {
  __shared__ float sh[CTHREADS];
  __shared__ unsigned char in_u[32];  // per level: whether the smoothed iterate is in u
  pdl_trigger();
  const CoarsePrm& p = g.p[blockIdx.x / cluster];
  const Cycle C{p, cluster_rank() * (CTHREADS / 32) + (int)(threadIdx.x >> 5), cluster * (CTHREADS / 32),
                     (int)(threadIdx.x & 31)};
  pdl_wait();
  auto b_of = [&](int l) { return l == p.top ? p.b : (const float*)p.lv[l].b; };
  auto u_of = [&](int l) { return l == p.top ? p.u : p.lv[l].u; };
  bool done = p.first_done;
  for (int l = p.top; l > 0; --l) {
    const CoarseLev L = p.lv[l], Lc = p.lv[l - 1];
    const float* const b = b_of(l);
    float* const u = u_of(l);
    float* cur = done ? L.y : u;
    float* alt = done ? u : L.y;
    for (int i = done ? 1 : 0; i < p.nu1; ++i) {
      C.sweep<MODE_JACOBI>(L, cur, b, alt);
      cluster_sync();
      float* t = cur;
      cur = alt, alt = t;
    }
    C.sweep<MODE_RESIDUAL>(L, cur, b, L.r);
    if (threadIdx.x == 0) in_u[l] = cur == u;
    cluster_sync();
    const bool first = p.nu1 >= 1 && l - 1 > 0;
    C.restrict_to(L, Lc, first);
    if (!first && l - 1 > 0) C.copy(Lc.u, nullptr, Lc.S * p.n_cells);
    cluster_sync();
    done = first;
  }
  C.level0(b_of(0), u_of(0), sh);
  cluster_sync();
  for (int l = 1; l <= p.top; ++l) {
    const CoarseLev L = p.lv[l], Lc = p.lv[l - 1];
    const float* const b = b_of(l);
    float* const u = u_of(l);
    const bool inu = in_u[l];
    float* cur = inu ? u : L.y;
    float* alt = inu ? L.y : u;
    C.prolong(Lc, L, cur);
    cluster_sync();
    for (int i = 0; i < p.nu2; ++i) {
      C.sweep<MODE_JACOBI>(L, cur, b, alt);
      cluster_sync();
      float* t = cur;
      cur = alt, alt = t;
    }
    if (cur != u) {
      C.copy(u, cur, L.S * p.n_cells);
      cluster_sync();
    }
  }
}

// Blocks per cluster: 16 where the current device places such clusters, else 8.
cudaError_t cluster_size(int* size) {
  static PerDevice sizes;
  return sizes.get(size, [](int* v) {
    *v = 8;
    if (cudaFuncSetAttribute(k_coarse, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(16);
      cfg.blockDim = dim3(CTHREADS);
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = 16, at[0].val.clusterDim.y = 1, at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k_coarse, &cfg) == cudaSuccess && n > 0) *v = 16;
    }
    cudaGetLastError();
    return cudaSuccess;
  });
}

}  // namespace

cudaError_t launch_coarse_cycle(Mesh* const* ms, int cnt, int l, const float* const* b, float* const* u,
                                bool first_done, cudaStream_t s) {
  int cluster = 8;
  const cudaError_t ec = cluster_size(&cluster);
  if (ec != cudaSuccess) return ec;
  for (int i0 = 0; i0 < cnt; i0 += kGroupMax) {
    CoarseArgs g;
    const int k = cnt - i0 < kGroupMax ? cnt - i0 : kGroupMax;
    for (int i = 0; i < k; ++i) {
      const Mesh& m = *ms[i0 + i];
      const Solver& sv = *m.solver;
      g.p[i] = CoarsePrm{sv.coarse,     b[i0 + i], u[i0 + i],       m.d_incs, sv.a0inv32, sv.v_of_slot0, sv.slot_of_v0,
                         sv.nv0,        int(m.n_cells), l,          sv.nu1,   sv.nu2,     first_done ? 1 : 0,
                         float(sv.omega)};
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cluster * k));
    cfg.blockDim = dim3(CTHREADS);
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster, at[0].val.clusterDim.y = 1, at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_coarse, g, cluster);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t coarse_cycle_prepare(int* warps) {
  int size = 0;
  const cudaError_t e = cluster_size(&size);
  *warps = size * (CTHREADS / 32);
  return e;
}

}  // namespace hyteg
