// 3D apply and sweeps (15-point Kuhn stencil): one launch completes the
// macro-interior and the interface points (iface3d.cuh).  Large vectors march
// columns through the slices (march3d.cuh); small ones take the direct form
// below, one thread per macro-interior point, neighbours straight from memory.
//
// The 15-point Kuhn stencil in the direct form reads every value 15 times,
// through L1 and L2; on a level whose vector stays in L2 what counts is the
// length of the chain of dependent loads, and here it is one table entry
// (read before the previous kernel has finished) and one round of loads.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "direct.cuh"
#include "march3d.cuh"
#include "per_device.h"
#include "rows3d.cuh"

namespace hyteg {

namespace {

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
    int n_if_blocks;
    Iface3<T> f;
    StencilPtr st;
    ModeArgs md;
    int n;
    int64_t S;
  };
  static __device__ __forceinline__ void run(const Prm& p, int block, int) {
    if (block < p.n_if_blocks) {
      const int u = (kThreads / 32) * block + (int)(threadIdx.x >> 5);
      if (u < p.f.n_units) iface3d_unit<MODE, P::kPoison, T>(p.x, p.y, p.f, u, p.n, p.S, p.st, p.md);
      return;
    }
    const int b = block - p.n_if_blocks;
    const int m = b / p.bpm;
    const int t = (b - m * p.bpm) * kThreads + (int)threadIdx.x;
    if (t >= p.n_pts) return;
    const int2 e = p.pts[t];
    const int64_t wb = (int64_t)m * (NCLS3 * NW3);
    InnerW<3, P> W;
    W.load(p.st, wb);
    const Off15 o(e.y >> 16, e.y & 0xFFFF);
    const int64_t i = (int64_t)m * p.S + e.x;
    pdl_wait();
    T bi = T(0), di = T(0), uc;
    if (MODE == MODE_JACOBI || MODE == MODE_RESIDUAL) bi = ld<false>(static_cast<const T*>(p.md.b) + i);
    if (MODE == MODE_JACOBI) di = __ldg(static_cast<const T*>(p.md.dinv) + i);
    const T r = inner_row<3, P, false>(p.x + i, o, W, p.st, wb, uc);
    p.y[i] = mode_out_staged<MODE, T>(r, uc, bi, di, p.md.omega);
  }
};

template <class T>
const T* face_table(const LevelDev& L);
template <>
const double* face_table<double>(const LevelDev& L) {
  return L.wf64;
}
template <>
const float* face_table<float>(const LevelDev& L) {
  return L.wf32;
}

template <class T>
Iface3<T> iface_of(const Mesh& m, const LevelDev& L) {
  Iface3<T> f;
  f.items = L.ifi;
  f.n_items = L.n_ifi_ev;
  f.per_face = std::max(1, (L.n_face_pts + 31) / 32);
  f.n_pts = L.n_face_pts;
  f.n_units = L.n_ifi_ev + f.per_face * L.n_face3;
  f.faces = L.face3;
  f.ab = L.face_ab;
  f.incs = m.d_incs;
  f.wf = face_table<T>(L);
  return f;
}

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
    p.f = iface_of<T>(m, L);
    p.st = StencilPtr{L.st64, L.st32, L.st_hi, L.st_lo};
    p.md = md ? md[i] : ModeArgs{nullptr, nullptr, 0.0};
    p.n = L.n;
    p.S = L.slots_per_macro;
    p.n_if_blocks = (p.f.n_units + B::kThreads / 32 - 1) / (B::kThreads / 32);
    prm.push_back(p);
    blocks.push_back(p.n_if_blocks + p.bpm * int(m.n_cells));
  }
  return launch_group<B>(prm.data(), blocks.data(), count, s);
}

// Work of the columns' march over one macro pair: (first column, z0, z1, -)
// per block, the longest first; the largest extent of a block's columns with
// their neighbour rows, in elements.
struct MarchList {
  std::vector<int4> work;
  int stride = 32;
};
MarchList march_list(int n, int chunks, bool dense) {
  MarchList r;
  auto row = [](int64_t t) {
    int64_t j = int64_t((std::sqrt(8.0 * double(t) + 1.0) - 1.0) / 2.0);
    while (j * (j + 1) / 2 > t) --j;
    while ((j + 1) * (j + 2) / 2 <= t) ++j;
    return int(j);
  };
  std::vector<std::pair<int64_t, int4>> items;
  for (const int4& z : z_ranges(n, chunks)) {
    const int zlo = std::max(1, z.y), kmax = n - 1 - zlo;
    if (kmax < 2 || z.z <= zlo) continue;
    // columns of rows 2 .. kmax: dense, the interior ones; else all as they lie
    const int first = dense ? 0 : 3, end = dense ? kmax * (kmax - 1) / 2 : (kmax + 1) * (kmax + 2) / 2;
    const int all = dense ? (n - 2) * (n - 3) / 2 : 0x7FFFFFFF;
    for (int t = first; t < end; t += MARCH_COLS) {
      int k0, k1, q0, q1;
      if (dense) {
        const int u = std::min(t + MARCH_COLS, all) - 1;
        k0 = row(t) + 2, k1 = row(u) + 2;
        q0 = k0 * (k0 + 1) / 2 + 1 + t - (k0 - 2) * (k0 - 1) / 2;
        q1 = k1 * (k1 + 1) / 2 + 1 + u - (k1 - 2) * (k1 - 1) / 2;
      } else {
        q0 = t, q1 = t + MARCH_COLS - 1;
        k0 = row(q0), k1 = row(q1);
      }
      r.stride = std::max(r.stride, (q1 + k1 + 2) - (q0 - k0 - 1) + 1);
      const int64_t len = std::min(z.z - 1, n - 1 - k0) - zlo + 3;
      items.push_back({len, make_int4(t, z.y, z.z, 0)});
    }
  }
  std::stable_sort(items.begin(), items.end(), [](const auto& a, const auto& b) { return a.first > b.first; });
  for (const auto& i : items) r.work.push_back(i.second);
  return r;
}

constexpr size_t kSmemMax = 226 * 1024;  // beside the 128 B of static shared memory
// macro pairs whose blocks lie together: about so many blocks (a few per
// SM), so that a column range finds its neighbour rows in L2
constexpr int kChunkBlocks = 4096;
// below so many march blocks the interface step takes blocks of its own
constexpr int kOwnIfaceBlocks = 1024;

template <class P, int MODE, int STRIDE>
cudaError_t march_attr() {
  using B = March3<P, MODE, STRIDE>;
  static_assert(B::smem_bytes() <= kSmemMax, "the ring does not fit");
  static PerDevice set;
  int value = 0;
  return set.get(&value, [](int*) {
    cudaError_t err =
        cudaFuncSetAttribute(k_group<B, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)B::smem_bytes());
    if constexpr (STRIDE <= 512) {
      if (err == cudaSuccess)
        err = cudaFuncSetAttribute(k_group<B, kGroupMax>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)B::smem_bytes());
    }
    return err;
  });
}

template <class P, int MODE, int STRIDE>
cudaError_t launch_march_s(const Mesh* const* ms, const int* levels, const void* const* xs, void* const* ys,
                           const ModeArgs* md, int count, cudaStream_t s, const March3Work* over) {
  using B = March3<P, MODE, STRIDE>;
  using T = typename P::T;
  constexpr int dt = sizeof(T) == 4 ? 2 : (P::kPoison ? 1 : 3);
  const cudaError_t attr = march_attr<P, MODE, STRIDE>();
  if (attr != cudaSuccess) return attr;
  std::vector<typename B::Prm> prm;
  std::vector<int> blocks;
  for (int i = 0; i < count; ++i) {
    const Mesh& m = *ms[i];
    const LevelDev& L = m.levels[levels[i]];
    const March3Work& w = over ? *over : L.march[dt];
    typename B::Prm p;
    p.x = static_cast<const T*>(xs[i]);
    p.y = static_cast<T*>(ys[i]);
    p.work = w.work;
    p.n_work = w.n_work;
    p.n_cells = int(m.n_cells);
    p.n_pairs = int((m.n_cells + 1) / 2);
    p.per_chunk = std::max(1, std::min(p.n_pairs, (kChunkBlocks + w.n_work - 1) / std::max(1, w.n_work)));
    p.f = iface_of<T>(m, L);
    p.st = StencilPtr{L.st64, L.st32, L.st_hi, L.st_lo};
    p.md = md ? md[i] : ModeArgs{nullptr, nullptr, 0.0};
    p.n = L.n;
    p.S = L.slots_per_macro;
    // n >= 4: there are points to march over, and a list that holds them
    if (w.stride > STRIDE || (w.n_work == 0 && L.n >= 4)) return cudaErrorInvalidValue;
    p.n_march = int64_t(p.n_work) * p.n_pairs;
    const int64_t all = p.n_march + (p.n_march < kOwnIfaceBlocks ? (p.f.n_units + 7) / 8 : 0);
    if (all > 0x7FFFFFFF) return cudaErrorInvalidValue;
    prm.push_back(p);
    blocks.push_back(int(all));
  }
  if constexpr (STRIDE <= 512) return launch_group<B>(prm.data(), blocks.data(), count, s, B::smem_bytes());
  cudaError_t e = cudaSuccess;  // large levels fill the device each by itself
  for (int i = 0; i < count && e == cudaSuccess; ++i) e = launch_one<B>(prm[i], blocks[i], s, B::smem_bytes());
  return e;
}

// The slot size is a constant of the kernel: the columns of a block with their
// neighbour rows, 256 + 2n, for n up to 128; native fp64, which has the point table
// up to there, for level 8.
template <class P, int MODE>
cudaError_t launch_march(const Mesh* const* ms, const int* levels, const void* const* xs, void* const* ys,
                         const ModeArgs* md, int count, cudaStream_t s, const March3Work* over) {
  return launch_march_s<P, MODE, std::is_same<P, ArF64Native>::value ? 1280 : 512>(ms, levels, xs, ys, md, count, s,
                                                                                   over);
}

template <class P, int MODE>
cudaError_t launch_rows(const Mesh* const* ms, const int* levels, const void* const* xs, void* const* ys,
                        const ModeArgs* md, int count, cudaStream_t s) {
  using B = Rows3<P, MODE>;
  using T = typename P::T;
  for (int i = 0; i < count; ++i) {  // such levels fill the device each by itself
    const Mesh& m = *ms[i];
    const LevelDev& L = m.levels[levels[i]];
    typename B::Prm p;
    p.x = static_cast<const T*>(xs[i]);
    p.y = static_cast<T*>(ys[i]);
    p.tiles = L.tiles3;
    p.n_tiles = L.n_tiles3;
    p.n_warps = int64_t(L.n_tiles3) * m.n_cells;
    p.f = iface_of<T>(m, L);
    p.st = StencilPtr{L.st64, L.st32, L.st_hi, L.st_lo};
    p.md = md ? md[i] : ModeArgs{nullptr, nullptr, 0.0};
    p.n = L.n;
    p.S = L.slots_per_macro;
    p.n_if_blocks = (p.f.n_units + B::kThreads / 32 - 1) / (B::kThreads / 32);
    const int64_t blocks = p.n_if_blocks + (p.n_warps * 32 + B::kThreads - 1) / B::kThreads;
    if (L.n_tiles3 == 0 || blocks > 0x7FFFFFFF) return cudaErrorInvalidValue;
    const cudaError_t e = launch_one<B>(p, int(blocks), s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// The members whose vectors are small take the direct kernel, the others the
// march or the rows (takes_rows3); each kind shares its launches.
template <class P, int MODE>
cudaError_t launch_t(const Mesh* const* ms, const int* levels, const void* const* xs, void* const* ys,
                     const ModeArgs* md, int count, cudaStream_t s) {
  // native fp64 is bound by the fp64 pipe either way, and the direct kernel's
  // occupancy suits it better (level 6, 384 macro-tets: 488 against 600 us)
  constexpr bool native = std::is_same<P, ArF64Native>::value;
  constexpr int dt = sizeof(typename P::T) == 4 ? 2 : (native ? 3 : 1);
  auto kind = [](const LevelDev& L) { return L.direct3 || (native && L.pts3) ? 0 : L.rows3[dt] ? 2 : 1; };
  auto go = [&](int k, const Mesh* const* m, const int* l, const void* const* x, void* const* y, const ModeArgs* a,
                int cnt) {
    return k == 0   ? launch_direct<P, MODE>(m, l, x, y, a, cnt, s)
           : k == 1 ? launch_march<P, MODE>(m, l, x, y, a, cnt, s, nullptr)
                    : launch_rows<P, MODE>(m, l, x, y, a, cnt, s);
  };
  if (count == 1) return go(kind(ms[0]->levels[levels[0]]), ms, levels, xs, ys, md, 1);
  for (int k = 0; k < 3; ++k) {
    std::vector<const Mesh*> mm;
    std::vector<int> lv;
    std::vector<const void*> xx;
    std::vector<void*> yy;
    std::vector<ModeArgs> mo;
    for (int i = 0; i < count; ++i) {
      if (kind(ms[i]->levels[levels[i]]) != k) continue;
      mm.push_back(ms[i]);
      lv.push_back(levels[i]);
      xx.push_back(xs[i]);
      yy.push_back(ys[i]);
      if (md) mo.push_back(md[i]);
    }
    if (mm.empty()) continue;
    const cudaError_t e = go(k, mm.data(), lv.data(), xx.data(), yy.data(), md ? mo.data() : nullptr, int(mm.size()));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int MODE>
cudaError_t launch_dt(int dtype, const Mesh* const* ms, const int* levels, const void* const* xs, void* const* ys,
                      int count, cudaStream_t s) {
  switch (dtype) {
    case 1: return launch_t<ArF64FF, MODE>(ms, levels, xs, ys, nullptr, count, s);
    case 2: return launch_t<ArF32, MODE>(ms, levels, xs, ys, nullptr, count, s);
    case 3: return launch_t<ArF64Native, MODE>(ms, levels, xs, ys, nullptr, count, s);
    default: return cudaErrorInvalidValue;
  }
}

// Sum of the copies' partial rows that y holds (Dirichlet points: y = x).
template <class T>
struct Sum3 {
  static constexpr int kThreads = 256;
  static constexpr bool kLateWait = true;
  struct Prm {
    const T* x;
    T* y;
    const IfItem* items;
    int n_items;
    const Inc* incs;
    int n;
    int64_t S;
  };
  static __device__ __forceinline__ void run(const Prm& p, int block, int) {
    const int item = (kThreads / 32) * block + (int)(threadIdx.x >> 5);
    if (item >= p.n_items) return;
    const IfItem it = p.items[item];
    pdl_wait();
    run_item<3, false, T>(
        it.work, (int)(threadIdx.x & 31), it.prim, p.incs, p.n, p.S,
        [&](int cell, const Pt<3>& q) { return p.y[(int64_t)cell * p.S + q.slot]; },
        [&](int64_t s) { return ld<false>(p.x + s); }, [&](T a, int64_t) { return a; },
        [&](int64_t s, T v) { p.y[s] = v; });
  }
};

}  // namespace

cudaError_t launch_apply3d_group(int dtype, bool partial, const Mesh* const* ms, const int* levels,
                                 const void* const* xs, void* const* ys, int count, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  return partial ? launch_dt<MODE_PARTIAL>(dtype, ms, levels, xs, ys, count, s)
                 : launch_dt<MODE_APPLY>(dtype, ms, levels, xs, ys, count, s);
}

cudaError_t launch_sweep3d_group(bool jacobi, const Mesh* const* ms, const int* levels, const void* const* u,
                                 const void* const* b, const void* const* dinv, const double* omega,
                                 void* const* out, int count, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  std::vector<ModeArgs> md(count);
  for (int i = 0; i < count; ++i) md[i] = ModeArgs{b[i], dinv[i], omega[i]};
  return jacobi ? launch_t<ArF32, MODE_JACOBI>(ms, levels, u, out, md.data(), count, s)
                : launch_t<ArF32, MODE_RESIDUAL>(ms, levels, u, out, md.data(), count, s);
}

cudaError_t launch_march3d_work(int dtype, const Mesh& m, int level, const March3Work& work, const void* x, void* y,
                                cudaStream_t s) {
  const Mesh* mp = &m;
  switch (dtype) {
    case 1: return launch_march<ArF64FF, MODE_APPLY>(&mp, &level, &x, &y, nullptr, 1, s, &work);
    case 2: return launch_march<ArF32, MODE_APPLY>(&mp, &level, &x, &y, nullptr, 1, s, &work);
    case 3: return launch_march<ArF64Native, MODE_APPLY>(&mp, &level, &x, &y, nullptr, 1, s, &work);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_sum_copies3d(const Mesh* const* ms, const int* levels, const double* const* xs, double* const* ys,
                                int count, cudaStream_t s) {
  using B = Sum3<double>;
  std::vector<B::Prm> prm;
  std::vector<int> blocks;
  for (int i = 0; i < count; ++i) {
    const LevelDev& L = ms[i]->levels[levels[i]];
    prm.push_back({xs[i], ys[i], L.ifi, L.n_ifi, ms[i]->d_incs, L.n, L.slots_per_macro});
    blocks.push_back((L.n_ifi + B::kThreads / 32 - 1) / (B::kThreads / 32));
  }
  return launch_group<B>(prm.data(), blocks.data(), count, s);
}

cudaError_t apply3d_prepare(int n) {
  if (n > 128) return cudaSuccess;
  const cudaError_t e = march_attr<ArF64FF, MODE_APPLY, 512>();
  return e == cudaSuccess ? march_attr<ArF32, MODE_APPLY, 512>() : e;
}

// us per apply, rows / march: float-float and fp32 on level 8, 1 macro 45 / 90 and
// 15 / 29, 6 macros 228 / 264 and 69 / 113, 48 macros 1804 / 2133 and 556 / 953; on
// level 7, 5 macros 41 / 46 and 15 / 18, 9 macros 62 / 46 and 20 / 18.  Native fp64
// on level 8, even numbers of macros 595 / 546 (6), odd ones, whose last pair of
// the march is half empty, 119 / 202 (1), 499 / 544 (5), 1457 / 1456 (15); on level
// 9, 6 macros 4228 / 4242.
bool takes_rows3(int n, int64_t n_cells, int dt) {
  if (dt == 3) return n >= 512 || (n >= 256 && n_cells % 2 && n_cells < 16);
  return n >= 256 || (n >= 128 && slots_per_macro(3, 7) * n_cells <= kRows3Slots);
}

std::vector<int4> tile_list_rows3(int n) {
  // chunks of 32 rows (level 7, 384 macro-tets: 3.94 -> 3.50 ms float-float and
  // 1.16 -> 1.11 ms fp32 against 64; a warp walks its rows serially)
  constexpr int kRows = 32;
  std::vector<int4> t;
  for (int z = 1; z <= n - 3; ++z) {
    const int M = n + 1 - z;
    for (int x0 = 1; x0 <= M - 3; x0 += ROWS3_WIDTH)
      for (int y0 = 1; y0 <= M - 2 - x0; y0 += kRows)
        t.push_back(make_int4(x0, y0, std::min(y0 + kRows, M - 1 - x0), z));
  }
  return t;
}

void march3d_lists(int n, int chunks, int dtype, std::vector<int4>& work, int& stride) {
  MarchList l = march_list(n, chunks, dtype == 1);
  work = std::move(l.work);
  stride = l.stride;
}

}  // namespace hyteg
