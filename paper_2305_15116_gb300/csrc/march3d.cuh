// 3D apply and sweeps of large vectors: columns of a macro marched through its
// slices.
//
// A macro array stacks triangular slices; slice z (side M = n+1-z) is one
// contiguous range.  Count the points of a slice from its END: point q lies
// on row k from the apex (q = k(k+1)/2 + j, 0 <= j <= k; row k holds k+1
// points; x = k - j, y = n-z-k).  The same q in the next slice is the point
// (x, y-1, z+1): a column of constant q runs along the Kuhn direction
// (0,-1,1), and every neighbour offset depends on the column's k alone
// (A = k+1):
//   slice z:   q, q -+ 1, q -+ A, q + A+1, q - A+1
//   slice z+1: (0,0,1) q-A, (-1,0,1) q-A+1, (0,-1,1) q, (1,-1,1) q-1
//   slice z-1: (0,0,-1) q+A+1, (1,0,-1) q+A, (0,1,-1) q, (-1,1,-1) q+1
// so the 15 points lie at 7 offsets q, each read from a slice once: a thread
// owns a column, reads 7 values of every slice from shared memory, finishes
// the point of the slice before with the four it needs "above", begins the
// point of this slice, and keeps the four that the next but one needs
// "below" in registers.  No point's position is decoded after the start, and
// a column costs no work outside the macro.
//
// Measured (us per apply, this kernel with its interface step / the kernels
// before it, which decoded each slice's points by index with 15 shared loads
// each, or above n = 64 walked along rows, and summed the interface in a launch
// of their own): level 6, 384 macro-tets float-float 235 / 298, fp32 86 / 131;
// level 7, 72 macro-tets 269 / 572, 94 / 244.  Executed instructions per slot:
// float-float 331 -> 160, fp32 181 -> 54 (level 7); without the interface step
// 157 and 47 us at level 6.  What bounds it: latency between the barriers with 16 warps per SM
// in float-float, 24 in fp32 (issue 40 / 50 %, L1 and shared memory 55 / 63 %;
// more blocks per SM with fewer registers ran slower), and the interface
// points' gathers, whose rows lie a slice apart.
//
// A block takes MARCH_COLS columns of TWO macros over a range of slices.  The
// macros' refinements are congruent, so the positions, predicates and
// addresses serve both, and the two points form the halves of packed f32x2
// operations without a register move.  The column range with its neighbour
// rows is one contiguous piece of every slice; cp.async stages the next slices
// into a ring, float-float values are split once per block (while the slice
// before is computed) into (hA, hB, lA, lB) quadruples.  One barrier per slice.
//
// Lane order: for float-float the interior columns are numbered densely (no
// idle lane); in fp32, which the shared-memory loads bound, columns are taken
// as they lie, so that a warp's loads fall on 32 consecutive words.
#pragma once

#include <type_traits>

#include "fallback.cuh"
#include "group.cuh"
#include "iface3d.cuh"

namespace hyteg {

constexpr int MARCH_COLS = 256;

// Values, weights and accumulators of two macros.
template <class P>
struct Two;
template <>
struct Two<ArF32> {
  using V = f2_t;
  using W = f2_t;
  struct Acc {
    f2_t s;
  };
  static constexpr bool kSplit = false;
  static __device__ __forceinline__ W weight(const StencilPtr& st, int64_t a, int64_t b) {
    return f2_pack(__ldg(st.f + a), __ldg(st.f + b));
  }
  static __device__ __forceinline__ V get(const float* a, const float* b) { return f2_pack(*a, *b); }
  static __device__ __forceinline__ void first(Acc& a, const W& w, const V& v) { a.s = f2_mul(w, v); }
  static __device__ __forceinline__ void sym(Acc& a, const W& w, const V& u, const V& v) {
    a.s = f2_fma(w, f2_add(u, v), a.s);
  }
  static __device__ __forceinline__ void finish(const Acc& a, float& ra, float& rb) { f2_unpack(a.s, ra, rb); }
  static __device__ __forceinline__ void value(const V& v, float& a, float& b) { f2_unpack(v, a, b); }
};
template <>
struct Two<ArF64Native> {
  using V = double2;
  using W = double2;
  struct Acc {
    double2 s;
  };
  static constexpr bool kSplit = false;
  static __device__ __forceinline__ W weight(const StencilPtr& st, int64_t a, int64_t b) {
    return make_double2(__ldg(st.d + a), __ldg(st.d + b));
  }
  static __device__ __forceinline__ V get(const double* a, const double* b) { return make_double2(*a, *b); }
  static __device__ __forceinline__ void first(Acc& a, const W& w, const V& v) {
    a.s = make_double2(__dmul_rn(w.x, v.x), __dmul_rn(w.y, v.y));
  }
  static __device__ __forceinline__ void sym(Acc& a, const W& w, const V& u, const V& v) {
    a.s.x = __fma_rn(w.x, __dadd_rn(u.x, v.x), a.s.x);
    a.s.y = __fma_rn(w.y, __dadd_rn(u.y, v.y), a.s.y);
  }
  static __device__ __forceinline__ void finish(const Acc& a, double& ra, double& rb) {
    ra = a.s.x;
    rb = a.s.y;
  }
  static __device__ __forceinline__ void value(const V& v, double& a, double& b) {
    a = v.x;
    b = v.y;
  }
};
template <>
struct Two<ArF64FF> {
  using V = ArF64FF::P2;
  struct W {
    f2_t h, l;
  };
  using Acc = ArF64FF::Acc;
  static constexpr bool kSplit = true;
  static __device__ __forceinline__ W weight(const StencilPtr& st, int64_t a, int64_t b) {
    return W{f2_pack(__ldg(st.hi + a), __ldg(st.hi + b)), f2_pack(__ldg(st.lo + a), __ldg(st.lo + b))};
  }
  static __device__ __forceinline__ V get(const ulonglong2* p) {
    const ulonglong2 v = *p;
    return V{v.x, v.y};
  }
  // the roundings of ArF64FF::first / add / add_sym, with a weight per half
  static __device__ __forceinline__ f2_t neg_products(const W& w, const f2_t& vh) {
    float va, vb, wa, wb;
    f2_unpack(vh, va, vb);
    f2_unpack(w.h, wa, wb);
    return f2_pack(__fmul_rn(-wa, va), __fmul_rn(-wb, vb));
  }
  static __device__ __forceinline__ void first(Acc& a, const W& w, const V& v) {
    const f2_t pm = neg_products(w, v.h);
    a.s = f2_sub(f2_pack(0.0f, 0.0f), pm);
    f2_t e = f2_fma(w.h, v.h, pm);
    e = f2_fma(w.h, v.l, e);
    a.e = f2_fma(w.l, v.h, e);
  }
  static __device__ __forceinline__ void sym(Acc& a, const W& w, const V& u, const V& v) {
    const f2_t sh = f2_add(u.h, v.h);
    const f2_t bb = f2_sub(sh, u.h);
    const f2_t er = f2_add(f2_sub(u.h, f2_sub(sh, bb)), f2_sub(v.h, bb));
    const f2_t sl = f2_add(f2_add(u.l, v.l), er);
    f2_t e = f2_fma(w.h, sl, a.e);
    const f2_t pm = neg_products(w, sh);
    e = f2_fma(w.l, sh, e);
    const f2_t sn = f2_sub(a.s, pm);
    const f2_t nbp = f2_sub(a.s, sn);
    const f2_t t2 = f2_sub(a.s, f2_add(sn, nbp));
    a.s = sn;
    e = f2_add(e, f2_fma(w.h, sh, nbp));
    a.e = f2_add(e, t2);
  }
  static __device__ __forceinline__ void finish(const Acc& a, double& ra, double& rb) { ArF64FF::finish(a, ra, rb); }
};

// the row of point t of a triangle with rows of 1, 2, 3, .. points
__device__ __forceinline__ int apex_row(int t) {
  int j = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (j * (j + 1) / 2 > t) --j;
  while ((j + 1) * (j + 2) / 2 <= t) ++j;
  return j;
}

// Kept out of line: a rare call that would otherwise cost the march registers.
__device__ __noinline__ double march_native_row(const double* xm, int n, int px, int py, int pz, const double* w) {
  return native_row3d(xm, n, px, py, pz, w);
}

// STRIDE: elements of a slot per macro, the largest extent of a block's
// columns with their neighbour rows.
template <class P, int MODE, int STRIDE>
struct March3 {
  using T = typename P::T;
  using Q = Two<P>;
  static constexpr bool kSplit = Q::kSplit;
  static constexpr bool kDense = kSplit;
  static constexpr int kThreads = MARCH_COLS;
  static constexpr bool kLateWait = true;  // the tables first
  // slices in the ring; float-float: split slices kept, from which the values
  // "below" are read again (32 registers fewer)
  static constexpr int kPlanes = kSplit ? 4 : 0;
  static constexpr bool kReread = kSplit;
  static constexpr int kDepth = kReread ? 4 : sizeof(T) == 4 ? 6 : 3;
  // fp32: three blocks per SM.  At four the 64 registers spill around the
  // interface step and in the marching (level 7, 72 macro-tets: 105 against 94 us).
  static constexpr int kMinBlocks = STRIDE > 512 ? 1 : sizeof(T) == 4 ? 3 : 2;
  static constexpr int kRounds = (STRIDE + MARCH_COLS - 1) / MARCH_COLS;
  static constexpr bool kSweep = MODE == MODE_JACOBI || MODE == MODE_RESIDUAL;
  struct Prm {
    const T* x;
    T* y;
    const int4* work;  // (first column, z0, z1, -), the longest first
    int n_work, n_pairs, n_cells;
    int per_chunk;     // macro pairs whose blocks are neighbours in the launch
    int64_t n_march;   // blocks that march; further ones take the interface step
    Iface3<T> f;
    StencilPtr st;
    ModeArgs md;
    int n;
    int64_t S;
  };
  // shared memory: ring [kDepth][2][STRIDE] T, float-float planes [kPlanes][STRIDE] 16 B
  static constexpr size_t smem_bytes() {
    return (size_t)STRIDE * (2 * (size_t)kDepth * sizeof(T) + kPlanes * 16);
  }

  static __device__ __forceinline__ void run(const Prm& p, int idx, int nb) {
    if (idx >= p.n_march) {
      const int u = (int)(idx - p.n_march) * (MARCH_COLS / 32) + (int)(threadIdx.x >> 5);
      if (u < p.f.n_units) iface3d_unit<MODE, P::kPoison, T>(p.x, p.y, p.f, u, p.n, p.S, p.st, p.md);
      return;
    }
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = threadIdx.x;
    const int n = p.n;
    // block -> chunk of pairs, work entry, pair
    const int chunk = idx / (p.n_work * p.per_chunk);
    const int rest = idx - chunk * (p.n_work * p.per_chunk);
    const int in_chunk = min(p.per_chunk, p.n_pairs - chunk * p.per_chunk);
    const int wi = rest / in_chunk;
    const int pair = chunk * p.per_chunk + (rest - wi * in_chunk);
    const int4 wk = p.work[wi];
    const int m0 = 2 * pair, m1 = min(2 * pair + 1, p.n_cells - 1);
    const bool two = m1 > m0;

    // this thread's column and the block's range of columns
    int k, q, k0, q0, k1, q1;  // own, first, last
    bool live;
    if (kDense) {  // interior columns: rows k = 2 .. n-2, j = 1 .. k-1
      const int nt = (n - 3) * (n - 2) / 2;
      auto col = [&](int t, int& kk, int& qq) {
        const int j = apex_row(t);
        kk = j + 2;
        qq = kk * (kk + 1) / 2 + 1 + (t - j * (j + 1) / 2);
      };
      live = wk.x + tid < nt;
      col(min(wk.x + tid, nt - 1), k, q);
      col(wk.x, k0, q0);
      col(min(wk.x + MARCH_COLS, nt) - 1, k1, q1);
    } else {
      q = wk.x + tid;
      k = apex_row(q);
      const int j = q - k * (k + 1) / 2;
      live = j >= 1 && j <= k - 1 && k <= n - 2;
      q0 = wk.x;
      k0 = apex_row(q0);
      q1 = wk.x + MARCH_COLS - 1;
      k1 = apex_row(q1);
    }
    const int A = k + 1;
    const int qmin = q0 - (k0 + 1), qmax = q1 + k1 + 2;
    const int zlo = max(1, wk.y);
    const int zhi = live ? min(wk.z - 1, n - 1 - k) : -2;    // this column's last point
    const int s0 = zlo - 1;
    const int s1 = min(wk.z, n - max(k0, 2));                // last slice read by the block
    const int sw = min(s1, __reduce_max_sync(0xFFFFFFFFu, zhi) + 1);  // and by this warp

    const int64_t wa = (int64_t)m0 * (NCLS3 * NW3), wb = (int64_t)m1 * (NCLS3 * NW3);
    // weights: the centre's, then one per pair of opposite neighbours; 8-byte
    // types read them from shared memory (broadcast), whose 32 registers decide
    // how many blocks fit
    __shared__ __align__(16) typename Q::W wsm[8];
    typename Q::W wreg[8];
    constexpr bool kWSmem = sizeof(T) == 8;
    {
      const int slot_of[8] = {0, 1, 3, 5, 7, 8, 9, 10};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (kWSmem) {
          if (tid == i) wsm[i] = Q::weight(p.st, wa + slot_of[i], wb + slot_of[i]);
        } else {
          wreg[i] = Q::weight(p.st, wa + slot_of[i], wb + slot_of[i]);
        }
      }
    }
    auto W = [&](int i) -> typename Q::W { return kWSmem ? wsm[i] : wreg[i]; };
    const T* const xa = p.x + (int64_t)m0 * p.S;
    const T* const xb = p.x + (int64_t)m1 * p.S;

    T* const ring = reinterpret_cast<T*>(smem);
    ulonglong2* const planes = reinterpret_cast<ulonglong2*>(smem + (size_t)STRIDE * 2 * kDepth * sizeof(T));

    // Element e of a slot is column qmax - e; slice z holds the columns
    // q < c(z) = M(M+1)/2, the last slot of slice z is E(z).
    auto count = [&](int z) { return (n + 1 - z) * (n + 2 - z) / 2; };
    const int64_t N1 = n + 1, B1 = N1 - s0;
    const int c0 = count(s0);
    const int E0 = (int)((N1 * (N1 + 1) * (N1 + 2) - B1 * (B1 + 1) * (B1 + 2)) / 6) + c0 - 1;
    // The elements e = tid + r MARCH_COLS, qmax - c(z) < e <= emax, are staged
    // (and split) by this thread: one bound for the tests of all of them, and
    // the second macro's addresses as an offset, which kept 18 registers free.
    const int emax = qmax - max(qmin, 0);
    const int below = emax - tid;
    auto staged = [&](int r, int cz) { return (unsigned)(below - r * MARCH_COLS) < (unsigned)max(cz + emax - qmax, 0); };
    const int pair_off = two ? (int)p.S : 0;
    int z_st = s0, c_st = c0;  // the next slice to stage
    const T* ga = xa + (E0 - qmax + tid);
    auto stage = [&](auto slot_c) {
      constexpr int at = decltype(slot_c)::value % kDepth * 2 * STRIDE;
      if (z_st <= s1) {
#pragma unroll
        for (int r = 0; r < kRounds; ++r)
          if (staged(r, c_st)) {
            cp_async_one(ring + at + tid + r * MARCH_COLS, ga + r * MARCH_COLS);
            cp_async_one(ring + at + STRIDE + tid + r * MARCH_COLS, ga + pair_off + r * MARCH_COLS);
          }
        ++z_st;
        c_st -= n + 2 - z_st;  // c(z) - c(z+1) = n+1-z
        ga += c_st;
      }
      cp_async_commit();
    };
    int c_sp = c0;  // float-float: of the next slice to split
    int z_sp = s0;
    auto split = [&](auto slot_c) {
      constexpr int at = decltype(slot_c)::value % kDepth * 2 * STRIDE;
      constexpr int pl = decltype(slot_c)::value % kPlanes * STRIDE;
      if (z_sp <= s1) {
        double va[kRounds], vb[kRounds];
#pragma unroll
        for (int r = 0; r < kRounds; ++r) {  // reads first: also elements that are not needed
          const int e = min(tid + r * MARCH_COLS, STRIDE - 1);
          va[r] = (double)ring[at + e];
          vb[r] = (double)ring[at + STRIDE + e];
        }
#pragma unroll
        for (int r = 0; r < kRounds; ++r)
          if (staged(r, c_sp)) {
            const FF a = ff_split(va[r]), b = ff_split(vb[r]);
            planes[pl + tid + r * MARCH_COLS] = make_ulonglong2(f2_pack(a.h, b.h), f2_pack(a.l, b.l));
          }
        ++z_sp;
        c_sp -= n + 2 - z_sp;
      }
    };

    const int c = qmax - q;  // this column's element
    const int cp = c + A, cm = c - A;
    T* ya = p.y + (int64_t)m0 * p.S + (E0 - c0 - q);  // at the point of slice s-1
    int c_now = c0;
    const T* bp = nullptr;  // sweep modes: b at the point of slice s
    T ba = T(0), bb = T(0), da = T(0), db = T(0);
    if (kSweep) {
      bp = static_cast<const T*>(p.md.b) + (int64_t)m0 * p.S + (E0 - q);
    }
    if (MODE == MODE_JACOBI && zhi >= zlo) {  // the inverse diagonal is one value inside a macro
      const T* dv = static_cast<const T*>(p.md.dinv);
      const int64_t in = (int64_t)E0 + count(s0 + 1) - q;  // slice zlo
      da = __ldg(dv + (int64_t)m0 * p.S + in);
      db = __ldg(dv + (int64_t)m1 * p.S + in);
    }

    struct Below {  // of one slice: what the point two slices up needs
      typename Q::V c, p1, A0, A1;  // q, q+1, q+A, q+A+1
    };
    Below X[kReread ? 1 : 3] = {};
    typename Q::Acc acc;

    // slice s has arrived in slot I: its values
    typename Q::V vm, l0, l1;
    auto fetch = [&](auto slot_c) {
      constexpr int I = decltype(slot_c)::value;
      Below& now = X[kReread ? 0 : I % 3];
      auto get = [&](int e) -> typename Q::V {
        if constexpr (kSplit)
          return Q::get(planes + I % kPlanes * STRIDE + e);
        else
          return Q::get(ring + I % kDepth * 2 * STRIDE + e, ring + I % kDepth * 2 * STRIDE + STRIDE + e);
      };
      now.c = get(c);                               // q
      vm = get(c + 1);                              // q-1
      l0 = get(cp);                                 // q-A
      l1 = get(cp - 1);                             // q-A+1
      now.p1 = get(c - 1);                          // q+1
      now.A0 = get(cm);                             // q+A
      now.A1 = get(cm - 1);                         // q+A+1
    };
    // finish the point of slice s-1, begin that of s
    auto arrive = [&](int s, auto slot_c) {
      constexpr int I = decltype(slot_c)::value;
      const Below& now = X[kReread ? 0 : I % 3];
      const Below& one = X[kReread ? 0 : (I + 2) % 3];
      const Below& two_back = X[kReread ? 0 : (I + 1) % 3];
      if (s > zlo) {
        if constexpr (kReread) {
          const ulonglong2* const bk = planes + (I + 2) % 4 * STRIDE;
          Q::sym(acc, W(4), l0, Q::get(bk + cm - 1));
          Q::sym(acc, W(5), l1, Q::get(bk + cm));
          Q::sym(acc, W(6), now.c, Q::get(bk + c));
          Q::sym(acc, W(7), vm, Q::get(bk + c - 1));
        } else {
          Q::sym(acc, W(4), l0, two_back.A1);
          Q::sym(acc, W(5), l1, two_back.A0);
          Q::sym(acc, W(6), now.c, two_back.c);
          Q::sym(acc, W(7), vm, two_back.p1);
        }
        T ra, rb;
        Q::finish(acc, ra, rb);
        const bool mine = s - 1 <= zhi;
        if constexpr (P::kPoison) {
          if (mine && P::bad(acc)) {  // an input outside the float-float range: native fp64 rows
            const int z = s - 1, px = k - (q - k * (k + 1) / 2), py = n - z - k;
            float sa, sb;
            f2_unpack(acc.s, sa, sb);
            if (sa != sa) ra = march_native_row(xa, n, px, py, z, p.st.d + wa);
            if (sb != sb) rb = march_native_row(xb, n, px, py, z, p.st.d + wb);
          }
        }
        if constexpr (kSweep) {
          T ua, ub;
          Q::value(one.c, ua, ub);
          ra = mode_out_staged<MODE, T>(ra, ua, ba, da, p.md.omega);
          rb = mode_out_staged<MODE, T>(rb, ub, bb, db, p.md.omega);
        }
        if (mine) {
          *ya = ra;
          if (pair_off) ya[pair_off] = rb;
        }
      }
      if constexpr (kSweep) {
        if (s >= zlo && s <= zhi) {
          ba = ld<false>(bp);
          bb = ld<false>(bp + pair_off);
        }
        bp += c_now - (n + 1 - s);
      }
      Q::first(acc, W(0), now.c);
      Q::sym(acc, W(1), vm, now.p1);
      Q::sym(acc, W(2), l0, now.A1);
      Q::sym(acc, W(3), now.A0, l1);
      ya += c_now;
      c_now -= n + 1 - s;
    };

    pdl_wait();  // the vectors after the previous kernel in the stream
    {
      stage(std::integral_constant<int, 0>{});
      stage(std::integral_constant<int, 1>{});
      if constexpr (kDepth == 6) {
        stage(std::integral_constant<int, 2>{});
        stage(std::integral_constant<int, 3>{});
        stage(std::integral_constant<int, 4>{});
      } else if constexpr (kSplit) {
        stage(std::integral_constant<int, 2>{});
        stage(std::integral_constant<int, 3>{});
      }
    }
    // While the first slices land: this block's share of the interface step, in
    // the order of the macros.  (Interface blocks between the marching ones
    // held a block's registers for the latency of a gather: 247 against 233 us
    // at level 6 with 384 macro-tets in float-float.)
    if (nb == p.n_march) {
      const int w = tid >> 5, faces = p.f.n_units - p.f.n_items;
      const int i0 = (int)((int64_t)p.f.n_items * idx / nb), i1 = (int)((int64_t)p.f.n_items * (idx + 1) / nb);
      const int f0 = (int)((int64_t)faces * idx / nb), f1 = (int)((int64_t)faces * (idx + 1) / nb);
      for (int u = i0 + w; u < i1 + (f1 - f0); u += MARCH_COLS / 32)
        iface3d_unit<MODE, P::kPoison, T>(p.x, p.y, p.f, u < i1 ? u : p.f.n_items + f0 + (u - i1), n, p.S, p.st, p.md);
    }
    if constexpr (kSplit) {
      cp_async_wait<kDepth - 1>();
      __syncthreads();
      split(std::integral_constant<int, 0>{});
    }
    // One pass per slice.  fp32, native: slice s has landed and the slot of
    // slice s-1 is free.  Float-float: slice s is split, slice s+1 has landed.
    auto pass = [&](int s, auto slot_c) {
      constexpr int I = decltype(slot_c)::value;
      cp_async_wait<kDepth - 2>();
      __syncthreads();
      if constexpr (kSplit) {
        split(std::integral_constant<int, I + 1>{});
        stage(std::integral_constant<int, I>{});
      } else {
        stage(std::integral_constant<int, (I + kDepth - 1) % kDepth>{});
      }
      if (s <= sw) {
        fetch(slot_c);
        arrive(s, slot_c);
      }
    };
    int s = s0;
    // the warp's own slices, then the ones only other warps need
#define HY_PASS(I)                                  \
  pass(s, std::integral_constant<int, I>{});        \
  if (++s > s1) break;
    for (;;) {
      HY_PASS(0)
      HY_PASS(1)
      HY_PASS(2)
      if constexpr (kDepth > 3) {
        HY_PASS(3)
      }
      if constexpr (kDepth > 4) {
        HY_PASS(4)
        HY_PASS(5)
      }
    }
#undef HY_PASS
    cp_async_wait<0>();
  }
};

}  // namespace hyteg
