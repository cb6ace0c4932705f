// mf_kernels.cuh -- sum-factorised apply, duplicate summation (DSS), geometry, diagonal and
// layout kernels.  The apply kernels are templated on the storage type S of the vectors
// (double, float, or double-float dd) and the compute type T (double, dd, or the FP32 pair f2),
// and on n = k+1; each comes as a one-operator kernel and a batched kernel over several.
//
// Included once per degree by mf_apply_k<k>.cu so the eight degrees compile in parallel.
#pragma once
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "mf_dd.cuh"
#include "mf_internal.h"
#include "mf_launch.cuh"
#include "mf_reduce.cuh"

namespace mf {

// Cells processed by one CTA of the apply kernels (a divisor of BL).  One thread owns one
// pencil (a 1D line of n values) of one cell -- of two cells for f2 -- in every sweep, so a
// CTA has n^2 * CB threads.
// Launch configurations of the pencil kernels, chosen per operator by the autotuner
// (mf_operator_autotune): base configuration Cfg 0 = CB0 cells per CTA with registers capped for 2
// resident CTAs per SM (launch variant 0 is the fastest of these per degree and path, or a plane
// kernel: see variant0 and mf_plane.cuh); variant 1 = CB0/2 cells per CTA, capped for 3 resident CTAs per SM;
// variant 2 = CB0/2 cells per CTA with no register cap (high degrees spill under a cap);
// variant 4 (double-float compute only) = CB0/2 cells per CTA, registers capped for 1.5x
// Cfg 0's resident threads per SM; variant 5 (double-float only) = CB0 cells per CTA,
// capped for three resident CTAs (also 1.5x).  The block-size sweep of Sec. 6 found the
// double-float apply faster in smaller blocks, and a later sweep of the register budget
// found it faster at higher occupancy: the Cartesian apply at k = 4..7 gains 5-17%.
// (Staging the streamed geometry into shared memory with cp.async was measured and lost:
// the 2-CTA configuration already hides its load latency.)
constexpr int MF_NUM_VARIANTS = 3;
// CB counts compute values per pencil position: cells for double / dd / float, cell pairs for
// the FP32 pair type f2 (CPL cells per value); a CTA holds CB * CPL cells.
template <typename T, int N, int V>
struct Cfg {
  static constexpr int CPL = CellsPer<T>::value;
  static constexpr int CELLS0 = (N <= 4) ? 32 : (N <= 6) ? 16 : (N <= 8) ? 8 : (IsF32<T>::value ? 8 : 4);
  static constexpr int CB0 = CELLS0 / CPL;
  static constexpr int CBH = (CB0 / 2) * CPL >= 4 ? CB0 / 2 : 4 / CPL;
  static constexpr int CB = (V == 0 || V == 5) ? CB0 : CBH;
  static constexpr int MINB = V == 0 ? 2 : (V == 1 || V == 5) ? 3 : (V == 4 ? 3 * CB0 / CBH : 1);
  static constexpr int NT = N * N * CB;
  static constexpr bool GENERAL = true; // kernels of the affine and curved paths built too
  static_assert(CB * CPL >= 4 && BL % (CB * CPL) == 0, "a CTA holds at least 4 cells of a tile (apply_max_blocks)");
};

__device__ __forceinline__ void cell_of(const GridInfo& g, long long t64, int lane, int& cx, int& cy, int& cz) {
  const int t = (int)t64; // tile counts are below 2^31 (checked at mesh creation)
  const int txy = g.ntx * g.nty;
  const int tz = t / txy;
  const int r = t - tz * txy;
  const int ty = r / g.ntx;
  const int tx = r - ty * g.ntx;
  cx = tx * TX + (lane & 3);
  cy = ty * TY + ((lane >> 2) & 3);
  cz = tz * TZ + (lane >> 4);
}

__device__ __forceinline__ long long native_index(const GridInfo& g, int n3, int cx, int cy, int cz, int l) {
  long long t = (long long)(cx / TX) + (long long)g.ntx * ((cy / TY) + (long long)g.nty * (cz / TZ));
  int lane = (cx % TX) + TX * ((cy % TY) + TY * (cz % TZ));
  return (t * n3 + l) * BL + lane;
}

template <int N>
__device__ __forceinline__ bool on_cube_boundary(const GridInfo& g, int cx, int cy, int cz, int i, int j, int k) {
  return (cx == 0 && i == 0) || (cx == g.nx - 1 && i == N - 1) || (cy == 0 && j == 0) ||
         (cy == g.ny - 1 && j == N - 1) || (cz == 0 && k == 0) || (cz == g.nz - 1 && k == N - 1);
}

// Accumulators of the fused CG pairing in store_xpencil: PairAcc sums p y of the stored
// values (Cartesian path); NoAcc when the kernel forms the pairing at the quadrature points.
template <typename S>
struct PairAcc {
  static constexpr bool active = true;
  typename AccOf<S>::type acc;
  __device__ __forceinline__ void add(S p, S y) { acc.add(p, y); }
  __device__ __forceinline__ double value() const { return acc.value(); }
};
struct NoAcc {
  static constexpr bool active = false;
  template <typename S>
  __device__ __forceinline__ void add(S, S) {}
};

__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(float v) { return (double)v; }
__device__ __forceinline__ double to_double(dd v) { return dd_to_double(v); }
__device__ __forceinline__ double to_double(f2 v) { return (double)v.x + (double)v.y; }

// Bulk prefetch of [p, p + bytes) into L2 (16-byte aligned, size a multiple of 16), split into
// 16 KB requests over the lanes of the calling warp.
__device__ __forceinline__ void prefetch_l2_warp(const void* p, unsigned long long bytes) {
  const unsigned long long chunk = 16384;
  for (unsigned long long o = (unsigned long long)(threadIdx.x & 31) * chunk; o < bytes; o += 32 * chunk) {
    const unsigned long long n = bytes - o < chunk ? bytes - o : chunk;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"((const char*)p + o), "r"((unsigned)n) : "memory");
  }
}

// Warp 0 of the first CTA of tile t starts moving tile t + pf_tiles (its input vector rows
// and, for streamed geometry, its metric) from HBM into L2, so that the CTAs of the next wave
// find their loads in L2.  Tiles are contiguous chunks of both arrays.
template <typename S, typename T, int N, int NC>
__device__ __forceinline__ void prefetch_next_wave(const ApplyJob<S, T>& a, long long t, int lane0) {
  constexpr int N3 = N * N * N;
  if (a.pf_tiles <= 0 || lane0 != 0 || threadIdx.x >= 32) return;
  const long long tn = t + a.pf_tiles;
  if (tn >= a.g.ntiles) return;
  const S* xin = (a.cg.st != nullptr && a.cg.update_p) ? a.cg.p : a.x;
  const unsigned long long xb = (unsigned long long)N3 * BL * sizeof(S);
  prefetch_l2_warp(xin + tn * (long long)N3 * BL, xb);
  if (a.cg.st != nullptr && a.cg.update_p) prefetch_l2_warp(a.cg.r + tn * (long long)N3 * BL, xb);
  if (NC > 0 && a.pf_geom && a.geom != nullptr) {
    const unsigned long long gb = (unsigned long long)NC * N3 * BL * sizeof(T);
    prefetch_l2_warp(a.geom + tn * (long long)NC * N3 * BL, gb);
  }
}

// Sum and difference of two values without renormalisation (inputs of further products).
__device__ __forceinline__ dd add_lazy(dd a, dd b) {
  const float s = a.hi + b.hi;
  const float v = s - a.hi;
  const float t = (a.hi - (s - v)) + (b.hi - v);
  return dd(s, t + (a.lo + b.lo));
}
__device__ __forceinline__ dd sub_lazy(dd a, dd b) { return add_lazy(a, dd(-b.hi, -b.lo)); }
__device__ __forceinline__ double add_lazy(double a, double b) { return a + b; }
__device__ __forceinline__ double sub_lazy(double a, double b) { return a - b; }
__device__ __forceinline__ float add_lazy(float a, float b) { return a + b; }
__device__ __forceinline__ float sub_lazy(float a, float b) { return a - b; }

// Where double-float products take the form of 10 instructions (fma_short): only where double
// input is converted with rounding, which outweighs their extra rounding -- n = 4, 5, and the
// forward sweeps of the Cartesian kernels to n = 8.  Vectors kept in double-float (CG) convert
// nothing, and at n = 2, 3 the conversion truncates.  Relative error against 64 bits over that
// with fma() everywhere and truncated conversion (L2, three inputs, 10^3 to 44^3 cells): applies at
// n >= 4 0.89-1.00; with fma_short at n = 3 too 1.00-1.01 there, and in CG 1.01-1.04.
template <typename S, typename T, int N>
struct ShortProducts {
  static constexpr bool rounded = std::is_same<S, double>::value && std::is_same<T, dd>::value && N >= 4;
  static constexpr bool all = rounded && N <= 5, forward = rounded && N <= 8;
};

// sum_i c[i] x[i], i < M (M >= 1), not renormalised
template <typename C, typename T, bool SHORT, int M>
__device__ __forceinline__ T chain(const C* c, const T* x) {
  T s = mul0(c[0], x[0]);
#pragma unroll
  for (int i = 1; i < M; ++i) s = fma_n<SHORT>(c[i], x[i], s);
  return s;
}
__device__ __forceinline__ f2 add_lazy(f2 a, f2 b) { return a + b; }
__device__ __forceinline__ f2 sub_lazy(f2 a, f2 b) { return a + (-b); }

// lo = u + w and hi = u - w (ANTI: w - u), w = sum_i c[i] x[i], i < N / 2.  In FP32 at n = 3 the one
// product goes into the sum by one rounding instead of two (with two, the apply's error against
// 64 bits was 1.005-1.02 times as large; Fold::add_to does the same).
template <bool SHORT, int N, bool ANTI, typename C, typename T>
__device__ __forceinline__ void chain_sum(const C* c, const T* x, T u, T& lo, T& hi) {
  if constexpr (N == 3 && IsF32<T>::value) {
    lo = fma(c[0], x[0], u);
    hi = ANTI ? fma(c[0], x[0], -u) : fma(-c[0], x[0], u);
  } else {
    const T w = chain<C, T, SHORT, N / 2>(c, x);
    lo = add_lazy(u, w);
    hi = ANTI ? sub_lazy(w, u) : sub_lazy(u, w);
  }
}

// Even-odd 1D contraction of one pencil (see EoTab): the pencil folded into its sum and
// difference halves, H (H + 1) products per half instead of n^2 in all.  ANTI: the matrix is
// centro-antisymmetric.  out[q] finished.
template <typename T, int N, bool ANTI, bool SHORT = false>
struct Fold {
  static constexpr int H = N / 2, HE = (N + 1) / 2;
  T e[HE], o[H > 0 ? H : 1];
  __device__ __forceinline__ explicit Fold(const T* in) {
#pragma unroll
    for (int i = 0; i < H; ++i) {
      e[i] = add_lazy(in[i], in[N - 1 - i]);
      o[i] = sub_lazy(in[i], in[N - 1 - i]);
    }
    if (N % 2) e[H] = in[H];
  }
  template <typename C>
  __device__ __forceinline__ void apply(const EoTab<C, N>& t, T* out) const {
#pragma unroll
    for (int q = 0; q < H; ++q) {
      const T u = chain<C, T, SHORT, HE>(t.F + q * HE, e);
      T lo, hi;
      chain_sum<SHORT, N, ANTI>(t.G + q * H, o, u, lo, hi);
      out[q] = finish(lo);
      out[N - 1 - q] = finish(hi);
    }
    if (N % 2) out[H] = finish(ANTI ? chain<C, T, SHORT, H>(t.Mid, o) : chain<C, T, SHORT, HE>(t.Mid, e));
  }
  // s + the contraction (in FP32 a row of one product by one rounding, see chain_sum)
  template <typename C>
  __device__ __forceinline__ void add_to(const T* s, const EoTab<C, N>& t, T* out) const {
    apply(t, out);
#pragma unroll
    for (int q = 0; q < N; ++q) out[q] = finish(add_lazy(s[q], out[q]));
    if constexpr (N == 3 && ANTI && IsF32<T>::value) out[1] = fma(t.Mid[0], o[0], s[1]);
  }
};

// Whether a kernel carries dd_from_double's general form in line (its registers) or calls it
// (its code).  Split apply, FP64, ms in line / called: Cartesian Q3 64^3 0.146 / 0.152, Q4 52^3 0.177 /
// 0.184, Q5 44^3 0.196 / 0.201, Q7 33^3 0.300 / 0.282, Q8 30^3 0.375 / 0.347; curved Q3 64^3 0.365 /
// 0.341, Q4 52^3 0.411 / 0.409.  (The Q2 Cartesian plane kernel, in line with the rest, takes 0.136 against
// 0.124 at 88^3; doubles there run on the tensor cores by default.)
template <int N>
struct InlineFrom { static constexpr bool cartesian = N <= 7; };
template <bool INL, bool NEAR, typename T, typename S>
__device__ __forceinline__ T load_value(S v) {
  if constexpr (std::is_same<T, dd>::value && std::is_same<S, double>::value)
    return dd_from_double<INL, NEAR>(v);
  else
    return to_compute<T, S>(v);
}

// N values of the input from element e0, `step` elements apart, of one cell (CPL = 1; real: v0) or a
// pair (CPL = 2, 8-byte accesses; real: v0, v1): x, or in a CG step with update_p the new
// direction p = r + beta p, written back (zero in padding cells).  Every load is issued before the
// first store, which the compiler must assume to change what a later load reads (mf_launch.cuh).
template <typename S, int CPL, int N>
struct LoadLine {
  typename std::conditional<CPL == 2, float2, S>::type x[N];
  template <typename T>
  __device__ __forceinline__ LoadLine(const ApplyJob<S, T>& a, bool fuse, S beta, long long e0, int step, bool v0,
                                      bool v1) {
    using V = typename std::conditional<CPL == 2, float2, S>::type;
    const S* src = fuse ? a.cg.p : a.x;
#pragma unroll
    for (int m = 0; m < N; ++m)
      if (CPL == 2 || v0) x[m] = *reinterpret_cast<const V*>(src + e0 + (long long)m * step);
    if (!fuse) return;
    V r[N];
#pragma unroll
    for (int m = 0; m < N; ++m)
      if (CPL == 2 || v0) r[m] = *reinterpret_cast<const V*>(a.cg.r + e0 + (long long)m * step);
#pragma unroll
    for (int m = 0; m < N; ++m) {
      if constexpr (CPL == 2) {
        x[m].x = v0 ? fmaf(beta, x[m].x, r[m].x) : 0.0f;
        x[m].y = v1 ? fmaf(beta, x[m].y, r[m].y) : 0.0f;
      } else {
        x[m] = v0 ? finish(fma(beta, x[m], r[m])) : S(0);
      }
      *reinterpret_cast<V*>(a.cg.p + e0 + (long long)m * step) = x[m];
    }
  }
};

// Load the CB values (CB * CPL cells from lane0) of tile t into smem as buf[l*CB + c] (cell
// fastest; a pair value holds cells lane0 + 2c and lane0 + 2c + 1), zeroing padding cells and,
// for Dirichlet, the constrained nodes (the P of P A P).  In a CG step with update_p the loaded
// vector is the new direction p = r + beta p, written back.
// Thread (l0, c) = (threadIdx.x / CB, threadIdx.x % CB) loads local dofs l0 + m n^2 of value c
// (m < n): its cell is the same in every trip, so its coordinates are found once.
template <bool INL, typename S, typename T, int N, int CB, int NT>
__device__ __forceinline__ void load_tile(const ApplyJob<S, T>& a, long long t, int lane0, T* buf) {
  constexpr int N2 = N * N, N3 = N2 * N, CPL = CellsPer<T>::value;
  static_assert(NT == N2 * CB, "one thread per pencil position and value");
  const long long base = t * (long long)N3 * BL + lane0;
  const bool fuse = a.cg.st != nullptr && a.cg.update_p;
  const S beta = fuse ? scalar_from_double<S>(a.cg.st->beta) : S(0);
  const int c = threadIdx.x % CB, l0 = threadIdx.x / CB;
  const long long e0 = base + (long long)l0 * BL + c * CPL; // local dof l0 + m n^2 at e0 + m n^2 BL
  int cx, cy, cz;
  cell_of(a.g, t, lane0 + c * CPL, cx, cy, cz); // for a pair: the second cell is at cx + 1
  const bool yz = cy < a.g.ny && cz < a.g.nz;
  const bool v0 = yz && cx < a.g.nx, v1 = yz && cx + 1 < a.g.nx;
  LoadLine<S, CPL, N> in(a, fuse, beta, e0, N2 * BL, v0, v1);
#pragma unroll
  for (int m = 0; m < N; ++m) {
    const int l = l0 + m * N2, idx = l * CB + c;
    if constexpr (CPL == 1) {
      T v = T(0);
      if (v0) {
        v = load_value<INL, (N >= 4), T, S>(in.x[m]);
        if (a.g.bc) {
          const int i = l % N, j = (l / N) % N, k = l / N2;
          if (on_cube_boundary<N>(a.g, cx, cy, cz, i, j, k)) v = T(0);
        }
      }
      buf[idx] = v;
    } else { // a pair of cells (FP32): 8-byte accesses
      const float2 xv = in.x[m];
      float vx = v0 ? xv.x : 0.0f, vy = v1 ? xv.y : 0.0f;
      if (a.g.bc) {
        const int i = l % N, j = (l / N) % N, k = l / N2;
        if (v0 && on_cube_boundary<N>(a.g, cx, cy, cz, i, j, k)) vx = 0.0f;
        if (v1 && on_cube_boundary<N>(a.g, cx + 1, cy, cz, i, j, k)) vy = 0.0f;
      }
      buf[idx] = T(vx, vy);
    }
  }
}

// Load one x-pencil (j, k) of value c straight into registers: load_tile's load of the
// pencil's n values (the same zeroing of padding cells and constrained nodes, the same fused
// p = r + beta p written back), for a kernel whose first sweep runs along x.
template <typename S, typename T, int N>
__device__ __forceinline__ void load_xpencil(const ApplyJob<S, T>& a, long long t, int lane0, int c, int j, int k,
                                             T* in) {
  constexpr int N2 = N * N, N3 = N2 * N, CPL = CellsPer<T>::value;
  const long long base = t * (long long)N3 * BL + lane0 + c * CPL;
  const bool fuse = a.cg.st != nullptr && a.cg.update_p;
  const S beta = fuse ? scalar_from_double<S>(a.cg.st->beta) : S(0);
  int cx, cy, cz;
  cell_of(a.g, t, lane0 + c * CPL, cx, cy, cz); // for a pair: the second cell is at cx + 1
  const bool yz = cy < a.g.ny && cz < a.g.nz;
  const bool v0 = yz && cx < a.g.nx, v1 = yz && cx + 1 < a.g.nx;
  LoadLine<S, CPL, N> ld(a, fuse, beta, base + (long long)(N * j + N2 * k) * BL, BL, v0, v1);
  if constexpr (CPL == 1) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      T v = T(0);
      if (v0) {
        v = load_value<InlineFrom<N>::cartesian, (N >= 4), T, S>(ld.x[i]);
        if (a.g.bc && on_cube_boundary<N>(a.g, cx, cy, cz, i, j, k)) v = T(0);
      }
      in[i] = v;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const float2 xv = ld.x[i];
      float vx = v0 ? xv.x : 0.0f, vy = v1 ? xv.y : 0.0f;
      if (a.g.bc) {
        if (v0 && on_cube_boundary<N>(a.g, cx, cy, cz, i, j, k)) vx = 0.0f;
        if (v1 && on_cube_boundary<N>(a.g, cx + 1, cy, cz, i, j, k)) vy = 0.0f;
      }
      in[i] = T(vx, vy);
    }
  }
}

// Store one x-pencil (j, k) of value c to global y, zeroing padding / constrained nodes.  In a
// CG step each stored value is also paired with p (acc += p y over real copies); pv holds p
// of the pencil, CPL values per node.
template <typename S, typename T, int N, int CB, typename Acc>
__device__ __forceinline__ void store_xpencil(const ApplyJob<S, T>& a, long long t, int lane0, int c, int j, int k,
                                              const T* out, Acc& acc, const S* pv) {
  constexpr int N2 = N * N, N3 = N2 * N, CPL = CellsPer<T>::value;
  int cx, cy, cz;
  cell_of(a.g, t, lane0 + c * CPL, cx, cy, cz);
  const long long base = t * (long long)N3 * BL + lane0 + c * CPL;
  if constexpr (CPL == 1) {
    const bool valid = cx < a.g.nx && cy < a.g.ny && cz < a.g.nz;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      S v = valid ? to_storage<S, T>(out[i]) : S(0);
      if (valid && a.g.bc && on_cube_boundary<N>(a.g, cx, cy, cz, i, j, k)) v = S(0);
      const long long e = base + (long long)(i + N * j + N2 * k) * BL;
      a.y[e] = v;
      if constexpr (Acc::active) {
        if (a.cg.st != nullptr && valid) acc.add(pv[i], v);
      }
    }
  } else {
    const bool yz = cy < a.g.ny && cz < a.g.nz;
    const bool v0 = yz && cx < a.g.nx, v1 = yz && cx + 1 < a.g.nx;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      float2 v;
      v.x = v0 ? out[i].x : 0.0f;
      v.y = v1 ? out[i].y : 0.0f;
      if (a.g.bc) {
        if (v0 && on_cube_boundary<N>(a.g, cx, cy, cz, i, j, k)) v.x = 0.0f;
        if (v1 && on_cube_boundary<N>(a.g, cx + 1, cy, cz, i, j, k)) v.y = 0.0f;
      }
      const long long e = base + (long long)(i + N * j + N2 * k) * BL;
      *reinterpret_cast<float2*>(a.y + e) = v;
      if constexpr (Acc::active) {
        if (a.cg.st != nullptr) {
          if (v0) acc.add(pv[2 * i], v.x);
          if (v1) acc.add(pv[2 * i + 1], v.y);
        }
      }
    }
  }
}

// A CTA's part of <p, A_K p> in a CG step: every thread parks its value in red[threadIdx.x]
// before a barrier the caller provides; after it, warp 0 folds red in a fixed order and
// writes partials[cta] with a plain store (the next kernel of the stream reads it, so
// no fence is needed and no thread waits for its stores to drain).
template <int NT>
__device__ __forceinline__ void cta_partial_after_barrier(const double* red, double* partials, long long cta) {
  if (threadIdx.x >= 32) return;
  double s = 0.0;
  for (int i = threadIdx.x; i < NT; i += 32) s += red[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (threadIdx.x == 0) partials[cta] = s;
}

// ---------------------------------------------------------------------------------------
// Cartesian cells (axis-aligned affine): Sec. 3.1, Eq. (eval_pipeline), the seven-
// contraction form  y = gx (M(x)M(x)K) x + gy (M(x)K(x)M) x + gz (K(x)M(x)M) x [+ c M(x)M(x)M x]
// (Kronecker factors listed z, y, x).  x-sweep: M and K (2); y-sweep: M on Mx, K on Mx, M on
// Kx (3); z-sweep: M on the combination and K on (M(x)M)x (2).
// ---------------------------------------------------------------------------------------
// One CTA: cells [lane0, lane0 + CB) of tile t; cta = the CTA's index in its operator's grid
// (where its CG partial goes).
template <typename S, typename T, int N, int CB, bool HELM>
__device__ __forceinline__ void cartesian_body(const ApplyJob<S, T>& a, const Tab<typename CoefOf<T>::type, N>& tab,
                                               long long t, int lane0,
                                               long long cta) {
  constexpr int N2 = N * N, N3 = N2 * N, NT = N2 * CB;
  constexpr bool SH = ShortProducts<S, T, N>::all;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf0 = reinterpret_cast<T*>(smem_raw);
  T* buf1 = buf0 + N3 * CB;
  if (a.cg.st != nullptr && a.cg.st->flag != 0) return; // CG step after convergence: no work
  prefetch_next_wave<S, T, N, 0>(a, t, lane0);
  load_tile<InlineFrom<N>::cartesian, S, T, N, CB, NT>(a, t, lane0, buf0);
  __syncthreads();
  const int c = threadIdx.x % CB, p = threadIdx.x / CB, pa = p % N, pb = p / N;
  { // x: pencil (j=pa, k=pb): M and K share one fold of the pencil
    T in[N], mo[N], ko[N];
#pragma unroll
    for (int i = 0; i < N; ++i) in[i] = buf0[(i + N * pa + N2 * pb) * CB + c];
    const Fold<T, N, false, SH> f(in);
    f.apply(tab.eM, mo);
    f.apply(tab.eK, ko);
#pragma unroll
    for (int q = 0; q < N; ++q) {
      buf0[(q + N * pa + N2 * pb) * CB + c] = mo[q];
      buf1[(q + N * pa + N2 * pb) * CB + c] = ko[q];
    }
  }
  __syncthreads();
  { // y: pencil (i=pa, k=pb)
    T am[N], ak[N], mm[N], km[N], mk[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
      am[j] = buf0[(pa + N * j + N2 * pb) * CB + c];
      ak[j] = buf1[(pa + N * j + N2 * pb) * CB + c];
    }
    {
      const Fold<T, N, false, SH> fa(am);
      fa.apply(tab.eM, mm);
      fa.apply(tab.eK, km);
    }
    Fold<T, N, false, SH>(ak).apply(tab.eM, mk);
#pragma unroll
    for (int q = 0; q < N; ++q) {
      T w = fma(a.gx, mk[q], mul0(a.gy, km[q]));
      if (HELM) w = fma(a.cmass, mm[q], w);
      buf0[(pa + N * q + N2 * pb) * CB + c] = finish(w);
      buf1[(pa + N * q + N2 * pb) * CB + c] = mm[q];
    }
  }
  __syncthreads();
  { // z: pencil (i=pa, j=pb); result rows go straight back to smem, then out by x-pencils
    T w[N], mm[N], so[N], ro[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      w[k] = buf0[(pa + N * pb + N2 * k) * CB + c];
      mm[k] = buf1[(pa + N * pb + N2 * k) * CB + c];
    }
    Fold<T, N, false, SH>(w).apply(tab.eM, so);
    Fold<T, N, false, SH>(mm).apply(tab.eK, ro);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < N; ++q) buf0[(pa + N * pb + N2 * q) * CB + c] = finish(fma(a.gz, ro[q], so[q]));
  }
  __syncthreads();
  PairAcc<S> acc;
  { // write out as x-pencils (j=pa, k=pb) so the Dirichlet mask indexes match; a fused CG step
    // pairs each stored value with p (this CTA wrote p during the load, before the barriers)
    constexpr int CPL = CellsPer<T>::value;
    S pv[N * CPL];
    if (a.cg.st != nullptr) {
      const S* pg = (a.cg.update_p ? a.cg.p : a.x) + t * (long long)N3 * BL + lane0 + c * CPL;
#pragma unroll
      for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < CPL; ++j) pv[i * CPL + j] = pg[(long long)(i + N * pa + N2 * pb) * BL + j];
    }
    T o[N];
#pragma unroll
    for (int i = 0; i < N; ++i) o[i] = buf0[(i + N * pa + N2 * pb) * CB + c];
    store_xpencil<S, T, N, CB>(a, t, lane0, c, pa, pb, o, acc, pv);
  }
  if (a.cg.st != nullptr) {
    __shared__ double red[NT];
    red[threadIdx.x] = acc.value();
    __syncthreads();
    cta_partial_after_barrier<NT>(red, a.cg.partials, cta);
  }
}

// ---------------------------------------------------------------------------------------
// Cartesian cells in fast-diagonalised form: with W = M V (V^T M V = I, V^T K V = diag(lam)),
// M = W W^T and K = W diag(lam) W^T, so the seven-contraction operator of Eq. (eval_pipeline)
// is A_e = (W(x)W(x)W) diag(d) (W(x)W(x)W)^T with d(i,j,k) = gx lam_i + gy lam_j + gz lam_k
// [+ c]: three forward sweeps W^T, a pointwise scale, three backward sweeps W.  Six
// single-input contractions (folded: every mode is symmetric or antisymmetric) instead of
// seven, and the pointwise scale replaces the combination of the contractions.
// ---------------------------------------------------------------------------------------
// forward: modes of a pencil (symmetric first), from its folded sums and differences
template <bool SHORT, typename C, typename T, int N>
__device__ __forceinline__ void fd_forward(const FdTab<C, N>& t, const T* in, T* out) {
  constexpr int H = N / 2, HE = (N + 1) / 2;
  const Fold<T, N, false> f(in);
#pragma unroll
  for (int m = 0; m < HE; ++m) out[m] = finish(chain<C, T, SHORT, HE>(t.Ff + m * HE, f.e));
#pragma unroll
  for (int m = 0; m < H; ++m) out[HE + m] = finish(chain<C, T, SHORT, H>(t.Gf + m * H, f.o));
}
// backward: nodal values of a pencil from its modes
template <bool SHORT, typename C, typename T, int N>
__device__ __forceinline__ void fd_backward(const FdTab<C, N>& t, const T* z, T* out) {
  constexpr int H = N / 2, HE = (N + 1) / 2;
#pragma unroll
  for (int j = 0; j < H; ++j) {
    const T u = chain<C, T, SHORT, HE>(t.Fb + j * HE, z);
    T lo, hi;
    chain_sum<SHORT, N, false>(t.Gb + j * H, z + HE, u, lo, hi);
    out[j] = finish(lo);
    out[N - 1 - j] = finish(hi);
  }
  if (N % 2) out[H] = finish(chain<C, T, SHORT, HE>(t.Fb + H * HE, z));
}

template <typename S, typename T, int N, int CB, bool HELM>
__device__ __forceinline__ void cartesian_fd_body(const ApplyJob<S, T>& a, const Tab<typename CoefOf<T>::type, N>& tab,
                                                  long long t, int lane0, long long cta) {
  using C = typename CoefOf<T>::type;
  constexpr int N2 = N * N, N3 = N2 * N, NT = N2 * CB;
  constexpr bool SH = ShortProducts<S, T, N>::all, SHF = ShortProducts<S, T, N>::forward;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf0 = reinterpret_cast<T*>(smem_raw);
  if (a.cg.st != nullptr && a.cg.st->flag != 0) return; // CG step after convergence: no work
  prefetch_next_wave<S, T, N, 0>(a, t, lane0);
  const int c = threadIdx.x % CB, p = threadIdx.x / CB, pa = p % N, pb = p / N;
  const FdTab<C, N>& fd = tab.fd;
  // At n = 6..8 each double-float thread loads its x-pencil straight from global memory (no
  // shared-memory round trip, one barrier fewer: k = 5..7 2-3% faster).  Elsewhere the tile
  // load through shared memory is kept: measured, the direct load made k = 4 9% and k = 8 5%
  // slower (its registers cost resident CTAs); the FP32 view was not measured.
  constexpr bool direct = N >= 6 && N <= 8 && !IsF32<T>::value;
  if constexpr (!direct) {
    load_tile<InlineFrom<N>::cartesian, S, T, N, CB, NT>(a, t, lane0, buf0);
    __syncthreads();
  }
  { // forward x: pencil (j=pa, k=pb)
    T in[N], out[N];
    if constexpr (direct) {
      load_xpencil<S, T, N>(a, t, lane0, c, pa, pb, in);
    } else {
#pragma unroll
      for (int i = 0; i < N; ++i) in[i] = buf0[(i + N * pa + N2 * pb) * CB + c];
    }
    fd_forward<SHF, C, T, N>(fd, in, out);
#pragma unroll
    for (int i = 0; i < N; ++i) buf0[(i + N * pa + N2 * pb) * CB + c] = out[i];
  }
  __syncthreads();
  { // forward y: pencil (i=pa, k=pb)
    T in[N], out[N];
#pragma unroll
    for (int j = 0; j < N; ++j) in[j] = buf0[(pa + N * j + N2 * pb) * CB + c];
    fd_forward<SHF, C, T, N>(fd, in, out);
#pragma unroll
    for (int j = 0; j < N; ++j) buf0[(pa + N * j + N2 * pb) * CB + c] = out[j];
  }
  __syncthreads();
  { // forward z, scale by d = gx lam_pa + gy lam_pb + gz lam_k (+ c), backward z: pencil (i=pa, j=pb)
    T in[N], z[N], out[N];
#pragma unroll
    for (int k = 0; k < N; ++k) in[k] = buf0[(pa + N * pb + N2 * k) * CB + c];
    fd_forward<SHF, C, T, N>(fd, in, z);
    T dxy = fma(fd.lam[pb], a.gy, mul0(fd.lam[pa], a.gx));
    if (HELM) dxy = add_lazy(dxy, a.cmass);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const T dk = finish(fma(fd.lam[k], a.gz, dxy));
      z[k] = finish(mul0(dk, z[k]));
    }
    fd_backward<SH, C, T, N>(fd, z, out);
#pragma unroll
    for (int k = 0; k < N; ++k) buf0[(pa + N * pb + N2 * k) * CB + c] = out[k];
  }
  __syncthreads();
  { // backward y: pencil (i=pa, k=pb)
    T z[N], out[N];
#pragma unroll
    for (int j = 0; j < N; ++j) z[j] = buf0[(pa + N * j + N2 * pb) * CB + c];
    fd_backward<SH, C, T, N>(fd, z, out);
#pragma unroll
    for (int j = 0; j < N; ++j) buf0[(pa + N * j + N2 * pb) * CB + c] = out[j];
  }
  __syncthreads();
  PairAcc<S> acc;
  { // backward x: pencil (j=pa, k=pb) -> global (a fused CG step pairs each stored value with p)
    constexpr int CPL = CellsPer<T>::value;
    S pv[N * CPL];
    if (a.cg.st != nullptr) {
      const S* pg = (a.cg.update_p ? a.cg.p : a.x) + t * (long long)N3 * BL + lane0 + c * CPL;
#pragma unroll
      for (int i = 0; i < N; ++i)
#pragma unroll
        for (int j = 0; j < CPL; ++j) pv[i * CPL + j] = pg[(long long)(i + N * pa + N2 * pb) * BL + j];
    }
    T z[N], o[N];
#pragma unroll
    for (int i = 0; i < N; ++i) z[i] = buf0[(i + N * pa + N2 * pb) * CB + c];
    fd_backward<SH, C, T, N>(fd, z, o);
    store_xpencil<S, T, N, CB>(a, t, lane0, c, pa, pb, o, acc, pv);
  }
  if (a.cg.st != nullptr) {
    __shared__ double red[NT];
    red[threadIdx.x] = acc.value();
    __syncthreads();
    cta_partial_after_barrier<NT>(red, a.cg.partials, cta);
  }
}

// 1 / b for b well inside the float range (here in [0.6, 1.4]): the hardware's approximation
// (1 ulp) and one Newton-Raphson step, x (2 - b x); within 1 ulp of the division, whose range
// handling costs several times as much (Q4 curved FP32 52^3, plane kernel: 0.110 -> 0.099 ms).
// The pencil kernels of n = 7, 8 keep the division (n = 7: 0.162 against 0.174 ms, n = 8: 0.175
// against 0.195 with the Newton step, which costs them registers).
template <int N>
__device__ __forceinline__ float metric_rcp(float b) {
  if constexpr (N == 7 || N == 8) return __frcp_rn(b);
  float x;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(b));
  return fmaf(x, fmaf(-b, x, 1.0f), x);
}

// Flux v = G d of the FP32 curved view at one Gauss point of one cell (d the reference
// gradient), and m = w |det J| c_m, from the sin and pi cos of pi xh per direction: the map
// x = xh + amp s(xh) (1,1,1) has J = (I + u v^T) D with u = amp (1,1,1), v = grad s, D = diag(h);
// Sherman-Morrison gives J^-1 = D^-1 (I - u v^T / beta), beta = 1 + v.u, and J^-1 J^-T = D^-1
// (I - (u v^T + v u^T)/beta + |v|^2 u u^T / beta^2) D^-1.  G is applied as it stands, one
// rank-one term at a time (23 operations instead of 21 to form its six entries and 9 to apply
// them).  Arguments: sx, pi cos x, and the products sy sz, pi cos y sz, sy pi cos z.  Every
// operation is rounded as written (no contraction), see f2.
template <int N, typename S, typename T>
__device__ __forceinline__ void curved_flux_f32(float sx, float px, float syz, float pyz, float spz, float w,
                                                const ApplyJob<S, T>& a, float d1, float d2, float d3, float* v,
                                                float* m) {
  const float v1 = __fmul_rn(px, syz), v2 = __fmul_rn(sx, pyz), v3 = __fmul_rn(sx, spz);
  const float beta = fmaf(a.amp, __fadd_rn(__fadd_rn(v1, v2), v3), 1.0f);
  const float au = __fmul_rn(a.amp, metric_rcp<N>(beta));
  const float vv = fmaf(v3, v3, fmaf(v2, v2, __fmul_rn(v1, v1)));
  const float c2 = __fmul_rn(__fmul_rn(au, au), vv);
  const float wd = __fmul_rn(__fmul_rn(w, a.hdet), fabsf(beta));
  const float e1 = __fmul_rn(a.ih[0], d1), e2 = __fmul_rn(a.ih[1], d2), e3 = __fmul_rn(a.ih[2], d3); // D^-1 d
  const float s = __fadd_rn(__fadd_rn(e1, e2), e3), t = fmaf(v3, e3, fmaf(v2, e2, __fmul_rn(v1, e1)));
  const float k = fmaf(c2, s, -__fmul_rn(au, t)), as = __fmul_rn(au, s);
  v[0] = __fmul_rn(__fmul_rn(wd, a.ih[0]), fmaf(-as, v1, __fadd_rn(e1, k)));
  v[1] = __fmul_rn(__fmul_rn(wd, a.ih[1]), fmaf(-as, v2, __fadd_rn(e2, k)));
  v[2] = __fmul_rn(__fmul_rn(wd, a.ih[2]), fmaf(-as, v3, __fadd_rn(e3, k)));
  *m = __fmul_rn(wd, a.cm);
}
// the same for a value (a pair of x-neighbours: sx, px per cell)
template <int N, typename S, typename T>
__device__ __forceinline__ void curved_flux(const float (&sx)[2], const float (&px)[2], float syz, float pyz, float spz,
                                            float w, const ApplyJob<S, T>& a, T d1, T d2, T d3, T& v1, T& v2, T& v3,
                                            T& m) {
  float v[3], mm;
  if constexpr (CellsPer<T>::value == 2) {
    float u[3], mu;
    curved_flux_f32<N>(sx[0], px[0], syz, pyz, spz, w, a, d1.x, d2.x, d3.x, v, &mm);
    curved_flux_f32<N>(sx[1], px[1], syz, pyz, spz, w, a, d1.y, d2.y, d3.y, u, &mu);
    v1 = T(v[0], u[0]);
    v2 = T(v[1], u[1]);
    v3 = T(v[2], u[2]);
    m = T(mm, mu);
  } else if constexpr (IsF32<T>::value) {
    curved_flux_f32<N>(sx[0], px[0], syz, pyz, spz, w, a, d1, d2, d3, v, &mm);
    v1 = v[0];
    v2 = v[1];
    v3 = v[2];
    m = mm;
  }
}

// ---------------------------------------------------------------------------------------
// General cells (affine with a full metric, or curved with per-point geometry):
// interpolate to Gauss points with S (three sweeps), reference gradients by the collocation
// derivative Dc (three sweeps), v = G grad u at every point (6 metric entries; Helmholtz adds
// m u), then the transposes: Dc^T per direction summed, and S^T along z, y, x.
// ---------------------------------------------------------------------------------------
template <typename S, typename T, int N, int CB, bool CURVED, bool HELM>
__device__ __forceinline__ void general_body(const ApplyJob<S, T>& a, const Tab<typename CoefOf<T>::type, N>& tab,
                                             long long t, int lane0,
                                             long long cta) {
  constexpr int N2 = N * N, N3 = N2 * N, NT = N2 * CB;
  constexpr int NC = HELM ? 7 : 6;
  constexpr bool SH = ShortProducts<S, T, N>::all;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* buf0 = reinterpret_cast<T*>(smem_raw);
  T* buf1 = buf0 + N3 * CB;
  T* buf2 = buf1 + N3 * CB;
  if (a.cg.st != nullptr && a.cg.st->flag != 0) return; // CG step after convergence: no work
  // streamed geometry exists only for the FP64 views (the FP32 view computes its metric)
  prefetch_next_wave<S, T, N, (CURVED && !IsF32<T>::value) ? NC : 0>(a, t, lane0);
  load_tile<false, S, T, N, CB, NT>(a, t, lane0, buf0);
  __syncthreads();
  const int c = threadIdx.x % CB, p = threadIdx.x / CB, pa = p % N, pb = p / N;
  { // x-sweep with S, pencil (j=pa, k=pb), in place
    T in[N], out[N];
#pragma unroll
    for (int i = 0; i < N; ++i) in[i] = buf0[(i + N * pa + N2 * pb) * CB + c];
    Fold<T, N, false, SH>(in).apply(tab.eS, out);
#pragma unroll
    for (int q = 0; q < N; ++q) buf0[(q + N * pa + N2 * pb) * CB + c] = out[q];
  }
  __syncthreads();
  { // y-sweep, pencil (i=pa, k=pb)
    T in[N], out[N];
#pragma unroll
    for (int j = 0; j < N; ++j) in[j] = buf0[(pa + N * j + N2 * pb) * CB + c];
    Fold<T, N, false, SH>(in).apply(tab.eS, out);
#pragma unroll
    for (int q = 0; q < N; ++q) buf0[(pa + N * q + N2 * pb) * CB + c] = out[q];
  }
  __syncthreads();
  // z-sweep, pencil (i=pa, j=pb): values U and the z-derivative stay in registers, U also goes
  // to buf1 for the x- and y-derivatives of the other pencils
  T U[N], d3[N];
  {
    T in[N];
#pragma unroll
    for (int k = 0; k < N; ++k) in[k] = buf0[(pa + N * pb + N2 * k) * CB + c];
    Fold<T, N, false, SH>(in).apply(tab.eS, U);
#pragma unroll
    for (int q = 0; q < N; ++q) buf1[(pa + N * pb + N2 * q) * CB + c] = U[q];
    Fold<T, N, true, SH>(U).apply(tab.eD, d3);
  }
  __syncthreads();
  { // x- and y-derivatives by Dc, folded like the z one: x-pencil (j=pa, k=pb) of buf1 -> buf0,
    // y-pencil (i=pa, k=pb) of buf1 -> buf2
    T in[N], out[N];
#pragma unroll
    for (int i = 0; i < N; ++i) in[i] = buf1[(i + N * pa + N2 * pb) * CB + c];
    Fold<T, N, true, SH>(in).apply(tab.eD, out);
#pragma unroll
    for (int q = 0; q < N; ++q) buf0[(q + N * pa + N2 * pb) * CB + c] = out[q];
#pragma unroll
    for (int j = 0; j < N; ++j) in[j] = buf1[(pa + N * j + N2 * pb) * CB + c];
    Fold<T, N, true, SH>(in).apply(tab.eD, out);
#pragma unroll
    for (int q = 0; q < N; ++q) buf2[(pa + N * q + N2 * pb) * CB + c] = out[q];
  }
  __syncthreads();
  // Per Gauss point (pa, pb, q): reference gradient (d1 from buf0, d2 from buf2, d3 in
  // registers), metric, and the fluxes v = G grad u, each written over its own derivative:
  // v1 -> buf0, v2 -> buf2, v3 -> d3 (Helmholtz: m u too).
  // A fused CG step also sums grad u . v (+ m u^2): p_K^T A_K p_K of this pencil's points,
  // equal to the pairing of p with the split product written below (Lemma 1).
  const long long gbase = (t * NC * (long long)N3) * BL + lane0 + c * CellsPer<T>::value;
  const bool fuse = a.cg.st != nullptr;
  T pap = T(0);
  // FP32 curved: sin and pi cos of pi xh at this thread's x and y points and at every z point of
  // the cell's layer, loaded before the point loop (per cell of the value: the cells of a
  // pair are x-neighbours, so only the x tables differ)
  constexpr int CPL = CellsPer<T>::value;
  float sx[2], px[2], sy = 0.f, py = 0.f, szq[N], pzq[N];
  if constexpr (CURVED && IsF32<T>::value) {
    int ccx, ccy, ccz;
    cell_of(a.g, t, lane0 + c * CPL, ccx, ccy, ccz);
    ccy = min(ccy, a.g.ny - 1);
    ccz = min(ccz, a.g.nz - 1);
#pragma unroll
    for (int j = 0; j < CPL; ++j) {
      const float* tx = a.gtab + 2 * (min(ccx + j, a.g.nx - 1) * N + pa);
      sx[j] = tx[0];
      px[j] = tx[1];
    }
    const float* ty = a.gtab + 2 * ((a.g.nx + ccy) * N + pb);
    const float* tz = a.gtab + 2 * ((a.g.nx + a.g.ny + ccz) * N);
    sy = ty[0]; py = ty[1];
#pragma unroll
    for (int q = 0; q < N; ++q) { szq[q] = tz[2 * q]; pzq[q] = tz[2 * q + 1]; }
  }
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int l = pa + N * pb + N2 * q;
    const T d1 = buf0[l * CB + c], d2 = buf2[l * CB + c], d3q = d3[q];
    T v1, v2, v3, m = T(0);
    if constexpr (CURVED && IsF32<T>::value) {
      curved_flux<N>(sx, px, __fmul_rn(sy, szq[q]), __fmul_rn(py, szq[q]), __fmul_rn(sy, pzq[q]),
                  tab.W[pa] * tab.W[pb] * tab.W[q], a, d1, d2, d3q, v1, v2, v3, m);
    } else {
      T g0, g1, g2, g3, g4, g5;
      if (CURVED) {
        const T* gp = a.geom + gbase + (long long)l * BL;
        g0 = gp[0];
        g1 = gp[(long long)1 * N3 * BL];
        g2 = gp[(long long)2 * N3 * BL];
        g3 = gp[(long long)3 * N3 * BL];
        g4 = gp[(long long)4 * N3 * BL];
        g5 = gp[(long long)5 * N3 * BL];
        if (HELM) m = gp[(long long)6 * N3 * BL];
      } else {
        const auto w = tab.W[pa] * tab.W[pb] * tab.W[q];
        g0 = w * a.G[0]; g1 = w * a.G[1]; g2 = w * a.G[2];
        g3 = w * a.G[3]; g4 = w * a.G[4]; g5 = w * a.G[5];
        if (HELM) m = w * a.mdet;
      }
      v1 = finish(fma_n<SH>(g0, d1, fma_n<SH>(g1, d2, mul0(g2, d3q))));
      v2 = finish(fma_n<SH>(g1, d1, fma_n<SH>(g3, d2, mul0(g4, d3q))));
      v3 = finish(fma_n<SH>(g2, d1, fma_n<SH>(g4, d2, mul0(g5, d3q))));
    }
    buf0[l * CB + c] = v1;
    buf2[l * CB + c] = v2;
    d3[q] = v3;
    if (fuse) { // <p, A_K p> as the quadrature form: sum over points of grad u . G grad u (+ m u^2)
      pap = fma(d1, v1, fma(d2, v2, fma(d3q, v3, pap)));
      if (HELM) pap = fma(U[q], m * U[q], pap);
    }
    if (HELM) U[q] = m * U[q];
  }
  __syncthreads();
  { // Dc^T along x of v1: x-pencil (j=pa, k=pb) of buf0 -> buf1 (U there is no longer read);
    // Dc^T along y of v2: y-pencil (i=pa, k=pb) of buf2, in place
    T in[N], out[N];
#pragma unroll
    for (int q = 0; q < N; ++q) in[q] = buf0[(q + N * pa + N2 * pb) * CB + c];
    Fold<T, N, true, SH>(in).apply(tab.eDt, out);
#pragma unroll
    for (int i = 0; i < N; ++i) buf1[(i + N * pa + N2 * pb) * CB + c] = out[i];
#pragma unroll
    for (int q = 0; q < N; ++q) in[q] = buf2[(pa + N * q + N2 * pb) * CB + c];
    Fold<T, N, true, SH>(in).apply(tab.eDt, out);
#pragma unroll
    for (int j = 0; j < N; ++j) buf2[(pa + N * j + N2 * pb) * CB + c] = out[j];
  }
  __syncthreads();
  // t = Dc^T_x v1 (+ m u) + Dc^T_y v2 + Dc^T_z v3 at points (pa, pb, q), then S^T along z
  {
    T s[N], tq[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const int l = pa + N * pb + N2 * q;
      s[q] = buf1[l * CB + c];
      if (HELM) s[q] = add_lazy(s[q], U[q]);
      s[q] = add_lazy(s[q], buf2[l * CB + c]);
    }
    Fold<T, N, true, SH>(d3).add_to(s, tab.eDt, tq); // Dc^T_z v3 along this pencil
    T out[N];
    Fold<T, N, false, SH>(tq).apply(tab.eSt, out);
#pragma unroll
    for (int k = 0; k < N; ++k) buf1[(pa + N * pb + N2 * k) * CB + c] = out[k];
  }
  __syncthreads();
  { // S^T along y, pencil (i=pa, k=pb), in place
    T in[N], out[N];
#pragma unroll
    for (int q = 0; q < N; ++q) in[q] = buf1[(pa + N * q + N2 * pb) * CB + c];
    Fold<T, N, false, SH>(in).apply(tab.eSt, out);
#pragma unroll
    for (int j = 0; j < N; ++j) buf1[(pa + N * j + N2 * pb) * CB + c] = out[j];
  }
  __syncthreads();
  NoAcc acc;
  { // S^T along x, pencil (j=pa, k=pb) -> global
    T in[N], o[N];
#pragma unroll
    for (int q = 0; q < N; ++q) in[q] = buf1[(q + N * pa + N2 * pb) * CB + c];
    Fold<T, N, false, SH>(in).apply(tab.eSt, o);
    store_xpencil<S, T, N, CB>(a, t, lane0, c, pa, pb, o, acc, static_cast<const S*>(nullptr));
  }
  if (fuse) { // after the last barrier, so that no warp waits for warp 0's fold
    __shared__ double red[NT];
    red[threadIdx.x] = to_double(finish(pap));
    __syncthreads();
    cta_partial_after_barrier<NT>(red, a.cg.partials, cta);
  }
}

} // namespace mf

#include "mf_plane.cuh"

namespace mf {

// Kernels: one operator per launch (CTA b = cells (b % GPT) * CB .. of tile b / GPT), or a
// batch of operators of one degree (see ApplyBatch): the CTA finds its job by binary search
// over the block offsets and copies the job's description into shared memory.
// MF_CART_FD=0 selects the seven-contraction Cartesian body instead of the fast-diagonalised one
#ifndef MF_CART_FD
#define MF_CART_FD 1
#endif
template <typename S, typename T, int N, int CB, bool HELM>
__device__ __forceinline__ void cartesian_apply(const ApplyJob<S, T>& a, const Tab<typename CoefOf<T>::type, N>& tab,
                                                long long t, int lane0, long long cta) {
  if (MF_CART_FD) cartesian_fd_body<S, T, N, CB, HELM>(a, tab, t, lane0, cta);
  else cartesian_body<S, T, N, CB, HELM>(a, tab, t, lane0, cta);
}
template <typename S, typename T, int N, int CB, int MINB, bool HELM>
__global__ void __launch_bounds__(N * N * CB, MINB) apply_cartesian(ApplyArgs<S, T, N> A) {
  constexpr int CC = CB * CellsPer<T>::value, GPT = BL / CC; // cells per CTA, CTAs per tile
  pdl_enter();
  cartesian_apply<S, T, N, CB, HELM>(A.j, A.tab, blockIdx.x / GPT, (blockIdx.x % GPT) * CC, blockIdx.x);
}
template <typename S, typename T, int N, int CB, int MINB, bool CURVED, bool HELM>
__global__ void __launch_bounds__(N * N * CB, MINB) apply_general(ApplyArgs<S, T, N> A) {
  constexpr int CC = CB * CellsPer<T>::value, GPT = BL / CC;
  pdl_enter();
  general_body<S, T, N, CB, CURVED, HELM>(A.j, A.tab, blockIdx.x / GPT, (blockIdx.x % GPT) * CC, blockIdx.x);
}

template <typename S, typename T, int N, bool HELM>
__global__ void __launch_bounds__(PlaneCfg<T, N>::NT, PlaneCfg<T, N>::MINB_C) apply_cartesian_plane(ApplyArgs<S, T, N> A) {
  pdl_enter();
  cartesian_plane<S, T, N, HELM>(A.j, A.tab, blockIdx.x);
}
template <typename S, typename T, int N, bool CURVED, bool HELM>
__global__ void __launch_bounds__(PlaneCfg<T, N>::NT, PlaneCfg<T, N>::MINB_G) apply_general_plane(ApplyArgs<S, T, N> A) {
  pdl_enter();
  general_plane<S, T, N, CURVED, HELM>(A.j, A.tab, blockIdx.x);
}

// The batched apply is one persistent launch: as many CTAs as fit the GPU at once, each
// taking work units u = blockIdx.x, blockIdx.x + gridDim.x, ... of the concatenated unit
// space of all jobs (a unit is what one CTA of the job's own launch does).  batch_unit finds
// the job of unit u (largest i with block0[i] <= u), copies its description into shared
// memory when it differs from the one held (jheld), and returns the unit's local index, so a
// unit computes exactly what the job's solo launch computes in that CTA.
template <typename S, typename T>
__device__ __forceinline__ long long batch_unit(const ApplyJob<S, T>* jobs, const long long* block0, int njobs,
                                                long long u, ApplyJob<S, T>& sj, int& jheld) {
  __shared__ int jsel;
  if (threadIdx.x == 0) {
    int lo = 0, hi = njobs - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (block0[mid] <= u) lo = mid;
      else hi = mid - 1;
    }
    jsel = lo;
  }
  __syncthreads();
  const int j = jsel;
  if (j != jheld) { // uniform: both are shared
    static_assert(sizeof(ApplyJob<S, T>) % 8 == 0, "job description copied as 8-byte words");
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(jobs + j);
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(&sj);
    for (int i = threadIdx.x; i < (int)(sizeof(ApplyJob<S, T>) / 8); i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    if (threadIdx.x == 0) jheld = j; // every thread has read jheld above; the next read follows
                                     // the barrier that ends the unit
  }
  return u - block0[j];
}
template <typename S, typename T, int N, int CB, int MINB, bool HELM>
__global__ void __launch_bounds__(N * N * CB, MINB) apply_cartesian_batch(ApplyBatch<S, T, N> B) {
  constexpr int CC = CB * CellsPer<T>::value, GPT = BL / CC;
  __shared__ __align__(16) ApplyJob<S, T> sj;
  __shared__ int jheld;
  if (threadIdx.x == 0) jheld = -1;
  pdl_enter();
  for (long long u = blockIdx.x; u < B.nunits; u += gridDim.x) {
    const long long b = batch_unit(B.jobs, B.block0, B.njobs, u, sj, jheld);
    cartesian_apply<S, T, N, CB, HELM>(sj, B.tab, b / GPT, (int)(b % GPT) * CC, b);
    __syncthreads(); // the next unit reuses the shared buffers (and may replace sj)
  }
}
template <typename S, typename T, int N, int CB, int MINB, bool CURVED, bool HELM>
__global__ void __launch_bounds__(N * N * CB, MINB) apply_general_batch(ApplyBatch<S, T, N> B) {
  constexpr int CC = CB * CellsPer<T>::value, GPT = BL / CC;
  __shared__ __align__(16) ApplyJob<S, T> sj;
  __shared__ int jheld;
  if (threadIdx.x == 0) jheld = -1;
  pdl_enter();
  for (long long u = blockIdx.x; u < B.nunits; u += gridDim.x) {
    const long long b = batch_unit(B.jobs, B.block0, B.njobs, u, sj, jheld);
    general_body<S, T, N, CB, CURVED, HELM>(sj, B.tab, b / GPT, (int)(b % GPT) * CC, b);
    __syncthreads(); // the next unit reuses the shared buffers (and may replace sj)
  }
}

template <typename S, typename T, int N, bool HELM>
__global__ void __launch_bounds__(PlaneCfg<T, N>::NT, PlaneCfg<T, N>::MINB_C)
    apply_cartesian_plane_batch(ApplyBatch<S, T, N> B) {
  __shared__ __align__(16) ApplyJob<S, T> sj;
  __shared__ int jheld;
  if (threadIdx.x == 0) jheld = -1;
  pdl_enter();
  for (long long u = blockIdx.x; u < B.nunits; u += gridDim.x) {
    const long long b = batch_unit(B.jobs, B.block0, B.njobs, u, sj, jheld);
    cartesian_plane<S, T, N, HELM>(sj, B.tab, b);
    __syncthreads();
  }
}
template <typename S, typename T, int N, bool CURVED, bool HELM>
__global__ void __launch_bounds__(PlaneCfg<T, N>::NT, PlaneCfg<T, N>::MINB_G)
    apply_general_plane_batch(ApplyBatch<S, T, N> B) {
  __shared__ __align__(16) ApplyJob<S, T> sj;
  __shared__ int jheld;
  if (threadIdx.x == 0) jheld = -1;
  pdl_enter();
  for (long long u = blockIdx.x; u < B.nunits; u += gridDim.x) {
    const long long b = batch_unit(B.jobs, B.block0, B.njobs, u, sj, jheld);
    general_plane<S, T, N, CURVED, HELM>(sj, B.tab, b);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------
// Duplicate summation y <- G G^T y (Sec. 4: embedding G and assembly G^T) in the canonical
// order of the dimension-split sweeps of Sec. 3: the copies of a node are summed pairwise
// along x, then the x-sums along y, then along z.  Each node belongs to its lowest copy (the
// cell with the smaller index in every direction), and that copy's lane reads and writes all
// of its copies, so no atomics and no races.
//
// A warp takes rows (local node (i, j, k)) of a tile, lane = cell: its own copies are one
// contiguous 32-element row, and the copies across a face are the row of the opposite local
// node, shifted by one cell inside the tile (3 of 4 lanes along x and y, half along z) and in
// the next tile for the rest.  In a tile away from the low mesh faces only the rows with
// i, j, k >= 1 and at least one of them K own shared nodes, every lane of them is at work, and
// a row's kind (which faces it lies on) is uniform in the warp.  The tiles on a low mesh face
// get further warps for the rows with a zero index, for the lanes on that face.
// Bound by the copies' traffic (each read and written once).  Measured on one GB300 against a
// kernel with one thread per node along a row of nodes, which this one replaced (it spent 77
// instructions per DoF on finding the copies, and half-used sectors in FP32): FP64 Q1 184^3
// 0.157 -> 0.131 ms, Q4 74^3 0.232 -> 0.125 ms (5.1 TB/s), Q8 41^3 0.234 -> 0.115 ms;
// FP32 Q4 64^3 0.153 -> 0.050 ms; Q2 8^3 4.4 -> 4.3 us.
// avg = 1: the average of the copies instead of their sum (mf_make_consistent): the sum in
// the same canonical order times 1/multiplicity (a power of two, so exact), and no Dirichlet
// mask.
// ---------------------------------------------------------------------------------------
constexpr int DSS_THREADS = 256;
template <int N>
struct DssCfg {
  static constexpr int K = N - 1, E = K - 1;
  // Rows of an inner tile by kind: (K-1)^2 on each of the three faces, K-1 on each edge, the
  // vertex.  A warp takes one chunk of U rows along a line (U loads in flight per copy and
  // lane), CL chunks per line, so that a copy's address is one pointer plus constant offsets.
  // (A loop over chunks made the compiler keep every kind's pointers: 160 registers.)
  static constexpr int U = E < 1 ? 1 : (E <= 4 ? E : (E + 1) / 2), CL = E < 1 ? 1 : (E + U - 1) / U;
  static constexpr int CHUNKS = E < 1 ? 1 : 1 + 3 * CL + 3 * CL * E;
  static constexpr int LOW = N * N * N - K * K * K; // rows with a zero index
};

// What a lane needs to find and sum the copies of its nodes.
struct DssLane {
  long long o[3]; // element distance to the copy across the high x / y / z face
  bool h[3];      // whether there is one
  bool mask;      // constrained nodes are zeroed
  int avg;
};

// `count` (<= U) rows of one kind (A / B / C: on the high x / y / z face of the cell), ST
// elements apart from y[0]; low: the rows lie on a low mesh face.
template <typename T, bool A, bool B, bool C, int U, int ST>
__device__ __forceinline__ void dss_rows(T* y, const DssLane& d, int count, bool low) {
  const bool X = A && d.h[0], Y = B && d.h[1], Z = C && d.h[2];
  const bool zero = d.mask && (low || (A && !X) || (B && !Y) || (C && !Z));
  if (!(X || Y || Z || zero)) return;
  T v[2][2][2][U];
#pragma unroll
  for (int c = 0; c <= (C ? 1 : 0); ++c)
#pragma unroll
    for (int b = 0; b <= (B ? 1 : 0); ++b)
#pragma unroll
      for (int a = 0; a <= (A ? 1 : 0); ++a) {
        const T* p = y + (a ? d.o[0] : 0) + (b ? d.o[1] : 0) + (c ? d.o[2] : 0);
        if (!zero && (a == 0 || X) && (b == 0 || Y) && (c == 0 || Z)) {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (u < count) v[c][b][a][u] = p[u * ST];
        }
      }
  T s[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    s[u] = T(0);
    if (!zero) {
      T sz[2];
#pragma unroll
      for (int c = 0; c <= (C ? 1 : 0); ++c) {
        T sy[2];
#pragma unroll
        for (int b = 0; b <= (B ? 1 : 0); ++b) {
          sy[b] = v[c][b][0][u];
          if (A && X) sy[b] = v[c][b][0][u] + v[c][b][1][u];
        }
        sz[c] = sy[0];
        if (B && Y) sz[c] = sy[0] + sy[1];
      }
      s[u] = sz[0];
      if (C && Z) s[u] = sz[0] + sz[1];
      if (d.avg) s[u] = s[u] * ((X ? T(0.5) : T(1)) * (Y ? T(0.5) : T(1)) * (Z ? T(0.5) : T(1)));
    }
  }
#pragma unroll
  for (int c = 0; c <= (C ? 1 : 0); ++c)
#pragma unroll
    for (int b = 0; b <= (B ? 1 : 0); ++b)
#pragma unroll
      for (int a = 0; a <= (A ? 1 : 0); ++a) {
        T* p = y + (a ? d.o[0] : 0) + (b ? d.o[1] : 0) + (c ? d.o[2] : 0);
        if ((a == 0 || X) && (b == 0 || Y) && (c == 0 || Z)) {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (u < count) p[u * ST] = s[u];
        }
      }
}

// Warp u of the launch: chunk u % CHUNKS of tile u / CHUNKS for u < nmain, then row by row the
// LOW rows of the low-face tiles (the layer tz = 0, then ty = 0, then tx = 0 of the rest).
template <typename T, int N>
__global__ void __launch_bounds__(DSS_THREADS) dss_kernel(T* y, GridInfo g, int avg, long long nmain, long long nunits) {
  using D = DssCfg<N>;
  constexpr int K = N - 1, N2 = N * N, N3 = N2 * N, U = D::U, CL = D::CL, E1 = D::E > 0 ? D::E : 1;
  pdl_enter();
  const long long u = (long long)blockIdx.x * (DSS_THREADS / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (u >= nunits) return;
  const bool low = u >= nmain;
  const long long v = low ? u - nmain : u;
  long long t = low ? v / D::LOW : v / D::CHUNKS;
  const int q = (int)(low ? v - t * D::LOW : v - t * D::CHUNKS);
  if (low) { // the t-th low-face tile
    const long long nxy = (long long)g.ntx * g.nty, nxz = (long long)g.ntx * (g.ntz - 1);
    if (t >= nxy) {
      long long r = t - nxy;
      if (r < nxz) { // ty = 0, tz >= 1
        t = (1 + r / g.ntx) * nxy + r % g.ntx;
      } else { // tx = 0, ty, tz >= 1
        r -= nxz;
        t = (1 + r / (g.nty - 1)) * nxy + (1 + r % (g.nty - 1)) * g.ntx;
      }
    }
  }
  int cx, cy, cz;
  cell_of(g, t, lane, cx, cy, cz);
  if (cx >= g.nx || cy >= g.ny || cz >= g.nz) return; // padding lane (no warp-wide operation below)
  const int lx = lane & 3, ly = (lane >> 2) & 3, lz = lane >> 4;
  const long long tile_el = (long long)N3 * BL;
  DssLane d;
  d.h[0] = cx < g.nx - 1;
  d.h[1] = cy < g.ny - 1;
  d.h[2] = cz < g.nz - 1;
  d.o[0] = lx < TX - 1 ? 1 - K * BL : tile_el - K * BL - (TX - 1);
  d.o[1] = ly < TY - 1 ? TX - K * N * BL : g.ntx * tile_el - K * N * BL - TX * (TY - 1);
  d.o[2] =
      lz < TZ - 1 ? TX * TY - K * N2 * BL : (long long)g.ntx * g.nty * tile_el - K * N2 * BL - TX * TY * (TZ - 1);
  d.mask = g.bc && !avg;
  d.avg = avg;
  T* y0 = y + t * tile_el + lane;
  if (low) {
    int i, j, k, r = q; // row q of those with a zero index: k = 0, then j = 0, then i = 0
    if (r < N2) {
      k = 0; j = r / N; i = r % N;
    } else if ((r -= N2) < N * K) {
      j = 0; k = 1 + r / N; i = r % N;
    } else {
      r -= N * K;
      i = 0; j = 1 + r % K; k = 1 + r / K;
    }
    if ((i == 0 && cx > 0) || (j == 0 && cy > 0) || (k == 0 && cz > 0)) return; // not the lowest copy
    T* p = y0 + (i + N * j + N2 * k) * BL;
    switch ((i == K ? 1 : 0) | (j == K ? 2 : 0) | (k == K ? 4 : 0)) { // uniform
      case 0: dss_rows<T, false, false, false, 1, 0>(p, d, 1, true); break;
      case 1: dss_rows<T, true, false, false, 1, 0>(p, d, 1, true); break;
      case 2: dss_rows<T, false, true, false, 1, 0>(p, d, 1, true); break;
      case 3: dss_rows<T, true, true, false, 1, 0>(p, d, 1, true); break;
      case 4: dss_rows<T, false, false, true, 1, 0>(p, d, 1, true); break;
      case 5: dss_rows<T, true, false, true, 1, 0>(p, d, 1, true); break;
      default: dss_rows<T, false, true, true, 1, 0>(p, d, 1, true); break; // one index is 0: never all three
    }
    return;
  }
  // rows with i, j, k >= 1 on a high face of the cell
  if (q == 0) {
    dss_rows<T, true, true, true, 1, 0>(y0 + (K + N * K + N2 * K) * BL, d, 1, false);
    return;
  }
  // line: 0..2 the edges along x, y, z; then E lines on each of the z, y and x faces
  const int line = (q - 1) / CL, first = 1 + ((q - 1) - line * CL) * U, count = min(U, K - first);
  if (line < 3) {
    if (line == 0) dss_rows<T, false, true, true, U, BL>(y0 + (first + N * K + N2 * K) * BL, d, count, false);
    else if (line == 1) dss_rows<T, true, false, true, U, N * BL>(y0 + (K + N * first + N2 * K) * BL, d, count, false);
    else dss_rows<T, true, true, false, U, N2 * BL>(y0 + (K + N * K + N2 * first) * BL, d, count, false);
  } else {
    const int f = (line - 3) / E1, m = 1 + (line - 3) - f * E1;
    if (f == 0) dss_rows<T, false, false, true, U, BL>(y0 + (first + N * m + N2 * K) * BL, d, count, false);
    else if (f == 1) dss_rows<T, false, true, false, U, BL>(y0 + (first + N * K + N2 * m) * BL, d, count, false);
    else dss_rows<T, true, false, false, U, N * BL>(y0 + (K + N * first + N2 * m) * BL, d, count, false);
  }
}

// ---------------------------------------------------------------------------------------
// Atomic duplicate summation (ablation of dss_kernel): pass 1 adds every copy into its
// unique node's accumulator with atomicAdd; pass 2 writes the accumulated sum (zero on the
// Dirichlet boundary) back to every copy.  One thread per native element in both passes.
// ---------------------------------------------------------------------------------------
template <int N>
__device__ __forceinline__ bool unique_of(const GridInfo& g, long long e, long long* I, bool* bnd) {
  constexpr int K = N - 1, N2 = N * N, N3 = N2 * N;
  const int lane = (int)(e % BL);
  const int l = (int)((e / BL) % N3);
  const long long t = e / ((long long)BL * N3);
  int cx, cy, cz;
  cell_of(g, t, lane, cx, cy, cz);
  if (cx >= g.nx || cy >= g.ny || cz >= g.nz) return false;
  const long long NX = (long long)g.nx * K + 1, NY = (long long)g.ny * K + 1, NZ = (long long)g.nz * K + 1;
  const long long gi = (long long)cx * K + l % N, gj = (long long)cy * K + (l / N) % N, gk = (long long)cz * K + l / N2;
  *I = gi + NX * (gj + NY * gk);
  *bnd = g.bc && (gi == 0 || gi == NX - 1 || gj == 0 || gj == NY - 1 || gk == 0 || gk == NZ - 1);
  return true;
}
template <typename T, int N>
__global__ void dss_atomic_add_kernel(const T* __restrict__ y, T* __restrict__ acc, GridInfo g, long long n) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    long long I;
    bool bnd;
    if (unique_of<N>(g, e, &I, &bnd) && !bnd) atomicAdd(&acc[I], y[e]);
  }
}
template <typename T, int N>
__global__ void dss_atomic_read_kernel(T* __restrict__ y, const T* __restrict__ acc, GridInfo g, long long n) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    long long I;
    bool bnd;
    if (unique_of<N>(g, e, &I, &bnd)) y[e] = bnd ? T(0) : acc[I];
  }
}
template <int N>
mf_status dss_atomic_n(const mf_operator* op, int elem, void* y, void* acc, cudaStream_t s) {
  const long long n = op->n_native;
  const int thr = 256;
  long long blocks = (n + thr - 1) / thr;
  if (blocks > 152 * 32) blocks = 152 * 32;
  mf_status st = cuda_check(cudaMemsetAsync(acc, 0, (size_t)op->n_unique * elem, s), "dss atomic clear");
  if (st) return st;
  if (elem == 8) {
    dss_atomic_add_kernel<double, N><<<(unsigned)blocks, thr, 0, s>>>((const double*)y, (double*)acc, op->g, n);
    dss_atomic_read_kernel<double, N><<<(unsigned)blocks, thr, 0, s>>>((double*)y, (const double*)acc, op->g, n);
  } else {
    dss_atomic_add_kernel<float, N><<<(unsigned)blocks, thr, 0, s>>>((const float*)y, (float*)acc, op->g, n);
    dss_atomic_read_kernel<float, N><<<(unsigned)blocks, thr, 0, s>>>((float*)y, (const float*)acc, op->g, n);
  }
  return cuda_check(cudaGetLastError(), "dss atomic launch");
}

// ---------------------------------------------------------------------------------------
// Stream twin of the apply (Sec. 6 times such memory-only kernels as the ceiling of an access
// pattern): the apply's grid and cells per CTA (CC) and its global accesses -- the x tile read
// into shared memory, the NC metric words of every point of the thread's z pencil read as the
// streamed geometry, y written by x-pencils -- and none of the contractions.  y is a bit-copy
// of x: the metric words are folded by XOR and tested against a mask that the host passes as
// zero, which keeps their loads live without changing y.
// ---------------------------------------------------------------------------------------
template <typename E, int N, int CC, int NC>
__global__ void __launch_bounds__(N * N * CC) stream_twin_kernel(const E* __restrict__ x, E* __restrict__ y,
                                                                  const unsigned long long* __restrict__ geom,
                                                                  unsigned long long mask) {
  constexpr int N2 = N * N, N3 = N2 * N, NT = N2 * CC, GPT = BL / CC;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  E* buf = reinterpret_cast<E*>(smem_raw);
  const long long t = blockIdx.x / GPT;
  const int lane0 = (int)(blockIdx.x % GPT) * CC;
  const long long base = t * (long long)N3 * BL + lane0;
  for (int idx = threadIdx.x; idx < N3 * CC; idx += NT) {
    const int l = idx / CC, c = idx - l * CC;
    buf[idx] = x[base + (long long)l * BL + c];
  }
  __syncthreads();
  const int c = threadIdx.x % CC, p = threadIdx.x / CC, pa = p % N, pb = p / N;
  if constexpr (NC > 0) {
    const unsigned long long* gp = geom + t * (long long)NC * N3 * BL + lane0 + c;
    unsigned long long acc = 0;
#pragma unroll
    for (int q = 0; q < N; ++q)
#pragma unroll
      for (int m = 0; m < NC; ++m) acc ^= gp[(long long)(m * N3 + pa + N * pb + N2 * q) * BL];
    if ((acc & mask) != 0) buf[(pa + N * pb) * CC + c] = E(0);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int l = i + N * pa + N2 * pb;
    y[base + (long long)l * BL + c] = buf[l * CC + c];
  }
}
template <typename E, int N, int CC>
static mf_status stream_twin_cc(const mf_operator* op, const void* x, void* y, const void* geom, int nc,
                                cudaStream_t s) {
  constexpr int NT = N * N * CC;
  const long long blocks = op->g.ntiles * (BL / CC);
  const size_t smem = sizeof(E) * N * N * N * CC;
  if (blocks <= 0) return MF_OK;
  void (*k)(const E*, E*, const unsigned long long*, unsigned long long) =
      nc == 7 ? stream_twin_kernel<E, N, CC, 7> : (nc == 6 ? stream_twin_kernel<E, N, CC, 6> : stream_twin_kernel<E, N, CC, 0>);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_check(e, "cudaFuncSetAttribute(stream twin)");
  }
  k<<<(unsigned)blocks, NT, smem, s>>>(static_cast<const E*>(x), static_cast<E*>(y),
                                       static_cast<const unsigned long long*>(geom), 0ull);
  return cuda_check(cudaGetLastError(), "stream twin launch");
}
// vk: the view mf_apply uses; geom / nc: the streamed metric (nullptr / 0 when there is none).
// Cells per CTA follow the view's compute type and the operator's launch variant.
template <int N>
mf_status stream_twin_n(const mf_operator* op, int vk, const void* x, void* y, const void* geom, int nc,
                        cudaStream_t s) {
  const int var = op->variant[vk == VK_DDS ? VK_DD : vk];
  const bool half = var == 1 || var == 2 || (var == MF_VARIANT_SMALL_CTA && vk != VK_F32);
  if (vk == VK_F32) {
    using C0 = Cfg<FP32C, N, 0>;
    using CH = Cfg<FP32C, N, 1>;
    return half ? stream_twin_cc<unsigned, N, CH::CB * CH::CPL>(op, x, y, nullptr, 0, s)
                : stream_twin_cc<unsigned, N, C0::CB * C0::CPL>(op, x, y, nullptr, 0, s);
  }
  using D0 = Cfg<dd, N, 0>;
  using DH = Cfg<dd, N, 1>;
  return half ? stream_twin_cc<unsigned long long, N, DH::CB>(op, x, y, geom, nc, s)
              : stream_twin_cc<unsigned long long, N, D0::CB>(op, x, y, geom, nc, s);
}

// ---------------------------------------------------------------------------------------
// Per-point geometry of the curved map (Sec. 2: six metric entries plus det J per point):
// G = w |det J| J^-1 J^-T (xx,xy,xz,yy,yz,zz) and, for Helmholtz, m = w |det J| c_m, computed
// in FP64 from the analytic Jacobian and stored in T, layout [tile][comp][l][lane].
// ---------------------------------------------------------------------------------------
struct GeomArgsQ {
  double qx[MAXN];
};

// FP32 curved view: sin(pi xh) and pi cos(pi xh) at the Gauss points of every cell layer, per
// direction ([(nx+ny+nz) * N][2] floats), computed in FP64 once at set-up.
template <int N>
__global__ void geom_table_kernel(float* tab, GridInfo g, GeomArgsQ q) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (g.nx + g.ny + g.nz) * N) return;
  const int r = e / N, qq = e - r * N;
  const int nd = r < g.nx ? g.nx : (r < g.nx + g.ny ? g.ny : g.nz);
  const int c = r < g.nx ? r : (r < g.nx + g.ny ? r - g.nx : r - g.nx - g.ny);
  double sp, cp;
  sincospi((c + q.qx[qq]) / nd, &sp, &cp);
  tab[2 * e] = (float)sp;
  tab[2 * e + 1] = (float)(3.141592653589793238462643383279502884 * cp);
}

template <typename T>
__device__ __forceinline__ T geom_value(double v) { return (T)v; }
template <>
__device__ __forceinline__ dd geom_value<dd>(double v) {
  const float h = __double2float_rn(v);
  return dd(h, __double2float_rn(v - (double)h));
}


struct GeomArgs {
  GridInfo g;
  double qx[MAXN], qw[MAXN];
  double amp, cm;
  int comps;
};

template <typename T, int N>
__global__ void geometry_kernel(T* __restrict__ geom, GeomArgs a) {
  constexpr int N2 = N * N, N3 = N2 * N;
  const long long total = a.g.ntiles * N3 * BL;
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int lane = (int)(e % BL);
  const int l = (int)((e / BL) % N3);
  const long long t = e / ((long long)BL * N3);
  int cx, cy, cz;
  cell_of(a.g, t, lane, cx, cy, cz);
  double out[7] = {0, 0, 0, 0, 0, 0, 0};
  if (cx < a.g.nx && cy < a.g.ny && cz < a.g.nz) {
    const int i = l % N, j = (l / N) % N, k = l / N2;
    const double xh[3] = {(cx + a.qx[i]) / a.g.nx, (cy + a.qx[j]) / a.g.ny, (cz + a.qx[k]) / a.g.nz};
    const double h[3] = {1.0 / a.g.nx, 1.0 / a.g.ny, 1.0 / a.g.nz};
    const double pi = 3.141592653589793238462643383279502884;
    double sn[3], cs[3];
    for (int d = 0; d < 3; ++d) sincospi(xh[d], &sn[d], &cs[d]);
    const double gs[3] = {pi * cs[0] * sn[1] * sn[2], pi * sn[0] * cs[1] * sn[2], pi * sn[0] * sn[1] * cs[2]};
    double J[3][3];
    for (int r = 0; r < 3; ++r)
      for (int d = 0; d < 3; ++d) J[r][d] = ((r == d) ? 1.0 : 0.0) * h[d] + a.amp * gs[d] * h[d];
    const double c00 = J[1][1] * J[2][2] - J[1][2] * J[2][1];
    const double c01 = J[1][2] * J[2][0] - J[1][0] * J[2][2];
    const double c02 = J[1][0] * J[2][1] - J[1][1] * J[2][0];
    const double det = J[0][0] * c00 + J[0][1] * c01 + J[0][2] * c02;
    const double id = 1.0 / det;
    double Ji[3][3]; // inverse
    Ji[0][0] = c00 * id; Ji[1][0] = c01 * id; Ji[2][0] = c02 * id;
    Ji[0][1] = (J[0][2] * J[2][1] - J[0][1] * J[2][2]) * id;
    Ji[1][1] = (J[0][0] * J[2][2] - J[0][2] * J[2][0]) * id;
    Ji[2][1] = (J[0][1] * J[2][0] - J[0][0] * J[2][1]) * id;
    Ji[0][2] = (J[0][1] * J[1][2] - J[0][2] * J[1][1]) * id;
    Ji[1][2] = (J[0][2] * J[1][0] - J[0][0] * J[1][2]) * id;
    Ji[2][2] = (J[0][0] * J[1][1] - J[0][1] * J[1][0]) * id;
    const double wd = a.qw[i] * a.qw[j] * a.qw[k] * fabs(det);
    const int pr[6][2] = {{0, 0}, {0, 1}, {0, 2}, {1, 1}, {1, 2}, {2, 2}};
    for (int m = 0; m < 6; ++m) {
      const int r = pr[m][0], s = pr[m][1];
      out[m] = wd * (Ji[r][0] * Ji[s][0] + Ji[r][1] * Ji[s][1] + Ji[r][2] * Ji[s][2]);
    }
    out[6] = wd * a.cm;
  }
  for (int m = 0; m < a.comps; ++m) geom[((t * a.comps + m) * N3 + l) * BL + lane] = geom_value<T>(out[m]);
}

// ---------------------------------------------------------------------------------------
// Diagonal of the operator (Jacobi preconditioning, FP32): per cell-local node i,
// (A_K)_ii = sum_q grad phi_i^T G_q grad phi_i + m_q phi_i^2 with the same quadrature and
// metric as the apply (grad phi_i = (D S S, S D S, S S D) from the 1D GLL basis S and its
// derivative D at the Gauss points); the split diagonal is then summed over copies.
// ---------------------------------------------------------------------------------------
struct DiagArgs {
  GridInfo g;
  float S[MAXN * MAXN], D[MAXN * MAXN], W[MAXN];
  int curved;
  float G[6], mdet;                 // affine metric (w-free) and mass * det
  const float* gtab;                // curved: sin and pi cos of pi xh per cell layer and direction
  float amp, cm, h[3];
};

template <int N>
__global__ void diag_kernel(float* __restrict__ dg, DiagArgs a) {
  constexpr int N2 = N * N, N3 = N2 * N;
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= a.g.ntiles * N3 * BL) return;
  const int lane = (int)(e % BL);
  const int l = (int)((e / BL) % N3);
  const long long t = e / ((long long)BL * N3);
  int cx, cy, cz;
  cell_of(a.g, t, lane, cx, cy, cz);
  if (cx >= a.g.nx || cy >= a.g.ny || cz >= a.g.nz) {
    dg[e] = 0.0f;
    return;
  }
  const int ix = l % N, iy = (l / N) % N, iz = l / N2;
  const float* tx = a.gtab + 2 * (cx * N);
  const float* ty = a.gtab + 2 * ((a.g.nx + cy) * N);
  const float* tz = a.gtab + 2 * ((a.g.nx + a.g.ny + cz) * N);
  float acc = 0.0f;
  for (int qz = 0; qz < N; ++qz) {
    const float Sz = a.S[qz * MAXN + iz], Dz = a.D[qz * MAXN + iz];
    for (int qy = 0; qy < N; ++qy) {
      const float Sy = a.S[qy * MAXN + iy], Dy = a.D[qy * MAXN + iy];
#pragma unroll
      for (int qx = 0; qx < N; ++qx) {
        const float Sx = a.S[qx * MAXN + ix], Dx = a.D[qx * MAXN + ix];
        const float gx = Dx * Sy * Sz, gy = Sx * Dy * Sz, gz = Sx * Sy * Dz, ph = Sx * Sy * Sz;
        const float w = a.W[qx] * a.W[qy] * a.W[qz];
        float g0, g1, g2, g3, g4, g5, m;
        if (a.curved) {
          // the metric of the curved map (same closed form as the FP32 apply)
          const float sx = tx[2 * qx], cxv = tx[2 * qx + 1], sy = ty[2 * qy], cyv = ty[2 * qy + 1];
          const float sz = tz[2 * qz], czv = tz[2 * qz + 1];
          const float v1 = cxv * sy * sz, v2 = sx * cyv * sz, v3 = sx * sy * czv;
          const float beta = fmaf(a.amp, v1 + v2 + v3, 1.0f);
          const float au = a.amp / beta;
          const float c2 = au * au * (v1 * v1 + v2 * v2 + v3 * v3);
          const float wd = w * (a.h[0] * a.h[1] * a.h[2]) * fabsf(beta);
          const float i0 = 1.0f / a.h[0], i1 = 1.0f / a.h[1], i2 = 1.0f / a.h[2];
          g0 = wd * i0 * i0 * (1.0f - 2.0f * au * v1 + c2);
          g1 = wd * i0 * i1 * (c2 - au * (v1 + v2));
          g2 = wd * i0 * i2 * (c2 - au * (v1 + v3));
          g3 = wd * i1 * i1 * (1.0f - 2.0f * au * v2 + c2);
          g4 = wd * i1 * i2 * (c2 - au * (v2 + v3));
          g5 = wd * i2 * i2 * (1.0f - 2.0f * au * v3 + c2);
          m = wd * a.cm;
        } else {
          g0 = w * a.G[0]; g1 = w * a.G[1]; g2 = w * a.G[2];
          g3 = w * a.G[3]; g4 = w * a.G[4]; g5 = w * a.G[5];
          m = w * a.mdet;
        }
        acc += gx * (g0 * gx + 2.0f * (g1 * gy + g2 * gz)) + gy * (g3 * gy + 2.0f * g4 * gz) + g5 * gz * gz +
               m * ph * ph;
      }
    }
  }
  dg[e] = acc;
}

// diag (n_native floats) = the assembled diagonal (consistent; 0 on Dirichlet nodes and
// padding); gtab: (nx + ny + nz) * N * 2 floats of scratch for curved meshes
template <int N>
mf_status diagonal_n(const mf_operator* op, float* diag, float* gtab, cudaStream_t s) {
  DiagArgs a;
  a.g = op->g;
  const HostTables& h = op->tab;
  for (int q = 0; q < MAXN * MAXN; ++q) {
    a.S[q] = (float)h.S[q];
    a.D[q] = (float)h.D[q];
  }
  for (int q = 0; q < MAXN; ++q) a.W[q] = (float)h.qw[q];
  a.curved = op->path == PATH_CURVED;
  for (int m = 0; m < 6; ++m) a.G[m] = (float)op->G[m];
  a.mdet = (float)(op->kind == MF_HELMHOLTZ ? op->mdet : 0.0);
  a.gtab = gtab;
  a.amp = (float)op->mesh.amp;
  a.cm = (float)(op->kind == MF_HELMHOLTZ ? op->mass : 0.0);
  a.h[0] = 1.0f / op->g.nx;
  a.h[1] = 1.0f / op->g.ny;
  a.h[2] = 1.0f / op->g.nz;
  if (a.curved) {
    GeomArgsQ q;
    for (int i = 0; i < N; ++i) q.qx[i] = op->tab.qx[i];
    const int nt = (op->g.nx + op->g.ny + op->g.nz) * N;
    geom_table_kernel<N><<<(nt + 127) / 128, 128, 0, s>>>(gtab, op->g, q);
  }
  const long long total = op->g.ntiles * (long long)N * N * N * BL;
  diag_kernel<N><<<(unsigned)((total + 255) / 256), 256, 0, s>>>(diag, a);
  mf_status st = cuda_check(cudaGetLastError(), "diagonal launch");
  if (st) return st;
  return dss_n<N>(op, 4, diag, s);
}

// ---------------------------------------------------------------------------------------
// Layout conversion: canonical <-> native, unique -> native (gather G), native -> unique.
// ---------------------------------------------------------------------------------------
template <typename T, int N>
__global__ void layout_kernel(const T* __restrict__ in, T* __restrict__ out, GridInfo g, int mode) {
  constexpr int K = N - 1, N2 = N * N, N3 = N2 * N;
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long NX = (long long)g.nx * K + 1, NY = (long long)g.ny * K + 1, NZ = (long long)g.nz * K + 1;
  if (mode == LAYOUT_GATHER_UNIQUE) {
    if (e >= NX * NY * NZ) return;
    const long long I = e % NX, J = (e / NX) % NY, L = e / (NX * NY);
    const int cx = (int)min(I / K, (long long)g.nx - 1), cy = (int)min(J / K, (long long)g.ny - 1),
              cz = (int)min(L / K, (long long)g.nz - 1);
    const int i = (int)(I - (long long)cx * K), j = (int)(J - (long long)cy * K), k = (int)(L - (long long)cz * K);
    out[e] = in[native_index(g, N3, cx, cy, cz, i + N * j + N2 * k)];
    return;
  }
  // the other modes run over native elements
  if (e >= g.ntiles * N3 * BL) return;
  const int lane = (int)(e % BL);
  const int l = (int)((e / BL) % N3);
  const long long t = e / ((long long)BL * N3);
  int cx, cy, cz;
  cell_of(g, t, lane, cx, cy, cz);
  const bool valid = cx < g.nx && cy < g.ny && cz < g.nz;
  const long long cell = ((long long)cz * g.ny + cy) * g.nx + cx;
  if (mode == LAYOUT_TO_NATIVE) {
    out[e] = valid ? in[cell * N3 + l] : T(0);
  } else if (mode == LAYOUT_FROM_NATIVE) {
    if (valid) out[cell * N3 + l] = in[e];
  } else { // LAYOUT_SCATTER_UNIQUE
    if (!valid) { out[e] = T(0); return; }
    const int i = l % N, j = (l / N) % N, k = l / N2;
    const long long I = (long long)cx * K + i, J = (long long)cy * K + j, L = (long long)cz * K + k;
    out[e] = in[I + NX * (J + NY * L)];
  }
}

// ---------------------------------------------------------------------------------------
// Host-side launchers for one degree.
// ---------------------------------------------------------------------------------------
template <typename S, typename T>
static void fill_job(const mf_operator* op, ApplyJob<S, T>& a) {
  a.g = op->g;
  for (int m = 0; m < 6; ++m) a.G[m] = host_from_double<T>(op->G[m]);
  a.mdet = host_from_double<T>(op->mdet);
  a.gx = host_from_double<T>(op->gx);
  a.gy = host_from_double<T>(op->gy);
  a.gz = host_from_double<T>(op->gz);
  a.cmass = host_from_double<T>(op->cmass);
  a.gtab = static_cast<const float*>(op->v32.geom);
  a.amp = (float)op->mesh.amp;
  a.cm = (float)(op->kind == MF_HELMHOLTZ ? op->mass : 0.0);
  a.ih[0] = (float)op->g.nx;
  a.ih[1] = (float)op->g.ny;
  a.ih[2] = (float)op->g.nz;
  a.hdet = (float)(1.0 / ((double)op->g.nx * op->g.ny * op->g.nz));
  a.cg = CgFuse<S>{};
  a.pf_tiles = 0;
  a.pf_geom = 0;
}
// A(q, i) = a[q * MAXN + i], or a[i * MAXN + q] for the transpose
template <typename T, int N>
static void fill_eo(const double* a, bool transpose, EoTab<T, N>& e) {
  constexpr int H = N / 2, HE = (N + 1) / 2;
  auto A = [&](int q, int i) { return transpose ? a[i * MAXN + q] : a[q * MAXN + i]; };
  for (int q = 0; q < H; ++q) {
    for (int i = 0; i < H; ++i) {
      e.F[q * HE + i] = host_from_double<T>(0.5 * (A(q, i) + A(q, N - 1 - i)));
      e.G[q * H + i] = host_from_double<T>(0.5 * (A(q, i) - A(q, N - 1 - i)));
    }
    if (N % 2) e.F[q * HE + H] = host_from_double<T>(A(q, H));
  }
  if (N % 2)
    for (int i = 0; i < HE; ++i) e.Mid[i] = host_from_double<T>(A(H, i));
}

template <typename T, int N>
static void fill_tab(const mf_operator* op, Tab<T, N>& tab) {
  const HostTables& h = op->tab;
  fill_eo<T, N>(h.S, false, tab.eS);
  fill_eo<T, N>(h.S, true, tab.eSt);
  fill_eo<T, N>(h.Dc, false, tab.eD);
  fill_eo<T, N>(h.Dc, true, tab.eDt);
  fill_eo<T, N>(h.M, false, tab.eM);
  fill_eo<T, N>(h.K, false, tab.eK);
  for (int q = 0; q < N; ++q) tab.W[q] = host_from_double<T>(h.qw[q]);
  // fast diagonalisation (modes: HE symmetric, then H antisymmetric)
  constexpr int H = N / 2, HE = (N + 1) / 2;
  auto Wm = [&](int j, int m) { return h.Wfd[j * MAXN + m]; };
  for (int m = 0; m < HE; ++m) {
    for (int j = 0; j < H; ++j) tab.fd.Ff[m * HE + j] = host_from_double<T>(Wm(j, m));
    if (N % 2) tab.fd.Ff[m * HE + H] = host_from_double<T>(Wm(H, m));
  }
  for (int m = 0; m < H; ++m)
    for (int j = 0; j < H; ++j) tab.fd.Gf[m * H + j] = host_from_double<T>(Wm(j, HE + m));
  for (int j = 0; j < HE; ++j)
    for (int m = 0; m < HE; ++m) tab.fd.Fb[j * HE + m] = host_from_double<T>(Wm(j, m));
  for (int j = 0; j < H; ++j)
    for (int m = 0; m < H; ++m) tab.fd.Gb[j * H + m] = host_from_double<T>(Wm(j, HE + m));
  for (int m = 0; m < N; ++m) tab.fd.lam[m] = host_from_double<T>(h.lam[m]);
}

// L2 prefetch distance of an apply launch: MF_PREFETCH_WAVES waves of resident CTAs, in
// tiles (gpt CTAs per tile).  Occupancy and SM count are looked up once per kernel.
#ifndef MF_PREFETCH_WAVES
#define MF_PREFETCH_WAVES 1
#endif
// CTAs of a kernel resident on the whole GPU at once (SMs x occupancy), cached per kernel,
// dynamic shared memory and device; 2^31 - 1 when the query fails (then the launch is simply
// not persistent).
[[maybe_unused]] static long long resident_ctas(const void* kernel, int threads, size_t smem) {
  struct Entry {
    const void* k;
    size_t smem;
    int dev;
    long long ctas;
  };
  static Entry cache[64];
  static int ncache = 0;
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(mu);
  for (int i = 0; i < ncache; ++i)
    if (cache[i].k == kernel && cache[i].smem == smem && cache[i].dev == dev) return cache[i].ctas;
  int sms = 0, per_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  cudaGetLastError();
  const long long ctas = (sms > 0 && per_sm > 0) ? (long long)sms * per_sm : 0x7fffffffLL;
  if (ncache < 64) cache[ncache++] = Entry{kernel, smem, dev, ctas};
  return ctas;
}

[[maybe_unused]] static int prefetch_distance_tiles(const void* kernel, int threads, size_t smem, int gpt) {
  if (MF_PREFETCH_WAVES <= 0) return 0;
  struct Entry {
    const void* k;
    size_t smem;
    int dev, tiles;
  };
  static Entry cache[64];
  static int ncache = 0;
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(mu);
  for (int i = 0; i < ncache; ++i)
    if (cache[i].k == kernel && cache[i].smem == smem && cache[i].dev == dev) return cache[i].tiles;
  int sms = 0, per_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  cudaGetLastError(); // a failed query only turns the prefetch off
  const int tiles = (sms > 0 && per_sm > 0) ? MF_PREFETCH_WAVES * ((sms * per_sm + gpt - 1) / gpt) : 0;
  if (ncache < 64) cache[ncache++] = Entry{kernel, smem, dev, tiles};
  return tiles;
}

// Block-size sweep of Sec. 6 (B cells per CTA; a measurement entry): the registers are capped
// so that the resident threads per SM equal those of the base configuration (MINB * NT = 2 * NT of
// Cfg 0), which separates the block size from the register budget.
template <typename T, int N, int B, bool G>
struct BCfg {
  static constexpr int CPL = CellsPer<T>::value;
  static constexpr int CB = B / CPL;
  static constexpr int MINB = 2 * Cfg<T, N, 0>::CB / CB > 0 ? 2 * Cfg<T, N, 0>::CB / CB : 1;
  static constexpr int NT = N * N * CB;
  static constexpr bool GENERAL = G;
  static_assert(B >= 4 && BL % B == 0 && CB * CPL == B && NT <= 1024 && NT >= 32, "B cells per CTA: 4, 8, 16 or 32");
};
// B cells per CTA: a CTA of n^2 * B threads, at most 1024 and at least one full warp (the
// CTA reductions fold in warp 0)
template <int N, int B>
constexpr bool block_fits() { return N * N * B <= 1024 && N * N * B >= 32; }

// What a launch needs besides its arguments: the kernel, its CTA and grid.  K: the one-operator
// kernel's type or the batched one's.
template <typename K>
struct Shape {
  K kernel = nullptr;
  int threads = 0, ctas_per_tile = 1, tiles_per_cta = 1;
  size_t smem = 0;
  long long blocks(long long ntiles) const {
    return (ntiles * ctas_per_tile + tiles_per_cta - 1) / tiles_per_cta;
  }
};
// C: the pencil kernels' launch configuration (cells per CTA CB * CPL, MINB resident CTAs, NT threads)
template <typename S, typename T, int N, typename C>
static mf_status pencil_shape(const mf_operator* op, Shape<void (*)(ApplyArgs<S, T, N>)>& h) {
  const bool helm = op->kind == MF_HELMHOLTZ;
  // buffers of n^3 values per cell: Cartesian 1 (fast-diagonalised) or 2, general 3
  h.smem = (op->path == PATH_CARTESIAN ? (MF_CART_FD ? 1 : 2) : 3) * sizeof(T) * N * N * N * C::CB;
  h.threads = C::NT;
  h.ctas_per_tile = BL / (C::CB * C::CPL);
  if (op->path == PATH_CARTESIAN) {
    h.kernel = helm ? apply_cartesian<S, T, N, C::CB, C::MINB, true> : apply_cartesian<S, T, N, C::CB, C::MINB, false>;
  } else if constexpr (C::GENERAL) {
    if (op->path == PATH_AFFINE)
      h.kernel = helm ? apply_general<S, T, N, C::CB, C::MINB, false, true>
                      : apply_general<S, T, N, C::CB, C::MINB, false, false>;
    else
      h.kernel =
          helm ? apply_general<S, T, N, C::CB, C::MINB, true, true> : apply_general<S, T, N, C::CB, C::MINB, true, false>;
  } else {
    return set_error(MF_ERR_UNSUPPORTED, "block-size sweep: built for the Cartesian path at this degree");
  }
  return MF_OK;
}
// Launch variant 0 in full: a plane kernel (CFG_PLANE) or the pencil configuration measured
// fastest per degree, path and size on one GB300.  Any two give bitwise equal vectors, but a
// batch's members must share one (their CTAs and CG partials differ): see apply_config.
constexpr int CFG_PLANE = 6;
// Planes need enough CTAs: one CTA's pass is a long serial stretch per thread (FP32 curved Q4:
// 9.1 us on any mesh up to 12^3 cells, the pencil kernel 3.7; at 24^3, 216 CTAs, 13.3 against 16.4).
// FP32: from one CTA per SM (two tiles each), always where the stretch is short (n = 2;
// Cartesian up to n = 4).  Double-float: from 2048 tiles (split apply, us, plane / pencil: Q2
// Cartesian 32^3, 1024 tiles, 14.6 / 10.0; 40^3, 2000 tiles, 17.1 / 17.7; 48^3 26.3 / 27.9; 64^3 56.6 / 64.5;
// Q2 sheared 22.0 / 21.0, 35.6 / 38.9, 56.8 / 62.7, 133 / 145; Q1 curved 9.5 / 7.3, 11.2 / 11.0, 15.7 / 17.2,
// 36.8 / 40.5).  On CG's double-float vectors planes win from about 500 tiles (Q2 Cartesian 32^3 12.6 /
// 15.7), but one line serves both.
template <typename T, int N, int PATH>
constexpr long long plane_from_tiles() {
  return std::is_same<T, dd>::value ? 2048 : (N == 2 || (PATH == PATH_CARTESIAN && N <= 4) ? 0 : 304);
}
template <typename T, int N>
static bool use_plane(const mf_operator* op) {
  const long long t = op->g.ntiles;
  if (op->path == PATH_CARTESIAN)
    return UsePlane<T, N, PATH_CARTESIAN>::value && t >= plane_from_tiles<T, N, PATH_CARTESIAN>();
  if (op->path == PATH_AFFINE) return UsePlane<T, N, PATH_AFFINE>::value && t >= plane_from_tiles<T, N, PATH_AFFINE>();
  return UsePlane<T, N, PATH_CURVED>::value && t >= plane_from_tiles<T, N, PATH_CURVED>();
}
// Whether a batch's members (at most BATCH_MAX_TILES) ever take a plane kernel: FP32 where planes have no
// line.  The others are not built.
template <typename T, int N, int PATH>
constexpr bool plane_in_batch() {
  return UsePlane<T, N, PATH>::value && plane_from_tiles<T, N, PATH>() <= BATCH_MAX_TILES;
}
// Small meshes take variant 1's smaller CTAs: FP32 below the plane kernels' line, double-float
// up to 64 tiles (curved Q4 8^3 12.4 -> 8.4 us, Q6 19.7 -> 13.1, Cartesian Q6 11.3 -> 8.3; at 128
// tiles curved Q4 19.9 against 21.6).  Above, double-float (split apply, ms at ~17M DoFs, base
// configuration -> the chosen one).  Cartesian: Q3 0.174 -> 0.147, Q4 0.221 -> 0.178, Q5 0.218 ->
// 0.196, Q6 0.305 -> 0.255, Q7 0.219 -> 0.210, Q8 0.392 -> 0.347.  Affine: Q3 0.362 -> 0.335, Q4
// 0.459 -> 0.397, Q6 0.683 -> 0.632, the others stay.  Curved: Q2 0.361 -> 0.354 (Helmholtz 0.428 ->
// 0.364), Q3 0.367 -> 0.342, Q4 (Laplace) 0.453 -> 0.408, Q5 (Helmholtz) 0.601 -> 0.577, Q6 (Laplace)
// 0.691 -> 0.681, the others stay (Q8 would gain above 20^3 cells and lose below).  CG's apply on double-float
// vectors takes the same: there the choice loses in Cartesian Q7 (0.216 -> 0.229) and gains or is even
// elsewhere (curved Q4 0.488 -> 0.469; with variant 4, whose 40 registers spill there, 0.528).
template <typename T, int N>
static int pencil_config(const mf_operator* op) {
  if (IsF32<T>::value) return N <= (op->path == PATH_CARTESIAN ? 7 : 6) && op->g.ntiles < 304 ? 1 : 0;
  if (!std::is_same<T, dd>::value) return 0;
  if (op->g.ntiles <= 64) return 1;
  if (op->path == PATH_CARTESIAN) return N >= 7 ? MF_VARIANT_OCCUPANCY : (N >= 4 ? MF_VARIANT_SMALL_CTA : 0);
  if (op->path == PATH_AFFINE) return N == 4 ? MF_VARIANT_SMALL_CTA : (N == 5 || N == 7 ? MF_VARIANT_OCCUPANCY : 0);
  if (N == 3) return MF_VARIANT_SMALL_CTA;
  if (N == 4 || (N == 6 && op->kind == MF_HELMHOLTZ)) return 1;
  return (N == 5 || N == 7) && op->kind == MF_LAPLACE ? MF_VARIANT_OCCUPANCY : 0;
}
// The configuration of a pencil / plane launch with this variant (the tensor-core variant's
// operators run variant 0 where their vectors are not plain doubles).
template <typename T, int N>
static int config_of(const mf_operator* op, int variant) {
  if (variant != 0 && variant != MF_VARIANT_TENSOR) return variant;
  return use_plane<T, N>(op) ? CFG_PLANE : pencil_config<T, N>(op);
}
template <typename S, typename T, int N>
static void plane_shape(const mf_operator* op, Shape<void (*)(ApplyArgs<S, T, N>)>& h) {
  using P = PlaneCfg<T, N>;
  const bool helm = op->kind == MF_HELMHOLTZ;
  h.threads = P::NT;
  h.tiles_per_cta = P::TPC;
  h.smem = (op->path == PATH_CARTESIAN ? 1 : 2) * sizeof(T) * N * N * N * P::CB;
  if constexpr (UsePlane<T, N, PATH_CARTESIAN>::value)
    if (op->path == PATH_CARTESIAN)
      h.kernel = helm ? apply_cartesian_plane<S, T, N, true> : apply_cartesian_plane<S, T, N, false>;
  if constexpr (UsePlane<T, N, PATH_AFFINE>::value)
    if (op->path == PATH_AFFINE)
      h.kernel = helm ? apply_general_plane<S, T, N, false, true> : apply_general_plane<S, T, N, false, false>;
  if constexpr (UsePlane<T, N, PATH_CURVED>::value)
    if (op->path == PATH_CURVED)
      h.kernel = helm ? apply_general_plane<S, T, N, true, true> : apply_general_plane<S, T, N, true, false>;
}

template <typename S, typename T, int N>
static mf_status apply_launch(const mf_operator* op, const Shape<void (*)(ApplyArgs<S, T, N>)>& h, const void* x,
                              void* y, const void* geom, const CgFuse<S>& cg, long long* nblocks, cudaStream_t s) {
  ApplyArgs<S, T, N> a;
  fill_job<S, T>(op, a.j);
  fill_tab<typename CoefOf<T>::type, N>(op, a.tab);
  a.j.cg = cg;
  a.j.x = static_cast<const S*>(x);
  a.j.y = static_cast<S*>(y);
  a.j.geom = static_cast<const T*>(geom);
  const long long blocks = h.blocks(op->g.ntiles);
  if (nblocks) *nblocks = blocks;
  if (blocks <= 0) return MF_OK;
  if (h.smem > 227 * 1024)
    return set_error(MF_ERR_UNSUPPORTED, "apply variant needs %zu bytes of shared memory", h.smem);
  // the kernels also hold static shared memory (the CG partial's park, NT doubles, and a few
  // bytes of the compiler's), and static + dynamic above 48 KB needs the opt-in
  if (h.smem + sizeof(double) * h.threads + 1024 > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(h.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)h.smem);
    if (e != cudaSuccess) return cuda_check(e, "cudaFuncSetAttribute(apply)");
  }
  a.j.pf_tiles = prefetch_distance_tiles((const void*)h.kernel, h.threads, h.smem, h.ctas_per_tile) * h.tiles_per_cta;
  a.j.pf_geom = (op->path == PATH_CURVED && !IsF32<T>::value) ? 1 : 0;
  return cuda_check(launch_pdl(h.kernel, (unsigned)blocks, h.threads, h.smem, s, a), "apply launch");
}
template <typename S, typename T, int N, typename C>
static mf_status apply_split_c(const mf_operator* op, const void* x, void* y, const void* geom, const CgFuse<S>& cg,
                               long long* nblocks, cudaStream_t s) {
  Shape<void (*)(ApplyArgs<S, T, N>)> h;
  mf_status st = pencil_shape<S, T, N, C>(op, h);
  if (st) return st;
  return apply_launch<S, T, N>(op, h, x, y, geom, cg, nblocks, s);
}
template <typename S, typename T, int N, int V>
static mf_status apply_split_v(const mf_operator* op, const void* x, void* y, const void* geom, const CgFuse<S>& cg,
                               long long* nblocks, cudaStream_t s) {
  return apply_split_c<S, T, N, Cfg<T, N, V>>(op, x, y, geom, cg, nblocks, s);
}

// Degree 3 (n = 4, the degree of the paper's block-size experiment): every path, the
// double-float and FP32 views.  Other degrees: the Cartesian double-float apply.
template <int N, int B>
static mf_status apply_block_t(const mf_operator* op, int vk, const void* x, void* y, cudaStream_t s) {
  if constexpr (!block_fits<N, B>()) {
    return set_error(MF_ERR_UNSUPPORTED, "mf_apply_split_block: %d cells of degree %d do not make a CTA of 32..1024 threads",
                     B, N - 1);
  } else {
    constexpr bool all = N == 4;
    if (vk == VK_DD)
      return apply_split_c<double, dd, N, BCfg<dd, N, B, all>>(op, x, y, op->v64.geom, CgFuse<double>{}, nullptr, s);
    if constexpr (all) {
      if (vk == VK_F32)
        return apply_split_c<float, FP32C, N, BCfg<FP32C, N, B, true>>(op, x, y, op->v32.geom, CgFuse<float>{},
                                                                       nullptr, s);
    }
    return set_error(MF_ERR_UNSUPPORTED, "mf_apply_split_block: MF_FP64 (double-float)%s operators only",
                     all ? " or MF_FP32" : "");
  }
}
template <int N>
mf_status apply_block_n(const mf_operator* op, int vk, int cells, const void* x, void* y, cudaStream_t s) {
  switch (cells) {
    case 4: return apply_block_t<N, 4>(op, vk, x, y, s);
    case 8: return apply_block_t<N, 8>(op, vk, x, y, s);
    case 16: return apply_block_t<N, 16>(op, vk, x, y, s);
    case 32: return apply_block_t<N, 32>(op, vk, x, y, s);
    default: return set_error(MF_ERR_ARG, "mf_apply_split_block: cells per CTA must be 4, 8, 16 or 32");
  }
}

template <typename S, typename T, int N>
static mf_status apply_split_t(const mf_operator* op, int variant, const void* x, void* y, const void* geom,
                               const CgFuse<S>& cg, long long* nblocks, cudaStream_t s) {
  variant = config_of<T, N>(op, variant);
  if (variant == CFG_PLANE) {
    Shape<void (*)(ApplyArgs<S, T, N>)> h;
    plane_shape<S, T, N>(op, h);
    return apply_launch<S, T, N>(op, h, x, y, geom, cg, nblocks, s);
  }
  if (variant == 1) return apply_split_v<S, T, N, 1>(op, x, y, geom, cg, nblocks, s);
  if (variant == 2) return apply_split_v<S, T, N, 2>(op, x, y, geom, cg, nblocks, s);
  if constexpr (std::is_same<T, dd>::value) {
    if (variant == MF_VARIANT_SMALL_CTA) return apply_split_v<S, T, N, 4>(op, x, y, geom, cg, nblocks, s);
    if (variant == MF_VARIANT_OCCUPANCY) return apply_split_v<S, T, N, 5>(op, x, y, geom, cg, nblocks, s);
  }
  return apply_split_v<S, T, N, 0>(op, x, y, geom, cg, nblocks, s);
}

template <int N>
int apply_config_n(const mf_operator* op, int vk) {
  const int v = op->variant[vk == VK_DDS ? VK_DD : vk];
  if (vk == VK_F32) return config_of<FP32C, N>(op, v);
  return vk == VK_F64 ? config_of<double, N>(op, v) : config_of<dd, N>(op, v);
}

// vk: VK_F64 (double storage, native FP64 compute), VK_DD (double storage, double-float
// compute), VK_F32 (float storage and compute).
template <int N>
mf_status apply_split_n(const mf_operator* op, int vk, const void* x, void* y, cudaStream_t s) {
  const int v = op->variant[vk == VK_DDS ? VK_DD : vk];
  // the tensor-core apply stages x with 16-byte bulk copies; other x take the variant-0 kernel
  if (vk == VK_DD && v == MF_VARIANT_TENSOR && (reinterpret_cast<uintptr_t>(x) & 15) == 0)
    return tc_apply(op, x, y, s);
  if (vk == VK_F64) return apply_split_t<double, double, N>(op, v, x, y, op->v64.geom, CgFuse<double>{}, nullptr, s);
  if (vk == VK_DD) return apply_split_t<double, dd, N>(op, v, x, y, op->v64.geom, CgFuse<double>{}, nullptr, s);
  if (vk == VK_DDS) return apply_split_t<dd, dd, N>(op, v, x, y, op->v64.geom, CgFuse<dd>{}, nullptr, s);
  return apply_split_t<float, FP32C, N>(op, v, x, y, op->v32.geom, CgFuse<float>{}, nullptr, s);
}

template <int N>
mf_status apply_cg_n(const mf_operator* op, int vk, void* p, const void* r, void* y, CgState* st, double* partials,
                     int update_p, long long* nblocks, cudaStream_t s) {
  const int v = op->variant[vk == VK_DDS ? VK_DD : vk];
  void* x = update_p ? nullptr : p;
  if (vk == VK_F32) {
    const CgFuse<float> cg{static_cast<float*>(p), static_cast<const float*>(r), st, partials, update_p};
    return apply_split_t<float, FP32C, N>(op, v, x, y, op->v32.geom, cg, nblocks, s);
  }
  if (vk == VK_DDS) {
    const CgFuse<dd> cg{static_cast<dd*>(p), static_cast<const dd*>(r), st, partials, update_p};
    return apply_split_t<dd, dd, N>(op, v, x, y, op->v64.geom, cg, nblocks, s);
  }
  const CgFuse<double> cg{static_cast<double*>(p), static_cast<const double*>(r), st, partials, update_p};
  if (vk == VK_F64) return apply_split_t<double, double, N>(op, v, x, y, op->v64.geom, cg, nblocks, s);
  return apply_split_t<double, dd, N>(op, v, x, y, op->v64.geom, cg, nblocks, s);
}

// ---------------------------------------------------------------------------------------
// Batched CG-step apply over several operators of one degree, path, kind, view and launch
// variant (the serving loop's continuous batch).  apply_batch_fill_n writes the jobs' device
// descriptions and block offsets into host staging; apply_batch_launch_n launches one kernel
// over all of them (tables from op0: they depend only on the degree).
// ---------------------------------------------------------------------------------------
template <typename S, typename T, int N, int V>
static mf_status batch_fill_v(const BatchMember* m, int n, int vk, void* jobs_host, long long* block0_host) {
  using C = Cfg<T, N, V>;
  ApplyJob<S, T>* jobs = static_cast<ApplyJob<S, T>*>(jobs_host);
  long long b = 0;
  for (int i = 0; i < n; ++i) {
    const mf_operator* op = m[i].op;
    ApplyJob<S, T>& a = jobs[i];
    fill_job<S, T>(op, a);
    a.cg = CgFuse<S>{static_cast<S*>(m[i].p), static_cast<const S*>(m[i].r), m[i].st, m[i].apart, 0};
    a.x = static_cast<const S*>(m[i].p);
    a.y = static_cast<S*>(m[i].q);
    a.geom = static_cast<const T*>(vk == VK_F32 ? op->v32.geom : op->v64.geom);
    block0_host[i] = b;
    b += V == CFG_PLANE ? PlaneCfg<T, N>::blocks(op->g.ntiles) : op->g.ntiles * (BL / (C::CB * C::CPL));
  }
  block0_host[n] = b;
  return MF_OK;
}

template <typename S, typename T, int N, int V>
static mf_status batch_launch_v(const mf_operator* op0, const void* jobs_dev, const long long* block0_dev, int njobs,
                                long long blocks, cudaStream_t s) {
  using C = Cfg<T, N, V>;
  ApplyBatch<S, T, N> B;
  fill_tab<typename CoefOf<T>::type, N>(op0, B.tab);
  B.jobs = static_cast<const ApplyJob<S, T>*>(jobs_dev);
  B.block0 = block0_dev;
  B.njobs = njobs;
  const bool helm = op0->kind == MF_HELMHOLTZ;
  if (blocks <= 0 || njobs <= 0) return MF_OK;
  Shape<void (*)(ApplyBatch<S, T, N>)> h;
  if constexpr (V == CFG_PLANE) {
    using P = PlaneCfg<T, N>;
    h.threads = P::NT;
    h.smem = (op0->path == PATH_CARTESIAN ? 1 : 2) * sizeof(T) * N * N * N * P::CB;
    if constexpr (plane_in_batch<T, N, PATH_CARTESIAN>())
      if (op0->path == PATH_CARTESIAN)
        h.kernel = helm ? apply_cartesian_plane_batch<S, T, N, true> : apply_cartesian_plane_batch<S, T, N, false>;
    if constexpr (plane_in_batch<T, N, PATH_AFFINE>())
      if (op0->path == PATH_AFFINE)
        h.kernel =
            helm ? apply_general_plane_batch<S, T, N, false, true> : apply_general_plane_batch<S, T, N, false, false>;
    if constexpr (plane_in_batch<T, N, PATH_CURVED>())
      if (op0->path == PATH_CURVED)
        h.kernel = helm ? apply_general_plane_batch<S, T, N, true, true> : apply_general_plane_batch<S, T, N, true, false>;
    if (!h.kernel) return set_error(MF_ERR_UNSUPPORTED, "batch: members above %lld tiles", BATCH_MAX_TILES);
  } else {
    h.threads = C::NT;
    h.smem = (op0->path == PATH_CARTESIAN ? (MF_CART_FD ? 1 : 2) : 3) * sizeof(T) * N * N * N * C::CB;
    if (op0->path == PATH_CARTESIAN)
      h.kernel =
          helm ? apply_cartesian_batch<S, T, N, C::CB, C::MINB, true> : apply_cartesian_batch<S, T, N, C::CB, C::MINB, false>;
    else if (op0->path == PATH_AFFINE)
      h.kernel = helm ? apply_general_batch<S, T, N, C::CB, C::MINB, false, true>
                      : apply_general_batch<S, T, N, C::CB, C::MINB, false, false>;
    else
      h.kernel = helm ? apply_general_batch<S, T, N, C::CB, C::MINB, true, true>
                      : apply_general_batch<S, T, N, C::CB, C::MINB, true, false>;
  }
  if (h.smem > 227 * 1024)
    return set_error(MF_ERR_UNSUPPORTED, "apply variant needs %zu bytes of shared memory", h.smem);
  if (h.smem + sizeof(double) * h.threads + sizeof(ApplyJob<S, T>) + 1024 > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(h.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)h.smem);
    if (e != cudaSuccess) return cuda_check(e, "cudaFuncSetAttribute(batched apply)");
  }
  // one persistent launch: the CTAs resident on the GPU at once, looping over the units
  B.nunits = blocks;
  const long long grid = std::min<long long>(blocks, resident_ctas((const void*)h.kernel, h.threads, h.smem));
  return cuda_check(launch_pdl(h.kernel, (unsigned)grid, h.threads, h.smem, s, B), "batched apply launch");
}

template <typename S, typename T, int N>
static mf_status batch_fill_t(const BatchMember* m, int n, int vk, int variant, void* jobs_host, long long* block0_host) {
  variant = config_of<T, N>(m[0].op, variant);
  if (variant == CFG_PLANE) return batch_fill_v<S, T, N, CFG_PLANE>(m, n, vk, jobs_host, block0_host);
  if (variant == 1) return batch_fill_v<S, T, N, 1>(m, n, vk, jobs_host, block0_host);
  if (variant == 2) return batch_fill_v<S, T, N, 2>(m, n, vk, jobs_host, block0_host);
  if constexpr (std::is_same<T, dd>::value) {
    if (variant == MF_VARIANT_SMALL_CTA) return batch_fill_v<S, T, N, 4>(m, n, vk, jobs_host, block0_host);
    if (variant == MF_VARIANT_OCCUPANCY) return batch_fill_v<S, T, N, 5>(m, n, vk, jobs_host, block0_host);
  }
  return batch_fill_v<S, T, N, 0>(m, n, vk, jobs_host, block0_host);
}
template <typename S, typename T, int N>
static mf_status batch_launch_t(const mf_operator* op0, int variant, const void* jobs_dev, const long long* block0_dev,
                                int njobs, long long blocks, cudaStream_t s) {
  variant = config_of<T, N>(op0, variant);
  if (variant == CFG_PLANE) return batch_launch_v<S, T, N, CFG_PLANE>(op0, jobs_dev, block0_dev, njobs, blocks, s);
  if (variant == 1) return batch_launch_v<S, T, N, 1>(op0, jobs_dev, block0_dev, njobs, blocks, s);
  if (variant == 2) return batch_launch_v<S, T, N, 2>(op0, jobs_dev, block0_dev, njobs, blocks, s);
  if constexpr (std::is_same<T, dd>::value) {
    if (variant == MF_VARIANT_SMALL_CTA)
      return batch_launch_v<S, T, N, 4>(op0, jobs_dev, block0_dev, njobs, blocks, s);
    if (variant == MF_VARIANT_OCCUPANCY)
      return batch_launch_v<S, T, N, 5>(op0, jobs_dev, block0_dev, njobs, blocks, s);
  }
  return batch_launch_v<S, T, N, 0>(op0, jobs_dev, block0_dev, njobs, blocks, s);
}

template <int N>
mf_status apply_batch_fill_n(const BatchMember* m, int n, int vk, void* jobs_host, long long* block0_host) {
  const int v = m[0].op->variant[vk == VK_DDS ? VK_DD : vk];
  if (vk == VK_F32) return batch_fill_t<float, FP32C, N>(m, n, vk, v, jobs_host, block0_host);
  if (vk == VK_DDS) return batch_fill_t<dd, dd, N>(m, n, vk, v, jobs_host, block0_host);
  if (vk == VK_DD) return batch_fill_t<double, dd, N>(m, n, vk, v, jobs_host, block0_host);
  return batch_fill_t<double, double, N>(m, n, vk, v, jobs_host, block0_host);
}
template <int N>
mf_status apply_batch_launch_n(const mf_operator* op0, int vk, const void* jobs_dev, const long long* block0_dev,
                               int njobs, long long blocks, cudaStream_t s) {
  const int v = op0->variant[vk == VK_DDS ? VK_DD : vk];
  if (vk == VK_F32) return batch_launch_t<float, FP32C, N>(op0, v, jobs_dev, block0_dev, njobs, blocks, s);
  if (vk == VK_DDS) return batch_launch_t<dd, dd, N>(op0, v, jobs_dev, block0_dev, njobs, blocks, s);
  if (vk == VK_DD) return batch_launch_t<double, dd, N>(op0, v, jobs_dev, block0_dev, njobs, blocks, s);
  return batch_launch_t<double, double, N>(op0, v, jobs_dev, block0_dev, njobs, blocks, s);
}
template <int N>
static mf_status dss_mode(const mf_operator* op, int elem, void* y, int avg, cudaStream_t s) {
  const GridInfo& g = op->g;
  const long long nlow = g.ntiles - (long long)(g.ntx - 1) * (g.nty - 1) * (g.ntz - 1);
  const long long nmain = g.ntiles * DssCfg<N>::CHUNKS, units = nmain + nlow * DssCfg<N>::LOW;
  const unsigned blocks = (unsigned)((units + DSS_THREADS / 32 - 1) / (DSS_THREADS / 32));
  const cudaError_t e =
      elem == 8 ? launch_pdl(dss_kernel<double, N>, blocks, DSS_THREADS, 0, s, static_cast<double*>(y), g, avg, nmain, units)
                : launch_pdl(dss_kernel<float, N>, blocks, DSS_THREADS, 0, s, static_cast<float*>(y), g, avg, nmain, units);
  return cuda_check(e, "dss launch");
}
template <int N>
mf_status dss_n(const mf_operator* op, int elem, void* y, cudaStream_t s) {
  return dss_mode<N>(op, elem, y, 0, s);
}
template <int N>
mf_status make_consistent_n(const mf_operator* op, int elem, void* y, cudaStream_t s) {
  return dss_mode<N>(op, elem, y, 1, s);
}

template <int N>
mf_status geometry_n(const mf_operator* op, int vk, void* geom, cudaStream_t s) {
  GeomArgs a;
  a.g = op->g;
  for (int q = 0; q < N; ++q) { a.qx[q] = op->tab.qx[q]; a.qw[q] = op->tab.qw[q]; }
  a.amp = op->mesh.amp;
  a.cm = op->kind == MF_HELMHOLTZ ? op->mass : 0.0;
  a.comps = geom_comps(op);
  const long long total = op->g.ntiles * (long long)N * N * N * BL;
  const int thr = 256;
  const long long blocks = (total + thr - 1) / thr;
  if (vk == VK_F64) geometry_kernel<double, N><<<(unsigned)blocks, thr, 0, s>>>(static_cast<double*>(geom), a);
  else if (vk == VK_DD) geometry_kernel<dd, N><<<(unsigned)blocks, thr, 0, s>>>(static_cast<dd*>(geom), a);
  else {
    GeomArgsQ q;
    for (int i = 0; i < N; ++i) q.qx[i] = op->tab.qx[i];
    const int nt = (op->g.nx + op->g.ny + op->g.nz) * N;
    geom_table_kernel<N><<<(nt + 127) / 128, 128, 0, s>>>(static_cast<float*>(geom), op->g, q);
  }
  return cuda_check(cudaGetLastError(), "geometry launch");
}

template <int N>
mf_status layout_n(const mf_operator* op, int elem, int mode, const void* in, void* out, cudaStream_t s) {
  const long long total = (mode == LAYOUT_GATHER_UNIQUE) ? op->n_unique : op->g.ntiles * (long long)N * N * N * BL;
  const int thr = 256;
  const long long blocks = (total + thr - 1) / thr;
  if (blocks == 0) return MF_OK;
  if (elem == 8)
    layout_kernel<double, N><<<(unsigned)blocks, thr, 0, s>>>(static_cast<const double*>(in), static_cast<double*>(out), op->g, mode);
  else
    layout_kernel<float, N><<<(unsigned)blocks, thr, 0, s>>>(static_cast<const float*>(in), static_cast<float*>(out), op->g, mode);
  return cuda_check(cudaGetLastError(), "layout launch");
}

} // namespace mf

// Two translation units per degree, compiled in parallel: the single-operator kernels, and
// the batched kernels of the serving loop.
#define MF_INSTANTIATE_DEGREE(NN)                                                                        \
  namespace mf {                                                                                        \
  template mf_status apply_split_n<NN>(const mf_operator*, int, const void*, void*, cudaStream_t);      \
  template int apply_config_n<NN>(const mf_operator*, int);                                              \
  template mf_status apply_block_n<NN>(const mf_operator*, int, int, const void*, void*, cudaStream_t);  \
  template mf_status apply_cg_n<NN>(const mf_operator*, int, void*, const void*, void*, CgState*, double*, \
                                    int, long long*, cudaStream_t);                                     \
  template mf_status dss_n<NN>(const mf_operator*, int, void*, cudaStream_t);                           \
  template mf_status make_consistent_n<NN>(const mf_operator*, int, void*, cudaStream_t);               \
  template mf_status dss_atomic_n<NN>(const mf_operator*, int, void*, void*, cudaStream_t);              \
  template mf_status stream_twin_n<NN>(const mf_operator*, int, const void*, void*, const void*, int,    \
                                       cudaStream_t);                                                   \
  template mf_status diagonal_n<NN>(const mf_operator*, float*, float*, cudaStream_t);                   \
  template mf_status geometry_n<NN>(const mf_operator*, int, void*, cudaStream_t);                      \
  template mf_status layout_n<NN>(const mf_operator*, int, int, const void*, void*, cudaStream_t);      \
  }
#define MF_INSTANTIATE_DEGREE_BATCH(NN)                                                                  \
  namespace mf {                                                                                        \
  template mf_status apply_batch_fill_n<NN>(const BatchMember*, int, int, void*, long long*);            \
  template mf_status apply_batch_launch_n<NN>(const mf_operator*, int, const void*, const long long*, int,  \
                                              long long, cudaStream_t);                                 \
  }
