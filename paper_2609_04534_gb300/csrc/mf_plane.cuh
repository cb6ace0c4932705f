// mf_plane.cuh -- the apply with one thread per plane of a cell.
//
// A thread owns an n x n plane of one value's cell (value: one cell, or a pair for FP32) in every
// stage and runs the two sweeps inside the plane in its registers, so data goes through shared
// memory only where the plane changes direction: 2 (Cartesian) or 4 (general) exchanges and as
// many barriers instead of one per sweep.  n independent pencils per thread give the
// instruction parallelism that the pencil kernels need many resident warps for.  32 values make
// a CTA: a warp is one plane index of 32 consecutive values, so every global access is a whole
// row.  Per pencil the arithmetic (Fold, chains, their order) is that of the pencil kernels, so
// both give bitwise equal results.
//
// What bounds it: instruction fetch.  The plane's sweeps are straight-line code (their arrays are
// registers), a few warps per scheduler run it, and at n = 5 (FP32, curved, 48^3) 0.95 warps are stalled
// on fetch per issued instruction, more than for any other reason; 56% of issue slots are used.
// The pencil loops between shared memory and shared memory are therefore not unrolled (with them
// unrolled Q4 curved FP32 52^3 took 0.099 ms, Q5 44^3 0.161), and double-float, whose code is six times
// longer, uses planes only where n is 2 or 3.
// Measured against the pencil kernels on one GB300 (split apply, ms, pencil -> plane): FP32 Q2 Cartesian
// 88^3 0.041 -> 0.025, Q4 Cartesian 52^3 0.038 -> 0.030 (69% of HBM), Q6 Cartesian 38^3 0.054 -> 0.053,
// Q4 curved 52^3 0.117 -> 0.089 (114 instructions per DoF), Q5 curved 44^3 0.116 -> 0.103, Q4 sheared
// 52^3 0.093 -> 0.072; FP64 (double-float) Q1 Cartesian 120^3 0.114 -> 0.092, Q2 Cartesian 88^3 0.161 ->
// 0.136, Q1 curved 120^3 0.242 -> 0.220, Q2 sheared 88^3 0.370 -> 0.332.
#pragma once

namespace mf {

template <typename T, int N>
struct PlaneCfg {
  static constexpr int CPL = CellsPer<T>::value, CB = 32, NT = N * CB, VPT = BL / CPL; // values per tile
  static long long blocks(long long ntiles) { return (ntiles * VPT + CB - 1) / CB; }
  static constexpr int TPC = CB / VPT; // tiles per CTA
  // resident CTAs the registers are capped for: general, Cartesian
  static constexpr int MINB_G = N == 2 ? 16 : (N == 3 ? 7 : (N == 4 ? 4 : 2));
  static constexpr int MINB_C = N == 2 ? 20 : (N == 3 ? 10 : (N == 4 ? 6 : (N == 5 ? 4 : (N == 6 ? 3 : 2))));
};

// Where the plane kernels are launch variant 0 (else a pencil kernel is): FP32 pairs while the
// plane's arrays fit the registers (n^2 values of 8 bytes, twice on the general path; Cartesian
// n = 8 lost, 0.084 -> 0.116 ms), double-float for n = 2 and on the Cartesian and affine paths
// n = 3 (curved n = 3: 0.50 against 0.41 ms of the pencil kernel).
template <typename T, int N, int PATH>
struct UsePlane {
  static constexpr bool value = CellsPer<T>::value == 2 ? N <= (PATH == PATH_CARTESIAN ? 7 : 6)
                                                        : std::is_same<T, dd>::value &&
                                                              N <= (PATH == PATH_CURVED ? 2 : 3);
};

// The cells of one value: its tile, first lane, coordinates, and which exist.
struct PlaneCell {
  long long t;
  int lane, cx, cy, cz;
  bool v0, v1; // first cell, second cell of a pair
};
template <typename T>
__device__ __forceinline__ PlaneCell plane_cell(const GridInfo& g, long long value) {
  constexpr int CPL = CellsPer<T>::value, VPT = BL / CPL;
  PlaneCell q;
  q.t = value / VPT;
  q.lane = (int)(value - q.t * VPT) * CPL;
  cell_of(g, q.t, q.lane, q.cx, q.cy, q.cz);
  const bool yz = q.t < g.ntiles && q.cy < g.ny && q.cz < g.nz;
  q.v0 = yz && q.cx < g.nx;
  q.v1 = CPL == 2 && yz && q.cx + 1 < g.nx;
  return q;
}
// Constrained nodes of the plane k: the whole plane, or by i / j.
template <int N>
struct PlaneMask {
  bool on, all, x0, x1, y0, y1;
  __device__ __forceinline__ PlaneMask(const GridInfo& g, int cx, int cy, int cz, int k) {
    on = g.bc != 0;
    all = (cz == 0 && k == 0) || (cz == g.nz - 1 && k == N - 1);
    x0 = cx == 0;
    x1 = cx == g.nx - 1;
    y0 = cy == 0;
    y1 = cy == g.ny - 1;
  }
  __device__ __forceinline__ bool operator()(int i, int j) const {
    return all || (i == 0 && x0) || (i == N - 1 && x1) || (j == 0 && y0) || (j == N - 1 && y1);
  }
};

// The plane k of a value into u[j][i]: load_tile's values (padding cells and constrained nodes
// zero; in a CG step with update_p the new direction p = r + beta p, written back).
template <bool INL, typename S, typename T, int N>
__device__ __forceinline__ void load_plane(const ApplyJob<S, T>& a, const PlaneCell& q, int k, T (&u)[N][N]) {
  constexpr int N2 = N * N, N3 = N2 * N, CPL = CellsPer<T>::value;
  const bool fuse = a.cg.st != nullptr && a.cg.update_p;
  const S beta = fuse ? scalar_from_double<S>(a.cg.st->beta) : S(0);
  const long long base = (q.t * N3 + (long long)N2 * k) * BL + q.lane;
  const bool in = q.t < a.g.ntiles;
  if constexpr (CPL == 1) {
    const PlaneMask<N> m(a.g, q.cx, q.cy, q.cz, k);
    S x[N][N];
    if (fuse) {
      S* pg = a.cg.p + base;
      const S* rg = a.cg.r + base;
      S r[N][N]; // every load before the first store (see LoadLine)
#pragma unroll
      for (int j = 0; j < N; ++j)
#pragma unroll
        for (int i = 0; i < N; ++i) {
          x[j][i] = r[j][i] = S(0);
          if (q.v0) {
            x[j][i] = pg[(i + N * j) * BL];
            r[j][i] = rg[(i + N * j) * BL];
          }
        }
#pragma unroll
      for (int j = 0; j < N; ++j)
#pragma unroll
        for (int i = 0; i < N; ++i) {
          x[j][i] = q.v0 ? finish(fma(beta, x[j][i], r[j][i])) : S(0);
          if (in) pg[(i + N * j) * BL] = x[j][i];
        }
    } else {
      const S* xg = a.x + base;
#pragma unroll
      for (int j = 0; j < N; ++j)
#pragma unroll
        for (int i = 0; i < N; ++i) {
          x[j][i] = S(0);
          if (q.v0) x[j][i] = xg[(i + N * j) * BL];
        }
    }
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int i = 0; i < N; ++i) u[j][i] = load_value<INL, (N >= 4), T, S>(x[j][i]);
    if (m.on) {
#pragma unroll
      for (int j = 0; j < N; ++j)
#pragma unroll
        for (int i = 0; i < N; ++i)
          if (m(i, j)) u[j][i] = T(0);
    }
  } else {
    const PlaneMask<N> m0(a.g, q.cx, q.cy, q.cz, k), m1(a.g, q.cx + 1, q.cy, q.cz, k);
    float2 x[N][N];
    if (fuse) { // row by row, a row's loads before the stores of the row before it (see LoadLine)
      S* pg = a.cg.p + base;
      const S* rg = a.cg.r + base;
      float2 r[2][N];
      auto load_row = [&](int j) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
          x[j][i] = r[j & 1][i] = make_float2(0.f, 0.f);
          if (in) {
            x[j][i] = *reinterpret_cast<const float2*>(pg + (i + N * j) * BL);
            r[j & 1][i] = *reinterpret_cast<const float2*>(rg + (i + N * j) * BL);
          }
        }
      };
      load_row(0);
#pragma unroll
      for (int j = 0; j < N; ++j) {
        if (j + 1 < N) load_row(j + 1);
#pragma unroll
        for (int i = 0; i < N; ++i) {
          x[j][i].x = q.v0 ? fmaf(beta, x[j][i].x, r[j & 1][i].x) : 0.0f;
          x[j][i].y = q.v1 ? fmaf(beta, x[j][i].y, r[j & 1][i].y) : 0.0f;
          if (in) *reinterpret_cast<float2*>(pg + (i + N * j) * BL) = x[j][i];
        }
      }
    } else {
      const S* xg = a.x + base;
#pragma unroll
      for (int j = 0; j < N; ++j)
#pragma unroll
        for (int i = 0; i < N; ++i) {
          x[j][i] = make_float2(0.f, 0.f);
          if (in) x[j][i] = *reinterpret_cast<const float2*>(xg + (i + N * j) * BL);
        }
    }
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int i = 0; i < N; ++i) u[j][i] = T(q.v0 ? x[j][i].x : 0.0f, q.v1 ? x[j][i].y : 0.0f);
    if (m0.on) {
#pragma unroll
      for (int j = 0; j < N; ++j)
#pragma unroll
        for (int i = 0; i < N; ++i) {
          if (m0(i, j)) u[j][i].x = 0.0f;
          if (m1(i, j)) u[j][i].y = 0.0f;
        }
    }
  }
}

// The plane k of a value to y (store_xpencil's values); PAIR: the sum of p y over the plane's
// real copies for a CG step, p re-read from where load_plane found (or wrote) it.
template <bool PAIR, typename S, typename T, int N>
__device__ __forceinline__ double store_plane(const ApplyJob<S, T>& a, const PlaneCell& q, int k, T (&u)[N][N]) {
  constexpr int N2 = N * N, N3 = N2 * N, CPL = CellsPer<T>::value;
  if (q.t >= a.g.ntiles) return 0.0;
  const long long base = (q.t * N3 + (long long)N2 * k) * BL + q.lane;
  S* yg = a.y + base;
  typename AccOf<S>::type acc;
  const bool pair = PAIR && a.cg.st != nullptr;
  const S* pg = pair ? (a.cg.update_p ? a.cg.p : a.x) + base : nullptr;
  if constexpr (CPL == 1) {
    const PlaneMask<N> m(a.g, q.cx, q.cy, q.cz, k);
    auto value = [&](int j, int i) {
      const S v = q.v0 ? to_storage<S, T>(u[j][i]) : S(0);
      return m.on && m(i, j) ? S(0) : v;
    };
    if (pair && q.v0) { // its loads before the first store (see LoadLine)
#pragma unroll
      for (int j = 0; j < N; ++j)
#pragma unroll
        for (int i = 0; i < N; ++i) acc.add(pg[(i + N * j) * BL], value(j, i));
    }
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int i = 0; i < N; ++i) yg[(i + N * j) * BL] = value(j, i);
  } else {
    const PlaneMask<N> m0(a.g, q.cx, q.cy, q.cz, k), m1(a.g, q.cx + 1, q.cy, q.cz, k);
    auto value = [&](int j, int i) {
      float2 v = make_float2(q.v0 ? u[j][i].x : 0.0f, q.v1 ? u[j][i].y : 0.0f);
      if (m0.on) {
        if (m0(i, j)) v.x = 0.0f;
        if (m1(i, j)) v.y = 0.0f;
      }
      return v;
    };
    if (pair) {
#pragma unroll
      for (int j = 0; j < N; ++j)
#pragma unroll
        for (int i = 0; i < N; ++i) {
          const float2 pv = *reinterpret_cast<const float2*>(pg + (i + N * j) * BL), v = value(j, i);
          if (q.v0) acc.add(pv.x, v.x);
          if (q.v1) acc.add(pv.y, v.y);
        }
    }
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int i = 0; i < N; ++i) *reinterpret_cast<float2*>(yg + (i + N * j) * BL) = value(j, i);
  }
  return pair ? acc.value() : 0.0;
}

// prefetch_next_wave for the tiles of this CTA
template <typename S, typename T, int N, int NC>
__device__ __forceinline__ void plane_prefetch(const ApplyJob<S, T>& a, long long cta) {
  constexpr int TPC = PlaneCfg<T, N>::TPC;
#pragma unroll
  for (int i = 0; i < TPC; ++i) prefetch_next_wave<S, T, N, NC>(a, cta * TPC + i, 0);
}

// A matrix applied to every row (x) or column (y) of a plane, in place.
template <bool ANTI, bool SHORT, typename C, typename T, int N>
__device__ __forceinline__ void plane_x(const EoTab<C, N>& m, T (&u)[N][N]) {
#pragma unroll
  for (int j = 0; j < N; ++j) {
    T out[N];
    Fold<T, N, ANTI, SHORT>(u[j]).apply(m, out);
#pragma unroll
    for (int i = 0; i < N; ++i) u[j][i] = out[i];
  }
}
template <bool ANTI, bool SHORT, typename C, typename T, int N>
__device__ __forceinline__ void plane_y(const EoTab<C, N>& m, T (&u)[N][N]) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    T in[N], out[N];
#pragma unroll
    for (int j = 0; j < N; ++j) in[j] = u[j][i];
    Fold<T, N, ANTI, SHORT>(in).apply(m, out);
#pragma unroll
    for (int j = 0; j < N; ++j) u[j][i] = out[j];
  }
}

// A thread's part of <p, A p> over its plane: every row of n points is summed like a pencil of
// general_body, and the rows are joined in double-float (FP32) or double.  (A plain FP32 sum over n^2
// points lost 1e-6 of a sum of one large and many small terms.)
template <typename T>
struct RowSum {
  double s = 0.0;
  __device__ __forceinline__ void add(T row) { s += to_double(finish(row)); }
  __device__ __forceinline__ double value() const { return s; }
};
template <>
struct RowSum<float> {
  AccF acc;
  __device__ __forceinline__ void add(float row) { acc.add2(row, 0.0f); }
  __device__ __forceinline__ double value() const { return acc.value(); }
};
template <>
struct RowSum<f2> {
  AccF acc;
  __device__ __forceinline__ void add(f2 row) {
    acc.add2(row.x, 0.0f);
    acc.add2(row.y, 0.0f);
  }
  __device__ __forceinline__ double value() const { return acc.value(); }
};

// General cells (see general_body).  Stages: plane k = p: load, S along x and y | plane j = p:
// S along z and the z-derivative | plane q = p: x- and y-derivatives, metric, Dc^T along x and
// y | plane j = p: Dc^T along z, S^T along z | plane k = p: S^T along y and x, store.
template <typename S, typename T, int N, bool CURVED, bool HELM>
__device__ __forceinline__ void general_plane(const ApplyJob<S, T>& a, const Tab<typename CoefOf<T>::type, N>& tab,
                                              long long cta) {
  constexpr int N2 = N * N, N3 = N2 * N, CB = PlaneCfg<T, N>::CB, NT = N * CB, CPL = CellsPer<T>::value;
  constexpr int NC = HELM ? 7 : 6;
  constexpr bool SH = ShortProducts<S, T, N>::all;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* A = reinterpret_cast<T*>(smem_raw);
  T* B = A + N3 * CB;
  if (a.cg.st != nullptr && a.cg.st->flag != 0) return; // CG step after convergence: no work
  plane_prefetch<S, T, N, (CURVED && !IsF32<T>::value) ? NC : 0>(a, cta);
  const int c = threadIdx.x % CB, p = threadIdx.x / CB;
  const PlaneCell cell = plane_cell<T>(a.g, cta * CB + c);
  A += c;
  B += c;
  {
    T u[N][N];
    load_plane<false, S, T, N>(a, cell, p, u);
    plane_x<false, SH>(tab.eS, u);
    plane_y<false, SH>(tab.eS, u);
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int i = 0; i < N; ++i) A[(i + N * j + N2 * p) * CB] = u[j][i];
  }
  __syncthreads();
#pragma unroll (N == 2 ? 2 : 1)
  for (int i = 0; i < N; ++i) { // pencils (i, j = p): values to A, z-derivatives to B (own slots)
    T in[N], U[N], d3[N];
#pragma unroll
    for (int k = 0; k < N; ++k) in[k] = A[(i + N * p + N2 * k) * CB];
    Fold<T, N, false, SH>(in).apply(tab.eS, U);
    Fold<T, N, true, SH>(U).apply(tab.eD, d3);
#pragma unroll
    for (int q = 0; q < N; ++q) {
      A[(i + N * p + N2 * q) * CB] = U[q];
      B[(i + N * p + N2 * q) * CB] = d3[q];
    }
  }
  __syncthreads();
  const bool fuse = a.cg.st != nullptr;
  RowSum<T> pap;
  { // plane q = p: u holds U, then Dc^T_x v1 (+ m U), row by row; d2 the y-derivatives, then v2
    T u[N][N], d2[N][N];
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int i = 0; i < N; ++i) u[j][i] = d2[j][i] = A[(i + N * j + N2 * p) * CB];
    plane_y<true, SH>(tab.eD, d2);
    float sx[N][2], px[N][2], sz = 0.f, pz = 0.f;
    const float* ty = nullptr;
    if constexpr (CURVED && IsF32<T>::value) { // sin and pi cos of pi xh, see general_body
      const int cy = min(cell.cy, a.g.ny - 1), cz = min(cell.cz, a.g.nz - 1);
#pragma unroll
      for (int m = 0; m < CPL; ++m) {
        const float* tx = a.gtab + 2 * (min(cell.cx + m, a.g.nx - 1) * N);
#pragma unroll
        for (int i = 0; i < N; ++i) {
          sx[i][m] = tx[2 * i];
          px[i][m] = tx[2 * i + 1];
        }
      }
      ty = a.gtab + 2 * ((a.g.nx + cy) * N);
      const float* tz = a.gtab + 2 * ((a.g.nx + a.g.ny + cz) * N + p);
      sz = tz[0];
      pz = tz[1];
    }
    const T* gp = nullptr;
    if constexpr (CURVED && !IsF32<T>::value)
      gp = a.geom + ((cell.t * NC) * (long long)N3 + (long long)N2 * p) * BL + cell.lane;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      T d1[N], mu[N], row = T(0);
      Fold<T, N, true, SH>(u[j]).apply(tab.eD, d1);
      float syz = 0.f, pyz = 0.f, spz = 0.f;
      if constexpr (CURVED && IsF32<T>::value) {
        syz = __fmul_rn(ty[2 * j], sz);
        pyz = __fmul_rn(ty[2 * j + 1], sz);
        spz = __fmul_rn(ty[2 * j], pz);
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const int l = i + N * j + N2 * p;
        const T e1 = d1[i], e2 = d2[j][i], e3 = B[l * CB];
        T v1, v2, v3, m = T(0);
        if constexpr (CURVED && IsF32<T>::value) {
          curved_flux<N>(sx[i], px[i], syz, pyz, spz, tab.W[i] * tab.W[j] * tab.W[p], a, e1, e2, e3, v1, v2, v3, m);
        } else {
          T g0, g1, g2, g3, g4, g5;
          if (CURVED) {
            const T* gq = gp + (i + N * j) * BL;
            g0 = gq[0];
            g1 = gq[1 * N3 * BL];
            g2 = gq[2 * N3 * BL];
            g3 = gq[3 * N3 * BL];
            g4 = gq[4 * N3 * BL];
            g5 = gq[5 * N3 * BL];
            if (HELM) m = gq[6 * N3 * BL];
          } else {
            const auto w = tab.W[i] * tab.W[j] * tab.W[p];
            g0 = w * a.G[0]; g1 = w * a.G[1]; g2 = w * a.G[2];
            g3 = w * a.G[3]; g4 = w * a.G[4]; g5 = w * a.G[5];
            if (HELM) m = w * a.mdet;
          }
          v1 = finish(fma_n<SH>(g0, e1, fma_n<SH>(g1, e2, mul0(g2, e3))));
          v2 = finish(fma_n<SH>(g1, e1, fma_n<SH>(g3, e2, mul0(g4, e3))));
          v3 = finish(fma_n<SH>(g2, e1, fma_n<SH>(g4, e2, mul0(g5, e3))));
        }
        d1[i] = v1;
        d2[j][i] = v2;
        B[l * CB] = v3;
        if (fuse) row = fma(e1, v1, fma(e2, v2, fma(e3, v3, row)));
        if (HELM) {
          mu[i] = m * u[j][i];
          if (fuse) row = fma(u[j][i], mu[i], row);
        }
      }
      if (fuse) pap.add(row);
      T out[N];
      Fold<T, N, true, SH>(d1).apply(tab.eDt, out);
#pragma unroll
      for (int i = 0; i < N; ++i) u[j][i] = HELM ? add_lazy(out[i], mu[i]) : out[i];
    }
    plane_y<true, SH>(tab.eDt, d2);
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int i = 0; i < N; ++i) A[(i + N * j + N2 * p) * CB] = add_lazy(u[j][i], d2[j][i]);
  }
  __syncthreads();
#pragma unroll (N == 2 ? 2 : 1)
  for (int i = 0; i < N; ++i) { // pencils (i, j = p)
    T v3[N], s[N], tq[N], out[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      v3[q] = B[(i + N * p + N2 * q) * CB];
      s[q] = A[(i + N * p + N2 * q) * CB];
    }
    Fold<T, N, true, SH>(v3).add_to(s, tab.eDt, tq);
    Fold<T, N, false, SH>(tq).apply(tab.eSt, out);
#pragma unroll
    for (int k = 0; k < N; ++k) A[(i + N * p + N2 * k) * CB] = out[k];
  }
  __syncthreads();
  {
    T u[N][N];
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int i = 0; i < N; ++i) u[j][i] = A[(i + N * j + N2 * p) * CB];
    plane_y<false, SH>(tab.eSt, u);
    plane_x<false, SH>(tab.eSt, u);
    store_plane<false, S, T, N>(a, cell, p, u);
  }
  if (fuse) {
    __shared__ double red[NT];
    red[threadIdx.x] = pap.value();
    __syncthreads();
    cta_partial_after_barrier<NT>(red, a.cg.partials, cta);
  }
}

// Cartesian cells in fast-diagonalised form (see cartesian_fd_body).  Stages: plane k = p:
// load, W^T along x and y | plane j = p: W^T along z, scale, W along z | plane k = p: W along y
// and x, store.
template <typename S, typename T, int N, bool HELM>
__device__ __forceinline__ void cartesian_plane(const ApplyJob<S, T>& a, const Tab<typename CoefOf<T>::type, N>& tab,
                                                long long cta) {
  using C = typename CoefOf<T>::type;
  constexpr int N2 = N * N, CB = PlaneCfg<T, N>::CB, NT = N * CB;
  constexpr bool SH = ShortProducts<S, T, N>::all, SHF = ShortProducts<S, T, N>::forward;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* A = reinterpret_cast<T*>(smem_raw);
  if (a.cg.st != nullptr && a.cg.st->flag != 0) return; // CG step after convergence: no work
  plane_prefetch<S, T, N, 0>(a, cta);
  const int c = threadIdx.x % CB, p = threadIdx.x / CB;
  const PlaneCell cell = plane_cell<T>(a.g, cta * CB + c);
  const FdTab<C, N>& fd = tab.fd;
  A += c;
  {
    T u[N][N];
    load_plane<InlineFrom<N>::cartesian, S, T, N>(a, cell, p, u);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      T out[N];
      fd_forward<SHF, C, T, N>(fd, u[j], out);
#pragma unroll
      for (int i = 0; i < N; ++i) u[j][i] = out[i];
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
      T in[N], out[N];
#pragma unroll
      for (int j = 0; j < N; ++j) in[j] = u[j][i];
      fd_forward<SHF, C, T, N>(fd, in, out);
#pragma unroll
      for (int j = 0; j < N; ++j) A[(i + N * j + N2 * p) * CB] = out[j];
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < N; ++i) { // pencils (i, j = p), own slots
    T in[N], z[N], out[N];
#pragma unroll
    for (int k = 0; k < N; ++k) in[k] = A[(i + N * p + N2 * k) * CB];
    fd_forward<SHF, C, T, N>(fd, in, z);
    T dxy = fma(fd.lam[p], a.gy, mul0(fd.lam[i], a.gx));
    if (HELM) dxy = add_lazy(dxy, a.cmass);
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const T dk = finish(fma(fd.lam[k], a.gz, dxy));
      z[k] = finish(mul0(dk, z[k]));
    }
    fd_backward<SH, C, T, N>(fd, z, out);
#pragma unroll
    for (int k = 0; k < N; ++k) A[(i + N * p + N2 * k) * CB] = out[k];
  }
  __syncthreads();
  double pap = 0.0;
  {
    T u[N][N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      T z[N], out[N];
#pragma unroll
      for (int j = 0; j < N; ++j) z[j] = A[(i + N * j + N2 * p) * CB];
      fd_backward<SH, C, T, N>(fd, z, out);
#pragma unroll
      for (int j = 0; j < N; ++j) u[j][i] = out[j];
    }
#pragma unroll
    for (int j = 0; j < N; ++j) {
      T out[N];
      fd_backward<SH, C, T, N>(fd, u[j], out);
#pragma unroll
      for (int i = 0; i < N; ++i) u[j][i] = out[i];
    }
    pap = store_plane<true, S, T, N>(a, cell, p, u);
  }
  if (a.cg.st != nullptr) {
    __shared__ double red[NT];
    red[threadIdx.x] = pap;
    __syncthreads();
    cta_partial_after_barrier<NT>(red, a.cg.partials, cta);
  }
}

} // namespace mf
