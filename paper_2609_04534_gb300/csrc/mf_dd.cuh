// mf_dd.cuh -- double-float ("dd") arithmetic: a value is the unevaluated sum hi + lo of two
// floats (about 48 significant bits).  GB300's FP32 pipe issues 64x more FMAs per clock than
// its FP64 pipe, so FP64-accurate sum factorisation runs faster in dd than in native double.
//
// Building blocks are the classical error-free transformations: Knuth's TwoSum
// (s + e = a + b exactly) and the FMA-based TwoProd (p + e = a * b exactly, e = fma(a, b, -p)).
// fma() below accumulates a*b + c without renormalising; finish() renormalises a chain result
// with Dekker's FastTwoSum.  A double is split by integer operations on its bits; a result is joined
// by the otherwise idle FP64 pipe (two conversions and an add per stored value).  The arithmetic
// between them issues no FP64 instruction.
#pragma once
#include <cstring>

#include <cuda_runtime.h>

namespace mf {

// bit casts that also compile for the host (the conversions below are tested on the CPU)
__host__ __device__ __forceinline__ unsigned fbits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  unsigned u;
  std::memcpy(&u, &f, sizeof(u));
  return u;
#endif
}
__host__ __device__ __forceinline__ double dbl_of_bits(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  std::memcpy(&d, &b, sizeof(d));
  return d;
#endif
}

struct __align__(8) dd {
  float hi, lo;
  __host__ __device__ dd() {}
  __host__ __device__ constexpr dd(float h, float l) : hi(h), lo(l) {}
  __host__ __device__ explicit constexpr dd(int v) : hi((float)v), lo(0.0f) {}
};

// Native overloads so that unqualified fma() inside namespace mf also serves double / float.
__device__ __forceinline__ double fma(double a, double b, double c) { return ::fma(a, b, c); }
__device__ __forceinline__ float fma(float a, float b, float c) { return fmaf(a, b, c); }

// a*b + c.  TwoProd of the leading parts, first-order cross terms, TwoSum with c.hi; the
// rounding errors collect in lo (not renormalised: call finish() at the end of a chain).
__device__ __forceinline__ dd fma(dd a, dd b, dd c) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  const float s = c.hi + p;
  const float v = s - c.hi;
  const float t = (c.hi - (s - v)) + (p - v);
  return dd(s, t + (c.lo + e));
}

// The same in 10 instructions instead of 12, for chains of up to three terms: TwoSum's last
// difference p - v and TwoProd's error a.hi b.hi - p are taken together, as a.hi b.hi - v in one
// fma, and the cross terms go straight into lo.  lo is rounded once more per term, so it is used
// only where the rounded conversion of double input outweighs that (ShortProducts, mf_kernels.cuh; split
// apply of doubles, against fma() everywhere: Q4 curved 52^3 0.438 -> 0.409 ms, Q4 Cartesian 52^3 0.189 ->
// 0.177, Q7 Cartesian 33^3 0.294 -> 0.282).
__device__ __forceinline__ dd fma_short(dd a, dd b, dd c) {
  const float p = a.hi * b.hi;
  const float s = __fadd_rn(c.hi, p);
  const float v = s - c.hi;
  const float t = (c.hi - (s - v)) + fmaf(a.hi, b.hi, -v);
  return dd(s, fmaf(a.lo, b.hi, fmaf(a.hi, b.lo, c.lo)) + t);
}
// fma() or, for double-float with SHORT, fma_short()
template <bool SHORT>
__device__ __forceinline__ dd fma_n(dd a, dd b, dd c) { return SHORT ? fma_short(a, b, c) : fma(a, b, c); }
template <bool SHORT, typename A, typename B>
__device__ __forceinline__ B fma_n(A a, B b, B c) { return fma(a, b, c); }

// a*b as the first term of a chain: TwoProd of the leading parts plus the cross terms, not
// renormalised (an fma() into a zero accumulator would spend a TwoSum on the zero).
__device__ __forceinline__ dd mul0(dd a, dd b) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return dd(p, e);
}
__device__ __forceinline__ double mul0(double a, double b) { return a * b; }
__device__ __forceinline__ float mul0(float a, float b) { return a * b; }

__device__ __forceinline__ dd finish(dd a) {
  const float h = a.hi + a.lo;
  return dd(h, a.lo - (h - a.hi));
}
__device__ __forceinline__ double finish(double a) { return a; }
__device__ __forceinline__ float finish(float a) { return a; }

__device__ __forceinline__ dd operator*(dd a, dd b) {
  const float p = a.hi * b.hi;
  float e = fmaf(a.hi, b.hi, -p);
  e = fmaf(a.hi, b.lo, e);
  e = fmaf(a.lo, b.hi, e);
  return finish(dd(p, e));
}

__host__ __device__ __forceinline__ dd operator-(dd a) { return dd(-a.hi, -a.lo); }

__device__ __forceinline__ dd operator+(dd a, dd b) {
  const float s = a.hi + b.hi;
  const float v = s - a.hi;
  const float t = (a.hi - (s - v)) + (b.hi - v);
  return finish(dd(s, t + (a.lo + b.lo)));
}

// double -> dd: hi keeps the leading 24 significant bits (truncated), lo the remaining 29
// bits rounded to 24.  Magnitudes below 2^-126 flush to zero; inf/nan go through hi.  The
// general form; dd_from_double takes the common range without its branches.
__device__ __forceinline__ dd dd_from_double_any(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned hi32 = (unsigned)(b >> 32), lo32 = (unsigned)b;
  const int e = (int)((hi32 >> 20) & 0x7ffu);
  const unsigned sign = hi32 & 0x80000000u;
  const int ef = e - 896; // float biased exponent of the same power of two
  if (e == 0x7ff) return dd(__double2float_rn(x), 0.0f);
  if (ef <= 0) return dd(0.0f, 0.0f);
  if (ef >= 255) return dd(__uint_as_float(sign | 0x7f800000u), 0.0f);
  const unsigned mant = ((hi32 & 0xfffffu) << 3) | (lo32 >> 29);
  const float h = __uint_as_float(sign | ((unsigned)ef << 23) | mant);
  const unsigned r = lo32 & 0x1fffffffu;
  const int es = e - 948; // float biased exponent of 2^(e - 1075)
  // below 2^-74 lo's power of two is no normal float: scaled in two steps (lo itself may be subnormal)
  float l = (es > 0) ? __uint2float_rn(r) * __uint_as_float((unsigned)es << 23)
            : (es > -64) ? __uint2float_rn(r) * 0x1p-64f * __uint_as_float((unsigned)(es + 64) << 23) : 0.0f;
  return dd(h, sign ? -l : l);
}

static __device__ __noinline__ dd dd_from_double_call(double x) { return dd_from_double_any(x); }
// Biased exponents 949..1149 (magnitudes 2^-74..2^127, where hi and lo are normal floats) without
// the branches: hi is the double's leading 24 bits shifted left by 3 with the exponent rebased by
// one exclusive or, lo the remaining bits as an integer times the double's power of two, 2^-52 of
// it.  NEAR: hi is rounded instead of truncated (half its last place added first; the rounding
// may carry, so lo keeps the double's own power), which halves the remainder and its rounding:
// the apply's error against 64 bits falls by 4-7% at n >= 4 (no change below, where it is not used).
// INL: the general form in line or called.
template <bool INL = false, bool NEAR = false>
__device__ __forceinline__ dd dd_from_double(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x), n = NEAR ? b + (1ull << 28) : b;
  const unsigned hi32 = (unsigned)(b >> 32), nh = (unsigned)(n >> 32);
  const unsigned h = ((__funnelshift_l((unsigned)n, nh, 3) ^ 0x40000000u) & 0x7fffffffu) | (nh & 0x80000000u);
  dd r(__uint_as_float(h), 0.0f);
  if (NEAR) {
    const float l = __int2float_rn((int)((unsigned)b << 3) >> 3) *
                    __uint_as_float((((hi32 << 3) ^ 0x40000000u) & 0x7f800000u) - (52u << 23));
    r.lo = __uint_as_float(__float_as_uint(l) ^ (hi32 & 0x80000000u));
  } else {
    r.lo = __uint2float_rn((unsigned)b & 0x1fffffffu) * __uint_as_float((h & 0xff800000u) - (52u << 23));
  }
  if ((hi32 & 0x7fffffffu) - (949u << 20) >= (201u << 20)) r = INL ? dd_from_double_any(x) : dd_from_double_call(x);
  return r;
}

// float -> double by bit manipulation (normal numbers; zero and subnormals give zero).
__host__ __device__ __forceinline__ double f2d_bits(float f) {
  const unsigned u = fbits(f);
  const unsigned ex = (u >> 23) & 0xffu;
  if (ex == 0u) return 0.0;
  if (ex == 0xffu) return (double)f;
  const unsigned long long s = (unsigned long long)(u & 0x80000000u) << 32;
  const unsigned long long de = (unsigned long long)(ex - 127u + 1023u) << 52;
  const unsigned long long m = (unsigned long long)(u & 0x7fffffu) << 29;
  return dbl_of_bits(s | de | m);
}

// dd -> double: exact sum of the two parts (one FP64 add, rounded to nearest).  A subnormal lo
// flushes to zero, as in dd_from_double.  On the device the parts are converted by the FP64
// pipe, which the apply otherwise leaves idle (3 of its slow instructions per stored value take 1.5 clocks
// of an SM, an apply 2.5 or more per value); the same conversion by bits takes about 20
// instructions of the issue-bound kernels (split apply, FP64: Q4 Cartesian 52^3 0.205 -> 0.193 ms, Q2
// 88^3 0.160 -> 0.137, Q2 sheared 88^3 0.329 -> 0.307).
__host__ __device__ __forceinline__ double dd_to_double(dd a) {
#ifdef __CUDA_ARCH__
  double h, l;
  asm("cvt.ftz.f64.f32 %0, %1;" : "=d"(h) : "f"(a.hi));
  asm("cvt.ftz.f64.f32 %0, %1;" : "=d"(l) : "f"(a.lo));
  return h + l;
#else
  return f2d_bits(a.hi) + f2d_bits(a.lo);
#endif
}

// Two FP32 values of neighbouring cells processed by one thread (the FP32 apply): every
// operation acts on both lanes; table coefficients stay scalar floats.  Products and sums that
// are not an fma() are single rounded operations (no contraction), so that kernels of different
// shape give bitwise equal results.
struct __align__(8) f2 {
  float x, y;
  __host__ __device__ f2() {}
  __host__ __device__ constexpr f2(float a, float b) : x(a), y(b) {}
  __host__ __device__ explicit constexpr f2(int v) : x((float)v), y((float)v) {}
};
__device__ __forceinline__ f2 fma(float c, f2 a, f2 b) { return f2(fmaf(c, a.x, b.x), fmaf(c, a.y, b.y)); }
__device__ __forceinline__ f2 fma(f2 c, f2 a, f2 b) { return f2(fmaf(c.x, a.x, b.x), fmaf(c.y, a.y, b.y)); }
__device__ __forceinline__ f2 mul0(float c, f2 a) { return f2(__fmul_rn(c, a.x), __fmul_rn(c, a.y)); }
__device__ __forceinline__ f2 mul0(f2 c, f2 a) { return f2(__fmul_rn(c.x, a.x), __fmul_rn(c.y, a.y)); }
__device__ __forceinline__ f2 finish(f2 a) { return a; }
__device__ __forceinline__ f2 operator*(float c, f2 a) { return mul0(c, a); }
__device__ __forceinline__ f2 operator*(f2 c, f2 a) { return mul0(c, a); }
__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return f2(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y)); }
__device__ __forceinline__ f2 operator-(f2 a) { return f2(-a.x, -a.y); }

// Coefficient type of the 1D tables for a compute type, and cells per compute value.
template <typename T>
struct CoefOf { using type = T; };
template <>
struct CoefOf<f2> { using type = float; };
template <typename T>
struct CellsPer { static constexpr int value = 1; };
template <>
struct CellsPer<f2> { static constexpr int value = 2; };
template <typename T>
struct IsF32 { static constexpr bool value = false; };
template <>
struct IsF32<float> { static constexpr bool value = true; };
template <>
struct IsF32<f2> { static constexpr bool value = true; };

// Compute type of the FP32 view: pairs of cells per thread (MF_FP32_PAIRS=0: one cell).
#ifndef MF_FP32_PAIRS
#define MF_FP32_PAIRS 1
#endif
#if MF_FP32_PAIRS
using FP32C = f2;
#else
using FP32C = float;
#endif

// A double scalar (a CG coefficient) in a vector element type.
template <typename S>
__device__ __forceinline__ S scalar_from_double(double v) { return (S)v; }
template <>
__device__ __forceinline__ dd scalar_from_double<dd>(double v) { return dd_from_double(v); }

// storage <-> compute conversions used by the kernels
template <typename C, typename S>
__device__ __forceinline__ C to_compute(S v) { return (C)v; }
template <>
__device__ __forceinline__ dd to_compute<dd, double>(double v) { return dd_from_double(v); }

template <typename S, typename C>
__device__ __forceinline__ S to_storage(C v) { return (S)v; }
template <>
__device__ __forceinline__ double to_storage<double, dd>(dd v) { return dd_to_double(v); }

// host: double -> compute type
template <typename C>
inline C host_from_double(double v) { return (C)v; }
template <>
inline f2 host_from_double<f2>(double v) { return f2((float)v, (float)v); }
template <>
inline dd host_from_double<dd>(double v) {
  const float h = (float)v;
  return dd(h, (float)(v - (double)h));
}

} // namespace mf
