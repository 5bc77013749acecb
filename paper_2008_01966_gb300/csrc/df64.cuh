// Pair-of-FP32 ("double-float") arithmetic for the residual operator of the
// mixed-precision solve.
//
// A value is hi + lo with hi = fl32(hi + lo); sums and products are formed
// with the error-free transformations of Knuth (two-sum: s = a + b exactly as
// s + e) and of the fused multiply-add (two-product: a b = p + fma(a, b, -p)),
// then renormalised (Dekker's fast two-sum).  The addition is the short form
// (hi parts by two-sum, lo parts added once), with a relative error of a few
// units of 2^-44 away from cancellation; products are within ~2^-45.  That is
// ~1e-12 relative for a whole transform pass, against ~1e-7 in FP32, at FP32
// instruction rates, which on this GPU are 64x the FP64 rate.
//
// Every step uses the _rn intrinsics, which the compiler never contracts into
// fused multiply-adds or reassociates, so the transformations stay exact.
#pragma once
#include "fft.cuh"

struct __align__(8) df {
  float hi, lo;
  df() = default;
  __host__ __device__ constexpr df(float h, float l) : hi(h), lo(l) {}
  __host__ __device__ constexpr df(int v) : hi((float)v), lo(0.0f) {}
  __host__ __device__ constexpr df(float v) : hi(v), lo(0.0f) {}
  __host__ __device__ constexpr df(double v)
      : hi((float)v), lo((float)(v - (double)(float)v)) {}
  __host__ __device__ explicit operator double() const { return (double)hi + (double)lo; }
};

// 16-byte aligned so that a complex value moves as one vector access
struct __align__(16) cdf {
  df x, y;
};
template <> struct cplx_t<df> { typedef cdf type; };
// Four points a thread, radix 4 (fft.cuh): 64 registers, so 32 warps per SM, where
// radix 8 takes 128 and 16 warps left the kernels waiting (issue slots 40-55 %
// busy).  A line has 256 threads at most, so that two CTAs share an SM; at 4096
// points, where shared memory holds one CTA, 512.  Operator on a GB300, with
// radix 8 and spills of 0.3-2 KB a thread, and now (128 threads a line of 1024
// points and 256 of 2048 then): 256 x 256, 6 vectors 2.35 -> 1.74 ms; 512 x 512,
// 8 vectors 10.0 -> 8.6 ms (10.4 with 512 threads a line and one CTA per SM);
// 1024 x 1024, 3 vectors 25.7 -> 14.8 ms; 32 x 32, one vector 96 -> 75 us.
template <> struct FftE<df> {
  static constexpr int E = 4, LRMAX = 2, THREADS = 512;
  __host__ __device__ static constexpr int max_tpl(int n) { return n < 4096 ? 256 : 512; }
};

__device__ __forceinline__ df df_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return df(s, e);
}
__device__ __forceinline__ df df_fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return df(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ df operator+(df a, df b) {
  const df s = df_two_sum(a.hi, b.hi);
  return df_fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ df operator-(df a) { return df(-a.hi, -a.lo); }
__device__ __forceinline__ df operator-(df a, df b) { return a + (-b); }
__device__ __forceinline__ df operator*(df a, df b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return df_fast_two_sum(p, e);
}
// quotient by one correction step of the FP32 quotient of the hi parts
__device__ __forceinline__ df operator/(df a, df b) {
  const float q1 = __fdiv_rn(a.hi, b.hi);
  const df r = a - b * df(q1);
  const float q2 = __fdiv_rn(r.hi, b.hi);
  return df_fast_two_sum(q1, q2);
}
__device__ __forceinline__ df& operator+=(df& a, df b) { return a = a + b; }
__device__ __forceinline__ df& operator-=(df& a, df b) { return a = a - b; }
__device__ __forceinline__ df& operator*=(df& a, df b) { return a = a * b; }

__device__ __forceinline__ cdf to_cdf(double2 v) { return cdf{df(v.x), df(v.y)}; }
__device__ __forceinline__ double2 to_d2(cdf v) { return make_double2((double)v.x, (double)v.y); }
