// Double-float arithmetic: a value held as an unevaluated sum of two FP32
// terms, x = hi + lo with |lo| <= ulp(hi) / 2 (about 48 significant bits).
//
// GB300 issues FP64 arithmetic (and FP64 conversions) at 1/64 of its FP32
// rate, so on the element-wise paths of the refined form every FP64
// operation per vector entry costs about as much as a gather. The refined
// form therefore keeps its FP64-accurate quantities (the outer iterate, the
// refinement residual, the outer Lanczos basis) as two FP32 terms and works
// on them with FP32 instructions only, through the error-free transforms
// below:
//   two_sum  (Knuth):   s + e == a + b exactly, any a, b
//   quick_two_sum (Dekker): the same when |a| >= |b| (or a == 0)
//   two_prod (FMA):     p + e == a * b exactly
// The compound operations (add, mul) are the usual "sloppy" double-float
// forms: their error is about 2^-46 of the operands' magnitudes, which is
// what an absolute residual or a normalised Lanczos vector needs.
#pragma once
#include <cuda_runtime.h>

namespace wl {

struct df {
  float hi, lo;
};

__device__ __forceinline__ df two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return df{s, e};
}

__device__ __forceinline__ df quick_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return df{s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ df two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return df{p, __fmaf_rn(a, b, -p)};
}

__device__ __forceinline__ df df_norm(float s, float e) { return quick_two_sum(s, e); }

__device__ __forceinline__ df df_add(df a, df b) {
  df s = two_sum(a.hi, b.hi);
  const float e = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
  return two_sum(s.hi, e);
}

__device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, df{-b.hi, -b.lo}); }

__device__ __forceinline__ df df_add_f(df a, float b) {
  df s = two_sum(a.hi, b);
  return two_sum(s.hi, __fadd_rn(s.lo, a.lo));
}

__device__ __forceinline__ df df_mul(df a, df b) {
  df p = two_prod(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.lo, p.lo);
  e = __fmaf_rn(a.lo, b.hi, e);
  return quick_two_sum(p.hi, e);
}

__device__ __forceinline__ df df_mul_f(df a, float b) {
  df p = two_prod(a.hi, b);
  return quick_two_sum(p.hi, __fmaf_rn(a.lo, b, p.lo));
}

// running sum (s, c) += a with the rounding error of every add kept in c
__device__ __forceinline__ void df_acc(float& s, float& c, float a) {
  const df t = two_sum(s, a);
  s = t.hi;
  c = __fadd_rn(c, t.lo);
}

// running sum (s, c) += a (double-float)
__device__ __forceinline__ void df_acc2(float& s, float& c, df a) {
  const df t = two_sum(s, a.hi);
  s = t.hi;
  c = __fadd_rn(c, __fadd_rn(t.lo, a.lo));
}

// host/device split of an FP64 constant
__host__ __device__ inline df df_from_double(double x) {
  const float h = (float)x;
  return df{h, (float)(x - (double)h)};
}

__device__ __forceinline__ double df_to_double(df a) { return (double)a.hi + (double)a.lo; }

// The same conversions for whole vectors, by integer instructions: a conversion
// between FP32 and FP64 goes through the FP64 pipe (2 lanes per clock and SM), so
// that passes that split or join vectors were bound by it and not by memory. Bit
// for bit the results of the above. 131072 x 64 doubles split, with column norms:
// 102 -> 39 us; joined: 51 -> 31 us; the batch's residual of 24 graphs x 5 x 32
// columns: 267 -> 207 us.
// 2^-63 <= |x| < 2^127; other values take the conversions
__device__ __forceinline__ df split_f64(double x) {
  const int uh = __double2hiint(x), ul = __double2loint(x);
  const int e = (uh >> 20) & 0x7ff;
  if (e < 960 || e >= 1023 + 127) {
    if (((uh & 0x7fffffff) | ul) == 0) return df{__int_as_float(uh), 0.f};
    return df_from_double(x);
  }
  // leading 24 bits rounded to nearest even, the other 29 less the carry as an integer
  const unsigned top = ((unsigned)uh << 3) | ((unsigned)ul >> 29);  // its low 23 bits: the fraction
  const int rem = ul & 0x1fffffff;
  const int up = rem > 0x10000000 || (rem == 0x10000000 && (top & 1u));
  const int hb = (uh & 0x80000000) | (int)((((unsigned)(e - 896) << 23) | (top & 0x7fffffu)) + (unsigned)up);
  const int r = rem - (up << 29);
  const float lo = (float)(uh < 0 ? -r : r) * __int_as_float((e - 948) << 23);
  return df{__int_as_float(hb), lo};
}
// an FP32 value as a double: normal values and zero by bits
__device__ __forceinline__ double widen_f32(float x) {
  const int b = __float_as_int(x), e = (b >> 23) & 0xff;
  if (e == 0 || e == 0xff) {
    if ((b & 0x7fffffff) == 0) return __hiloint2double(b, 0);
    return (double)x;
  }
  return __hiloint2double((b & 0x80000000) | (((b & 0x7fffffff) >> 3) + (896 << 20)), b << 29);
}
__device__ __forceinline__ double join_f64(float hi, float lo) { return widen_f32(hi) + widen_f32(lo); }

// sum type of the reductions: double-float for FP32 (error-free adds with
// FP32 instructions; FP64 adds run at 1/64 of their rate), FP64 for FP64
template <typename T>
struct CoopSum;
template <>
struct CoopSum<float> {
  using S = float2;
  static __device__ __forceinline__ S from(float v) { return make_float2(v, 0.f); }
  static __device__ __forceinline__ S add(S a, S b) {
    const df t = df_add(df{a.x, a.y}, df{b.x, b.y});
    return make_float2(t.hi, t.lo);
  }
  static __device__ __forceinline__ S shfl(S a, int off) {
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, off), __shfl_xor_sync(0xffffffffu, a.y, off));
  }
  static __device__ __forceinline__ S zero() { return make_float2(0.f, 0.f); }
  static __device__ __forceinline__ double out(S a) { return (double)a.x + (double)a.y; }
  static __device__ __forceinline__ S in(double v) {
    const df t = df_from_double(v);
    return make_float2(t.hi, t.lo);
  }
  static __device__ __forceinline__ float lead(S a) { return a.x; }
  // a / b to FP32: the leading quotient and one correction (an FP64 division waits a microsecond here)
  static __device__ __forceinline__ float quot(S a, S b) {
    const float q = a.x / b.x;
    const df r = df_sub(df{a.x, a.y}, df_mul_f(df{b.x, b.y}, q));
    return q + r.hi / b.x;
  }
  static __device__ __forceinline__ bool le(S a, S b) { return a.x < b.x || (a.x == b.x && a.y <= b.y); }
};
template <>
struct CoopSum<double> {
  using S = double;
  static __device__ __forceinline__ S from(double v) { return v; }
  static __device__ __forceinline__ S add(S a, S b) { return a + b; }
  static __device__ __forceinline__ S shfl(S a, int off) { return __shfl_xor_sync(0xffffffffu, a, off); }
  static __device__ __forceinline__ S zero() { return 0.0; }
  static __device__ __forceinline__ double out(S a) { return a; }
  static __device__ __forceinline__ S in(double v) { return v; }
  static __device__ __forceinline__ double lead(S a) { return a; }
  static __device__ __forceinline__ double quot(S a, S b) { return a / b; }
  static __device__ __forceinline__ bool le(S a, S b) { return a <= b; }
};

}  // namespace wl
