// Double-float ("df64") arithmetic on the FP32 pipe: a value is the unevaluated
// sum hi + lo of two floats with |lo| <= ulp(hi)/2, about 48 significant
// bits.  Built from error-free transformations: Knuth's TwoSum (The Art of
// Computer Programming vol. 2, 4.2.2), Dekker's FastTwoSum and the FMA form
// of Dekker's TwoProd (Dekker, "A floating-point technique for extending the
// available precision", 1971).  GB300 runs FP64 at 1/58 of the FP32 rate, so
// an FP64-accurate operation costs less as a handful of FP32 operations.
#pragma once

#include <cuda_runtime.h>

namespace mgar {

struct df {
  float hi, lo;
};

// s + e == a + b exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bv = __fsub_rn(s, a);
  const float av = __fsub_rn(s, bv);
  e = __fadd_rn(__fsub_rn(a, av), __fsub_rn(b, bv));
}

// s + e == a + b exactly, given |a| >= |b| (or a == 0)
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}

// p + e == a * b exactly
__device__ __forceinline__ void two_prod(float a, float b, float& p, float& e) {
  p = __fmul_rn(a, b);
  e = __fmaf_rn(a, b, -p);
}

__device__ __forceinline__ df df_make(float h, float l) {
  df r;
  fast_two_sum(h, l, r.hi, r.lo);
  return r;
}

// a + b (sloppy form: error ~2^-46 of max(|a|, |b|))
__device__ __forceinline__ df df_add(df a, df b) {
  float s, e;
  two_sum(a.hi, b.hi, s, e);
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return df_make(s, e);
}

__device__ __forceinline__ df df_neg(df a) { return df{-a.hi, -a.lo}; }

__device__ __forceinline__ df df_sub(df a, df b) { return df_add(a, df_neg(b)); }

// a * b
__device__ __forceinline__ df df_mul(df a, df b) {
  float p, e;
  two_prod(a.hi, b.hi, p, e);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return df_make(p, e);
}

// a * b for a float b
__device__ __forceinline__ df df_mulf(df a, float b) {
  float p, e;
  two_prod(a.hi, b, p, e);
  e = __fmaf_rn(a.lo, b, e);
  return df_make(p, e);
}

// 1 / sqrt(a), a > 0: an FP32 seed and two Newton steps y <- y + y (1 - a y^2) / 2
// with the residual 1 - a y^2 formed in df64 (each step doubles the correct bits)
__device__ __forceinline__ df df_rsqrt(df a) {
  df y{rsqrtf(a.hi), 0.f};
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const df e = df_sub(df{1.f, 0.f}, df_mul(df_mul(a, y), y));
    y = df_add(y, df_mulf(y, 0.5f * e.hi));
  }
  return y;
}

// Order of normalised pairs (|lo| <= ulp(hi)/2): by the high words, then the
// low words.
__device__ __forceinline__ bool df_le(df a, df b) {
  return a.hi < b.hi || (a.hi == b.hi && a.lo <= b.lo);
}
__device__ __forceinline__ df df_max(df a, df b) { return df_le(a, b) ? b : a; }
__device__ __forceinline__ df df_min(df a, df b) { return df_le(a, b) ? a : b; }
__device__ __forceinline__ df df_abs(df a) { return a.hi < 0.f ? df_neg(a) : a; }

// a / b to about 2^-44: the FP32 quotient of the high words and two corrections
// from the remainder
__device__ __forceinline__ df df_div(df a, df b) {
  const float q0 = __fdiv_rn(a.hi, b.hi);
  df r = df_sub(a, df_mulf(b, q0));
  const float q1 = __fdiv_rn(r.hi, b.hi);
  r = df_sub(r, df_mulf(b, q1));
  const float q2 = __fdiv_rn(r.hi, b.hi);
  return df_add(df_make(q0, q1), df{q2, 0.f});
}

// p = a / b in df64 without an FP64 division: the quotient of the significands,
// scaled.  False (nothing done) for zeros, denormal or non-finite operands and
// quotients outside [2^-100, 2^100].
__device__ __forceinline__ bool df_quotient(double a, double b, df& p);

// Conversions, rounded to nearest even: hi = fl32(x), lo = fl32(x - hi), and
// fl64(hi + lo).  Written with FP64 instructions they are four and three of
// them, and the FP64 pipe takes about 20 clocks per instruction of a warp (a
// pass that converts 17 M values: 124 us against 40 us of bytes).  On the
// device they work on the words instead, about 25 FP32 and integer
// instructions, with the same bits for every input: values whose exponent
// leaves the range below, and pairs that are not normalised, take the FP64
// instructions.
__host__ __device__ __forceinline__ df df_from_double_fp(double x) {
  df r;
  r.hi = (float)x;
  r.lo = (float)(x - (double)r.hi);
  return r;
}
__host__ __device__ __forceinline__ double df_to_double_fp(df a) { return (double)a.hi + (double)a.lo; }

__host__ __device__ __forceinline__ df df_from_double(double x) {
#ifdef __CUDA_ARCH__
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const unsigned e = (h >> 20) & 0x7ffu;
  if (e - 949u > 200u) {  // |x| outside [2^-74, 2^127)
    if (((h << 1) | l) == 0u) return df{__uint_as_float(h), 0.f};
    return df_from_double_fp(x);
  }
  // the significand's top 24 bits, the 29 below rounded: rem - 2^29 up is what
  // hi misses, an integer of the last place
  const unsigned b = (((h & 0x7fffffffu) - 0x38000000u) << 3) | (l >> 29);
  const unsigned rem = l & 0x1fffffffu, up = (rem + 0x0fffffffu + (b & 1u)) >> 29;
  const int r = (int)(rem - (up << 29));
  const unsigned sign = h & 0x80000000u;
  const float place = __uint_as_float(((e - 948u) << 23) | sign);  // +-2^(e - 1075)
  return df{__uint_as_float((b + up) | sign), r == 0 ? 0.f : __fmul_rn(__int2float_rn(r), place)};
#else
  return df_from_double_fp(x);
#endif
}

__host__ __device__ __forceinline__ double df_to_double(df a) {
#ifdef __CUDA_ARCH__
  const unsigned b = __float_as_uint(a.hi), mag = b & 0x7fffffffu;
  // lo in units of the last place that the FP64 result has in hi's binade; the
  // result stays in it unless hi is its lower end and lo points below
  const float t = __fmul_rn(a.lo, __uint_as_float(0x99000000u - (b & 0x7f800000u)));
  if (mag - 0x1a000000u < 0x65800000u && fabsf(t) <= 268435456.f && ((b & 0x7fffffu) != 0u || t == 0.f)) {
    const int sign = (int)b >> 31, n = (__float2int_rn(t) ^ sign) - sign;
    const unsigned long long w =
        (((unsigned long long)((mag >> 3) + 0x38000000u) << 32) | (unsigned)(b << 29)) + (long long)n;
    return __hiloint2double((int)((unsigned)(w >> 32) | (b & 0x80000000u)), (int)(unsigned)w);
  }
  const unsigned bl = __float_as_uint(a.lo);
  if ((mag | (bl << 1)) == 0u) return __hiloint2double((int)(b & bl & 0x80000000u), 0);
  return df_to_double_fp(a);
#else
  return df_to_double_fp(a);
#endif
}

__device__ __forceinline__ bool df_quotient(double a, double b, df& p) {
  const int ha = __double2hiint(a), hb = __double2hiint(b);
  const int ea = (ha >> 20) & 0x7ff, eb = (hb >> 20) & 0x7ff, e = ea - eb;
  if (ea == 0 || ea == 0x7ff || eb == 0 || eb == 0x7ff || e < -100 || e > 100) return false;
  const int one = 0x3ff00000, rest = (int)0x800fffff;
  p = df_div(df_from_double(__hiloint2double((ha & rest) | one, __double2loint(a))),
             df_from_double(__hiloint2double((hb & rest) | one, __double2loint(b))));
  const float scale = __uint_as_float((unsigned)(127 + e) << 23);
  p.hi *= scale;
  p.lo *= scale;
  return true;
}

}  // namespace mgar
