// Double-float sums: a value as an unevaluated FP32 pair (sum, error), accumulated with Knuth's
// TwoSum on the FP32 pipes, and its conversion to FP64 on the integer pipes.
#pragma once
#include <cmath>

#include "common.cuh"

namespace pcopt {

struct DF {
  float hi, lo;
};

// (hi, lo) += x exactly (TwoSum; no contraction into FMA)
__device__ __forceinline__ void df_add(DF& a, float x) {
  const float s = __fadd_rn(a.hi, x);
  const float bb = __fsub_rn(s, a.hi);
  const float err = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(x, bb));
  a.hi = s;
  a.lo = __fadd_rn(a.lo, err);
}

// (hi, lo) += (kh + kl) u
__device__ __forceinline__ void df_add_prod(DF& a, float kh, float kl, float u) {
  const float p = __fmul_rn(kh, u);
  const float e = fmaf(kh, u, -p);
  df_add(a, p);
  a.lo = __fadd_rn(a.lo, fmaf(kl, u, e));
}

// (hi + lo) 2^-p as the nearest FP64 value, without the FP64 unit.  With s + e = hi + lo, s the
// rounded sum, |e| is at most half a unit of s's 24th bit, so e moves the FP64 bit pattern of s
// by e / 2^(exponent of s - 52), an integer of at most 30 bits; below a power of two the
// pattern's step is half as long.  Zero, subnormal sums, infinities and NaN take the FP64 sum
// of the converted parts.  About 30 integer and FP32 operations where two conversions and the
// FP64 addition were 20 and one of the 12 FP64 operations a point that bounded the element
// products (12 x 2.06 M points = 47 of the 75 us at 127^2 x 128).
__device__ __forceinline__ double df_to_f64(const DF& a, int p) {
  const float s = __fadd_rn(a.hi, a.lo);
  const float bb = __fsub_rn(s, a.hi);
  const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(a.lo, bb));
  const unsigned us = __float_as_uint(s), ue = __float_as_uint(e);
  const int Es = (int)((us >> 23) & 0xFFu), Ee = (int)((ue >> 23) & 0xFFu);
  if (Es == 0 || Es == 0xFF) return scalbn(f32_to_f64(a.hi) + f32_to_f64(a.lo), -p);
  const unsigned ms = us & 0x7FFFFFu, me = (ue & 0x7FFFFFu) | 0x800000u;
  const bool minus = ((us ^ ue) >> 31) != 0;
  int sh = 29 - (Es - Ee) + (minus && ms == 0 ? 1 : 0);  // at most 6
  sh = sh < -30 ? -30 : sh;
  unsigned d = sh >= 0 ? me << sh : (me + ((1u << -sh) >> 1)) >> -sh;
  d = Ee == 0 ? 0u : d;
  unsigned long long bits = ((unsigned long long)((unsigned)(Es + 896 - p) << 20 | (ms >> 3)) << 32) | (ms << 29);
  bits = minus ? bits - d : bits + d;
  bits |= (unsigned long long)(us & 0x80000000u) << 32;
  return __longlong_as_double((long long)bits);
}

// Scale 2^p that brings tk into [1/2, 1): element products keep tk K 2^p in FP32 pairs, which no
// K in the FP32 range overflows, and take 2^-p in df_to_f64.
inline int df_scale_exponent(double tk) {
  int e = 0;
  std::frexp(tk, &e);
  return -e;
}
// whether the exponent field of df_to_f64's result, Es + 896 - p, holds for every FP32 sum
// (1 <= Es <= 254); beyond (tau below 1e-270 or above 1e269) the products take FP64 arithmetic
inline bool df_scale_fits(int p) { return p >= -896 && p <= 896; }

}  // namespace pcopt
