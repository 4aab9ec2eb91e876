// Float-float ("double-single") arithmetic: a value is the unevaluated sum hi + lo of two
// FP32 numbers with |lo| <= ulp(hi)/2, about 48 significant bits.  Error-free transformations
// after Dekker (1971) and Knuth (TAOCP vol. 2): two_sum exact by six additions, two_prod
// exact by one product and one FMA.  GB300 runs FP32 about 60x faster than FP64, so a few
// FP32 operations per FP64 operation still relieve the FP64 pipe where 2^-46 relative
// accuracy is enough.
#pragma once

struct ff {
  float hi, lo;
};

__device__ __forceinline__ ff ff_make(float hi, float lo) {
  ff r;
  r.hi = hi;
  r.lo = lo;
  return r;
}

// (hi + lo) 2^shift as a double by integer instructions (normalised float-float, hi normal or zero;
// low parts below 2^-46 of hi round away; zero below the double range, infinite above it, NaN when hi
// is not finite).
__device__ __forceinline__ double ff_join(ff a, int shift) {
  const unsigned hb = __float_as_uint(a.hi), sg = hb & 0x80000000u;
  const int e = (int)((hb >> 23) & 0xffu);
  // |hi| as an integer with 46 fraction bits, and the low part (at most 2^22) in the same unit, 2^(e - 173)
  const int up = e < 64 ? 64 : 0;
  const float unit = __uint_as_float((unsigned)max(300 - e - up, 1) << 23);
  const float l = __uint_as_float(__float_as_uint(a.lo) ^ sg) * unit * (up ? 0x1p64f : 1.f);
  const int q = __float_as_int(__fadd_rn(l, 12582912.f)) - 0x4B400000;
  long long m = ((long long)((hb & 0x7fffffu) | 0x800000u) << 23) + q;
  const int below = m < (1LL << 46);
  m <<= 6 + below;
  const int ex = e - 127 + 1023 - below + shift;
  long long r = ((long long)ex << 52) + (m & 0xfffffffffffffLL);
  if (e == 255 || ex >= 2047) r = e == 255 ? 0x7ff8000000000000LL : 0x7ff0000000000000LL;
  return e == 0 || ex <= 0 ? 0.0 : __longlong_as_double(r | ((long long)sg << 32));
}

// nearest float-float of a double (two conversions and one FP64 subtraction)
__device__ __forceinline__ ff ff_from_double(double x) {
  const float hi = __double2float_rn(x);
  const float lo = __double2float_rn(x - (double)hi);
  return ff_make(hi, lo);
}

// The same to 47 bits (nearest) by integer and FP32 instructions, for kernels whose FP64 pipe is the
// bound: hi = the top 24 bits, lo = the next 23 (rounded to FP32's smallest numbers below 2^-80 of the
// value).  Values below 2^-126 give zero; from 2^128 on, and for infinities and NaN, hi is not finite.
__device__ __forceinline__ ff ff_split(double v) {
  const unsigned hv = (unsigned)__double2hiint(v), top = hv & 0x7fffffffu;
  // half of the last bit kept is added to |v|, in words: as one 64-bit mask it becomes an FP64 abs, whose
  // result for a NaN has no fixed sign
  const unsigned l = (unsigned)__double2loint(v) + 32u, h = top + (l < 32u ? 1u : 0u);
  // exponent and 23 bits of the fraction, moved to FP32's place and bias: two upper exponent bits drop out, and
  // 1023 - 127 = 896 is -128 modulo 2^9
  unsigned hb = __funnelshift_l(l, h, 3) + (128u << 23);
  hb = top < (897u << 20) ? 0u : (top >= (1151u << 20) ? 0x7fc00000u : hb);
  hb |= hv & 0x80000000u;
  const float low = __fsub_rn(__uint_as_float(0x4B000000u | ((l >> 6) & 0x7fffffu)), 8388608.f);
  return ff_make(__uint_as_float(hb), __fmul_rn(__fmul_rn(low, 0x1p-46f), __uint_as_float(hb & 0xff800000u)));
}

// The same of v 2^shift, |shift| < 1000 (zero where that leaves the normal range of FP64 below).
__device__ __forceinline__ ff ff_split_scaled(double v, int shift) {
  const int hv = __double2hiint(v), e = (hv >> 20) & 0x7ff;
  if (e == 0 || e + shift <= 0) return ff_make(0.f, 0.f);
  return ff_split(e + shift >= 0x7ff ? v : __hiloint2double(hv + (shift << 20), __double2loint(v)));
}

__device__ __forceinline__ double ff_to_double(ff a) { return (double)a.hi + (double)a.lo; }

__device__ __forceinline__ ff ff_quick_two_sum(float a, float b) {   // |a| >= |b|
  const float s = __fadd_rn(a, b);
  const float e = __fsub_rn(b, __fsub_rn(s, a));
  return ff_make(s, e);
}

__device__ __forceinline__ ff ff_two_sum(float a, float b) {   // exact a + b
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return ff_make(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}

__device__ __forceinline__ ff ff_add(ff a, ff b) {
  const float s = __fadd_rn(a.hi, b.hi);
  const float bb = __fsub_rn(s, a.hi);
  float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
  e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return ff_quick_two_sum(s, e);
}

__device__ __forceinline__ ff ff_neg(ff a) { return ff_make(-a.hi, -a.lo); }

__device__ __forceinline__ ff ff_sub(ff a, ff b) { return ff_add(a, ff_neg(b)); }

__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return ff_quick_two_sum(p, e);
}

// a * b + c
__device__ __forceinline__ ff ff_fma(ff a, ff b, ff c) { return ff_add(ff_mul(a, b), c); }

__device__ __forceinline__ ff ff_scale(ff a, float s) {   // a * s for an exact FP32 factor s
  const float p = __fmul_rn(a.hi, s);
  float e = __fmaf_rn(a.hi, s, -p);
  e = __fmaf_rn(a.lo, s, e);
  return ff_quick_two_sum(p, e);
}

// Compensated accumulation of the product a b (float-float operands) into (h, l).
__device__ __forceinline__ void ff_mac(float& h, float& l, ff a, ff b) {
  const float v = __fmul_rn(a.hi, b.hi);
  const float e = __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -v)));
  const ff m = ff_two_sum(h, v);
  h = m.hi;
  l = __fadd_rn(l, __fadd_rn(m.lo, e));
}
