// Float-float ("double-FP32") arithmetic for the mixed-precision path.
//
// GB300 executes FP32 about 55x faster than FP64 (measured 68.6 vs 1.25
// TFLOP/s FMA), so the mixed path evaluates its FP64-class work - the
// temperature Newton solve, transport and the Arrhenius chemistry - on pairs
// of floats.  A value is hi + lo with |lo| <= ulp(hi)/2, about 48 significant
// bits (relative precision ~4e-15), with the exponent range of FP32.
//
// Error-free transformations (published methods):
//   two_sum       Knuth, TAOCP vol. 2: s + e = a + b exactly;
//   fast_two_sum  Dekker 1971: the same when |a| >= |b|;
//   two_prod      with a fused multiply-add: p + e = a * b exactly.
// exp: Tang's table-driven reduction to |r| <= ln2/128 with a 64-entry
// float-float table of 2^(j/64) and a degree-6 polynomial for e^r.
// log: from the FP32 logarithm y, log x = y + log(1 + t) with
// t = x e^(-y) - 1, log(1 + t) to second order (|t| ~ 1e-7).
// Intrinsics with explicit rounding keep the compiler from contracting or
// reassociating the transformations.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

struct ff {
  float hi, lo;
  __host__ __device__ ff() : hi(0.f), lo(0.f) {}
  __host__ __device__ ff(float h, float l) : hi(h), lo(l) {}
  __host__ __device__ explicit ff(float h) : hi(h), lo(0.f) {}
};

__device__ __forceinline__ ff two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return ff(s, e);
}
__device__ __forceinline__ ff fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return ff(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ ff two_prod(float a, float b) {
  const float p = __fmul_rn(a, b);
  return ff(p, __fmaf_rn(a, b, -p));
}

__device__ __forceinline__ ff operator+(ff a, ff b) {
  ff s = two_sum(a.hi, b.hi);
  const ff t = two_sum(a.lo, b.lo);
  s.lo = __fadd_rn(s.lo, t.hi);
  s = fast_two_sum(s.hi, s.lo);
  s.lo = __fadd_rn(s.lo, t.lo);
  return fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ ff operator-(ff a) { return ff(-a.hi, -a.lo); }
__device__ __forceinline__ ff operator-(ff a, ff b) { return a + (-b); }
__device__ __forceinline__ ff operator*(ff a, ff b) {
  ff p = two_prod(a.hi, b.hi);
  p.lo = __fmaf_rn(a.hi, b.lo, p.lo);
  p.lo = __fmaf_rn(a.lo, b.hi, p.lo);
  return fast_two_sum(p.hi, p.lo);
}
__device__ __forceinline__ ff operator/(ff a, ff b) {
  const float q1 = __fdiv_rn(a.hi, b.hi);
  const ff r = a - b * ff(q1);
  const float q2 = __fdiv_rn(r.hi, b.hi);
  const ff r2 = r - b * ff(q2);
  const float q3 = __fdiv_rn(r2.hi, b.hi);
  return fast_two_sum(q1, q2) + ff(q3);
}
__device__ __forceinline__ ff& operator+=(ff& a, ff b) { return a = a + b; }
__device__ __forceinline__ ff& operator-=(ff& a, ff b) { return a = a - b; }
__device__ __forceinline__ ff& operator*=(ff& a, ff b) { return a = a * b; }

// scale by 2^k exactly (k small)
__device__ __forceinline__ ff ff_ldexp(ff a, int k) {
  return ff(ldexpf(a.hi, k), ldexpf(a.lo, k));
}

// 2^(j/64), j = 0..63, each as the nearest float plus the nearest float to
// the remainder (generated in 40-digit arithmetic)
static __device__ const float2 kExp2Tab64[64] = {
    {1.000000000e+00f, 0.000000000e+00f}, {1.010889292e+00f, -5.711605411e-09f},
    {1.021897197e+00f, -4.811559862e-08f}, {1.033024907e+00f, -2.809089317e-08f},
    {1.044273734e+00f, 4.833470157e-08f}, {1.055645227e+00f, -4.907169426e-08f},
    {1.067140460e+00f, -5.933751979e-08f}, {1.078760743e+00f, 5.461594554e-08f},
    {1.090507746e+00f, -1.307753994e-08f}, {1.102382541e+00f, 4.260501996e-08f},
    {1.114386797e+00f, -5.435540018e-08f}, {1.126521587e+00f, 3.123641434e-08f},
    {1.138788581e+00f, 5.386222313e-08f}, {1.151189208e+00f, 2.192228266e-08f},
    {1.163724899e+00f, -4.051441493e-08f}, {1.176396966e+00f, 2.566975077e-08f},
    {1.189207077e+00f, 3.797635273e-08f}, {1.202156782e+00f, -5.069756526e-08f},
    {1.215247393e+00f, -3.267394888e-08f}, {1.228480577e+00f, -4.136200360e-08f},
    {1.241857767e+00f, 4.496838102e-08f}, {1.255380750e+00f, 7.322237483e-09f},
    {1.269050956e+00f, 1.419333318e-09f}, {1.282870054e+00f, -3.816621685e-08f},
    {1.296839595e+00f, -4.018999533e-08f}, {1.310961246e+00f, -3.496571566e-08f},
    {1.325236678e+00f, -3.496373324e-08f}, {1.339667559e+00f, -3.461673970e-08f},
    {1.354255557e+00f, -1.012334927e-08f}, {1.369002461e+00f, -3.845881835e-08f},
    {1.383909941e+00f, -5.875577358e-08f}, {1.398979664e+00f, 8.689434061e-09f},
    {1.414213538e+00f, 2.420323497e-08f}, {1.429613352e+00f, -1.342992917e-08f},
    {1.445180774e+00f, 3.324199938e-08f}, {1.460917830e+00f, -3.628657552e-08f},
    {1.476826191e+00f, -4.500898854e-08f}, {1.492907763e+00f, -3.423620143e-08f},
    {1.509164453e+00f, -2.495937323e-08f}, {1.525598168e+00f, -1.762856883e-08f},
    {1.542210817e+00f, 8.070904833e-09f}, {1.559004426e+00f, -2.576466507e-08f},
    {1.575980902e+00f, -5.661025426e-08f}, {1.593142152e+00f, -4.903136785e-10f},
    {1.610490322e+00f, 9.836217174e-09f}, {1.628027439e+00f, -1.726008314e-08f},
    {1.645755529e+00f, -5.124972091e-08f}, {1.663676620e+00f, -3.920298752e-08f},
    {1.681792855e+00f, -2.475532668e-08f}, {1.700106382e+00f, -2.865147231e-08f},
    {1.718619347e+00f, -4.849617596e-08f}, {1.737333894e+00f, -5.850223417e-08f},
    {1.756252170e+00f, -9.235770371e-09f}, {1.775376439e+00f, 5.343197884e-08f},
    {1.794709086e+00f, -1.141504491e-08f}, {1.814252138e+00f, 3.736258236e-08f},
    {1.834008098e+00f, -1.123927795e-08f}, {1.853979111e+00f, 1.436561181e-08f},
    {1.874167681e+00f, -4.663005626e-08f}, {1.894575953e+00f, 2.810338451e-08f},
    {1.915206552e+00f, 9.845328108e-09f}, {1.936061740e+00f, 5.357072297e-08f},
    {1.957144141e+00f, -1.702180441e-08f}, {1.978456020e+00f, 6.032726318e-09f},
};

__device__ __forceinline__ ff ff_exp(ff x) {
  if (x.hi > 88.7f) return ff(__int_as_float(0x7f800000), 0.f);   // +inf
  if (x.hi < -103.0f) return ff(0.f, 0.f);
  // Table-driven reduction (Tang, ACM TOMS 15(2), 1989): x = (64 n + j) ln2/64
  // + r with |r| <= ln2/128; ln2/64 = L1 + L2 + L3, L1 with 9 significant
  // bits so that k * L1 is exact for every k reached here, and x.hi - k L1
  // is exact too (the operands are within a factor 2 of each other, Sterbenz
  // lemma, or k = 0).  k L3 is below 3e-10 and goes into the low part.
  const float L1 = 0.010833740234375f, L2 = -3.3155381515825866e-06f,
              L3 = 2.572804640231345e-14f;
  const float k = rintf(__fmul_rn(x.hi, 92.33248138427734f));   // 64 / ln2
  // r = x - k ln2/64 = (x.hi - k L1) - hi(k L2) + x.lo - lo(k L2) - k L3:
  // the first difference is exact, the next two terms join it by exact
  // two-sums (x.lo is as large as r's own rounding scale), and the last two
  // (below 1e-9) with the two-sums' errors in FP32.
  const float t = __fsub_rn(x.hi, __fmul_rn(k, L1));
  const ff kL2 = two_prod(k, L2);
  const ff s1 = two_sum(t, -kL2.hi);
  const ff s2 = two_sum(s1.hi, x.lo);
  ff r = two_sum(s2.hi, __fadd_rn(__fadd_rn(s1.lo, s2.lo), -__fmaf_rn(k, L3, kL2.lo)));
  // e^r - 1 = r + r^2/2 + r^2 c, c = r/6 + r^2/24 + r^3/120 + r^4/720: c is
  // below 1e-3 and needs only FP32 (its rounding is below 1e-15 of e^r);
  // the Taylor remainder r^7/5040 is below 1e-19.  |r| <= ln2/128, so
  // r^2/2 < |r|/256: the head sum needs no magnitude test, and the terms
  // below ulp(r.hi) (r.lo, the low part of r^2/2, r^2 c) go in FP32.
  const float rh = r.hi;
  const float c = __fmul_rn(rh, __fmaf_rn(rh, __fmaf_rn(rh, __fmaf_rn(rh, 1.3888889225e-3f,
                                                                           8.3333337680e-3f),
                                                       4.1666667908e-2f),
                                          1.6666667163e-1f));
  const ff r2 = two_prod(rh, rh);                       // r.hi^2 exactly
  const float h2 = __fmul_rn(0.5f, r2.hi);
  ff em1 = fast_two_sum(rh, h2);
  float tail = __fmaf_rn(r2.hi, c, __fmaf_rn(0.5f, r2.lo, r.lo));
  tail = __fmaf_rn(rh, r.lo, tail);                     // the cross term r.hi r.lo
  em1 = fast_two_sum(em1.hi, __fadd_rn(em1.lo, tail));
  const int ki = (int)k;
  const float2 t64 = __ldg(&kExp2Tab64[ki & 63]);
  // y = 2^(j/64) (1 + em1): the head product exactly, the rest in FP32
  const ff p = two_prod(t64.x, em1.hi);
  ff y = fast_two_sum(t64.x, p.hi);
  const float lo = __fmaf_rn(t64.x, em1.lo, __fmaf_rn(t64.y, em1.hi, __fadd_rn(p.lo, t64.y)));
  y = fast_two_sum(y.hi, __fadd_rn(y.lo, lo));
  // scale by 2^e: an exact multiply while 2^e is a normal float
  const int e = ki >> 6;
  if (e >= -126) {
    const float sc = __int_as_float((e + 127) << 23);
    return ff(__fmul_rn(y.hi, sc), __fmul_rn(y.lo, sc));
  }
  return ff_ldexp(y, e);
}

__device__ __forceinline__ ff ff_log(ff x) {
  // y0 = log(x.hi) in FP32 (error d below a few 1e-7 relative), then
  // log x = y0 + log(1 + t), t = x e^(-y0) - 1 (|t| ~ |d|): log(1 + t) =
  // t - t^2/2 + O(t^3), the t^2 term in FP32 (a plain Newton step y0 + t
  // would leave t^2/2, up to 1e-11 for large |log x|)
  const ff y0(logf(x.hi));
  ff t = x * ff_exp(-y0) - ff(1.f);
  t = fast_two_sum(t.hi, __fmaf_rn(-0.5f * t.hi, t.hi, t.lo));
  return y0 + t;
}

// Sums kept as hi + lo without renormalising after every term: the head by
// an exact two-sum, the errors and low parts in one FP32 word (8 operations
// against 20 for operator+; each term's rounding stays below 2^-47 of the
// largest partial sum).  ff_norm closes a sum.
__device__ __forceinline__ void ff_acc(ff& s, ff b) {
  const ff t = two_sum(s.hi, b.hi);
  s.hi = t.hi;
  s.lo = __fadd_rn(s.lo, __fadd_rn(t.lo, b.lo));
}
// s += a b, the product's head exact (12 operations against 27)
__device__ __forceinline__ void ff_fma_acc(ff& s, ff a, ff b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  const ff t = two_sum(s.hi, p);
  s.hi = t.hi;
  s.lo = __fadd_rn(s.lo, __fadd_rn(t.lo, e));
}
__device__ __forceinline__ ff ff_norm(ff s) { return fast_two_sum(s.hi, s.lo); }

// Conversions through the bit patterns.  GB300's FP32 <-> FP64 conversion
// instructions run at the rate of its FP64 pipes (measured: 17 cycles per
// warp and SM, as a DFMA, against 0.26 for an FP32 or integer instruction),
// so the moves between the two formats are integer work here.
//
// |d| < 2^-126 becomes 0, |d| >= 2^128 (and infinities, NaN) NaN; hi is the
// nearest float, lo the 24 leading of the 28 bits that remain (dropped, 0, for
// |d| < 2^-74).
__device__ __forceinline__ ff ff_of_double(double d) {
  const int h = __double2hiint(d), l = __double2loint(d);
  const int mag = h & 0x7fffffff, sgn = h & 0x80000000;
  const int tr = (int)(__funnelshift_l(l, mag, 3) - (896u << 23));   // truncated
  const int up = (l >> 28) & 1;                       // the first bit below it
  const int rest = (l & 0x1fffffff) - (up << 29);
  int hb = tr + up;
  if (mag < 0x38100000) hb = 0;                       // below 2^-126
  if (mag >= 0x47f00000) hb = 0x7fffffff;             // 2^128 and above
  const int sc = max((tr & 0x7f800000) - (52 << 23), 0);
  const float lo = __fmul_rn(__int2float_rn(rest), __int_as_float(sc | sgn));
  return ff(__int_as_float(hb | sgn), mag < 0x38100000 ? 0.f : lo);
}
// exact for 0 and normal numbers; denormals become 0
__device__ __forceinline__ double double_of_float(float f) {
  const int b = __float_as_int(f);
  const int m = b & 0x7fffffff;
  int h = (m >> 3) + (896 << 20);
  if (m < 0x00800000) h = 0;
  if (m >= 0x7f800000) h = m > 0x7f800000 ? 0x7ff80000 : 0x7ff00000;
  return __hiloint2double(h | (b & 0x80000000), m < 0x00800000 ? 0 : b << 29);
}
// exact for denormals too
__device__ __forceinline__ double double_of_float_exact(float f) {
  const bool sub = (__float_as_int(f) & 0x7fffffff) < 0x00800000;
  const double d = double_of_float(sub ? f * 16777216.f : f);
  const int h = __double2hiint(d), l = __double2loint(d);
  return __hiloint2double(sub && (h << 1) != 0 ? h - (24 << 20) : h, l);
}
// rounded to nearest (the conversion instruction for results that are denormal
// or infinite)
__device__ __forceinline__ float float_of_double(double d) {
  const int h = __double2hiint(d), l = __double2loint(d), mag = h & 0x7fffffff;
  if ((unsigned)(mag - 0x38100000) >= 0x0fe00000u)
    return mag < 0x36900000 ? __int_as_float(h & 0x80000000) : __double2float_rn(d);
  const unsigned up = (unsigned)(l & 0x1fffffff) + ((l >> 29) & 1) > 0x10000000u;
  return __int_as_float(((int)(__funnelshift_l(l, mag, 3) - (896u << 23)) + (int)up) |
                        (h & 0x80000000));
}
__device__ __forceinline__ double double_of_ff(ff a) {
  return double_of_float(a.hi) + double_of_float(a.lo);
}
// The same for a normalised pair (|lo| <= ulp(hi) / 2), the low part joined to
// the head's mantissa by an integer addition; through the FP64 pipe below
// 2^-75, where lo's weight leaves FP32's range.
__device__ __forceinline__ double double_join(ff a) {
  const int b = __float_as_int(a.hi), m = b & 0x7fffffff;
  if (m < (52 << 23) || m >= 0x7f800000) return double_of_ff(a);
  const float w = __int_as_float((int)((306u << 23) - (m & 0x7f800000u)));   // 2^(52 - exponent)
  int l = __float2int_rn(__fmul_rn(a.lo, w));
  if (b < 0) l = -l;
  if (l < 0 && (m & 0x007fffff) == 0) l += l;   // below a power of two the last bit counts half
  const unsigned long long d =
      ((unsigned long long)((m >> 3) + (896 << 20)) << 32 | ((unsigned)b << 29)) + (long long)l;
  return __longlong_as_double((long long)(d | (unsigned long long)(b & 0x80000000u) << 32));
}
// d = m 2^e, 1 <= |m| < 2 (0 and denormals: m = 0; infinities, NaN: m = NaN)
__device__ __forceinline__ ff ff_mantissa(double d, int& e) {
  const int h = __double2hiint(d), ex = (h >> 20) & 0x7ff;
  e = ex - 1023;
  if (ex == 0x7ff) return ff(__int_as_float(0x7fffffff), 0.f);
  return ex == 0 ? ff() : ff_of_double(__hiloint2double((h & 0x800fffff) | 0x3ff00000,
                                                        __double2loint(d)));
}
// a 2^e for a normalised pair, 0 below FP64's normal numbers
__device__ __forceinline__ double double_join(ff a, int e) {
  const double d = double_join(a);
  const int h = __double2hiint(d), ex = (h >> 20) & 0x7ff;
  if (ex == 0x7ff) return d;
  if (ex == 0 || ex + e <= 0) return 0.0;
  return __hiloint2double(h + (e << 20), __double2loint(d));
}
// 1 / a
__device__ __forceinline__ ff ff_rcp(ff a) {
  const float q = __fdiv_rn(1.f, a.hi);
  float e = __fmaf_rn(-q, a.hi, 1.f);
  e = __fmaf_rn(-q, a.lo, e);
  return fast_two_sum(q, __fmul_rn(q, e));
}
// a / b to ~46 bits (a Newton update's quotient)
__device__ __forceinline__ ff ff_quotient(ff a, ff b) {
  const float r = __fdiv_rn(1.f, b.hi);
  const float q = __fmul_rn(a.hi, r);
  const ff p = two_prod(q, b.hi);
  float e = __fsub_rn(__fsub_rn(a.hi, p.hi), p.lo);
  e = __fadd_rn(e, __fmaf_rn(-q, b.lo, a.lo));
  return fast_two_sum(q, __fmul_rn(e, r));
}
// a pair in a double's place
__device__ __forceinline__ double ff_pack(ff a) {
  return __hiloint2double(__float_as_int(a.hi), __float_as_int(a.lo));
}
__device__ __forceinline__ ff ff_unpack(double d) {
  return ff(__int_as_float(__double2hiint(d)), __int_as_float(__double2loint(d)));
}

// 0 <= d < 2^(63 - bits) as an integer with `bits` fraction bits; the largest
// integer above
__device__ __forceinline__ long long fixed_of(double d, int bits) {
  const int h = __double2hiint(d);
  const unsigned long long m =
      ((unsigned long long)(unsigned)((h & 0xfffff) | 0x100000) << 42) |
      ((unsigned long long)(unsigned)__double2loint(d) << 10);    // 62 fraction bits
  const int sh = 62 + 1023 - bits - (h >> 20);
  return sh < 0 ? 0x7fffffffffffffffLL : (long long)(m >> min(sh, 63));
}

// Exponentials of the float-float reaction rates.  The argument comes in units
// of ln2/64 (the mechanism's coefficients are scaled by 64/ln2 on the host), as
// the nearest integer n and the rest r = rh + rl, |r| <= 1/2; e^x = y 2^e with
// e = floor(n / 64) and y = 2^(j/64) e^z, z = r ln2/64 (Tang's reduction,
// as ff_exp).
struct ExpArg {
  int n;
  float rh, rl;
};
// arguments beyond +-16000 (e^+-173) are held at that bound; NaN stays NaN
constexpr float kExpArgMax = 16000.f;

// x = xh + xl in units of ln2/64
__device__ __forceinline__ ExpArg exp_arg(ff x) {
  ExpArg a;
  const float xh = fminf(fmaxf(x.hi, -kExpArgMax), kExpArgMax);   // NaN: -kExpArgMax
  const float t = __fadd_rn(xh, 12582912.f);                       // 1.5 2^23: rounds
  a.n = __float_as_int(t) - 0x4b400000;
  const ff r = two_sum(__fsub_rn(xh, __fsub_rn(t, 12582912.f)),
                       fabsf(x.hi) <= kExpArgMax ? x.lo : (x.hi != x.hi ? x.hi : 0.f));
  a.rh = r.hi;
  a.rl = r.lo;
  return a;
}

__device__ __forceinline__ ff exp_frac(const ExpArg& a) {
  // z = r ln2/64 as p + e
  const float C1 = 0x1.62e43p-7f, C2 = -0x1.05c61p-35f;   // ln2/64 = C1 + C2
  const float p = __fmul_rn(a.rh, C1);
  float e = __fmaf_rn(a.rh, C1, -p);
  e = __fmaf_rn(a.rh, C2, e);
  e = __fmaf_rn(a.rl, C1, e);
  // e^z - 1 = z + z^2/2 + z^3 (1/6 + z/24 + z^2/120 + z^3/720), the last
  // group (below 3e-8) in FP32
  const float q = __fmul_rn(p, p);
  const float qe = __fmaf_rn(p, p, -q);
  float c = __fmaf_rn(p, 1.3888889225e-3f, 8.3333337680e-3f);
  c = __fmaf_rn(p, c, 4.1666667908e-2f);
  c = __fmaf_rn(p, c, 1.6666667163e-1f);
  const ff s = fast_two_sum(p, __fmul_rn(0.5f, q));
  float lo = __fmaf_rn(0.5f, qe, __fmaf_rn(p, e, e));
  lo = __fmaf_rn(__fmul_rn(p, q), c, lo);
  lo = __fadd_rn(s.lo, lo);
  // 2^(j/64) (1 + em1)
  const float2 t = __ldg(&kExp2Tab64[a.n & 63]);
  const ff w = two_prod(t.x, s.hi);
  const ff y = fast_two_sum(t.x, w.hi);
  lo = __fmaf_rn(t.x, lo, __fmaf_rn(t.y, s.hi, __fadd_rn(w.lo, t.y)));
  return fast_two_sum(y.hi, __fadd_rn(y.lo, lo));
}
// a 2^e, |e| <= 256, in two exact factors
__device__ __forceinline__ ff ff_scale(ff a, int e) {
  const int e1 = e >> 1;
  const float s1 = __int_as_float((e1 + 127) << 23);
  const float s2 = __int_as_float((e - e1 + 127) << 23);
  return ff(__fmul_rn(__fmul_rn(a.hi, s1), s2), __fmul_rn(__fmul_rn(a.lo, s1), s2));
}

__device__ __forceinline__ double ff_to_double(ff a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ ff ff_from_double(double d) {
  const float h = __double2float_rn(d);
  return ff(h, __double2float_rn(d - (double)h));
}
__host__ inline ff ff_host(double d) {
  const float h = (float)d;
  return ff(h, (float)(d - (double)h));
}

}  // namespace lbm
