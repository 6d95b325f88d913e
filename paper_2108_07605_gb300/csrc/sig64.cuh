// Reaction rates in 64-bit significands: a value is m 2^e, m a signed 64-bit
// integer, e an int, so that a rate constant, the concentrations and their
// products neither round at 53 bits nor leave FP64's range on the way.
//
// On GB300 an FP64 instruction occupies an SM quarter for 64 to 75 cycles per
// warp, an integer one for 1 or 2: this keeps ~35 FP64 instructions per reaction
// off that pipe, with errors below FP64's.  Pairs of FP32 (48 bits, FP32's range)
// in its place are a little faster (10 steps of the 600x40x40 tube 57.1 ms
// against 58.8), but lose trace species and rates below 1e-38.
#pragma once

#include "ff.cuh"

namespace lbm {

struct Sig {
  long long m;
  int e;
};
constexpr int kSigNaN = 1 << 20;      // e from half of this on: not a number

// exact for 0 and normal numbers, |m| in [2^62, 2^63); denormals become 0
__device__ __forceinline__ Sig sig_of(double v) {
  const int h = __double2hiint(v), ex = (h >> 20) & 0x7ff;
  long long m = (long long)((unsigned long long)(unsigned)((h & 0xfffff) | 0x100000) << 42 |
                            (unsigned long long)(unsigned)__double2loint(v) << 10);
  if (ex == 0) m = 0;
  return Sig{h < 0 ? -m : m, ex == 0x7ff ? kSigNaN : ex - 1085};
}
// rounded to nearest; 0 below FP64's normal numbers, infinite above them
__device__ __forceinline__ double double_of_sig(Sig s) {
  if (s.m == 0) return 0.0;
  const unsigned sgn = (unsigned)(s.m >> 32) & 0x80000000u;
  unsigned long long a =
      s.m < 0 ? 0ull - (unsigned long long)s.m : (unsigned long long)s.m;
  const int z = __clzll((long long)a);
  a <<= z;                                     // leading bit at 63
  const unsigned long long r = ((a >> 10) + 1) >> 1;          // 53 bits, rounded
  const int ex = s.e + 1086 - z;               // biased exponent of the leading bit
  unsigned long long d = ex <= 0 ? 0 : ((unsigned long long)(ex - 1) << 52) + r;
  if (ex >= 0x7ff) d = s.e >= kSigNaN / 2 ? 0x7ff8000000000000ull : 0x7ff0000000000000ull;
  return __longlong_as_double((long long)(d | (unsigned long long)sgn << 32));
}
__device__ __forceinline__ Sig operator*(Sig a, Sig b) {
  return Sig{__mul64hi(a.m, b.m), a.e + b.e + 64};
}
// |a.m|, |b.m| < 2^62
__device__ __forceinline__ Sig operator-(Sig a, Sig b) {
  const int ea = a.m == 0 ? -(1 << 22) : a.e, eb = b.m == 0 ? -(1 << 22) : b.e;
  const int e = max(ea, eb);
  return Sig{(a.m >> min(e - ea, 63)) - (b.m >> min(e - eb, 63)), e};
}

// 2^(j/64) 2^62 (60-digit arithmetic)
static __device__ const long long kExp2Sig64[64] = {
    0x4000000000000000LL, 0x40b268f9de0183baLL, 0x4166c34c5615d0ecLL, 0x421d1461d66f2023LL,
    0x42d561b3e6243d8aLL, 0x438fb0cb4f468808LL, 0x444c0740496d4294LL, 0x450a6abaa4b77ecdLL,
    0x45cae0f1f545eb73LL, 0x468d6fadbf2dd4f3LL, 0x47521cc5a2e6a9e0LL, 0x4818ee218a3358eeLL,
    0x48e1e9b9d588e19bLL, 0x49ad159789f37496LL, 0x4a7a77d47f7b84b1LL, 0x4b4a169b900c2d00LL,
    0x4c1bf828c6dc54b8LL, 0x4cf022c9905bfd32LL, 0x4dc69cdceaa72a9cLL, 0x4e9f6cd3967fdba8LL,
    0x4f7a993048d088d7LL, 0x50582887dcb8a7e1LL, 0x513821818624b40cLL, 0x521a8ad704f3404fLL,
    0x52ff6b54d8a89c75LL, 0x53e6c9da74b29ab5LL, 0x54d0ad5a753e077cLL, 0x55bd1cdad49f699cLL,
    0x56ac1f752150a563LL, 0x579dbc56b48521baLL, 0x5891fac0e95612c8LL, 0x5988e20954889245LL,
    0x5a827999fcef3242LL, 0x5b7ec8f19468bbc9LL, 0x5c7dd7a3b17dcf75LL, 0x5d7fad59099f22feLL,
    0x5e8451cfac061b5fLL, 0x5f8bccdb3d398841LL, 0x6096266533384a2bLL, 0x61a3666d124bb204LL,
    0x62b39508aa836d6fLL, 0x63c6ba6455dcd8aeLL, 0x64dcdec3371793d1LL, 0x65f60a7f79393e2eLL,
    0x6712460a8fc24072LL, 0x683199ed779592caLL, 0x69540ec8f895722dLL, 0x6a79ad55e7f6fd10LL,
    0x6ba27e656b4eb57aLL, 0x6cce8ae13c57ebdbLL, 0x6dfddbcbed791babLL, 0x6f307a412f074892LL,
    0x70666f76154a7089LL, 0x719fc4b95f452d29LL, 0x72dc8373be41a454LL, 0x741cb5281e25ee34LL,
    0x75606373ee921c97LL, 0x76a7980f6cca15c2LL, 0x77f25ccdee6d7ae6LL, 0x7940bb9e2cffd89dLL,
    0x7a92be8a92436616LL, 0x7be86fb985689ddcLL, 0x7d41d96db915019dLL, 0x7e9f06067a4360baLL,
};
// e^x, the argument v in units of ln2/64 with 46 fraction bits, |v| < 2^62:
// n = v to the nearest integer, j = n mod 64, e^x = 2^(n div 64) 2^(j/64) e^z,
// z = r ln2/64, |r| <= 1/2 (Tang's reduction, ACM TOMS 15(2), 1989), by the
// Taylor polynomial z + z^2 (1/2 + z/6 + z^2 (1/24 + z/120 + z^2/720)) in fixed
// point (remainder below 2^-64).  Relative error below 2^-56; 0 < m < 2^62.
__device__ __forceinline__ Sig exp_sig(long long v) {
  const int n = ((int)(v >> 32) + (1 << 13)) >> 14;
  const long long r = (long long)((unsigned long long)v << 18);       // 64 fraction bits
  const long long z = __mul64hi(r, 6393154322601327830LL);               // 69
  const long long zz = __mul64hi(z, z);                               // z^2: 74
  const int zh = (int)(z >> 32), z2 = (int)(zz >> 32);                // 37, 42
  const int c = 178956971 + __mulhi(zh, 1118481) + __mulhi(z2, 5825); // 32
  const long long h = (1LL << 61) + __mul64hi(z, 24019198012642645LL) +
                      ((long long)__mulhi(z2, c) << 20);              // 62
  const long long em1 = z + (__mul64hi(zz, h) >> 3);                  // e^z - 1: 69
  const long long t = __ldg(&kExp2Sig64[n & 63]);
  return Sig{(t + (__mul64hi(t, em1) >> 5)) >> 1, (n >> 6) - 61};
}
// x in units of ln2/64: infinite from 65536 (e^709.8) on, 0 below -65536
__device__ __forceinline__ Sig exp_sig(double x) {
  const int h = __double2hiint(x);
  if ((h & 0x7fffffff) >= 0x40f00000) {
    if (x != x) return Sig{1LL << 61, kSigNaN};
    return Sig{h < 0 ? 0 : 1LL << 61, 1 << 16};
  }
  const long long v = fixed_of(__hiloint2double(h & 0x7fffffff, __double2loint(x)), 46);
  return exp_sig(h < 0 ? -v : v);
}

}  // namespace lbm
