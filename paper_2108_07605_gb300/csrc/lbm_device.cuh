// Device-side building blocks of the reactive-mixture LBM step.
//
// Lattice: D3Q27 / D2Q9 product-form velocity sets, index
// i = (cz+1)*9 + (cy+1)*3 + (cx+1) (x fastest), opposite = Q-1-i (Sec. 2.2).
// Thermodynamics, rates and transport are evaluated from the precomputed
// polynomial forms in DevMech (filled on the host from lbm_mechanism).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "exp64.cuh"
#include "log64.cuh"
#include "sig64.cuh"
#include "lbm_internal.h"

namespace lbm {

template <int D> struct Lat;
template <> struct Lat<3> {
  static constexpr int Q = 27;
  static constexpr int NP = 6;   // xx, yy, zz, xy, xz, yz
};
template <> struct Lat<2> {
  static constexpr int Q = 9;
  static constexpr int NP = 3;   // xx, yy, xy
};

// component a (0 = x, 1 = y, 2 = z) of velocity i
__host__ __device__ constexpr int cvel(int i, int a) {
  return a == 0 ? (i % 3) - 1 : (a == 1 ? ((i / 3) % 3) - 1 : (i / 9) - 1);
}
__host__ __device__ constexpr int csq(int i, int D) {
  return cvel(i, 0) * cvel(i, 0) + cvel(i, 1) * cvel(i, 1) +
         (D == 3 ? cvel(i, 2) * cvel(i, 2) : 0);
}
// Per-axis product-form factor Psi_c(xi, P), Eqs. phi0, phiPlus, phis.
template <typename R>
__device__ __forceinline__ R psi1(int c, R xi, R P) {
  return c == 0 ? (R(1) - P) : (c == 1 ? R(0.5) * (P + xi) : R(0.5) * (P - xi));
}

// Reading R5 of Eq. momentum1: u_a := u when rho_a <= 1e-300 or when some
// |j_a| >= rho_a (impossible for non-negative populations; it arises only
// from cancellation in near-zero densities, where j_a / rho_a is noise).
template <int D, typename R>
__host__ __device__ __forceinline__ bool species_velocity_undefined(R rho_a, const R* j_a) {
  bool bad = sizeof(R) == 4 ? rho_a <= R(0)              // FP32: no value below 1e-300
                            : double(rho_a) <= RHO_TINY;
  for (int d = 0; d < D; ++d) bad |= fabs(j_a[d]) >= rho_a;
  return bad;
}

// Moment-record field offsets ([field][N] scratch in the lattice compute
// type, written by the moments and boundary kernels, read by the collision
// kernel).  Neighbours read H and PHI only.
template <int D, int M> struct Rec {
  static constexpr int RHO = 0;
  static constexpr int U = 1;
  static constexpr int Z = U + D;               // q - u . P (energy flux less the work of P)
  static constexpr int E = Z + D;
  static constexpr int Y = E + 1;
  // sum_a Y_a H_a(T)/c^2 as a polynomial in T: its gradient at a node's own T
  // is sum_a H_a grad Y_a, from four fields per neighbour instead of M
  static constexpr int H = Y + M;
  static constexpr int US = H + 4;              // u_a - u (record_us)
  static constexpr int PHI = US + M * D;
  static constexpr int DRHO = PHI + D;          // reaction increments, species a < M
  static constexpr int TH = DRHO + M - 1;       // theta = R T / c^2
  static constexpr int LNT = TH + 1;            // ln(T / T0)
  static constexpr int NF = LNT + 1;
};

// u_a - u as the record holds it: in FP64 a float-float pair, the type of the
// diffusion velocities it becomes
__device__ __forceinline__ float record_us(float v) { return v; }
__device__ __forceinline__ double record_us(double v) { return ff_pack(ff_of_double(v)); }

// ------------------------------------------------------------------------
// Sums of FP64 values in fixed point.  An FP64 addition occupies an SM quarter
// of GB300 for 75 cycles, an integer one for 1: a group of values (one
// lattice's populations at a node) is shifted to a common exponent, that of
// the largest, and added in integers.  A value is cut at 2^-63 of the largest
// one's power of two (a double's own last bit lies at 2^-52 of it), and the
// sums of a lattice's 27 terms are exact (31 fit a); with the small differences that a momentum
// is made of, this is what FP64 differences keep, and more.
//
// Fix: the value modulo 2^64 in units of 2^(e - 63), and a, the same in units
// of 2^(e - 25), each term rounded towards 0, which says which multiple of
// 2^64 was lost.
struct Fix {
  unsigned long long lo;
  int a;
  __device__ Fix() : lo(0), a(0) {}
  __device__ Fix(unsigned long long l, int a_) : lo(l), a(a_) {}
};
__device__ __forceinline__ Fix operator+(Fix x, Fix y) { return Fix(x.lo + y.lo, x.a + y.a); }
__device__ __forceinline__ Fix operator-(Fix x, Fix y) { return Fix(x.lo - y.lo, x.a - y.a); }

// biased exponent of v; the common one is the maximum over the group
__device__ __forceinline__ int fix_exponent(double v) {
  return (__double2hiint(v) >> 20) & 0x7ff;
}
__device__ __forceinline__ Fix fix_of(double v, int e) {
  const int h = __double2hiint(v), l = __double2loint(v);
  const int ev = (h >> 20) & 0x7ff;
  const unsigned hm = (unsigned)((h & 0xfffff) | 0x100000);
  unsigned long long m = ((unsigned long long)(hm << 11 | (unsigned)l >> 21) << 32) |
                         (unsigned)(l << 11);
  m >>= min(e - ev, 63);
  if (ev == 0 || e - ev > 63) m = 0;           // zeros, denormals, values far below
  const int a = (int)(m >> 38);
  return h < 0 ? Fix(0ull - m, -a) : Fix(m, a);
}
// The sum as a signed integer s in units of 2^(e - 1023 - 57), e the biased
// exponent to be used with it: six bits finer than asked for where it fits.
struct FixSum {
  long long s;
  int e;
};
__device__ __forceinline__ FixSum fix_sum(Fix v, int e) {
  // |value / 2^38 - a| <= the number of terms
  const int k = (v.a - (int)(v.lo >> 38) + (1 << 25)) >> 26;
  const long long f = (long long)v.lo;
  if (k == (int)(f >> 63)) return FixSum{f, e - 6};
  return FixSum{((long long)k << 58) + (long long)(((v.lo >> 5) + 1) >> 1), e};
}
// s shifted down by sh >= 0 exponents, rounded
__device__ __forceinline__ long long fix_down(long long s, int sh) {
  return sh <= 0 ? s : ((s >> min(sh - 1, 62)) + 1) >> 1;
}
// the value, rounded to nearest; NaN when e is near that of infinities
__device__ __forceinline__ double double_of_fix(long long s, int e) {
  return e >= 0x7f0 ? __longlong_as_double(0x7ff8000000000000LL) : double_of_sig(Sig{s, e - 1080});
}
__device__ __forceinline__ double double_of_fix(FixSum v) { return double_of_fix(v.s, v.e); }

// ------------------------------------------------------------------------
// thermodynamics (Sec. 3.1)
// U_a(T) = u0 + u1 T + u2 T^2 + u3 T^3 (J/kg), C_av = dU_a/dT.

template <int M>
__device__ __forceinline__ void mixture_energy_poly(const DevMech& m, const double* Y,
                                                    double c[4]) {
  c[0] = c[1] = c[2] = c[3] = 0.0;
#pragma unroll
  for (int a = 0; a < M; ++a) {
    c[0] += Y[a] * m.u0[a];
    c[1] += Y[a] * m.u1[a];
    c[2] += Y[a] * m.u2[a];
    c[3] += Y[a] * m.u3[a];
  }
}

// Newton on sum_a Y_a U_a(T) = U (Eq. temperature) for the polynomial's
// coefficients c; stops when the update satisfies |dT| <= rtol |T| after it is
// applied; ok = false after max_iter.  The residual and T are FP64, the
// derivative and the quotient (46 bits of a correction) float-float: four
// FP64 instructions per iteration instead of ~22.
__device__ __forceinline__ double newton_poly(const double (&c)[4], double U, double T,
                                              int max_iter, double rtol, bool& ok) {
  const double c0 = c[0] - U;
  const ff d1 = ff_of_double(c[1]);
  ff d2 = ff_of_double(c[2]), d3 = ff_of_double(c[3]);
  d2 = ff(2.f * d2.hi, 2.f * d2.lo);
  d3 = ff(3.f) * d3;
  const float tol = (float)rtol;
  ok = false;
  for (int it = 0; it < max_iter; ++it) {
    const double F = fma(T, fma(T, fma(T, c[3], c[2]), c[1]), c0);
    const ff Tf = ff_of_double(T);
    ff e = d2;
    ff_fma_acc(e, d3, Tf);
    ff dF = d1;
    ff_fma_acc(dF, ff_norm(e), Tf);
    const ff dT = -ff_quotient(ff_of_double(F), ff_norm(dF));
    T += double_join(dT);
    if (fabsf(dT.hi) <= tol * fabsf(Tf.hi)) { ok = true; break; }
  }
  return T;
}

// c receives the polynomial's coefficients
template <int M>
__device__ __forceinline__ double newton_T(const DevMech& m, const double* Y, double U,
                                           double T, int max_iter, double rtol, bool& ok,
                                           double (&c)[4]) {
  mixture_energy_poly<M>(m, Y, c);
  return newton_poly(c, U, T, max_iter, rtol, ok);
}
template <int M>
__device__ __forceinline__ double newton_T(const DevMech& m, const double* Y, double U,
                                           double T, int max_iter, double rtol, bool& ok) {
  double c[4];
  return newton_T<M>(m, Y, U, T, max_iter, rtol, ok, c);
}

__device__ __forceinline__ double species_U(const DevMech& m, int a, double T) {
  return m.u0[a] + T * (m.u1[a] + T * (m.u2[a] + T * m.u3[a]));
}

// ------------------------------------------------------------------------
// The same temperature solve in float-float (mixed path).  The formulas are
// those of newton_T; the stopping rule uses max(rtol, 4e-13), the resolution
// of float-float sums of the formation-energy-sized terms.
__device__ __forceinline__ ff species_U_ff(const DevMech& m, int a, ff T) {
  return m.u0_f[a] + T * (m.u1_f[a] + T * (m.u2_f[a] + T * m.u3_f[a]));
}

__device__ __forceinline__ ff newton_poly(const ff (&c)[4], ff U, ff T, int max_iter,
                                          float rtol, bool& ok) {
  const ff d2(2.f * c[2].hi, 2.f * c[2].lo), d3 = ff(3.f) * c[3];
  const ff c0 = c[0] - U;
  ok = false;
  for (int it = 0; it < max_iter; ++it) {
    const ff F = c0 + T * (c[1] + T * (c[2] + T * c[3]));
    ff e = d2;
    ff_fma_acc(e, d3, T);
    ff dF = c[1];
    ff_fma_acc(dF, ff_norm(e), T);
    const ff dT = -ff_quotient(F, ff_norm(dF));
    T += dT;
    if (fabsf(dT.hi) <= rtol * fabsf(T.hi)) { ok = true; break; }
  }
  return T;
}

template <int M>
__device__ __forceinline__ ff newton_T_ff(const DevMech& m, const ff* Y, ff U, ff T,
                                          int max_iter, float rtol, bool& ok, ff (&c)[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) c[k] = ff();
#pragma unroll
  for (int a = 0; a < M; ++a) {
    ff_fma_acc(c[0], Y[a], m.u0_f[a]);
    ff_fma_acc(c[1], Y[a], m.u1_f[a]);
    ff_fma_acc(c[2], Y[a], m.u2_f[a]);
    ff_fma_acc(c[3], Y[a], m.u3_f[a]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) c[k] = ff_norm(c[k]);
  return newton_poly(c, U, T, max_iter, rtol, ok);
}

// The record's enthalpy polynomial from the energy polynomial c (J/kg) and
// sum Y_a/m_a: H_a = U_a + R_a T.
__device__ __forceinline__ void enthalpy_poly(const double (&c)[4], double Rm, const Units& un,
                                              double (&H)[4]) {
  H[0] = c[0] * un.inv_c2;
  H[1] = fma(Rm, R_U, c[1]) * un.inv_c2;
  H[2] = c[2] * un.inv_c2;
  H[3] = c[3] * un.inv_c2;
}
__device__ __forceinline__ void enthalpy_poly(const double (&c)[4], float Rm, const Units& un,
                                              float (&H)[4]) {
  H[0] = float(c[0] * un.inv_c2);
  H[1] = float((c[1] + double(Rm) * R_U) * un.inv_c2);
  H[2] = float(c[2] * un.inv_c2);
  H[3] = float(c[3] * un.inv_c2);
}
__device__ __forceinline__ void enthalpy_poly(const ff (&c)[4], float Rm, const Units& un,
                                              float (&H)[4]) {
  H[0] = (c[0] * un.inv_c2_f).hi;
  H[1] = ((c[1] + ff(Rm * float(R_U))) * un.inv_c2_f).hi;
  H[2] = (c[2] * un.inv_c2_f).hi;
  H[3] = (c[3] * un.inv_c2_f).hi;
}
// ln(T / T0)
__device__ __forceinline__ float ln_T0(float T) { return log(T * float(1.0 / T_REF)); }
__device__ __forceinline__ double ln_T0(double T) { return log_tang(T) - LN_T_REF; }
// q - u . P
template <int D, typename R, typename QT, typename PT>
__device__ __forceinline__ R flux_less_work(int d, const R (&u)[D], const QT& q, const PT& P) {
  R v = q[d];
#pragma unroll
  for (int b = 0; b < D; ++b)
    v = fma(-u[b], P[b == d ? b : (D == 3 ? (b + d == 1 ? 3 : (b + d == 2 ? 4 : 5)) : 2)], v);
  return v;
}

// ------------------------------------------------------------------------
// Chemistry: rates of progress and mass production rates (Sec. 2.4, Sec.
// 3.6), the temperature in CT: FP64 (the FP64 path, and FP32 storage with
// chem_fp64) or float-float.
//
// What bounds it is the arithmetic of two exponentials per reaction.  In
// FP64 the whole took ~42 FP64 instructions per reaction of 64 to 75 cycles
// each per SM quarter, in float-float ~410 FP32 instructions.  So (1) the
// logarithm of each rate constant is one sum over the basis (1, ln T, 1/T, T,
// T^2) with coefficients folded on the host, which replaces the species' Gibbs
// functions; (2) of FP64 temperatures these sums are taken in 64-bit fixed
// point, the exponentials and their products with the concentrations in 64-bit
// significands (Sig), and only a rate of progress becomes a double: FP64 is
// left with the third body and the sums over the reactions (~6 instructions per
// reaction), its range and rounding with all of it; (3) float-float sums stay
// unnormalised (ff_acc); (4) the third-body sums are formed once per distinct
// row of efficiencies.
template <typename CT> struct TBasis { CT lnT, invT, T, T2; };
// FP64: also in fixed point, in which a sum takes no FP64 instruction (and is
// exact to 2^-46; FP64's own rounding of it is up to 2^-40); usable for
// mechanisms and temperatures inside its range
template <> struct TBasis<double> {
  double lnT, invT, T, T2;
  long long q[5];
  bool fixed;
};

__device__ __forceinline__ TBasis<double> tbasis(const DevMech& m, double T) {
  TBasis<double> b;
  b.lnT = log_tang(T);
  b.invT = 1.0 / T;
  b.T = T;
  b.T2 = T * T;
  // 128 < T < 16384: at 128 K itself 1/T = 2^-7 is one past its kBitsInvT bits
  // (one bit fewer of it would leave the coefficients no room for activation
  // energies above 377 kJ/mol)
  const long long Tb = __double_as_longlong(T);
  b.fixed = m.fixed_args && Tb > 0x4060000000000000LL && Tb < 0x40d0000000000000LL;
  b.q[0] = 0;
  b.q[1] = fixed_of(b.lnT, kBitsLnT);
  b.q[2] = fixed_of(b.invT, kBitsInvT);
  b.q[3] = fixed_of(T, kBitsT);
  b.q[4] = fixed_of(b.T2, kBitsT2);
  return b;
}
__device__ __forceinline__ TBasis<ff> tbasis(const DevMech&, ff T) {
  return TBasis<ff>{ff_log(T), ff(1.f) / T, T, T * T};
}
// the rate constants
__device__ __forceinline__ Sig forward_constant(const DevReaction& x, const TBasis<double>& b) {
  if (b.fixed)
    return exp_sig(x.fq[0] + __mul64hi(x.fq[1], b.q[1]) + __mul64hi(x.fq[2], b.q[2]));
  return exp_sig(fma(x.f[2], b.invT, fma(x.f[1], b.lnT, x.f[0])));
}
__device__ __forceinline__ Sig reverse_constant(const DevReaction& x, const TBasis<double>& b) {
  if (b.fixed)
    return exp_sig(x.rq[0] + __mul64hi(x.rq[1], b.q[1]) + __mul64hi(x.rq[2], b.q[2]) +
                   __mul64hi(x.rq[3], b.q[3]) + __mul64hi(x.rq[4], b.q[4]));
  return exp_sig(fma(x.r[2], b.invT,
                     fma(x.r[1], b.lnT, fma(x.r[4], b.T2, fma(x.r[3], b.T, x.r[0])))));
}
__device__ __forceinline__ ExpArg forward_arg(const DevReaction& x, const TBasis<ff>& b) {
  ff s = x.f_f[0];
  ff_fma_acc(s, x.f_f[1], b.lnT);
  ff_fma_acc(s, x.f_f[2], b.invT);
  return exp_arg(ff_norm(s));
}
__device__ __forceinline__ ExpArg reverse_arg(const DevReaction& x, const TBasis<ff>& b) {
  ff s = x.r_f[0];
  ff_fma_acc(s, x.r_f[3], b.T);
  ff_fma_acc(s, x.r_f[4], b.T2);
  ff_fma_acc(s, x.r_f[1], b.lnT);
  ff_fma_acc(s, x.r_f[2], b.invT);
  return exp_arg(ff_norm(s));
}

// The arrays the reaction loop indexes by species (concentrations, molar
// rates) live in a per-thread slice of shared memory: a runtime index into a
// register array would put it in local memory.  ST: threads per block (or more),
// the stride of a slice's entries; kBytes: the block's slices.
constexpr int kChemThreads = 128;
template <int M, typename CT, int ST = kChemThreads> struct ChemSlice;
template <int M, int ST> struct ChemSlice<M, ff, ST> {
  static constexpr size_t kBytes = (size_t)2 * M * ST * sizeof(ff);
  ff* p;
  __device__ __forceinline__ ChemSlice(void* block, int t) : p(static_cast<ff*>(block) + t) {}
  __device__ __forceinline__ ff c(int a) const { return p[a * ST]; }
  __device__ __forceinline__ void set(int a, ff c) { p[a * ST] = c; }
  __device__ __forceinline__ void clear(int a) { p[(M + a) * ST] = ff(); }
  __device__ __forceinline__ void add(int a, ff q) { ff_acc(p[(M + a) * ST], q); }
  __device__ __forceinline__ ff sum(int a) const { return p[(M + a) * ST]; }   // unnormalised
  __device__ __forceinline__ ff rate(int a) const { return ff_norm(sum(a)); }
  __device__ __forceinline__ ff third_body(const DevMech& m, int row) const {
    ff s;
#pragma unroll
    for (int a = 0; a < M; ++a) ff_fma_acc(s, m.eff_f[row][a], c(a));
    return ff_norm(s);
  }
};
// FP64: the concentrations also as significand and exponent
template <int M, int ST> struct ChemSlice<M, double, ST> {
  static constexpr size_t kBytes = (size_t)M * ST * (3 * sizeof(double) + sizeof(int));
  double* p;      // C, W, then the significands
  int* e;
  __device__ __forceinline__ ChemSlice(void* block, int t)
      : p(static_cast<double*>(block) + t), e(static_cast<int*>(block) + 6 * M * ST + t) {}
  __device__ __forceinline__ double c(int a) const { return p[a * ST]; }
  __device__ __forceinline__ Sig sig(int a) const {
    return Sig{__double_as_longlong(p[(2 * M + a) * ST]), e[a * ST]};
  }
  __device__ __forceinline__ void set(int a, double c) {
    const Sig s = sig_of(c);
    p[a * ST] = c;
    p[(2 * M + a) * ST] = __longlong_as_double(s.m);
    e[a * ST] = s.e;
  }
  __device__ __forceinline__ void clear(int a) { p[(M + a) * ST] = 0.0; }
  __device__ __forceinline__ void add(int a, double q) { p[(M + a) * ST] += q; }
  __device__ __forceinline__ double sum(int a) const { return p[(M + a) * ST]; }
  __device__ __forceinline__ double rate(int a) const { return sum(a); }
  __device__ __forceinline__ double third_body(const DevMech& m, int row) const {
    double s = 0.0;
#pragma unroll
    for (int a = 0; a < M; ++a) s = fma(m.eff[row][a], c(a), s);
    return s;
  }
};

// Rate of progress of a reaction without its third body, from this thread's
// concentrations.
template <int M, int ST>
__device__ __forceinline__ double reaction_rate(const DevReaction& x, const TBasis<double>& b,
                                                const ChemSlice<M, double, ST>& s) {
  // both constants together: two chains in flight (an irreversible reaction's
  // reverse one goes unused)
  Sig q = forward_constant(x, b), rev = reverse_constant(x, b);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    if (j < x.nr) q = q * s.sig(x.reac[j]);
    if (j < x.np) rev = rev * s.sig(x.prod[j]);
  }
  return double_of_sig(x.reversible ? q - rev : q);
}
// Float-float: of a rate constant 2^e1 y, what FP32 holds of 2^e1 goes before the
// concentrations and the rest after them.
template <int M, int ST>
__device__ __forceinline__ ff scaled_product(const ExpArg& x, int n, const int* species,
                                             const ChemSlice<M, ff, ST>& s) {
  const int e = x.n >> 6, e1 = min(max(e, -100), 126);
  ff q = ff_scale(exp_frac(x), e1);
  for (int j = 0; j < n; ++j) q *= s.c(species[j]);
  return e == e1 ? q : ff_scale(q, e - e1);
}
template <int M, int ST>
__device__ __forceinline__ ff reaction_rate(const DevReaction& x, const TBasis<ff>& b,
                                            const ChemSlice<M, ff, ST>& s) {
  ff q = scaled_product(forward_arg(x, b), x.nr, x.reac, s);
  if (x.reversible) {
    ff_acc(q, -scaled_product(reverse_arg(x, b), x.np, x.prod, s));
    q = ff_norm(q);
  }
  return q;
}

// The reactions first, first + step, ... added to this thread's molar rates.
template <int M, typename CT, int ST>
__device__ __forceinline__ void add_reactions(const DevMech& m, const TBasis<CT>& b,
                                              ChemSlice<M, CT, ST>& s, int first, int step) {
  int row = -1;
  CT cm = CT();
  for (int k = first; k < m.R; k += step) {
    const DevReaction& x = m.rx[k];
    CT q = reaction_rate(x, b, s);
    if (x.third_body >= 0) {
      if (x.third_body != row) {
        row = x.third_body;
        cm = s.third_body(m, row);
      }
      q *= cm;
    }
    for (int j = 0; j < x.nr; ++j) s.add(x.reac[j], -q);
    for (int j = 0; j < x.np; ++j) s.add(x.prod[j], q);
  }
}

// Molar rates (mol/(m^3 s)) at T of the concentrations already in this
// thread's slice; the slice's rates are overwritten.
template <int M, typename CT, int ST>
__device__ __forceinline__ void molar_rates(const DevMech& m, CT T, ChemSlice<M, CT, ST>& s) {
#pragma unroll
  for (int a = 0; a < M; ++a) s.clear(a);
  add_reactions(m, tbasis(m, T), s, 0, 1);
}

// ------------------------------------------------------------------------
// Gaussian elimination without pivoting for A V = B with 3 right-hand sides,
// the matrix stored with entry (r, c) at A[(r M + c) st].
// A is strictly row diagonally dominant (diagonal 1 + sum of |off-diagonal|),
// so every pivot is at least 1.
template <int M, int D, typename R>
__device__ __forceinline__ void solve_dd_strided(R* A, int st, R (&B)[M][D]) {
#pragma unroll
  for (int k = 0; k < M; ++k) {
    const R inv = R(1) / A[(k * M + k) * st];
#pragma unroll
    for (int r = k + 1; r < M; ++r) {
      const R f = A[(r * M + k) * st] * inv;
#pragma unroll
      for (int c = k + 1; c < M; ++c) A[(r * M + c) * st] -= f * A[(k * M + c) * st];
#pragma unroll
      for (int d = 0; d < D; ++d) B[r][d] -= f * B[k][d];
    }
  }
#pragma unroll
  for (int k = M - 1; k >= 0; --k) {
    const R inv = R(1) / A[(k * M + k) * st];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      R s = B[k][d];
#pragma unroll
      for (int c = k + 1; c < M; ++c) s -= A[(k * M + c) * st] * B[c][d];
      B[k][d] = s * inv;
    }
  }
}

// The same in float-float (the FP64 path's diffusion velocities, which enter
// the collision only through corrections a thousand times below what they
// correct: 48 bits of a correction are beyond FP64's rounding of the sum.  In
// FP64 the elimination took ~800 instructions of 64 cycles), the right-hand
// sides in the matrix's columns M .. M + D - 1 (rows of M + D entries); they
// become the solution.  The loop over the rows below the pivot is rolled:
// unrolled, the code (a dozen instructions per update) outgrows the
// instruction cache, and fetching it took half of the time.
template <int M, int D>
__device__ __forceinline__ void solve_dd_ff(ff* A, int st) {
  constexpr int W = M + D;
#pragma unroll
  for (int k = 0; k < M; ++k) {
    const ff inv = ff_rcp(A[(k * W + k) * st]);
    A[(k * W + k) * st] = inv;
    ff piv[W];
#pragma unroll
    for (int c = k + 1; c < W; ++c) piv[c] = A[(k * W + c) * st];
#pragma unroll 1
    for (int r = k + 1; r < M; ++r) {
      ff* const row = A + r * W * st;
      const ff f = -(row[k * st] * inv);
#pragma unroll
      for (int c = k + 1; c < W; ++c) {
        ff v = row[c * st];
        ff_fma_acc(v, f, piv[c]);
        row[c * st] = ff_norm(v);
      }
    }
  }
#pragma unroll 1
  for (int d = 0; d < D; ++d) {
    ff x[M];
#pragma unroll
    for (int k = M - 1; k >= 0; --k) {
      ff s = A[(k * W + M + d) * st];
#pragma unroll
      for (int c = k + 1; c < M; ++c) ff_fma_acc(s, -A[(k * W + c) * st], x[c]);
      x[k] = ff_norm(s) * A[(k * W + k) * st];
      A[(k * W + M + d) * st] = x[k];
    }
  }
}

}  // namespace lbm
