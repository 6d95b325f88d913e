// Kernels of the reactive-mixture LBM step (templates; instantiated per
// lattice, species count and precision by lbm_inst.cu).
//
//   k_bnode     one thread per interface node: gather, bounce-back / TMS /
//               inlet / LODI outlet reconstruction, the node's moment record
//               (lbm_bnode.cuh).
//   k_bnode_warp  the same and the node's reaction sub-steps with one warp per
//               interface node (few of them).
//   k_iface_chem, k_chem  the interface nodes' reaction sub-steps after k_bnode
//               (a thread or eight lanes per node).
//   k_moments   one thread per bulk node: pull-stream all lattices, moments,
//               temperature Newton, the reaction sub-steps, the moment
//               record (scratch) and the T guess.
//   k_mchem     the same with a group of lanes per node (small grids).
//   k_collide   gradients from neighbour records, relaxation parameters,
//               diffusion velocities, collision of all lattices on a second
//               pull gather, store to the other buffer (fused collision).
//   k_prep, k_coll  the same collision split into a per-node parameter
//               kernel and a nine-threads-per-node direction kernel.
//   k_*_batch   the same bodies over the tiles of several handles.
//   k_step_persist  a whole batched step as one launch over a work-list.
//   k_init      populations at the equilibria of given fields.
//   k_out       fields of the stored state (SI units).
//   k_diag      per-node heat release and flame diagnostics.
//
// Template parameters: D (2 or 3), M (species), S (storage type), RT (type
// of the lattice arithmetic: moments, equilibria, collision).  FP64 storage
// computes to FP64 rounding; what can runs beside the FP64 pipe (population sums
// in fixed point, rates, diffusion velocities and the Stefan-Maxwell term in
// float-float).  FP32 and FP16 storage compute the lattice
// arithmetic and transport in FP32 and the temperature Newton solve and the
// chemistry in float-float (ff.cuh) or, with LBM_CHEM64, in FP64.
#include <atomic>
#include <climits>
#include <cmath>
#include <type_traits>

#pragma once

#include "lbm_device.cuh"
#include "lbm_sync.cuh"

// Chemistry mode of the mixed path in this translation unit: with FP32
// lattice arithmetic, the temperature Newton solve and the reaction
// chemistry run in float-float (LBM_CHEM64 = 0) or as in the FP64 path
// (LBM_CHEM64 = 1).  The two modes' templates live in distinct inline
// namespaces, so both can be instantiated in one library.
#ifndef LBM_CHEM64
#define LBM_CHEM64 0
#endif

namespace lbm {
#if LBM_CHEM64
inline namespace chem64 {
#else
inline namespace chemff {
#endif

// float-float Newton and chemistry: FP32 lattice arithmetic, float-float mode
template <typename RT> constexpr bool kFF = sizeof(RT) == 4 && !LBM_CHEM64;
template <typename RT> struct ChemType { using type = double; };
template <> struct ChemType<float> { using type = std::conditional_t<LBM_CHEM64 != 0, double, ff>; };
// resident blocks per SM the moments kernels are compiled for (register cap):
// four (128 registers, FP64 spills 340 bytes): with three (168) ten FP64 steps of
// the 600x40x40 tube took 63.7 ms against 60.9, a 61x37x29 box 13.5 against 10.7, an
// uneven FP32 batch 43.6 against 40.2
constexpr int kMomentsMinBlocks = 4;
// ... of the single-domain kernel with float-float chemistry five: 24 steps of
// the tube 45.4 against 44.3 ms; the batch kernel, which holds its domain's
// descriptor as well, four (uneven FP32 batch 39.7 against 41.0 with five)
template <typename RT> constexpr int kMoments1MinBlocks = kFF<RT> ? 5 : kMomentsMinBlocks;
// Blocks per SM that k_prep's registers are held to.  FP32 (latency of the
// gradients' loads and of the elimination): four, 128 registers; with three, as
// the compiler chose, 600x40x40 tube 47.5 against 45.4 ms per 24 steps, uneven
// FP32 batch 43.0 against 39.7.  FP64: two, by its shared memory (110 KB).
template <typename RT> constexpr int kPrepMinBlocks = sizeof(RT) == 4 ? 4 : 2;

// Arithmetic type of a storage type: FP16 storage computes in FP32.
template <typename S> struct ComputeType { using type = S; };
template <> struct ComputeType<__half> { using type = float; };

// Stored-population codec.  FP64 and FP32 storage hold the value itself.
// FP16 storage holds offsets (reading R19): h = (f - o_li) / s_l, o_li the
// equilibrium population at the mean initial state and s_l a per-lattice
// scale, both fixed by lbm_init_fields (codec entry li = {o, s, 1/s, 0}).
template <typename S> struct Codec {
  template <typename R>
  __device__ static R dec(S v, const float4*, int) { return R(v); }
  template <typename R>
  __device__ static S enc(R v, const float4*, int) { return S(v); }
};
template <> struct Codec<__half> {
  template <typename R>
  __device__ static R dec(__half v, const float4* t, int li) {
    const float4 c = __ldg(t + li);
    return R(fmaf(c.y, __half2float(v), c.x));
  }
  template <typename R>
  __device__ static __half enc(R v, const float4* t, int li) {
    const float4 c = __ldg(t + li);
    return __float2half_rn((float(v) - c.x) * c.z);
  }
};

__device__ __forceinline__ int wrap1(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

template <int D>
__device__ __forceinline__ long long node_shift(int x, int y, int z, int i, int sgn,
                                                const Geom& g) {
  const int sx = wrap1(x + sgn * cvel(i, 0), g.nx);
  const int sy = wrap1(y + sgn * cvel(i, 1), g.ny);
  const int sz = D == 3 ? wrap1(z + sgn * cvel(i, 2), g.nz) : 0;
  return sx + (long long)g.nx * (sy + (long long)g.ny * sz);
}

// Population (lattice l, direction i) entering node n's collision: the
// reconstructed value for interface nodes (tag >= 0), else the streamed one.
template <typename RT, typename S>
__device__ __forceinline__ RT pop_in(const S* __restrict__ src, const BCDev& bc, int tag,
                                     long long N, long long sn, int li, const float4* codec) {
  return tag >= 0 ? static_cast<const RT*>(bc.pops)[(long long)li * bc.n_if + tag]
                  : Codec<S>::template dec<RT>(__ldg(src + (long long)li * N + sn), codec, li);
}

// 1/tau_ab = s * K_ab: the coefficient table in the lattice compute type
template <typename RT> __device__ __forceinline__ RT kcoef(const DevMech& m, int a, int b);
template <> __device__ __forceinline__ double kcoef<double>(const DevMech& m, int a, int b) {
  return m.K[a][b];
}
template <> __device__ __forceinline__ float kcoef<float>(const DevMech& m, int a, int b) {
  return m.Kf[a][b];
}

// threads per block of the node kernels (the shared-memory columns use it)
constexpr int kBS = 128;
static_assert(kBS == kChemThreads, "the chemistry's shared-memory slices assume kBS threads");

// shared-memory entries per thread of the diffusion-velocity solve: the
// matrix, in FP64 (float-float pairs) with the right-hand sides
template <int D, int M, typename RT> constexpr int solve_smem_entries() {
  return sizeof(RT) == 8 ? M * (M + D) : M * M;
}

// shared memory of the collision kernel per thread: the diffusion-velocity
// matrix, then the axis-factor tables (FP32: every axis; FP64 in 3D: the y
// and z axes, the whole table would halve the occupancy)
template <int D, int M, typename RT> constexpr int collide_smem_entries() {
  constexpr int tab = sizeof(RT) == 4 ? 2 * M * D * 3 : (D == 3 ? 2 * M * 2 * 3 : 0);
  constexpr int solve = solve_smem_entries<D, M, RT>();
  return tab > solve ? tab : solve;
}

template <int D>
__device__ __forceinline__ constexpr int pidx(int a, int b) {
  return a == b ? a : (D == 3 ? (a + b == 1 ? 3 : (a + b == 2 ? 4 : 5)) : 2);
}

// ---------------------------------------------------------------------------
// Reaction sub-steps of one node by one thread at frozen internal energy
// (Sec. 2.4 Eq. R3): rs the post-stream species densities (the slaved one
// included), rho, ER = E / rho and usqR = |u|^2 of the moments, T_0 = T
// their temperature; dr receives the increments drho_a (a < M - 1).  The
// temperature solve in float-float (mixed path) or FP64; the rate arrays live
// in the thread's slice of shared memory (chem_slice: the block's slices).
// Blocks of at most kChemThreads threads.
template <int M, typename CT, int ST = kChemThreads>
__device__ __forceinline__ void* chem_static_slice() {
  __shared__ __align__(8) unsigned char chem_raw[ChemSlice<M, CT, ST>::kBytes];
  return chem_raw;
}

template <int M, typename RT>
__device__ __forceinline__ void node_substeps(const RT (&rs)[M], RT rho, RT ER, RT usqR,
                                              double T, const Units& un, const DevMech& mech,
                                              int* __restrict__ status, void* chem_slice,
                                              RT (&dr)[M - 1]) {
  ChemSlice<M, typename ChemType<RT>::type> cs(chem_slice, threadIdx.x);
  if constexpr (kFF<RT>) {
    const ff Uphys = (ff(ER) + ff(-0.5f * usqR)) * un.c2_f;
    ff r[M];
#pragma unroll
    for (int a = 0; a < M; ++a) r[a] = ff(rs[a]);
    ff Ts = ff_from_double(T);
    const ff rho_f(rho);
    for (int s = 0; s < un.substeps; ++s) {
      if (s > 0) {
        ff Ys[M];
#pragma unroll
        for (int a = 0; a < M; ++a) Ys[a] = r[a] / rho_f;
        bool oks;
        ff c[4];
        Ts = newton_T_ff<M>(mech, Ys, Uphys, Ts, un.newton_max_iter, un.newton_rtol_f, oks, c);
        if (!oks) atomicOr(status, ST_NEWTON);
      }
#pragma unroll
      for (int a = 0; a < M; ++a) cs.set(a, r[a] * mech.inv_mm_f[a]);
      molar_rates(mech, Ts, cs);
#pragma unroll
      for (int a = 0; a < M; ++a) r[a] += un.dt_sub_f * (cs.rate(a) * mech.mm_f[a]);
    }
#pragma unroll
    for (int a = 0; a < M - 1; ++a) dr[a] = (r[a] - ff(rs[a])).hi;
  } else {
    const double Uphys = (double(ER) - 0.5 * double(usqR)) * un.c * un.c;
    const double dtr = un.dt_sub, ir = 1.0 / double(rho);
    double r[M];
#pragma unroll
    for (int a = 0; a < M; ++a) r[a] = double(rs[a]);
    double Ts = T;
    for (int s = 0; s < un.substeps; ++s) {
      if (s > 0) {
        double Ys[M];
#pragma unroll
        for (int a = 0; a < M; ++a) Ys[a] = r[a] * ir;
        bool oks;
        Ts = newton_T<M>(mech, Ys, Uphys, Ts, un.newton_max_iter, un.newton_rtol, oks);
        if (!oks) atomicOr(status, ST_NEWTON);
      }
#pragma unroll
      for (int a = 0; a < M; ++a) cs.set(a, r[a] * mech.inv_mm[a]);
      molar_rates(mech, Ts, cs);
#pragma unroll
      for (int a = 0; a < M; ++a) r[a] = fma(cs.rate(a), dtr * mech.mm[a], r[a]);
    }
#pragma unroll
    for (int a = 0; a < M - 1; ++a) dr[a] = RT(r[a] - double(rs[a]));
  }
}

// ---------------------------------------------------------------------------
// Reaction sub-steps with several lanes per node (Sec. 2.4 Eq. R3), for
// grids too small to fill the GPU at one thread per node: the node's
// reactions are dealt out over the lanes, which cuts the latency of a node's
// chemistry by about the lane count.  The formulas are those of node_substeps;
// only the production rates are summed in another order (partial sums per
// lane), so the placements agree to rounding.  CT: double (FP64 path) or
// float-float (mixed path).
__device__ __forceinline__ double shfl_xor_ct(unsigned mask, double v, int o) {
  return __shfl_xor_sync(mask, v, o);
}
__device__ __forceinline__ ff shfl_xor_ct(unsigned mask, ff v, int o) {
  return ff(__shfl_xor_sync(mask, v.hi, o), __shfl_xor_sync(mask, v.lo, o));
}

template <typename CT> struct Chem;
template <> struct Chem<double> {
  __device__ static double inv(double x) { return 1.0 / x; }
  __device__ static double of(double v) { return v; }
  __device__ static double of_T(double T) { return T; }
  __device__ static double of_ff(ff v) { return double_of_ff(v); }
  __device__ static double concentration(const DevMech& m, int a, double r) {
    return r * m.inv_mm[a];
  }
  __device__ static double increment(const DevMech& m, const Units& u, int a, double w) {
    return w * (u.dt_sub * m.mm[a]);
  }
  // sum over the group, the same in every lane: significands shifted to the
  // largest exponent and added in integers (a butterfly of FP64 additions would
  // occupy the FP64 pipe for 75 cycles per stage)
  template <int L> __device__ __forceinline__ static double group_sum(double v, unsigned gmask) {
    constexpr int G = L == 32 ? 6 : (L == 8 ? 4 : 3);       // log2 L and the sign
    const Sig s = sig_of(v);
    int e = s.m == 0 ? -(1 << 16) : s.e;
#pragma unroll
    for (int o = 1; o < L; o <<= 1) e = max(e, __shfl_xor_sync(gmask, e, o));
    long long m = s.m >> min(e - s.e + G, 63);
#pragma unroll
    for (int o = 1; o < L; o <<= 1) m += __shfl_xor_sync(gmask, m, o);
    return e >= kSigNaN / 2 ? __longlong_as_double(0x7ff8000000000000LL)
                            : double_of_sig(Sig{m, e + G});
  }
  __device__ static double ucoef(const DevMech& m, int k, int a) {
    return k == 0 ? m.u0[a] : (k == 1 ? m.u1[a] : (k == 2 ? m.u2[a] : m.u3[a]));
  }
  __device__ static double rtol(const Units& u) { return u.newton_rtol; }
};
template <> struct Chem<ff> {
  __device__ static ff inv(ff x) { return ff(1.f) / x; }
  __device__ static ff of(float v) { return ff(v); }
  __device__ static ff of_T(double T) { return ff_from_double(T); }
  __device__ static ff of_ff(ff v) { return v; }
  __device__ static ff concentration(const DevMech& m, int a, ff r) { return r * m.inv_mm_f[a]; }
  __device__ static ff increment(const DevMech& m, const Units& u, int a, ff w) {
    return u.dt_sub_f * (ff_norm(w) * m.mm_f[a]);
  }
  // (unnormalised)
  template <int L> __device__ __forceinline__ static ff group_sum(ff v, unsigned gmask) {
#pragma unroll
    for (int o = 1; o < L; o <<= 1) ff_acc(v, shfl_xor_ct(gmask, v, o));
    return v;
  }
  __device__ static ff ucoef(const DevMech& m, int k, int a) {
    return k == 0 ? m.u0_f[a] : (k == 1 ? m.u1_f[a] : (k == 2 ? m.u2_f[a] : m.u3_f[a]));
  }
  __device__ static float rtol(const Units& u) { return u.newton_rtol_f; }
};

// Register r[a] for a lane-dependent species index a (a select per species:
// a runtime index into a register array would put it in local memory).
template <int M, typename CT>
__device__ __forceinline__ CT pick(const CT (&r)[M], int a) {
  CT v = r[0];
#pragma unroll
  for (int b = 1; b < M; ++b)
    if (b == a) v = r[b];
  return v;
}

// Temperature Newton on Eq. temperature for a lane group (the formulas of
// newton_T / newton_T_ff): lane `sub` sums the mixture energy polynomial's
// coefficients over the species a = sub, sub + L, ..., the group adds them
// with a butterfly (every lane ends with the same sums, so every lane takes
// the same iterates), and every lane iterates.
template <int M, int L, typename CT>
__device__ __forceinline__ CT group_newton(const DevMech& m, const CT (&r)[M], CT irho, CT U,
                                           CT T, const Units& un, int sub, unsigned gmask,
                                           bool& ok, CT (&c)[4]) {
  using X = Chem<CT>;
#pragma unroll
  for (int k = 0; k < 4; ++k) c[k] = CT();
#pragma unroll
  for (int j = 0; j < (M + L - 1) / L; ++j) {
    const int a = sub + j * L;
    if (a < M) {
      const CT Ya = pick<M, CT>(r, a) * irho;
#pragma unroll
      for (int k = 0; k < 4; ++k) c[k] += Ya * X::ucoef(m, k, a);
    }
  }
#pragma unroll
  for (int o = 1; o < L; o <<= 1)
#pragma unroll
    for (int k = 0; k < 4; ++k) c[k] += shfl_xor_ct(gmask, c[k], o);
  return newton_poly(c, U, T, un.newton_max_iter, X::rtol(un), ok);
}

// The reaction sub-steps of one node by its lane group (Sec. 2.4 Eq. R3),
// from the post-stream species densities r (replaced by the densities after
// the sub-steps), 1/rho, the internal energy U and the temperature T_0 of
// the moments.  cs: this thread's slice for concentrations and rates.
template <int M, typename CT, int L, int ST>
__device__ __forceinline__ void chem_group_substeps(CT (&r)[M], const CT irho, const CT U,
                                                    CT Ts, const Units& un, const DevMech& m,
                                                    int sub, unsigned gmask,
                                                    int* __restrict__ status,
                                                    ChemSlice<M, CT, ST>& cs) {
  using X = Chem<CT>;
  for (int s = 0; s < un.substeps; ++s) {
    if (s > 0) {
      bool ok;
      CT c[4];
      Ts = group_newton<M, L, CT>(m, r, irho, U, Ts, un, sub, gmask, ok, c);
      if (!ok && sub == 0) atomicOr(status, ST_NEWTON);
    }
#pragma unroll
    for (int a = 0; a < M; ++a) {
      cs.set(a, X::concentration(m, a, r[a]));
      cs.clear(a);
    }
    add_reactions(m, tbasis(m, Ts), cs, sub, L);
    // the group's sums: every lane ends with the same total
#pragma unroll
    for (int a = 0; a < M; ++a)
      r[a] += X::increment(m, un, a, X::template group_sum<L>(cs.sum(a), gmask));
  }
}

// Reaction sub-steps of node n by a group of L lanes (L = 4 or 8, aligned
// within the warp): every lane forms the node's state, temperature and
// concentrations; lane `sub` takes the reactions
// k = sub, sub + L, ...; the species production rates are summed across the
// group with shuffles, after which every lane holds the same densities.
template <int D, int M, typename RT, int L>
__device__ __forceinline__ void chem_lanes_body(RT* __restrict__ rec,
                                                const double* __restrict__ Tf,
                                                int* __restrict__ status, long long N,
                                                const Units& un, const DevMech& m,
                                                long long n, int sub, unsigned gmask) {
  using CT = typename ChemType<RT>::type;
  using X = Chem<CT>;
  using RC = Rec<D, M>;
  const RT rho = rec[RC::RHO * N + n];
  RT usq = RT(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const RT ud = rec[(RC::U + d) * N + n];
    usq += ud * ud;
  }
  const RT ER = rec[RC::E * N + n];
  CT U;
  if constexpr (kFF<RT>) U = (ff(ER) + ff(-0.5f * usq)) * un.c2_f;
  else U = (double(ER) - 0.5 * double(usq)) * un.c * un.c;
  // the post-stream species densities the moments kernel left in the
  // increment slots; the slaved species from the mixture density
  CT r[M], r0[M - 1];
  RT last = rho;
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    const RT v = rec[(RC::DRHO + a) * N + n];
    last -= v;
    r0[a] = X::of(v);
    r[a] = r0[a];
  }
  r[M - 1] = X::of(last);
  ChemSlice<M, CT> cs(chem_static_slice<M, CT>(), threadIdx.x);
  chem_group_substeps<M, CT, L>(r, X::inv(X::of(rho)), U, X::of_T(Tf[n]), un, m, sub, gmask,
                                status, cs);
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    if (a % L != sub) continue;
    if constexpr (kFF<RT>) rec[(RC::DRHO + a) * N + n] = (r[a] - r0[a]).hi;
    else rec[(RC::DRHO + a) * N + n] = RT(r[a] - r0[a]);
  }
}

// Moments and reaction sub-steps of node n by a group of L lanes (grids too
// small to fill the GPU at one thread per node; chem_lanes = L).  Lane `sub`
// pulls the directions sub, sub + L, ... of every lattice, the group adds the
// partial sums with a butterfly, every lane forms the node's fields (the
// formulas of moments_body), the temperature solve is shared as in
// group_newton, the lanes split the record's stores, and the group runs the
// sub-steps from the post-stream densities (chem_group_substeps).  m: the
// mechanism for compile-time indices; mg: its global copy, indexed by lane.
template <int D, int M, typename S, typename RT, int L>
__device__ __forceinline__ void mchem_body(const S* __restrict__ src, RT* __restrict__ rec,
                                           double* __restrict__ Tf, int* __restrict__ status,
                                           const Geom& g, const Units& un, const BCDev& bc,
                                           const DevMech& m, const DevMech& mg, long long n,
                                           int tag, int sub, unsigned gmask) {
  constexpr int Q = Lat<D>::Q, NP = Lat<D>::NP;
  using RC = Rec<D, M>;
  using CT = typename ChemType<RT>::type;
  using X = Chem<CT>;
  const long long N = g.N;
  const int x = (int)(n % g.nx);
  const int y = (int)((n / g.nx) % g.ny);
  const int z = (int)(n / ((long long)g.nx * g.ny));
  RT rho = RT(0), rhoE = RT(0), j[D], q[D], P[NP], rs[M], js[M][D];
#pragma unroll
  for (int d = 0; d < D; ++d) { j[d] = RT(0); q[d] = RT(0); }
#pragma unroll
  for (int k = 0; k < NP; ++k) P[k] = RT(0);
#pragma unroll
  for (int a = 0; a < M; ++a) {
    rs[a] = RT(0);
#pragma unroll
    for (int d = 0; d < D; ++d) js[a][d] = RT(0);
  }
#pragma unroll
  for (int jd = 0; jd < (Q + L - 1) / L; ++jd) {
    const int i = sub + jd * L;
    if (i < Q) {
      RT c[D];
#pragma unroll
      for (int d = 0; d < D; ++d) c[d] = RT(cvel(i, d));
      const long long sn = node_shift<D>(x, y, z, i, -1, g);
#pragma unroll
      for (int a = 0; a < M - 1; ++a) {
        const RT v = pop_in<RT>(src, bc, tag, N, sn, a * Q + i, g.codec);
        rs[a] += v;
#pragma unroll
        for (int d = 0; d < D; ++d) js[a][d] += c[d] * v;
      }
      const RT f = pop_in<RT>(src, bc, tag, N, sn, (M - 1) * Q + i, g.codec);
      rho += f;
#pragma unroll
      for (int d = 0; d < D; ++d) {
        j[d] += c[d] * f;
#pragma unroll
        for (int e = d; e < D; ++e) P[pidx<D>(d, e)] += c[d] * c[e] * f;
      }
      const RT gv = pop_in<RT>(src, bc, tag, N, sn, M * Q + i, g.codec);
      rhoE += gv;
#pragma unroll
      for (int d = 0; d < D; ++d) q[d] += c[d] * gv;
    }
  }
#pragma unroll
  for (int o = 1; o < L; o <<= 1) {
    rho += __shfl_xor_sync(gmask, rho, o);
    rhoE += __shfl_xor_sync(gmask, rhoE, o);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      j[d] += __shfl_xor_sync(gmask, j[d], o);
      q[d] += __shfl_xor_sync(gmask, q[d], o);
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) P[k] += __shfl_xor_sync(gmask, P[k], o);
#pragma unroll
    for (int a = 0; a < M - 1; ++a) {
      rs[a] += __shfl_xor_sync(gmask, rs[a], o);
#pragma unroll
      for (int d = 0; d < D; ++d) js[a][d] += __shfl_xor_sync(gmask, js[a][d], o);
    }
  }
  // slaved species M (Eq. strongest)
  rs[M - 1] = rho;
#pragma unroll
  for (int d = 0; d < D; ++d) js[M - 1][d] = j[d];
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    rs[M - 1] -= rs[a];
#pragma unroll
    for (int d = 0; d < D; ++d) js[M - 1][d] -= js[a][d];
  }
  const RT inv_rho = RT(1) / rho;
  RT uR[D], YR[M], usqR = RT(0);
#pragma unroll
  for (int d = 0; d < D; ++d) { uR[d] = j[d] * inv_rho; usqR += uR[d] * uR[d]; }
#pragma unroll
  for (int a = 0; a < M; ++a) YR[a] = rs[a] * inv_rho;
  const RT ER = rhoE * inv_rho;
  // temperature (Eq. temperature) from the node's previous T, shared solve
  CT U, r[M];
  if constexpr (kFF<RT>) U = (ff(ER) + ff(-0.5f * usqR)) * un.c2_f;
  else U = (double(ER) - 0.5 * double(usqR)) * un.c * un.c;
#pragma unroll
  for (int a = 0; a < M; ++a) r[a] = X::of(rs[a]);
  const CT irho = X::inv(X::of(rho));
  bool ok;
  CT c[4];
  const CT Tx = group_newton<M, L, CT>(mg, r, irho, U, X::of_T(Tf[n]), un, sub, gmask, ok, c);
  double T;
  RT thR, H[4];
  if constexpr (sizeof(RT) == 4) {
    float Rm = 0.f;
#pragma unroll
    for (int a = 0; a < M; ++a) Rm += YR[a] * m.inv_mm_s[a];
    if constexpr (kFF<RT>) T = ff_to_double(Tx);
    else T = Tx;
    thR = Rm * float(R_U) * float(T) * un.inv_c2_s;
    enthalpy_poly(c, Rm, un, H);
  } else {
    double Rm = 0.0;
#pragma unroll
    for (int a = 0; a < M; ++a) Rm += YR[a] * m.inv_mm[a];
    T = Tx;
    thR = RT(Rm * R_U * T * un.inv_c2);
    enthalpy_poly(c, Rm, un, H);
  }
  if (sub == 0) {
    if (!ok) atomicOr(status, ST_NEWTON);
    if (!(rho > RT(0)) || !isfinite(double(rho)) || !isfinite(T)) atomicOr(status, ST_NONFINITE);
    Tf[n] = T;
  }
  // the record's fields, each stored by one lane of the group
  auto put = [&](int f, RT v) {
    if (f % L == sub) rec[(long long)f * N + n] = v;
  };
  put(RC::RHO, rho);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    put(RC::U + d, uR[d]);
    put(RC::Z + d, flux_less_work<D, RT>(d, uR, q, P));
    put(RC::PHI + d, rho * uR[d] * (RT(1) - RT(3) * thR) - rho * uR[d] * uR[d] * uR[d]);
  }
  put(RC::E, ER);
  put(RC::TH, thR);
  put(RC::LNT, ln_T0(RT(T)));
#pragma unroll
  for (int k = 0; k < 4; ++k) put(RC::H + k, H[k]);
#pragma unroll
  for (int a = 0; a < M; ++a) {
    put(RC::Y + a, YR[a]);
    const bool tiny = species_velocity_undefined<D, RT>(rs[a], js[a]);
#pragma unroll
    for (int d = 0; d < D; ++d)
      put(RC::US + a * D + d, record_us(tiny ? RT(0) : js[a][d] / rs[a] - uR[d]));
  }
  // reaction sub-steps at frozen U (Sec. 2.4 Eq. R3), T_0 the T just solved
  CT r0[M - 1];
#pragma unroll
  for (int a = 0; a < M - 1; ++a) r0[a] = r[a];
  ChemSlice<M, CT> cs(chem_static_slice<M, CT>(), threadIdx.x);
  chem_group_substeps<M, CT, L>(r, irho, U, X::of_T(T), un, mg, sub, gmask, status, cs);
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    if constexpr (kFF<RT>) put(RC::DRHO + a, (r[a] - r0[a]).hi);
    else put(RC::DRHO + a, RT(r[a] - r0[a]));
  }
}

// ---------------------------------------------------------------------------
// Shared memory of the moments kernels: per thread the chemistry's slice and
// the sums of its rates over the sub-steps.
template <int M, typename RT> constexpr size_t moments_bytes() {
  return ChemSlice<M, typename ChemType<RT>::type>::kBytes +
         (size_t)M * kChemThreads * sizeof(double);
}
template <int M, typename RT>
__device__ __forceinline__ void* moments_static() {
  __shared__ __align__(16) unsigned char mom_raw[moments_bytes<M, RT>()];
  return mom_raw;
}

// Sums over a lattice's 27 (9) populations: density, momentum, momentum flux.
// FP32: plain sums, row by row and plane by plane; FP64: fixed point.
template <typename RT> struct SumType { using type = RT; };
template <> struct SumType<double> { using type = Fix; };
__device__ __forceinline__ float sum_of(float v, int) { return v; }
__device__ __forceinline__ Fix sum_of(double v, int e) { return fix_of(v, e); }

template <int D, typename RT>
__device__ __forceinline__ void lattice_sums(const RT (&v)[Lat<D>::Q], int e,
                                             typename SumType<RT>::type& sum,
                                             typename SumType<RT>::type (&sj)[D],
                                             typename SumType<RT>::type (&sP)[Lat<D>::NP]) {
  using ST = typename SumType<RT>::type;
  constexpr int NZ = Lat<D>::Q / 9;
  sum = ST();
#pragma unroll
  for (int d = 0; d < D; ++d) sj[d] = ST();
#pragma unroll
  for (int k = 0; k < Lat<D>::NP; ++k) sP[k] = ST();
#pragma unroll
  for (int pz = 0; pz < NZ; ++pz) {
    ST ps = ST(), pd = ST(), py = ST(), pxy = ST();
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int i = 9 * pz + 3 * r;
      const ST f0 = sum_of(v[i], e), f1 = sum_of(v[i + 1], e), f2 = sum_of(v[i + 2], e);
      const ST sx = f0 + f2, sr = sx + f1, dx = f2 - f0;
      ps = ps + sr;
      pd = pd + dx;
      sP[pidx<D>(0, 0)] = sP[pidx<D>(0, 0)] + sx;
      if (r != 1) {
        py = r == 2 ? py + sr : py - sr;
        pxy = r == 2 ? pxy + dx : pxy - dx;
        sP[pidx<D>(1, 1)] = sP[pidx<D>(1, 1)] + sr;
      }
    }
    sum = sum + ps;
    sj[0] = sj[0] + pd;
    sj[1] = sj[1] + py;
    sP[pidx<D>(0, 1)] = sP[pidx<D>(0, 1)] + pxy;
    if constexpr (D == 3) {
      if (pz != 1) {
        sj[2] = pz == 2 ? sj[2] + ps : sj[2] - ps;
        sP[pidx<D>(2, 2)] = sP[pidx<D>(2, 2)] + ps;
        sP[pidx<D>(0, 2)] = pz == 2 ? sP[pidx<D>(0, 2)] + pd : sP[pidx<D>(0, 2)] - pd;
        sP[pidx<D>(1, 2)] = pz == 2 ? sP[pidx<D>(1, 2)] + py : sP[pidx<D>(1, 2)] - py;
      }
    }
  }
}

// The slaved species' sums: the f lattice's less the other species' (Eq.
// strongest).  FP64: in fixed point at exponent eR (momenta: eR - 6); ex: sums
// that do not fit there (beyond any physical state).
template <int D, typename RT> struct Remainder {
  RT v[1 + D];
  __device__ Remainder() {
#pragma unroll
    for (int d = 0; d <= D; ++d) v[d] = RT(0);
  }
  __device__ __forceinline__ void start(int) {}
  __device__ __forceinline__ void add(int d, RT, RT value, bool first) {
    v[d] = first ? value : v[d] - value;
  }
  __device__ __forceinline__ RT get(int d) const { return v[d]; }
};
template <int D> struct Remainder<D, double> {
  long long rem[1 + D];
  double ex[1 + D];
  int eR;
  __device__ Remainder() : eR(0) {
#pragma unroll
    for (int d = 0; d <= D; ++d) { rem[d] = 0; ex[d] = 0.0; }
  }
  __device__ __forceinline__ void start(int e) { eR = e + 2; }
  __device__ __forceinline__ void add(int d, FixSum t, double value, bool first) {
    const int to = d == 0 ? eR : eR - 6;
    if (t.e <= to) {
      const long long r = fix_down(t.s, to - t.e);
      rem[d] += first ? r : -r;
    } else {
      ex[d] += first ? value : -value;
    }
  }
  __device__ __forceinline__ double get(int d) const {
    const double r = double_of_fix(rem[d], d == 0 ? eR : eR - 6);
    return ex[d] != 0.0 ? r + ex[d] : r;
  }
};
__device__ __forceinline__ float sum_value(float s) { return s; }
__device__ __forceinline__ double sum_value(FixSum s) { return double_of_fix(s); }
__device__ __forceinline__ float close_sum(float s, int) { return s; }
__device__ __forceinline__ FixSum close_sum(Fix s, int e) { return fix_sum(s, e); }

// (j_a - rho_a u) / rho_a where u_a is defined (reading R5), else 0, as the
// record holds it.  FP64: the quotient in float-float, numerator and rho_a
// scaled by rho_a's power of two, comparisons on the bit patterns (positive
// doubles order as integers; a negative rho_a is below every |j_a|).
template <int D>
__device__ __forceinline__ void record_velocities(double rs, const double (&js)[D],
                                                  const double (&u)[D], double (&out)[D]) {
  const long long rb = __double_as_longlong(rs);
  bool undef = rb <= __double_as_longlong(RHO_TINY);
#pragma unroll
  for (int d = 0; d < D; ++d)
    undef |= (__double_as_longlong(js[d]) & 0x7fffffffffffffffLL) >= rb;
  const int de = 1023 - ((__double2hiint(rs) >> 20) & 0x7ff);
  const ff ir = ff_rcp(ff_of_double(
      __hiloint2double((__double2hiint(rs) & 0x800fffff) | 0x3ff00000, __double2loint(rs))));
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const double w = fma(-rs, u[d], js[d]);
    const int h = __double2hiint(w), ew = ((h >> 20) & 0x7ff) + de;
    const double ws = ew <= 0 || undef
                          ? 0.0
                          : __hiloint2double((h & 0x800fffff) | (ew << 20), __double2loint(w));
    out[d] = ff_pack(ff_of_double(ws) * ir);
  }
}
template <int D>
__device__ __forceinline__ void record_velocities(float rs, const float (&js)[D],
                                                  const float (&u)[D], float (&out)[D]) {
  // where defined, |j_a| < rho_a, so the quotient lies in (-1, 1) even when
  // rho_a is denormal (its reciprocal would overflow)
  const bool undef = species_velocity_undefined<D, float>(rs, js);
#pragma unroll
  for (int d = 0; d < D; ++d) out[d] = undef ? 0.f : js[d] / rs - u[d];
}

// The moments (Sec. 2.1, Sec. 3.1-3.2, Sec. 3.7 slaving, Sec. 4.1 pull
// streaming), record and reaction sub-steps (Sec. 2.4 Eq. R3) of bulk node n by
// one thread, lattice by lattice.
//
// What bounds it: in FP64 the count of FP64 instructions (75 cycles of an SM
// quarter each), in FP32 instruction issue, and in both the latency of the
// loads at the few warps that the registers leave.  So a lattice's 27
// populations are loaded together (27 loads in flight), and the loop over the
// lattices is rolled: its sums need no register arrays and the code stays in
// the instruction cache.  FP64: the sums run in fixed point (fix_of), u_a - u,
// which only becomes a diffusion velocity, is a float-float quotient, and a
// sub-step's energy coefficients are those of the moments plus float-float
// increments (~300 FP64 instructions per node remain of ~1500).
// smem: the block's shared memory (moments_bytes).
template <int D, int M, typename S, typename RT>
__device__ __forceinline__ void moments_body(const S* __restrict__ src, RT* __restrict__ rec,
                                             double* __restrict__ Tf, int* __restrict__ status,
                                             const Geom& g, const Units& un, const BCDev& bc,
                                             const DevMech& mech, long long n, void* smem) {
  constexpr int Q = Lat<D>::Q, NP = Lat<D>::NP;
  using RC = Rec<D, M>;
  using ST = typename SumType<RT>::type;
  using CT = typename ChemType<RT>::type;
  const long long N = g.N;
  if (n >= N) return;
  if (bc.tag && bc.tag[n] == TAG_SOLID) return;
  double* const Wd = static_cast<double*>(smem) + threadIdx.x;
  ChemSlice<M, CT> cs(static_cast<double*>(smem) + M * kChemThreads, threadIdx.x);
  const int x = (int)(n % g.nx);
  const int y = (int)((n / g.nx) % g.ny);
  const int z = (int)(n / ((long long)g.nx * g.ny));
  // pull sources: x of c_x = -1, 0, 1 and the offsets of (c_y, c_z)
  const int xs[3] = {wrap1(x + 1, g.nx), x, wrap1(x - 1, g.nx)};
  int row[Q / 3];      // (a grid of 2^31 nodes would not fit any memory)
#pragma unroll
  for (int r = 0; r < Q / 3; ++r)
    row[r] = g.nx * (wrap1(y - (r % 3 - 1), g.ny) +
                     g.ny * (D == 3 ? wrap1(z - (r / 3 - 1), g.nz) : 0));

  RT rho = RT(0), inv_rho = RT(0), u[D], usq = RT(0), ER = RT(0), Z[D];
  RT Rm = RT(0);                                   // sum Y_a / m_a
  CT cU[4] = {CT(), CT(), CT(), CT()};             // energy polynomial
  Remainder<D, RT> rest;
#pragma unroll
  for (int d = 0; d < D; ++d) u[d] = Z[d] = RT(0);

  // species a's state from its sums: record, concentration, energy polynomial
  auto species = [&](int a, RT rs, const RT (&js)[D]) {
    const RT Y = rs * inv_rho;
    rec[(RC::Y + a) * N + n] = Y;
    if constexpr (kFF<RT>) {
      Rm += Y * mech.inv_mm_s[a];
      ff_fma_acc(cU[0], ff(Y), mech.u0_f[a]);
      ff_fma_acc(cU[1], ff(Y), mech.u1_f[a]);
      ff_fma_acc(cU[2], ff(Y), mech.u2_f[a]);
      ff_fma_acc(cU[3], ff(Y), mech.u3_f[a]);
      cs.set(a, ff(rs) * mech.inv_mm_f[a]);
      Wd[a * kChemThreads] = ff_pack(ff());
    } else {
      double Yd, rd;
      if constexpr (sizeof(RT) == 8) {
        Yd = Y;
        rd = rs;
        Rm = fma(Y, mech.inv_mm[a], Rm);
      } else {
        Yd = double_of_float_exact(Y);
        rd = double_of_float_exact(rs);
        Rm += Y * mech.inv_mm_s[a];
      }
      cU[0] = fma(Yd, mech.u0[a], cU[0]);
      cU[1] = fma(Yd, mech.u1[a], cU[1]);
      cU[2] = fma(Yd, mech.u2[a], cU[2]);
      cU[3] = fma(Yd, mech.u3[a], cU[3]);
      cs.set(a, rd * mech.inv_mm[a]);
      Wd[a * kChemThreads] = 0.0;
    }
    RT us[D];
    record_velocities<D>(rs, js, u, us);
#pragma unroll
    for (int d = 0; d < D; ++d) rec[(RC::US + a * D + d) * N + n] = us[d];
  };

#pragma unroll 1
  for (int it = 0; it <= M; ++it) {
    const int l = it == 0 ? M - 1 : (it == 1 ? M : it - 2);   // f, g, the species
    RT v[Q];
    int e = 0;
    const S* pl = src + (long long)l * Q * N;
#pragma unroll
    for (int i = 0; i < Q; ++i, pl += N)
      v[i] = Codec<S>::template dec<RT>(__ldg(pl + (row[i / 3] + xs[i % 3])), g.codec, l * Q + i);
    if constexpr (sizeof(RT) == 8) {
#pragma unroll
      for (int i = 0; i < Q; ++i) e = max(e, fix_exponent(v[i]));
    }
    ST sum, sj[D], sP[NP];
    lattice_sums<D, RT>(v, e, sum, sj, sP);
    const auto t0 = close_sum(sum, e);
    const RT s0 = sum_value(t0);
    RT s1[D];
#pragma unroll
    for (int d = 0; d < D; ++d) s1[d] = sum_value(close_sum(sj[d], e));
    if (it == 0) {
      rho = s0;
      inv_rho = RT(1) / rho;
      rec[RC::RHO * N + n] = rho;
#pragma unroll
      for (int d = 0; d < D; ++d) {
        u[d] = s1[d] * inv_rho;
        usq = fma(u[d], u[d], usq);
        rec[(RC::U + d) * N + n] = u[d];
      }
      RT P[NP];
#pragma unroll
      for (int k = 0; k < NP; ++k) P[k] = sum_value(close_sum(sP[k], e));
#pragma unroll
      for (int d = 0; d < D; ++d) Z[d] = flux_less_work<D, RT>(d, u, Z, P);
      rest.start(e);
    } else if (it == 1) {
      ER = s0 * inv_rho;
      rec[RC::E * N + n] = ER;
#pragma unroll
      for (int d = 0; d < D; ++d) rec[(RC::Z + d) * N + n] = s1[d] + Z[d];
    }
    if (it != 1) {
      rest.add(0, t0, s0, it == 0);
#pragma unroll
      for (int d = 0; d < D; ++d) rest.add(1 + d, close_sum(sj[d], e), s1[d], it == 0);
      if (it > 1) species(l, s0, s1);
    }
  }
  {   // slaved species M (Eq. strongest)
    RT js[D];
#pragma unroll
    for (int d = 0; d < D; ++d) js[d] = rest.get(1 + d);
    species(M - 1, rest.get(0), js);
  }

  // temperature (Eq. temperature) from the node's previous T
  using X = Chem<CT>;
  CT U;
  ff irho;
  if constexpr (kFF<RT>) {
    irho = ff_rcp(ff(rho));
#pragma unroll
    for (int k = 0; k < 4; ++k) cU[k] = ff_norm(cU[k]);
    U = (ff(ER) + ff(-0.5f * usq)) * un.c2_f;
  } else {
    if constexpr (sizeof(RT) == 8) irho = ff_of_double(inv_rho);
    else irho = ff_rcp(ff(rho));
    U = (double(ER) - 0.5 * double(usq)) * un.c * un.c;
  }
  bool ok;
  CT Ts = newton_poly(cU, U, X::of_T(__ldcg(Tf + n)), un.newton_max_iter, X::rtol(un), ok);
  double T;
  RT th, H[4];
  if constexpr (kFF<RT>) {
    T = ff_to_double(Ts);
    th = Rm * float(R_U) * Ts.hi * un.inv_c2_s;
  } else if constexpr (sizeof(RT) == 4) {
    T = Ts;
    th = Rm * float(R_U) * float(T) * un.inv_c2_s;
  } else {
    T = Ts;
    th = R_U * Rm * T * un.inv_c2;
  }
  if (!ok) atomicOr(status, ST_NEWTON);
  if (!(rho > RT(0)) || !isfinite(rho) || !isfinite(T)) atomicOr(status, ST_NONFINITE);
  Tf[n] = T;
  enthalpy_poly(cU, Rm, un, H);
#pragma unroll
  for (int k = 0; k < 4; ++k) rec[(RC::H + k) * N + n] = H[k];
  rec[RC::TH * N + n] = th;
  const RT b3 = fma(RT(-3), th, RT(1));                            // 1 - 3 theta
#pragma unroll
  for (int d = 0; d < D; ++d)
    rec[(RC::PHI + d) * N + n] = rho * u[d] * fma(-u[d], u[d], b3);
  if constexpr (sizeof(RT) == 4) rec[RC::LNT * N + n] = ln_T0(RT(T));

  // reaction sub-steps at frozen U (Sec. 2.4 Eq. R3): a zero-dimensional
  // reactor per node from its post-stream species densities; T_0 is the T just
  // solved
  ff dU[4];                              // increments of rho cU
#pragma unroll 1
  for (int s = 0; s < un.substeps; ++s) {
    if (s > 0) {
      CT c[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) c[k] = cU[k] + X::of_ff(ff_norm(dU[k]) * irho);
      bool oks;
      Ts = newton_poly(c, U, Ts, un.newton_max_iter, X::rtol(un), oks);
      if (!oks) atomicOr(status, ST_NEWTON);
    }
#pragma unroll
    for (int a = 0; a < M; ++a) cs.clear(a);
    const TBasis<CT> tb = tbasis(mech, Ts);
    if constexpr (sizeof(RT) == 8)
      if (s == 0) rec[RC::LNT * N + n] = tb.lnT - LN_T_REF;
    add_reactions(mech, tb, cs, 0, 1);
    const bool last = s + 1 == un.substeps;
#pragma unroll 1
    for (int a = 0; a < M; ++a) {
      const CT w = cs.rate(a);
      // FP32: with what its rounding took off rho Y_a, so that the sub-steps'
      // energies are those of rho_a / rho in the chemistry's precision
      float e = 0.f;
      if constexpr (sizeof(RT) == 4) {
        if (s == 0 && !last) {
          ff c;
          if constexpr (kFF<RT>) c = cs.c(a);
          else c = ff_of_double(cs.c(a));
          const float rs = (c * mech.mm_f[a]).hi;       // rho_a again
          e = __fmaf_rn(-(rs * inv_rho), rho, rs);
        }
      }
      ff inc;
      if constexpr (kFF<RT>) {
        Wd[a * kChemThreads] = ff_pack(ff_unpack(Wd[a * kChemThreads]) + w);
        if (last) continue;
        cs.set(a, cs.c(a) + un.dt_sub_f * w);
        inc = w * un.dtmm_f[a];
      } else {
        Wd[a * kChemThreads] += w;
        if (last) continue;
        cs.set(a, fma(w, un.dt_sub, cs.c(a)));
        inc = ff_of_double(w) * un.dtmm_f[a];
      }
      if constexpr (sizeof(RT) == 4) ff_acc(inc, ff(e));
      ff_fma_acc(dU[0], inc, mech.u0_f[a]);
      ff_fma_acc(dU[1], inc, mech.u1_f[a]);
      ff_fma_acc(dU[2], inc, mech.u2_f[a]);
      ff_fma_acc(dU[3], inc, mech.u3_f[a]);
    }
  }
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    if constexpr (kFF<RT>)
      rec[(RC::DRHO + a) * N + n] = (ff_unpack(Wd[a * kChemThreads]) * un.dtmm_f[a]).hi;
    else
      rec[(RC::DRHO + a) * N + n] = RT(Wd[a * kChemThreads] * un.dtmm[a]);
  }
}

// Transport and lattice constants in the parameter type: FP64 for the FP64
// path, FP32 for the mixed path.
template <typename PT> struct MixParams;
template <> struct MixParams<double> {
  __device__ static double inv_mm(const DevMech& m, int a) { return m.inv_mm[a]; }
  __device__ static double Ra(const DevMech& m, int a) { return m.Ra[a]; }
  __device__ static double D_T_exp(const DevMech& m) { return m.D_T_exp; }
  __device__ static double mu0(const DevMech& m) { return m.mu0; }
  __device__ static double mu_T_exp(const DevMech& m) { return m.mu_T_exp; }
  __device__ static double inv_prandtl(const DevMech& m) { return m.inv_prandtl; }
  __device__ static double inv_c2(const Units& u) { return u.inv_c2; }
  __device__ static double s_pref(const Units& u) { return u.s_pref; }
  __device__ static double nu_pref(const Units& u) { return u.nu_pref; }
  __device__ static double mu0_sp(const DevMech& m, int a) { return m.mu0_sp[a]; }
  __device__ static double wilke_phi(const DevMech& m, int a, int b) {
    return m.wilke_phi[a][b];
  }
};
template <> struct MixParams<float> {
  __device__ static float inv_mm(const DevMech& m, int a) { return m.inv_mm_s[a]; }
  __device__ static float Ra(const DevMech& m, int a) { return m.Ra_s[a]; }
  __device__ static float D_T_exp(const DevMech& m) { return m.D_T_exp_s; }
  __device__ static float mu0(const DevMech& m) { return m.mu0_s; }
  __device__ static float mu_T_exp(const DevMech& m) { return m.mu_T_exp_s; }
  __device__ static float inv_prandtl(const DevMech& m) { return m.inv_prandtl_s; }
  __device__ static float inv_c2(const Units& u) { return u.inv_c2_s; }
  __device__ static float s_pref(const Units& u) { return u.s_pref_s; }
  __device__ static float nu_pref(const Units& u) { return u.nu_pref_s; }
  __device__ static float mu0_sp(const DevMech& m, int a) { return m.mu0_sp_s[a]; }
  __device__ static float wilke_phi(const DevMech& m, int a, int b) {
    return m.wilke_phi_s[a][b];
  }
};

__device__ __forceinline__ float exp_of(float x) { return exp(x); }
__device__ __forceinline__ double exp_of(double x) { return exp_tang(x); }

// ---------------------------------------------------------------------------
// Per-node collision parameters: everything the direction loop needs
// (Sec. 2.3 Eqs. betaa, taua, transform1; Sec. 3.3 Eq. Pex; Sec. 3.4 Eqs.
// gstar, qdiff, corrFourier; Sec. 2.4 Eq. R3).
// The diffusion velocities and what only they need: float-float in the FP64
// path (solve_dd_ff), FP32 in the mixed path (solve_dd_strided).
template <typename RT> struct DiffType { using type = RT; };
template <> struct DiffType<double> { using type = ff; };
template <int D, int M, typename RT> struct NodePar {
  RT rho, om, U, theta;          // density, omega, internal energy, R T (lattice)
  RT u[D], Pex[D], W[D];         // velocity, extended diagonal pressure, energy-flux term
  RT th[M], rs[M];               // theta_b, rho_b
  typename DiffType<RT>::type V[M][D];             // diffusion velocities
  // (beta_a - 1) Y_a s, 1 - 2 beta_a, 2 beta_a rho_a + drho_a
  RT cF[M - 1], om1[M - 1], hh[M - 1];
};

// Field offsets of NodePar stored field-major [field][N] (split collision);
// float-float fields as packed pairs (ff_pack).
template <int D, int M> struct CPar {
  static constexpr int TH = 0;
  static constexpr int V = TH + M;
  static constexpr int RS = V + M * D;
  static constexpr int CF = RS + M;
  static constexpr int OM1 = CF + M - 1;
  static constexpr int HH = OM1 + M - 1;
  static constexpr int U = HH + M - 1;
  static constexpr int PEX = U + D;
  static constexpr int W = PEX + D;
  static constexpr int RHO = W + D;
  static constexpr int OM = RHO + 1;
  static constexpr int UL = OM + 1;
  static constexpr int THETA = UL + 1;
  static constexpr int NF = THETA + 1;
};

// The per-node part of the collision of node n (not solid, n < N):
// moments from the record, isotropic gradients, relaxation parameters,
// diffusion velocities, energy-flux correction.  The diffusion-velocity
// solve uses this thread's shared-memory column (M*M entries, stride kBS).
// kLive: the records were written earlier in the same launch (k_step_persist),
// so the neighbours' fields may not come through the read-only path.
template <bool kLive, typename RT>
__device__ __forceinline__ RT record_load(const RT* p) {
  if constexpr (kLive) return __ldcg(p);
  else return __ldg(p);
}
template <int D, int M, bool kLive, typename RT>
__device__ __forceinline__ void node_params(const RT* __restrict__ rec,
                                            const double* __restrict__ Tf, const Geom& g,
                                            const Units& un, const BCDev& bc,
                                            const DevMech& mech, long long n, int tag,
                                            NodePar<D, M, RT>& p) {
  constexpr int Q = Lat<D>::Q;
  using RC = Rec<D, M>;
  const long long N = g.N;
  const int x = (int)(n % g.nx);
  const int y = (int)((n / g.nx) % g.ny);
  const int z = (int)(n / ((long long)g.nx * g.ny));

  // node scalars in the lattice type; the diffusion velocities in VT
  using MP = MixParams<RT>;
  using VT = typename DiffType<RT>::type;
  const RT rho = rec[RC::RHO * N + n];
  const double T_d = __ldcg(Tf + n);
  const RT T = RT(T_d);
  const RT E = rec[RC::E * N + n];
  const RT theta = rec[RC::TH * N + n];
  RT u[D], Y[M], Z[D], usq = RT(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    u[d] = rec[(RC::U + d) * N + n];
    Z[d] = rec[(RC::Z + d) * N + n];
    usq += u[d] * u[d];
  }
#pragma unroll
  for (int a = 0; a < M; ++a) Y[a] = rec[(RC::Y + a) * N + n];

  // isotropic gradients 3 sum_i w_i c_i phi(x + c_i): d_a Phi_a, and
  // sum_a H_a grad Y_a with this node's H_a, from the neighbours' enthalpy
  // polynomials at this node's T (three multiply-adds per neighbour instead of
  // M, and M - 4 fewer loads)
  RT dPhi[D], corr[D];
#pragma unroll
  for (int d = 0; d < D; ++d) dPhi[d] = corr[d] = RT(0);
  auto enthalpy = [&](long long nb) {
    const RT* h = rec + (long long)RC::H * N + nb;
    auto H = [&](int k) { return record_load<kLive>(h + k * N); };
    return fma(T, fma(T, fma(T, H(3), H(2)), H(1)), H(0));
  };
  const RT HYself = enthalpy(n);
  // ghost values beyond non-periodic faces and on solid nodes: walls Phi = 0,
  // inlet the inlet state's Phi, outlet the node's own Phi; Y the node's own
  RT phi_self[D], phi_in[D];
#pragma unroll
  for (int d = 0; d < D; ++d) {
    phi_self[d] = RT(0);
    phi_in[d] = RT(0);
  }
  if (bc.tag) {
#pragma unroll
    for (int d = 0; d < D; ++d) {
      phi_self[d] = rec[(RC::PHI + d) * N + n];
      const RT ui = tag >= 0 ? RT(bc.if_uin[(long long)d * bc.n_if + tag]) : RT(0);
      const RT rin = RT(bc.rho_in);
      phi_in[d] = rin * ui * (RT(1) - RT(3) * RT(bc.theta_in)) - rin * ui * ui * ui;
    }
  }
  // x-rows of neighbours unrolled, rows rolled (instruction footprint, as in
  // the moments kernel)
#pragma unroll 1
  for (int r = 0; r < Q / 3; ++r) {
    const int cyi = r % 3 - 1, czi = D == 3 ? r / 3 - 1 : 0;
#pragma unroll
    for (int ix = 0; ix < 3; ++ix) {
      const int cxi = ix - 1;
      if (ix == 1 && cyi == 0 && czi == 0) continue;          // the rest velocity
      const int cvi[3] = {cxi, cyi, czi};
      long long nb = 0;
      int gk = BK_NONE;
      if (!bc.tag) {
        nb = node_shift<D>(x, y, z, 3 * r + ix, +1, g);
      } else {
        int cc[3] = {x + cxi, y + cyi, D == 3 ? z + czi : z};
        const int ext[3] = {g.nx, g.ny, g.nz};
#pragma unroll
        for (int a = 0; a < D; ++a) {
          if (cc[a] < 0) {
            if (bc.face[2 * a]) { if (!gk) gk = bc.face[2 * a]; } else cc[a] += ext[a];
          } else if (cc[a] >= ext[a]) {
            if (bc.face[2 * a + 1]) { if (!gk) gk = bc.face[2 * a + 1]; } else cc[a] -= ext[a];
          }
        }
        if (!gk) {
          nb = cc[0] + (long long)g.nx * (cc[1] + (long long)g.ny * cc[2]);
          if (bc.has_solid && bc.tag[nb] == TAG_SOLID) gk = bc.solid_kind;
        }
      }
      // 3 w_i: the product of 2/3 (c = 0) and 1/6 (c = +-1) per axis
      const RT wy = cyi == 0 ? RT(2.0 / 3.0) : RT(1.0 / 6.0);
      const RT wz = D == 3 ? (czi == 0 ? RT(2.0 / 3.0) : RT(1.0 / 6.0)) : RT(1);
      const RT w3 = RT(3) * ((ix == 1 ? RT(2.0 / 3.0) : RT(1.0 / 6.0)) * wy * wz);
      const RT hy = gk == BK_NONE ? enthalpy(nb) : HYself;
#pragma unroll
      for (int d = 0; d < D; ++d) {
        if (cvi[d] == 0) continue;
        const RT wc = w3 * RT(cvi[d]);
        const RT pv = gk == BK_NONE ? record_load<kLive>(rec + (RC::PHI + d) * N + nb)
                      : (gk == BK_INLET ? phi_in[d] : (gk == BK_OUTLET ? phi_self[d] : RT(0)));
        dPhi[d] += wc * pv;
        corr[d] += wc * hy;
      }
    }
  }

  // relaxation parameters (Sec. 2.3 Eqs. betaa, taua; Sec. 3.5 Eqs. mu,
  // lambda): 1/tau_ab = s K_ab; with xr = nu/theta, omega = 1/(xr + 1/2),
  // omega1 = 1/(xr/Pr + 1/2) and (2 - omega)/(2 omega) = xr
  const RT lnTr = rec[RC::LNT * N + n];
  const RT s_tau = MP::s_pref(un) * rho * T * T * exp_of(-MP::D_T_exp(mech) * lnTr);
  RT mu = MP::mu0(mech);
  if (mech.wilke) {
    // Wilke's mixing rule over the species viscosities (the mole fractions'
    // normalisation cancels between numerator and denominator)
    RT X[M];
#pragma unroll
    for (int a = 0; a < M; ++a) X[a] = Y[a] * MP::inv_mm(mech, a);
    mu = RT(0);
#pragma unroll
    for (int a = 0; a < M; ++a) {
      RT den = RT(0);
#pragma unroll
      for (int b = 0; b < M; ++b) den += X[b] * MP::wilke_phi(mech, a, b);
      mu += X[a] * MP::mu0_sp(mech, a) / den;
    }
  }
  mu *= exp_of(MP::mu_T_exp(mech) * lnTr);
  const RT Pres = rho * theta;
  const RT iP = RT(1) / Pres;
  const RT xr = mu * MP::nu_pref(un) * iP;
  const RT h0 = xr + RT(0.5), h1 = xr * MP::inv_prandtl(mech) + RT(0.5);
  const RT ih = RT(1) / (h0 * h1);
  const RT omega = h1 * ih, omega1 = h0 * ih;

  // diffusion velocities, Eq. transform1: A V = u_a - u  (V holds the rhs),
  // A_aa = 1 + 1/(2 tau_a), A_ab = -Y_b/(2 tau_ab).  Each thread's matrix lives
  // in shared memory, entry-major with the block's threads contiguous (no
  // bank conflicts): in registers it would not fit beside the node's other
  // state and spills to local memory.
  VT V[M][D], sv;
  RT inv_tau_a[M];               // FP64: 2 + 1/tau_a
  {
    extern __shared__ unsigned char smem_raw[];
    VT* As = reinterpret_cast<VT*>(smem_raw) + threadIdx.x;
    const int st = kBS;
    if constexpr (sizeof(RT) == 8) {
      sv = ff_of_double(s_tau * mech.K_unit);
      constexpr int W = M + D;
      ff Yv[M], yh[M];
#pragma unroll
      for (int a = 0; a < M; ++a) {
        Yv[a] = ff_of_double(Y[a]);
        yh[a] = ff(-0.5f * sv.hi, -0.5f * sv.lo) * Yv[a];
      }
#pragma unroll 1
      for (int a = 0; a < M; ++a) {
#pragma unroll
        for (int b = 0; b < M; ++b) As[(a * W + b) * st] = yh[b] * mech.K_f[a][b];
#pragma unroll
        for (int d = 0; d < D; ++d)
          As[(a * W + M + d) * st] = ff_unpack(rec[(RC::US + a * D + d) * N + n]);
      }
#pragma unroll
      for (int a = 0; a < M; ++a) {
        // in FP64: beta_a moves whole populations, not a correction (in
        // float-float the lightest species lost two bits of FP64's accuracy)
        double acc = 0.0;
#pragma unroll
        for (int b = 0; b < M; ++b)
          if (b != a) acc = fma(mech.K[a][b], Y[b], acc);
        inv_tau_a[a] = fma(s_tau, acc, 2.0);
        const ff dg = ff_of_double(inv_tau_a[a]);
        As[(a * W + a) * st] = ff(0.5f * dg.hi, 0.5f * dg.lo);
      }
      solve_dd_ff<M, D>(As, st);
#pragma unroll
      for (int a = 0; a < M; ++a)
#pragma unroll
        for (int d = 0; d < D; ++d) V[a][d] = As[(a * W + M + d) * st];
    } else {
      sv = s_tau;
#pragma unroll
      for (int a = 0; a < M; ++a) {
        RT acc = RT(0);
#pragma unroll
        for (int b = 0; b < M; ++b)
          if (b != a) acc += Y[b] * kcoef<RT>(mech, a, b);
        inv_tau_a[a] = s_tau * acc;
        As[(a * M + a) * st] = RT(1) + RT(0.5) * inv_tau_a[a];
#pragma unroll
        for (int d = 0; d < D; ++d) V[a][d] = rec[(RC::US + a * D + d) * N + n];
      }
#pragma unroll
      for (int b = 0; b < M; ++b) {
        const RT y = RT(-0.5) * s_tau * Y[b];
#pragma unroll
        for (int a = 0; a < M; ++a)
          if (b != a) As[(a * M + b) * st] = y * kcoef<RT>(mech, a, b);
      }
      solve_dd_strided<M, D, RT>(As, st, V);
    }
  }

  // species densities; the reaction increments come from the moments kernel
  RT rs[M];
#pragma unroll
  for (int a = 0; a < M; ++a) rs[a] = rho * Y[a];

  // energy-flux correction W = (omega - omega1)(q* - q^eq), folded form
  const RT U_lat = E - RT(0.5) * usq;
  RT W[D];
  {
    // diffusion flux sum_a H_a Y_a V_a, H_a/c^2 in float-float
    VT diff[D];
#pragma unroll
    for (int d = 0; d < D; ++d) diff[d] = VT();
    const ff T1 = ff_of_double(T_d), T2 = T1 * T1, T3 = T2 * T1;
#pragma unroll
    for (int a = 0; a < M; ++a) {
      ff h = un.hl_f[0][a];
      ff_fma_acc(h, un.hl_f[1][a], T1);
      ff_fma_acc(h, un.hl_f[2][a], T2);
      ff_fma_acc(h, un.hl_f[3][a], T3);
      if constexpr (sizeof(RT) == 8) {
        const ff HY = ff_norm(h) * ff_of_double(Y[a]);
#pragma unroll
        for (int d = 0; d < D; ++d) ff_fma_acc(diff[d], HY, V[a][d]);
      } else {
        const RT HY = ff_norm(h).hi * Y[a];
#pragma unroll
        for (int d = 0; d < D; ++d) diff[d] += HY * V[a][d];
      }
    }
    // q - q^eq - u . (P - P^eq) = (q - u . P) - rho u (E - u^2)
    const RT b = rho * (E - usq);
#pragma unroll
    for (int d = 0; d < D; ++d) {
      RT df;
      if constexpr (sizeof(RT) == 8) df = double_of_ff(diff[d]);
      else df = diff[d];
      const RT qd = fma(-b, u[d], Z[d]) - RT(0.5) * u[d] * dPhi[d];     // with q^ex
      W[d] = (omega - omega1) * qd + omega1 * rho * df +
             (RT(0.5) * (RT(2) - omega1)) * Pres * corr[d];
    }
  }

  // per-lattice parameters
#pragma unroll
  for (int a = 0; a < M; ++a) {
    p.th[a] = MP::Ra(mech, a) * T * MP::inv_c2(un);
    p.rs[a] = rs[a];
#pragma unroll
    for (int d = 0; d < D; ++d) p.V[a][d] = V[a][d];
  }
#pragma unroll
  for (int d = 0; d < D; ++d) {
    p.u[d] = u[d];
    p.Pex[d] = theta + u[d] * u[d] + xr * (iP * theta) * dPhi[d];
    p.W[d] = W[d];
  }
  p.rho = rho;
  p.om = omega;
  p.U = U_lat;
  p.theta = theta;
  // species coefficients of the update
  //   f_a + 2 beta_a (rho_a psi_a - f_a) + cF_a sum_b K_ab d_b + drho_a psi_a
  //     = f_a om1_a + psi_a hh_a + cF_a sum_b K_ab d_b,
  // cF_a = (beta_a - 1) Y_a s (1/tau_ab = s K_ab), om1_a = 1 - 2 beta_a,
  // hh_a = 2 beta_a rho_a + drho_a; beta = 1 / (2 tau + 1) = 1 - 2 r, r =
  // 1 / (2 + 1/tau) (om1 and hh share its rounding, so that mass is conserved)
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    RT beta;
    if constexpr (sizeof(RT) == 8) {
      // r in float-float and a Newton step in FP64
      int e;
      const ff x = ff_mantissa(inv_tau_a[a], e);
      const double r0 = double_join(ff_rcp(x), -e);
      const double r = fma(r0, fma(-inv_tau_a[a], r0, 1.0), r0);
      beta = fma(-2.0, r, 1.0);
      // beta - 1 = -2 r; FP64's range, which trace species need
      p.cF[a] = r * (Y[a] * (-2.0 * s_tau));
    } else {
      beta = inv_tau_a[a] / (RT(2) + inv_tau_a[a]);
      p.cF[a] = (beta - RT(1)) * Y[a] * s_tau;
    }
    p.om1[a] = RT(1) - RT(2) * beta;
    p.hh[a] = RT(2) * beta * rs[a] + rec[(RC::DRHO + a) * N + n];
  }
}

// Energy-equilibrium axis factors (the closed form of g^eq, Sec. 3.4 Eq.
// geq_i): A_c acting on 1 and B_c acting on u^2/2, c = -1, 0, 1.
template <int D, typename RT>
__device__ __forceinline__ void energy_factors(const RT (&u)[D], RT theta, RT (&Af)[D][3],
                                               RT (&Bf)[D][3]) {
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const RT ua = u[d];
    const RT O1 = theta * ua + RT(0.5) * ua * ua * ua;
    const RT O2 = theta * theta + RT(2.5) * theta * ua * ua + RT(0.5) * ua * ua * ua * ua;
    const RT Pd = theta + ua * ua;
    Af[d][0] = RT(0.5) * (Pd - ua);
    Af[d][1] = RT(1) - Pd;
    Af[d][2] = RT(0.5) * (Pd + ua);
    Bf[d][0] = RT(0.5) * (O2 - O1);
    Bf[d][1] = RT(0.5) * ua * ua - O2;
    Bf[d][2] = RT(0.5) * (O2 + O1);
  }
}

// Axis factors of psi(u, theta_b) (set 0) and psi(u + V_b, theta_b) (set 1)
// (Eq. prod): entry e = ((set*M + b)*D + d)*3 + c + 1 of a table.
template <int D, int M, typename RT>
__device__ __forceinline__ RT axis_factor(int e, const RT* th, const RT* u, const RT* V) {
  const int c = e % 3 - 1;
  const int d = (e / 3) % D;
  const int b = (e / (3 * D)) % M;
  const int set = e / (3 * D * M);
  const RT xs = set ? u[d] + V[b * D + d] : u[d];
  const RT Ps = th[b] + xs * xs;
  return c == 0 ? RT(1) - Ps : (c > 0 ? RT(0.5) * (Ps + xs) : RT(0.5) * (Ps - xs));
}

// The M + 1 populations of direction i entering node n's collision (pulled
// from node sn, or the boundary-reconstructed ones).
template <int D, int M, typename S, typename RT>
__device__ __forceinline__ void load_direction(const S* __restrict__ src, const BCDev& bc,
                                               int tag, long long N, long long sn, int i,
                                               const float4* codec, RT (&fin)[M + 1]) {
  constexpr int Q = Lat<D>::Q;
#pragma unroll
  for (int l = 0; l <= M; ++l) fin[l] = pop_in<RT>(src, bc, tag, N, sn, l * Q + i, codec);
}

// The part of the equilibria of direction (c_x, c_y, c_z) that depends on
// (c_x, c_y) only, shared by the directions that differ in c_z (the product
// form, Sec. 3.3 Eqs. prod, feqmix; Sec. 3.4 Eq. geq_i):
//   species  e_b = psi_x psi_y of psi(u, theta_b), s_b the same of psi(u + V_b, theta_b);
//   momentum rho psi_x psi_y of the extended equilibrium;
//   energy   g^eq = rho [A_z (U A_x A_y + B_x A_y + A_x B_y) + A_x A_y B_z].
template <int D, int M, typename RT> struct XYPart {
  RT e[M], s[M];
  RT fxy, gP, gQ;
};

template <int D, int M, typename RT, typename PS>
__device__ __forceinline__ void xy_part(const PS& ps, int cx, int cy, XYPart<D, M, RT>& h) {
#pragma unroll
  for (int b = 0; b < M; ++b) {
    h.e[b] = ps.sp(0, b, 0, cx) * ps.sp(0, b, 1, cy);
    h.s[b] = ps.sp(1, b, 0, cx) * ps.sp(1, b, 1, cy);
  }
  h.fxy = ps.rho() * psi1<RT>(cx, ps.u(0), ps.Pex(0)) * psi1<RT>(cy, ps.u(1), ps.Pex(1));
  const RT ax = ps.Af(0, cx), ay = ps.Af(1, cy);
  h.gP = ax * ay;
  h.gQ = ps.U() * h.gP + ps.Bf(0, cx) * ay + ax * ps.Bf(1, cy);
}

// Collision of every lattice in direction i = (c_x, c_y, cz) of node n
// (Sec. 2.3 Eq. finalNumericalEquationsReactive; Sec. 3.2 Eqs. f, g; Sec.
// 3.3 Eq. feqmix), from the shared (c_x, c_y) part h.  PS supplies the
// node's parameters (registers, or the block's shared memory in the split
// placement).  The species update
//   f_a + 2 beta_a (rho_a psi_a - f_a) + cF_a sum_b K_ab d_b + drho_a psi_a
// is evaluated as f_a om1_a + psi_a hh_a + cF_a F_a with the per-node
// om1_a = 1 - 2 beta_a and hh_a = 2 beta_a rho_a + drho_a.
template <int D, int M, typename S, typename RT, typename PS>
__device__ __forceinline__ void collide_direction(const PS& ps, const XYPart<D, M, RT>& h,
                                                  int i, const RT (&fin)[M + 1],
                                                  S* __restrict__ dst, long long N, long long n,
                                                  const DevMech& mech, const float4* codec) {
  constexpr int Q = Lat<D>::Q;
  const int cz = D == 3 ? cvel(i, 2) : 0;
  RT pe[M], dd[M];
#pragma unroll
  for (int b = 0; b < M; ++b) {
    RT e = h.e[b], st = h.s[b];
    if constexpr (D == 3) {
      e *= ps.sp(0, b, 2, cz);
      st *= ps.sp(1, b, 2, cz);
    }
    pe[b] = e;
    dd[b] = ps.rs(b) * (e - st);
  }
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    RT F = RT(0);
#pragma unroll
    for (int b = 0; b < M; ++b)
      if (b != a) F += kcoef<RT>(mech, a, b) * dd[b];
    const long long off = (long long)(a * Q + i) * N;
    const RT fn = fin[a] * ps.om1(a) + pe[a] * ps.hh(a) + ps.cF(a) * F;
    dst[off + n] = Codec<S>::enc(fn, codec, a * Q + i);
  }
  {
    RT fex = h.fxy;
    if constexpr (D == 3) fex *= psi1<RT>(cz, ps.u(2), ps.Pex(2));
    const long long off = (long long)((M - 1) * Q + i) * N;
    const RT f = fin[M - 1];
    dst[off + n] = Codec<S>::enc(f + ps.om() * (fex - f), codec, (M - 1) * Q + i);
  }
  {
    RT geq = h.gQ;
    if constexpr (D == 3) geq = ps.Af(2, cz) * h.gQ + h.gP * ps.Bf(2, cz);
    geq *= ps.rho();
    const long long off = (long long)(M * Q + i) * N;
    const RT gv = fin[M];
    RT gn = gv + ps.om() * (geq - gv);
    if (csq(i, D) == 1) {
#pragma unroll
      for (int d = 0; d < D; ++d)
        if (cvel(i, d) != 0) gn += (cvel(i, d) > 0 ? RT(0.5) : RT(-0.5)) * ps.W(d);
    }
    dst[off + n] = Codec<S>::enc(gn, codec, M * Q + i);
  }
}

__device__ __forceinline__ float value_of(float v) { return v; }
__device__ __forceinline__ double value_of(ff v) { return double_of_ff(v); }
__device__ __forceinline__ float stored(float v) { return v; }
__device__ __forceinline__ double stored(ff v) { return ff_pack(v); }

// Parameters held in registers (fused placement).  The species axis factors
// come from a table in this thread's shared-memory column (FP32, entry stride
// kBS) or are formed directly, except, in FP64 3D, those of the y and z axes,
// tabulated in the column (yztab: entry (((set M + b) 2 + d - 1) 3 + c + 1)
// kBS, d = 1, 2).
template <int D, int M, typename RT> struct RegPar {
  const NodePar<D, M, RT>& p;
  RT Afv[D][3], Bfv[D][3], Vx[M];
  const RT* tab;
  const RT* yztab;
  __device__ RegPar(const NodePar<D, M, RT>& p_, const RT* tab_, const RT* yztab_ = nullptr)
      : p(p_), tab(tab_), yztab(yztab_) {
    energy_factors<D, RT>(p.u, p.theta, Afv, Bfv);
#pragma unroll
    for (int b = 0; b < M; ++b) Vx[b] = value_of(p.V[b][0]);
  }
  __device__ RT rho() const { return p.rho; }
  __device__ RT om() const { return p.om; }
  __device__ RT U() const { return p.U; }
  __device__ RT u(int d) const { return p.u[d]; }
  __device__ RT Pex(int d) const { return p.Pex[d]; }
  __device__ RT W(int d) const { return p.W[d]; }
  __device__ RT rs(int a) const { return p.rs[a]; }
  __device__ RT cF(int a) const { return p.cF[a]; }
  __device__ RT om1(int a) const { return p.om1[a]; }
  __device__ RT hh(int a) const { return p.hh[a]; }
  __device__ RT Af(int d, int c) const { return c == 0 ? Afv[d][1] : (c > 0 ? Afv[d][2] : Afv[d][0]); }
  __device__ RT Bf(int d, int c) const { return c == 0 ? Bfv[d][1] : (c > 0 ? Bfv[d][2] : Bfv[d][0]); }
  // species axis factor (set 0: psi(u, theta_b); set 1: psi(u + V_b, theta_b))
  __device__ RT sp(int set, int b, int d, int c) const {
    if (tab) return tab[(((set * M + b) * D + d) * 3 + c + 1) * kBS];
    if (D == 3 && d > 0 && yztab) return yztab[(((set * M + b) * 2 + d - 1) * 3 + c + 1) * kBS];
    const RT xs = set ? p.u[d] + (d == 0 ? Vx[b] : RT(value_of(p.V[b][d]))) : p.u[d];
    return psi1<RT>(c, xs, p.th[b] + xs * xs);
  }
};

// Fused placement: one thread per node does the per-node part and then every
// direction (Sec. 2.3, 3.2-3.4).
template <int D, int M, bool kLive, typename S, typename RT>
__device__ __forceinline__ void collide_body(const S* __restrict__ src, S* __restrict__ dst,
                                             const RT* __restrict__ rec,
                                             const double* __restrict__ Tf,
                                             int* __restrict__ status, const Geom& g,
                                             const Units& un, const BCDev& bc,
                                             const DevMech& mech, long long n) {
  constexpr int Q = Lat<D>::Q;
  const long long N = g.N;
  if (n >= N) return;
  const int tag = bc.tag ? bc.tag[n] : TAG_BULK;
  if (tag == TAG_SOLID) return;
  NodePar<D, M, RT> p;
  node_params<D, M, kLive, RT>(rec, Tf, g, un, bc, mech, n, tag, p);
  const int x = (int)(n % g.nx);
  const int y = (int)((n / g.nx) % g.ny);
  const int z = (int)(n / ((long long)g.nx * g.ny));
  // FP32: the species axis factors tabulated once per node in this thread's
  // shared-memory column (the solve's space, now free)
  extern __shared__ unsigned char smem_raw[];
  RT* tab = nullptr;
  RT* yztab = nullptr;
  if constexpr (sizeof(RT) == 4) {
    tab = reinterpret_cast<RT*>(smem_raw) + threadIdx.x;
    constexpr int NT = 2 * M * D * 3;
#pragma unroll
    for (int e = 0; e < NT; ++e)
      tab[e * kBS] = axis_factor<D, M, RT>(e, p.th, p.u, &p.V[0][0]);
  } else if constexpr (D == 3) {
    // FP64: the y- and z-axis factors, psi_c(x_s, theta_b + x_s^2) with
    // x_s = u_d (set 0) or u_d + V_bd (set 1)
    yztab = reinterpret_cast<RT*>(smem_raw) + threadIdx.x;
#pragma unroll
    for (int set = 0; set < 2; ++set)
#pragma unroll
      for (int b = 0; b < M; ++b)
#pragma unroll
        for (int d = 1; d < 3; ++d) {
          const RT xs = set ? p.u[d] + RT(value_of(p.V[b][d])) : p.u[d];
          const RT Ps = p.th[b] + xs * xs;
#pragma unroll
          for (int c = -1; c <= 1; ++c)
            yztab[(((set * M + b) * 2 + d - 1) * 3 + c + 1) * kBS] = psi1<RT>(c, xs, Ps);
        }
  }
  const RegPar<D, M, RT> ps(p, tab, yztab);
  // directions i = j + 9 k share (c_x, c_y) = direction j's
#pragma unroll 1
  for (int j = 0; j < 9; ++j) {
    XYPart<D, M, RT> h;
    xy_part<D, M, RT>(ps, cvel(j, 0), cvel(j, 1), h);
#pragma unroll 1
    for (int i = j; i < Q; i += 9) {
      RT fin[M + 1];
      load_direction<D, M, S, RT>(src, bc, tag, N, node_shift<D>(x, y, z, i, -1, g), i,
                                  g.codec, fin);
      collide_direction<D, M, S, RT>(ps, h, i, fin, dst, N, n, mech, g.codec);
    }
  }
}

// ---------------------------------------------------------------------------
// Split placement of the collision (the default): k_prep (one thread per node)
// stores each node's parameters field-major; k_coll gives every node kCollTPN
// threads (one warp per direction group, lanes over 32 consecutive nodes),
// stages the block's parameters and axis-factor tables in shared memory, and
// updates each direction as the fused kernel does.
template <int D, int M, bool kLive, typename RT>
__device__ __forceinline__ void prep_body(const RT* __restrict__ rec,
                                          const double* __restrict__ Tf, RT* __restrict__ cp,
                                          const Geom& g, const Units& un, const BCDev& bc,
                                          const DevMech& mech, long long n) {
  using CP = CPar<D, M>;
  const long long N = g.N;
  if (n >= N) return;
  const int tag = bc.tag ? bc.tag[n] : TAG_BULK;
  if (tag == TAG_SOLID) return;
  NodePar<D, M, RT> p;
  node_params<D, M, kLive, RT>(rec, Tf, g, un, bc, mech, n, tag, p);
#pragma unroll
  for (int b = 0; b < M; ++b) {
    cp[(CP::TH + b) * N + n] = p.th[b];
    cp[(CP::RS + b) * N + n] = p.rs[b];
#pragma unroll
    for (int d = 0; d < D; ++d) cp[(CP::V + b * D + d) * N + n] = stored(p.V[b][d]);
  }
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    cp[(CP::CF + a) * N + n] = p.cF[a];
    cp[(CP::OM1 + a) * N + n] = p.om1[a];
    cp[(CP::HH + a) * N + n] = p.hh[a];
  }
#pragma unroll
  for (int d = 0; d < D; ++d) {
    cp[(CP::U + d) * N + n] = p.u[d];
    cp[(CP::PEX + d) * N + n] = p.Pex[d];
    cp[(CP::W + d) * N + n] = p.W[d];
  }
  cp[CP::RHO * N + n] = p.rho;
  cp[CP::OM * N + n] = p.om;
  cp[CP::UL * N + n] = p.U;
  cp[CP::THETA * N + n] = p.theta;
}

constexpr int kCollNodes = kCollNodesPerBlock;   // nodes per block of k_coll (the lanes)
constexpr int kCollTPN = 9;      // threads per node (warps per block)
constexpr int kColl32Blocks = 3; // FP32 blocks per SM the registers are held to

// shared-memory entries per node of k_coll: parameters, energy factors,
// species axis-factor tables
template <int D, int M, typename RT> constexpr int coll_smem_entries();

// Layout of k_coll's shared memory in FP64 (8-byte entries per node): the FP64
// axis factors E of the stored species' equilibria (x: times hh_a), float-float
// tables (packed pairs) of the Stefan-Maxwell term's factors, the extended
// equilibrium's and the energy factors, the species coefficients cF (a pair with
// an exponent of its own, cF being as small as Y_a) and 1 - 2 beta, and the
// scalars.  The pairs:
//   e_d(c), the axis factor of psi(u, theta_b), and t_d(c) = s_d(c) - e_d(c),
//   s_d(c) that of psi(u + V_b, theta_b), formed without cancellation from
//   V_b (t(0) = -V (2u + V), t(+-1) = (V (2u + V) +- V)/2); for x, s and t
//   times -rho_b.
template <int D, int M> struct Coll64 {
  static constexpr int E = 0, F = E + (M - 1) * D * 3;
  static constexpr int EX = F + M * D * 6, AF = EX + 3 * D, BF = AF + 3 * D;
  static constexpr int CF = BF + 3 * D, OM1 = CF + M - 1;
  static constexpr int RHO = OM1 + M - 1, OM = RHO + 1, U = OM + 1, W = U + 1;
  static constexpr int CE = W + D, N = CE + M / 2;       // CE: M - 1 ints per node
  static constexpr int e(int a, int d, int c) { return E + (a * D + d) * 3 + c + 1; }
  // first of a pair: x: -rho s(c), then -rho t(c); y, z: e(c), then t(c)
  static constexpr int f(int b, int d, int c) { return F + (b * D + d) * 6 + c + 1; }
};
// ... and in FP32 (4-byte entries per node): per axis d and c the species' axis
// factors e of psi(u, theta_b) and s of psi(u + V_b, theta_b) (x: times rho_b, and
// e times hh_b), the factors of the extended equilibrium and the energy
// factors, then the species coefficients cF and 1 - 2 beta and the scalars.
template <int D, int M> struct Coll32 {
  static constexpr int E = 0, S = E + D * 3 * M, H = S + D * 3 * M;
  static constexpr int EX = H + 3 * M, AF = EX + 3 * D, BF = AF + 3 * D;
  static constexpr int CF = BF + 3 * D, OM1 = CF + M - 1;
  static constexpr int RHO = OM1 + M - 1, OM = RHO + 1, U = OM + 1, W = U + 1;
  static constexpr int N = W + D;
  static constexpr int f(int b, int d, int c) { return (d * 3 + c + 1) * M + b; }
};
template <int D, int M, typename RT> constexpr int coll_smem_entries() {
  return sizeof(RT) == 8 ? Coll64<D, M>::N + kCollTPN * (M + 1) : Coll32<D, M>::N;
}

// Asynchronous 8-byte copy from global to this thread's shared memory (8-byte
// aligned), and the wait for this thread's copies.
__device__ __forceinline__ void copy_async8(double* to, const double* from) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(to)),
               "l"(from)
               : "memory");
}
__device__ __forceinline__ void copy_async_wait() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// The FP64 collision of one block of TPN warps, 32 nodes (lane = node), the
// directions dealt to the warps as in coll_block.
//
// What bounds it is the FP64 pipe: an FP64 instruction occupies an SM quarter
// for 64 cycles, an FP32 one for 1.  So only what must carry 53 bits runs
// there: per population the equilibrium and the relaxation (two fused
// multiply-adds for a species, f om1 + cF F + psi hh with hh folded into the
// (c_x, c_y) part), f^ex, g^eq and the axis factors.  The Stefan-Maxwell term
//   F_a = sum_b K_ab d_b,  d_b = rho_b (psi(u) - psi(u + V_b)),
// half of the FP64 work before, is a correction of the relative size of V:
// float-float (48 bits) differences and sums of it stay below FP64's
// rounding of the population.  d_b is formed from the differences t of the
// axis factors, without the cancellation of psi(u) - psi(u + V_b):
//   -d_b / rho_b = (t_x e_y + s_x t_y) e_z + s_x s_y t_z.
template <int D, int M, typename S, int TPN>
__device__ __forceinline__ void coll_block64(const S* __restrict__ src, S* __restrict__ dst,
                                             const double* __restrict__ cp, const Geom& g,
                                             const BCDev& bc, const DevMech& mech,
                                             long long n0, double* __restrict__ sm) {
  using CP = CPar<D, M>;
  using T = Coll64<D, M>;
  constexpr int Q = Lat<D>::Q;
  const long long N = g.N;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long n = n0 + lane;
  const int tag = n < N ? (bc.tag ? bc.tag[n] : TAG_BULK) : TAG_SOLID;
  const bool valid = tag != TAG_SOLID;
  double* const s = sm + lane;
  int* const ce = reinterpret_cast<int*>(sm + T::CE * kCollNodes) + lane;
  const int x = (int)(n % g.nx);
  const int y = (int)((n / g.nx) % g.ny);
  const int z = (int)(n / ((long long)g.nx * g.ny));
  constexpr int NZ = D == 3 ? 3 : 1;
  constexpr int CH = (Q + TPN - 1) / TPN;
  const int k0 = w * CH, k1 = min(k0 + CH, Q);
  // This lane's slots of the warp's buffer hold the populations of one
  // direction; the next direction's are copied into them once all are read (a
  // barrier of the warp between: nothing else orders a copy after its own
  // thread's loads), the first direction's while the tables are built.
  double* const fin = sm + T::N * kCollNodes + w * (M + 1) * kCollNodes + lane;
  const long long stride = Q * (tag >= 0 ? (long long)bc.n_if : N);
  auto first_of = [&](int i) {
    return tag >= 0 ? static_cast<const double*>(bc.pops) + (long long)i * bc.n_if + tag
                    : src + i * N + node_shift<D>(x, y, z, i, -1, g);
  };
  if (valid && k0 < k1) {
    const double* p = first_of(k0 / NZ + 9 * (k0 % NZ));
#pragma unroll
    for (int l = 0; l <= M; ++l, p += stride) copy_async8(fin + l * kCollNodes, p);
  }
  if (valid) {
    auto G = [&](int f) { return __ldcg(cp + (long long)f * N + n); };
    for (int e = w; e < M * D; e += TPN) {
      const int b = e / D, d = e % D;
      const double u = G(CP::U + d), th = G(CP::TH + b);
      const ff V = ff_unpack(G(CP::V + b * D + d));
      const ff mr = d == 0 ? -ff_of_double(G(CP::RS + b)) : ff(1.f);
      const double hh = d == 0 && b < M - 1 ? G(CP::HH + b) : 1.0;
      const double P = fma(u, u, th), hu = 0.5 * u;
      const double E[3] = {fma(0.5, P, -hu), 1.0 - P, fma(0.5, P, hu)};
      ff uf = ff_of_double(u);
      uf = ff(2.f * uf.hi, 2.f * uf.lo) + V;
      const ff dP = V * uf;                     // V (2u + V)
      const ff t0 = -dP, tp = dP + V, tm = dP - V;
      const ff t[3] = {ff(0.5f * tm.hi, 0.5f * tm.lo), t0, ff(0.5f * tp.hi, 0.5f * tp.lo)};
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (b < M - 1) s[(T::E + e * 3 + c) * kCollNodes] = d == 0 ? hh * E[c] : E[c];
        const ff ef = ff_of_double(E[c]);
        const ff first = d == 0 ? mr * (ef + t[c]) : ef;
        const ff second = d == 0 ? mr * t[c] : t[c];
        s[(T::F + e * 6 + c) * kCollNodes] = ff_pack(first);
        s[(T::F + e * 6 + 3 + c) * kCollNodes] = ff_pack(second);
      }
    }
    if (w == TPN - 1) {
      double u[D], Af[D][3], Bf[D][3];
#pragma unroll
      for (int d = 0; d < D; ++d) u[d] = G(CP::U + d);
      energy_factors<D, double>(u, G(CP::THETA), Af, Bf);
#pragma unroll
      for (int d = 0; d < D; ++d) {
        const double px = G(CP::PEX + d);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          s[(T::AF + d * 3 + k) * kCollNodes] = Af[d][k];
          s[(T::BF + d * 3 + k) * kCollNodes] = Bf[d][k];
          s[(T::EX + d * 3 + k) * kCollNodes] = psi1<double>(k - 1, u[d], px);
        }
        s[(T::W + d) * kCollNodes] = G(CP::W + d);
      }
      s[T::RHO * kCollNodes] = G(CP::RHO);
      s[T::OM * kCollNodes] = G(CP::OM);
      s[T::U * kCollNodes] = G(CP::UL);
    }
    for (int a = w; a < M - 1; a += TPN) {
      int e;
      s[(T::CF + a) * kCollNodes] = ff_pack(ff_mantissa(G(CP::CF + a), e));
      ce[a * kCollNodes] = e + mech.K_exp;
      s[(T::OM1 + a) * kCollNodes] = G(CP::OM1 + a);
    }
  }
  __syncthreads();
  const unsigned lanes = __ballot_sync(0xffffffffu, valid);
  if (!valid) return;
  auto P = [&](int f) { return s[f * kCollNodes]; };
  auto PF = [&](int f) { return ff_unpack(s[f * kCollNodes]); };
  if (k0 >= k1) return;
  ff A[M], SS[M];              // t_x e_y + s_x t_y and s_x s_y, times -rho_b
  double eh[M - 1];            // hh_a e_x e_y
  double fxy = 0.0, gP = 0.0, gQ = 0.0;
  const double rho = P(T::RHO), om = P(T::OM);
  int jcur = -1;
#pragma unroll 1
  for (int k = k0; k < k1; ++k) {
    const int j = k / NZ, i = j + 9 * (k % NZ);
    const int cx = cvel(j, 0), cy = cvel(j, 1), cz = D == 3 ? k % NZ - 1 : 0;
    // the next direction
    const bool more = k + 1 < k1;
    const double* pn = more ? first_of((k + 1) / NZ + 9 * ((k + 1) % NZ)) : src;
    if (j != jcur) {
      jcur = j;
#pragma unroll
      for (int b = 0; b < M; ++b) {
        const ff sx = PF(T::f(b, 0, cx)), tx = PF(T::f(b, 0, cx) + 3);
        const ff ey = PF(T::f(b, 1, cy)), ty = PF(T::f(b, 1, cy) + 3);
        ff v = tx * ey;
        ff_fma_acc(v, sx, ty);
        A[b] = ff_norm(v);
        if constexpr (D == 3) {
          ff sy = ey;
          ff_acc(sy, ty);
          SS[b] = sx * ff_norm(sy);
        }
        if (b < M - 1) eh[b] = P(T::e(b, 0, cx)) * P(T::e(b, 1, cy));
      }
      fxy = rho * P(T::EX + cx + 1) * P(T::EX + 3 + cy + 1);
      const double ax = P(T::AF + cx + 1), ay = P(T::AF + 3 + cy + 1);
      gP = ax * ay;
      gQ = fma(P(T::U), gP, fma(P(T::BF + cx + 1), ay, ax * P(T::BF + 3 + cy + 1)));
    }
    ff dd[M];
#pragma unroll
    for (int b = 0; b < M; ++b) {
      if constexpr (D == 3) {
        ff v = A[b] * PF(T::f(b, 2, cz));
        ff_fma_acc(v, SS[b], PF(T::f(b, 2, cz) + 3));
        dd[b] = ff_norm(v);
      } else {
        dd[b] = A[b];
      }
    }
    copy_async_wait();
    double in[M + 1];
#pragma unroll
    for (int l = 0; l <= M; ++l) in[l] = fin[l * kCollNodes];
    __syncwarp(lanes);
    if (more) {
#pragma unroll
      for (int l = 0; l <= M; ++l, pn += stride) copy_async8(fin + l * kCollNodes, pn);
    }
#pragma unroll
    for (int a = 0; a < M - 1; ++a) {
      ff F;
#pragma unroll
      for (int b = 0; b < M; ++b)
        if (b != a) ff_fma_acc(F, mech.K_f[a][b], dd[b]);
      F = PF(T::CF + a) * ff_norm(F);
      const double ez = D == 3 ? P(T::e(a, D - 1, cz)) : 1.0;
      const double base = fma(in[a], P(T::OM1 + a), double_join(F, ce[a * kCollNodes]));
      dst[(long long)(a * Q + i) * N + n] = D == 3 ? fma(eh[a], ez, base) : eh[a] + base;
    }
    double fex = fxy, geq = gQ;
    if constexpr (D == 3) {
      fex *= P(T::EX + 6 + cz + 1);
      geq = fma(P(T::AF + 6 + cz + 1), gQ, gP * P(T::BF + 6 + cz + 1));
    }
    const double fm = in[M - 1];
    dst[(long long)((M - 1) * Q + i) * N + n] = fma(om, fex - fm, fm);
    const double gm = in[M];
    double gn = fma(om, fma(rho, geq, -gm), gm);
    if (csq(i, D) == 1) {
#pragma unroll
      for (int d = 0; d < D; ++d)
        if (cvel(i, d) != 0) gn = fma(cvel(i, d) > 0 ? 0.5 : -0.5, P(T::W + d), gn);
    }
    dst[(long long)(M * Q + i) * N + n] = gn;
  }
}

// One block of TPN warps: nodes n0 .. n0 + 31.  sm holds coll_smem_entries *
// kCollNodes.  The Q directions, taken in the order k = 0 .. Q - 1 with
// direction (k / NZ) + 9 (k % NZ) (NZ = 3 in 3D: the directions of one
// (c_x, c_y) pair in a row), are dealt to the warps in contiguous chunks.
//
// FP32 lattice arithmetic: bound by instruction issue (of 744 instructions per
// direction and warp, most formed addresses and shared (c_x, c_y) products
// again; now ~250), then by HBM.  The products with rho_b, hh_b and of x and y
// are taken once per (c_x, c_y) pair, a species update is two multiply-adds
// beside its Stefan-Maxwell sum, and every lattice's address is the
// direction's plus a constant stride.
template <int D, int M, typename S, typename RT, int TPN = kCollTPN>
__device__ __forceinline__ void coll_block(const S* __restrict__ src, S* __restrict__ dst,
                                           const RT* __restrict__ cp, const Geom& g,
                                           const BCDev& bc, const DevMech& mech, long long n0,
                                           RT* __restrict__ sm) {
  if constexpr (sizeof(RT) == 8) {
    coll_block64<D, M, S, TPN>(src, dst, cp, g, bc, mech, n0, sm);
  } else {
    using CP = CPar<D, M>;
    using T = Coll32<D, M>;
    constexpr int Q = Lat<D>::Q, CN = kCollNodes;
    const long long N = g.N;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long n = n0 + lane;
    const int tag = n < N ? (bc.tag ? bc.tag[n] : TAG_BULK) : TAG_SOLID;
    const bool valid = tag != TAG_SOLID;
    RT* const s = sm + lane;
    const int x = (int)(n % g.nx);
    const int y = (int)((n / g.nx) % g.ny);
    const int z = (int)(n / ((long long)g.nx * g.ny));
    constexpr int NZ = D == 3 ? 3 : 1;
    constexpr int CH = (Q + TPN - 1) / TPN;
    const int k0 = w * CH, k1 = min(k0 + CH, Q);
    // populations entering direction i of lattice l (pop_in)
    const long long ls = (long long)Q * N;              // stride of a lattice
    auto load = [&](long long sn, int i, RT (&fin)[M + 1]) {
      if (tag >= 0) {
        const RT* p = static_cast<const RT*>(bc.pops) + (long long)i * bc.n_if + tag;
        const long long st = (long long)Q * bc.n_if;
#pragma unroll
        for (int l = 0; l <= M; ++l, p += st) fin[l] = *p;
      } else {
        const S* p = src + (long long)i * N + sn;
#pragma unroll
        for (int l = 0; l <= M; ++l, p += ls)
          fin[l] = Codec<S>::template dec<RT>(__ldg(p), g.codec, l * Q + i);
      }
    };
    RT fin[M + 1];
#pragma unroll
    for (int l = 0; l <= M; ++l) fin[l] = RT(0);
    if (valid) {
      // the first direction's populations are in flight while the block's
      // tables are built
      if (k0 < k1) {
        const int i = k0 / NZ + 9 * (k0 % NZ);
        load(node_shift<D>(x, y, z, i, -1, g), i, fin);
      }
      auto P = [&](int f) { return __ldcg(cp + (long long)f * N + n); };
      for (int e = w; e < M * D; e += TPN) {
        const int b = e / D, d = e % D;
        const RT u = P(CP::U + d), th = P(CP::TH + b), us = u + P(CP::V + b * D + d);
        const RT pe = th + u * u, ps = th + us * us;
        const RT r = d == 0 ? P(CP::RS + b) : RT(1);
        const RT ee[3] = {RT(0.5) * (pe - u), RT(1) - pe, RT(0.5) * (pe + u)};
        const RT ss[3] = {RT(0.5) * (ps - us), RT(1) - ps, RT(0.5) * (ps + us)};
        const RT hh = d == 0 && b < M - 1 ? P(CP::HH + b) : RT(0);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          s[(T::E + T::f(b, d, c - 1)) * CN] = r * ee[c];
          s[(T::S + T::f(b, d, c - 1)) * CN] = r * ss[c];
          if (d == 0) s[(T::H + c * M + b) * CN] = hh * ee[c];
        }
      }
      if (w == TPN - 1) {
        RT u[D], Af[D][3], Bf[D][3];
#pragma unroll
        for (int d = 0; d < D; ++d) u[d] = P(CP::U + d);
        energy_factors<D, RT>(u, P(CP::THETA), Af, Bf);
#pragma unroll
        for (int d = 0; d < D; ++d) {
          const RT px = P(CP::PEX + d);
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            s[(T::AF + d * 3 + k) * CN] = Af[d][k];
            s[(T::BF + d * 3 + k) * CN] = Bf[d][k];
            s[(T::EX + d * 3 + k) * CN] = psi1<RT>(k - 1, u[d], px);
          }
          s[(T::W + d) * CN] = P(CP::W + d);
        }
        s[T::RHO * CN] = P(CP::RHO);
        s[T::OM * CN] = P(CP::OM);
        s[T::U * CN] = P(CP::UL);
      }
      for (int a = w; a < M - 1; a += TPN) {
        s[(T::CF + a) * CN] = P(CP::CF + a);
        s[(T::OM1 + a) * CN] = P(CP::OM1 + a);
      }
    }
    __syncthreads();
    if (!valid || k0 >= k1) return;
    RT re[M], rss[M], eh[M - 1];     // rho_b e_x e_y, rho_b s_x s_y, hh_a e_x e_y
    RT fxy = RT(0), gP = RT(0), gQ = RT(0);
    const RT rho = s[T::RHO * CN], om = s[T::OM * CN];
    int jcur = -1;
#pragma unroll 1
    for (int k = k0; k < k1; ++k) {
      const int j = k / NZ, i = j + 9 * (k % NZ);
      const int cx = cvel(j, 0), cy = cvel(j, 1), cz = D == 3 ? k % NZ - 1 : 0;
      if (j != jcur) {
        jcur = j;
        const RT *ex = s + (T::E + T::f(0, 0, cx)) * CN, *ey = s + (T::E + T::f(0, 1, cy)) * CN;
        const RT *sx = s + (T::S + T::f(0, 0, cx)) * CN, *sy = s + (T::S + T::f(0, 1, cy)) * CN;
        const RT* hx = s + (T::H + (cx + 1) * M) * CN;
#pragma unroll
        for (int b = 0; b < M; ++b) {
          const RT e = ey[b * CN];
          re[b] = ex[b * CN] * e;
          rss[b] = sx[b * CN] * sy[b * CN];
          if (b < M - 1) eh[b] = hx[b * CN] * e;
        }
        fxy = rho * s[(T::EX + cx + 1) * CN] * s[(T::EX + 3 + cy + 1) * CN];
        const RT ax = s[(T::AF + cx + 1) * CN], ay = s[(T::AF + 3 + cy + 1) * CN];
        gP = ax * ay;
        gQ = s[T::U * CN] * gP + s[(T::BF + cx + 1) * CN] * ay + ax * s[(T::BF + 3 + cy + 1) * CN];
      }
      RT dd[M], pe[M - 1];
      if constexpr (D == 3) {
        const RT *ez = s + (T::E + T::f(0, 2, cz)) * CN, *sz = s + (T::S + T::f(0, 2, cz)) * CN;
#pragma unroll
        for (int b = 0; b < M; ++b) {
          const RT e = ez[b * CN];
          dd[b] = re[b] * e - rss[b] * sz[b * CN];
          if (b < M - 1) pe[b] = eh[b] * e;
        }
      } else {
#pragma unroll
        for (int b = 0; b < M; ++b) {
          dd[b] = re[b] - rss[b];
          if (b < M - 1) pe[b] = eh[b];
        }
      }
      S* out = dst + (long long)i * N + n;
      const RT f = fin[M - 1], gv = fin[M];
#pragma unroll
      for (int a = 0; a < M - 1; ++a) {
        RT F = RT(0);
#pragma unroll
        for (int b = 0; b < M; ++b)
          if (b != a) F += kcoef<RT>(mech, a, b) * dd[b];
        const RT fn = fin[a] * s[(T::OM1 + a) * CN] + (pe[a] + s[(T::CF + a) * CN] * F);
        *out = Codec<S>::enc(fn, g.codec, a * Q + i);
        out += ls;
      }
      // the next direction's populations (the last direction's again)
      const int kn = min(k + 1, k1 - 1), in = kn / NZ + 9 * (kn % NZ);
      load(node_shift<D>(x, y, z, in, -1, g), in, fin);
      RT fex = fxy, geq = gQ;
      if constexpr (D == 3) {
        fex *= s[(T::EX + 6 + cz + 1) * CN];
        geq = s[(T::AF + 6 + cz + 1) * CN] * gQ + gP * s[(T::BF + 6 + cz + 1) * CN];
      }
      *out = Codec<S>::enc(f + om * (fex - f), g.codec, (M - 1) * Q + i);
      RT gn = gv + om * (rho * geq - gv);
      if (csq(i, D) == 1) {
#pragma unroll
        for (int d = 0; d < D; ++d)
          if (cvel(i, d) != 0) gn += (cvel(i, d) > 0 ? RT(0.5) : RT(-0.5)) * s[(T::W + d) * CN];
      }
      out[ls] = Codec<S>::enc(gn, g.codec, M * Q + i);
    }
  }
}

#include "lbm_bnode.cuh"

// ---------------------------------------------------------------------------
// Single-domain kernels: one thread per node (moments, collision), one thread
// per interface node (k_bnode: boundary reconstruction and record).
// Node sets: every node, or the nodes without boundary reconstruction (the
// bulk; the interface nodes run on a side stream concurrent with it).
enum { NODES_ALL = 0, NODES_BULK = 1 };

template <int D, int M, typename S, typename RT>
__global__ void __launch_bounds__(128, kMoments1MinBlocks<RT>)
k_moments(const S* __restrict__ src, RT* __restrict__ rec, double* __restrict__ Tf,
          int* __restrict__ status, const __grid_constant__ Geom g,
          const __grid_constant__ Units un, const __grid_constant__ BCDev bc,
          const __grid_constant__ DevMech mech, int node_set) {
  // node_set: NODES_ALL or NODES_BULK
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (node_set == NODES_BULK && bc.tag && n < g.N && bc.tag[n] >= 0) return;
  moments_body<D, M, S, RT>(src, rec, Tf, status, g, un, bc, mech, n, moments_static<M, RT>());
}

// The reaction sub-steps of the interface nodes from entry `first` of their
// list, after the boundary kernel: kIfLanes lanes per node, 128 threads per block.
constexpr int kIfLanes = 8;
static_assert(128 / kIfLanes == kIfChemNodesPerBlock, "the interface-chemistry grid");
template <int D, int M, typename RT>
__device__ __forceinline__ void chem_entry(RT* rec, const double* Tf, int* status, long long N,
                                           const Units& un, const DevMech& m, long long first,
                                           const int* if_node, int n_if) {
  const int lane = threadIdx.x & 31;
  const long long k = first + threadIdx.x / kIfLanes;
  if (k >= n_if) return;                                // the whole group leaves
  const unsigned gmask = ((1u << kIfLanes) - 1u) << (lane & ~(kIfLanes - 1));
  chem_lanes_body<D, M, RT, kIfLanes>(rec, Tf, status, N, un, m, if_node[k],
                                      lane & (kIfLanes - 1), gmask);
}

template <int D, int M, typename RT>
__global__ void __launch_bounds__(128)
k_chem(RT* __restrict__ rec, const double* __restrict__ Tf, int* __restrict__ status,
       long long N, const __grid_constant__ Units un, const DevMech* __restrict__ mech,
       const int* __restrict__ if_node, int n_if) {
  chem_entry<D, M, RT>(rec, Tf, status, N, un, *mech, blockIdx.x * (128LL / kIfLanes), if_node,
                       n_if);
}

// moments and reaction sub-steps, L lanes per node, 128 threads per block,
// over every node or the nodes without boundary reconstruction
template <int D, int M, typename S, typename RT, int L>
__global__ void __launch_bounds__(128)
k_mchem(const S* __restrict__ src, RT* __restrict__ rec, double* __restrict__ Tf,
        int* __restrict__ status, const __grid_constant__ Geom g,
        const __grid_constant__ Units un, const __grid_constant__ BCDev bc,
        const __grid_constant__ DevMech mech, const DevMech* __restrict__ mech_g,
        int node_set) {
  const int lane = threadIdx.x & 31;
  const long long n = blockIdx.x * (128LL / L) + threadIdx.x / L;
  if (n >= g.N) return;                                  // the whole group leaves
  const int tag = bc.tag ? bc.tag[n] : TAG_BULK;
  if (tag == TAG_SOLID || (node_set == NODES_BULK && tag >= 0)) return;
  const unsigned gmask = ((1u << L) - 1u) << (lane & ~(L - 1));
  mchem_body<D, M, S, RT, L>(src, rec, Tf, status, g, un, bc, mech, *mech_g, n, tag,
                             lane & (L - 1), gmask);
}

template <int D, int M, typename S, typename RT>
__global__ void __launch_bounds__(128)
k_collide(const S* __restrict__ src, S* __restrict__ dst, const RT* __restrict__ rec,
          const double* __restrict__ Tf, int* __restrict__ status,
          const __grid_constant__ Geom g, const __grid_constant__ Units un,
          const __grid_constant__ BCDev bc, const __grid_constant__ DevMech mech) {
  collide_body<D, M, false, S, RT>(src, dst, rec, Tf, status, g, un, bc, mech,
                            blockIdx.x * (long long)blockDim.x + threadIdx.x);
}

template <int D, int M, typename RT>
__global__ void __launch_bounds__(128, kPrepMinBlocks<RT>)
k_prep(const RT* __restrict__ rec, const double* __restrict__ Tf, RT* __restrict__ cp,
       const __grid_constant__ Geom g, const __grid_constant__ Units un,
       const __grid_constant__ BCDev bc, const __grid_constant__ DevMech mech) {
  prep_body<D, M, false, RT>(rec, Tf, cp, g, un, bc, mech,
                      blockIdx.x * (long long)blockDim.x + threadIdx.x);
}

// 288-thread blocks: FP64 two per SM (96 registers, 97 KB of shared memory each),
// FP32 three (72 registers; two or four: 46.4 and 45.7 ms per 24 steps of the
// 600x40x40 tube against 45.4)
template <int D, int M, typename S, typename RT>
__global__ void __launch_bounds__(32 * kCollTPN, sizeof(RT) == 4 ? kColl32Blocks : 2)
k_coll(const S* __restrict__ src, S* __restrict__ dst, const RT* __restrict__ cp,
       const __grid_constant__ Geom g, const __grid_constant__ BCDev bc,
       const __grid_constant__ DevMech mech) {
  extern __shared__ __align__(16) unsigned char coll_raw[];
  coll_block<D, M, S, RT>(src, dst, cp, g, bc, mech, blockIdx.x * (long long)kCollNodes,
                          reinterpret_cast<RT*>(coll_raw));
}

// One thread per interface node: reconstruction and record (lbm_bnode.cuh);
// the interface nodes' reaction sub-steps follow in k_chem.
template <int D, int M, typename S>
__global__ void __launch_bounds__(kBnd, kBnodeMinBlocks<S>)
k_bnode(const S* __restrict__ src, const __grid_constant__ BCDev bc, double* __restrict__ Tf,
        int* __restrict__ status, const __grid_constant__ Geom g,
        const __grid_constant__ Units un, const __grid_constant__ DevMech mech,
        typename ComputeType<S>::type* __restrict__ rec) {
  using R = typename ComputeType<S>::type;
  extern __shared__ __align__(16) unsigned char bnd_raw[];
  const int k = blockIdx.x * kBnd + threadIdx.x;
  if (k >= bc.n_if) return;
  bnode_body<D, M, S, R>(src, bc, rec, Tf, status, g, un, mech, k,
                         reinterpret_cast<R*>(bnd_raw) + threadIdx.x,
                         reinterpret_cast<long long*>(
                             bnd_raw + sizeof(R) * bnode_col_entries<D, M>() * kBnd) +
                             threadIdx.x);
}

// The interface nodes with a warp each: reconstruction, record and reaction
// sub-steps (lbm_bnode.cuh).
template <int D, int M, typename S>
__global__ void __launch_bounds__(32 * kBnodeWarps)
k_bnode_warp(const S* __restrict__ src, const __grid_constant__ BCDev bc,
             double* __restrict__ Tf, int* __restrict__ status, const __grid_constant__ Geom g,
             const __grid_constant__ Units un, const DevMech* __restrict__ mech,
             typename ComputeType<S>::type* __restrict__ rec) {
  using R = typename ComputeType<S>::type;
  __shared__ R ws[kBnodeWarps][WB<D, M>::N];
  const int w = threadIdx.x >> 5, k = blockIdx.x * kBnodeWarps + w;
  if (k >= bc.n_if) return;
  using CT = typename ChemType<R>::type;
  ChemSlice<M, CT, 32 * kBnodeWarps> cs(chem_static_slice<M, CT, 32 * kBnodeWarps>(), threadIdx.x);
  bnode_warp<D, M, S, R>(src, bc, rec, Tf, status, g, un, *mech, k, ws[w], threadIdx.x & 31, cs);
}

// ---------------------------------------------------------------------------
// Batched kernels: the grid is the concatenation of every domain's tiles; a
// block finds its domain by binary search over the domains' first blocks.
enum { GRID_NODE = 0, GRID_BOUNDARY = 1, GRID_CHEM = 2, GRID_COLL = 3, GRID_BNODE = 4 };
__device__ __forceinline__ int domain_of_block(const DomainDev* __restrict__ d, int ndom,
                                               int b, int grid) {
  int lo = 0, hi = ndom - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    const int first = grid == GRID_BOUNDARY ? d[mid].bblock_begin
                      : grid == GRID_CHEM   ? d[mid].cblock_begin
                      : grid == GRID_COLL   ? d[mid].kblock_begin
                      : grid == GRID_BNODE  ? d[mid].tblock_begin
                                            : d[mid].block_begin;
    if (first <= b) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Every batched kernel walks its grid's blocks b = blockIdx.x, + gridDim.x,
// ... below nblk: launched with one block per tile it runs each tile once;
// launched persistent (a grid sized to the blocks resident on the GPU) each
// block processes several tiles in turn.
//
// The block's domain descriptor is copied to shared memory whenever the
// block moves to another domain (k block-uniform, every thread calls it),
// so the bodies read its fields from shared memory rather than reloading
// them from global memory around every store.
struct BlockDomain {
  unsigned char* raw;   // __shared__ storage of sizeof(DomainDev) bytes
  int cur = -1;
  __device__ const DomainDev& get(const DomainDev* __restrict__ doms, int k) {
    if (k != cur) {
      __syncthreads();   // the previous domain's readers are done
      const unsigned* src = reinterpret_cast<const unsigned*>(doms + k);
      unsigned* dst = reinterpret_cast<unsigned*>(raw);
      for (int i = threadIdx.x; i < (int)(sizeof(DomainDev) / 4); i += blockDim.x)
        dst[i] = src[i];
      __syncthreads();
      cur = k;
    }
    return *reinterpret_cast<const DomainDev*>(raw);
  }
};
static_assert(sizeof(DomainDev) % 4 == 0, "domain descriptor copied in 4-byte words");
#define LBM_BLOCK_DOMAIN(name)                                          \
  __shared__ __align__(16) unsigned char name##_raw[sizeof(DomainDev)]; \
  BlockDomain name{name##_raw}
template <int D, int M, typename S, typename RT>
__global__ void __launch_bounds__(128, kMomentsMinBlocks)
k_moments_batch(const DomainDev* __restrict__ doms, int ndom, int parity, int node_set,
                int nblk) {
  LBM_BLOCK_DOMAIN(bd);
  // node_set: NODES_ALL or NODES_BULK (the interface nodes' records come from
  // k_bnode_batch)
  for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
    const DomainDev& d = bd.get(doms, domain_of_block(doms, ndom, b, GRID_NODE));
    const int c = d.cur0 ^ parity;
    const long long n = (b - d.block_begin) * (long long)blockDim.x + threadIdx.x;
    if (node_set == NODES_BULK && d.bc.tag && n < d.g.N && d.bc.tag[n] >= 0) continue;
    moments_body<D, M, S, RT>(static_cast<const S*>(d.pops[c]), static_cast<RT*>(d.rec), d.Tf,
                              d.status, d.g, d.un, d.bc, *d.mech, n, moments_static<M, RT>());
  }
}

// k_chem over the interface nodes of several handles
template <int D, int M, typename RT>
__global__ void __launch_bounds__(128)
k_chem_batch(const DomainDev* __restrict__ doms, int ndom, int nblk) {
  LBM_BLOCK_DOMAIN(bd);
  for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
    const DomainDev& d = bd.get(doms, domain_of_block(doms, ndom, b, GRID_BOUNDARY));
    chem_entry<D, M, RT>(static_cast<RT*>(d.rec), d.Tf, d.status, d.g.N, d.un, *d.mech,
                         (b - d.bblock_begin) * (128LL / kIfLanes), d.bc.if_node, d.bc.n_if);
  }
}

// the chemistry grid (128 / L nodes per block)
template <int D, int M, typename S, typename RT, int L>
__global__ void __launch_bounds__(128)
k_mchem_batch(const DomainDev* __restrict__ doms, int ndom, int parity, int node_set,
              int nblk) {
  LBM_BLOCK_DOMAIN(bd);
  for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
    const DomainDev& d = bd.get(doms, domain_of_block(doms, ndom, b, GRID_CHEM));
    const int c = d.cur0 ^ parity;
    const int lane = threadIdx.x & 31;
    const long long n = (b - d.cblock_begin) * (128LL / L) + threadIdx.x / L;
    if (n >= d.g.N) continue;
    const int tag = d.bc.tag ? d.bc.tag[n] : TAG_BULK;
    if (tag == TAG_SOLID || (node_set == NODES_BULK && tag >= 0)) continue;
    const unsigned gmask = ((1u << L) - 1u) << (lane & ~(L - 1));
    mchem_body<D, M, S, RT, L>(static_cast<const S*>(d.pops[c]), static_cast<RT*>(d.rec), d.Tf,
                               d.status, d.g, d.un, d.bc, *d.mech, *d.mech, n, tag,
                               lane & (L - 1), gmask);
  }
}

template <int D, int M, typename S, typename RT>
__global__ void __launch_bounds__(128)
k_collide_batch(const DomainDev* __restrict__ doms, int ndom, int parity, int nblk) {
  LBM_BLOCK_DOMAIN(bd);
  for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
    const DomainDev& d = bd.get(doms, domain_of_block(doms, ndom, b, GRID_NODE));
    const int c = d.cur0 ^ parity;
    collide_body<D, M, false, S, RT>(static_cast<const S*>(d.pops[c]),
                              static_cast<S*>(const_cast<void*>(d.pops[1 - c])),
                              static_cast<const RT*>(d.rec), d.Tf, d.status, d.g, d.un, d.bc,
                              *d.mech, (b - d.block_begin) * (long long)blockDim.x + threadIdx.x);
  }
}

template <int D, int M, typename RT>
__global__ void __launch_bounds__(128, kPrepMinBlocks<RT>)
k_prep_batch(const DomainDev* __restrict__ doms, int ndom, int nblk) {
  LBM_BLOCK_DOMAIN(bd);
  for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
    const DomainDev& d = bd.get(doms, domain_of_block(doms, ndom, b, GRID_NODE));
    prep_body<D, M, false, RT>(static_cast<const RT*>(d.rec), d.Tf, static_cast<RT*>(d.cpar), d.g,
                        d.un, d.bc, *d.mech,
                        (b - d.block_begin) * (long long)blockDim.x + threadIdx.x);
  }
}

template <int D, int M, typename S, typename RT>
__global__ void __launch_bounds__(32 * kCollTPN, sizeof(RT) == 4 ? kColl32Blocks : 2)
k_coll_batch(const DomainDev* __restrict__ doms, int ndom, int parity, int nblk) {
  LBM_BLOCK_DOMAIN(bd);
  extern __shared__ __align__(16) unsigned char coll_raw[];
  for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
    const DomainDev& d = bd.get(doms, domain_of_block(doms, ndom, b, GRID_COLL));
    const int c = d.cur0 ^ parity;
    // the previous tile's threads are done with the shared memory
    if (b != blockIdx.x) __syncthreads();
    coll_block<D, M, S, RT>(static_cast<const S*>(d.pops[c]),
                            static_cast<S*>(const_cast<void*>(d.pops[1 - c])),
                            static_cast<const RT*>(d.cpar), d.g, d.bc, *d.mech,
                            (b - d.kblock_begin) * (long long)kCollNodes,
                            reinterpret_cast<RT*>(coll_raw));
  }
}

// One thread per interface node over every domain (the batched k_bnode).
template <int D, int M, typename S>
__global__ void __launch_bounds__(kBnd, kBnodeMinBlocks<S>)
k_bnode_batch(const DomainDev* __restrict__ doms, int ndom, int parity, int nblk) {
  LBM_BLOCK_DOMAIN(bd);
  using R = typename ComputeType<S>::type;
  extern __shared__ __align__(16) unsigned char bnd_raw[];
  R* col = reinterpret_cast<R*>(bnd_raw) + threadIdx.x;
  long long* sncol =
      reinterpret_cast<long long*>(bnd_raw + sizeof(R) * bnode_col_entries<D, M>() * kBnd) +
      threadIdx.x;
  for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
    const DomainDev& d = bd.get(doms, domain_of_block(doms, ndom, b, GRID_BNODE));
    const int k = (b - d.tblock_begin) * kBnd + threadIdx.x;
    if (k >= d.bc.n_if) continue;
    bnode_body<D, M, S, R>(static_cast<const S*>(d.pops[d.cur0 ^ parity]), d.bc,
                           static_cast<R*>(d.rec), d.Tf, d.status, d.g, d.un, *d.mech, k, col,
                           sncol);
  }
}

template <int D, int M, typename S>
__global__ void __launch_bounds__(32 * kBnodeWarps)
k_bnode_warp_batch(const DomainDev* __restrict__ doms, int ndom, int parity, int nblk) {
  LBM_BLOCK_DOMAIN(bd);
  using R = typename ComputeType<S>::type;
  using CT = typename ChemType<R>::type;
  __shared__ R ws[kBnodeWarps][WB<D, M>::N];
  ChemSlice<M, CT, 32 * kBnodeWarps> cs(chem_static_slice<M, CT, 32 * kBnodeWarps>(), threadIdx.x);
  const int w = threadIdx.x >> 5;
  for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
    const DomainDev& d = bd.get(doms, domain_of_block(doms, ndom, b, GRID_BNODE));
    const int k = (b - d.tblock_begin) * kBnodeWarps + w;
    if (k >= d.bc.n_if) continue;
    bnode_warp<D, M, S, R>(static_cast<const S*>(d.pops[d.cur0 ^ parity]), d.bc,
                           static_cast<R*>(d.rec), d.Tf, d.status, d.g, d.un, *d.mech, k, ws[w],
                           threadIdx.x & 31, cs);
  }
}

// ---------------------------------------------------------------------------
// The whole batched step as one persistent launch over a work-list (PItem,
// lbm_internal.h).  Dependencies go through sync words: a producer block
// fences its stores and then releases a count or a flag; a consumer's first
// thread acquires it (bounded by timeout_ns on the global timer, after which
// it sets the abort word and ST_TIMEOUT in the item's domain) before the
// block reads.  Data written earlier in the same launch is read only after
// such an acquire, and the reads that could meet a line fetched before its
// last write (the temperature guesses and the collision parameters) bypass
// the L1 (ld.global.cg).
// Reaction sub-steps of interface node n (Sec. 2.4 Eq. R3) by one thread,
// from the record the boundary reconstruction left (post-stream species
// densities in the increment slots), as chem_lanes_body does with lanes.
template <int D, int M, typename RT>
__device__ __forceinline__ void iface_substeps(RT* __restrict__ rec, const double* __restrict__ Tf,
                                               int* __restrict__ status, long long N,
                                               const Units& un, const DevMech& mech, long long n,
                                               void* chem_slice) {
  using RC = Rec<D, M>;
  const RT rho = __ldcg(rec + RC::RHO * N + n);
  RT usq = RT(0);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const RT ud = __ldcg(rec + (RC::U + d) * N + n);
    usq += ud * ud;
  }
  const RT ER = __ldcg(rec + RC::E * N + n);
  RT rs[M];
  RT last = rho;
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    rs[a] = __ldcg(rec + (RC::DRHO + a) * N + n);
    last -= rs[a];
  }
  rs[M - 1] = last;
  RT dr[M - 1];
  node_substeps<M, RT>(rs, rho, ER, usq, __ldcg(Tf + n), un, mech, status, chem_slice, dr);
#pragma unroll
  for (int a = 0; a < M - 1; ++a) rec[(RC::DRHO + a) * N + n] = dr[a];
}

// The interface nodes' sub-steps with one thread per node (grids with at
// least kIfChemThreadNodes interface nodes, which fill the GPU this way):
// the same arithmetic as the lane groups of k_chem without their redundant
// per-lane temperature solves.  Rate arrays in dynamic shared memory.  Measured
// with the tube's steps, eight lanes / a thread per node, us: FP64 20896 interface
// nodes 1596 / 1598, 31552 2217 / 2177, 90752 6004 / 5828; FP32 20896 529 / 553,
// 31552 739 / 742, 90752 1850 / 1767; FP32 with FP64 chemistry 20896 682 / 676.
constexpr long long kIfChemThreadNodes = 152LL * 128;

template <int D, int M, typename RT>
__global__ void __launch_bounds__(kChemThreads)
k_iface_chem(RT* __restrict__ rec, const double* __restrict__ Tf, int* __restrict__ status,
             long long N, const int* __restrict__ if_node, int n_if,
             const __grid_constant__ Units un, const DevMech* __restrict__ mech) {
  extern __shared__ __align__(16) unsigned char ic_raw[];
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (k >= n_if) return;
  iface_substeps<D, M, RT>(rec, Tf, status, N, un, *mech, if_node[k], ic_raw);
}

// The same over the interface nodes of several handles (batch plans whose
// handles hold at least kIfChemThreadNodes interface nodes in all), on the
// thread-per-interface-node grid of k_bnode_batch.
template <int D, int M, typename RT>
__global__ void __launch_bounds__(kBnd)
k_iface_chem_batch(const DomainDev* __restrict__ doms, int ndom, int nblk) {
  LBM_BLOCK_DOMAIN(bd);
  extern __shared__ __align__(16) unsigned char icb_raw[];
  for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
    const DomainDev& d = bd.get(doms, domain_of_block(doms, ndom, b, GRID_BNODE));
    const long long k = (b - d.tblock_begin) * (long long)kBnd + threadIdx.x;
    if (k >= d.bc.n_if) continue;
    iface_substeps<D, M, RT>(static_cast<RT*>(d.rec), d.Tf, d.status, d.g.N, d.un, *d.mech,
                             d.bc.if_node[k], icb_raw);
  }
}

template <typename RT> constexpr int kPersistMinBlocks = sizeof(RT) == 8 ? 2 : 3;
// a boundary item of up to this many interface nodes gives each a warp (the
// thread-per-node procedure of a 128-node item takes as long as ~15 nodes of a
// warp each)
constexpr int kPersistWarpNodes = 32;
constexpr int kPersistCollWarps = kPersistThreads / 32;

template <int D, int M, typename S, typename RT>
__global__ void __launch_bounds__(kPersistThreads, kPersistMinBlocks<RT>)
k_step_persist(const DomainDev* __restrict__ doms, int ndom, int parity,
               const PItem* __restrict__ items, int nitems, int npt, int* __restrict__ sync,
               long long timeout_ns) {
  LBM_BLOCK_DOMAIN(bd);
  using R = typename ComputeType<S>::type;
  constexpr int Q = Lat<D>::Q;
  extern __shared__ __align__(16) unsigned char ps_raw[];
  __shared__ int s_item, s_go;
  int* const next = sync;
  int* const abort_w = sync + 1;
  int* const done1 = sync + kSyncHead;
  int* const pflag = done1 + ndom;
  for (;;) {
    if (threadIdx.x == 0) {
      const int it = atomicAdd(next, 1);
      int go = it < nitems && !ld_acquire_gpu(abort_w);
      if (go) {
        const PItem w = items[it];
        if (w.kind == PI_PREP || w.kind == PI_COLLIDE)
          go = wait_at_least(done1 + w.dom, w.dep, abort_w, timeout_ns);
        else if (w.kind == PI_COLL) go = wait_at_least(pflag + w.dep, 1, abort_w, timeout_ns);
        if (!go) atomicOr(doms[w.dom].status, ST_TIMEOUT);
      }
      s_item = it;
      s_go = go;
    }
    __syncthreads();
    if (!s_go) break;
    const PItem w = items[s_item];
    const DomainDev& d = bd.get(doms, w.dom);
    const int c = d.cur0 ^ parity;
    const S* src = static_cast<const S*>(d.pops[c]);
    RT* rec = static_cast<RT*>(d.rec);
    if (w.kind == PI_BND && d.bc.n_if - w.first <= kPersistWarpNodes) {
      // few interface nodes: the block's warps take them in turn
      const int wp = threadIdx.x >> 5;
      using CT = typename ChemType<R>::type;
      R* ws = reinterpret_cast<R*>(ps_raw + ChemSlice<M, CT>::kBytes) + wp * WB<D, M>::N;
      ChemSlice<M, CT> cs(ps_raw, threadIdx.x);
      for (int k = (int)w.first + wp; k < d.bc.n_if; k += kPersistThreads / 32)
        bnode_warp<D, M, S, R>(src, d.bc, static_cast<R*>(d.rec), d.Tf, d.status, d.g, d.un,
                               *d.mech, k, ws, threadIdx.x & 31, cs);
    } else if (w.kind == PI_BND) {
      // two groups of kBnd threads, each with its boundary columns
      const int grp = threadIdx.x / kBnd, t = threadIdx.x % kBnd;
      constexpr int E = bnode_col_entries<D, M>();
      R* col = reinterpret_cast<R*>(ps_raw) + grp * E * kBnd + t;
      long long* sncol =
          reinterpret_cast<long long*>(ps_raw + sizeof(R) * E * kBnd * (kPersistThreads / kBnd)) +
          grp * (Q / 3) * kBnd + t;
      const long long k = w.first + threadIdx.x;
      if (k < d.bc.n_if)
        bnode_body<D, M, S, R>(src, d.bc, static_cast<R*>(d.rec), d.Tf, d.status, d.g, d.un,
                               *d.mech, (int)k, col, sncol);
      __syncthreads();   // the columns become the sub-steps' shared-memory slices
      if (k < d.bc.n_if)
        iface_substeps<D, M, RT>(rec, d.Tf, d.status, d.g.N, d.un, *d.mech, d.bc.if_node[k],
                                 ps_raw);
    } else if (w.kind == PI_MOM) {
      for (int j = 0; j < npt; ++j) {
        const long long n = w.first + (long long)j * kPersistThreads + threadIdx.x;
        if (n >= d.g.N) break;
        if (d.bc.tag && d.bc.tag[n] >= 0) continue;   // interface node: PI_BND
        moments_body<D, M, S, RT>(src, rec, d.Tf, d.status, d.g, d.un, d.bc, *d.mech, n, ps_raw);
      }
    } else if (w.kind == PI_PREP) {
      for (int j = 0; j < npt; ++j)
        prep_body<D, M, true, RT>(rec, d.Tf, static_cast<RT*>(d.cpar), d.g, d.un, d.bc, *d.mech,
                            w.first + (long long)j * kPersistThreads + threadIdx.x);
    } else if (w.kind == PI_COLLIDE) {
      for (int j = 0; j < npt; ++j)
        collide_body<D, M, true, S, RT>(src, static_cast<S*>(const_cast<void*>(d.pops[1 - c])), rec,
                                  d.Tf, d.status, d.g, d.un, d.bc, *d.mech,
                                  w.first + (long long)j * kPersistThreads + threadIdx.x);
    } else {
      coll_block<D, M, S, RT, kPersistCollWarps>(
          src, static_cast<S*>(const_cast<void*>(d.pops[1 - c])),
          static_cast<const RT*>(d.cpar), d.g, d.bc, *d.mech, w.first,
          reinterpret_cast<RT*>(ps_raw));
    }
    // publish the item: every thread's stores, then the block's release
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      if (w.kind == PI_BND || w.kind == PI_MOM) add_release_gpu(done1 + w.dom, 1);
      else if (w.kind == PI_PREP) st_release_gpu(pflag + w.flag, 1);
    }
  }
}

// dynamic shared memory of k_step_persist: the largest of its items' needs
// (split: parameter and collision items; else fused collision items)
template <int D, int M, typename S, typename RT> constexpr size_t persist_smem(bool split) {
  using R = typename ComputeType<S>::type;
  const size_t bnd = bnode_smem<D, M, R>() * (kPersistThreads / kBnd);
  const size_t prep = (size_t)solve_smem_entries<D, M, RT>() * kBS * sizeof(RT);
  const size_t coll = (size_t)coll_smem_entries<D, M, RT>() * kCollNodes * sizeof(RT);
  const size_t fused = (size_t)collide_smem_entries<D, M, RT>() * kBS * sizeof(RT);
  const size_t chem = ChemSlice<M, typename ChemType<RT>::type>::kBytes +
                      sizeof(R) * WB<D, M>::N * (kPersistThreads / 32);
  size_t m = bnd > chem ? bnd : chem;
  m = m > moments_bytes<M, RT>() ? m : moments_bytes<M, RT>();
  if (split) {
    m = m > prep ? m : prep;
    m = m > coll ? m : coll;
  } else {
    m = m > fused ? m : fused;
  }
  return m;
}

// ---------------------------------------------------------------------------
// A double in the storage type of its lattice li (FP32: rounded through the bit
// pattern, the conversion instruction runs at the FP64 pipe's rate).
__device__ __forceinline__ void store_pop(double* p, double v, const float4*, int) { *p = v; }
__device__ __forceinline__ void store_pop(float* p, double v, const float4*, int) {
  *p = float_of_double(v);
}
__device__ __forceinline__ void store_pop(__half* p, double v, const float4* codec, int li) {
  *p = Codec<__half>::enc(v, codec, li);
}

// Initial populations at the equilibria of (rho or P, u, T, Y), in both
// population buffers (solid nodes keep them).  Lattice by lattice from axis
// factors; one product per population and row instead of three factors each
// (600x40x40 tube: 1.59 ms and a 0.65 ms copy of the buffer before).
template <int D, int M, typename S>
__global__ void __launch_bounds__(128)
k_init(const double* __restrict__ rho_or_P, int is_pressure, const double* __restrict__ uin,
       const double* __restrict__ Tin, const double* __restrict__ Yin, S* __restrict__ pops,
       S* __restrict__ pops2, double* __restrict__ Tf, int* __restrict__ status, Geom g, Units un,
       const __grid_constant__ DevMech mech) {
  constexpr int Q = Lat<D>::Q, NZ = Q / 9;
  const long long N = g.N;
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= N) return;
  const double T = Tin[n];
  double Rmix = 0.0, U = 0.0;
#pragma unroll
  for (int a = 0; a < M; ++a) {
    const double Y = Yin[a * N + n];
    Rmix += Y * mech.inv_mm[a];
    U += Y * species_U(mech, a, T);
  }
  Rmix *= R_U;
  const double rho = is_pressure ? rho_or_P[n] / (Rmix * T) : rho_or_P[n];
  if (!(rho > 0.0) || !isfinite(rho) || !(T > 0.0)) atomicOr(status, ST_NONFINITE);
  double u[D];
#pragma unroll
  for (int d = 0; d < D; ++d) u[d] = uin[d * N + n] * un.inv_c;
  const double theta = Rmix * T * un.inv_c2;
  const double U_lat = U * un.inv_c2;
  auto put = [&](int l, int i, double v) {
    store_pop(pops + (long long)(l * Q + i) * N + n, v, g.codec, l * Q + i);
    if (pops2) store_pop(pops2 + (long long)(l * Q + i) * N + n, v, g.codec, l * Q + i);
  };
#pragma unroll 1
  for (int l = 0; l < M; ++l) {
    const double th = l < M - 1 ? mech.Ra[l] * T * un.inv_c2 : theta;
    const double p = l < M - 1 ? rho * Yin[l * N + n] : rho;
    double t[D][3];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const double P = fma(u[d], u[d], th), hu = 0.5 * u[d];
      t[d][0] = fma(0.5, P, -hu);
      t[d][1] = 1.0 - P;
      t[d][2] = fma(0.5, P, hu);
    }
#pragma unroll
    for (int z = 0; z < NZ; ++z)
#pragma unroll
      for (int y = 0; y < 3; ++y) {
        double q = p * t[1][y];
        if constexpr (D == 3) q *= t[2][z];
#pragma unroll
        for (int x = 0; x < 3; ++x) put(l, 9 * z + 3 * y + x, q * t[0][x]);
      }
  }
  double A[D][3], Bf[D][3];
  energy_factors<D, double>(u, theta, A, Bf);
#pragma unroll
  for (int z = 0; z < NZ; ++z)
#pragma unroll
    for (int y = 0; y < 3; ++y) {
      // g^eq = rho [A_x (U A_y A_z + B_y A_z + A_y B_z) + B_x A_y A_z]
      double P = A[1][y], Qv = fma(U_lat, P, Bf[1][y]);
      if constexpr (D == 3) {
        Qv = fma(Qv, A[2][z], P * Bf[2][z]);
        P *= A[2][z];
      }
#pragma unroll
      for (int x = 0; x < 3; ++x)
        put(M, 9 * z + 3 * y + x, rho * fma(A[0][x], Qv, Bf[0][x] * P));
    }
  Tf[n] = T;
}

// Sums of node n's stored populations in FP64 (fixed point): rho, j, rho E, and
// species(a, rho_a) for every species, the slaved one last.

// Q populations of a lattice from pl, N apart, times 2^shift, and their largest
// biased exponent.  FP32: from the largest bit pattern, so that all loads are in
// flight before the first is widened; shift: 64 where FP32's denormals count.
template <typename S, int Q>
__device__ __forceinline__ int load_lattice(const S* __restrict__ pl, long long N,
                                            const float4* codec, int li, double (&v)[Q],
                                            int& shift) {
  int e = 0;
  shift = 0;
  if constexpr (sizeof(S) == 8) {
#pragma unroll
    for (int i = 0; i < Q; ++i, pl += N) v[i] = __ldg(pl);
#pragma unroll
    for (int i = 0; i < Q; ++i) e = max(e, fix_exponent(v[i]));
  } else {
    float f[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i, pl += N)
      f[i] = Codec<S>::template dec<float>(__ldg(pl), codec, li + i);
#pragma unroll
    for (int i = 0; i < Q; ++i) e = max(e, __float_as_int(f[i]) & 0x7fffffff);
    if (e < (67 << 23)) {                          // all below 2^-60
      shift = 64;
      e = __float_as_int(0x1p64f * __int_as_float(e));
#pragma unroll
      for (int i = 0; i < Q; ++i) f[i] *= 0x1p64f;
    }
    e = fix_exponent(double_of_float(__int_as_float(e)));
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = double_of_float(f[i]);
  }
  return e;
}

template <int D, int M, typename S, typename F>
__device__ __forceinline__ void stored_sums(const S* __restrict__ pops, long long N, long long n,
                                            const float4* codec, double& rho, double (&j)[D],
                                            double& rhoE, F&& species) {
  constexpr int Q = Lat<D>::Q, NP = Lat<D>::NP;
  Remainder<D, double> rest;
#pragma unroll 1
  for (int it = 0; it <= M; ++it) {
    const int l = it == 0 ? M - 1 : (it == 1 ? M : it - 2);   // f, g, the species
    double v[Q];
    const S* pl = pops + (long long)l * Q * N + n;
    int shift, e = load_lattice<S>(pl, N, codec, l * Q, v, shift);
    Fix sum, sj[D], sP[NP];
    lattice_sums<D, double>(v, e, sum, sj, sP);
    e -= shift;
    const FixSum t = fix_sum(sum, e);
    const double s0 = double_of_fix(t);
    if (it == 0) {
      rho = s0;
#pragma unroll
      for (int d = 0; d < D; ++d) j[d] = double_of_fix(fix_sum(sj[d], e));
      rest.start(e);
      rest.add(0, t, s0, true);
    } else if (it == 1) {
      rhoE = s0;
    } else {
      rest.add(0, t, s0, false);
      species(l, s0);
    }
  }
  species(M - 1, rest.get(0));
}

// ---------------------------------------------------------------------------
// Flame diagnostics of the stored state (Sec. 5.3 quantities), one pass:
// per node the moments, T by Newton from the guess, the mass production
// rates and q = -sum_a H_a(T) rho_dot_a (W/m^3, H_a with the enthalpy of
// formation); per block the sum of q, the largest q with its node (the
// smallest index among equal maxima), the largest T and |u| (m/s).  FP64
// whatever the storage.
template <int D, int M, typename S>
__global__ void __launch_bounds__(128)
k_diag(const S* __restrict__ pops, const double* __restrict__ Tf, const int* __restrict__ tag,
       DiagPart* __restrict__ part, int* __restrict__ status, Geom g, Units un,
       const __grid_constant__ DevMech mech, int x0, int x1) {
  __shared__ double s_sum[128], s_qmax[128], s_T[128], s_u[128];
  __shared__ long long s_n[128];
  const long long N = g.N;
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  double q = 0.0, qmax = -INFINITY, Tmax = -INFINITY, umax = -INFINITY;
  long long nmax = LLONG_MAX;
  const int xn = (int)(n % g.nx);   // the nodes with x in [x0, x1) only
  if (n < N && xn >= x0 && xn < x1 && !(tag && tag[n] == TAG_SOLID)) {
    double rho, rhoE, j[D], c[4] = {0.0, 0.0, 0.0, 0.0}, ir = 0.0, usq = 0.0;
    ChemSlice<M, double> cs(chem_static_slice<M, double>(), threadIdx.x);
    stored_sums<D, M, S>(pops, N, n, g.codec, rho, j, rhoE, [&](int a, double rs) {
      if (a == 0) ir = 1.0 / rho;
      const double Y = rs * ir;
      c[0] = fma(Y, mech.u0[a], c[0]);
      c[1] = fma(Y, mech.u1[a], c[1]);
      c[2] = fma(Y, mech.u2[a], c[2]);
      c[3] = fma(Y, mech.u3[a], c[3]);
      cs.set(a, rs * mech.inv_mm[a]);
    });
    for (int d = 0; d < D; ++d) usq += (j[d] * ir) * (j[d] * ir);
    bool ok;
    const double T = newton_poly(c, (rhoE * ir - 0.5 * usq) * un.c * un.c, Tf[n],
                                 un.newton_max_iter, un.newton_rtol, ok);
    if (!ok) atomicOr(status, ST_NEWTON);
    molar_rates(mech, T, cs);
    for (int a = 0; a < M; ++a)
      q -= (species_U(mech, a, T) + mech.Ra[a] * T) * (cs.rate(a) * mech.mm[a]);
    qmax = q;
    nmax = n;
    Tmax = T;
    umax = sqrt(usq) * un.c;
  }
  const int t = threadIdx.x;
  s_sum[t] = q;
  s_qmax[t] = qmax;
  s_n[t] = nmax;
  s_T[t] = Tmax;
  s_u[t] = umax;
  __syncthreads();
  for (int o = 64; o > 0; o >>= 1) {
    if (t < o) {
      s_sum[t] += s_sum[t + o];
      if (s_qmax[t + o] > s_qmax[t] || (s_qmax[t + o] == s_qmax[t] && s_n[t + o] < s_n[t])) {
        s_qmax[t] = s_qmax[t + o];
        s_n[t] = s_n[t + o];
      }
      s_T[t] = fmax(s_T[t], s_T[t + o]);
      s_u[t] = fmax(s_u[t], s_u[t + o]);
    }
    __syncthreads();
  }
  if (t == 0) part[blockIdx.x] = DiagPart{s_sum[0], s_qmax[0], s_n[0], s_T[0], s_u[0]};
}

// Fields of the stored state: rho, u (m/s), T (Newton, not stored), Y, E (J/kg).
// Bound by its one pass over the populations (600x40x40 tube: 0.40 ms in FP64,
// 0.98 with the sums in FP64 instructions; 0.47 in FP32, 1.5 with a lattice's
// loads one after the other).
template <int D, int M, typename S>
__global__ void __launch_bounds__(128)
k_out(const S* __restrict__ pops, const double* __restrict__ Tf, double* __restrict__ orho,
      double* __restrict__ ou, double* __restrict__ oT, double* __restrict__ oY,
      double* __restrict__ oE, int* __restrict__ status, Geom g, Units un,
      const __grid_constant__ DevMech mech) {
  const long long N = g.N;
  const long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (n >= N) return;
  double rho, rhoE, j[D], u[D], c[4] = {0.0, 0.0, 0.0, 0.0}, ir = 0.0, usq = 0.0;
  stored_sums<D, M, S>(pops, N, n, g.codec, rho, j, rhoE, [&](int a, double rs) {
    if (a == 0) ir = 1.0 / rho;
    const double Y = rs * ir;
    if (oY) oY[a * N + n] = Y;
    c[0] = fma(Y, mech.u0[a], c[0]);
    c[1] = fma(Y, mech.u1[a], c[1]);
    c[2] = fma(Y, mech.u2[a], c[2]);
    c[3] = fma(Y, mech.u3[a], c[3]);
  });
  for (int d = 0; d < D; ++d) { u[d] = j[d] * ir; usq += u[d] * u[d]; }
  const double E = rhoE * ir;
  bool ok;
  const double T = newton_poly(c, (E - 0.5 * usq) * un.c * un.c, Tf[n], un.newton_max_iter,
                               un.newton_rtol, ok);
  if (!ok) atomicOr(status, ST_NEWTON);
  if (orho) orho[n] = rho;
  if (ou) {
    for (int d = 0; d < 3; ++d) ou[d * N + n] = d < D ? u[d] * un.c : 0.0;
  }
  if (oT) oT[n] = T;
  if (oE) oE[n] = E * un.c * un.c;
}


// ---------------------------------------------------------------------------
// dispatch

static inline unsigned blocks_for(long long N, int bs) { return (unsigned)((N + bs - 1) / bs); }

// dynamic shared memory of the collision kernels and of k_prep (bytes)
template <int D, int M, typename RT> constexpr size_t fused_smem() {
  return (size_t)collide_smem_entries<D, M, RT>() * kBS * sizeof(RT);
}
template <int D, int M, typename RT> constexpr size_t prep_smem() {
  return (size_t)solve_smem_entries<D, M, RT>() * kBS * sizeof(RT);
}
template <int D, int M, typename RT> constexpr size_t coll_smem() {
  return (size_t)coll_smem_entries<D, M, RT>() * kCollNodes * sizeof(RT);
}

// Kernel attributes (shared memory above the 48 KB default) of every kernel a
// step may launch; idempotent, and required before a stream capture, where
// attribute calls are not recorded.
template <int D, int M, typename S, typename RT>
static cudaError_t prepare_impl() {
  cudaError_t e = cudaSuccess;
  auto big = [&](const void* f, size_t bytes) {
    if (e == cudaSuccess && bytes > 48 * 1024)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  };
  big((const void*)k_collide<D, M, S, RT>, fused_smem<D, M, RT>());
  big((const void*)k_collide_batch<D, M, S, RT>, fused_smem<D, M, RT>());
  big((const void*)k_prep<D, M, RT>, prep_smem<D, M, RT>());
  big((const void*)k_prep_batch<D, M, RT>, prep_smem<D, M, RT>());
  big((const void*)k_coll<D, M, S, RT>, coll_smem<D, M, RT>());
  big((const void*)k_coll_batch<D, M, S, RT>, coll_smem<D, M, RT>());
  big((const void*)k_bnode<D, M, S>, bnode_smem<D, M, RT>());
  big((const void*)k_bnode_batch<D, M, S>, bnode_smem<D, M, RT>());
  big((const void*)k_step_persist<D, M, S, RT>,
      std::max(persist_smem<D, M, S, RT>(true), persist_smem<D, M, S, RT>(false)));
  return e;
}

// the interface nodes' reaction sub-steps after k_bnode: a thread each where
// these fill the GPU, else eight lanes
template <int D, int M, typename RT>
static void launch_chem(cudaStream_t s, RT* rec, const double* Tf, int* status, long long N,
                        const BCDev& bc, const Units& un, const DevMech* mech) {
  if (bc.n_if >= kIfChemThreadNodes)
    k_iface_chem<D, M, RT>
        <<<blocks_for(bc.n_if, kChemThreads), kChemThreads,
           ChemSlice<M, typename ChemType<RT>::type>::kBytes, s>>>(
            rec, Tf, status, N, bc.if_node, bc.n_if, un, mech);
  else
    k_chem<D, M, RT><<<blocks_for(bc.n_if, kIfChemNodesPerBlock), 128, 0, s>>>(
        rec, Tf, status, N, un, mech, bc.if_node, bc.n_if);
}

// prepare_impl once per device and instantiation
template <int D, int M, typename S, typename RT>
static cudaError_t prepare_once() {
  static std::atomic<unsigned long long> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (done.load() & bit) return cudaSuccess;
  e = prepare_impl<D, M, S, RT>();
  if (e == cudaSuccess) done.fetch_or(bit);
  return e;
}

template <int D, int M, typename S, typename RT>
static cudaError_t step_impl(const DevMech& mech, const StepArgs& a, cudaStream_t s,
                             int which) {
  const int bs = kBS;
  const unsigned nb = blocks_for(a.g.N, bs);
  const cudaError_t pe = prepare_once<D, M, S, RT>();
  if (pe != cudaSuccess) return pe;
  const Launch& lc = a.lc;
  const bool chem_sep = lc.chem_lanes > 1 && a.mech_dev;
  const bool split = lc.coll_split && a.cpar;
  if (which != 1) {
    const S* src = static_cast<const S*>(a.src);
    RT* rec = reinterpret_cast<RT*>(a.rec);
    // chem_lanes > 1: the bulk nodes' moments and reaction sub-steps in one
    // kernel with chem_lanes lanes per node (k_mchem).  chem_lanes = 1:
    // k_moments with the sub-steps inline.
    auto mchem = [&](cudaStream_t st, int node_set) {
      const unsigned nbm = blocks_for(a.g.N, 128 / lc.chem_lanes);
      if (lc.chem_lanes == 4)
        k_mchem<D, M, S, RT, 4><<<nbm, 128, 0, st>>>(src, rec, a.Tfield, a.status, a.g, a.un,
                                                     a.bc, mech, a.mech_dev, node_set);
      else
        k_mchem<D, M, S, RT, 8><<<nbm, 128, 0, st>>>(src, rec, a.Tfield, a.status, a.g, a.un,
                                                     a.bc, mech, a.mech_dev, node_set);
    };
    // the boundary kernel and the interface nodes' sub-steps run on a side
    // stream beside the bulk moments.  Interface nodes need the handle's
    // device copy of the mechanism (every handle has one; the
    // allocation-free step accepts no interface nodes).
    if (a.bc.n_if > 0 && !a.mech_dev) return cudaErrorInvalidValue;
    const bool fork = a.bc.n_if > 0 && a.side && a.ev_fork && a.ev_join;
    // the boundary kernel and the interface nodes' sub-steps
    auto boundary = [&](cudaStream_t st) {
      if (a.bc.n_if <= boundary_warp_nodes(sizeof(S) == 8, LBM_CHEM64 != 0)) {
        k_bnode_warp<D, M, S><<<blocks_for(a.bc.n_if, kBnodeWarps), 32 * kBnodeWarps, 0, st>>>(
            src, a.bc, a.Tfield, a.status, a.g, a.un, a.mech_dev, rec);
        return;
      }
      k_bnode<D, M, S><<<blocks_for(a.bc.n_if, kBnd), kBnd, bnode_smem<D, M, RT>(), st>>>(
          src, a.bc, a.Tfield, a.status, a.g, a.un, mech, rec);
      launch_chem<D, M, RT>(st, rec, a.Tfield, a.status, a.g.N, a.bc, a.un, a.mech_dev);
    };
    auto bulk = [&](int node_set) {
      if (chem_sep)
        mchem(s, node_set);
      else
        k_moments<D, M, S, RT><<<nb, bs, 0, s>>>(src, rec, a.Tfield, a.status, a.g, a.un, a.bc,
                                                 mech, node_set);
    };
    if (fork) {
      cudaError_t e = cudaEventRecord(a.ev_fork, s);
      if (e == cudaSuccess) e = cudaStreamWaitEvent(a.side, a.ev_fork, 0);
      if (e != cudaSuccess) return e;
      boundary(a.side);
      e = cudaEventRecord(a.ev_join, a.side);
      if (e != cudaSuccess) return e;
      bulk(NODES_BULK);
      e = cudaStreamWaitEvent(s, a.ev_join, 0);
      if (e != cudaSuccess) return e;
    } else {
      const bool bnd = a.bc.n_if > 0;
      if (bnd) boundary(s);
      bulk(bnd ? NODES_BULK : NODES_ALL);
    }
  }
  if (which != 0) {
    if (split) {
      k_prep<D, M, RT><<<nb, bs, prep_smem<D, M, RT>(), s>>>(
          reinterpret_cast<const RT*>(a.rec), a.Tfield, static_cast<RT*>(a.cpar), a.g, a.un,
          a.bc, mech);
      k_coll<D, M, S, RT><<<blocks_for(a.g.N, kCollNodes), 32 * kCollTPN, coll_smem<D, M, RT>(),
                            s>>>(static_cast<const S*>(a.src), static_cast<S*>(a.dst),
                                 static_cast<const RT*>(a.cpar), a.g, a.bc, mech);
    } else {
      k_collide<D, M, S, RT><<<nb, bs, fused_smem<D, M, RT>(), s>>>(
          static_cast<const S*>(a.src), static_cast<S*>(a.dst),
          reinterpret_cast<const RT*>(a.rec), a.Tfield, a.status, a.g, a.un, a.bc, mech);
    }
  }
  return cudaGetLastError();
}

template <int D, int M, typename S>
static cudaError_t init_impl(const DevMech& mech, const Geom& g, const Units& un,
                             const double* rho_or_P, int is_pressure, const double* u,
                             const double* T, const double* Y, void* pops, void* pops2,
                             double* Tfield, int* status, cudaStream_t s) {
  k_init<D, M, S><<<blocks_for(g.N, 128), 128, 0, s>>>(rho_or_P, is_pressure, u, T, Y,
                                                        static_cast<S*>(pops),
                                                        static_cast<S*>(pops2), Tfield, status,
                                                        g, un, mech);
  return cudaGetLastError();
}

template <int D, int M, typename S>
static cudaError_t diag_impl(const DevMech& mech, const Geom& g, const Units& un,
                             const void* pops, const double* Tfield, const int* tag,
                             DiagPart* part, int* status, int x0, int x1, cudaStream_t s) {
  k_diag<D, M, S><<<blocks_for(g.N, 128), 128, 0, s>>>(static_cast<const S*>(pops), Tfield, tag,
                                                        part, status, g, un, mech, x0, x1);
  return cudaGetLastError();
}

template <int D, int M, typename S>
static cudaError_t out_impl(const DevMech& mech, const Geom& g, const Units& un,
                            const void* pops, const double* Tfield, double* rho, double* u,
                            double* T, double* Y, double* E, int* status, cudaStream_t s) {
  k_out<D, M, S><<<blocks_for(g.N, 128), 128, 0, s>>>(static_cast<const S*>(pops), Tfield,
                                                       rho, u, T, Y, E, status, g, un, mech);
  return cudaGetLastError();
}

// Grid of a batched kernel: one block per tile, or (persistent) at most the
// blocks the GPU holds at once, from the occupancy calculator.
template <typename K>
static int batch_grid(K kernel, int nblk, int threads, size_t smem, bool persistent) {
  if (!persistent || nblk <= 0) return nblk;
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) !=
          cudaSuccess ||
      per_sm <= 0)
    return nblk;
  return std::min(nblk, sms * per_sm);
}

template <int D, int M, typename S, typename RT>
static cudaError_t batch_impl(const DomainDev* doms, int ndom, const BatchGrids& gr,
                              const Launch& lc, int parity, cudaStream_t s,
                              const SideStream& side) {
  const int bs = kBS;
  const cudaError_t pe = prepare_once<D, M, S, RT>();
  if (pe != cudaSuccess) return pe;
  if (lc.persistent == 2) {
    // the whole step as one launch over the work-list (sync words zeroed
    // first)
    if (gr.nitems == 0) return cudaSuccess;
    auto kp = k_step_persist<D, M, S, RT>;
    const size_t sm = persist_smem<D, M, S, RT>(lc.coll_split != 0);
    cudaError_t e = cudaMemsetAsync(gr.sync, 0, (size_t)gr.nsync * sizeof(int), s);
    if (e != cudaSuccess) return e;
    kp<<<batch_grid(kp, gr.nitems, kPersistThreads, sm, true), kPersistThreads, sm, s>>>(
        doms, ndom, parity, gr.items, gr.nitems, lc.npt, gr.sync, gr.timeout_ns);
    return cudaGetLastError();
  }
  const int chem_inline = lc.chem_lanes <= 1;
  const bool ps = lc.persistent != 0;
  auto kmom = k_moments_batch<D, M, S, RT>;
  // the boundary kernel: a warp or a thread per interface node
  auto bnd = [&](cudaStream_t st) {
    if (gr.bnd_warp) {
      auto k = k_bnode_warp_batch<D, M, S>;
      k<<<batch_grid(k, gr.ntblocks, 32 * kBnodeWarps, 0, ps), 32 * kBnodeWarps, 0, st>>>(
          doms, ndom, parity, gr.ntblocks);
    } else {
      auto k = k_bnode_batch<D, M, S>;
      const size_t sm = bnode_smem<D, M, RT>();
      k<<<batch_grid(k, gr.ntblocks, kBnd, sm, ps), kBnd, sm, st>>>(doms, ndom, parity,
                                                                    gr.ntblocks);
    }
  };
  // the interface nodes' reaction sub-steps after the thread-per-node kernel
  auto chem = [&](cudaStream_t st) {
    if (gr.bnd_warp) return;          // done by the boundary kernel
    if (gr.n_if_total >= kIfChemThreadNodes) {
      // enough interface nodes to fill the GPU with one thread each
      auto k = k_iface_chem_batch<D, M, RT>;
      const size_t sm = ChemSlice<M, typename ChemType<RT>::type>::kBytes;
      k<<<batch_grid(k, gr.ntblocks, kBnd, sm, ps), kBnd, sm, st>>>(doms, ndom, gr.ntblocks);
    } else {
      auto k = k_chem_batch<D, M, RT>;
      k<<<batch_grid(k, gr.nbblocks, 128, 0, ps), 128, 0, st>>>(doms, ndom, gr.nbblocks);
    }
  };
  // chem_lanes > 1: moments and sub-steps of the nodes in one kernel with
  // chem_lanes lanes per node, on the chemistry grid
  auto mchem = [&](int node_set) {
    if (gr.ncblocks == 0) return;
    if (lc.chem_lanes == 4) {
      auto k = k_mchem_batch<D, M, S, RT, 4>;
      k<<<batch_grid(k, gr.ncblocks, 128, 0, ps), 128, 0, s>>>(doms, ndom, parity, node_set,
                                                               gr.ncblocks);
    } else {
      auto k = k_mchem_batch<D, M, S, RT, 8>;
      k<<<batch_grid(k, gr.ncblocks, 128, 0, ps), 128, 0, s>>>(doms, ndom, parity, node_set,
                                                               gr.ncblocks);
    }
  };
  if (gr.nbblocks > 0 && side.stream && side.fork && side.join) {
    // on the side stream, concurrent with the bulk moments: the boundary
    // kernel and the interface nodes' sub-steps
    cudaError_t e = cudaEventRecord(side.fork, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(side.stream, side.fork, 0);
    if (e != cudaSuccess) return e;
    bnd(side.stream);
    chem(side.stream);
    e = cudaEventRecord(side.join, side.stream);
    if (e != cudaSuccess) return e;
    if (chem_inline)
      kmom<<<batch_grid(kmom, gr.nblocks, bs, 0, ps), bs, 0, s>>>(doms, ndom, parity,
                                                                  NODES_BULK, gr.nblocks);
    else
      mchem(NODES_BULK);
    e = cudaStreamWaitEvent(s, side.join, 0);
    if (e != cudaSuccess) return e;
  } else {
    const bool bnd_rec = gr.nbblocks > 0;
    if (gr.nbblocks > 0)
      bnd(s);
    if (chem_inline)
      kmom<<<batch_grid(kmom, gr.nblocks, bs, 0, ps), bs, 0, s>>>(
          doms, ndom, parity, bnd_rec ? NODES_BULK : NODES_ALL, gr.nblocks);
    else
      mchem(bnd_rec ? NODES_BULK : NODES_ALL);
    if (bnd_rec) chem(s);
  }
  if (lc.coll_split) {
    auto kp = k_prep_batch<D, M, RT>;
    auto kc = k_coll_batch<D, M, S, RT>;
    const size_t sp = prep_smem<D, M, RT>(), sc = coll_smem<D, M, RT>();
    kp<<<batch_grid(kp, gr.nblocks, bs, sp, ps), bs, sp, s>>>(doms, ndom, gr.nblocks);
    kc<<<batch_grid(kc, gr.nkblocks, 32 * kCollTPN, sc, ps), 32 * kCollTPN, sc, s>>>(
        doms, ndom, parity, gr.nkblocks);
  } else {
    auto kf = k_collide_batch<D, M, S, RT>;
    const size_t sf = fused_smem<D, M, RT>();
    kf<<<batch_grid(kf, gr.nblocks, bs, sf, ps), bs, sf, s>>>(doms, ndom, parity, gr.nblocks);
  }
  return cudaGetLastError();
}

// The kernel set of one (D, M, precision).
template <int D, int M, typename S, typename RT>
const KernelSet* make_kernel_set() {
  static const KernelSet ks = {&step_impl<D, M, S, RT>, &batch_impl<D, M, S, RT>,
                               &prepare_once<D, M, S, RT>, &init_impl<D, M, S>,
                               &out_impl<D, M, S>, &diag_impl<D, M, S>, Rec<D, M>::NF,
                               CPar<D, M>::NF};
  return &ks;
}

}  // inline namespace
}  // namespace lbm
