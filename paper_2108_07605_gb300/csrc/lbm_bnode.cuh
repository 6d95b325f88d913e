// Boundary reconstruction with one thread per interface node (Sec. 4):
// bounce-back (Eq. bb), Tamm-Mott-Smith wall (Sec. 4.2.2, Eqs. BBrho-fatms),
// flux inlet (Sec. 4.3, Eqs. in_f-fa_inlet, and the simplified inlet of the
// same section) and LODI outlet (Sec. 4.4, Eqs. convectiveBC-fa_outlet),
// followed by the node's moment record.  Included by lbm_kernels.cuh inside
// its namespace.
//
// Why a thread per node.  A node's procedure is a chain of scalar steps
// (moment sums over the 270 populations, up to four temperature Newton
// solves, equilibrium parameters) around three passes over its populations.
// Spread over a warp (lane = direction), every scalar step and every
// cross-lane reduction is a full-warp instruction: on GB300, whose FP64
// pipes run two lanes per clock per SM, that made the FP64 boundary kernel
// execute ~63k FP64 FLOP per interface node.  With a thread per node the
// sums are sequential adds and the scalar steps run once per node.  The
// passes run lattice by lattice (compile-time l) and, inside, direction by
// direction: the direction index is the same for every thread of a warp,
// so the branches on c_i are uniform, and each equilibrium population is a
// product of three entries of per-lattice axis-factor tables (Eq. prod)
// built once per lattice and state.  Threads are consecutive interface
// nodes (the list is in node order), so the pull loads of a wall row
// coalesce.
//
// Per-thread arrays (species mass fractions, the TMS local species
// velocities, the pull-source node of every direction) live in this
// thread's shared-memory column, stride kBnd.

constexpr int kBnd = kBndNodesPerBlock;   // threads per block of the boundary kernel
// Blocks per SM its registers are held to.  FP64 is bound by its FP64 instructions
// (pipe 72 % of the active cycles) and the tail of its one wave and a half, FP32 by
// instruction fetch and latency (19 % of the issue slots): what counts is loads in
// flight, by the directions unrolled three rows deep, and warps.
// 600x40x40 tube, 91k interface nodes: FP64 1.22 -> 1.11 ms (255 registers);
// FP32 0.44 -> 0.32 ms at 168 registers and six blocks, 0.41 at eight (128
// registers, spills) and at four (240); FP16 0.52 -> 0.37.
template <typename S> constexpr int kBnodeMinBlocks = sizeof(S) == 8 ? 4 : 6;

// shared memory per thread: target Y, local Y, a spare Y, the local u_a and
// the target u_a (off-grid TMS targets) (R entries), then the pull sources of
// the Q / 3 rows of directions (long long)
template <int D, int M> constexpr int bnode_col_entries() { return 3 * M + 2 * M * D; }
template <int D, int M, typename R> constexpr size_t bnode_smem() {
  return (sizeof(R) * bnode_col_entries<D, M>() + sizeof(long long) * (Lat<D>::Q / 3)) * kBnd;
}

// An equilibrium state of the boundary procedures (Eqs. faEqGeneral,
// fEqGeneral, gEqGeneral): rho, T, theta, U/c^2, u in registers; Y and the
// species velocities in shared memory.
template <int D, int M, typename R> struct BState {
  R rho, T, th, U;
  R u[D];
  R* Y;           // [M], stride kBnd
  R* us;          // [M D] species velocities, stride kBnd (nullptr: u for every species)
  double T_full;  // T to the solve's precision
};

// theta, U/c^2 of a state from its T and Y (the mixture energy as a sum over
// species, float-float in the mixed path)
template <int D, int M, typename R>
__device__ __forceinline__ void bstate_prepare(BState<D, M, R>& s, const DevMech& m,
                                               const Units& un) {
  if constexpr (!kFF<R>) {
    double Rm = 0.0, U = 0.0;
#pragma unroll
    for (int a = 0; a < M; ++a) {
      const double Ya = double(s.Y[a * kBnd]);
      Rm += Ya * m.inv_mm[a];
      U += Ya * species_U(m, a, double(s.T));
    }
    s.th = R(R_U * Rm * double(s.T) * un.inv_c2);
    s.U = R(U * un.inv_c2);
  } else {
    float Rm = 0.f;
    const ff T(s.T);
    ff U;
#pragma unroll
    for (int a = 0; a < M; ++a) {
      Rm += s.Y[a * kBnd] * m.inv_mm_s[a];
      U += ff(s.Y[a * kBnd]) * species_U_ff(m, a, T);
    }
    s.th = float(R_U) * Rm * s.T * un.inv_c2_s;
    s.U = (U * un.inv_c2_f).hi;
  }
}

// Population sums of a node (every lattice): rho, j, the momentum flux
// tensor P of the f lattice, rho E and q of the g lattice, rho_a and j_a of
// the stored species.
template <int D, int M, typename R> struct BSums {
  R rho, rhoE, j[D], q[D], P[Lat<D>::NP], rs[M], js[M][D];
};

// The macroscopic state of population sums (Eqs. density1, momentum1,
// fdensity, f1momMomentum, g0momTotalEnergy, slaving Eq. strongest): rho,
// u, Y, u_a (reading R5) and T by Newton on Eq. temperature from T_guess,
// then theta and U/c^2 as bstate_prepare; the record's enthalpy polynomial in
// H if given.
template <int D, int M, typename R>
__device__ __forceinline__ void bstate_of(BState<D, M, R>& s, const BSums<D, M, R>& z,
                                          double T_guess, const DevMech& m, const Units& un,
                                          int* status, R* H = nullptr) {
  s.rho = z.rho;
  const R irho = R(1) / z.rho;
  R usq = R(0);
#pragma unroll
  for (int d = 0; d < D; ++d) { s.u[d] = z.j[d] * irho; usq += s.u[d] * s.u[d]; }
  R rM = z.rho, jM[D];
#pragma unroll
  for (int d = 0; d < D; ++d) jM[d] = z.j[d];
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    rM -= z.rs[a];
#pragma unroll
    for (int d = 0; d < D; ++d) jM[d] -= z.js[a][d];
  }
#pragma unroll
  for (int a = 0; a < M; ++a) {
    const R ra = a < M - 1 ? z.rs[a] : rM;
    s.Y[a * kBnd] = ra * irho;
    if (s.us) {
      R ja[D];
#pragma unroll
      for (int d = 0; d < D; ++d) ja[d] = a < M - 1 ? z.js[a][d] : jM[d];
      const bool tiny = species_velocity_undefined<D, R>(ra, ja);
      if constexpr (sizeof(R) == 8) {
        // rho_a > 1e-300 when not tiny: 1/rho_a is finite
        const R ira = tiny ? R(0) : R(1) / ra;
#pragma unroll
        for (int d = 0; d < D; ++d) s.us[(a * D + d) * kBnd] = tiny ? s.u[d] : ja[d] * ira;
      } else {
        // FP32: a positive rho_a below ~3e-39 has no finite reciprocal
#pragma unroll
        for (int d = 0; d < D; ++d) s.us[(a * D + d) * kBnd] = tiny ? s.u[d] : ja[d] / ra;
      }
    }
  }
  bool ok;
  if constexpr (!kFF<R>) {
    double Y[M];
#pragma unroll
    for (int a = 0; a < M; ++a) Y[a] = double(s.Y[a * kBnd]);
    const double U = (double(z.rhoE * irho) - 0.5 * double(usq)) * un.c * un.c;
    double c[4];
    const double T = newton_T<M>(m, Y, U, T_guess, un.newton_max_iter, un.newton_rtol, ok, c);
    s.T = R(T);
    s.T_full = T;
    if (H) {
      R Rm = R(0), h[4];
#pragma unroll
      for (int a = 0; a < M; ++a) {
        if constexpr (sizeof(R) == 8) Rm += Y[a] * m.inv_mm[a];
        else Rm += s.Y[a * kBnd] * m.inv_mm_s[a];
      }
      enthalpy_poly(c, Rm, un, h);
#pragma unroll
      for (int k = 0; k < 4; ++k) H[k] = h[k];
    }
  } else {
    ff Yf[M];
#pragma unroll
    for (int a = 0; a < M; ++a) Yf[a] = ff(s.Y[a * kBnd]);
    const ff U = (ff(z.rhoE * irho) + ff(-0.5f * usq)) * un.c2_f;
    ff c[4];
    const ff T = newton_T_ff<M>(m, Yf, U, ff_from_double(T_guess), un.newton_max_iter,
                                un.newton_rtol_f, ok, c);
    s.T = T.hi;
    s.T_full = ff_to_double(T);
    if (H) {
      float Rm = 0.f, h[4];
#pragma unroll
      for (int a = 0; a < M; ++a) Rm += s.Y[a * kBnd] * m.inv_mm_s[a];
      enthalpy_poly(c, Rm, un, h);
#pragma unroll
      for (int k = 0; k < 4; ++k) H[k] = h[k];
    }
  }
  if (!ok) atomicOr(status, ST_NEWTON);
  bstate_prepare<D, M, R>(s, m, un);
}

// Per-lattice axis-factor tables of a state (Eqs. phi0, phiPlus, phis,
// prod): entry k of an axis is the factor for c = k - 1.  PTab: a species
// or the f lattice, population = pref * prod_d t[d][c_d + 1].  GTab: the g
// lattice by the closed form of Eq. geq_i, A = Psi_c(u_d, theta + u_d^2),
// B = Psi_c applied to u_d^2 / 2.
template <int D, typename R> struct PTab { R pref, t[D][3]; };
template <int D, typename R> struct GTab { R rho, U, A[D][3], B[D][3]; };

template <typename R> __device__ __forceinline__ R sel3(int c, const R (&t)[3]) {
  return c < 0 ? t[0] : (c == 0 ? t[1] : t[2]);
}

// FP32 products rounded on their own, and below sums fused explicitly: left
// to the compiler, a thread's and a warp's procedure (bnode_body, bnode_warp)
// would not be fused alike
__device__ __forceinline__ float mul1(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul1(double a, double b) { return a * b; }

template <int D, int M, int l, typename R>
__device__ __forceinline__ void ptab(const BState<D, M, R>& s, PTab<D, R>& e, const DevMech& m,
                                     const Units& un) {
  R th;
  if constexpr (l < M - 1) {
    if constexpr (sizeof(R) == 8) th = R(m.Ra[l] * double(s.T) * un.inv_c2);
    else th = m.Ra_s[l] * s.T * un.inv_c2_s;
    e.pref = s.rho * s.Y[l * kBnd];
  } else {
    th = s.th;
    e.pref = s.rho;
  }
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const R xi = (l < M - 1 && s.us) ? s.us[(l * D + d) * kBnd] : s.u[d];
    const R P = th + xi * xi;
    e.t[d][0] = R(0.5) * (P - xi);
    e.t[d][1] = R(1) - P;
    e.t[d][2] = R(0.5) * (P + xi);
  }
}

template <int D, int M, typename R>
__device__ __forceinline__ void gtab(const BState<D, M, R>& s, GTab<D, R>& g) {
  g.rho = s.rho;
  g.U = s.U;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const R ua = s.u[d];
    const R q = mul1(ua, ua), hq = R(0.5) * q;
    const R O1 = mul1(ua, s.th + hq);                                  // theta u + u^3/2
    const R O2 = fma(s.th, s.th, mul1(q, fma(R(2.5), s.th, hq)));
    const R P = s.th + q;
    g.A[d][0] = R(0.5) * (P - ua);
    g.A[d][1] = R(1) - P;
    g.A[d][2] = R(0.5) * (P + ua);
    g.B[d][0] = R(0.5) * (O2 - O1);
    g.B[d][1] = hq - O2;
    g.B[d][2] = R(0.5) * (O2 + O1);
  }
}

// Tables of one state for the lattice of the current pass.  row<l>(c_y,
// c_z) forms the part shared by a row of three directions (the population's
// pref t_y t_z; for g, A_y A_z and U A_y A_z + B_y A_z + A_y B_z, since
// g^eq = rho [A_x (U A_y A_z + B_y A_z + A_y B_z) + B_x A_y A_z]); evalx<l>(c_x)
// then finishes a direction of that row.
template <int D, int M, typename R> struct ETab {
  PTab<D, R> p;
  GTab<D, R> g;
  R rp, rP, rQ;
  template <int l>
  __device__ __forceinline__ void build(const BState<D, M, R>& s, const DevMech& m,
                                        const Units& un) {
    if constexpr (l == M) gtab<D, M, R>(s, g);
    else ptab<D, M, l, R>(s, p, m, un);
  }
  template <int l> __device__ __forceinline__ void row(int cy, int cz) {
    if constexpr (l == M) {
      const R ay = sel3(cy, g.A[1]), by = sel3(cy, g.B[1]);
      if constexpr (D == 3) {
        const R az = sel3(cz, g.A[2]), bz = sel3(cz, g.B[2]);
        rP = mul1(ay, az);
        rQ = fma(g.U, rP, fma(by, az, mul1(ay, bz)));
      } else {
        rP = ay;
        rQ = fma(g.U, ay, by);
      }
    } else {
      rp = p.pref * sel3(cy, p.t[1]);
      if constexpr (D == 3) rp *= sel3(cz, p.t[2]);
    }
  }
  template <int l> __device__ __forceinline__ R evalx(int cx) const {
    if constexpr (l == M)
      return mul1(g.rho, fma(sel3(cx, g.A[0]), rQ, mul1(sel3(cx, g.B[0]), rP)));
    else return mul1(rp, sel3(cx, p.t[0]));
  }
};

// Compile-time loop l = B .. E-1: f(std::integral_constant<int, l>{}).
template <int B, int E> struct ForL {
  template <typename Fn> __device__ __forceinline__ static void run(Fn&& f) {
    f(std::integral_constant<int, B>{});
    ForL<B + 1, E>::run(f);
  }
};
template <int E> struct ForL<E, E> {
  template <typename Fn> __device__ __forceinline__ static void run(Fn&&) {}
};

// Population sums of a pass, lattice by lattice: fn.template setup<l>()
// once per lattice, then, row by row, fn.template row<l>(c_y, c_z) and
// fn.template get<l>(i, c) for the row's three directions.
// Directions in rows of three (c_x = -1, 0, 1 at compile time), three rows'
// loads in flight together; a row enters through its sum s and difference
// d = f_+ - f_- (and f_+ + f_- for P_xx).  kDensOnly: the densities rho_a,
// rho and rho E only (the bounce-back pass of a wall).
template <int D, int M, typename R, bool kDensOnly = false, typename F>
__device__ __forceinline__ void bsums(F& fn, BSums<D, M, R>& z) {
  constexpr int Q = Lat<D>::Q, NP = Lat<D>::NP;
  ForL<0, M + 1>::run([&](auto lc) {
    constexpr int l = decltype(lc)::value;
    fn.template setup<l>();
    R sum = R(0), sj[D], sP[NP];
#pragma unroll
    for (int d = 0; d < D; ++d) sj[d] = R(0);
#pragma unroll
    for (int p = 0; p < NP; ++p) sP[p] = R(0);
#pragma unroll 3
    for (int yz = 0; yz < Q / 3; ++yz) {
      const int cy = yz % 3 - 1, cz = D == 3 ? yz / 3 - 1 : 0;
      fn.template row<l>(cy, cz);
      R v[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int c[3] = {k - 1, cy, cz};
        v[k] = fn.template get<l>(3 * yz + k, c);
      }
      const R sx = v[0] + v[2], sr = sx + v[1];
      sum += sr;
      if constexpr (!kDensOnly) {
        const R dx = v[2] - v[0];
        sj[0] += dx;
        if (cy != 0) sj[1] += cy > 0 ? sr : -sr;
        if constexpr (D == 3)
          if (cz != 0) sj[2] += cz > 0 ? sr : -sr;
        if constexpr (l == M - 1) {
          sP[pidx<D>(0, 0)] += sx;
          if (cy != 0) {
            sP[pidx<D>(1, 1)] += sr;
            sP[pidx<D>(0, 1)] += cy > 0 ? dx : -dx;
          }
          if constexpr (D == 3) {
            if (cz != 0) {
              sP[pidx<D>(2, 2)] += sr;
              sP[pidx<D>(0, 2)] += cz > 0 ? dx : -dx;
              if (cy != 0) sP[pidx<D>(1, 2)] += cy == cz ? sr : -sr;
            }
          }
        }
      }
    }
    if constexpr (l < M - 1) {
      z.rs[l] = sum;
#pragma unroll
      for (int d = 0; d < D; ++d) z.js[l][d] = sj[d];
    } else if constexpr (l == M - 1) {
      z.rho = sum;
#pragma unroll
      for (int d = 0; d < D; ++d) z.j[d] = sj[d];
#pragma unroll
      for (int p = 0; p < NP; ++p) z.P[p] = sP[p];
    } else {
      z.rhoE = sum;
#pragma unroll
      for (int d = 0; d < D; ++d) z.q[d] = sj[d];
    }
  });
}

// Value functors of bsums.  BPull: the pulled population (source node from
// this thread's column) or, with bbk and an incoming link, the node's own
// opposite post-collision population (Eq. bb).
template <int D, int M, typename S, typename R> struct BPull {
  static constexpr int Q = Lat<D>::Q;
  const S* src;
  const float4* codec;
  long long N, n;
  const long long* sn;      // row r's pull source is node sn[r kBnd] + dx[k], c_x = k - 1
  int dx[3];
  unsigned inc;
  bool bbk;
  __device__ __forceinline__ bool incoming(int i) const { return inc >> i & 1u; }
  template <int l> __device__ __forceinline__ void setup() {}
  template <int l> __device__ __forceinline__ void row(int, int) {}
  template <int l> __device__ __forceinline__ R pull(int i, int k) const {
    const bool bb = bbk && incoming(i);
    const long long mm = bb ? n : sn[i / 3 * kBnd] + dx[k];
    const int ii = bb ? Q - 1 - i : i;
    return Codec<S>::template dec<R>(__ldg(src + (long long)(l * Q + ii) * N + mm), codec,
                                     l * Q + ii);
  }
  template <int l> __device__ __forceinline__ R get(int i, const int (&c)[3]) const {
    return pull<l>(i, c[0] + 1);
  }
};

// BPull whose values are also stored as the node's reconstructed populations.
template <int D, int M, typename S, typename R> struct BStorePull {
  static constexpr int Q = Lat<D>::Q;
  BPull<D, M, S, R> p;
  R* P;
  long long st;
  template <int l> __device__ __forceinline__ void setup() {}
  template <int l> __device__ __forceinline__ void row(int, int) {}
  template <int l> __device__ __forceinline__ R get(int i, const int (&c)[3]) const {
    const R v = p.template pull<l>(i, c[0] + 1);
    P[(long long)(l * Q + i) * st] = v;
    return v;
  }
};

// The stored populations of one node.
template <int D, int M, typename S, typename R> struct BNode {
  static constexpr int Q = Lat<D>::Q;
  const S* src;
  const float4* codec;
  long long N, node;
  template <int l> __device__ __forceinline__ void setup() {}
  template <int l> __device__ __forceinline__ void row(int, int) {}
  template <int l> __device__ __forceinline__ R get(int i, const int (&)[3]) const {
    return Codec<S>::template dec<R>(__ldg(src + (long long)(l * Q + i) * N + node), codec,
                                     l * Q + i);
  }
};

// The local populations: incoming links at the state A, the others pulled.
template <int D, int M, typename S, typename R> struct BLocal {
  BPull<D, M, S, R> p;
  const BState<D, M, R>* A;
  const DevMech* m;
  const Units* un;
  ETab<D, M, R> ta;
  template <int l> __device__ __forceinline__ void setup() {
    ta.template build<l>(*A, *m, *un);
  }
  template <int l> __device__ __forceinline__ void row(int cy, int cz) {
    ta.template row<l>(cy, cz);
  }
  template <int l> __device__ __forceinline__ R get(int i, const int (&c)[3]) const {
    return p.incoming(i) ? ta.template evalx<l>(c[0]) : p.template pull<l>(i, c[0] + 1);
  }
};

// Step 4: the target + the local populations - the local equilibria L, stored
// as the node's reconstructed populations (the simplified inlet: the local
// equilibria).  same: the target is the state A of the incoming links, else Bt.
template <int D, int M, typename S, typename R> struct BFinal {
  static constexpr int Q = Lat<D>::Q;
  BLocal<D, M, S, R> lo;
  const BState<D, M, R>* Bt;
  const BState<D, M, R>* L;
  bool simple, same;
  R* P;
  long long st;
  ETab<D, M, R> tb, tl;
  __device__ __forceinline__ void store() {
    ForL<0, M + 1>::run([&](auto lc) {
      constexpr int l = decltype(lc)::value;
      lo.template setup<l>();
      if (!same) tb.template build<l>(*Bt, *lo.m, *lo.un);
      tl.template build<l>(*L, *lo.m, *lo.un);
#pragma unroll 1
      for (int yz = 0; yz < Q / 3; ++yz) {
        const int cy = yz % 3 - 1, cz = D == 3 ? yz / 3 - 1 : 0;
        lo.template row<l>(cy, cz);
        if (!same) tb.template row<l>(cy, cz);
        tl.template row<l>(cy, cz);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const int i = 3 * yz + k;
          const R loc = tl.template evalx<l>(k - 1), a = lo.ta.template evalx<l>(k - 1);
          const R t = same ? a : tb.template evalx<l>(k - 1);
          const R v = t + (lo.p.incoming(i) ? a : lo.p.template pull<l>(i, k)) - loc;
          P[(long long)(l * Q + i) * st] = simple ? loc : v;
        }
      }
    });
  }
};

// The sums of the reconstructed populations, target t + local populations
// (whose sums these are) - local equilibria l: the two equilibria's moments are
// known, so no pass over the populations is needed.  Explicitly fused (see
// mul1).
template <typename R>
__device__ __forceinline__ R final_momentum(R rt, R ut, R j, R rl, R ul) {
  return fma(rt, ut, fma(-rl, ul, j));
}
template <int D, int M, typename R, typename ST>
__device__ __forceinline__ R final_flux(int a, int b, const ST& t, R P, const ST& l) {
  const R pt = a == b ? fma(t.u[a], t.u[a], t.th) : mul1(t.u[a], t.u[b]);
  const R pl = a == b ? fma(l.u[a], l.u[a], l.th) : mul1(l.u[a], l.u[b]);
  return fma(t.rho, pt, fma(-l.rho, pl, P));
}
template <int D, typename R, typename ST>
__device__ __forceinline__ R state_energy(const ST& s) {       // U + u^2/2
  R q = mul1(s.u[0], s.u[0]);
#pragma unroll
  for (int d = 1; d < D; ++d) q = fma(s.u[d], s.u[d], q);
  return fma(R(0.5), q, s.U);
}
template <int D, int M, typename R>
__device__ __forceinline__ void final_sums(BSums<D, M, R>& z, const BState<D, M, R>& t,
                                           const BState<D, M, R>& l) {
  const R Et = state_energy<D, R>(t), El = state_energy<D, R>(l);
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    const R rt = mul1(t.rho, t.Y[a * kBnd]), rl = mul1(l.rho, l.Y[a * kBnd]);
#pragma unroll
    for (int d = 0; d < D; ++d)
      z.js[a][d] = final_momentum(rt, t.us ? t.us[(a * D + d) * kBnd] : t.u[d], z.js[a][d], rl,
                                  l.us ? l.us[(a * D + d) * kBnd] : l.u[d]);
    z.rs[a] = rt;
  }
#pragma unroll
  for (int d = 0; d < D; ++d) {
    z.j[d] = mul1(t.rho, t.u[d]);
    z.q[d] = final_momentum(mul1(t.rho, Et + t.th), t.u[d], z.q[d], mul1(l.rho, El + l.th),
                            l.u[d]);
  }
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int b = a; b < D; ++b)
      z.P[pidx<D>(a, b)] = final_flux<D, M, R>(a, b, t, z.P[pidx<D>(a, b)], l);
  z.rhoE = final_momentum(t.rho, Et, z.rhoE, l.rho, El);
  z.rho = t.rho;
}
// ... and of the local equilibria alone (simplified inlet)
template <int D, int M, typename R>
__device__ __forceinline__ void equilibrium_sums(BSums<D, M, R>& z, const BState<D, M, R>& l) {
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    z.rs[a] = mul1(l.rho, l.Y[a * kBnd]);
#pragma unroll
    for (int d = 0; d < D; ++d) z.js[a][d] = mul1(z.rs[a], l.u[d]);
  }
  const R E = state_energy<D, R>(l);
#pragma unroll
  for (int d = 0; d < D; ++d) {
    z.j[d] = mul1(l.rho, l.u[d]);
    z.q[d] = mul1(mul1(l.rho, E + l.th), l.u[d]);
  }
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int b = a; b < D; ++b)
      z.P[pidx<D>(a, b)] =
          mul1(l.rho, a == b ? fma(l.u[a], l.u[a], l.th) : mul1(l.u[a], l.u[b]));
  z.rhoE = mul1(l.rho, E);
  z.rho = l.rho;
}

// The boundary procedure of interface node k and its moment record.
// col: this thread's shared-memory column of R entries, sncol: its column of
// pull sources (both stride kBnd).
template <int D, int M, typename S, typename R>
__device__ __forceinline__ void bnode_body(const S* __restrict__ src, const BCDev& bc,
                                           R* __restrict__ rec, double* __restrict__ Tf,
                                           int* __restrict__ status, const Geom& g,
                                           const Units& un, const DevMech& m, int k,
                                           R* col, long long* sncol) {
  constexpr int Q = Lat<D>::Q;
  using RC = Rec<D, M>;
  using Pull = BPull<D, M, S, R>;
  const long long N = g.N;
  const long long n = bc.if_node[k];
  const int info = bc.if_info[k];
  const int kind = info & 15;
  const unsigned inc = bc.if_inc[k];
  // the pull sources: a row's directions share y and z
  const int x = (int)(n % g.nx);
  const int dx[3] = {wrap1(x + 1, g.nx), x, wrap1(x - 1, g.nx)};
  {
    const int y = (int)((n / g.nx) % g.ny);
    const int z = (int)(n / ((long long)g.nx * g.ny));
#pragma unroll 1
    for (int r = 0; r < Q / 3; ++r)
      sncol[r * kBnd] = node_shift<D>(x, y, z, 3 * r + 1, -1, g) - x;
  }
  const long long st = bc.n_if;
  const float4* codec = g.codec;
  BState<D, M, R> A, B, L;
  A.Y = col;
  L.Y = col + M * kBnd;
  B.Y = col + 2 * M * kBnd;                // spare column (outlet upstream state)
  L.us = col + 3 * M * kBnd;
  A.us = B.us = nullptr;
  BSums<D, M, R> z;

  if (kind == BK_BB) {
    // Eq. bb: incoming links take the node's own opposite post-collision
    // populations
    BStorePull<D, M, S, R> out{Pull{src, codec, N, n, sncol, {dx[0], dx[1], dx[2]}, inc, true},
                               static_cast<R*>(bc.pops) + k, st};
    bsums<D, M, R>(out, z);
  } else {
    if (kind == BK_TMS) {
      // step 1, Eqs. BBrho and BBY: bounce-back density and mass fractions
      Pull pull{src, codec, N, n, sncol, {dx[0], dx[1], dx[2]}, inc, true};
      bsums<D, M, R, true>(pull, z);
      A.rho = z.rho;
      const R irho = R(1) / z.rho;
      R ysum = R(0);
#pragma unroll
      for (int a = 0; a < M - 1; ++a) {
        const R Ya = z.rs[a] * irho;
        A.Y[a * kBnd] = Ya;
        ysum += Ya;
      }
      A.Y[(M - 1) * kBnd] = R(1) - ysum;
#pragma unroll
      for (int d = 0; d < D; ++d) A.u[d] = R(0);     // u^tgt = u_a^tgt = 0
      A.T = R(bc.if_wallT[k]);
      if (bc.if_nbr && bc.if_nbr[k] >= 0) {
        // off-grid targets (last paragraph of Sec. 4.2.2; reading R20): the
        // stored state of the fluid node x_f (Newton from this node's own T
        // guess, as for the outlet), interpolated along the wall normal
        // between the wall (at -delta) and x_f (at h)
        BState<D, M, R> sf = B;            // the spare and local-u_a columns, free now
        sf.us = L.us;
        BNode<D, M, S, R> nf{src, codec, N, (long long)bc.if_nbr[k]};
        bsums<D, M, R>(nf, z);
        bstate_of<D, M, R>(sf, z, __ldcg(Tf + n), m, un, status);
        const double h = bc.if_wh[k], dl = bc.if_wd[k];
        const R w = R(dl / (h + dl));
#pragma unroll
        for (int d = 0; d < D; ++d) A.u[d] = w * sf.u[d];
        A.us = col + (3 * M + M * D) * kBnd;
#pragma unroll
        for (int e = 0; e < M * D; ++e) A.us[e * kBnd] = w * sf.us[e * kBnd];
        A.T = R((h * bc.if_wallT[k] + dl * sf.T_full) / (h + dl));
      }
      bstate_prepare<D, M, R>(A, m, un);              // step 2: target (Eqs. tgtf-tgtfa)
    } else if (kind == BK_INLET) {
      A.rho = R(bc.rho_in);
#pragma unroll
      for (int a = 0; a < M; ++a) A.Y[a * kBnd] = R(bc.Y_in[a]);
#pragma unroll
      for (int d = 0; d < D; ++d) A.u[d] = R(bc.if_uin[(long long)d * st + k]);
      A.T = R(bc.T_in);
      bstate_prepare<D, M, R>(A, m, un);              // step 1 (Eqs. in_f-in_fa)
    } else {
      // LODI data from the stored state at x and x - n (Eq. convectiveBC,
      // reading R13); the upstream node's Newton starts from this node's T
      // guess (the bulk moments kernel may be rewriting the upstream one)
      const int ax = (info >> 4) & 3;
      const int sg = (info >> 6) & 1 ? 1 : -1;
      const long long stride =
          ax == 0 ? 1 : (ax == 1 ? (long long)g.nx : (long long)g.nx * g.ny);
      const long long up = n - sg * stride;
      BState<D, M, R> s0 = L, s1 = B;      // the local and spare columns, free until later
      s0.us = s1.us = nullptr;
      BNode<D, M, S, R> n0{src, codec, N, n};
      bsums<D, M, R>(n0, z);
      bstate_of<D, M, R>(s0, z, __ldcg(Tf + n), m, un, status);
      BNode<D, M, S, R> n1{src, codec, N, up};
      bsums<D, M, R>(n1, z);
      bstate_of<D, M, R>(s1, z, __ldcg(Tf + n), m, un, status);
      double R0 = 0.0, R1 = 0.0, Cv = 0.0;
      const double T0 = s0.T, T1 = s1.T;
#pragma unroll
      for (int a = 0; a < M; ++a) {
        const double Y0 = double(s0.Y[a * kBnd]), Y1 = double(s1.Y[a * kBnd]);
        R0 += Y0 * m.inv_mm[a];
        R1 += Y1 * m.inv_mm[a];
        Cv += Y0 * (m.u1[a] + T0 * (2.0 * m.u2[a] + 3.0 * T0 * m.u3[a]));
      }
      R0 *= R_U;
      R1 *= R_U;
      const double r0 = s0.rho, r1 = s1.rho;
      const double p0 = r0 * R0 * T0 * un.inv_c2;
      const double p1 = r1 * R1 * T1 * un.inv_c2;
      const double un0 = sg * double(s0.u[ax]), un1 = sg * double(s1.u[ax]);
      const double gamma = (Cv + R0) / Cv;
      const double cs = sqrt(gamma * R0 * T0 * un.inv_c2);
      const double Ma = un0 / cs;
      const double Ln = bc.outlet_L > 0.0 ? bc.outlet_L : (ax == 0 ? g.nx : (ax == 1 ? g.ny : g.nz));
      const double K = bc.sigma * (1.0 - Ma * Ma) * cs / Ln;
      const double L1 = K * (p0 - bc.p_out_lat);
      const double L2 = un0 * (cs * cs * (r0 - r1) - (p0 - p1));
      const double L5 = (un0 + cs) * ((p0 - p1) + r0 * cs * (un0 - un1));
      const double rho_o = r0 - (L2 + 0.5 * (L5 + L1)) / (cs * cs);
      const double p_o = p0 - 0.5 * (L5 + L1);
      const double un_o = un0 - (L5 - L1) / (2.0 * r0 * cs);
      A.rho = R(rho_o);
#pragma unroll
      for (int d = 0; d < D; ++d)
        A.u[d] = R(double(s0.u[d]) - un0 * double(s0.u[d] - s1.u[d]));
      A.u[ax] = R(sg * un_o);
      double Ro = 0.0;
#pragma unroll
      for (int a = 0; a < M; ++a) {
        const double Y0 = double(s0.Y[a * kBnd]);
        const double Ya = Y0 - un0 * (Y0 - double(s1.Y[a * kBnd]));
        A.Y[a * kBnd] = R(Ya);
        Ro += Ya * m.inv_mm[a];
      }
      A.T = R(p_o * un.c * un.c / (rho_o * R_U * Ro));
      bstate_prepare<D, M, R>(A, m, un);              // step 1 (Eqs. out_f-out_fa)
    }
    // the local state: incoming links at A, the others pulled (Eqs.
    // locRho-locT and their inlet / outlet analogues)
    BLocal<D, M, S, R> local{Pull{src, codec, N, n, sncol, {dx[0], dx[1], dx[2]}, inc, false},
                             &A, &m, &un, {}};
    bsums<D, M, R>(local, z);
    if (kind != BK_TMS) L.us = nullptr;               // TMS local species use u_a^loc
    bstate_of<D, M, R>(L, z, __ldcg(Tf + n), m, un, status);
    if (kind == BK_INLET) {                           // target (Eqs. in_tgt_*)
      B.rho = L.rho;
      B.Y = L.Y;
#pragma unroll
      for (int d = 0; d < D; ++d) B.u[d] = A.u[d];
      B.T = R(bc.T_in);
      bstate_prepare<D, M, R>(B, m, un);
    }
    // step 4 (Eqs. ftms-fatms, f_inlet-fa_inlet, f_outlet-fa_outlet)
    const bool simple = kind == BK_INLET && bc.inlet_simplified != 0, same = kind != BK_INLET;
    BFinal<D, M, S, R> fin{local, &B, &L, simple, same, static_cast<R*>(bc.pops) + k, st, {}, {}};
    fin.store();
    if (simple) equilibrium_sums<D, M, R>(z, L);
    else final_sums<D, M, R>(z, same ? A : B, L);
  }

  // the record from the sums of the reconstructed populations (the fields the
  // moments kernel records, T by Newton from the node's previous T); the
  // reaction sub-steps follow in their own kernel
  BState<D, M, R> s;
  s.Y = A.Y;                                    // the target columns are free now
  s.us = col + 3 * M * kBnd;
  R H[4];
  bstate_of<D, M, R>(s, z, __ldcg(Tf + n), m, un, status, H);
  if (!(s.rho > R(0)) || !isfinite(double(s.rho)) || !isfinite(s.T_full))
    atomicOr(status, ST_NONFINITE);
  Tf[n] = s.T_full;
  const R rr = s.rho;
#pragma unroll
  for (int a = 0; a < M - 1; ++a) rec[(RC::DRHO + a) * N + n] = s.Y[a * kBnd] * rr;
  rec[RC::RHO * N + n] = rr;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    rec[(RC::U + d) * N + n] = s.u[d];
    rec[(RC::Z + d) * N + n] = flux_less_work<D, R>(d, s.u, z.q, z.P);
    rec[(RC::PHI + d) * N + n] =
        rr * s.u[d] * (R(1) - R(3) * s.th) - rr * s.u[d] * s.u[d] * s.u[d];
  }
  rec[RC::E * N + n] = z.rhoE * (R(1) / rr);
  rec[RC::TH * N + n] = s.th;
  rec[RC::LNT * N + n] = ln_T0(s.T);
#pragma unroll
  for (int k = 0; k < 4; ++k) rec[(RC::H + k) * N + n] = H[k];
#pragma unroll
  for (int a = 0; a < M; ++a) {
    rec[(RC::Y + a) * N + n] = s.Y[a * kBnd];
#pragma unroll
    for (int d = 0; d < D; ++d)
      rec[(RC::US + a * D + d) * N + n] = record_us(s.us[(a * D + d) * kBnd] - s.u[d]);
  }
}

// ---------------------------------------------------------------------------
// The same procedure with one warp per interface node, for grids with few of
// them (boundary_warp_nodes): a thread per node is then a single chain of some
// thousand dependent loads and sums, whatever the node count (444 us in FP64,
// 355 us in FP32 for the 32 interface nodes of the 1024x4x4 flame, the
// critical path of its step; with a warp each, sub-steps included, 75 and 59).
// Lane 3 l + p holds lattice l's directions of
// c_z = p - 1 (D3Q27: 9 populations; D2Q9: 3, of c_y = p - 1); its loads are
// in flight together, its sums go through shared memory to every lane, and
// the sums over the species are butterflies over 16 lanes (lane & 15 = the
// species).  In FP64 the sums are taken in another order than in bnode_body
// (the two agree to rounding); FP32 sums keep its order, whose rounding a
// flame's front would amplify.

template <int D, int M> struct WB {
  static constexpr int Q = Lat<D>::Q, NP = Lat<D>::NP;
  static constexpr int NR = D == 3 ? 9 : 3;        // populations per lane
  static constexpr int ZS = 1 + D;                 // sums per lattice
  static constexpr int Z = 0, P = Z + (M + 1) * ZS;    // sums, momentum flux of f
  static constexpr int ST = P + NP;                // states: Y [M], u_a [M D]
  static constexpr int SS = M + M * D;
  static constexpr int N = ST + 4 * SS;            // R entries per warp
};

// A state: scalars in every lane, Y and the species velocities (us; used:
// nullptr when u serves every species) in the warp's shared memory.
template <int D, int M, typename R> struct WState {
  R rho, T, th, U;
  R u[D];
  R *Y, *us;
  bool own_us;
  double T_full;
};

__device__ __forceinline__ float shfl_xor_ct(unsigned mask, float v, int o) {
  return __shfl_xor_sync(mask, v, o);
}
template <typename V>
__device__ __forceinline__ V species_sum(V v) {
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) v += shfl_xor_ct(0xffffffffu, v, o);
  return v;
}

// theta, U/c^2 from T and Y (bstate_prepare)
template <int D, int M, typename R>
__device__ __forceinline__ void wprepare(WState<D, M, R>& s, const DevMech& m, const Units& un,
                                         int lane) {
  using CT = typename ChemType<R>::type;
  const int a = min(lane & 15, M - 1);
  const R Ya = (lane & 15) < M ? s.Y[a] : R(0);
  if constexpr (!kFF<R>) {
    const double Rm = species_sum(double(Ya) * m.inv_mm[a]);
    const double U = species_sum(double(Ya) * species_U(m, a, double(s.T)));
    s.th = R(R_U * Rm * double(s.T) * un.inv_c2);
    s.U = R(U * un.inv_c2);
  } else {
    float Rm = 0.f;
#pragma unroll
    for (int b = 0; b < M; ++b) Rm += s.Y[b] * m.inv_mm_s[b];
    const CT U = species_sum(ff(Ya) * species_U_ff(m, a, ff(s.T)));
    s.th = float(R_U) * Rm * s.T * un.inv_c2_s;
    s.U = (U * un.inv_c2_f).hi;
  }
}

// This lane's partial sums of its populations v; the lattice's totals (and
// the f lattice's momentum flux) in z.
template <int D, int M, typename R>
__device__ __forceinline__ void wsums(const R (&v)[WB<D, M>::NR], R* z, int lane) {
  using W = WB<D, M>;
  const int l = lane / 3, p = lane % 3;
  const bool on = lane < 3 * (M + 1);
  R sum = R(0), sj[D], sP[W::NP];
#pragma unroll
  for (int d = 0; d < D; ++d) sj[d] = R(0);
#pragma unroll
  for (int q = 0; q < W::NP; ++q) sP[q] = R(0);
  // a row (c_y, c_z) of sum sr, difference dx and sx = f_+ + f_-
  auto add_row = [&](R sr, R dx, R sx, int cy, int cz) {
    sum += sr;
    sj[0] += dx;
    sP[pidx<D>(0, 0)] += sx;
    if (cy != 0) {
      sj[1] += cy > 0 ? sr : -sr;
      sP[pidx<D>(1, 1)] += sr;
      sP[pidx<D>(0, 1)] += cy > 0 ? dx : -dx;
    }
    if constexpr (D == 3) {
      if (cz != 0) {
        sj[2] += cz > 0 ? sr : -sr;
        sP[pidx<D>(2, 2)] += sr;
        sP[pidx<D>(0, 2)] += cz > 0 ? dx : -dx;
        if (cy != 0) sP[pidx<D>(1, 2)] += cy == cz ? sr : -sr;
      }
    }
  };
  const int l0 = min(3 * l, 27);
  if constexpr (sizeof(R) == 4) {
    // bsums' order: row after row, every lane of the lattice the whole sum
#pragma unroll
    for (int pp = 0; pp < 3; ++pp)
#pragma unroll
      for (int r = 0; r < W::NR / 3; ++r) {
        R w[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) w[q] = __shfl_sync(0xffffffffu, v[3 * r + q], l0 + pp);
        const R sx = w[0] + w[2];
        if constexpr (D == 3) add_row(sx + w[1], w[2] - w[0], sx, r - 1, pp - 1);
        else add_row(sx + w[1], w[2] - w[0], sx, pp - 1, 0);
      }
  } else {
#pragma unroll
    for (int r = 0; r < W::NR / 3; ++r) {
      const R sx = v[3 * r] + v[3 * r + 2], dx = v[3 * r + 2] - v[3 * r];
      add_row(sx + v[3 * r + 1], dx, sx, D == 3 ? r - 1 : 0, 0);
    }
    // the terms with this lane's own velocity component p - 1 (c_z; D2Q9: c_y)
    const R c = on ? R(p - 1) : R(0);
    sj[D - 1] = c * sum;
    if constexpr (D == 3) {
      sP[pidx<D>(2, 2)] = c * c * sum;
      sP[pidx<D>(0, 2)] = c * sj[0];
      sP[pidx<D>(1, 2)] = c * sj[1];
    } else {
      sP[pidx<D>(1, 1)] = c * c * sum;
      sP[pidx<D>(0, 1)] = c * sj[0];
    }
    auto total = [&](R x) {
      const R y0 = __shfl_sync(0xffffffffu, x, l0), y1 = __shfl_sync(0xffffffffu, x, l0 + 1),
              y2 = __shfl_sync(0xffffffffu, x, l0 + 2);
      return y0 + y1 + y2;
    };
    sum = total(sum);
#pragma unroll
    for (int d = 0; d < D; ++d) sj[d] = total(sj[d]);
#pragma unroll
    for (int q = 0; q < W::NP; ++q) sP[q] = total(sP[q]);
  }
  __syncwarp();                        // the previous sums' readers are done
  if (on && p == 0) {
    z[W::Z + l * W::ZS] = sum;
#pragma unroll
    for (int d = 0; d < D; ++d) z[W::Z + l * W::ZS + 1 + d] = sj[d];
    if (l == M - 1)
#pragma unroll
      for (int q = 0; q < W::NP; ++q) z[W::P + q] = sP[q];
  }
  __syncwarp();
}

// The macroscopic state of the sums in z (bstate_of).
template <int D, int M, typename R>
__device__ __forceinline__ void wstate_of(WState<D, M, R>& s, const R* z, double T_guess,
                                          const DevMech& m, const Units& un, int* status,
                                          int lane, R* H = nullptr) {
  using W = WB<D, M>;
  using CT = typename ChemType<R>::type;
  using X = Chem<CT>;
  const int sp = lane & 15, a = min(sp, M - 1);
  const R* zf = z + W::Z + (M - 1) * W::ZS;
  s.rho = zf[0];
  const R irho = R(1) / s.rho;
  R usq = R(0);
#pragma unroll
  for (int d = 0; d < D; ++d) { s.u[d] = zf[1 + d] * irho; usq += s.u[d] * s.u[d]; }
  // rho_a, j_a: the slaved species from the mixture
  R q[W::ZS];
#pragma unroll
  for (int e = 0; e < W::ZS; ++e) {
    const R mine = sp < M - 1 ? z[W::Z + a * W::ZS + e] : R(0);
    R rest = zf[e];
    if constexpr (sizeof(R) == 4) {
#pragma unroll
      for (int b = 0; b < M - 1; ++b) rest -= z[W::Z + b * W::ZS + e];
    } else {
      rest -= species_sum(mine);
    }
    q[e] = sp < M - 1 ? mine : rest;
  }
  const R Ya = sp < M ? q[0] * irho : R(0);
  if (lane < M) {
    s.Y[a] = Ya;
    if (s.own_us) {
      R ja[D];
#pragma unroll
      for (int d = 0; d < D; ++d) ja[d] = q[1 + d];
      const bool tiny = species_velocity_undefined<D, R>(q[0], ja);
#pragma unroll
      for (int d = 0; d < D; ++d) s.us[a * D + d] = tiny ? s.u[d] : ja[d] / q[0];
    }
  }
  __syncwarp();
  CT c[4], U;
#pragma unroll
  for (int k = 0; k < 4; ++k) c[k] = species_sum(X::of(Ya) * X::ucoef(m, k, a));
  const R rhoE = z[W::Z + M * W::ZS];
  if constexpr (!kFF<R>) U = (double(rhoE * irho) - 0.5 * double(usq)) * un.c * un.c;
  else U = (ff(rhoE * irho) + ff(-0.5f * usq)) * un.c2_f;
  bool ok;
  const CT T = newton_poly(c, U, X::of_T(T_guess), un.newton_max_iter, X::rtol(un), ok);
  if constexpr (!kFF<R>) {
    s.T = R(T);
    s.T_full = T;
  } else {
    s.T = T.hi;
    s.T_full = ff_to_double(T);
  }
  if (!ok && lane == 0) atomicOr(status, ST_NEWTON);
  if (H) {
    R Rm = R(0), h[4];
    if constexpr (sizeof(R) == 4) {
#pragma unroll
      for (int b = 0; b < M; ++b) Rm += s.Y[b] * m.inv_mm_s[b];
    } else {
      Rm = species_sum(Ya * m.inv_mm[a]);
    }
    enthalpy_poly(c, Rm, un, h);
#pragma unroll
    for (int k = 0; k < 4; ++k) H[k] = h[k];
  }
  wprepare<D, M, R>(s, m, un, lane);
}

// Equilibrium populations of a state in this lane's lattice and directions.
template <int D, int M, typename R>
__device__ __forceinline__ void wequilibrium(const WState<D, M, R>& s, const DevMech& m,
                                             const Units& un, int lane, R (&e)[WB<D, M>::NR]) {
  using W = WB<D, M>;
  const int l = min(lane / 3, M), p = lane % 3;
  if (l < M) {
    R th = s.th, pref = s.rho;
    if (l < M - 1) {
      if constexpr (sizeof(R) == 8) th = R(m.Ra[l] * double(s.T) * un.inv_c2);
      else th = m.Ra_s[l] * s.T * un.inv_c2_s;
      pref = s.rho * s.Y[l];
    }
    R t[D][3];
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const R xi = l < M - 1 && s.own_us ? s.us[l * D + d] : s.u[d];
      const R P = th + xi * xi;
      t[d][0] = R(0.5) * (P - xi);
      t[d][1] = R(1) - P;
      t[d][2] = R(0.5) * (P + xi);
    }
    const R tp = sel3(p - 1, t[D - 1]);
#pragma unroll
    for (int r = 0; r < W::NR / 3; ++r) {
      const R w = D == 3 ? pref * t[1][r] * tp : pref * tp;
#pragma unroll
      for (int k = 0; k < 3; ++k) e[3 * r + k] = mul1(w, t[0][k]);
    }
  } else {
    BState<D, M, R> b;
    b.rho = s.rho;
    b.th = s.th;
    b.U = s.U;
#pragma unroll
    for (int d = 0; d < D; ++d) b.u[d] = s.u[d];
    GTab<D, R> g;
    gtab<D, M, R>(b, g);
    const R az = sel3(p - 1, g.A[D - 1]), bz = sel3(p - 1, g.B[D - 1]);
#pragma unroll
    for (int r = 0; r < W::NR / 3; ++r) {
      const R P = D == 3 ? mul1(g.A[1][r], az) : az;
      const R Qv = D == 3 ? fma(g.U, P, fma(g.B[1][r], az, mul1(g.A[1][r], bz)))
                          : fma(g.U, az, bz);
#pragma unroll
      for (int k = 0; k < 3; ++k)
        e[3 * r + k] = mul1(g.rho, fma(g.A[0][k], Qv, mul1(g.B[0][k], P)));
    }
  }
}

// Interface node k by one warp; sm: the warp's WB::N entries; m: the
// mechanism's global copy (indexed by lane); cs: this thread's slice for the
// sub-steps.
template <int D, int M, typename S, typename R, typename Slice>
__device__ __forceinline__ void bnode_warp(const S* __restrict__ src, const BCDev& bc,
                                           R* __restrict__ rec, double* __restrict__ Tf,
                                           int* __restrict__ status, const Geom& g,
                                           const Units& un, const DevMech& m, int k, R* sm,
                                           int lane, Slice& cs) {
  using W = WB<D, M>;
  using RC = Rec<D, M>;
  constexpr int Q = W::Q;
  const long long N = g.N;
  const long long n = bc.if_node[k];
  const int info = bc.if_info[k], kind = info & 15;
  const unsigned inc = bc.if_inc[k];
  const bool on = lane < 3 * (M + 1);
  const int l = min(lane / 3, M), p = lane % 3;
  const int i0 = p * W::NR;                        // the lane's directions i0 .. i0 + NR - 1
  const int x = (int)(n % g.nx);
  const int y = (int)((n / g.nx) % g.ny);
  const int z = (int)(n / ((long long)g.nx * g.ny));
  auto at = [&](long long node, int i) {
    return Codec<S>::template dec<R>(__ldg(src + (long long)(l * Q + i) * N + node), g.codec,
                                     l * Q + i);
  };
  auto stored = [&](long long node, R (&v)[W::NR]) {
#pragma unroll
    for (int j = 0; j < W::NR; ++j) v[j] = at(node, i0 + j);
  };
  R pull[W::NR], v[W::NR];
#pragma unroll
  for (int j = 0; j < W::NR; ++j) pull[j] = at(node_shift<D>(x, y, z, i0 + j, -1, g), i0 + j);
  const double Tg = __ldcg(Tf + n);
  auto incoming = [&](int j) { return (inc >> (i0 + j) & 1u) != 0; };
  WState<D, M, R> A, B, L;
  A.Y = sm + W::ST;
  B.Y = A.Y + W::SS;
  L.Y = B.Y + W::SS;
  R* const Fs = L.Y + W::SS;
  A.us = A.Y + M;
  B.us = B.Y + M;
  L.us = L.Y + M;
  A.own_us = B.own_us = L.own_us = false;

  if (kind == BK_BB) {
#pragma unroll
    for (int j = 0; j < W::NR; ++j) v[j] = incoming(j) ? at(n, Q - 1 - i0 - j) : pull[j];
  } else {
    if (kind == BK_TMS) {
#pragma unroll
      for (int j = 0; j < W::NR; ++j) v[j] = incoming(j) ? at(n, Q - 1 - i0 - j) : pull[j];
      wsums<D, M, R>(v, sm, lane);
      A.rho = sm[W::Z + (M - 1) * W::ZS];
      const R irho = R(1) / A.rho;
      const int sp = lane & 15;
      const R Ya = sp < M - 1 ? sm[W::Z + min(sp, M - 1) * W::ZS] * irho : R(0);
      R last = R(1);
      if constexpr (sizeof(R) == 4) {
        R ysum = R(0);
#pragma unroll
        for (int b = 0; b < M - 1; ++b) ysum += mul1(sm[W::Z + b * W::ZS], irho);
        last -= ysum;
      } else {
        last -= species_sum(Ya);
      }
      if (lane < M) A.Y[lane] = lane < M - 1 ? Ya : last;
#pragma unroll
      for (int d = 0; d < D; ++d) A.u[d] = R(0);
      A.T = R(bc.if_wallT[k]);
      __syncwarp();
      if (bc.if_nbr && bc.if_nbr[k] >= 0) {
        B.own_us = true;
        stored(bc.if_nbr[k], v);
        wsums<D, M, R>(v, sm, lane);
        wstate_of<D, M, R>(B, sm, Tg, m, un, status, lane);
        const double h = bc.if_wh[k], dl = bc.if_wd[k];
        const R w = R(dl / (h + dl));
#pragma unroll
        for (int d = 0; d < D; ++d) A.u[d] = w * B.u[d];
        A.own_us = true;
        for (int e = lane; e < M * D; e += 32) A.us[e] = w * B.us[e];
        A.T = R((h * bc.if_wallT[k] + dl * B.T_full) / (h + dl));
        B.own_us = false;
        __syncwarp();
      }
    } else if (kind == BK_INLET) {
      A.rho = R(bc.rho_in);
      if (lane < M) A.Y[lane] = R(bc.Y_in[lane]);
#pragma unroll
      for (int d = 0; d < D; ++d) A.u[d] = R(bc.if_uin[(long long)d * bc.n_if + k]);
      A.T = R(bc.T_in);
      __syncwarp();
    } else {
      const int ax = (info >> 4) & 3;
      const int sg = (info >> 6) & 1 ? 1 : -1;
      const long long stride =
          ax == 0 ? 1 : (ax == 1 ? (long long)g.nx : (long long)g.nx * g.ny);
      R v1[W::NR];
      stored(n, v);
      stored(n - sg * stride, v1);
      wsums<D, M, R>(v, sm, lane);
      wstate_of<D, M, R>(L, sm, Tg, m, un, status, lane);
      wsums<D, M, R>(v1, sm, lane);
      wstate_of<D, M, R>(B, sm, Tg, m, un, status, lane);
      auto pick3 = [&](const R (&u)[D]) {
        R w = u[0];
#pragma unroll
        for (int d = 1; d < D; ++d)
          if (ax == d) w = u[d];
        return double(w);
      };
      const int sp = lane & 15, a = min(sp, M - 1);
      const double T0 = L.T, T1 = B.T;
      const double Y0 = sp < M ? double(L.Y[a]) : 0.0, Y1 = sp < M ? double(B.Y[a]) : 0.0;
      const double R0 = R_U * species_sum(Y0 * m.inv_mm[a]);
      const double R1 = R_U * species_sum(Y1 * m.inv_mm[a]);
      const double Cv =
          species_sum(Y0 * (m.u1[a] + T0 * (2.0 * m.u2[a] + 3.0 * T0 * m.u3[a])));
      const double r0 = L.rho, r1 = B.rho;
      const double p0 = r0 * R0 * T0 * un.inv_c2;
      const double p1 = r1 * R1 * T1 * un.inv_c2;
      const double un0 = sg * pick3(L.u), un1 = sg * pick3(B.u);
      const double gamma = (Cv + R0) / Cv;
      const double cs = sqrt(gamma * R0 * T0 * un.inv_c2);
      const double Ma = un0 / cs;
      const double Ln =
          bc.outlet_L > 0.0 ? bc.outlet_L : (ax == 0 ? g.nx : (ax == 1 ? g.ny : g.nz));
      const double K = bc.sigma * (1.0 - Ma * Ma) * cs / Ln;
      const double L1 = K * (p0 - bc.p_out_lat);
      const double L2 = un0 * (cs * cs * (r0 - r1) - (p0 - p1));
      const double L5 = (un0 + cs) * ((p0 - p1) + r0 * cs * (un0 - un1));
      const double rho_o = r0 - (L2 + 0.5 * (L5 + L1)) / (cs * cs);
      const double p_o = p0 - 0.5 * (L5 + L1);
      const double un_o = un0 - (L5 - L1) / (2.0 * r0 * cs);
      A.rho = R(rho_o);
#pragma unroll
      for (int d = 0; d < D; ++d)
        A.u[d] = d == ax ? R(sg * un_o) : R(double(L.u[d]) - un0 * double(L.u[d] - B.u[d]));
      const double Ya = Y0 - un0 * (Y0 - Y1);
      const double Ro = species_sum(Ya * m.inv_mm[a]);
      if (lane < M) A.Y[lane] = R(Ya);
      A.T = R(p_o * un.c * un.c / (rho_o * R_U * Ro));
      __syncwarp();
    }
    wprepare<D, M, R>(A, m, un, lane);
    // the local state: incoming links at A, the others pulled
    R ea[W::NR], el[W::NR];
    wequilibrium<D, M, R>(A, m, un, lane, ea);
#pragma unroll
    for (int j = 0; j < W::NR; ++j) v[j] = incoming(j) ? ea[j] : pull[j];
    wsums<D, M, R>(v, sm, lane);
    L.own_us = kind == BK_TMS;
    wstate_of<D, M, R>(L, sm, Tg, m, un, status, lane);
    wequilibrium<D, M, R>(L, m, un, lane, el);
    if (kind == BK_INLET && bc.inlet_simplified != 0) {
#pragma unroll
      for (int j = 0; j < W::NR; ++j) v[j] = el[j];
    } else if (kind == BK_INLET) {
      R eb[W::NR];
      B.rho = L.rho;
      B.Y = L.Y;
#pragma unroll
      for (int d = 0; d < D; ++d) B.u[d] = A.u[d];
      B.T = R(bc.T_in);
      wprepare<D, M, R>(B, m, un, lane);
      wequilibrium<D, M, R>(B, m, un, lane, eb);
#pragma unroll
      for (int j = 0; j < W::NR; ++j) v[j] = eb[j] + (incoming(j) ? ea[j] : pull[j]) - el[j];
    } else {
#pragma unroll
      for (int j = 0; j < W::NR; ++j) v[j] = ea[j] + (incoming(j) ? ea[j] : pull[j]) - el[j];
    }
    // their sums (final_sums, equilibrium_sums), a lattice per lane
    const bool simple = kind == BK_INLET && bc.inlet_simplified != 0;
    const WState<D, M, R>& t = simple ? L : (kind == BK_INLET ? B : A);
    const R Et = state_energy<D, R>(t), El = state_energy<D, R>(L);
    __syncwarp();                        // the sums' readers (wstate_of) are done
    if (lane <= M) {
      R* zl = sm + W::Z + lane * W::ZS;
      if (lane < M - 1) {
        const R rt = mul1(t.rho, t.Y[lane]), rl = mul1(L.rho, L.Y[lane]);
#pragma unroll
        for (int d = 0; d < D; ++d) {
          const R ut = t.own_us ? t.us[lane * D + d] : t.u[d];
          zl[1 + d] = simple ? mul1(rt, ut)
                             : final_momentum(rt, ut, zl[1 + d], rl,
                                              L.own_us ? L.us[lane * D + d] : L.u[d]);
        }
        zl[0] = rt;
      } else if (lane == M - 1) {
        zl[0] = t.rho;
#pragma unroll
        for (int d = 0; d < D; ++d) zl[1 + d] = mul1(t.rho, t.u[d]);
#pragma unroll
        for (int a = 0; a < D; ++a)
#pragma unroll
          for (int b = a; b < D; ++b) {
            R& P = sm[W::P + pidx<D>(a, b)];
            P = simple ? mul1(t.rho, a == b ? fma(t.u[a], t.u[a], t.th) : mul1(t.u[a], t.u[b]))
                       : final_flux<D, M, R>(a, b, t, P, L);
          }
      } else {
        zl[0] = simple ? mul1(t.rho, Et) : final_momentum(t.rho, Et, zl[0], L.rho, El);
#pragma unroll
        for (int d = 0; d < D; ++d)
          zl[1 + d] = simple ? mul1(mul1(t.rho, Et + t.th), t.u[d])
                             : final_momentum(mul1(t.rho, Et + t.th), t.u[d], zl[1 + d],
                                              mul1(L.rho, El + L.th), L.u[d]);
      }
    }
    __syncwarp();
  }
  if (kind == BK_BB) wsums<D, M, R>(v, sm, lane);
  if (on)
#pragma unroll
    for (int j = 0; j < W::NR; ++j)
      static_cast<R*>(bc.pops)[(long long)(l * Q + i0 + j) * bc.n_if + k] = v[j];

  // the record
  WState<D, M, R> s;
  s.Y = Fs;
  s.us = Fs + M;
  s.own_us = true;
  R H[4];
  wstate_of<D, M, R>(s, sm, Tg, m, un, status, lane, H);
  const R rr = s.rho;
  if (lane == 0) {
    if (!(rr > R(0)) || !isfinite(double(rr)) || !isfinite(s.T_full))
      atomicOr(status, ST_NONFINITE);
    Tf[n] = s.T_full;
    rec[RC::RHO * N + n] = rr;
    rec[RC::E * N + n] = sm[W::Z + M * W::ZS] * (R(1) / rr);
    rec[RC::TH * N + n] = s.th;
    rec[RC::LNT * N + n] = ln_T0(s.T);
#pragma unroll
    for (int k = 0; k < 4; ++k) rec[(RC::H + k) * N + n] = H[k];
  }
#pragma unroll
  for (int d = 0; d < D; ++d) {
    if (lane == 1 + d) {
      rec[(RC::U + d) * N + n] = s.u[d];
      rec[(RC::Z + d) * N + n] =
          flux_less_work<D, R>(d, s.u, sm + W::Z + M * W::ZS + 1, sm + W::P);
      rec[(RC::PHI + d) * N + n] =
          rr * s.u[d] * (R(1) - R(3) * s.th) - rr * s.u[d] * s.u[d] * s.u[d];
    }
  }
  for (int a = lane; a < M; a += 32) rec[(RC::Y + a) * N + n] = s.Y[a];
#pragma unroll
  for (int d = 0; d < D; ++d)
    for (int a = lane; a < M; a += 32)
      rec[(RC::US + a * D + d) * N + n] = record_us(s.us[a * D + d] - s.u[d]);

  // the reaction sub-steps, the reactions over the warp's lanes
  using CT = typename ChemType<R>::type;
  using X = Chem<CT>;
  CT r[M], r0[M - 1], U;
  R last = rr, usq = R(0);
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    const R ra = s.Y[a] * rr;
    last -= ra;
    r0[a] = r[a] = X::of(ra);
  }
  r[M - 1] = X::of(last);
#pragma unroll
  for (int d = 0; d < D; ++d) usq += s.u[d] * s.u[d];
  const R ER = sm[W::Z + M * W::ZS] * (R(1) / rr);
  if constexpr (kFF<R>) U = (ff(ER) + ff(-0.5f * usq)) * un.c2_f;
  else U = (double(ER) - 0.5 * double(usq)) * un.c * un.c;
  chem_group_substeps<M, CT, 32>(r, X::inv(X::of(rr)), U, X::of_T(s.T_full), un, m, lane,
                                 0xffffffffu, status, cs);
#pragma unroll
  for (int a = 0; a < M - 1; ++a) {
    if (a != lane) continue;
    if constexpr (kFF<R>) rec[(RC::DRHO + a) * N + n] = (r[a] - r0[a]).hi;
    else rec[(RC::DRHO + a) * N + n] = R(r[a] - r0[a]);
  }
}
