// lbm_split.cuh -- the fused collide + stream with the lattices of a node
// shared out over the warps of a block.
//
// A block takes tiles of 32 nodes, one per lane.  Per tile:
//   1. the warps share out the velocities (16-bit storage: the nine rows of
//      three, each in two parts): the populations of every lattice are
//      loaded, decoded, given the terms still due (lbm_stencil.cuh,
//      lbm_eqcodec.cuh) and staged in shared memory.  The velocity is data of a
//      loop, not unrolled: unrolled, 16-bit decoding overflows the
//      instruction cache;
//   2. warp r < NP takes the species pair (2r, 2r + 1), its two species the
//      lanes of paired FP32 instructions, warp NP takes f, warp NP + 1 takes
//      g, and each sums its lattices' moments;
//   3. the node closure (coupling, thermodynamics, transport, the
//      Stefan-Maxwell system) runs with LPN lanes per node, a species pair and
//      two rows of the system per lane, sums and pivot rows by shuffles;
//   4. each warp updates and stores its lattices.
// Species and momentum updates are formed in moment space.  The product form
// of Sec. 2.4 is Psi_c = (sum over p of) t_cp m_p per axis with
// m = (1, xi, xi^2 + zeta), so a lattice's 27 values are one fixed transform
// (t x t x t) of its 27 product moments, and everything added to a species
// (its equilibrium and the forces of all other species, Eq. fstar1) is summed
// as moments and transformed once.  Moments are kept halved per axis index
// (hx = xi / 2, hs = (xi^2 + zeta) / 2), which makes the transform
//   c = -1: m2 - m1,   c = 0: m0 - 2 m2,   c = +1: m2 + m1.
// Equilibria enter as deviations from the reference rest state, telescoped
// over the axes, as in lbm_collide.cuh.
#pragma once

#include "lbm_stencil.cuh"
#include "lbm_collide.cuh"

namespace lbm {

// Product moments of a lattice's equilibrium deviation from the reference
// rest state, divided by the lattice's density:
//   e_pqr = a_p a_q a_r - r_p r_q r_r,  a = (1, hx, hs), r = (1, 0, hr),
// telescoped with da = a - r = (0, hx, hd).
template <class V>
struct RestDeviation {
  V h1[3], h2[3], d2[3], r2;
  template <int P> __device__ __forceinline__ V a(int ax) const { return P == 1 ? h1[ax] : h2[ax]; }
  template <int P> __device__ __forceinline__ V d(int ax) const { return P == 1 ? h1[ax] : d2[ax]; }
  // (y, z) part: a_q a_r, and da_q a_r + r_q da_r
  template <int Qy, int R> __device__ __forceinline__ V ayz() const {
    if constexpr (Qy == 0) return a<R>(2);
    else if constexpr (R == 0) return a<Qy>(1);
    else return vmul(a<Qy>(1), a<R>(2));
  }
  template <int Qy, int R> __device__ __forceinline__ V fyz() const {
    if constexpr (Qy == 0) return d<R>(2);
    else if constexpr (R == 0) return d<Qy>(1);
    else if constexpr (Qy == 1) return vmul(h1[1], a<R>(2));
    else return vfma(d2[1], a<R>(2), vmul(r2, d<R>(2)));
  }
  template <int Pp, int Qy, int R> __device__ __forceinline__ V e() const {
    constexpr bool yz0 = Qy == 0 && R == 0;
    if constexpr (Pp == 0) return fyz<Qy, R>();
    else if constexpr (yz0) return d<Pp>(0);
    else if constexpr (Pp == 1) return vmul(h1[0], ayz<Qy, R>());
    else return vfma(d2[0], ayz<Qy, R>(), vmul(r2, fyz<Qy, R>()));
  }
  // the moment of the rest state itself (zero unless every index is even)
  template <int Pp, int Qy, int R> static constexpr int rest_power() {
    return (Pp == 1 || Qy == 1 || R == 1) ? -1 : (Pp + Qy + R) / 2;
  }
};

// The 27 velocities of moments given plane by plane (plane<R>(m): m[3q + p]).
// emit<I>(value) for every velocity but the rest one, rest(value) last; the
// rest value is the remainder of the zeroth moment m000.
template <class Scalar, class V, class Plane, class Emit, class Rest>
__device__ __forceinline__ void from_moments(V m000, Plane&& plane, Emit&& emit, Rest&& rest) {
  auto xy = [&](auto R_, V (&t)[9]) {
    V m[9];
    plane(R_, m);
    const V two = bcast<V>(Scalar(-2));
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const V a = m[3 * q], b = m[3 * q + 1], c = m[3 * q + 2];
      t[3 * q] = vsub(c, b); t[3 * q + 1] = vfma(two, c, a); t[3 * q + 2] = vadd(c, b);
    }
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const V a = t[x], b = t[3 + x], c = t[6 + x];
      t[x] = vsub(c, b); t[3 + x] = vfma(two, c, a); t[6 + x] = vadd(c, b);
    }
  };
  V t1[9], t2[9], s;
  xy(std::integral_constant<int, 1>{}, t1);
  xy(std::integral_constant<int, 2>{}, t2);
  static_for<0, 9>([&](auto K_) {
    constexpr int k = decltype(K_)::value;
    const V lo = vsub(t2[k], t1[k]), hi = vadd(t2[k], t1[k]);
    emit(std::integral_constant<int, k>{}, lo);
    emit(std::integral_constant<int, 18 + k>{}, hi);
    const V both = vadd(lo, hi);
    s = k == 0 ? both : vadd(s, both);
  });
  xy(std::integral_constant<int, 0>{}, t1);
  static_for<0, 9>([&](auto K_) {
    constexpr int k = decltype(K_)::value;
    if constexpr (k != 4) {
      const V v = vsub(t1[k], vadd(t2[k], t2[k]));
      emit(std::integral_constant<int, 9 + k>{}, v);
      s = vadd(s, v);
    }
  });
  rest(vsub(m000, s));
}

template <int M>
struct Split {
  static constexpr int NP = (M + 1) / 2;                       // species pairs, species warps
  static constexpr int WARPS = NP + 2, THREADS = 32 * WARPS;
  static constexpr int LPN = NP <= 1 ? 1 : (NP <= 2 ? 2 : 4);  // closure lanes per node, a species pair each
  // Row stride of the closure's per-node pairs: its lanes (32 / LPN
  // neighbouring nodes of LPN rows) fall in distinct banks.
  static constexpr int LD = LPN == 1 ? 32 : 32 + 32 / LPN;
  // Shared memory, in Reals; arrays of pairs first.
  static constexpr int TAB = 0;                                // [8][LPN] constants, [M][LPN] phi_ab / m_b, C_ab
  static constexpr int TABC = TAB + 2 * LPN * (8 + 2 * M);     // C_ab as [M a][NP b pairs]
  static constexpr int STAGE = TABC + 2 * M * NP;              // species populations [27][NP][32] pairs
  static constexpr int DIF = STAGE + 27 * NP * 64;             // force moments [26][NP][32] pairs
  static constexpr int MOM = DIF;                              // species moments [4][LPN][LD] pairs (before DIF is written)
  static constexpr int DIF_SIZE = NP > 1 ? 26 * NP * 64 : 0, MOM_SIZE = 8 * LPN * LD;
  static constexpr int SP = DIF + (DIF_SIZE > MOM_SIZE ? DIF_SIZE : MOM_SIZE);   // closed species [7][LPN][LD] pairs
  static constexpr int FG = SP + 14 * LPN * LD;                // f, g populations [27][2][32]
  static constexpr int ND = FG + 27 * 64;                      // node rows [.][32]
  static constexpr int REALS = ND + 24 * 32;
};
enum SplitTab { ST_RL, ST_YR, ST_IM, ST_CV, ST_CP, ST_MU, ST_LAM, ST_ILAM };
enum SplitSp { SS_RA, SS_RD, SS_V, SS_BETA = SS_V + 3, SS_TY };
enum SplitNode { SN_RHOD, SN_J, SN_RHOED = SN_J + 3, SN_S, SN_DT = SN_S + 6, SN_DTH, SN_OM, SN_OM1, SN_CP, SN_HYV,
                 SN_USP = SN_HYV + 3, SN_RHOSP = SN_USP + 3 };
static_assert(SN_RHOSP < 24, "node rows");

// Sum of a quantity over the species of a node.
template <int LPN, class V>
__device__ __forceinline__ auto species_sum(V v) -> decltype(v.x) {
  auto s = v.x + v.y;
#pragma unroll
  for (int o = LPN / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, LPN);
  return s;
}

// Gauss-Jordan elimination of the M x M system whose rows 2a, 2a + 1 lane a
// of the group holds (columns diagonally dominant: no pivoting, see
// sm_eliminate).
template <int M, int LPN, class V>
__device__ __forceinline__ void lanes_solve(V (&A)[M], V (&r)[3], int a) {
  using T = decltype(A[0].x);
  V dinv = bcast<V>(T(1));
  auto from = [&](V v, int k) {
    const T s = k % 2 ? v.y : v.x;
    return LPN == 1 ? s : __shfl_sync(0xffffffffu, s, k / 2, LPN);
  };
#pragma unroll
  for (int k = 0; k < M; ++k) {
    const T inv = T(1) / from(A[k], k);
    V l = vmul(A[k], bcast<V>(-inv));
    if (a == k / 2) {
      if (k % 2) { dinv.y = inv; l.y = T(0); } else { dinv.x = inv; l.x = T(0); }
    }
#pragma unroll
    for (int b = k + 1; b < M; ++b) A[b] = vfma(l, bcast<V>(from(A[b], k)), A[b]);
#pragma unroll
    for (int c = 0; c < 3; ++c) r[c] = vfma(l, bcast<V>(from(r[c], k)), r[c]);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) r[c] = vmul(r[c], dinv);
}

// Node closure, species pair a of node nd (thermo_state, omega1_of, sm_solve
// and the relaxation times, a lane per species pair).  Species past M hold
// zeros and identity rows.
template <int M, class Real>
__device__ __forceinline__ void split_closure(const DevParams<Real>& p, Real* sm, int nd, int a, bool active,
                                              unsigned* __restrict__ err) {
  using C = Split<M>;
  using V = typename Pair<Real>::T;
  constexpr int LPN = C::LPN, LD = C::LD;
  const V* tab = reinterpret_cast<const V*>(sm + C::TAB) + a;
  auto cst = [&](int k) { return tab[k * LPN]; };
  const V* mom = reinterpret_cast<const V*>(sm + C::MOM) + a * LD + nd;
  V* sp = reinterpret_cast<V*>(sm + C::SP) + a * LD + nd;
  Real* node = sm + C::ND + nd;
  const V zero = bcast<V>(Real(0));
  const bool on0 = 2 * a < M, on1 = 2 * a + 1 < M;
  V rd = zero, ja[3] = {zero, zero, zero};
  if (on0) {
    rd = mom[0];
#pragma unroll
    for (int c = 0; c < 3; ++c) ja[c] = mom[(c + 1) * LPN * LD];
  }
  const Real rho_dev = node[SN_RHOD * 32], rhoE_dev = node[SN_RHOED * 32];
  Real j[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) j[c] = node[(SN_J + c) * 32];
  const Real rho = p.RL[M] + rho_dev, inv_rho = Real(1) / rho;
  const Real u[3] = {j[0] * inv_rho, j[1] * inv_rho, j[2] * inv_rho};
  Real usp[3], rho_sp, sp_dev;
  if (!p.weak) {
    // Eqs. (rhoMATCH), (uMATCH): the slaved species takes the deficits
    const bool s0 = 2 * a == p.slaved, s1 = 2 * a + 1 == p.slaved;
    auto match = [&](V& v, Real total) {
      if (s0) v.x = Real(0);
      if (s1) v.y = Real(0);
      const Real d = total - species_sum<LPN>(v);
      if (s0) v.x = d;
      if (s1) v.y = d;
    };
    match(rd, p.cS + rho_dev);
#pragma unroll
    for (int c = 0; c < 3; ++c) { match(ja[c], j[c]); usp[c] = u[c]; }
    rho_sp = rho;
    sp_dev = p.cS + rho_dev;
  } else {
    sp_dev = species_sum<LPN>(rd);
    rho_sp = p.Rsp + sp_dev;
    const Real is = Real(1) / rho_sp;
#pragma unroll
    for (int c = 0; c < 3; ++c) usp[c] = species_sum<LPN>(ja[c]) * is;
  }
  const V ra = vadd(cst(ST_RL), rd);
  const V inv_sp = bcast<V>(Real(1) / rho_sp);
  const V Y = vmul(ra, inv_sp);
  const V dY = vmul(vfma(cst(ST_YR), bcast<V>(-sp_dev), rd), inv_sp);
  const V im = cst(ST_IM), cv = cst(ST_CV), cp = cst(ST_CP);
  const Real inv_m = species_sum<LPN>(vmul(Y, im)), d_inv_m = species_sum<LPN>(vmul(dY, im));
  const Real Cv = species_sum<LPN>(vmul(Y, cv)), dCv = species_sum<LPN>(vmul(dY, cv));
  const Real Cp = species_sum<LPN>(vmul(Y, cp));
  const Real m = Real(1) / inv_m, R = p.R_U * inv_m, dR = p.R_U * d_inv_m;
  const Real usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  // Eq. (temperature2), T0 = 0
  const Real dT = (p.cE + rhoE_dev - Real(0.5) * rho * usq - rho_dev * p.Cvr * p.Tr - rho * dCv * p.Tr) / (rho * Cv);
  const Real T = p.Tr + dT, theta = R * T, dth = dR * T + p.Rr * dT, P = rho * theta;
  if (a == 0 && active && (!(rho > Real(0)) || !(T > Real(0)) || !(rho_sp > Real(0)))) atomicOr(err, 1u);
  Real Yb[M];
#pragma unroll
  for (int b = 0; b < M; ++b) {
    const Real y = b % 2 ? Y.y : Y.x;
    Yb[b] = LPN == 1 ? y : __shfl_sync(0xffffffffu, y, b / 2, LPN);
  }
  const V X = vmul(bcast<V>(m), vmul(Y, im));
  Real om, om1;
  if (p.omega_is_fixed) {
    om = p.omega_fixed;
  } else {
    // Wilke, Eqs. (viscosityMixture), (wilkePhi); phi = phi_ab / m_b
    const V* phi = tab + 8 * LPN;
    V den = zero;
#pragma unroll
    for (int b = 0; b < M; ++b) den = vfma(phi[b * LPN], bcast<V>(Yb[b]), den);
    const V num = vmul(cst(ST_MU), X);
    V q;
    q.x = on0 ? num.x / (m * den.x) : Real(0);
    q.y = on1 ? num.y / (m * den.y) : Real(0);
    om = Real(2) * P / (P + Real(2) * species_sum<LPN>(q));
  }
  if (p.omega1_is_fixed) {
    om1 = p.omega1_fixed;
  } else {
    const Real s1 = species_sum<LPN>(vmul(X, cst(ST_LAM))), s2 = species_sum<LPN>(vmul(X, cst(ST_ILAM)));
    const Real lam = Real(0.5) * (s1 + Real(1) / s2), pc = P * Cp;
    om1 = Real(2) * pc / (pc + Real(2) * lam);
  }
  // Eqs. (tauab), (tau), (transform12): rows of the system for J_a = rho_a V_a
  const V* cab = tab + (8 + M) * LPN;
  const Real tm = p.R_U * T * m;
  V A[M], r[3], diag = bcast<V>(Real(1)), it = zero;
  const V hY = vmul(bcast<V>(Real(-0.5)), Y);
#pragma unroll
  for (int b = 0; b < M; ++b) {
    const V itab = vmul(bcast<V>(tm), cab[b * LPN]);
    const V f = vmul(itab, bcast<V>(Yb[b]));
    it = vadd(it, f);
    V h = vmul(bcast<V>(Real(0.5)), f);
    if (a == b / 2) { if (b % 2) h.y = Real(0); else h.x = Real(0); }
    diag = vadd(diag, h);
    A[b] = vmul(hY, itab);
  }
#pragma unroll
  for (int b = 0; b < M; ++b)
    if (a == b / 2) { if (b % 2) A[b].y = diag.y; else A[b].x = diag.x; }
#pragma unroll
  for (int c = 0; c < 3; ++c) r[c] = vfma(ra, bcast<V>(-usp[c]), ja[c]);
  if constexpr (sizeof(Real) == 4) {
    // ill-conditioned systems are solved in FP64 (see sm_solve)
    Real cond = Real(2) * (fmax(diag.x, diag.y) - Real(1));
#pragma unroll
    for (int o = LPN / 2; o > 0; o >>= 1) cond = fmax(cond, __shfl_xor_sync(0xffffffffu, cond, o, LPN));
    const bool ill = cond + Real(1) > p.cond_bound;
    if (__any_sync(0xffffffffu, ill)) {
      const double tm64 = (double)p.R_U * (double)T * (double)m;
      double2 A64[M], r64[3], d64 = make_double2(1.0, 1.0);
#pragma unroll
      for (int b = 0; b < M; ++b) {
        const double hx = on0 ? 0.5 * tm64 * p.Cab64[on0 ? 2 * a : 0][b] : 0.0;
        const double hy = on1 ? 0.5 * tm64 * p.Cab64[on1 ? 2 * a + 1 : 0][b] : 0.0;
        if (2 * a != b) d64.x += hx * (double)Yb[b];
        if (2 * a + 1 != b) d64.y += hy * (double)Yb[b];
        A64[b] = make_double2(-hx * (double)Y.x, -hy * (double)Y.y);
      }
#pragma unroll
      for (int b = 0; b < M; ++b)
        if (a == b / 2) { if (b % 2) A64[b].y = d64.y; else A64[b].x = d64.x; }
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        r64[c] = make_double2((double)ja[c].x - (double)ra.x * (double)usp[c], (double)ja[c].y - (double)ra.y * (double)usp[c]);
        const double sr = species_sum<LPN>(r64[c]);
        r64[c].x -= (double)Y.x * sr;
        r64[c].y -= (double)Y.y * sr;
      }
      lanes_solve<M, LPN>(A64, r64, a);
      lanes_solve<M, LPN>(A, r, a);
      if (ill) {
#pragma unroll
        for (int c = 0; c < 3; ++c) { r[c].x = (Real)r64[c].x; r[c].y = (Real)r64[c].y; }
      }
    } else {
      lanes_solve<M, LPN>(A, r, a);
    }
  } else {
    lanes_solve<M, LPN>(A, r, a);
  }
  V ir;
  ir.x = (on0 && ra.x > p.rho_eps * rho_sp) ? Real(1) / ra.x : Real(0);
  ir.y = (on1 && ra.y > p.rho_eps * rho_sp) ? Real(1) / ra.y : Real(0);
  V beta;                                          // dt / (2 tau_a + dt)
  beta.x = it.x / (Real(2) + it.x);
  beta.y = it.y / (Real(2) + it.y);
  sp[SS_RA * LPN * LD] = ra;
  sp[SS_RD * LPN * LD] = rd;
  sp[SS_BETA * LPN * LD] = beta;
  sp[SS_TY * LPN * LD] = vmul(bcast<V>(tm), Y);
  const V cr = vmul(cp, ra);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const V v = vmul(r[c], ir);
    sp[(SS_V + c) * LPN * LD] = v;
    const Real h = species_sum<LPN>(vmul(cr, v));  // sum_a (H_a / T) rho_a V_a
    if (a == 0) node[(SN_HYV + c) * 32] = h;
  }
  if (a == 0) {
    node[SN_DT * 32] = dT; node[SN_DTH * 32] = dth;
    node[SN_OM * 32] = om; node[SN_OM1 * 32] = om1; node[SN_CP * 32] = Cp;
#pragma unroll
    for (int c = 0; c < 3; ++c) node[(SN_USP + c) * 32] = usp[c];
    node[SN_RHOSP * 32] = rho_sp;
  }
}

// Where the host takes this kernel (constant heats, exact closure), by the
// 32-node tiles per SM of the grid.  Measured (GB300, 152 SMs), collide here
// against a thread per node:
//   * From four species in FP64 and with 16-bit storage, and from seven in FP32,
//     always.  There a thread per node needs 255 registers and a stage of 690 to
//     1080 bytes, which leaves 4 to 8 warps on an SM.  FP64 48^3: M = 4 0.89
//     against 2.06 ms, 5 1.60 / 2.78, 6 1.63 / 3.37, 7 1.89 / 4.86; BF16 96^3
//     (thread per node before it formed the senders' terms by rows): M = 4 0.55 /
//     1.02 ms, 5 0.72 / 1.10, 6 0.76 / 1.29, 7 0.92 / 1.69; 192^3 M = 8 7.5 /
//     15.7.  FP32 128^3: M = 7 2.00 / 2.67 ms, M = 8 2.05 / 3.16; 48^3 M = 7 0.115 /
//     0.136; ragged rows and walls by more.
//   * FP32, four to six species.  The fewer the species, the less a thread per
//     node suffers, and on large grids its time per node falls (bulk row loads,
//     no last wave) where the split's stays.  M = 4: 16,384 nodes 15.9 / 19.2 us,
//     32,768 24.5 / 23.8, 49,152 33.1 / 38.9, 65,536 42.4 / 39.5, 80,400 in the
//     opposed-jets frame 57.0 / 57.6, 110,592 63.5 / 59.3, 262,144 169 / 143, 96^3
//     554 / 428, 128^3 1290 / 1035.  M = 5: 8192 nodes 14.6 / 22.0 us, 16,384 23.0 /
//     22.1, 32,768 33.2 / 26.8, 49,152 42.4 / 45.2, 147,456 129 / 100, 96^3 724 / 490.
//     M = 6, rows of whole 128-node blocks: 262,144 nodes 217 / 229 us, 524,288
//     431 / 431, 128^3 1705 / 1535; other rows 96^3 722 / 745, 127 x 129 x 130 1694 /
//     1775.  With walls the thread per node loses its bulk loads and reads the
//     wall per population: M = 4 65,536 nodes 40.1 / 45.3, 96^3 504 / 512; M = 5 65,536
//     51.4 / 52.4, 147,456 124 / 120, 96^3 676 / 613; M = 6 96^3 692 / 795, 128^3 1628 /
//     1824.
//   * With two or three species on grids of few tiles, where the time is one
//     node's latency.  The crossings lie where a second wave of tiles begins:
//     three species FP32 1024 nodes 12.1 / 14.8 us, 14,336 14.5 / 15.2, 19,008 15.0 /
//     16.5, 20,064 21.9 / 16.4; FP64 three species 1024 nodes 59 / 121 us, 4608 60 /
//     114, 8448 82 / 114, 10,560 134 / 126; two species 1024 nodes 52 / 97 us, 4608
//     52 / 97, 8448 63 / 97, 10,560 109 / 97.  The lines taken are 14,592 nodes (FP32)
//     and 4864 (FP64), the measured side of each.  FP32 with two species not:
//     1024 nodes 12.0 / 10.3.
//     Not with 16-bit storage (three species BF16 1024 nodes 14.2 / 22.4 us): a step
//     whose network is rejected at every node runs a thread per node, and at
//     M <= 3 it is held to the exact step within 1e-6 over steps, less than a
//     changed rounding moves a stored value.  From four species the two agree to
//     one unit of the stored part (after a step, 1e-7 to 5e-7 of the largest
//     population at M = 4, 5, 8).
// The tiles are those of the whole grid where the handle holds a slab of it
// (LaunchCtx::grid_nodes): the two collides differ in rounding, and a slab
// agrees with the undivided grid bit for bit.
template <int M, class Real, class Store>
constexpr bool kSplit = M >= 4 || (sizeof(Store) >= 4 && (M == 3 || (M == 2 && sizeof(Real) == 8)));
// The largest number of tiles per SM taken.  walls: bounce-back walls normal to
// x; segments: rows of whole blocks of the thread-per-node collide (bulk loads).
constexpr int kAnyTiles = 1 << 30;
template <int M, class Real, class Store>
constexpr int split_tiles_per_sm(bool walls, bool segments) {
  if (M <= 3) return sizeof(Real) == 8 ? 1 : 3;
  if (sizeof(Store) != 4 || M >= 7) return kAnyTiles;
  if (M == 4) return walls ? kAnyTiles : 12;
  if (M == 5) return walls ? 14 : 3;
  return segments && !walls ? 108 : kAnyTiles;
}
template <int M, class Real, class Store>
constexpr bool kSplitAlways = kSplit<M, Real, Store> && split_tiles_per_sm<M, Real, Store>(false, true) == kAnyTiles;
template <int M, class Real, class Store>
constexpr bool kSplitWallsAlways = kSplit<M, Real, Store> && split_tiles_per_sm<M, Real, Store>(true, false) == kAnyTiles;

// Blocks per SM asked of the register allocator.
#ifndef LBM_SPLIT_THREADS
#define LBM_SPLIT_THREADS 576
#endif
template <int M, class Real>
constexpr int split_min_blocks() {
  constexpr long long bytes = (long long)Split<M>::REALS * sizeof(Real) + 1024;
  constexpr int fit = (int)(227LL * 1024 / bytes);
  constexpr int want = sizeof(Real) == 8 ? 1 : LBM_SPLIT_THREADS / Split<M>::THREADS;
  return want < 1 ? 1 : (want < fit ? want : (fit < 1 ? 1 : fit));
}

// Constants by species pair (a lane-indexed read of the parameter block would
// be serialised).
template <int M, class Real>
__device__ __forceinline__ void split_constants(const DevParams<Real>& p, Real* sm) {
  using C = Split<M>;
  constexpr int NP = C::NP, LPN = C::LPN;
  const int tid = threadIdx.x;
  Real* t = sm + C::TAB;
  for (int k = tid; k < 2 * LPN; k += C::THREADS) {
    const bool on = k < M;
    const int a = on ? k : 0;
    t[ST_RL * 2 * LPN + k] = on ? p.RL[a] : Real(0);
    t[ST_YR * 2 * LPN + k] = on ? p.Yr[a] : Real(0);
    t[ST_IM * 2 * LPN + k] = on ? p.inv_mass[a] : Real(0);
    t[ST_CV * 2 * LPN + k] = on ? p.Cv_a[a] : Real(0);
    t[ST_CP * 2 * LPN + k] = on ? p.Cp_a[a] : Real(0);
    t[ST_MU * 2 * LPN + k] = on ? p.mu[a] : Real(0);
    t[ST_LAM * 2 * LPN + k] = on ? p.lam[a] : Real(0);
    t[ST_ILAM * 2 * LPN + k] = on ? p.inv_lam[a] : Real(0);
  }
  t += 16 * LPN;
  for (int k = tid; k < M * 2 * LPN; k += C::THREADS) {
    const int b = k / (2 * LPN), a = k % (2 * LPN);
    t[k] = a < M ? p.phi[a][b] * p.inv_mass[b] : Real(0);
    t[2 * LPN * M + k] = a < M ? p.Cab[a][b] : Real(0);
  }
  for (int k = tid; k < 2 * M * NP; k += C::THREADS) {
    const int a = k / (2 * NP), b = k % (2 * NP);
    sm[C::TABC + k] = b < M ? p.Cab[a][b] : Real(0);
  }
}

// One tile of 32 nodes.  All threads of the block take part; it ends on a
// barrier, and reads the constants only behind its first.
// BND: 0 periodic, 1 bounce-back walls normal to x, 2 opposed-jets frame.
template <int M, class Real, class Store, int PAR, int BND>
__device__ __forceinline__ void split_tile(const DevParams<Real>& p, Store* __restrict__ pops, Real* __restrict__ side,
                                           unsigned* __restrict__ err, const PlaneOffsets& po, Real* const sm, int tile) {
  using C = Split<M>;
  using V = typename Pair<Real>::T;
  constexpr int NP = C::NP, LPN = C::LPN, LD = C::LD;
  constexpr bool EQ = kEqCodec<Store, Real>, WALL = BND == 1;
  const int tid = threadIdx.x, lane = tid & 31, role = tid >> 5;
  V* const stage = reinterpret_cast<V*>(sm + C::STAGE) + lane;
  Real* const fg = sm + C::FG + lane;
  V* const dif = reinterpret_cast<V*>(sm + C::DIF) + lane;
  Real* const node = sm + C::ND + lane;
  const long long N = p.N;
  const long long n_raw = (long long)tile * 32 + lane;
  bool active = n_raw < N;
  const long long n = active ? n_raw : N - 1;
  if constexpr (BND == 2) {
    const long long x = n % p.nx, y = (n / p.nx) % p.ny;
    if (x == 0 || x == p.nx - 1 || y == 0 || y == p.ny - 1) active = false;
  }
  const unsigned act = __ballot_sync(0xffffffffu, active);
  const Nbr nb = make_nbr(p, n);
  // Lattice 0's slot `slot` at node `nn`; lattice L is po.off[L * Q] further.
  auto slot_at = [&](int slot, long long nn) { return reinterpret_cast<char*>(pops + nn) + po.off[slot]; };
  auto lat = [&](char* q, int L) { return reinterpret_cast<Store*>(q + po.off[L * Q]); };

  // ---- 1. load -------------------------------------------------------------
  // 16-bit storage: rows shared out over the warps.  A row is the three
  // velocities of one (c_y, c_z), in two parts: 0 its species but, from
  // five, the last pair, 1 the rest.  What a population lacks is formed at
  // its sender's x and handed to the neighbouring lane (lbm_eqcodec.cuh);
  // needL / needR: the lane's sender at x - 1 / x + 1 is in no lane of the warp.
  auto ysel = [&](const Nbr& b, int cy) { return cy == 0 ? b.ys[1] : (cy > 0 ? b.ys[0] : b.ys[2]); };   // of y - c_y
  auto zsel = [&](const Nbr& b, int cz) { return cz == 0 ? b.zs[1] : (cz > 0 ? b.zs[0] : b.zs[2]); };
  const bool needL = EQ && active && (lane == 0 || nb.xs[1] == 0);
  const bool needR = EQ && active && (lane == 31 || (int)nb.xs[1] == p.nx - 1);
  if constexpr (EQ) {
    const float* const rin = eq_rec_buf(side, N, p.rec_w, 1 - PAR);
    const unsigned long long need = (unsigned long long)__ballot_sync(0xffffffffu, needL) |
                                    ((unsigned long long)__ballot_sync(0xffffffffu, needR) << 32);
    const int cnt = 9 * __popcll(need);
#pragma unroll 1
    for (int e = tid; e < cnt; e += C::THREADS) {
      unsigned long long rest = need;
      for (int k = e / 9; k > 0; --k) rest &= rest - 1;
      const int who = __ffsll((long long)rest) - 1, row = e % 9;
      const int cx = who < 32 ? 1 : -1, cy = row % 3 - 1, cz = row / 3 - 1, k = who & 31;
      const long long nk = (long long)tile * 32 + k;
      const Nbr nbk = make_nbr(p, nk);
      const bool refl = WALL && arrives_from_wall_c(nbk, cx);
      const long long snd = refl ? nk : (long long)(zsel(nbk, cz) + ysel(nbk, cy) + (cx > 0 ? nbk.xs[0] : nbk.xs[2]));
      const RowLoad<M> in(p, side, rin, snd, cy, cz);
      float2 v[NP];
      float fv, gv;
      edge_terms<M>(p, in, refl, cx, cy, cz, v, fv, gv);
      const int i = (cx + 1) + 3 * row;
#pragma unroll
      for (int q = 0; q < NP; ++q) stage[i * NP * 32 + q * 32 + k - lane] = v[q];
      fg[2 * i * 32 + k - lane] = fv;
      fg[(2 * i + 1) * 32 + k - lane] = gv;
    }
    __syncthreads();
  }
  if constexpr (EQ) {
    // Warps take the two parts in turn: WARPS may be even.
    const float* const rin = eq_rec_buf(side, N, p.rec_w, 1 - PAR);
#pragma unroll 1
    for (int it = role, turn = 0; it < 18; it += C::WARPS, turn ^= 1) {
      const int pair = it >> 1, part = C::WARPS % 2 == 0 ? (it & 1) ^ turn : it & 1;
      const int row = pair, cy = row % 3 - 1, cz = row / 3 - 1, i0 = 3 * row;
      const unsigned rb = ysel(nb, cy) + zsel(nb, cz);
      const long long own = (long long)(rb + nb.xs[1]);                 // the sender at this x
      char* src[3];
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        const bool here = PAR == 0 || (WALL && arrives_from_wall_c(nb, x - 1));        // aa_read_loc
        src[x] = slot_at(here ? i0 + x : Q - 1 - i0 - x, here ? n : (long long)(rb + nb.xs[2 - x]));
      }
      const float4* rec = reinterpret_cast<const float4*>(rin) + own;
      // pairs [q0, q0 + K) of the row
      auto species = [&](auto Q0_, auto K_, const float4& A) {
        constexpr int q0 = decltype(Q0_)::value, K = decltype(K_)::value;
        Store raw[K][3][2];
        float2 d[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const int q = q0 + k;
          d[k] = reinterpret_cast<const float2*>(rec + (2 + q / 2) * N)[q % 2];
#pragma unroll
          for (int x = 0; x < 3; ++x) {
            raw[k][x][0] = *lat(src[x], 2 * q);
            if (2 * q + 1 < M) raw[k][x][1] = *lat(src[x], 2 * q + 1);
          }
        }
        const float4 w = p.weak ? rec[(2 + (1 + M + 3) / 4) * N] : A;
        const RowSpecies r(w.x, w.y, w.z, add1(p.Tr, A.w), cy, cz);
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const int q = q0 + k;
          float2 t[3];
          row_species(p, r, 2 * q, 2 * q + 1 < M ? 2 * q + 1 : 2 * q, d[k], t);
          t[2].x = __shfl_up_sync(0xffffffffu, t[2].x, 1);
          t[2].y = __shfl_up_sync(0xffffffffu, t[2].y, 1);
          t[0].x = __shfl_down_sync(0xffffffffu, t[0].x, 1);
          t[0].y = __shfl_down_sync(0xffffffffu, t[0].y, 1);
          if (needL) t[2] = stage[((i0 + 2) * NP + q) * 32];
          if (needR) t[0] = stage[(i0 * NP + q) * 32];
#pragma unroll
          for (int x = 0; x < 3; ++x) {
            float2 v;
            v.x = codec_decode<Store, float>(p, raw[k][x][0], 2 * q) + t[x].x;
            v.y = 2 * q + 1 < M ? codec_decode<Store, float>(p, raw[k][x][1], 2 * q + 1) + t[x].y : 0.0f;
            stage[((i0 + x) * NP + q) * 32] = v;
          }
        }
      };
      constexpr int Q1 = NP >= 3 ? NP - 1 : NP;          // pairs of part 0
      using Zero = std::integral_constant<int, 0>;
      using First = std::integral_constant<int, Q1>;
      using Last = std::integral_constant<int, NP - Q1>;
      const float4 A = *rec;
      if (part == 0) {
        species(Zero{}, First{}, A);
      } else {
        Store raw[3][2];
#pragma unroll
        for (int x = 0; x < 3; ++x) { raw[x][0] = *lat(src[x], M); raw[x][1] = *lat(src[x], M + 1); }
        const float4 B = rec[N];
        const float hq = reinterpret_cast<const float*>(rec + (2 + M / 4) * N)[M % 4];
        const RowSide<false> sd(side, N, own, cy, cz);
        if constexpr (Last::value > 0) species(First{}, Last{}, A);
        float f[3], g[3];
        row_fg<false>(p, M, A, B, hq, sd.k, sd.x, cy, cz, f, g, nullptr, nullptr);
        f[2] = __shfl_up_sync(0xffffffffu, f[2], 1);
        g[2] = __shfl_up_sync(0xffffffffu, g[2], 1);
        f[0] = __shfl_down_sync(0xffffffffu, f[0], 1);
        g[0] = __shfl_down_sync(0xffffffffu, g[0], 1);
        if (needL) { f[2] = fg[2 * (i0 + 2) * 32]; g[2] = fg[(2 * (i0 + 2) + 1) * 32]; }
        if (needR) { f[0] = fg[2 * i0 * 32]; g[0] = fg[(2 * i0 + 1) * 32]; }
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          fg[2 * (i0 + x) * 32] = codec_decode<Store, float>(p, raw[x][0], M) + f[x];
          fg[(2 * (i0 + x) + 1) * 32] = codec_decode<Store, float>(p, raw[x][1], M + 1) + g[x];
        }
      }
    }
  } else {
    // FP64 and FP32: the velocities in turn.  (Asynchronous copies of the whole
    // tile into the stage with the deferred terms formed by rows meanwhile
    // measured slower: eight species 128^3 FP32 2.07 against 1.95 ms.)
#pragma unroll 1
    for (int i = role; i < Q; i += C::WARPS) {
      const int cz = i / 9 - 1, cy = (i / 3) % 3 - 1, cx = i % 3 - 1;
      const bool refl = WALL && arrives_from_wall_c(nb, cx);
      const unsigned xs = cx == 0 ? nb.xs[1] : (cx > 0 ? nb.xs[0] : nb.xs[2]);
      const long long snd = refl ? n : (long long)(xs + ysel(nb, cy) + zsel(nb, cz));   // n - c_i, or n itself at a wall
      const bool own = PAR == 0 || refl;                                                // aa_read_loc
      char* const q = slot_at(own ? i : Q - 1 - i, own ? n : snd);
      Real v[M + 2];
#pragma unroll
      for (int L = 0; L < M + 2; ++L) v[L] = *lat(q, L);
      if (i != 13) {
        // the deferred terms (incoming_corr_th)
        const Real th = side[SP_THR * N + snd];
        Real kc = Real(0);
        if (cx) { const Real k = side[(SP_K + 0) * N + snd]; kc += cx > 0 ? k : -k; }
        if (cy) { const Real k = side[(SP_K + 1) * N + snd]; kc += cy > 0 ? k : -k; }
        if (cz) { const Real k = side[(SP_K + 2) * N + snd]; kc += cz > 0 ? k : -k; }
        const Real w0 = Real(1) - th, w1 = Real(0.5) * th;
        const Real cg = (cx ? w1 : w0) * (cy ? w1 : w0) * (cz ? w1 : w0) * kc;
        v[M + 1] += refl ? -cg : cg;
        if (cx * cx + cy * cy + cz * cz == 1) {
          const Real X = side[(SP_X + (cx ? 0 : (cy ? 1 : 2))) * N + snd];
          const Real cf = (cx + cy + cz > 0 ? Real(0.5) : Real(-0.5)) * X;
          v[M] += refl ? -cf : cf;
        }
      }
#pragma unroll
      for (int a = 0; a < M; a += 2) {
        V d;
        d.x = v[a];
        d.y = a + 1 < M ? v[a + 1] : Real(0);
        stage[(i * NP + a / 2) * 32] = d;
      }
      fg[2 * i * 32] = v[M];
      fg[(2 * i + 1) * 32] = v[M + 1];
    }
  }
  __syncthreads();

  // ---- 2. moments, each warp its own lattices' ---------------------------
  Real q3[3] = {Real(0), Real(0), Real(0)};     // g: energy flux
  if (role < NP) {
    V r4[4];
    static_for<0, Q>([&](auto I_) {
      constexpr int i = decltype(I_)::value;
      const V v = stage[(i * NP + role) * 32];
      r4[0] = i == 0 ? v : vadd(r4[0], v);
      static_for<0, 3>([&](auto A_) {
        constexpr int c = c_of(i, decltype(A_)::value);
        V& t = r4[1 + decltype(A_)::value];
        if constexpr (i == 0) t = vsub(bcast<V>(Real(0)), v);         // c = (-1, -1, -1)
        else if constexpr (c > 0) t = vadd(t, v);
        else if constexpr (c < 0) t = vsub(t, v);
      });
    });
    V* mom = reinterpret_cast<V*>(sm + C::MOM) + role * LD + lane;
#pragma unroll
    for (int c = 0; c < 4; ++c) mom[c * LPN * LD] = r4[c];
  } else if (role == NP) {
    Real rho_dev = Real(0), j[3] = {Real(0), Real(0), Real(0)}, S[6] = {Real(0), Real(0), Real(0), Real(0), Real(0), Real(0)};
    static_for<0, Q>([&](auto I_) {
      constexpr int i = decltype(I_)::value;
      constexpr int cx = cx_of(i), cy = cy_of(i), cz = cz_of(i);
      const Real v = fg[2 * i * 32];
      rho_dev += v;
      if (cx) { j[0] += cx * v; S[0] += v; }
      if (cy) { j[1] += cy * v; S[1] += v; }
      if (cz) { j[2] += cz * v; S[2] += v; }
      if (cx && cy) S[3] += (cx * cy) * v;
      if (cx && cz) S[4] += (cx * cz) * v;
      if (cy && cz) S[5] += (cy * cz) * v;
    });
    node[SN_RHOD * 32] = rho_dev;
#pragma unroll
    for (int c = 0; c < 3; ++c) node[(SN_J + c) * 32] = j[c];
#pragma unroll
    for (int c = 0; c < 6; ++c) node[(SN_S + c) * 32] = S[c];
  } else {
    Real rhoE_dev = Real(0);
    static_for<0, Q>([&](auto I_) {
      constexpr int i = decltype(I_)::value;
      const Real v = fg[(2 * i + 1) * 32];
      rhoE_dev += v;
      if (cx_of(i)) q3[0] += cx_of(i) * v;
      if (cy_of(i)) q3[1] += cy_of(i) * v;
      if (cz_of(i)) q3[2] += cz_of(i) * v;
    });
    node[SN_RHOED * 32] = rhoE_dev;
  }
  __syncthreads();

  // ---- 3. node closure -----------------------------------------------------
  if (role < LPN) split_closure<M, Real>(p, sm, tid / LPN, tid % LPN, (act >> (tid / LPN)) & 1u, err);
  __syncthreads();

  // ---- 4. update, store --------------------------------------------------
  const Nbr nbw = opaque(nb);
  const long long nw = opaque_idx(n);
  const Real dT = node[SN_DT * 32];
  if (role < NP) {
    const int a0 = 2 * role;
    const bool two = M % 2 == 0 || role < NP - 1;
    const V* sp = reinterpret_cast<const V*>(sm + C::SP) + lane;
    auto pick = [&](int k) { return sp[(k * LPN + role) * LD]; };
    V z, dz;                                        // R_a T and R_a (T - T_r)
    z.x = p.R_a[a0]; z.y = p.R_a[a0 + (two ? 1 : 0)];
    RestDeviation<V> e;
    const V half = bcast<V>(Real(0.5));
    e.r2 = vmul(z, bcast<V>(Real(0.5) * p.Tr));
    dz = vmul(z, bcast<V>(dT));
    z = vmul(z, bcast<V>(p.Tr + dT));
    V b1[3], b2[3], f1[3], f2[3];                   // halved moments of u + V; differences Psi(u) - Psi(u + V)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const Real x = node[(SN_USP + c) * 32];
      const V Vc = pick(SS_V + c);
      const V x2 = bcast<V>(x * x);
      e.h1[c] = bcast<V>(Real(0.5) * x);
      e.h2[c] = vmul(half, vadd(x2, z));
      e.d2[c] = vmul(half, vadd(x2, dz));
      f1[c] = vmul(bcast<V>(Real(-0.5)), Vc);
      f2[c] = vmul(f1[c], vadd(bcast<V>(x + x), Vc));
      b1[c] = vsub(e.h1[c], f1[c]);
      b2[c] = vsub(e.h2[c], f2[c]);
    }
    // Force moments of each species (density apart): a_p a_q a_r - b_p b_q b_r
    // with f = a - b, telescoped: f_p a_q a_r + b_p (f_q a_r + b_q f_r).
    V own[NP > 1 ? 1 : 26];
    auto fsel = [&](auto P_, int ax) { return decltype(P_)::value == 1 ? f1[ax] : f2[ax]; };
    auto bsel = [&](auto P_, int ax) { return decltype(P_)::value == 1 ? b1[ax] : b2[ax]; };
    static_for<0, 9>([&](auto K_) {
      constexpr int qy = decltype(K_)::value % 3, r = decltype(K_)::value / 3;
      using QC = std::integral_constant<int, qy>;
      using RC = std::integral_constant<int, r>;
      V E;
      if constexpr (qy == 0 && r == 0) E = bcast<V>(Real(0));
      else if constexpr (qy == 0) E = fsel(RC{}, 2);
      else if constexpr (r == 0) E = fsel(QC{}, 1);
      else E = vfma(fsel(QC{}, 1), e.template a<r>(2), vmul(bsel(QC{}, 1), fsel(RC{}, 2)));
      static_for<0, 3>([&](auto P_) {
        constexpr int pp = decltype(P_)::value, t = pp + 3 * qy + 9 * r - 1;
        if constexpr (t >= 0) {
          V D;
          if constexpr (pp == 0) D = E;
          else if constexpr (qy == 0 && r == 0) D = fsel(P_, 0);
          else D = vfma(fsel(P_, 0), e.template ayz<qy, r>(), vmul(bsel(P_, 0), E));
          if constexpr (NP > 1) dif[(t * NP + role) * 32] = D;
          else own[t] = D;
        }
      });
    });
    // weights of the force moments: (beta_a - 1) (Y_a / tau_ab) rho_b, species b in pairs
    const V beta = pick(SS_BETA), tY = pick(SS_TY), ra = pick(SS_RA), rd = pick(SS_RD);
    const V bm = vsub(beta, bcast<V>(Real(1))), w = vmul(bm, tY);
    const V cv = vsub(bcast<V>(Real(1)), vadd(beta, beta));       // 1 - 2 beta
    const V ce = EQ ? vsub(bcast<V>(Real(0)), cv) : vadd(beta, beta);
    V k0[NP], k1[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      const V* cab = reinterpret_cast<const V*>(sm + C::TABC) + a0 * NP + q;
      const V rb = sp[(SS_RA * LPN + q) * LD];
      k0[q] = vmul(vmul(bcast<V>(w.x), cab[0]), rb);
      k1[q] = two ? vmul(vmul(bcast<V>(w.y), cab[NP]), rb) : bcast<V>(Real(0));
    }
    if constexpr (NP > 1) asm volatile("bar.sync 1, %0;" ::"n"(NP * 32) : "memory");
    const V cra = vmul(ce, ra), crd = vmul(ce, rd);
    V rest_w[4];                                     // crd times the rest moments
    rest_w[0] = crd;
#pragma unroll
    for (int k = 1; k < 4; ++k) rest_w[k] = vmul(rest_w[k - 1], e.r2);
    auto plane = [&](auto R_, V (&mm)[9]) {
      constexpr int r = decltype(R_)::value;
      static_for<0, 9>([&](auto K_) {
        constexpr int k = decltype(K_)::value, pp = k % 3, qy = k / 3, t = pp + 3 * qy + 9 * r - 1;
        constexpr int rp = RestDeviation<V>::template rest_power<pp, qy, r>();
        V s;
        if constexpr (t < 0) {
          s = crd;
        } else {
          if constexpr (rp >= 0) s = vfma(cra, e.template e<pp, qy, r>(), rest_w[rp]);
          else s = vmul(cra, e.template e<pp, qy, r>());
          V s0 = bcast<V>(Real(0)), s1 = s0;
#pragma unroll
          for (int q = 0; q < NP; ++q) {
            V D;
            if constexpr (NP > 1) D = dif[(t * NP + q) * 32]; else D = own[t];
            s0 = q == 0 ? vmul(k0[q], D) : vfma(k0[q], D, s0);
            s1 = q == 0 ? vmul(k1[q], D) : vfma(k1[q], D, s1);
          }
          s.x += s0.x + s0.y;
          s.y += s1.x + s1.y;
        }
        mm[k] = s;
      });
    };
    char* const first = reinterpret_cast<char*>(pops) + (long long)a0 * po.off[Q];
    auto put = [&](auto I_, V val) {
      constexpr int i = decltype(I_)::value;
      long long nn; int slot;
      aa_write_loc<WALL>(PAR, nbw, nw, i, nn, slot);
      char* const q = first + (nn * (long long)sizeof(Store) + po.off[slot]);
      const V out = vfma(cv, stage[(i * NP + role) * 32], val);
      if (active) {
        codec_store<Store, Real>(p, reinterpret_cast<Store*>(q), 0, a0, out.x);
        if (two) codec_store<Store, Real>(p, lat(q, 1), 0, a0 + 1, out.y);
      }
    };
    from_moments<Real, V>(crd, plane, put, [&](V val) { put(std::integral_constant<int, 13>{}, val); });
  } else {
    const Real rho_dev = node[SN_RHOD * 32], dth = node[SN_DTH * 32], om = node[SN_OM * 32], om1 = node[SN_OM1 * 32];
    const Real rho = p.RL[M] + rho_dev, inv_rho = Real(1) / rho, theta = p.thr + dth, T = p.Tr + dT;
    const Real j[3] = {node[SN_J * 32], node[(SN_J + 1) * 32], node[(SN_J + 2) * 32]};
    const Real u[3] = {j[0] * inv_rho, j[1] * inv_rho, j[2] * inv_rho};
    const Real P = rho * theta, Cp = node[SN_CP * 32];
    const Real usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    if (role == NP) {
      if (active) {
        // side fields (Eqs. Xalpha, corrFourier; see collide_node)
        const Real a3 = Real(1) - Real(3) * theta;
#pragma unroll
        for (int c = 0; c < 3; ++c) side[(SP_PHI + c) * N + n] = j[c] * a3 - rho * u[c] * u[c] * u[c];
        side[SP_COM * N + n] = Real(1) / om - Real(0.5);
        side[SP_CP * N + n] = Cp;
        side[SP_S * N + n] = Real(0.5) * (Real(2) - om1) * P * T / theta;
        side[SP_TH * N + n] = theta;
      }
      // momentum lattice, Eqs. (feq), (fwithcorrection)
      RestDeviation<Real> e;
      e.r2 = Real(0.5) * p.thr;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const Real x2 = u[c] * u[c];
        e.h1[c] = Real(0.5) * u[c];
        e.h2[c] = Real(0.5) * (x2 + theta);
        e.d2[c] = Real(0.5) * (x2 + dth);
      }
      const Real cv = Real(1) - om, ce = EQ ? -cv : om;
      const Real cra = ce * rho, crd = ce * rho_dev;
      const Real rest_w[4] = {crd, crd * e.r2, crd * e.r2 * e.r2, crd * e.r2 * e.r2 * e.r2};
      auto plane = [&](auto R_, Real (&mm)[9]) {
        constexpr int r = decltype(R_)::value;
        static_for<0, 9>([&](auto K_) {
          constexpr int k = decltype(K_)::value, pp = k % 3, qy = k / 3;
          constexpr int rp = RestDeviation<Real>::template rest_power<pp, qy, r>();
          if constexpr (pp + qy + r == 0) mm[k] = crd;
          else if constexpr (rp >= 0) mm[k] = cra * e.template e<pp, qy, r>() + rest_w[rp];
          else mm[k] = cra * e.template e<pp, qy, r>();
        });
      };
      auto put = [&](auto I_, Real val) {
        constexpr int i = decltype(I_)::value;
        long long nn; int slot;
        aa_write_loc<WALL>(PAR, nbw, nw, i, nn, slot);
        if (active) codec_store<Store, Real>(p, lat(slot_at(slot, nn), M), 0, M, cv * fg[2 * i * 32] + val);
      };
      from_moments<Real, Real>(crd, plane, put, [&](Real val) { put(std::integral_constant<int, 13>{}, val); });
    } else {
      // energy lattice (see collide_node for the closed form)
      const Real rhoE_dev = node[SN_RHOED * 32];
      const Real dP = rho_dev * theta + p.RL[M] * dth;
      const Real hk = Cp * T + Real(0.5) * usq, inv_theta = Real(1) / theta;
      const Real Gc = rho * (hk + theta) * Real(0.5) * inv_theta;
      const Real dE0 = rhoE_dev - Real(1.5) * dP - Gc * usq;
      Real dZ[3], mvec[3], qt[3];
      {
        const Real z1 = Real(1) - Real(3) * theta;
        const Real zb = Real(0.5) * (z1 * dP - Real(3) * dth * p.Pr);
#pragma unroll
        for (int c = 0; c < 3; ++c) dZ[c] = zb + z1 * Gc * u[c] * u[c];
        Real S[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) S[c] = node[(SN_S + c) * 32];
        Real dP6[6];                                       // Pi - P^eq
#pragma unroll
        for (int c = 0; c < 3; ++c) dP6[c] = p.cPi + S[c] - dP - rho * u[c] * u[c];
        dP6[3] = S[3] - rho * u[0] * u[1];
        dP6[4] = S[4] - rho * u[0] * u[2];
        dP6[5] = S[5] - rho * u[1] * u[2];
        const Real qb[3] = {q3[0] - (u[0] * dP6[0] + u[1] * dP6[3] + u[2] * dP6[4]),
                            q3[1] - (u[0] * dP6[3] + u[1] * dP6[1] + u[2] * dP6[5]),
                            q3[2] - (u[0] * dP6[4] + u[1] * dP6[5] + u[2] * dP6[2])};
        const Real rY = p.weak ? rho / node[SN_RHOSP * 32] : Real(1);
        const Real c1 = om1 * T * rY, dw = om - om1;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const Real qeq = hk * j[c];
          qt[c] = qeq * inv_theta;
          mvec[c] = (om * qeq + dw * (qb[c] - qeq) + c1 * node[(SN_HYV + c) * 32]) * inv_theta;
        }
      }
      if constexpr (EQ) {
        if (active) {
          EqRec<M> r;
#pragma unroll
          for (int c = 0; c < 3; ++c) { r.u[c] = u[c]; r.usp[c] = node[(SN_USP + c) * 32]; }
          r.dth = dth; r.dT = dT; r.drho = rho_dev; r.dE0 = dE0;
          r.Gq = Gc * inv_theta; r.hq = hk * rho * inv_theta;
#pragma unroll
          for (int a = 0; a < M; ++a) {
            const V d = reinterpret_cast<const V*>(sm + C::SP)[(SS_RD * LPN + a / 2) * LD + lane];
            r.ra[a] = a % 2 ? d.y : d.x;
          }
          store_rec<M>(eq_rec_buf(side, N, p.rec_w, PAR), N, n, p.weak, r);
        }
      }
      const Real w0 = Real(1) - theta, w1 = Real(0.5) * theta;          // Eq. (w0)
      const Real r0 = Real(1) - p.thr, r1 = Real(0.5) * p.thr;
      const Real d0 = -dth, d1 = Real(0.5) * dth;
      Real s_g = Real(0);
      static_for<0, 13>([&](auto I_) {
        constexpr int i = decltype(I_)::value, o = Q - 1 - i;
        constexpr int cx = cx_of(i), cy = cy_of(i), cz = cz_of(i);
        long long node_i, node_o; int slot_i, slot_o;
        aa_write_loc<WALL>(PAR, nbw, nw, i, node_i, slot_i);
        aa_write_loc<WALL>(PAR, nbw, nw, o, node_o, slot_o);
        const Real uc = dotc<Real, i>(u);
        const Real cc = Real(0.5) * Real(c2_of(i));
        const Real ucu = Gc * uc * uc * inv_theta;
        const Real dEi = dE0 + cc * rho_dev + ucu;
        const Real wx = cx ? w1 : w0, wy = cy ? w1 : w0, wz = cz ? w1 : w0;
        const Real rx = cx ? r1 : r0, ry = cy ? r1 : r0;
        const Real dx = cx ? d1 : d0, dy = cy ? d1 : d0, dzz = cz ? d1 : d0;
        const Real wi = wx * wy * wz;
        const Real dwi = dx * wy * wz + rx * dy * wz + rx * ry * dzz;
        const Real eg = wi * dEi + dwi * energy_rest(p, M, c2_of(i)) + BdotZ<Real, i>(dZ);
        s_g += eg + eg;
        const Real fl = wi * dotc<Real, i>(mvec);
        const Real gi = fg[(2 * i + 1) * 32], go = fg[(2 * o + 1) * 32];
        const Real out_i = gi + om * (eg - gi) + fl;
        const Real out_o = go + om * (eg - go) - fl;
        if (active) {
          const Real sq = EQ ? wi * dotc<Real, i>(qt) : Real(0);
          codec_store<Store, Real>(p, lat(slot_at(slot_i, node_i), M + 1), 0, M + 1, EQ ? out_i - (eg + sq) : out_i);
          codec_store<Store, Real>(p, lat(slot_at(slot_o, node_o), M + 1), 0, M + 1, EQ ? out_o - (eg - sq) : out_o);
        }
      });
      long long nn; int slot;
      aa_write_loc<WALL>(PAR, nbw, nw, 13, nn, slot);
      const Real e13 = rhoE_dev - s_g;
      const Real gr = fg[(2 * 13 + 1) * 32];
      const Real out = gr + om * (e13 - gr);
      if (active) codec_store<Store, Real>(p, lat(slot_at(slot, nn), M + 1), 0, M + 1, EQ ? out - e13 : out);
    }
  }
  __syncthreads();      // the next tile's moments take the place of this tile's
}

template <int M, class Real, class Store, int PAR, int BND>
__global__ void __launch_bounds__(Split<M>::THREADS, split_min_blocks<M, Real>())
collide_split_kernel(const __grid_constant__ DevParams<Real> p, Store* __restrict__ pops, Real* __restrict__ side,
                     unsigned* __restrict__ err, int ntiles, const __grid_constant__ PlaneOffsets po) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  Real* const sm = reinterpret_cast<Real*>(smem_raw);
  split_constants<M, Real>(p, sm);
  wait_previous();
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x)
    split_tile<M, Real, Store, PAR, BND>(p, pops, side, err, po, sm, tile);
}

}  // namespace lbm
