// lbm_stencil.cuh -- the deferred non-local terms of the step, the two stencil
// passes that build them, and the readers of the state (observables,
// checkpoint copies) that apply them.
//
// The D3Q27 correction A_i . X (Eq. fwithcorrection) and the grad C_p part of
// q^corr (Eq. corrFourier) enter the post-collision populations additively,
// but they need the neighbours' time-t moments, which a node does not have
// when it collides.  Each collision therefore writes its populations without
// them, and the node that receives a population at the next step adds the
// sender's term before using it:
//   f_i += 1/2 c_i . X(x)             (the six face directions)
//   g_i += w_i(theta_x) c_i . K(x),   K = (1/2)(2 - omega_1) P T grad C_p / theta
// with x = y - c_i the sender.  X and K are built between steps by the two
// stencil passes below from side fields each collision writes, so every
// population is exact (synchronous in time t) when it is used.
#pragma once

#include "lbm_helpers.cuh"
#include "lbm_eqcodec.cuh"

namespace lbm {

// Four consecutive values (16-byte aligned for FP32, 32-byte for FP64).
template <class Real>
__device__ __forceinline__ void load4(const Real* __restrict__ f, Real* v) {
  if constexpr (sizeof(Real) == 4) {
    const float4 q = *reinterpret_cast<const float4*>(f);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    const double2 a = *reinterpret_cast<const double2*>(f);
    const double2 b = *reinterpret_cast<const double2*>(f + 2);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
  }
}
template <class Real>
__device__ __forceinline__ void store4(Real* __restrict__ f, const Real* v) {
  if constexpr (sizeof(Real) == 4) {
    *reinterpret_cast<float4*>(f) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    *reinterpret_cast<double2*>(f) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2*>(f + 2) = make_double2(v[2], v[3]);
  }
}

// The deferred terms of the population that `sender` sent in direction I,
// for a sender whose theta is th.
template <class Real, int I, bool NC>
__device__ __forceinline__ void incoming_corr_th(const Real* __restrict__ side, long long N, long long sender,
                                                 Real th, Real& cf, Real& cg) {
  constexpr int cx = cx_of(I), cy = cy_of(I), cz = cz_of(I);
  Real kc = Real(0);
  if constexpr (cx != 0) kc += (cx > 0 ? ld<NC>(side + (SP_K + 0) * N + sender) : -ld<NC>(side + (SP_K + 0) * N + sender));
  if constexpr (cy != 0) kc += (cy > 0 ? ld<NC>(side + (SP_K + 1) * N + sender) : -ld<NC>(side + (SP_K + 1) * N + sender));
  if constexpr (cz != 0) kc += (cz > 0 ? ld<NC>(side + (SP_K + 2) * N + sender) : -ld<NC>(side + (SP_K + 2) * N + sender));
  const Real w0 = Real(1) - th, w1 = Real(0.5) * th;
  const Real w = (cx ? w1 : w0) * (cy ? w1 : w0) * (cz ? w1 : w0);   // Eq. (weights)
  cg = w * kc;
  cf = Real(0);
  if constexpr (c2_of(I) == 1) {
    constexpr int a = cx ? 0 : (cy ? 1 : 2);
    constexpr int sg = cx + cy + cz;
    cf = (sg > 0 ? Real(0.5) : Real(-0.5)) * ld<NC>(side + (SP_X + a) * N + sender);
  }
}
template <class Real, int I, bool NC = false>
__device__ __forceinline__ void incoming_corr(const Real* __restrict__ side, long long N, long long sender,
                                              Real& cf, Real& cg) {
  incoming_corr_th<Real, I, NC>(side, N, sender, ld<NC>(side + SP_THR * N + sender), cf, cg);
}

// Reduced-precision storage: the record of the node that sent the population
// arriving at n in direction I, the equilibrium shifts of every lattice for
// that population (lbm_eqcodec.cuh) and its deferred terms.  The sender is
// n - c_I; with walls, a population arriving from beyond a wall is n's own
// population of direction opp(I) reflected, so it was stored with n's shift
// for opp(I) and carries n's terms for I negated.  For the readers of the state
// and its initialisation.
template <int M, int I, bool WALL>
__device__ __forceinline__ void eq_incoming(const DevParams<float>& p, const float* __restrict__ side,
                                            const Nbr& nb, long long n, int parity, float& cf, float& cg,
                                            float (&sh)[M + 2]) {
  const long long N = p.N;
  const float* rin = eq_rec_buf(side, N, p.rec_w, 1 - parity);
  bool refl = false;
  long long snd = n;
  if constexpr (I != 13) {
    if (WALL && arrives_from_wall(nb, I)) refl = true;
    else snd = nb.idx(-cx_of(I), -cy_of(I), -cz_of(I));
  }
  const EqRec<M> r = load_rec<M>(rin, N, snd, p.weak);
  if (WALL && refl) eq_shift<M, opp_of(I)>(p, r, sh);
  else eq_shift<M, I>(p, r, sh);
  cf = 0.0f; cg = 0.0f;
  if constexpr (I != 13) {
    incoming_corr_th<float, I, true>(side, N, snd, p.thr + r.dth, cf, cg);
    if (WALL && refl) { cf = -cf; cg = -cg; }
  }
}

// The deferred terms of the population arriving in direction I at node n.
// With walls (WALL), one arriving from beyond a wall is the node's own
// population of direction opp(I) reflected, so its terms are the node's own
// for opp(I): those of I at the node, negated (w_opp(I) = w_I, c_opp(I) = -c_I).
template <class Real, int I, bool WALL, bool NC = false>
__device__ __forceinline__ void deferred_terms(const Real* __restrict__ side, long long N, const Nbr& nb,
                                               long long n, Real& cf, Real& cg) {
  if constexpr (WALL) {
    if (arrives_from_wall(nb, I)) {
      incoming_corr<Real, I, NC>(side, N, n, cf, cg);
      cf = -cf;
      cg = -cg;
      return;
    }
  }
  incoming_corr<Real, I, NC>(side, N, nb.idx(-cx_of(I), -cy_of(I), -cz_of(I)), cf, cg);
}

// The decoding terms of the population arriving at n in direction I for the
// readers of the state: the deferred non-local terms cf (f) and cg (g), and
// with 16-bit storage the equilibrium shifts sh of every lattice (zero
// otherwise); walls are handled whether or not the grid has them.
template <int M, class Real, class Store, int I>
__device__ __forceinline__ void incoming_terms(const DevParams<Real>& p, const Real* __restrict__ side,
                                               const Nbr& nb, long long n, int parity, Real& cf, Real& cg,
                                               Real (&sh)[M + 2]) {
  cf = Real(0); cg = Real(0);
  if constexpr (kEqCodec<Store, Real>) {
    eq_incoming<M, I, true>(p, side, nb, n, parity, cf, cg, sh);
  } else {
#pragma unroll
    for (int L = 0; L < M + 2; ++L) sh[L] = Real(0);
    if constexpr (I != 13) deferred_terms<Real, I, true, true>(side, p.N, nb, n, cf, cg);
  }
}

// 16-bit storage, for the readers of the state: every population arriving at
// node n, a (c_y, c_z) row at a time, as f(i, cx, cy, cz, slot, node, sh, cf, cg)
// with the AA place it is stored in and what it lacks: the shifts sh of every
// lattice and the deferred terms of f and g, added to sh or (SEP) apart in cf
// and cg.  As in the collide, a row's terms are
// formed once at the lane's x and exchanged between lanes; a lane whose sender
// is in no lane of the warp forms it itself.  All lanes of a warp call it;
// those past the grid with active = false and the last node.  Measured (GB300):
// observables of the 192^3 eight-species BF16 state 4.4 against 9.3 ms with
// every population's terms formed from its own gathered record, restart copies
// of 96^3 FP16 0.86 against 0.92 ms, two-species 256^3 BF16 4.2 ms either way.
template <int M, class Store, bool SEP, class F>
__device__ __forceinline__ void row_populations(const DevParams<float>& p, const float* __restrict__ side, int parity,
                                                const Nbr& nb, long long n, bool active, F&& f) {
  constexpr int NP = (M + 1) / 2;
  const float* const rin = eq_rec_buf(side, p.N, p.rec_w, 1 - parity);
  const int lane = threadIdx.x & 31;
  const bool needL = active && (lane == 0 || nb.xs[1] == 0);
  const bool needR = active && (lane == 31 || (int)nb.xs[1] == p.nx - 1);
#pragma unroll 1
  for (int row = 0; row < 9; ++row) {
    const int cy = row % 3 - 1, cz = row / 3 - 1;
    const unsigned rb = (cy == 0 ? nb.ys[1] : (cy > 0 ? nb.ys[0] : nb.ys[2])) +
                        (cz == 0 ? nb.zs[1] : (cz > 0 ? nb.zs[0] : nb.zs[2]));
    RowTerms<M, SEP> t;
    row_terms<M>(p, RowLoad<M, true>(p, side, rin, (long long)(rb + nb.xs[1]), cy, cz), cy, cz, t);
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      t.sp[q][2].x = __shfl_up_sync(0xffffffffu, t.sp[q][2].x, 1);
      t.sp[q][0].x = __shfl_down_sync(0xffffffffu, t.sp[q][0].x, 1);
      if (2 * q + 1 < M) {
        t.sp[q][2].y = __shfl_up_sync(0xffffffffu, t.sp[q][2].y, 1);
        t.sp[q][0].y = __shfl_down_sync(0xffffffffu, t.sp[q][0].y, 1);
      }
    }
    t.f[2] = __shfl_up_sync(0xffffffffu, t.f[2], 1);
    t.g[2] = __shfl_up_sync(0xffffffffu, t.g[2], 1);
    t.f[0] = __shfl_down_sync(0xffffffffu, t.f[0], 1);
    t.g[0] = __shfl_down_sync(0xffffffffu, t.g[0], 1);
    if constexpr (SEP) {
      t.cf[2] = __shfl_up_sync(0xffffffffu, t.cf[2], 1);
      t.cg[2] = __shfl_up_sync(0xffffffffu, t.cg[2], 1);
      t.cf[0] = __shfl_down_sync(0xffffffffu, t.cf[0], 1);
      t.cg[0] = __shfl_down_sync(0xffffffffu, t.cg[0], 1);
    }
    // the lane's first need, then (rows of one node) a second
    for (int k = 0; k < 2; ++k) {
      if (k == 0 ? !(needL || needR) : !(needL && needR)) continue;
      const int cx = k == 0 && needL ? 1 : -1;
      const bool refl = arrives_from_wall_c(nb, cx);
      float2 sp[NP];
      float fv, gv, cfv, cgv;
      edge_terms<M, true, SEP>(p, RowLoad<M, true>(p, side, rin, refl ? n : (long long)(rb + (cx > 0 ? nb.xs[0] : nb.xs[2])), cy, cz), refl,
                    cx, cy, cz, sp, fv, gv, &cfv, &cgv);
#pragma unroll
      for (int q = 0; q < NP; ++q) { if (cx > 0) t.sp[q][2] = sp[q]; else t.sp[q][0] = sp[q]; }
      if (cx > 0) { t.f[2] = fv; t.g[2] = gv; } else { t.f[0] = fv; t.g[0] = gv; }
      if constexpr (SEP) {
        if (cx > 0) { t.cf[2] = cfv; t.cg[2] = cgv; } else { t.cf[0] = cfv; t.cg[0] = cgv; }
      }
    }
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const int i = 3 * row + x;
      const bool own = parity == 0 || arrives_from_wall_c(nb, x - 1);          // aa_read_loc
      float sh[M + 2];
#pragma unroll
      for (int a = 0; a < M; ++a) sh[a] = a % 2 ? t.sp[a / 2][x].y : t.sp[a / 2][x].x;
      sh[M] = t.f[x];
      sh[M + 1] = t.g[x];
      f(i, x - 1, cy, cz, own ? i : Q - 1 - i, own ? n : (long long)(rb + nb.xs[2 - x]), sh,
        SEP ? t.cf[SEP ? x : 0] : 0.0f, SEP ? t.cg[SEP ? x : 0] : 0.0f);
    }
  }
}

// Zeroth/first moments of the (corrected) deviations needed by the
// thermodynamic state (Eqs. densitya, auxua, f0momDensity, f1momMomentum,
// g0momTotalEnergy).
template <int M, class Real, class Store>
__device__ __forceinline__ void load_state_moments(const DevParams<Real>& p, const Store* __restrict__ pops,
                                                   const Real* __restrict__ side, int parity, const Nbr& nb,
                                                   long long n, bool active, Real (&rdev)[M], Real (&ja)[M][3],
                                                   Real& rho_dev, Real (&j)[3], Real& rhoE_dev) {
  const long long N = p.N;
#pragma unroll
  for (int a = 0; a < M; ++a) { rdev[a] = Real(0); ja[a][0] = ja[a][1] = ja[a][2] = Real(0); }
  rho_dev = Real(0); j[0] = j[1] = j[2] = Real(0); rhoE_dev = Real(0);
  if constexpr (kEqCodec<Store, Real>) {
    row_populations<M, Store, false>(p, side, parity, nb, n, active,
                                     [&](int, int cx, int cy, int cz, int slot, long long node, const float (&sh)[M + 2],
                                         float, float) {
      const Store* q = pops + ((long long)slot * N + node);
      const float fx = (float)cx, fy = (float)cy, fz = (float)cz;
#pragma unroll
      for (int a = 0; a < M; ++a) {
        const float v = codec_decode<Store, float>(p, q[(long long)a * Q * N], a) + sh[a];
        rdev[a] += v;
        ja[a][0] += fx * v; ja[a][1] += fy * v; ja[a][2] += fz * v;
      }
      const float fv = codec_decode<Store, float>(p, q[(long long)M * Q * N], M) + sh[M];
      rho_dev += fv;
      j[0] += fx * fv; j[1] += fy * fv; j[2] += fz * fv;
      rhoE_dev += codec_decode<Store, float>(p, q[(long long)(M + 1) * Q * N], M + 1) + sh[M + 1];
    });
  } else {
    (void)active;
    static_for<0, Q>([&](auto I_) {
      constexpr int i = decltype(I_)::value;
      constexpr int cx = cx_of(i), cy = cy_of(i), cz = cz_of(i);
      long long node; int slot;
      aa_read_loc<true>(parity, nb, n, i, node, slot);
      Real cf = Real(0), cg = Real(0);
      if constexpr (i != 13) deferred_terms<Real, i, true, true>(side, N, nb, n, cf, cg);
#pragma unroll
      for (int a = 0; a < M; ++a) {
        const Real v = pops[(a * Q + slot) * N + node];
        rdev[a] += v;
        if (cx) ja[a][0] += cx * v;
        if (cy) ja[a][1] += cy * v;
        if (cz) ja[a][2] += cz * v;
      }
      const Real fv = pops[(M * Q + slot) * N + node] + cf;
      rho_dev += fv;
      if (cx) j[0] += cx * fv;
      if (cy) j[1] += cy * fv;
      if (cz) j[2] += cz * fv;
      rhoE_dev += pops[((M + 1) * Q + slot) * N + node] + cg;
    });
  }
}

// Stencil pass 1 (after a collision): G_alpha = c_omega d_alpha Phi_alpha (the
// inner derivative of Eq. Xalpha) and K_alpha = s d_alpha C_p with s = c2 / theta;
// the sender's theta is copied for the receivers' weights.
// With temperature-dependent heats (tvar) the enthalpy field differentiated
// is H-like: Phi_1 + T_n Phi_2 + T_n^2 Phi_3 of the neighbours with this
// node's T_n, so that K = s sum_k T^(k-1) grad Phi_k = (s / T) sum_a H_a grad Y_a.
// The passes exist as four nodes of a row per thread, a node per thread, and a
// thread per node and field.  Which of them a grid takes depends on its number
// of nodes; the sums a node gets do not.  They run over the nine neighbour rows
// (c_y, c_z), c_z outermost, and add a row's three values in one of two forms:
//   ROWS (rows of a multiple of ROWV nodes, constant heats): the D3Q27 weights
//     factor per axis, w_i = w(c_ix) w(c_iy) w(c_iz) with w(0) = 2/3, w(+-1) = 1/6,
//     so the isotropic gradient separates,
//       d_x phi = (1/72) sum_{cy,cz} W(cy) W(cz) [phi(x+1) - phi(x-1)]
//       d_y phi = (1/72) sum_{cz} W(cz) [s(+1, cz) - s(-1, cz)]
//       d_z phi = (1/72) sum_{cy} W(cy) [s(cy, +1) - s(cy, -1)]
//     with W(0) = 4, W(+-1) = 1 and s = phi(x-1) + 4 phi(x) + phi(x+1) on the row
//     (products with powers of two: exact, so the sums round the same whether
//     or not the compiler contracts them; with explicit fused operations the
//     four-node first pass took 140 registers in place of 64 and, at 256^3, 363
//     us in place of 212);
//   else velocity by velocity, grad = 3 sum_i w_i c_i phi(x + c_i), one product
//     to a sum, contracted alike everywhere (written as fused operations, the
//     per-node first pass took 60 registers in place of 42 and, at 45 x 75 x 101,
//     18.6 us in place of 15.0).
// Slabs of a grid and the batched domains thus agree with the undivided grid
// and the single domain bit for bit, whatever passes those take.
#ifndef LBM_STENCIL_ROW
#define LBM_STENCIL_ROW 4
#endif
constexpr int ROWV = LBM_STENCIL_ROW;
static_assert(ROWV == 4 || ROWV == 8, "row blocking of 4 or 8 nodes");

// Adds row (cy, cz), its values lo, mid, hi at x-1, x, x+1, to the sum d of the A-derivative.
template <class Real, int A, bool ROWS>
__device__ __forceinline__ Real row_term(Real lo, Real mid, Real hi, int cy, int cz, Real d) {
  if constexpr (ROWS) {
    const Real Wy = cy ? Real(1) : Real(4), Wz = cz ? Real(1) : Real(4);
    const Real W = A == 0 ? Wy * Wz : (A == 1 ? cy * Wz : cz * Wy);
    const Real s = A == 0 ? hi - lo : lo + Real(4) * mid + hi;
    return d + W * s;
  } else {
    const int i = 3 * (cy + 1) + 9 * (cz + 1);
    const Real w1 = iso_w<Real>(i), w0 = iso_w<Real>(i + 1), c = A == 0 ? Real(1) : (A == 1 ? Real(cy) : Real(cz));
    if constexpr (A == 0) {
      d += -w1 * lo;
    } else {
      d += (c * w1) * lo;
      d += (c * w0) * mid;
    }
    d += (c * w1) * hi;
    return d;
  }
}
// The factors of the sums: G = c_omega grad Phi, K = s grad C_p; X = -div.
template <class Real, bool ROWS>
__device__ __forceinline__ Real scaled_gradient(Real c, Real d) {
  return ROWS ? c * (d * (Real(1) / Real(72))) : Real(3) * c * d;
}
template <class Real, bool ROWS>
__device__ __forceinline__ Real minus_gradient(Real d) {
  return d * (ROWS ? Real(-1) / Real(72) : Real(-3));
}

template <class Real, bool ROWS, class G>
__device__ __forceinline__ void grad_GK_node(const G& p, Real* __restrict__ side, long long n, bool tvar = false) {
  if (n >= p.N) return;
  const long long N = p.N;
  const Nbr nb = make_nbr(p, n);
  Real d[3] = {Real(0), Real(0), Real(0)}, dc[3] = {Real(0), Real(0), Real(0)};
  const Real Tn = tvar ? side[SP_T * N + n] : Real(0);
  if constexpr (ROWS) {
#pragma unroll
    for (int cz = -1; cz <= 1; ++cz)
#pragma unroll
      for (int cy = -1; cy <= 1; ++cy) {
        const long long lo = nb.idx(-1, cy, cz), mid = nb.idx(0, cy, cz), hi = nb.idx(1, cy, cz);
        auto row = [&](int plane, auto A_, bool odd, Real acc) {
          const Real* f = side + plane * N;
          const Real l = f[lo], m = f[mid], h = f[hi];
          return row_term<Real, decltype(A_)::value, true>(odd && (nb.wall & 1u) ? -l : l, m,
                                                           odd && (nb.wall & 2u) ? -h : h, cy, cz, acc);
        };
        using A0 = std::integral_constant<int, 0>;
        using A1 = std::integral_constant<int, 1>;
        using A2 = std::integral_constant<int, 2>;
        d[0] = row(SP_PHI, A0{}, true, d[0]);              // beyond a wall Phi_x is odd, the others even
        if (cy) d[1] = row(SP_PHI + 1, A1{}, false, d[1]);
        if (cz) d[2] = row(SP_PHI + 2, A2{}, false, d[2]);
        dc[0] = row(SP_CP, A0{}, false, dc[0]);
        if (cy) dc[1] = row(SP_CP, A1{}, false, dc[1]);
        if (cz) dc[2] = row(SP_CP, A2{}, false, dc[2]);
      }
  } else {
    // velocity by velocity, all fields of one neighbour at a time (row by row
    // this took 18.5 against 15.0 us at 45 x 75 x 101 FP32)
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int cx = cx_of(i), cy = cy_of(i), cz = cz_of(i);
      if (i == 13) continue;
      const long long nn = nb.idx(cx, cy, cz);
      const Real w = iso_w<Real>(i);
      Real cp = side[SP_CP * N + nn];
      if (tvar) cp += Tn * (side[SP_HC2 * N + nn] + Tn * side[SP_HC3 * N + nn]);
      // beyond a wall the mirror image of Phi_x is odd, the other fields even
      const bool mirror = (cx < 0 && (nb.wall & 1u)) || (cx > 0 && (nb.wall & 2u));
      if (cx) {
        const Real phx = side[(SP_PHI + 0) * N + nn];
        d[0] += (cx * w) * (mirror ? -phx : phx);
        dc[0] += (cx * w) * cp;
      }
      if (cy) { d[1] += (cy * w) * side[(SP_PHI + 1) * N + nn]; dc[1] += (cy * w) * cp; }
      if (cz) { d[2] += (cz * w) * side[(SP_PHI + 2) * N + nn]; dc[2] += (cz * w) * cp; }
    }
  }
  const Real co = side[SP_COM * N + n], sv = side[SP_S * N + n];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    side[(SP_G + c) * N + n] = scaled_gradient<Real, ROWS>(co, d[c]);
    side[(SP_K + c) * N + n] = scaled_gradient<Real, ROWS>(sv, dc[c]);
  }
  side[SP_THR * N + n] = side[SP_TH * N + n];
}

// Stencil pass 2: X_alpha = -d_alpha G_alpha (Eq. Xalpha).
template <class Real, bool ROWS, class G>
__device__ __forceinline__ void grad_X_node(const G& p, Real* __restrict__ side, long long n) {
  if (n >= p.N) return;
  const long long N = p.N;
  const Nbr nb = make_nbr(p, n);
  Real d[3] = {Real(0), Real(0), Real(0)};
  auto g = [&](int c, long long nn) { return side[(SP_G + c) * N + nn]; };
#pragma unroll
  for (int cz = -1; cz <= 1; ++cz)
#pragma unroll
    for (int cy = -1; cy <= 1; ++cy) {
      const long long lo = nb.idx(-1, cy, cz), mid = nb.idx(0, cy, cz), hi = nb.idx(1, cy, cz);
      d[0] = row_term<Real, 0, ROWS>(g(0, lo), Real(0), g(0, hi), cy, cz, d[0]);
      if (cy) d[1] = row_term<Real, 1, ROWS>(g(1, lo), g(1, mid), g(1, hi), cy, cz, d[1]);
      if (cz) d[2] = row_term<Real, 2, ROWS>(g(2, lo), g(2, mid), g(2, hi), cy, cz, d[2]);
    }
#pragma unroll
  for (int c = 0; c < 3; ++c) side[(SP_X + c) * N + n] = minus_gradient<Real, ROWS>(d[c]);
}

// ---------------------------------------------------------------------------
// Row-blocked stencil passes (grids with nx a multiple of ROWV): one thread
// computes ROWV consecutive nodes of a row.  Each row is read once as ROWV + 2
// values (x0-1 .. x0+ROWV) shared by the thread's nodes: the middle ones as
// 16-byte vector loads, the two ends as scalar loads or (SHFL) from the
// neighbouring lanes, which hold them as their own middle values, except at
// warp and row edges.  Every lane of a warp takes part in the shuffles; lanes
// past the grid compute on the last nodes and store nothing.
// ---------------------------------------------------------------------------
// Row coordinates of the nodes n0 .. n0+ROWV-1 (x0 = n0 mod nx, a multiple of ROWV).
struct RowV {
  unsigned x0, xm, xp;       // first x, its left neighbour, the right neighbour of the last node (periodic)
  unsigned ys[3], zs[3];     // wrapped row offsets for c_y, c_z = -1, 0, +1
  bool from_left, from_right;   // the end values are held by lane - 1 / lane + 1 (same row)
  bool wlo, whi;                // walls: the left / right end value is a mirror image
  __device__ __forceinline__ unsigned row(int cy, int cz) const { return zs[cz + 1] + ys[cy + 1]; }
};
template <class P>
__device__ __forceinline__ RowV make_row(const P& p, unsigned n0) {
  RowV r;
  const unsigned nx = (unsigned)p.nx, ny = (unsigned)p.ny, nz = (unsigned)p.nz;
  r.x0 = n0 % nx;
  const unsigned t = n0 / nx, y = t % ny, z = t / ny, pl = nx * ny;
  const bool w = p.wall_x != 0;
  r.wlo = w && r.x0 == 0;
  r.whi = w && r.x0 + ROWV == nx;
  r.xm = r.x0 == 0 ? (w ? 0 : nx - 1) : r.x0 - 1;
  r.xp = r.x0 + ROWV == nx ? (w ? nx - 1 : 0) : r.x0 + ROWV;
  const unsigned lane = threadIdx.x & 31u;
  r.from_left = lane > 0 && r.x0 != 0;
  r.from_right = lane < 31 && r.x0 + ROWV != nx;
  r.ys[0] = (y == 0 ? ny - 1 : y - 1) * nx;  r.ys[1] = y * nx;  r.ys[2] = (y == ny - 1 ? 0 : y + 1) * nx;
  r.zs[0] = (z == 0 ? nz - 1 : z - 1) * pl;  r.zs[1] = z * pl;  r.zs[2] = (z == nz - 1 ? 0 : z + 1) * pl;
  return r;
}
// ODD: the field is odd under the mirror at a wall (Phi_x).
template <class Real, bool SHFL, bool ODD = false>
__device__ __forceinline__ void load_row(const Real* __restrict__ f, const RowV& r, unsigned rb, Real (&v)[ROWV + 2]) {
  if constexpr (SHFL) {
#pragma unroll
    for (int q = 0; q < ROWV; q += 4) load4<Real>(f + rb + r.x0 + q, v + 1 + q);
    const Real left = __shfl_up_sync(0xffffffffu, v[ROWV], 1);
    const Real right = __shfl_down_sync(0xffffffffu, v[1], 1);
    v[0] = r.from_left ? left : f[rb + r.xm];
    v[ROWV + 1] = r.from_right ? right : f[rb + r.xp];
  } else {
    v[0] = f[rb + r.xm];
#pragma unroll
    for (int q = 0; q < ROWV; q += 4) load4<Real>(f + rb + r.x0 + q, v + 1 + q);
    v[ROWV + 1] = f[rb + r.xp];
  }
  if constexpr (ODD) {
    if (r.wlo) v[0] = -v[0];
    if (r.whi) v[ROWV + 1] = -v[ROWV + 1];
  }
}
// End values by shuffle in the second pass only: in the first (four fields
// per row) the shuffles raised it from 64 to 80 registers and it ran slower,
// also when held to 64 (measured on GB300, 128^3 acoustic pulse).  Without
// shuffles the end loads go first: issued after the vector load the pass
// took 58 registers and ran 9 % slower.
#ifndef LBM_GK_SHFL
#define LBM_GK_SHFL 0
#endif
#ifndef LBM_X_SHFL
#define LBM_X_SHFL 1
#endif
// Adds row (cy, cz) of a field to the a-derivative accumulators d[ROWV] (a = 0, 1, 2).
template <class Real, int A>
__device__ __forceinline__ void row_derivative(const Real (&v)[ROWV + 2], int cy, int cz, Real (&d)[ROWV]) {
#pragma unroll
  for (int j = 0; j < ROWV; ++j) d[j] = row_term<Real, A, true>(v[j], v[j + 1], v[j + 2], cy, cz, d[j]);
}

// Pass 1 on ROWV nodes: G_a = c_omega d_a Phi_a, K = s grad C_p, theta copied.
template <class Real>
__device__ __forceinline__ void grad_GK_row(const DevParams<Real>& p, Real* __restrict__ side, unsigned n0,
                                            bool store) {
  const long long N = p.N;
  const RowV r = make_row(p, n0);
  Real dp[3][ROWV], dc[3][ROWV];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int j = 0; j < ROWV; ++j) dp[a][j] = dc[a][j] = Real(0);
#pragma unroll
  for (int cz = -1; cz <= 1; ++cz)
#pragma unroll
    for (int cy = -1; cy <= 1; ++cy) {
      const unsigned rb = r.row(cy, cz);
      Real v[ROWV + 2];
      load_row<Real, LBM_GK_SHFL, true>(side + (SP_PHI + 0) * N, r, rb, v);
      row_derivative<Real, 0>(v, cy, cz, dp[0]);
      if (cy) { load_row<Real, LBM_GK_SHFL>(side + (SP_PHI + 1) * N, r, rb, v); row_derivative<Real, 1>(v, cy, cz, dp[1]); }
      if (cz) { load_row<Real, LBM_GK_SHFL>(side + (SP_PHI + 2) * N, r, rb, v); row_derivative<Real, 2>(v, cy, cz, dp[2]); }
      load_row<Real, LBM_GK_SHFL>(side + SP_CP * N, r, rb, v);
      row_derivative<Real, 0>(v, cy, cz, dc[0]);
      if (cy) row_derivative<Real, 1>(v, cy, cz, dc[1]);
      if (cz) row_derivative<Real, 2>(v, cy, cz, dc[2]);
    }
  if (!store) return;
  const unsigned own = r.row(0, 0) + r.x0;
#pragma unroll
  for (int q = 0; q < ROWV; q += 4) {
    Real co[4], sv[4], th[4];
    load4<Real>(side + SP_COM * N + own + q, co);
    load4<Real>(side + SP_S * N + own + q, sv);
    load4<Real>(side + SP_TH * N + own + q, th);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Real g[4], k[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        g[j] = scaled_gradient<Real, true>(co[j], dp[a][q + j]);
        k[j] = scaled_gradient<Real, true>(sv[j], dc[a][q + j]);
      }
      store4<Real>(side + (SP_G + a) * N + own + q, g);
      store4<Real>(side + (SP_K + a) * N + own + q, k);
    }
    store4<Real>(side + SP_THR * N + own + q, th);
  }
}

// Pass 2 on ROWV nodes: X_a = -d_a G_a.
template <class Real>
__device__ __forceinline__ void grad_X_row(const DevParams<Real>& p, Real* __restrict__ side, unsigned n0,
                                           bool store) {
  const long long N = p.N;
  const RowV r = make_row(p, n0);
  Real d[3][ROWV];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int j = 0; j < ROWV; ++j) d[a][j] = Real(0);
#pragma unroll
  for (int cz = -1; cz <= 1; ++cz)
#pragma unroll
    for (int cy = -1; cy <= 1; ++cy) {
      const unsigned rb = r.row(cy, cz);
      Real v[ROWV + 2];
      load_row<Real, LBM_X_SHFL>(side + (SP_G + 0) * N, r, rb, v);
      row_derivative<Real, 0>(v, cy, cz, d[0]);
      if (cy) { load_row<Real, LBM_X_SHFL>(side + (SP_G + 1) * N, r, rb, v); row_derivative<Real, 1>(v, cy, cz, d[1]); }
      if (cz) { load_row<Real, LBM_X_SHFL>(side + (SP_G + 2) * N, r, rb, v); row_derivative<Real, 2>(v, cy, cz, d[2]); }
    }
  if (!store) return;
  const unsigned own = r.row(0, 0) + r.x0;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int q = 0; q < ROWV; q += 4) {
      Real x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = minus_gradient<Real, true>(d[a][q + j]);
      store4<Real>(side + (SP_X + a) * N + own + q, x);
    }
}

// Small grids: a thread per node and field, so that few nodes still spread
// over the SMs.  F = 0..2: G_F; 3: K and the copy of theta.
template <class Real, bool ROWS, int F>
__device__ __forceinline__ void grad_GK_field(const DevParams<Real>& p, Real* __restrict__ side, long long n) {
  if (n >= p.N) return;
  const long long N = p.N;
  const Nbr nb = make_nbr(p, n);
  const Real Tn = F == 3 && p.tvar ? side[SP_T * N + n] : Real(0);
  auto value = [&](int cx, int cy, int cz) {
    const long long nn = nb.idx(cx, cy, cz);
    if constexpr (F < 3) {
      const Real v = side[(SP_PHI + F) * N + nn];
      return F == 0 && ((cx < 0 && (nb.wall & 1u)) || (cx > 0 && (nb.wall & 2u))) ? -v : v;   // Phi_x is odd beyond a wall
    } else {
      Real v = side[SP_CP * N + nn];
      if (p.tvar) v += Tn * (side[SP_HC2 * N + nn] + Tn * side[SP_HC3 * N + nn]);
      return v;
    }
  };
  Real d[3] = {Real(0), Real(0), Real(0)};
#pragma unroll
  for (int cz = -1; cz <= 1; ++cz)
#pragma unroll
    for (int cy = -1; cy <= 1; ++cy) {
      if ((F == 1 && cy == 0) || (F == 2 && cz == 0)) continue;
      const Real lo = value(-1, cy, cz), hi = value(1, cy, cz);
      const Real mid = F == 0 || (cy == 0 && cz == 0) ? Real(0) : value(0, cy, cz);
      if (F == 0 || F == 3) d[0] = row_term<Real, 0, ROWS>(lo, mid, hi, cy, cz, d[0]);
      if (F == 1 || (F == 3 && cy)) d[1] = row_term<Real, 1, ROWS>(lo, mid, hi, cy, cz, d[1]);
      if (F == 2 || (F == 3 && cz)) d[2] = row_term<Real, 2, ROWS>(lo, mid, hi, cy, cz, d[2]);
    }
  if constexpr (F < 3) {
    side[(SP_G + F) * N + n] = scaled_gradient<Real, ROWS>(side[SP_COM * N + n], d[F]);
  } else {
    const Real sv = side[SP_S * N + n];
#pragma unroll
    for (int c = 0; c < 3; ++c) side[(SP_K + c) * N + n] = scaled_gradient<Real, ROWS>(sv, d[c]);
    side[SP_THR * N + n] = side[SP_TH * N + n];
  }
}
template <class Real, bool ROWS, int F>
__device__ __forceinline__ void grad_X_field(const DevParams<Real>& p, Real* __restrict__ side, long long n) {
  if (n >= p.N) return;
  const long long N = p.N;
  const Nbr nb = make_nbr(p, n);
  auto g = [&](int cx, int cy, int cz) { return side[(SP_G + F) * N + nb.idx(cx, cy, cz)]; };
  Real d = Real(0);
#pragma unroll
  for (int cz = -1; cz <= 1; ++cz)
#pragma unroll
    for (int cy = -1; cy <= 1; ++cy) {
      if ((F == 1 && cy == 0) || (F == 2 && cz == 0)) continue;
      d = row_term<Real, F, ROWS>(g(-1, cy, cz), F == 0 ? Real(0) : g(0, cy, cz), g(1, cy, cz), cy, cz, d);
    }
  side[(SP_X + F) * N + n] = minus_gradient<Real, ROWS>(d);
}
constexpr int BLOCK_FIELD = 32;
template <class Real, bool ROWS>
__global__ void __launch_bounds__(BLOCK_FIELD)
grad_GK_field_kernel(const __grid_constant__ DevParams<Real> p, Real* __restrict__ side) {
  wait_previous();
  if (blockIdx.y == 0) grad_GK_field<Real, ROWS, 0>(p, side, gtid());
  else if (blockIdx.y == 1) grad_GK_field<Real, ROWS, 1>(p, side, gtid());
  else if (blockIdx.y == 2) grad_GK_field<Real, ROWS, 2>(p, side, gtid());
  else grad_GK_field<Real, ROWS, 3>(p, side, gtid());
}
template <class Real, bool ROWS>
__global__ void __launch_bounds__(BLOCK_FIELD)
grad_X_field_kernel(const __grid_constant__ DevParams<Real> p, Real* __restrict__ side) {
  wait_previous();
  if (blockIdx.y == 0) grad_X_field<Real, ROWS, 0>(p, side, gtid());
  else if (blockIdx.y == 1) grad_X_field<Real, ROWS, 1>(p, side, gtid());
  else grad_X_field<Real, ROWS, 2>(p, side, gtid());
}

// LBM_GK_MINB > 0 sets a minimum of resident blocks per SM (FP32); by
// default the compiler chooses (64 registers, four blocks of 256).
#ifndef LBM_GK_MINB
#define LBM_GK_MINB 0
#endif
template <class Real>
__global__ void
#if LBM_GK_MINB > 0
__launch_bounds__(BLOCK_LIGHT, sizeof(Real) == 4 ? LBM_GK_MINB : 1)
#else
__launch_bounds__(BLOCK_LIGHT)
#endif
grad_GK_row_kernel(const __grid_constant__ DevParams<Real> p, Real* __restrict__ side) {
  wait_previous();
  const long long t = gtid();
  const bool in = ROWV * t < p.N;
  grad_GK_row<Real>(p, side, (unsigned)(in ? ROWV * t : p.N - ROWV), in);
}
template <class Real>
__global__ void __launch_bounds__(BLOCK_LIGHT)
grad_X_row_kernel(const __grid_constant__ DevParams<Real> p, Real* __restrict__ side) {
  wait_previous();
  const long long t = gtid();
  const bool in = ROWV * t < p.N;
  grad_X_row<Real>(p, side, (unsigned)(in ? ROWV * t : p.N - ROWV), in);
}

template <class Real>
__global__ void __launch_bounds__(BLOCK_LIGHT)
grad_GK_kernel(const __grid_constant__ DevParams<Real> p, Real* __restrict__ side) {
  wait_previous();
  grad_GK_node<Real, false>(p, side, gtid(), p.tvar != 0);
}
template <class Real>
__global__ void __launch_bounds__(BLOCK_LIGHT)
grad_X_kernel(const __grid_constant__ DevParams<Real> p, Real* __restrict__ side) {
  wait_previous();
  grad_X_node<Real, false>(p, side, gtid());
}

}  // namespace lbm
