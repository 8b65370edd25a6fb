// lbm_eqcodec.cuh -- reduced-precision (FP16 / BF16) storage of the
// populations as shifted deviations from the local equilibrium.
//
// The stored 16-bit value of a population is s_L (f_i - f^eq_i(y)) with y the
// node that wrote it (the sender, x - c_i for the population arriving at x
// in direction i), f^eq_i(y) that node's equilibrium of lattice L in
// direction i (Eqs. 27eq, feq, gieq: the lattice weights at the node's
// velocity and temperature times its density, and the energy lattice's
// equilibrium from its total energy and enthalpy), and s_L a per-lattice
// scale.  After a collision f' - f^eq is the non-equilibrium part, a small
// fraction of f even where the flow moves fast or the composition varies by
// factors, so the 8 (BF16) or 11 (FP16) significant bits are spent on it.
//
// The receiver needs the sender's equilibrium: every collision writes a
// per-node FP32 record of the quantities its equilibria are built from, and
// the receiver rebuilds f^eq_i(y) from the sender's record.  A record is
// rec_w floats (a multiple of 4), held as rec_w / 4 planes of one float4 per
// node, in two buffers after the side planes: the step of AA parity q reads
// buffer 1 - q (written by the previous step) and writes buffer q.  A warp
// gathers 32 neighbouring nodes' records: as planes each float4 load is one
// contiguous 512-byte row, four cache lines, where node-major records of 48
// bytes spread it over twelve (GB300, BF16: 256^3 two-species layers collide
// 6.01 against 6.64 ms, ternary ensemble step 3.44 against 3.72 ms).
//
// Record slots (floats), as deviations from the reference rest state where
// the quantity has one (T_r, theta_r, RL of each lattice):
//   [0..3]     u_x, u_y, u_z, dT                  mixture velocity, T - T_r
//   [4..7]     dtheta, drho, dE0, Gq              theta - theta_r, rho - RL_f, E_0 less its rest value, Gq = Gc / theta
//   [8..8+M)   drho_1 .. drho_M                   coupled species densities - RL_a
//   [8+M]      hq = (H + u^2/2) rho / theta       first-moment factor of g^eq (then padding to 4)
//   [..+3]     u_sp (weak coupling only)          velocity of the species subsystem
// with Gc = rho (h + theta) / (2 theta), h = H + u^2/2, E_0 = rho E - 3P/2 - Gc u^2.  The momentum and
// energy shifts are formed as deviations without cancellation (the same
// telescoped forms as the collision's equilibria), so the receiver recovers
// the populations to FP32 rounding of their deviations.
#pragma once

#include "lbm_helpers.cuh"

namespace lbm {

template <class Store, class Real>
constexpr bool kEqCodec = (sizeof(Store) == 2) && sizeof(Real) == 4;

__host__ __device__ constexpr int eq_rec_width(int M, int weak) {
  return 8 + ((1 + M + 3) / 4) * 4 + (weak ? 4 : 0);
}

// Offset (in floats) of the record buffers inside the side/scratch buffer:
// after the NSIDE planes, rounded up to 256 bytes.
__host__ __device__ constexpr long long eq_rec_offset(long long N) {
  return ((long long)NSIDE * N + 63) / 64 * 64;
}

__device__ __forceinline__ float* eq_rec_buf(float* side, long long N, int rw, int buf) {
  return side + eq_rec_offset(N) + (long long)buf * rw * N;
}
__device__ __forceinline__ const float* eq_rec_buf(const float* side, long long N, int rw, int buf) {
  return side + eq_rec_offset(N) + (long long)buf * rw * N;
}

template <int M>
struct EqRec {
  float u[3], dth, dT, drho, dE0, Gq, hq;
  float ra[M];      // species densities minus RL_a
  float usp[3];
};

// buf: a record buffer of N nodes (eq_rec_buf).  For the readers of the state.
template <int M>
__device__ __forceinline__ EqRec<M> load_rec(const float* __restrict__ buf, long long N, long long node, int weak) {
  const float4* q = reinterpret_cast<const float4*>(buf) + node;
  EqRec<M> r;
  const float4 a = ld<true>(q), b = ld<true>(q + N);
  r.u[0] = a.x; r.u[1] = a.y; r.u[2] = a.z; r.dT = a.w;
  r.dth = b.x; r.drho = b.y; r.dE0 = b.z; r.Gq = b.w;
  constexpr int NT = (1 + M + 3) / 4;
  float t[4 * NT];
#pragma unroll
  for (int k = 0; k < NT; ++k) {
    const float4 c = ld<true>(q + (2 + k) * N);
    t[4 * k] = c.x; t[4 * k + 1] = c.y; t[4 * k + 2] = c.z; t[4 * k + 3] = c.w;
  }
#pragma unroll
  for (int s = 0; s < M; ++s) r.ra[s] = t[s];
  r.hq = t[M];
  if (weak) {
    const float4 d = ld<true>(q + (2 + NT) * N);
    r.usp[0] = d.x; r.usp[1] = d.y; r.usp[2] = d.z;
  } else {
    r.usp[0] = r.u[0]; r.usp[1] = r.u[1]; r.usp[2] = r.u[2];
  }
  return r;
}

template <int M>
__device__ __forceinline__ void store_rec(float* __restrict__ buf, long long N, long long node, int weak,
                                          const EqRec<M>& r) {
  float4* q = reinterpret_cast<float4*>(buf) + node;
  q[0] = make_float4(r.u[0], r.u[1], r.u[2], r.dT);
  q[N] = make_float4(r.dth, r.drho, r.dE0, r.Gq);
  constexpr int NT = (1 + M + 3) / 4;
  float t[4 * NT];
#pragma unroll
  for (int k = 0; k < 4 * NT; ++k) t[k] = 0.0f;
#pragma unroll
  for (int s = 0; s < M; ++s) t[s] = r.ra[s];
  t[M] = r.hq;
#pragma unroll
  for (int k = 0; k < NT; ++k) q[(2 + k) * N] = make_float4(t[4 * k], t[4 * k + 1], t[4 * k + 2], t[4 * k + 3]);
  if (weak) q[(2 + NT) * N] = make_float4(r.usp[0], r.usp[1], r.usp[2], 0.0f);
}

// The shifts of direction I of every lattice, as deviations from the
// reference rest state (the arithmetic works on d = f - b_ref):
//   sh_L = f^eq_{L,I}(record) - b_ref_{L,I}.
// Species (Eq. 27eq) as rho_a Psi_I(u_sp, R_a T) - b_ref; momentum (Eq. feq)
// and energy (Eqs. gansatz, gieq) lattices in the telescoped deviation forms
// of the collision (lbm_collide.cuh), which carry no O(f) cancellation.
// f (lattice M): rho (Psi_I(u, theta) - W_I(theta_r)) + (rho - RL_f) W_I(theta_r)
template <int I>
__device__ __forceinline__ float eq_shift_f(const DevParams<float>& p, int M, const float (&u)[3], float dth,
                                            float drho) {
  const float x2[3] = {u[0] * u[0], u[1] * u[1], u[2] * u[2]};
  return (p.RL[M] + drho) * pf_diff<float, I>(u, x2, p.thr, dth) + drho * pf_ref<float, I>(p.thr);
}
// g (lattice M + 1): w_I(theta) [E_I + q^eq . c_I / theta] + B_I . Z relative
// to its rest value.  E_I less its rest value, dE_I = dE_0 + (drho/2) |c|^2 +
// Gq (u . c)^2, and E_I itself differ by a constant of the velocity's length
// (energy_rest), so the bracket's deviation is w_I dE_I + (w_I - W_I) (E_I - dE_I).
template <class Real>
__device__ __forceinline__ Real energy_rest(const DevParams<Real>& p, int M, int k2) {
  return fma1(Real(0.5) * Real(k2), p.RL[M], fma1(Real(-1.5) * p.RL[M], p.thr, p.RL[M + 1]));
}
template <int I>
__device__ __forceinline__ float eq_shift_g(const DevParams<float>& p, int M, const float (&u)[3], float dth,
                                            float drho, float dE0, float Gq, float hq) {
  constexpr int k2 = c2_of(I);
  constexpr int cx = cx_of(I), cy = cy_of(I), cz = cz_of(I);
  const float theta = p.thr + dth;
  const float uc = dotc<float, I>(u);
  const float dEi = dE0 + 0.5f * (float)k2 * drho + Gq * uc * uc;
  const float w0 = 1.0f - theta, w1 = 0.5f * theta;
  const float r0 = 1.0f - p.thr, r1 = 0.5f * p.thr;
  const float d0 = -dth, d1 = 0.5f * dth;
  const float wx = cx ? w1 : w0, wy = cy ? w1 : w0, wz = cz ? w1 : w0;
  const float rx = cx ? r1 : r0, ry = cy ? r1 : r0;
  const float ddx = cx ? d1 : d0, ddy = cy ? d1 : d0, ddz = cz ? d1 : d0;
  const float wyz = wy * wz;
  const float dwi = ddx * wyz + rx * (ddy * wz + ry * ddz);
  float sh = wx * wyz * (dEi + hq * uc) + dwi * energy_rest(p, M, k2);
  if constexpr (k2 <= 1) {
    const float z1 = 1.0f - 3.0f * theta;
    const float zb = 0.5f * (z1 * (drho * theta + p.RL[M] * dth) - 3.0f * dth * p.Pr);
    const float zG = z1 * Gq * theta;
    if constexpr (k2 == 0) {
      sh += 3.0f * zb + zG * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    } else {
      constexpr int ax = cx ? 0 : (cy ? 1 : 2);
      sh -= 0.5f * (zb + zG * u[ax] * u[ax]);
    }
  }
  return sh;
}
// Species (Eq. 27eq): per axis Psi_c = b + k z with (b, k) = (1 - x^2, -1) or
// ((x^2 +- x) / 2, 1/2), two species at a time in the lanes of paired FP32
// instructions.
template <int M, int I>
__device__ __forceinline__ void eq_shift(const DevParams<float>& p, const EqRec<M>& r, float (&sh)[M + 2]) {
  constexpr int k2 = c2_of(I);
  constexpr int cs[3] = {cx_of(I), cy_of(I), cz_of(I)};
  const float T = p.Tr + r.dT;
  float b[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float x = p.weak ? r.usp[d] : r.u[d];
    b[d] = cs[d] == 0 ? 1.0f - x * x : 0.5f * ((cs[d] > 0 ? x : -x) + x * x);
  }
#pragma unroll
  for (int a = 0; a + 1 < M; a += 2) {
    const float2 z = mul2(make_float2(p.R_a[a], p.R_a[a + 1]), make_float2(T, T));
    float2 f[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float2 bb = make_float2(b[d], b[d]);
      f[d] = cs[d] == 0 ? sub2(bb, z) : fma2(make_float2(0.5f, 0.5f), z, bb);
    }
    const float2 ra = add2(make_float2(p.RL[a], p.RL[a + 1]), make_float2(r.ra[a], r.ra[a + 1]));
    const float2 s = fma2(mul2(ra, f[0]), mul2(f[1], f[2]), make_float2(-p.bref[a][k2], -p.bref[a + 1][k2]));
    sh[a] = s.x;
    sh[a + 1] = s.y;
  }
  if constexpr (M % 2) {
    constexpr int a = M - 1;
    const float z = p.R_a[a] * T;
    float f[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) f[d] = cs[d] == 0 ? b[d] - z : b[d] + 0.5f * z;
    sh[a] = (p.RL[a] + r.ra[a]) * f[0] * (f[1] * f[2]) - p.bref[a][k2];
  }
  sh[M] = eq_shift_f<I>(p, M, r.u, r.dth, r.drho);
  sh[M + 1] = eq_shift_g<I>(p, M, r.u, r.dth, r.drho, r.dE0, r.Gq, r.hq);
}

// A record as loaded (the species velocity only under weak coupling).
template <int M, bool NC>
struct RecLoad {
  static constexpr int NT = (1 + M + 3) / 4;
  float4 q[3 + NT];
  __device__ __forceinline__ RecLoad(const float* __restrict__ buf, long long N, long long node, int weak) {
    const float4* r = reinterpret_cast<const float4*>(buf) + node;
#pragma unroll
    for (int k = 0; k < 2 + NT; ++k) q[k] = ld<NC>(r + k * N);
    q[2 + NT] = weak ? ld<NC>(r + (2 + NT) * N) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
};

// What one sender adds to the populations it sent along the three velocities
// (c_x = -1, 0, 1; c_y; c_z) of a row: the equilibrium shifts of every
// lattice (the values of eq_shift) and, on f and g, the deferred terms
// c . X / 2 (faces) and w(theta) c . K.  The (y, z) factors, and all that
// depends on the sender alone, are formed once for the three.
// Which lane forms a sender's terms depends on where the receiver falls in its
// warp, so every operation's rounding is fixed here (paired instructions, and
// the scalar operations of lbm_helpers.cuh that the compiler does not
// contract): the same sender gives the same bits wherever its terms are
// formed, and a node's result does not depend on its place in a warp.
// (y, z) factors of a row for the species: per axis Psi_c = a + be z.
struct RowSpecies {
  float by, bz, ay, az, x2, hx;
  float T;
  int k2;
  __device__ __forceinline__ RowSpecies(float ux, float uy, float uz, float T_, int cy, int cz)
      : by(cy ? 0.5f : -1.0f), bz(cz ? 0.5f : -1.0f), x2(mul1(ux, ux)), hx(mul1(0.5f, ux)), T(T_), k2(cy * cy + cz * cz) {
    ay = fma1(mul1(by, uy), uy, fma1(0.5f * cy, uy, cy ? 0.0f : 1.0f));
    az = fma1(mul1(bz, uz), uz, fma1(0.5f * cz, uz, cz ? 0.0f : 1.0f));
  }
};
// Shifts of species a0, a1 with densities RL + d.
__device__ __forceinline__ void row_species(const DevParams<float>& p, const RowSpecies& r, int a0, int a1, float2 d,
                                            float2 (&out)[3]) {
  const float2 z = mul2(make_float2(p.R_a[a0], p.R_a[a1]), bcast<float2>(r.T));
  const float2 ra = add2(make_float2(p.RL[a0], p.RL[a1]), d);
  const float2 yz = mul2(mul2(ra, fma2(bcast<float2>(r.by), z, bcast<float2>(r.ay))),
                         fma2(bcast<float2>(r.bz), z, bcast<float2>(r.az)));
  const float2 s = add2(bcast<float2>(r.x2), z), hs = mul2(bcast<float2>(0.5f), s);
  const float2 r0 = make_float2(-p.bref[a0][r.k2], -p.bref[a1][r.k2]);
  const float2 r1 = make_float2(-p.bref[a0][r.k2 + 1], -p.bref[a1][r.k2 + 1]);
  out[0] = fma2(yz, sub2(hs, bcast<float2>(r.hx)), r1);
  out[1] = fma2(yz, sub2(bcast<float2>(1.0f), s), r0);
  out[2] = fma2(yz, add2(hs, bcast<float2>(r.hx)), r1);
}
// f and g: A, B the record's first two float4s, hq, K, and the component x of
// X that a face velocity of the row needs.  SEP: the deferred terms apart, in
// cf and cg (for the readers that add the parts in FP64).
template <bool SEP>
__device__ __forceinline__ void row_fg(const DevParams<float>& p, int M, float4 A, float4 B, float hq,
                                       const float (&k)[3], float x, int cy, int cz, float (&f)[3], float (&g)[3],
                                       float* cf_out, float* cg_out) {
  const float dth = B.x, drho = B.y;
  const float by = cy ? 0.5f : -1.0f, bz = cz ? 0.5f : -1.0f, sy = (float)cy, sz = (float)cz;
  const int kyz = cy * cy + cz * cz;
  const float x2 = mul1(A.x, A.x), hx = mul1(0.5f, A.x);
  const float r1 = mul1(0.5f, p.thr), r0 = sub1(1.0f, p.thr);
  const float ry = cy ? r1 : r0, rz = cz ? r1 : r0, ryz = mul1(ry, rz);
  const float wy = mul1(by, dth), wz = mul1(bz, dth), wx = mul1(0.5f, dth);    // w_c(theta) - w_c(theta_r); x: c = 0 gives -dth
  {
    const float rho = add1(p.RL[M], drho);
    const float dy = fma1(mul1(by, A.y), A.y, fma1(mul1(0.5f, sy), A.y, wy));
    const float dz = fma1(mul1(bz, A.z), A.z, fma1(mul1(0.5f, sz), A.z, wz));
    const float az = add1(rz, dz), ayz = mul1(add1(ry, dy), az), fyz = fma1(dy, az, mul1(ry, dz));
    const float hs = mul1(0.5f, fma1(A.x, A.x, dth)), cf = mul1(0.5f, x);
    const float e1 = mul1(r1, fyz), d1 = mul1(drho, mul1(r1, ryz));
    f[0] = fma1(rho, fma1(sub1(hs, hx), ayz, e1), d1);
    f[1] = fma1(rho, fma1(mul1(-2.0f, hs), ayz, mul1(r0, fyz)), mul1(drho, mul1(r0, ryz)));
    f[2] = fma1(rho, fma1(add1(hs, hx), ayz, e1), d1);
    if constexpr (SEP) {
      cf_out[0] = kyz == 0 ? -cf : 0.0f;
      cf_out[1] = kyz == 1 ? mul1(add1(sy, sz), cf) : 0.0f;
      cf_out[2] = kyz == 0 ? cf : 0.0f;
    } else {
      if (kyz == 0) { f[0] = sub1(f[0], cf); f[2] = add1(f[2], cf); }
      if (kyz == 1) f[1] = fma1(add1(sy, sz), cf, f[1]);
    }
  }
  const float oz = add1(rz, wz), oyz = mul1(add1(ry, wy), oz), dyz = fma1(wy, oz, mul1(ry, wz));
  const float w1 = mul1(add1(r1, wx), oyz), w0 = mul1(sub1(r0, dth), oyz);
  const float c0 = mul1(fma1(-dth, oyz, mul1(r0, dyz)), energy_rest(p, M, kyz));
  const float c1 = mul1(fma1(wx, oyz, mul1(r1, dyz)), energy_rest(p, M, kyz + 1));
  const float uyz = fma1(sy, A.y, mul1(sz, A.z)), kk = fma1(sy, k[1], mul1(sz, k[2]));
  const float es = fma1(mul1(0.5f, (float)kyz), drho, B.z), e0 = SEP ? es : add1(es, kk), e1 = fma1(0.5f, drho, e0);
  const float um = sub1(uyz, A.x), up = add1(uyz, A.x);
  const float b0 = fma1(um, fma1(B.w, um, hq), e1), b2 = fma1(up, fma1(B.w, up, hq), e1);
  g[0] = fma1(w1, SEP ? b0 : sub1(b0, k[0]), c1);
  g[1] = fma1(w0, fma1(uyz, fma1(B.w, uyz, hq), e0), c0);
  g[2] = fma1(w1, SEP ? b2 : add1(b2, k[0]), c1);
  if constexpr (SEP) {
    cg_out[0] = mul1(w1, sub1(kk, k[0]));
    cg_out[1] = mul1(w0, kk);
    cg_out[2] = mul1(w1, add1(kk, k[0]));
  }
  if (kyz <= 1) {
    const float theta = add1(p.thr, dth), z1 = fma1(-3.0f, theta, 1.0f);
    const float zb = mul1(0.5f, fma1(z1, fma1(drho, theta, mul1(p.RL[M], dth)), mul1(mul1(-3.0f, dth), p.Pr)));
    const float zG = mul1(mul1(z1, B.w), theta);
    if (kyz == 0) {
      const float bx = mul1(0.5f, fma1(zG, x2, zb)), u2 = fma1(A.x, A.x, fma1(A.y, A.y, mul1(A.z, A.z)));
      g[0] = sub1(g[0], bx);
      g[1] = add1(g[1], fma1(zG, u2, mul1(3.0f, zb)));
      g[2] = sub1(g[2], bx);
    } else {
      const float c = cy ? A.y : A.z;
      g[1] = fma1(-0.5f, fma1(zG, mul1(c, c), zb), g[1]);
    }
  }
}
template <int M, bool SEP = false>
struct RowTerms {
  static constexpr int NP = (M + 1) / 2;
  float2 sp[NP][3];
  float f[3], g[3];
  float cf[SEP ? 3 : 1], cg[SEP ? 3 : 1];
};
// K and the component of X that a face velocity of the row needs.
template <bool NC>
struct RowSide {
  float k[3], x;
  __device__ __forceinline__ RowSide(const float* __restrict__ side, long long N, long long snd, int cy, int cz) {
    k[0] = ld<NC>(side + (SP_K + 0) * N + snd);
    k[1] = cy ? ld<NC>(side + (SP_K + 1) * N + snd) : 0.0f;
    k[2] = cz ? ld<NC>(side + (SP_K + 2) * N + snd) : 0.0f;
    x = cy * cz == 0 ? ld<NC>(side + (SP_X + (cy ? 1 : (cz ? 2 : 0))) * N + snd) : 0.0f;
  }
};
// What a sender's RowTerms are formed from, as loaded.
template <int M, bool NC = false>
struct RowLoad {
  RecLoad<M, NC> rec;
  RowSide<NC> s;
  __device__ __forceinline__ RowLoad(const DevParams<float>& p, const float* __restrict__ side,
                                     const float* __restrict__ rin, long long snd, int cy, int cz)
      : rec(rin, p.N, snd, p.weak), s(side, p.N, snd, cy, cz) {}
};
template <int M, bool NC, bool SEP>
__device__ __forceinline__ void row_terms(const DevParams<float>& p, const RowLoad<M, NC>& in, int cy, int cz,
                                          RowTerms<M, SEP>& out) {
  constexpr int NT = RecLoad<M, NC>::NT, NP = (M + 1) / 2;
  const float4 A = in.rec.q[0], W = p.weak ? in.rec.q[2 + NT] : A;
  float t[4 * NT];
#pragma unroll
  for (int k = 0; k < NT; ++k) {
    const float4 c = in.rec.q[2 + k];
    t[4 * k] = c.x; t[4 * k + 1] = c.y; t[4 * k + 2] = c.z; t[4 * k + 3] = c.w;
  }
  const RowSpecies r(W.x, W.y, W.z, add1(p.Tr, A.w), cy, cz);
#pragma unroll
  for (int q = 0; q < NP; ++q)
    row_species(p, r, 2 * q, 2 * q + 1 < M ? 2 * q + 1 : 2 * q, make_float2(t[2 * q], t[2 * q + 1]), out.sp[q]);
  row_fg<SEP>(p, M, A, in.rec.q[1], t[M], in.s.k, in.s.x, cy, cz, out.f, out.g, out.cf, out.cg);
}
// The same for one velocity (c_x = -1 or 1 given) of one sender.  refl: the
// population is the node's own of the opposite velocity, reflected by a wall;
// f^eq of the opposite velocity is that of -u, and the deferred terms change
// sign, so the row is formed with the sender's vectors reversed.
template <int M, bool NC, bool SEP = false>
__device__ __forceinline__ void edge_terms(const DevParams<float>& p, RowLoad<M, NC> in, bool refl, int cx, int cy,
                                           int cz, float2 (&sp)[(M + 1) / 2], float& f, float& g,
                                           float* cf = nullptr, float* cg = nullptr) {
  if (refl) {
    float4& A = in.rec.q[0];
    float4& W = in.rec.q[2 + RecLoad<M, NC>::NT];
    A.x = -A.x; A.y = -A.y; A.z = -A.z;
    W.x = -W.x; W.y = -W.y; W.z = -W.z;
#pragma unroll
    for (int c = 0; c < 3; ++c) in.s.k[c] = -in.s.k[c];
    in.s.x = -in.s.x;
  }
  RowTerms<M, SEP> t;
  row_terms<M>(p, in, cy, cz, t);
#pragma unroll
  for (int q = 0; q < RowTerms<M>::NP; ++q) sp[q] = cx > 0 ? t.sp[q][2] : t.sp[q][0];
  f = cx > 0 ? t.f[2] : t.f[0];
  g = cx > 0 ? t.g[2] : t.g[0];
  if constexpr (SEP) {
    *cf = cx > 0 ? t.cf[2] : t.cf[0];
    *cg = cx > 0 ? t.cg[2] : t.cg[0];
  }
}

// The record of a node from its coupled moments, in FP64 (initialisation
// and set_populations): rho_a the coupled species densities, rho, j and rho E
// of the mixture lattices, u_sp the species velocity.
template <int M>
__device__ __forceinline__ EqRec<M> eq_record64(const DevParams<double>& p, const double (&rho_a)[M], double rho,
                                               const double (&j)[3], double rhoE, const double (&u_sp)[3]) {
  double rsp = 0.0;
#pragma unroll
  for (int a = 0; a < M; ++a) rsp += rho_a[a];
  double inv_m = 0.0, Y[M];
#pragma unroll
  for (int a = 0; a < M; ++a) {
    Y[a] = rho_a[a] / rsp;
    inv_m += Y[a] * p.inv_mass[a];
  }
  const double u[3] = {j[0] / rho, j[1] / rho, j[2] / rho};
  const double usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  const double T = T_from_energy64(p, Y, M, rhoE / rho - 0.5 * usq);   // Eqs. (temperature), (temperature2)
  const double th = p.R_U * inv_m * T;
  double H = 0.0;
#pragma unroll
  for (int a = 0; a < M; ++a) H += Y[a] * H_a64(p, a, T);
  const double hk = H + 0.5 * usq;
  const double Gc = rho * (hk + th) / (2.0 * th);
  EqRec<M> r;
#pragma unroll
  for (int c = 0; c < 3; ++c) { r.u[c] = (float)u[c]; r.usp[c] = (float)u_sp[c]; }
  r.dth = (float)(th - p.thr); r.dT = (float)(T - p.Tr);
  r.drho = (float)(rho - p.RL[M]);
  r.dE0 = (float)(rhoE - 1.5 * rho * th - Gc * usq - (p.RL[M + 1] - 1.5 * p.RL[M] * p.thr));
  r.Gq = (float)(Gc / th);
  r.hq = (float)(hk * rho / th);
#pragma unroll
  for (int a = 0; a < M; ++a) r.ra[a] = (float)(rho_a[a] - p.RL[a]);
  return r;
}

}  // namespace lbm
