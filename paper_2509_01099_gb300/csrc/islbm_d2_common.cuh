// Shared by the 2-D kernels: the parameters of a step, the rest weights and the
// collision.
#pragma once

#include "islbm_internal.h"
#include "islbm_lanes.cuh"

namespace islbm {
namespace {

template <typename R>
struct P2 {
  int nx, ny, pitch;
  int y0, y1;           // rows the step computes: [y0, y1) (all rows unless a slab is set)
  long long plane;
  const int* bx[2];
  const R* wx[2];
  const int* by[2];
  const R* wy[2];
  const float4* px[2];  // packed FP32 tables of the tiled kernel
  const float4* py[2];
  // The temperature populations carry T - T_s (T_s: mean wall temperature);
  // the buoyancy force is rho g beta (T - T_ref) = rho g beta (T - T_s + Fb).
  R gbeta, s_e, s_eps, s_q, s_nu, q_j, q_e, q_nu, a_T;
  R Ts, Fb;             // T_s and T_s - T_ref
  R abb_hot, abb_cold;  // omega (T_w - T_s) of the anti-bounce-back rule
  unsigned step;        // step counter (seeds the stochastic rounding of 16-bit stores)
};

// Rest weights w_i of the D2Q9 populations.
template <typename R>
__device__ __forceinline__ R wrest(int i) {
  return i == 0 ? R(4.0 / 9.0) : (i < 5 ? R(1.0 / 9.0) : R(1.0 / 36.0));
}

// Rest weights (t_0, t_i) of the D2Q5 temperature equilibrium, (1 - a_T)/5 and
// (4 + a_T)/20.
__device__ __forceinline__ void trest(float aT, float& t0, float& ti) {
  t0 = (1.f - aT) * 0.2f;
  ti = (4.f + aT) * 0.05f;
}

// MRT collision in deviation form (Sec. 2.1), of one node (L = R) or of two
// nodes at once (L = float2, R = float: paired FP32 instructions).
//   m = M f with the Lallemand-Luo rows (rho, e, eps, jx, qx, jy, qy, pxx, pxy);
//   m+ = m - S (m - m_eq) + (I - S/2) M F~ with the printed m_eq and M F~;
//   f+ = f + M^-1 (m+ - m), M^-1 = M^T diag(1/|row_k|^2).
//   g: n = N g with rows (T, jx, jy, -4+5|c|^2, cx^2-cy^2), n+ = n - Q (n - n_eq).
// The buoyancy F = rho g beta (T - T_ref) acts along +y; u = (sum e f + F/2)/rho.
// The populations carry T - T_s, which is also the temperature of the
// equilibrium fluxes u T and of a_T T.
// Returns rho, u and T of the pre-collision state, and in m_o the moments of
// the post-collision state: drho, jx, jy + F_y, T - T_s.
template <typename L, typename R>
__device__ __forceinline__ void collide_m(L (&f)[9], L (&g)[5], const P2<R>& p, L& rho_o,
                                          L& ux_o, L& uy_o, L& T_o, L (&m_o)[4]) {
  using K = Lanes<L>;
  auto c = [](double v) { return K::bc((typename K::S)v); };
  // pre-collision moments
  const L d13 = lsub(f[1], f[3]), d56 = lsub(f[5], f[6]), d87 = lsub(f[8], f[7]);
  const L d24 = lsub(f[2], f[4]), p56 = ladd(f[5], f[6]), p78 = ladd(f[7], f[8]);
  const L drho = ladd(ladd(ladd(ladd(f[0], f[1]), ladd(f[2], f[3])),
                           ladd(ladd(f[4], f[5]), ladd(f[6], f[7]))), f[8]);
  const L rho = ladd(c(1), drho);
  const L jx = ladd(ladd(d13, d56), d87);
  const L jy = lsub(ladd(d24, p56), p78);
  const L Tr = ladd(ladd(ladd(g[0], g[1]), ladd(g[2], g[3])), g[4]);  // T - T_s
  const L Fy = lmul(lmul(rho, K::bc(p.gbeta)), ladd(Tr, K::bc(p.Fb)));
  const L inv = lrcp(rho);
  const L ux = lmul(jx, inv);
  const L uy = lmul(lfma(c(0.5), Fy, jy), inv);
  const L ux2 = lmul(ux, ux), uy2 = lmul(uy, uy);
  const L rusq = lmul(rho, ladd(ux2, uy2));
  const L uF = lmul(uy, Fy);

  const L sax = ladd(ladd(f[1], f[2]), ladd(f[3], f[4]));
  const L sdg = ladd(p56, p78);
  const L m1 = lfma(c(2), sdg, lsub(lmul(c(-4), f[0]), sax));
  const L m2 = lfma(c(-2), sax, lfma(c(4), f[0], sdg));
  const L m4 = lfma(c(-2), d13, ladd(d56, d87));
  const L m6 = lfma(c(-2), d24, lsub(p56, p78));
  const L m7 = lsub(ladd(f[1], f[3]), ladd(f[2], f[4]));
  const L m8 = lsub(ladd(f[5], f[7]), ladd(f[6], f[8]));

  // moment increments; the deviation form moves M w = (1,-2,1,0,...) into m_eq
  const R he = R(1) - R(0.5) * p.s_e, heps = R(1) - R(0.5) * p.s_eps;
  const R hq = R(1) - R(0.5) * p.s_q, hnu = R(1) - R(0.5) * p.s_nu;
  const L dm1 = lfma(K::bc(-p.s_e), lfma(c(-3), rusq, lfma(c(2), drho, m1)),
                     lmul(K::bc(R(6) * he), uF));
  const L dm2 = lfma(K::bc(-p.s_eps), lfma(c(3), rusq, lsub(m2, drho)),
                     lmul(K::bc(R(-6) * heps), uF));
  const L dm4 = lmul(K::bc(-p.s_q), lfma(rho, ux, m4));
  const L dm5 = Fy;  // j_y gains exactly F_y (independent of s_j)
  const L dm6 = lfma(K::bc(-p.s_q), lfma(rho, uy, m6), lmul(K::bc(-hq), Fy));
  const L dm7 = lfma(K::bc(-p.s_nu), lfma(rho, lsub(uy2, ux2), m7),
                     lmul(K::bc(R(-2) * hnu), uF));
  const L dm8 = lfma(K::bc(-p.s_nu), lsub(m8, lmul(lmul(rho, ux), uy)),
                     lmul(K::bc(hnu), lmul(ux, Fy)));

  // f+ = f + M^-1 dm
  const L a1 = lmul(dm1, c(1.0 / 36.0)), a2 = lmul(dm2, c(1.0 / 36.0));
  const L a4 = lmul(dm4, c(1.0 / 12.0)), a5 = lmul(dm5, c(1.0 / 6.0));
  const L a6 = lmul(dm6, c(1.0 / 12.0)), a7 = lmul(dm7, c(0.25)), a8 = lmul(dm8, c(0.25));
  const L cax = lsub(lmul(c(-2), a2), a1);   // -a1 - 2 a2
  const L cdg = lfma(c(2), a1, a2);          // 2 a1 + a2
  f[0] = lfma(c(4), lsub(a2, a1), f[0]);
  const L t13 = ladd(cax, a7);
  f[1] = ladd(f[1], lfma(c(-2), a4, t13));
  f[3] = ladd(f[3], lfma(c(2), a4, t13));
  const L t24 = lsub(cax, a7), v24 = lfma(c(-2), a6, a5);   // a5 - 2 a6
  f[2] = ladd(f[2], ladd(t24, v24));
  f[4] = ladd(f[4], lsub(t24, v24));
  const L w56 = ladd(a5, a6), p48 = ladd(a4, a8), m48 = lsub(a4, a8);
  const L cp = ladd(cdg, w56), cm = lsub(cdg, w56);
  f[5] = ladd(f[5], ladd(cp, p48));
  f[6] = ladd(f[6], lsub(cp, p48));
  f[7] = ladd(f[7], lsub(cm, m48));
  f[8] = ladd(f[8], ladd(cm, m48));

  const L n1 = lsub(g[1], g[3]), n2 = lsub(g[2], g[4]);
  const L n3 = lfma(c(-4), g[0], ladd(ladd(g[1], g[2]), ladd(g[3], g[4])));
  const L n4 = lsub(ladd(g[1], g[3]), ladd(g[2], g[4]));
  const L b1 = lmul(K::bc(R(-0.5) * p.q_j), lsub(n1, lmul(ux, Tr)));
  const L b2 = lmul(K::bc(R(-0.5) * p.q_j), lsub(n2, lmul(uy, Tr)));
  const L b3 = lmul(K::bc(R(-0.05) * p.q_e), lsub(n3, lmul(K::bc(p.a_T), Tr)));
  const L b4 = lmul(K::bc(R(-0.25) * p.q_nu), n4);
  g[0] = lfma(c(-4), b3, g[0]);
  const L s34 = ladd(b3, b4), d34 = lsub(b3, b4);
  g[1] = ladd(g[1], ladd(b1, s34));
  g[3] = ladd(g[3], lsub(s34, b1));
  g[2] = ladd(g[2], ladd(b2, d34));
  g[4] = ladd(g[4], lsub(d34, b2));

  rho_o = rho;
  ux_o = ux;
  uy_o = uy;
  T_o = Tr;
  m_o[0] = drho;
  m_o[1] = jx;
  m_o[2] = ladd(jy, Fy);
  m_o[3] = Tr;
}

// Constants of the paired collision, both lanes equal.  As kernel parameters
// the paired instructions take them as 64-bit operands; a literal or a scalar
// would have to be copied into a register pair at every use.
struct PairC {
  float2 gbeta, Fb, ms_e, he6, ms_eps, heps6, ms_q, mhq, ms_nu, hnu2, hnu, hq_j, hq_e, a_T, hq_nu;
  float2 one, half, two, m4, m2, four, m3, three, r36, r12, r6, quarter;
};

inline PairC make_pair_constants(const P2<float>& p) {
  auto d = [](double v) { return make_float2((float)v, (float)v); };
  const float he = 1.f - 0.5f * p.s_e, heps = 1.f - 0.5f * p.s_eps;
  const float hq = 1.f - 0.5f * p.s_q, hnu = 1.f - 0.5f * p.s_nu;
  PairC k;
  k.gbeta = d(p.gbeta);
  k.Fb = d(p.Fb);
  k.ms_e = d(-p.s_e);
  k.he6 = d(6.f * he);
  k.ms_eps = d(-p.s_eps);
  k.heps6 = d(-6.f * heps);
  k.ms_q = d(-p.s_q);
  k.mhq = d(-hq);
  k.ms_nu = d(-p.s_nu);
  k.hnu2 = d(-2.f * hnu);
  k.hnu = d(hnu);
  k.hq_j = d(-0.5f * p.q_j);
  k.hq_e = d(-0.05f * p.q_e);
  k.a_T = d(p.a_T);
  k.hq_nu = d(-0.25f * p.q_nu);
  k.one = d(1.0);
  k.half = d(0.5);
  k.two = d(2.0);
  k.m4 = d(-4.0);
  k.m2 = d(-2.0);
  k.four = d(4.0);
  k.m3 = d(-3.0);
  k.three = d(3.0);
  k.r36 = d(1.0 / 36.0);
  k.r12 = d(1.0 / 12.0);
  k.r6 = d(1.0 / 6.0);
  k.quarter = d(0.25);
  return k;
}

// collide_m of two nodes with the constants of PairC: the same operations in the
// same order, so the same bits.
__device__ __forceinline__ void collide_pair(float2 (&f)[9], float2 (&g)[5], const PairC& k,
                                             float2 (&m_o)[4]) {
  using L = float2;
  // pre-collision moments
  const L d13 = lsub(f[1], f[3]), d56 = lsub(f[5], f[6]), d87 = lsub(f[8], f[7]);
  const L d24 = lsub(f[2], f[4]), p56 = ladd(f[5], f[6]), p78 = ladd(f[7], f[8]);
  const L drho = ladd(ladd(ladd(ladd(f[0], f[1]), ladd(f[2], f[3])),
                           ladd(ladd(f[4], f[5]), ladd(f[6], f[7]))), f[8]);
  const L rho = ladd(k.one, drho);
  const L jx = ladd(ladd(d13, d56), d87);
  const L jy = lsub(ladd(d24, p56), p78);
  const L Tr = ladd(ladd(ladd(g[0], g[1]), ladd(g[2], g[3])), g[4]);  // T - T_s
  const L Fy = lmul(lmul(rho, k.gbeta), ladd(Tr, k.Fb));
  const L inv = lrcp(rho);
  const L ux = lmul(jx, inv);
  const L uy = lmul(lfma(k.half, Fy, jy), inv);
  const L ux2 = lmul(ux, ux), uy2 = lmul(uy, uy);
  const L rusq = lmul(rho, ladd(ux2, uy2));
  const L uF = lmul(uy, Fy);

  const L sax = ladd(ladd(f[1], f[2]), ladd(f[3], f[4]));
  const L sdg = ladd(p56, p78);
  const L m1 = lfma(k.two, sdg, lsub(lmul(k.m4, f[0]), sax));
  const L m2 = lfma(k.m2, sax, lfma(k.four, f[0], sdg));
  const L m4 = lfma(k.m2, d13, ladd(d56, d87));
  const L m6 = lfma(k.m2, d24, lsub(p56, p78));
  const L m7 = lsub(ladd(f[1], f[3]), ladd(f[2], f[4]));
  const L m8 = lsub(ladd(f[5], f[7]), ladd(f[6], f[8]));

  // moment increments; the deviation form moves M w = (1,-2,1,0,...) into m_eq
  const L dm1 = lfma(k.ms_e, lfma(k.m3, rusq, lfma(k.two, drho, m1)),
                     lmul(k.he6, uF));
  const L dm2 = lfma(k.ms_eps, lfma(k.three, rusq, lsub(m2, drho)),
                     lmul(k.heps6, uF));
  const L dm4 = lmul(k.ms_q, lfma(rho, ux, m4));
  const L dm5 = Fy;  // j_y gains exactly F_y (independent of s_j)
  const L dm6 = lfma(k.ms_q, lfma(rho, uy, m6), lmul(k.mhq, Fy));
  const L dm7 = lfma(k.ms_nu, lfma(rho, lsub(uy2, ux2), m7),
                     lmul(k.hnu2, uF));
  const L dm8 = lfma(k.ms_nu, lsub(m8, lmul(lmul(rho, ux), uy)),
                     lmul(k.hnu, lmul(ux, Fy)));

  // f+ = f + M^-1 dm
  const L a1 = lmul(dm1, k.r36), a2 = lmul(dm2, k.r36);
  const L a4 = lmul(dm4, k.r12), a5 = lmul(dm5, k.r6);
  const L a6 = lmul(dm6, k.r12), a7 = lmul(dm7, k.quarter), a8 = lmul(dm8, k.quarter);
  const L cax = lsub(lmul(k.m2, a2), a1);   // -a1 - 2 a2
  const L cdg = lfma(k.two, a1, a2);          // 2 a1 + a2
  f[0] = lfma(k.four, lsub(a2, a1), f[0]);
  const L t13 = ladd(cax, a7);
  f[1] = ladd(f[1], lfma(k.m2, a4, t13));
  f[3] = ladd(f[3], lfma(k.two, a4, t13));
  const L t24 = lsub(cax, a7), v24 = lfma(k.m2, a6, a5);   // a5 - 2 a6
  f[2] = ladd(f[2], ladd(t24, v24));
  f[4] = ladd(f[4], lsub(t24, v24));
  const L w56 = ladd(a5, a6), p48 = ladd(a4, a8), m48 = lsub(a4, a8);
  const L cp = ladd(cdg, w56), cm = lsub(cdg, w56);
  f[5] = ladd(f[5], ladd(cp, p48));
  f[6] = ladd(f[6], lsub(cp, p48));
  f[7] = ladd(f[7], lsub(cm, m48));
  f[8] = ladd(f[8], ladd(cm, m48));

  const L n1 = lsub(g[1], g[3]), n2 = lsub(g[2], g[4]);
  const L n3 = lfma(k.m4, g[0], ladd(ladd(g[1], g[2]), ladd(g[3], g[4])));
  const L n4 = lsub(ladd(g[1], g[3]), ladd(g[2], g[4]));
  const L b1 = lmul(k.hq_j, lsub(n1, lmul(ux, Tr)));
  const L b2 = lmul(k.hq_j, lsub(n2, lmul(uy, Tr)));
  const L b3 = lmul(k.hq_e, lsub(n3, lmul(k.a_T, Tr)));
  const L b4 = lmul(k.hq_nu, n4);
  g[0] = lfma(k.m4, b3, g[0]);
  const L s34 = ladd(b3, b4), d34 = lsub(b3, b4);
  g[1] = ladd(g[1], ladd(b1, s34));
  g[3] = ladd(g[3], lsub(s34, b1));
  g[2] = ladd(g[2], ladd(b2, d34));
  g[4] = ladd(g[4], lsub(d34, b2));

  m_o[0] = drho;
  m_o[1] = jx;
  m_o[2] = ladd(jy, Fy);
  m_o[3] = Tr;
}

template <typename L, typename R>
__device__ __forceinline__ void collide(L (&f)[9], L (&g)[5], const P2<R>& p, L& rho_o,
                                        L& ux_o, L& uy_o, L& T_o) {
  L m[4];
  collide_m(f, g, p, rho_o, ux_o, uy_o, T_o, m);
}

template <typename R>
P2<R> make_params(const Solver& s) {
  P2<R> p;
  p.nx = s.n[0];
  p.ny = s.n[1];
  p.y0 = s.row_end > 0 ? s.row_begin : 0;
  p.y1 = s.row_end > 0 ? s.row_end : s.n[1];
  p.pitch = s.pitch;
  p.plane = s.plane;
  for (int k = 0; k < 2; ++k) {
    p.bx[k] = s.dax[0].base[k];
    p.wx[k] = static_cast<const R*>(s.dax[0].w[k]);
    p.by[k] = s.dax[1].base[k];
    p.wy[k] = static_cast<const R*>(s.dax[1].w[k]);
    p.px[k] = s.dax[0].packed[k];
    p.py[k] = s.dax[1].packed[k];
  }
  const Physics& h = s.ph;
  p.gbeta = R(h.gbeta);
  p.Ts = R(h.Ts);
  p.Fb = R(h.Ts - h.T0);
  p.s_e = R(h.s_e);
  p.s_eps = R(h.s_eps);
  p.s_q = R(h.s_q);
  p.s_nu = R(h.s_nu);
  p.q_j = R(h.q_j);
  p.q_e = R(h.q_e);
  p.q_nu = R(h.q_nu);
  p.a_T = R(h.a_T);
  p.abb_hot = R(h.omega * (h.T_hot - h.Ts));
  p.abb_cold = R(h.omega * (h.T_cold - h.Ts));
  p.step = (unsigned)s.time;
  return p;
}

// rows of the step: the slab [row_begin, row_end) when one is set
int step_rows(const Solver& s) { return s.row_end > 0 ? s.row_end - s.row_begin : s.n[1]; }

}  // namespace
}  // namespace islbm
