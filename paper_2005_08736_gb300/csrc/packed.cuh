// Packed FP32 pairs for the sweep kernels: one instruction applies an add,
// multiply or fused multiply-add to both halves of a float2 (__fadd2_rn /
// __fmul2_rn / __ffma2_rn, sm_100 and later).  The FP32 sweeps are bound by
// instruction issue before the FMA pipe, so evaluating two reconstructions in
// the halves of one float2 halves the issue slots of their arithmetic.
//
// In k_march (march.cuh) the halves are two adjacent face layers, from the
// cells to the flux; in k_sweep (sweep_tile.cuh) and the adjoint two fields of
// one point, in its face fields the two cells of a face.  The formulas are
// those of recon.cuh, compat.cuh and physics.cuh, evaluated pairwise; only the
// rounding of the fused operations can differ from the scalar code.
#pragma once

#include <cmath>

#include "physics.cuh"
#include "recon.cuh"

namespace hgks {

// On the host (the checks of tests/support) each pair operation is the two
// scalar operations it stands for.
HGKS_HD float2 bc2(float s) { return make_float2(s, s); }
HGKS_HD float2 add2(float2 a, float2 b) {
#if defined(__CUDA_ARCH__)
  return __fadd2_rn(a, b);
#else
  return make_float2(a.x + b.x, a.y + b.y);
#endif
}
HGKS_HD float2 mul2(float2 a, float2 b) {
#if defined(__CUDA_ARCH__)
  return __fmul2_rn(a, b);
#else
  return make_float2(a.x * b.x, a.y * b.y);
#endif
}
HGKS_HD float2 fma2(float2 a, float2 b, float2 c) {
#if defined(__CUDA_ARCH__)
  return __ffma2_rn(a, b, c);
#else
  return make_float2(std::fma(a.x, b.x, c.x), std::fma(a.y, b.y, c.y));
#endif
}
// a - b
HGKS_HD float2 sub2(float2 a, float2 b) { return fma2(b, bc2(-1.f), a); }
HGKS_HD float2 rcp2(float2 a) { return make_float2(1.f / a.x, 1.f / a.y); }

// Linear-weight tangential reconstruction (the quartic through five face
// averages) of two columns at once: values v[m] and derivatives d[m] (per
// unit cell length) at the Gauss abscissae s_m = -+1/(2 sqrt 3):
//   P(+-g) = E +- O,  P'(+-g) = A +- B  with
//   E = f2 + (-f2/720 + (f1+f3)/1080 - (f0+f4)/4320), in this grouping: a
//   rounded 719/720 would scale every face value,
//   O = sqrt3 (7/432 (f0-f4) + 25/216 (f3-f1)),
//   A = (f0-f4)/12 + 2(f3-f1)/3,  B = sqrt3/54 (13 (f1+f3) - 24 f2 - (f0+f4)).
// The host checks alone call it: k_march takes tangential_linear_scaled_x2.
HGKS_HD void tangential_linear_x2(float2 f0, float2 f1, float2 f2, float2 f3,
                                                     float2 f4, float2 v[2], float2 d[2]) {
  const float sq3 = 1.7320508075688772f;
  const float2 s13 = add2(f1, f3), s04 = add2(f0, f4);
  const float2 d04 = sub2(f0, f4), d31 = sub2(f3, f1);
  const float2 E = add2(f2, fma2(f2, bc2(-1.f / 720.f), fma2(s13, bc2(1.f / 1080.f), mul2(s04, bc2(-1.f / 4320.f)))));
  const float2 O = fma2(d04, bc2(sq3 * 7.f / 432.f), mul2(d31, bc2(sq3 * 25.f / 216.f)));
  const float2 A = fma2(d04, bc2(1.f / 12.f), mul2(d31, bc2(2.f / 3.f)));
  const float k = sq3 / 54.f;
  const float2 B = fma2(s13, bc2(13.f * k), fma2(f2, bc2(-24.f * k), mul2(s04, bc2(-k))));
  v[0] = sub2(E, O);
  v[1] = add2(E, O);
  d[0] = sub2(A, B);
  d[1] = add2(A, B);
}

HGKS_HD void tangential_linear_val_x2(float2 f0, float2 f1, float2 f2, float2 f3,
                                                         float2 f4, float2 v[2]) {
  const float sq3 = 1.7320508075688772f;
  const float2 s13 = add2(f1, f3), s04 = add2(f0, f4);
  const float2 d04 = sub2(f0, f4), d31 = sub2(f3, f1);
  const float2 E = add2(f2, fma2(f2, bc2(-1.f / 720.f), fma2(s13, bc2(1.f / 1080.f), mul2(s04, bc2(-1.f / 4320.f)))));
  const float2 O = fma2(d04, bc2(sq3 * 7.f / 432.f), mul2(d31, bc2(sq3 * 25.f / 216.f)));
  v[0] = sub2(E, O);
  v[1] = add2(E, O);
}

// Two point states (deviation value and derivatives along n, t1, t2, local
// frame), one per half.
struct PointStateX2 {
  float2 q[5];
  float2 dq[3][5];
};

// Smooth BGK flux at two points (physics.cuh, flux_smooth, through the
// primitive derivatives and their time derivatives): F - E(Q_ref) (WANT_F)
// and dF are added to Fs[0..4] and Fs[5..9].  The time derivatives are formed
// with the opposite sign (they enter dF linearly).
template <bool WANT_F>
__device__ __forceinline__ void flux_smooth_x2(const PointStateX2& st, const Gas<float>& g, float2 Fs[10]) {
  // Primitive state (prim_of).
  const float2 rho = add2(bc2(g.rho_r), st.q[0]);
  const float2 inv = rcp2(rho);
  const float2 U[3] = {mul2(st.q[1], inv), mul2(st.q[2], inv), mul2(st.q[3], inv)};
  const float2 nU[3] = {mul2(U[0], bc2(-1.f)), mul2(U[1], bc2(-1.f)), mul2(U[2], bc2(-1.f))};
  const float2 hq2 = mul2(bc2(0.5f), fma2(U[0], U[0], fma2(U[1], U[1], mul2(U[2], U[2]))));
  const float2 dp = mul2(bc2(g.gm1), fma2(mul2(hq2, bc2(-1.f)), rho, st.q[4]));
  const float2 p = add2(bc2(g.p_r), dp);
  const float2 H = add2(add2(bc2(g.h_r), st.q[4]), dp);

  // Derivatives along n, t1, t2 (prim_rates).
  float2 du[3][3], dpd[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float2* dQ = st.dq[d];
#pragma unroll
    for (int k = 0; k < 3; ++k) du[d][k] = mul2(fma2(nU[k], dQ[0], dQ[1 + k]), inv);
    float2 t = fma2(nU[0], dQ[1], dQ[4]);
    t = fma2(nU[1], dQ[2], t);
    t = fma2(nU[2], dQ[3], t);
    t = fma2(hq2, dQ[0], t);
    dpd[d] = mul2(bc2(g.gm1), t);
  }
  const float2 div = add2(add2(du[0][0], du[1][1]), du[2][2]);
  // minus the time derivatives of density, velocity and pressure
  const float2 rt = fma2(U[0], st.dq[0][0], fma2(U[1], st.dq[1][0], fma2(U[2], st.dq[2][0], mul2(rho, div))));
  float2 ut[3];
#pragma unroll
  for (int i = 0; i < 3; ++i)
    ut[i] = fma2(U[0], du[0][i], fma2(U[1], du[1][i], fma2(U[2], du[2][i], mul2(dpd[i], inv))));
  const float2 pt = fma2(U[0], dpd[0], fma2(U[1], dpd[1], fma2(U[2], dpd[2], mul2(mul2(bc2(g.gamma), p), div))));
  // minus the time derivative of the Euler flux (euler_flux_rate)
  const float2 m = st.q[1];
  const float2 mt = fma2(rt, U[0], mul2(rho, ut[0]));
  const float2 uu = fma2(U[0], ut[0], fma2(U[1], ut[1], mul2(U[2], ut[2])));
  const float2 Ht = fma2(bc2(g.gamma / g.gm1), pt, fma2(hq2, rt, mul2(rho, uu)));
  float2 dF[5];
  dF[0] = mt;
  dF[1] = fma2(mt, U[0], fma2(m, ut[0], pt));
  dF[2] = fma2(mt, U[1], mul2(m, ut[1]));
  dF[3] = fma2(mt, U[2], mul2(m, ut[2]));
  dF[4] = fma2(ut[0], H, mul2(U[0], Ht));
#pragma unroll
  for (int i = 0; i < 5; ++i) Fs[5 + i] = sub2(Fs[5 + i], dF[i]);
  if constexpr (WANT_F) {
    // Viscosity mu(T) of the gas law at T = p/rho.
    const float2 theta = mul2(p, inv);
    float2 mu = bc2(g.mu_ref);
    if (g.visc_law == 1) {
      mu = make_float2(g.mu_ref * tpow(theta.x * g.T_ref_inv, g.visc_exp),
                       g.mu_ref * tpow(theta.y * g.T_ref_inv, g.visc_exp));
    }
    // Viscous stress row of the normal direction and the heat flux
    // (ns_viscous_rates).
    const float2 dT0 = mul2(fma2(theta, mul2(st.dq[0][0], bc2(-1.f)), dpd[0]), inv);
    const float2 s00 = mul2(mu, fma2(div, bc2(-2.f / (g.K + 3.f)), mul2(bc2(2.f), du[0][0])));
    const float2 s01 = mul2(mu, add2(du[0][1], du[1][0]));
    const float2 s02 = mul2(mu, add2(du[0][2], du[2][0]));
    const float hc = -(g.pr_fix + 1.f) * 0.5f * (g.K + 5.f);
    float2 F[5];
    F[0] = m;
    F[1] = sub2(fma2(m, U[0], dp), s00);
    F[2] = sub2(mul2(m, U[1]), s01);
    F[3] = sub2(mul2(m, U[2]), s02);
    const float2 work = fma2(s00, U[0], fma2(s01, U[1], mul2(s02, U[2])));
    F[4] = fma2(mul2(mu, bc2(hc)), dT0, sub2(mul2(U[0], H), work));
#pragma unroll
    for (int i = 0; i < 5; ++i) Fs[i] = add2(Fs[i], F[i]);
  }
}

// Nonlinear WENO5 end values of two columns at once, as six times their
// deviations from the centre averages (weno5_dev in recon.cuh, the same
// differences, candidates and weights in pair arithmetic; |beta0 - beta2| and
// the reciprocals per half).
template <int MODE>
HGKS_HD void weno5_dev_x2(float2 q0, float2 q1, float2 q2, float2 q3, float2 q4, float2& rL, float2& rR) {
  const float2 one = bc2(1.f), two = bc2(2.f);
  const float2 D1 = sub2(q1, q0), D2 = sub2(q2, q1), D3 = sub2(q3, q2), D4 = sub2(q4, q3);
  const float2 s0 = sub2(D2, D1), s1 = sub2(D3, D2), s2 = sub2(D4, D3);
  const float2 t0 = fma2(two, D2, s0), t1 = add2(D2, D3), t2 = sub2(add2(D3, D3), s2);
  const float2 w = add2(t0, D2), z = add2(t2, D3);
  const float2 c0 = add2(w, s0), c1 = add2(t1, D3), e0 = sub2(z, s2), e1 = add2(t1, D2);
  const float2 k = bc2(3.f / 13.f);
  const float2 b0 = fma2(mul2(k, t0), t0, mul2(s0, s0));
  const float2 b1 = fma2(mul2(k, t1), t1, mul2(s1, s1));
  const float2 b2 = fma2(mul2(k, t2), t2, mul2(s2, s2));
  float2 f0, f1, f2;
  if constexpr (MODE == RECON_WENO_JS) {
    const float2 e = bc2(12e-6f / 13.f);
    const float2 B0 = add2(b0, e), B1 = add2(b1, e), B2 = add2(b2, e);
    f0 = rcp2(mul2(B0, B0));
    f1 = rcp2(mul2(B1, B1));
    f2 = rcp2(mul2(B2, B2));
  } else {
    const float2 e = bc2(12e-20f / 13.f);
    const float2 d02 = sub2(b0, b2);
    const float2 tau5 = make_float2(fabsf(d02.x), fabsf(d02.y));
    f0 = fma2(tau5, rcp2(add2(b0, e)), one);
    f1 = fma2(tau5, rcp2(add2(b1, e)), one);
    f2 = fma2(tau5, rcp2(add2(b2, e)), one);
  }
  const float2 g0 = mul2(bc2(3.f), f0), g1 = mul2(bc2(6.f), f1), g2 = mul2(bc2(3.f), f2);
  const float2 nR = fma2(f0, c0, fma2(g1, c1, mul2(g2, z))), SR = add2(add2(f0, g1), g2);
  const float2 nL = fma2(f2, e0, fma2(g1, e1, mul2(g0, w))), SL = add2(add2(f2, g1), g0);
  const float2 iL = rcp2(SL);
  rR = mul2(nR, rcp2(SR));
  rL = mul2(nL, make_float2(-iL.x, -iL.y));
}

// WENO5 end values with nonlinear weights (weno5_pair) of two columns at once.
template <int MODE>
HGKS_HD void weno5_pair_x2(float2 q0, float2 q1, float2 q2, float2 q3, float2 q4,
                                              float2& qL, float2& qR) {
  float2 rL, rR;
  weno5_dev_x2<MODE>(q0, q1, q2, q3, q4, rL, rR);
  const float2 c6 = bc2(1.f / 6.f);
  qR = fma2(rR, c6, q2);
  qL = fma2(rL, c6, q2);
}

// Tangential reconstruction with nonlinear weights (tangential, WENO modes)
// of two columns at once: values v[m] and derivatives d[m] at the two Gauss
// abscissae from the quadratic through the WENO5 end values and the average.
template <int MODE>
HGKS_HD void tangential_weno_x2(float2 f0, float2 f1, float2 f2, float2 f3, float2 f4,
                                                   float2 v[2], float2 d[2]) {
  float2 rL, rR;
  weno5_dev_x2<MODE>(f0, f1, f2, f3, f4, rL, rR);
  const float gs = 0.5f / 1.7320508075688772f, c6 = 1.f / 6.f;
  const float2 b = sub2(rR, rL), r = add2(rL, rR);
  v[0] = fma2(b, bc2(-gs * c6), f2);
  v[1] = fma2(b, bc2(gs * c6), f2);
  const float2 cs = mul2(r, bc2(gs)), b6 = mul2(b, bc2(c6));
  d[0] = sub2(b6, cs);
  d[1] = add2(b6, cs);
}

}  // namespace hgks
