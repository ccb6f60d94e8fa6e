// Device arithmetic of the high-order gas-kinetic scheme (HGKS) of Cao, Pan &
// Xu (arXiv:2005.08736), templated on the floating type T (float or double).
//
// All conservative states handled here are DEVIATIONS from a reference state
// at rest, dQ = Q - Q_ref with Q_ref = (rho_r, 0, 0, 0, p_r/(gamma-1)).  Every
// quantity whose magnitude is set by the reference pressure (pressure,
// enthalpy flux, the Euler momentum flux) is formed from deviations, so that
// FP32 keeps the low-Mach variations instead of rounding them against p_r.
//
// Units: R = 1, p = rho T, lambda = rho / (2 p), theta = 1 / (2 lambda) = T.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

// The arithmetic below is compiled for the device and, where host code
// instantiates it (the operation tally of flopcount.cu), for the host.
#ifndef HGKS_HD
#define HGKS_HD __host__ __device__ __forceinline__
#endif

namespace hgks {

// Problem constants passed by value to every kernel.
template <class T>
struct Gas {
  T gamma, gm1;     // gamma, gamma - 1
  T K;              // internal degrees of freedom N = (5 - 3 gamma)/(gamma - 1), Sec. 2.1
  T pr_fix;         // 1/Pr - 1 (Prandtl fix of the energy flux)
  int visc_law;     // 0 constant, 1 power law
  T mu_ref, T_ref_inv, visc_exp;
  T tau_num_C;      // C of the numerical collision time, Sec. 3 opening
  T rho_r, p_r;     // reference state at rest
  T h_r;            // rho_r E_r + p_r = gamma/(gamma-1) p_r
};

template <class T> HGKS_HD T tsqrt(T x);
template <> HGKS_HD float tsqrt<float>(float x) { return sqrtf(x); }
template <> HGKS_HD double tsqrt<double>(double x) { return sqrt(x); }
template <class T> HGKS_HD T texp(T x);
template <> HGKS_HD float texp<float>(float x) { return expf(x); }
template <> HGKS_HD double texp<double>(double x) { return exp(x); }
template <class T> HGKS_HD T texpm1(T x);
template <> HGKS_HD float texpm1<float>(float x) { return expm1f(x); }
template <> HGKS_HD double texpm1<double>(double x) { return expm1(x); }
template <class T> HGKS_HD T terf(T x);
template <> HGKS_HD float terf<float>(float x) { return erff(x); }
template <> HGKS_HD double terf<double>(double x) { return erf(x); }
template <class T> HGKS_HD T tpow(T x, T y);
template <> HGKS_HD float tpow<float>(float x, float y) { return powf(x, y); }
template <> HGKS_HD double tpow<double>(double x, double y) { return pow(x, y); }
template <class T> HGKS_HD T tabs(T x) { return x < T(0) ? -x : x; }

template <class T>
struct Prim {
  T rho, inv_rho;  // density and its reciprocal
  T U, V, W;       // local-frame velocity
  T dp, p;         // pressure deviation and pressure
  T lam, theta;    // lambda = rho/(2p), theta = 1/(2 lambda)
};

// Primitive variables of the state Q_ref + dq (local frame).
template <class T>
HGKS_HD Prim<T> prim_of(const T dq[5], const Gas<T>& g) {
  Prim<T> s;
  s.rho = g.rho_r + dq[0];
  const T inv = T(1) / s.rho;
  s.inv_rho = inv;
  s.U = dq[1] * inv;
  s.V = dq[2] * inv;
  s.W = dq[3] * inv;
  // p - p_r = (gamma-1) (dE - |m|^2 / (2 rho)); the reference is at rest.
  s.dp = g.gm1 * (dq[4] - T(0.5) * (dq[1] * s.U + dq[2] * s.V + dq[3] * s.W));
  s.p = g.p_r + s.dp;
  s.theta = s.p * inv;
  s.lam = T(0.5) / s.theta;
  return s;
}

template <class T>
HGKS_HD void gauss_recursion(T* m, T U, T theta) {
  // <c^(n+2)> = U <c^(n+1)> + (n+1) theta <c^n>, on the line and on half lines.
#pragma unroll
  for (int n = 0; n < 5; ++n) m[n + 2] = U * m[n + 1] + T(n + 1) * theta * m[n];
}

// rho <u psi> - E(Q_ref): the Euler flux of the state minus that of the
// reference state (0, p_r, 0, 0, 0), formed from deviations.
template <class T>
HGKS_HD void euler_flux_dev(const Prim<T>& s, const T dq[5], const Gas<T>& g,
                                               T out[5]) {
  const T m = s.rho * s.U;
  out[0] = m;
  out[1] = m * s.U + s.dp;
  out[2] = m * s.V;
  out[3] = m * s.W;
  out[4] = s.U * (g.h_r + dq[4] + s.dp);
}

// One reconstructed state at a Gauss point: deviation value and derivatives
// along n, t1, t2 (local frame, physical units).
template <class T>
struct PointState {
  T q[5];
  T dq[3][5];
};

// Directional derivative of the Euler flux along local axis J at the state s
// (H = rho E + p) in the direction dQ: J_J(Q) dQ.
template <int J, class T>
HGKS_HD void euler_jvp(const Prim<T>& s, T H, const T dQ[5], const Gas<T>& g,
                                          T out[5]) {
  const T inv = s.inv_rho;
  const T U[3] = {s.U, s.V, s.W};
  const T du[3] = {(dQ[1] - U[0] * dQ[0]) * inv, (dQ[2] - U[1] * dQ[0]) * inv,
                   (dQ[3] - U[2] * dQ[0]) * inv};
  const T dp = g.gm1 * (dQ[4] - U[0] * dQ[1] - U[1] * dQ[2] - U[2] * dQ[3] +
                        T(0.5) * (U[0] * U[0] + U[1] * U[1] + U[2] * U[2]) * dQ[0]);
  const T mJ = s.rho * U[J];
  out[0] = dQ[1 + J];
#pragma unroll
  for (int i = 0; i < 3; ++i) out[1 + i] = dQ[1 + J] * U[i] + mJ * du[i];
  out[1 + J] += dp;
  out[4] = du[J] * H + U[J] * (dQ[4] + dp);
}

// Time derivative of the conservative state of the equilibrium,
// Q_t = rho <A psi> = -rho sum_d <(a_d.psi) u_d psi> = -sum_d J_d(Q) dQ/dx_d:
// each moment of (a.psi) g is the derivative of the Maxwellian's moment along
// the parameter change that a encodes.
template <class T>
HGKS_HD void state_time_derivative(const Prim<T>& s, T H, const T dq[3][5],
                                                      const Gas<T>& g, T Qt[5]) {
  T j0[5], j1[5], j2[5];
  euler_jvp<0>(s, H, dq[0], g, j0);
  euler_jvp<1>(s, H, dq[1], g, j1);
  euler_jvp<2>(s, H, dq[2], g, j2);
#pragma unroll
  for (int i = 0; i < 5; ++i) Qt[i] = -(j0[i] + j1[i] + j2[i]);
}

// Non-equilibrium flux of the smooth BGK solution, -tau rho (<u (a.u) psi> +
// <u A psi>), in its exact closed form: the Navier-Stokes viscous flux of the
// BGK model with mu = tau p, stress mu (grad U + grad U^T) - 2 mu/(K+3) div U I
// (bulk viscosity 2K/(3(K+3)) mu, Sec. 3.1), and heat flux -mu c_p dT/dn
// with c_p = (K+5)/2; `heat_scale` multiplies the heat flux (1/Pr for the
// Prandtl fix).
template <class T>
HGKS_HD void ns_viscous_flux(const Prim<T>& s, const T dq[3][5], const Gas<T>& g,
                                                T mu, T heat_scale, T Fv[5]) {
  const T inv = s.inv_rho;
  const T U[3] = {s.U, s.V, s.W};
  // du[j][i] = d u_i / d x_j (local frame) for the entries the normal row needs.
  T du0[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) du0[i] = (dq[0][1 + i] - U[i] * dq[0][0]) * inv;
  const T du10 = (dq[1][1] - U[0] * dq[1][0]) * inv, du11 = (dq[1][2] - U[1] * dq[1][0]) * inv;
  const T du20 = (dq[2][1] - U[0] * dq[2][0]) * inv, du22 = (dq[2][3] - U[2] * dq[2][0]) * inv;
  const T divU = du0[0] + du11 + du22;
  const T q2 = U[0] * U[0] + U[1] * U[1] + U[2] * U[2];
  const T dp0 = g.gm1 * (dq[0][4] - U[0] * dq[0][1] - U[1] * dq[0][2] - U[2] * dq[0][3] +
                         T(0.5) * q2 * dq[0][0]);
  const T dT0 = (dp0 - s.theta * dq[0][0]) * inv;
  const T s00 = mu * (T(2) * du0[0] - T(2) / (g.K + T(3)) * divU);
  const T s01 = mu * (du0[1] + du10);
  const T s02 = mu * (du0[2] + du20);
  Fv[0] = T(0);
  Fv[1] = -s00;
  Fv[2] = -s01;
  Fv[3] = -s02;
  Fv[4] = -(s00 * U[0] + s01 * U[1] + s02 * U[2]) - heat_scale * mu * T(0.5) * (g.K + T(5)) * dT0;
}

template <class T>
HGKS_HD T viscosity(const Prim<T>& s, const Gas<T>& g) {
  if (g.visc_law == 1) return g.mu_ref * tpow(s.theta * g.T_ref_inv, g.visc_exp);
  return g.mu_ref;
}

// The equilibrium state's derivatives in primitive variables: per direction
// d the velocity gradients du[d][i] and dp[d], and the Euler equations' time
// derivatives rt, ut[i], pt of density, velocity and pressure.  J_n Q_t then
// costs 15 operations and Q_t = -sum_d J_d dQ/dx_d is never formed in
// conservative variables (71 operations for both, 94 with three
// Jacobian-vector products and a fourth for J_n; the smooth flux is evaluated
// at four Gauss points of every face).  FP64 Taylor-Green 128^3, linear
// weights: 53.2 -> 49.8 ms a step.
template <class T>
struct PrimRates {
  T du[3][3], dp[3];
  T div;  // velocity divergence
  T rt, ut[3], pt;
  T hq2;  // |U|^2 / 2
};

template <class T>
HGKS_HD void prim_rates(const Prim<T>& s, const T dq[3][5], const Gas<T>& g, PrimRates<T>& r) {
  const T inv = s.inv_rho;
  const T U[3] = {s.U, s.V, s.W};
  r.hq2 = T(0.5) * (U[0] * U[0] + U[1] * U[1] + U[2] * U[2]);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int i = 0; i < 3; ++i) r.du[d][i] = (dq[d][1 + i] - U[i] * dq[d][0]) * inv;
    r.dp[d] = g.gm1 * (dq[d][4] - U[0] * dq[d][1] - U[1] * dq[d][2] - U[2] * dq[d][3] + r.hq2 * dq[d][0]);
  }
  r.div = r.du[0][0] + r.du[1][1] + r.du[2][2];
  r.rt = -(U[0] * dq[0][0] + U[1] * dq[1][0] + U[2] * dq[2][0] + s.rho * r.div);
#pragma unroll
  for (int i = 0; i < 3; ++i)
    r.ut[i] = -(U[0] * r.du[0][i] + U[1] * r.du[1][i] + U[2] * r.du[2][i] + r.dp[i] * inv);
  r.pt = -(U[0] * r.dp[0] + U[1] * r.dp[1] + U[2] * r.dp[2] + g.gamma * s.p * r.div);
}

// J_n(Q) Q_t, the time derivative of the Euler flux (H = rho E + p).
template <class T>
HGKS_HD void euler_flux_rate(const Prim<T>& s, T H, const PrimRates<T>& r, const Gas<T>& g, T out[5]) {
  const T mt = r.rt * s.U + s.rho * r.ut[0];
  const T m = s.rho * s.U;
  out[0] = mt;
  out[1] = mt * s.U + (m * r.ut[0] + r.pt);
  out[2] = mt * s.V + m * r.ut[1];
  out[3] = mt * s.W + m * r.ut[2];
  // (rho E + p)_t = gamma/(gamma-1) p_t + |U|^2/2 rho_t + rho U.U_t
  const T Ht = (g.gamma / g.gm1) * r.pt + r.hq2 * r.rt +
               s.rho * (s.U * r.ut[0] + s.V * r.ut[1] + s.W * r.ut[2]);
  out[4] = r.ut[0] * H + s.U * Ht;
}

// ns_viscous_flux from the primitive derivatives; dT0 is the normal
// temperature derivative (dp0 - theta drho0)/rho.
template <class T>
HGKS_HD void ns_viscous_rates(const Prim<T>& s, const PrimRates<T>& r, const Gas<T>& g, T mu, T heat_scale,
                              T dT0, T Fv[5]) {
  const T s00 = mu * (T(2) * r.du[0][0] - T(2) / (g.K + T(3)) * r.div);
  const T s01 = mu * (r.du[0][1] + r.du[1][0]);
  const T s02 = mu * (r.du[0][2] + r.du[2][0]);
  Fv[0] = T(0);
  Fv[1] = -s00;
  Fv[2] = -s01;
  Fv[3] = -s02;
  Fv[4] = -(s00 * s.U + s01 * s.V + s02 * s.W) - heat_scale * T(0.5) * (g.K + T(5)) * mu * dT0;
}

// Simplified smooth flux (Sec. 2.1, Remark 1): f = g0 [1 - tau (a.u + A) + t A],
// F = rho0 [<u psi> - tau (<u (a.u) psi> + <u A psi>)], dF = rho0 <u A psi>,
// with tau = mu/p (Sec. 3).  Evaluated through the exact identities
// rho0 <u psi> = Euler flux, -tau rho0 (<u(a.u)psi> + <u A psi>) = BGK
// Navier-Stokes viscous flux, rho0 <u A psi> = J_n(Q0) Q_t.  The Prandtl fix
// scales the heat flux by 1/Pr.  Returns F - E(Q_ref) and dF; want_F = false
// skips F (second S2O4 stage).
template <class T>
HGKS_HD void flux_smooth(const PointState<T>& st0, const Gas<T>& g, bool want_F,
                                            T F[5], T dF[5]) {
  const Prim<T> s = prim_of(st0.q, g);
  const T H = g.h_r + st0.q[4] + s.dp;
  PrimRates<T> r;
  prim_rates(s, st0.dq, g, r);
  euler_flux_rate(s, H, r, g, dF);
  if (!want_F) return;
  T E[5], Fv[5];
  euler_flux_dev(s, st0.q, g, E);
  const T dT0 = (r.dp[0] - s.theta * st0.dq[0][0]) * s.inv_rho;
  ns_viscous_rates(s, r, g, viscosity(s, g), g.pr_fix + T(1), dT0, Fv);
#pragma unroll
  for (int i = 0; i < 5; ++i) F[i] = E[i] + Fv[i];
}

// Coefficients of the linear fit F(t) = F + dF t (Eq. (7)) of the six
// time-integrated terms of Eq. (5), in closed form with y = 1 - exp(-dt/(2 tau)),
// r = tau/dt: term k contributes Fq[k] V_k to F and dFq[k] V_k to dF.
template <class T>
HGKS_HD void fit_coefficients(T tau, T dt, T Fq[6], T dFq[6]) {
  const T y = -texpm1(-dt / (T(2) * tau));
  const T eh = T(1) - y;
  const T r = tau / dt;
  const T S = y * (T(2) + y);  // 3 - 4 e^{-dt/2tau} + e^{-dt/tau}
  const T D = y * y;           // (1 - e^{-dt/2tau})^2
  Fq[0] = T(1) - r * S;
  Fq[3] = r * S;
  dFq[0] = T(4) * r * D / dt;
  dFq[3] = -dFq[0];
  Fq[1] = tau * (T(2) * r * S + D - T(2));
  Fq[4] = -tau - Fq[1];
  dFq[1] = T(4) * tau / dt * (eh * y - T(2) * r * D);
  dFq[4] = -dFq[1];
  Fq[2] = -tau * (T(1) - r * S);
  Fq[5] = -tau * r * S;
  dFq[2] = T(1) - T(4) * r * r * D;
  dFq[5] = T(4) * r * r * D;
}

// The full second-order flux (Eq. (5)) in parts, shared by the forward flux
// and its vector-Jacobian product:
//   equilibrium part (state 0): V0 = rho0 <u psi> - E(Q_ref) (Euler flux),
//     V2 = rho0 <u A psi> = J_n Q_t, V1 = rho0 <u (a.u) psi> =
//     -(viscous flux with mu = p, Pr = 1) - V2; mu0, p0 and the normal
//     temperature slope dT0 for tau and the Prandtl fix;
//   half-space part of side l (u > 0, g_l) or r (u < 0, g_r): rho <u psi>,
//     rho <u (a.psi) u_d psi>, rho <u A psi> over the half space, and p;
//   tau = mu0/p0 + C |p_l - p_r|/(p_l + p_r) dt (Sec. 3 opening);
//   the linear fit (Eq. (7)) F = sum_k Fq_k V_k, dF = sum_k dFq_k V_k, and
//   the Prandtl fix of the heat flux.
template <class T>
struct FullEq {
  T V[3][5];
  T mu, p, dT;
};
template <class T>
struct FullSide {
  T V[3][5];
  T p;
};

template <class T>
HGKS_HD void flux_full_eq(const PointState<T>& st0, const Gas<T>& g, FullEq<T>& o) {
  const Prim<T> s = prim_of(st0.q, g);
  const T H = g.h_r + st0.q[4] + s.dp;
  euler_flux_dev(s, st0.q, g, o.V[0]);
  PrimRates<T> r;
  prim_rates(s, st0.dq, g, r);
  euler_flux_rate(s, H, r, g, o.V[2]);
  // Normal temperature derivative, also for the Prandtl fix of the heat flux.
  o.dT = (r.dp[0] - s.theta * st0.dq[0][0]) * s.inv_rho;
  T Fv[5];
  ns_viscous_rates(s, r, g, s.p, T(1), o.dT, Fv);
#pragma unroll
  for (int i = 0; i < 5; ++i) o.V[1][i] = -Fv[i] - o.V[2][i];
  o.mu = viscosity(s, g);
  o.p = s.p;
}

// side = 0: g_l over u > 0; side = 1: g_r over u < 0.
//
// The moments are taken in the frame that moves with the state's tangential
// velocities V and W, where the odd moments of v' = v - V and w' = w - W
// vanish and <v'^2> = <w'^2> = theta: of the 15 entries of each moment matrix
// <u^k psi' psi'^T> seven remain (built from U_k = <u^k> alone), of
// <u v' psi' psi'^T> three.  The slopes go in as derivatives of the primitive
// variables per unit density (drho/rho, du_i, dp/rho): with d theta = dp/rho -
// theta drho/rho the slope coefficients are a4 = d theta/theta^2, a_i =
// du_i/theta, a0 = drho/rho - (K+3)/2 d theta/theta about the mean velocity,
// and the time coefficients A are the same form of the Euler equations' time
// derivatives.  The moment vectors go back to the frame of the face at the
// end.  About 235 fused operations, against 600 with full matrices in the
// frame of the face; the full flux evaluates this eight times per face.
// (Full flux in characteristic variables, FP32 90x75x67: 3.83 -> 2.94 ms a
// step together with weno5_dev, recon.cuh.)
template <class T>
HGKS_HD void flux_full_side(const PointState<T>& st, const Gas<T>& g, int side,
                                               FullSide<T>& o) {
  const Prim<T> s = prim_of(st.q, g);
  const T inv = s.inv_rho, th = s.theta, U = s.U, V = s.V, W = s.W;
  const T il = T(1) / th;
  const T hk3 = T(0.5) * (g.K + T(3));
  const T hv2 = T(0.5) * (V * V + W * W);
  // Primitive derivatives along n, t1, t2: r = drho/rho, du_i, pi = dp/rho.
  T r[3], du[3][3], pi[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    r[d] = st.dq[d][0] * inv;
    du[d][0] = st.dq[d][1] * inv - U * r[d];
    du[d][1] = st.dq[d][2] * inv - V * r[d];
    du[d][2] = st.dq[d][3] * inv - W * r[d];
    // internal energy per unit mass: (dE - u.dm + |u|^2/2 drho)/rho
    const T e = st.dq[d][4] * inv - V * du[d][1] - W * du[d][2] - U * du[d][0] - (hv2 + T(0.5) * U * U) * r[d];
    pi[d] = g.gm1 * e;
  }
  // a[d]: coefficients of 1, u, v', w', (u^2 + v'^2 + w'^2 + xi^2)/2.
  T a[3][5], A[5];
  const T il2 = il * il, hu2 = T(0.5) * U * U;
  auto slope = [&](const T dr, const T* dv, const T dpi, T* c) {
    const T dth = dpi - th * dr;
    const T c1 = dv[0] * il;
    c[4] = dth * il2;
    c[3] = dv[2] * il;
    c[2] = dv[1] * il;
    c[1] = c1 - U * c[4];
    c[0] = dr - hk3 * (dth * il) - U * c1 + hu2 * c[4];
  };
#pragma unroll
  for (int d = 0; d < 3; ++d) slope(r[d], du[d], pi[d], a[d]);
  {
    const T div = du[0][0] + du[1][1] + du[2][2];
    const T rt = -(U * r[0] + V * r[1] + W * r[2] + div);
    T ut[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) ut[i] = -(U * du[0][i] + V * du[1][i] + W * du[2][i] + pi[i]);
    const T pt = -(U * pi[0] + V * pi[1] + W * pi[2] + g.gamma * th * div);
    slope(rt, ut, pt, A);
  }
  // U_k = <u^k> over the half line, times rho.
  T m[7];
  {
    const T R = tsqrt(th + th);  // 1/sqrt(lam)
    const T x = U / R;
    const T e = texp(-x * x) * T(0.28209479177387814) * R;  // exp(-x^2) / (2 sqrt(pi lam))
    const T sg = T(side == 0 ? 1 : -1);
    m[0] = T(0.5) * s.rho * (T(1) + sg * terf(x));
    m[1] = U * m[0] + sg * (s.rho * e);
    gauss_recursion(m, U, th);
  }
  const T c1 = (g.K + T(2)) * th;           // <v'^2 + w'^2 + xi^2>
  const T c2 = c1 * (c1 + T(2) * th);       // <(v'^2 + w'^2 + xi^2)^2>
  const T P1 = T(0.5) * (m[3] + c1 * m[1]), P2 = T(0.5) * (m[4] + c1 * m[2]), P3 = T(0.5) * (m[5] + c1 * m[3]);
  const T R1 = T(0.25) * (m[5] + T(2) * c1 * m[3] + c2 * m[1]);
  const T R2 = T(0.25) * (m[6] + T(2) * c1 * m[4] + c2 * m[2]);
  const T t1 = th * m[1], t2 = th * m[2];
  const T B1 = T(0.5) * (th * m[3] + (c1 + T(2) * th) * t1);  // <u v'^2 psi4>
  // <u A psi'> and <u (a.u) psi'>: the u_t V and u_t W parts of a.u act
  // through <u psi' psi'^T> on V a_1 + W a_2.
  T uA[5], ua[5], h[5];
  uA[0] = m[1] * A[0] + m[2] * A[1] + P1 * A[4];
  uA[1] = m[2] * A[0] + m[3] * A[1] + P2 * A[4];
  uA[2] = t1 * A[2];
  uA[3] = t1 * A[3];
  uA[4] = P1 * A[0] + P2 * A[1] + R1 * A[4];
#pragma unroll
  for (int i = 0; i < 5; ++i) h[i] = V * a[1][i] + W * a[2][i];
  const T cross = a[1][2] + a[2][3];
  ua[0] = m[2] * a[0][0] + m[3] * a[0][1] + P2 * a[0][4] + m[1] * h[0] + m[2] * h[1] + P1 * h[4] + t1 * cross;
  ua[1] = m[3] * a[0][0] + m[4] * a[0][1] + P3 * a[0][4] + m[2] * h[0] + m[3] * h[1] + P2 * h[4] + t2 * cross;
  ua[2] = t2 * a[0][2] + t1 * (h[2] + a[1][0]) + t2 * a[1][1] + B1 * a[1][4];
  ua[3] = t2 * a[0][3] + t1 * (h[3] + a[2][0]) + t2 * a[2][1] + B1 * a[2][4];
  ua[4] = P2 * a[0][0] + P3 * a[0][1] + R2 * a[0][4] + P1 * h[0] + P2 * h[1] + R1 * h[4] + B1 * cross;
  // Back to the frame of the face.
  o.V[0][0] = m[1];
  o.V[0][1] = m[2];
  o.V[0][2] = V * m[1];
  o.V[0][3] = W * m[1];
  o.V[0][4] = P1 + hv2 * m[1];
  auto back = [&](const T* x, T* y) {
    y[0] = x[0];
    y[1] = x[1];
    y[2] = x[2] + V * x[0];
    y[3] = x[3] + W * x[0];
    y[4] = x[4] + V * x[2] + W * x[3] + hv2 * x[0];
  };
  back(ua, o.V[1]);
  back(uA, o.V[2]);
  o.p = s.p;
}

// |p_l - p_r| / (p_l + p_r)
template <class T>
HGKS_HD T pressure_jump(T pl, T pr) {
  return tabs((pl - pr) / (pl + pr));
}

template <class T>
HGKS_HD T collision_time_full(T mu0, T p0, T pl, T pr, const Gas<T>& g, T dt) {
  return mu0 / p0 + g.tau_num_C * pressure_jump(pl, pr) * dt;
}

// The parts of the full flux gathered for one Gauss point: the equilibrium
// part, the sum of the two half-space parts and the pressures of the l and r
// states (the full flux evaluated part by part, state by state).
template <class T>
struct FullParts {
  FullEq<T> e;
  T Vs[3][5];  // half-space parts, side l then + side r
  T pl, pr;
};

// Add the half-space part of side `side` (0: l, assigns; 1: r, adds) of the
// state st to the parts.
template <class T>
HGKS_HD void flux_full_add_side(const PointState<T>& st, const Gas<T>& g, int side, FullParts<T>& a) {
  FullSide<T> h;
  flux_full_side(st, g, side, h);
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 5; ++i) a.Vs[k][i] = side == 0 ? h.V[k][i] : a.Vs[k][i] + h.V[k][i];
  if (side == 0) a.pl = h.p; else a.pr = h.p;
}

// The full flux from its equilibrium part, the sums Vs of the half-space
// parts and the pressure jump: tau, the fit of Eq. (7), the Prandtl fix.
template <class T>
HGKS_HD void flux_full_close(const FullEq<T>& e, const T Vs[3][5], T jump, const Gas<T>& g, T dt, T F[5], T dF[5]) {
  const T tau = e.mu / e.p + g.tau_num_C * jump * dt;
  T Fq[6], dFq[6];
  fit_coefficients(tau, dt, Fq, dFq);
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    T f = T(0), df = T(0);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      // the half-space sum minus the reference Euler flux
      const T v = k < 3 ? e.V[k][i] : (k == 3 && i == 1 ? Vs[0][1] - g.p_r : Vs[k - 3][i]);
      f += Fq[k] * v;
      df += dFq[k] * v;
    }
    F[i] = f;
    dF[i] = df;
  }
  // Prandtl fix: (1/Pr - 1) times the heat flux -tau rho0 <h (a.u + A)> =
  // -tau p0 c_p dT/dn of the equilibrium part (tau includes the numerical term).
  F[4] -= g.pr_fix * tau * e.p * (T(0.5) * (g.K + T(5))) * e.dT;
}

// Full second-order flux (Eq. (5)) with the Heaviside factor H(u) on g_l and
// 1 - H(u) on g_r, integrated over [0, dt] and [0, dt/2] and fitted linearly
// (Eq. (7)).  Returns F - E(Q_ref) and dF.
template <class T>
HGKS_HD void flux_full(const PointState<T>& stl, const PointState<T>& str,
                                          const PointState<T>& st0, const Gas<T>& g, T dt,
                                          T F[5], T dF[5]) {
  FullParts<T> a;
  flux_full_eq(st0, g, a.e);
#pragma unroll 1  // one copy of the half-space code for both sides
  for (int side = 0; side < 2; ++side) flux_full_add_side(side == 0 ? stl : str, g, side, a);
  flux_full_close(a.e, a.Vs, pressure_jump(a.pl, a.pr), g, dt, F, dF);
}

// Equilibrium state of the compatibility condition, Q0 = int_{u>0} psi g_l +
// int_{u<0} psi g_r, as a deviation: Q0 - Q_ref = (dQl + dQr)/2 + (S_l - S_r)/2
// with S = int sign(u) psi g = rho (D0, D1, V D0, W D0, (D2 + D0 (V^2+W^2+(K+2) theta))/2),
// D0 = erf(sqrt(lam) U), D1 = U D0 + exp(-lam U^2)/sqrt(pi lam), D2 = U D1 + theta D0.
template <class T>
HGKS_HD void sign_moments(const T dq[5], const Gas<T>& g, T S[5]) {
  const Prim<T> s = prim_of(dq, g);
  const T R = tsqrt(s.theta + s.theta);  // 1/sqrt(lam)
  const T x = s.U / R;
  const T D0 = terf(x);
  const T D1 = s.U * D0 + texp(-x * x) * T(0.5641895835477563) * R;  // 1/sqrt(pi lam)
  const T D2 = s.U * D1 + s.theta * D0;
  S[0] = s.rho * D0;
  S[1] = s.rho * D1;
  S[2] = s.rho * s.V * D0;
  S[3] = s.rho * s.W * D0;
  S[4] = T(0.5) * s.rho * (D2 + D0 * (s.V * s.V + s.W * s.W + (g.K + T(2)) * s.theta));
}

template <class T>
HGKS_HD void compat_dev(const T dql[5], const T dqr[5], const Gas<T>& g,
                                           T dq0[5]) {
  T Sl[5], Sr[5];
  sign_moments(dql, g, Sl);
  sign_moments(dqr, g, Sr);
#pragma unroll
  for (int i = 0; i < 5; ++i) dq0[i] = T(0.5) * (dql[i] + dqr[i]) + T(0.5) * (Sl[i] - Sr[i]);
}

}  // namespace hgks
