// Reverse-mode derivatives (vector-Jacobian products) of the fluxes at one
// Gauss point with respect to their input states, values q and slopes dq
// together, in one backward pass per part: the half-space parts of the full
// flux (flux_full_side), its equilibrium part (flux_full_eq), the full flux
// assembled from them with the collision time and the fit of Eq. (7)
// (flux_full_vjp), the smooth flux (flux_smooth_rev) and the sign moments of
// the compatibility state.  Every function is the transpose of the forward
// function it names, with the forward intermediates recomputed; the
// slopes enter each part linearly, through the same intermediates as the
// values, so their cotangents come out of the same pass.  No counterpart in
// the paper.
#pragma once

#include "dual.cuh"
#include "physics.cuh"

namespace hgks {

// Cotangents of the fields of Prim.
template <class T>
struct PrimBar {
  T rho, inv, U, V, W, dp, p, lam, theta;
};

template <class T>
HGKS_HD void prim_bar_zero(PrimBar<T>& b) {
  b.rho = b.inv = b.U = b.V = b.W = b.dp = b.p = b.lam = b.theta = T(0);
}

// prim_of transposed: b holds the cotangents of the fields of s = prim_of(q);
// adds the cotangent of q to qb.
template <class T>
HGKS_HD void prim_of_rev(const T q[5], const Prim<T>& s, const Gas<T>& g, PrimBar<T> b, T qb[5]) {
  // lam = 1/(2 theta)
  b.theta += b.lam * (-T(0.5) / (s.theta * s.theta));
  // theta = p inv
  b.p += b.theta * s.inv_rho;
  b.inv += b.theta * s.p;
  // p = p_r + dp
  b.dp += b.p;
  // dp = gm1 (q4 - (q1 U + q2 V + q3 W)/2)
  const T h = g.gm1 * b.dp;
  qb[4] += h;
  qb[1] += -T(0.5) * h * s.U;
  qb[2] += -T(0.5) * h * s.V;
  qb[3] += -T(0.5) * h * s.W;
  b.U += -T(0.5) * h * q[1];
  b.V += -T(0.5) * h * q[2];
  b.W += -T(0.5) * h * q[3];
  // U = q1 inv, V = q2 inv, W = q3 inv
  qb[1] += b.U * s.inv_rho;
  qb[2] += b.V * s.inv_rho;
  qb[3] += b.W * s.inv_rho;
  b.inv += b.U * q[1] + b.V * q[2] + b.W * q[3];
  // inv = 1/rho, rho = rho_r + q0
  b.rho += -b.inv * s.inv_rho * s.inv_rho;
  qb[0] += b.rho;
}

// euler_jvp<J> transposed in the state (dQ held fixed): out = J_J(Q) dQ;
// given ob adds to sb and Hb.
template <int J, class T>
HGKS_HD void euler_jvp_rev_state(const Prim<T>& s, T H, const T dQ[5], const Gas<T>& g,
                                 const T ob[5], PrimBar<T>& sb, T& Hb) {
  const T inv = s.inv_rho;
  const T U[3] = {s.U, s.V, s.W};
  T du[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) du[i] = (dQ[1 + i] - U[i] * dQ[0]) * inv;
  const T dp = g.gm1 * (dQ[4] - U[0] * dQ[1] - U[1] * dQ[2] - U[2] * dQ[3] +
                        T(0.5) * (U[0] * U[0] + U[1] * U[1] + U[2] * U[2]) * dQ[0]);
  const T mJ = s.rho * U[J];
  T Ub[3] = {T(0), T(0), T(0)}, dub[3] = {T(0), T(0), T(0)};
  T mJb = T(0), dpb = T(0);
  // out[1+i] = dQ[1+J] U_i + mJ du_i (+ dp for i = J)
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Ub[i] += ob[1 + i] * dQ[1 + J];
    mJb += ob[1 + i] * du[i];
    dub[i] += ob[1 + i] * mJ;
  }
  dpb += ob[1 + J];
  // out4 = du_J H + U_J (dQ4 + dp)
  dub[J] += ob[4] * H;
  Hb += ob[4] * du[J];
  Ub[J] += ob[4] * (dQ[4] + dp);
  dpb += ob[4] * U[J];
  // mJ = rho U_J
  sb.rho += mJb * U[J];
  Ub[J] += mJb * s.rho;
  // dp = gm1 (dQ4 - U.dQm + |U|^2/2 dQ0)
#pragma unroll
  for (int i = 0; i < 3; ++i) Ub[i] += dpb * g.gm1 * (U[i] * dQ[0] - dQ[1 + i]);
  // du_i = (dQ[1+i] - U_i dQ0) inv
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Ub[i] += -dub[i] * dQ[0] * inv;
    sb.inv += dub[i] * (dQ[1 + i] - U[i] * dQ[0]);
  }
  sb.U += Ub[0];
  sb.V += Ub[1];
  sb.W += Ub[2];
}

// gauss_recursion transposed (m[n+2] = U m[n+1] + (n+1) theta m[n]).
template <class T>
HGKS_HD void gauss_recursion_rev(const T* m, T U, T theta, T* mb, T& Ub, T& thb) {
#pragma unroll
  for (int n = 4; n >= 0; --n) {
    const T b = mb[n + 2];
    Ub += b * m[n + 1];
    mb[n + 1] += b * U;
    thb += b * T(n + 1) * m[n];
    mb[n] += b * T(n + 1) * theta;
  }
}

// euler_jvp<J> transposed in dQ (the state held fixed): adds J_J(Q)^T ob to dQb.
template <int J, class T>
HGKS_HD void euler_jvp_rev_dq(const Prim<T>& s, T H, const Gas<T>& g, const T ob[5], T dQb[5]) {
  const T inv = s.inv_rho;
  const T U[3] = {s.U, s.V, s.W};
  const T mJ = s.rho * U[J];
  T dub[3] = {T(0), T(0), T(0)};
  T dpb = T(0);
  dQb[1 + J] += ob[0];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    dQb[1 + J] += ob[1 + i] * U[i];
    dub[i] += ob[1 + i] * mJ;
  }
  dpb += ob[1 + J];
  dub[J] += ob[4] * H;
  dQb[4] += ob[4] * U[J];
  dpb += ob[4] * U[J];
  // dp = gm1 (dQ4 - U.dQm + |U|^2/2 dQ0)
  const T h = g.gm1 * dpb;
  dQb[4] += h;
#pragma unroll
  for (int k = 0; k < 3; ++k) dQb[1 + k] += -h * U[k];
  dQb[0] += h * T(0.5) * (U[0] * U[0] + U[1] * U[1] + U[2] * U[2]);
  // du_i = (dQ[1+i] - U_i dQ0) inv
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    dQb[1 + i] += dub[i] * inv;
    dQb[0] += -dub[i] * U[i] * inv;
  }
}

// Cotangents of the values q and slopes dq of the state of flux_full_side
// (side 0: u > 0, side 1: u < 0) as it enters the full flux through the
// fit weights w_k = Fq[k] (F) and dFq[k] (dF) of its three moment vectors V_k
// (flux_full_close), given the flux cotangents gF, gdF; added to cot.  The
// weights are dual numbers carrying d/dtau; returns the part's share of
// gF . dF/dtau + gdF . d(dF)/dtau.  The cotangent of its pressure (through
// tau) is applied by pressure_viscosity_rev.
//
// The transpose of flux_full_side line by line: in the frame of the
// tangential velocity, with the slopes as primitive derivatives and the seven
// distinct entries of each moment matrix (a prefix g marks a cotangent).  About
// 700 operations; forming the four full moment matrices forward and again
// backward took some 2800, in straight-line code that the instruction cache
// did not hold (0.9 fetch stalls per issue).  FP32 64^3 WENO-JS, one adjoint
// step: 7.89 -> 6.30 ms.
template <class T>
HGKS_HD T flux_full_side_rev(const PointState<T>& st, const Gas<T>& g, int side, const T gF[5],
                             const T gdF[5], const Dual<T> Fq[3], const Dual<T> dFq[3], PointState<T>& cot) {
  // ---- forward (flux_full_side) ----
  const Prim<T> s = prim_of(st.q, g);
  const T inv = s.inv_rho, th = s.theta, U = s.U, V = s.V, W = s.W;
  const T il = T(1) / th, il2 = il * il;
  const T hk3 = T(0.5) * (g.K + T(3));
  const T hv2 = T(0.5) * (V * V + W * W), hu2 = T(0.5) * U * U;
  T r[3], du[3][3], pi[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    r[d] = st.dq[d][0] * inv;
    du[d][0] = st.dq[d][1] * inv - U * r[d];
    du[d][1] = st.dq[d][2] * inv - V * r[d];
    du[d][2] = st.dq[d][3] * inv - W * r[d];
    pi[d] = g.gm1 * (st.dq[d][4] * inv - V * du[d][1] - W * du[d][2] - U * du[d][0] - (hv2 + hu2) * r[d]);
  }
  auto slope = [&](const T dr, const T* dv, const T dpi, T* c) {
    const T dth = dpi - th * dr;
    const T c1 = dv[0] * il;
    c[4] = dth * il2;
    c[3] = dv[2] * il;
    c[2] = dv[1] * il;
    c[1] = c1 - U * c[4];
    c[0] = dr - hk3 * (dth * il) - U * c1 + hu2 * c[4];
  };
  T a[3][5], A[5];
#pragma unroll
  for (int d = 0; d < 3; ++d) slope(r[d], du[d], pi[d], a[d]);
  const T div = du[0][0] + du[1][1] + du[2][2];
  const T rt = -(U * r[0] + V * r[1] + W * r[2] + div);
  T ut[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) ut[i] = -(U * du[0][i] + V * du[1][i] + W * du[2][i] + pi[i]);
  const T pt = -(U * pi[0] + V * pi[1] + W * pi[2] + g.gamma * th * div);
  slope(rt, ut, pt, A);
  const T R = tsqrt(th + th), iR = T(1) / R, x = U * iR;
  const T e = texp(-x * x) * T(0.28209479177387814) * R;  // exp(-x^2) / (2 sqrt(pi lam))
  const T sg = T(side == 0 ? 1 : -1);
  const T half = T(0.5) * (T(1) + sg * terf(x));
  T m[7];
  m[0] = s.rho * half;
  m[1] = U * m[0] + sg * (s.rho * e);
  gauss_recursion(m, U, th);
  const T c1 = (g.K + T(2)) * th, c2 = c1 * (c1 + T(2) * th);
  const T P1 = T(0.5) * (m[3] + c1 * m[1]), P2 = T(0.5) * (m[4] + c1 * m[2]), P3 = T(0.5) * (m[5] + c1 * m[3]);
  const T R1 = T(0.25) * (m[5] + T(2) * c1 * m[3] + c2 * m[1]);
  const T R2 = T(0.25) * (m[6] + T(2) * c1 * m[4] + c2 * m[2]);
  const T t1 = th * m[1], t2 = th * m[2];
  const T B1 = T(0.5) * (th * m[3] + (c1 + T(2) * th) * t1);
  T uA[5], ua[5], h[5];
  uA[0] = m[1] * A[0] + m[2] * A[1] + P1 * A[4];
  uA[1] = m[2] * A[0] + m[3] * A[1] + P2 * A[4];
  uA[2] = t1 * A[2];
  uA[3] = t1 * A[3];
  uA[4] = P1 * A[0] + P2 * A[1] + R1 * A[4];
#pragma unroll
  for (int i = 0; i < 5; ++i) h[i] = V * a[1][i] + W * a[2][i];
  const T cross = a[1][2] + a[2][3], ah = a[0][0] + h[1];
  ua[0] = m[2] * ah + m[3] * a[0][1] + P2 * a[0][4] + m[1] * h[0] + P1 * h[4] + t1 * cross;
  ua[1] = m[3] * ah + m[4] * a[0][1] + P3 * a[0][4] + m[2] * h[0] + P2 * h[4] + t2 * cross;
  ua[2] = t2 * (a[0][2] + a[1][1]) + t1 * (h[2] + a[1][0]) + B1 * a[1][4];
  ua[3] = t2 * (a[0][3] + a[2][1]) + t1 * (h[3] + a[2][0]) + B1 * a[2][4];
  ua[4] = P2 * ah + P3 * a[0][1] + R2 * a[0][4] + P1 * h[0] + R1 * h[4] + B1 * cross;

  // ---- backward ----
  // Back to the frame of the face: y = (x0, x1, x2 + V x0, x3 + W x0, x4 + V x2
  // + W x3 + hv2 x0) for V0 (x = (m1, m2, 0, 0, P1)), V1 (ua) and V2 (uA).
  T gU = T(0), gV, gW, ghv2, gth = T(0), phi;
  T w0[5], z[5], y[5];  // cotangents of the three x
  {
    const T GF[5] = {gF[0] + V * gF[2] + W * gF[3] + hv2 * gF[4], gF[1], gF[2] + V * gF[4], gF[3] + W * gF[4], gF[4]};
    const T GD[5] = {gdF[0] + V * gdF[2] + W * gdF[3] + hv2 * gdF[4], gdF[1], gdF[2] + V * gdF[4],
                     gdF[3] + W * gdF[4], gdF[4]};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      w0[i] = GF[i] * Fq[0].v + GD[i] * dFq[0].v;
      z[i] = GF[i] * Fq[1].v + GD[i] * dFq[1].v;
      y[i] = GF[i] * Fq[2].v + GD[i] * dFq[2].v;
    }
    auto dot = [](const T* p, const T* q) {
      return p[0] * q[0] + p[1] * q[1] + p[2] * q[2] + p[3] * q[3] + p[4] * q[4];
    };
    phi = Fq[0].d * (GF[0] * m[1] + GF[1] * m[2] + GF[4] * P1) + dFq[0].d * (GD[0] * m[1] + GD[1] * m[2] + GD[4] * P1) +
          Fq[1].d * dot(GF, ua) + dFq[1].d * dot(GD, ua) + Fq[2].d * dot(GF, uA) + dFq[2].d * dot(GD, uA);
    const T S0 = Fq[0].v * m[1] + Fq[1].v * ua[0] + Fq[2].v * uA[0];
    const T D0 = dFq[0].v * m[1] + dFq[1].v * ua[0] + dFq[2].v * uA[0];
    const T S2 = Fq[1].v * ua[2] + Fq[2].v * uA[2], D2 = dFq[1].v * ua[2] + dFq[2].v * uA[2];
    const T S3 = Fq[1].v * ua[3] + Fq[2].v * uA[3], D3 = dFq[1].v * ua[3] + dFq[2].v * uA[3];
    gV = gF[2] * S0 + gF[4] * S2 + gdF[2] * D0 + gdF[4] * D2;
    gW = gF[3] * S0 + gF[4] * S3 + gdF[3] * D0 + gdF[4] * D3;
    ghv2 = gF[4] * S0 + gdF[4] * D0;
  }
  // <u A psi'> and <u (a.u) psi'>
  T gA[5], ga[3][5];
  gA[0] = m[1] * y[0] + m[2] * y[1] + P1 * y[4];
  gA[1] = m[2] * y[0] + m[3] * y[1] + P2 * y[4];
  gA[2] = t1 * y[2];
  gA[3] = t1 * y[3];
  gA[4] = P1 * y[0] + P2 * y[1] + R1 * y[4];
  const T gh0 = m[1] * z[0] + m[2] * z[1] + P1 * z[4], gh1 = m[2] * z[0] + m[3] * z[1] + P2 * z[4];
  const T gh2 = t1 * z[2], gh3 = t1 * z[3], gh4 = P1 * z[0] + P2 * z[1] + R1 * z[4];
  const T gcross = t1 * z[0] + t2 * z[1] + B1 * z[4];
  ga[0][0] = gh1;
  ga[0][1] = m[3] * z[0] + m[4] * z[1] + P3 * z[4];
  ga[0][2] = t2 * z[2];
  ga[0][3] = t2 * z[3];
  ga[0][4] = P2 * z[0] + P3 * z[1] + R2 * z[4];
  ga[1][0] = V * gh0 + gh2;
  ga[1][1] = V * gh1 + t2 * z[2];
  ga[1][2] = V * gh2 + gcross;
  ga[1][3] = V * gh3;
  ga[1][4] = V * gh4 + B1 * z[2];
  ga[2][0] = W * gh0 + gh3;
  ga[2][1] = W * gh1 + t2 * z[3];
  ga[2][2] = W * gh2;
  ga[2][3] = W * gh3 + gcross;
  ga[2][4] = W * gh4 + B1 * z[3];
  gV += a[1][0] * gh0 + a[1][1] * gh1 + a[1][2] * gh2 + a[1][3] * gh3 + a[1][4] * gh4;
  gW += a[2][0] * gh0 + a[2][1] * gh1 + a[2][2] * gh2 + a[2][3] * gh3 + a[2][4] * gh4;
  T gm[7];
  gm[0] = T(0);
  gm[1] = w0[0] + y[0] * A[0] + z[0] * h[0];
  gm[2] = w0[1] + y[0] * A[1] + y[1] * A[0] + z[0] * ah + z[1] * h[0];
  gm[3] = y[1] * A[1] + z[0] * a[0][1] + z[1] * ah;
  gm[4] = z[1] * a[0][1];
  const T gP1 = w0[4] + y[0] * A[4] + y[4] * A[0] + z[0] * h[4] + z[4] * h[0];
  const T gP2 = y[1] * A[4] + y[4] * A[1] + z[0] * a[0][4] + z[1] * h[4] + z[4] * ah;
  const T gP3 = z[1] * a[0][4] + z[4] * a[0][1];
  const T gR1 = y[4] * A[4] + z[4] * h[4], gR2 = z[4] * a[0][4];
  const T gB1 = z[2] * a[1][4] + z[3] * a[2][4] + z[4] * cross;
  const T gt1 = y[2] * A[2] + y[3] * A[3] + z[0] * cross + z[2] * (h[2] + a[1][0]) + z[3] * (h[3] + a[2][0]) +
                T(0.5) * gB1 * (c1 + T(2) * th);
  const T gt2 = z[1] * cross + z[2] * (a[0][2] + a[1][1]) + z[3] * (a[0][3] + a[2][1]);
  // the moments, from the combinations down the recursion
  T gc1 = T(0.5) * (gB1 * t1 + gP1 * m[1] + gP2 * m[2] + gP3 * m[3] + gR1 * m[3] + gR2 * m[4]);
  const T gc2 = T(0.25) * (gR1 * m[1] + gR2 * m[2]);
  gm[1] += gt1 * th + T(0.5) * c1 * gP1 + T(0.25) * c2 * gR1;
  gm[2] += gt2 * th + T(0.5) * c1 * gP2 + T(0.25) * c2 * gR2;
  gm[3] += T(0.5) * (gB1 * th + gP1 + c1 * (gP3 + gR1));
  gm[4] += T(0.5) * (gP2 + c1 * gR2);
  gm[5] = T(0.5) * gP3 + T(0.25) * gR1;
  gm[6] = T(0.25) * gR2;
  gc1 += gc2 * T(2) * (c1 + th);
  gth += T(0.5) * gB1 * (m[3] + T(2) * t1) + gt1 * m[1] + gt2 * m[2] + T(2) * c1 * gc2 + (g.K + T(2)) * gc1;
  gauss_recursion_rev(m, U, th, gm, gU, gth);
  PrimBar<T> sb;
  prim_bar_zero(sb);
  {
    gU += gm[1] * m[0];
    gm[0] += gm[1] * U;
    sb.rho = sg * gm[1] * e + gm[0] * half;
    const T ge = sg * gm[1] * s.rho, eR = e * iR;          // d erf/dx / 4 = e / R
    const T gx = T(2) * (sg * gm[0] * s.rho * eR - ge * e * x);
    gU += gx * iR;
    gth += (ge * eR - gx * x * iR) * iR;
  }
  // the slopes
  T gr[3] = {T(0), T(0), T(0)}, gdu[3][3], gpi[3], gil = T(0), gil2 = T(0), ghu2 = T(0);
  auto slope_rev = [&](const T dr, const T* dv, const T dpi, const T* gc, T& gdr, T* gdv, T& gdpi) {
    const T dth = dpi - th * dr, c4 = dth * il2;
    const T gl = gc[1] - U * gc[0], g4 = gc[4] - U * gc[1] + hu2 * gc[0];
    gU -= gc[1] * c4 + gc[0] * (dv[0] * il);
    ghu2 += gc[0] * c4;
    const T gdth = g4 * il2 - gc[0] * (hk3 * il);
    gil += gl * dv[0] + gc[2] * dv[1] + gc[3] * dv[2] - gc[0] * (hk3 * dth);
    gil2 += g4 * dth;
    gdv[0] = gl * il;
    gdv[1] = gc[2] * il;
    gdv[2] = gc[3] * il;
    gdpi = gdth;
    gth -= gdth * dr;
    gdr = gc[0] - gdth * th;
  };
#pragma unroll
  for (int d = 0; d < 3; ++d) slope_rev(r[d], du[d], pi[d], ga[d], gr[d], gdu[d], gpi[d]);
  {
    T nr, nu[3], np;
    slope_rev(rt, ut, pt, gA, nr, nu, np);
    nr = -nr;
    np = -np;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      nu[i] = -nu[i];
      gpi[i] += nu[i];
      gdu[0][i] += nu[i] * U;
      gdu[1][i] += nu[i] * V;
      gdu[2][i] += nu[i] * W;
    }
    gU += nr * r[0] + nu[0] * du[0][0] + nu[1] * du[0][1] + nu[2] * du[0][2] + np * pi[0];
    gV += nr * r[1] + nu[0] * du[1][0] + nu[1] * du[1][1] + nu[2] * du[1][2] + np * pi[1];
    gW += nr * r[2] + nu[0] * du[2][0] + nu[1] * du[2][1] + nu[2] * du[2][2] + np * pi[2];
    gr[0] += nr * U;
    gr[1] += nr * V;
    gr[2] += nr * W;
    gpi[0] += np * U;
    gpi[1] += np * V;
    gpi[2] += np * W;
    const T gdiv = nr + np * (g.gamma * th);
    gth += np * (g.gamma * div);
    gdu[0][0] += gdiv;
    gdu[1][1] += gdiv;
    gdu[2][2] += gdiv;
  }
  // the primitive derivatives
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const T ge = g.gm1 * gpi[d];
    const T g0 = gdu[d][0] - U * ge, g1 = gdu[d][1] - V * ge, g2 = gdu[d][2] - W * ge;
    const T gr0 = gr[d] - (hv2 + hu2) * ge - U * g0 - V * g1 - W * g2;
    gU -= ge * du[d][0] + g0 * r[d];
    gV -= ge * du[d][1] + g1 * r[d];
    gW -= ge * du[d][2] + g2 * r[d];
    ghv2 -= ge * r[d];
    ghu2 -= ge * r[d];
    sb.inv += ge * st.dq[d][4] + g0 * st.dq[d][1] + g1 * st.dq[d][2] + g2 * st.dq[d][3] + gr0 * st.dq[d][0];
    cot.dq[d][0] += gr0 * inv;
    cot.dq[d][1] += g0 * inv;
    cot.dq[d][2] += g1 * inv;
    cot.dq[d][3] += g2 * inv;
    cot.dq[d][4] += ge * inv;
  }
  sb.U = gU + U * ghu2;
  sb.V = gV + V * ghv2;
  sb.W = gW + W * ghv2;
  sb.theta = gth - il2 * (gil + T(2) * il * gil2);
  prim_of_rev(st.q, s, g, sb, cot.q);
  return phi;
}

// ns_viscous_flux transposed in the state and the viscosity (dq held fixed):
// given Fvb adds to sb and mub.
template <class T>
HGKS_HD void ns_viscous_flux_rev(const Prim<T>& s, const T dq[3][5], const Gas<T>& g, T mu, T heat_scale,
                                 const T Fvb[5], PrimBar<T>& sb, T& mub) {
  const T inv = s.inv_rho;
  const T U[3] = {s.U, s.V, s.W};
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
  const T c2 = T(2) / (g.K + T(3));
  const T s00 = mu * (T(2) * du0[0] - c2 * divU);
  const T s01 = mu * (du0[1] + du10);
  const T s02 = mu * (du0[2] + du20);
  const T ch = heat_scale * T(0.5) * (g.K + T(5));
  T Ub[3] = {T(0), T(0), T(0)};
  // Fv = (0, -s00, -s01, -s02, -(s00 U0 + s01 U1 + s02 U2) - ch mu dT0)
  const T s00b = -Fvb[1] - Fvb[4] * U[0];
  const T s01b = -Fvb[2] - Fvb[4] * U[1];
  const T s02b = -Fvb[3] - Fvb[4] * U[2];
  Ub[0] += -Fvb[4] * s00;
  Ub[1] += -Fvb[4] * s01;
  Ub[2] += -Fvb[4] * s02;
  mub += -Fvb[4] * ch * dT0;
  const T dT0b = -Fvb[4] * ch * mu;
  mub += s00b * (T(2) * du0[0] - c2 * divU) + s01b * (du0[1] + du10) + s02b * (du0[2] + du20);
  T du0b[3] = {s00b * mu * T(2), s01b * mu, s02b * mu};
  const T du10b = s01b * mu, du20b = s02b * mu;
  const T divUb = -s00b * mu * c2;
  du0b[0] += divUb;
  const T du11b = divUb, du22b = divUb;
  // dT0 = (dp0 - theta dq00) inv
  const T dp0b = dT0b * inv;
  sb.theta += -dT0b * dq[0][0] * inv;
  sb.inv += dT0b * (dp0 - s.theta * dq[0][0]);
#pragma unroll
  for (int i = 0; i < 3; ++i) Ub[i] += dp0b * g.gm1 * (U[i] * dq[0][0] - dq[0][1 + i]);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Ub[i] += -du0b[i] * dq[0][0] * inv;
    sb.inv += du0b[i] * (dq[0][1 + i] - U[i] * dq[0][0]);
  }
  Ub[0] += -du10b * dq[1][0] * inv;
  sb.inv += du10b * (dq[1][1] - U[0] * dq[1][0]);
  Ub[1] += -du11b * dq[1][0] * inv;
  sb.inv += du11b * (dq[1][2] - U[1] * dq[1][0]);
  Ub[0] += -du20b * dq[2][0] * inv;
  sb.inv += du20b * (dq[2][1] - U[0] * dq[2][0]);
  Ub[2] += -du22b * dq[2][0] * inv;
  sb.inv += du22b * (dq[2][3] - U[2] * dq[2][0]);
  sb.U += Ub[0];
  sb.V += Ub[1];
  sb.W += Ub[2];
}

// euler_flux_dev transposed: E = (m, m U + dp, m V, m W, U (h_r + q4 + dp)),
// m = rho U; given gE adds to sb and qb.
template <class T>
HGKS_HD void euler_flux_dev_rev(const Prim<T>& s, const T q[5], const Gas<T>& g, const T gE[5],
                                PrimBar<T>& sb, T qb[5]) {
  const T m = s.rho * s.U;
  const T mb = gE[0] + gE[1] * s.U + gE[2] * s.V + gE[3] * s.W;
  sb.U += gE[1] * m + gE[4] * (g.h_r + q[4] + s.dp);
  sb.V += gE[2] * m;
  sb.W += gE[3] * m;
  sb.dp += gE[1] + gE[4] * s.U;
  qb[4] += gE[4] * s.U;
  sb.rho += mb * s.U;
  sb.U += mb * s.rho;
}

// sign_moments transposed (the half-space sign moments S of the
// compatibility state): given gS adds the cotangent of dq to qb.
template <class T>
HGKS_HD void sign_moments_rev(const T dq[5], const Gas<T>& g, const T gS[5], T qb[5]) {
  const Prim<T> s = prim_of(dq, g);
  const T sl = tsqrt(s.lam);
  const T x = sl * s.U;
  const T D0 = terf(x);
  const T ex = texp(-x * x);
  const T R = tsqrt(s.theta + s.theta);
  const T c = T(0.5641895835477563);  // 1/sqrt(pi)
  const T D1 = s.U * D0 + ex * c * R;
  const T D2 = s.U * D1 + s.theta * D0;
  const T G = s.V * s.V + s.W * s.W + (g.K + T(2)) * s.theta;
  PrimBar<T> sb;
  prim_bar_zero(sb);
  const T h = T(0.5) * gS[4];
  sb.rho += gS[0] * D0 + gS[1] * D1 + gS[2] * s.V * D0 + gS[3] * s.W * D0 + h * (D2 + D0 * G);
  T D0b = gS[0] * s.rho + gS[2] * s.rho * s.V + gS[3] * s.rho * s.W + h * s.rho * G;
  T D1b = gS[1] * s.rho;
  const T D2b = h * s.rho;
  sb.V += gS[2] * s.rho * D0 + h * s.rho * D0 * T(2) * s.V;
  sb.W += gS[3] * s.rho * D0 + h * s.rho * D0 * T(2) * s.W;
  sb.theta += h * s.rho * D0 * (g.K + T(2));
  // D2 = U D1 + theta D0
  sb.U += D2b * D1;
  D1b += D2b * s.U;
  sb.theta += D2b * D0;
  D0b += D2b * s.theta;
  // D1 = U D0 + exp(-x^2) R / sqrt(pi), R = sqrt(2 theta)
  sb.U += D1b * D0;
  D0b += D1b * s.U;
  const T exb = D1b * c * R;
  sb.theta += D1b * ex * c / R;
  // ex = exp(-x^2), D0 = erf(x), x = sqrt(lam) U
  const T xb = exb * ex * (-T(2) * x) + D0b * T(2) * c * ex;
  sb.U += xb * sl;
  sb.lam += xb * s.U * T(0.5) / sl;
  prim_of_rev(dq, s, g, sb, qb);
}

// c0 += cotangent of dq along n from tb, the cotangent of the temperature
// slope dT0 = (dp0 - theta dq[0])/rho, dp0 = (gamma-1)(dq[4] - U.dm + |U|^2/2 dq[0]).
template <class T>
HGKS_HD void temperature_slope_vjp(const Prim<T>& s, const Gas<T>& g, T tb, T c0[5]) {
  const T inv = s.inv_rho;
  const T dpb = tb * inv * g.gm1;
  const T q2 = s.U * s.U + s.V * s.V + s.W * s.W;
  c0[0] += -s.theta * tb * inv + T(0.5) * q2 * dpb;
  c0[1] -= s.U * dpb;
  c0[2] -= s.V * dpb;
  c0[3] -= s.W * dpb;
  c0[4] += dpb;
}

// cd += (d Fv / d dq)^T w for ns_viscous_flux (linear in dq).
template <class T>
HGKS_HD void ns_viscous_vjp(const Prim<T>& s, const Gas<T>& g, T mu, T heat_scale, const T w[5],
                           T cd[3][5]) {
  const T inv = s.inv_rho;
  const T U[3] = {s.U, s.V, s.W};
  const T s00 = -w[1] - w[4] * U[0], s01 = -w[2] - w[4] * U[1], s02 = -w[3] - w[4] * U[2];
  const T divb = -mu * T(2) / (g.K + T(3)) * s00;
  const T du0b[3] = {T(2) * mu * s00 + divb, mu * s01, mu * s02};
  const T du10 = mu * s01, du20 = mu * s02, du11 = divb, du22 = divb;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    cd[0][1 + i] += du0b[i] * inv;
    cd[0][0] -= U[i] * du0b[i] * inv;
  }
  cd[1][1] += du10 * inv;
  cd[1][2] += du11 * inv;
  cd[1][0] -= (U[0] * du10 + U[1] * du11) * inv;
  cd[2][1] += du20 * inv;
  cd[2][3] += du22 * inv;
  cd[2][0] -= (U[0] * du20 + U[2] * du22) * inv;
  temperature_slope_vjp(s, g, -w[4] * heat_scale * mu * T(0.5) * (g.K + T(5)), cd[0]);
}

// Cotangents of the values q and slopes dq of the state of the smooth flux
// (flux_smooth) given the cotangents gF of F (if want_F) and gdF of dF;
// added to cot.
template <class T>
HGKS_HD void flux_smooth_rev(const PointState<T>& st0, const Gas<T>& g, bool want_F, const T gF[5],
                             const T gdF[5], PointState<T>& cot) {
  const T* q = st0.q;
  const Prim<T> s = prim_of(q, g);
  const T H = g.h_r + q[4] + s.dp;
  T Qt[5];
  state_time_derivative(s, H, st0.dq, g, Qt);
  PrimBar<T> sb;
  prim_bar_zero(sb);
  T Hb = T(0);
  // dF = J_n(Q) Q_t, Q_t = -(J_0 dq_0 + J_1 dq_1 + J_2 dq_2)
  euler_jvp_rev_state<0>(s, H, Qt, g, gdF, sb, Hb);
  T Qtb[5] = {0, 0, 0, 0, 0};
  euler_jvp_rev_dq<0>(s, H, g, gdF, Qtb);
  T nQtb[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) nQtb[i] = -Qtb[i];
  euler_jvp_rev_state<0>(s, H, st0.dq[0], g, nQtb, sb, Hb);
  euler_jvp_rev_state<1>(s, H, st0.dq[1], g, nQtb, sb, Hb);
  euler_jvp_rev_state<2>(s, H, st0.dq[2], g, nQtb, sb, Hb);
  euler_jvp_rev_dq<0>(s, H, g, nQtb, cot.dq[0]);
  euler_jvp_rev_dq<1>(s, H, g, nQtb, cot.dq[1]);
  euler_jvp_rev_dq<2>(s, H, g, nQtb, cot.dq[2]);
  if (want_F) {
    // F = Euler flux + viscous flux (mu = viscosity(s), heat flux scaled by 1/Pr)
    euler_flux_dev_rev(s, q, g, gF, sb, cot.q);
    const T mu = viscosity(s, g);
    T mub = T(0);
    ns_viscous_flux_rev(s, st0.dq, g, mu, g.pr_fix + T(1), gF, sb, mub);
    if (g.visc_law == 1) sb.theta += mub * mu * g.visc_exp / s.theta;
    ns_viscous_vjp(s, g, mu, g.pr_fix + T(1), gF, cot.dq);
  }
  cot.q[4] += Hb;
  sb.dp += Hb;
  prim_of_rev(q, s, g, sb, cot.q);
}

// Cotangents of the values q and slopes dq of the equilibrium state of
// flux_full_eq as it enters the full flux (flux_full_close): its three
// moment vectors V_k with the fit weights Fq[k] (F) and dFq[k] (dF), dual
// numbers carrying d/dtau, and the Prandtl fix -wpr tau p0 dT0 of F[4]
// (wpr = gF[4] pr_fix c_p), given the flux cotangents gF, gdF and the
// collision time tau; added to cot.  Returns the part's share of
// gF . dF/dtau + gdF . d(dF)/dtau.  The cotangents of mu0 and p0 through tau
// are applied by pressure_viscosity_rev.
template <class T>
HGKS_HD T flux_full_eq_rev(const PointState<T>& st0, const Gas<T>& g, const T gF[5], const T gdF[5],
                           const Dual<T> Fq[3], const Dual<T> dFq[3], T wpr, T tau, PointState<T>& cot) {
  const T* q = st0.q;
  const T* d0 = st0.dq[0];
  const Prim<T> s = prim_of(q, g);
  const T H = g.h_r + q[4] + s.dp;
  T Qt[5];
  state_time_derivative(s, H, st0.dq, g, Qt);
  // forward: V0 = Euler flux, V2 = J_n Q_t, V1 = -Fv(mu = p, Pr = 1) - V2, dT0
  T V0[5], V2[5], Fv[5];
  euler_flux_dev(s, q, g, V0);
  euler_jvp<0>(s, H, Qt, g, V2);
  ns_viscous_flux(s, st0.dq, g, s.p, T(1), Fv);
  const T q2 = s.U * s.U + s.V * s.V + s.W * s.W;
  const T dp0 = g.gm1 * (d0[4] - s.U * d0[1] - s.V * d0[2] - s.W * d0[3] + T(0.5) * q2 * d0[0]);
  const T dT = (dp0 - s.theta * d0[0]) * s.inv_rho;
  T phi = -wpr * s.p * dT;
  T gV0[5], Fvb[5], V2b[5];  // cotangents of V0, of Fv and of V2 (V1 = -Fv - V2)
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const T gt0 = gF[i] * Fq[0].d + gdF[i] * dFq[0].d, gt1 = gF[i] * Fq[1].d + gdF[i] * dFq[1].d;
    const T gt2 = gF[i] * Fq[2].d + gdF[i] * dFq[2].d;
    phi += gt0 * V0[i] + gt1 * (-Fv[i] - V2[i]) + gt2 * V2[i];
    const T gv1 = gF[i] * Fq[1].v + gdF[i] * dFq[1].v, gv2 = gF[i] * Fq[2].v + gdF[i] * dFq[2].v;
    gV0[i] = gF[i] * Fq[0].v + gdF[i] * dFq[0].v;
    Fvb[i] = -gv1;
    V2b[i] = gv2 - gv1;
  }
  // backward; the Prandtl fix gives p0 and dT0 the cotangents -wpr tau dT0
  // and -wpr tau p0
  const T gdT = -wpr * tau * s.p;
  PrimBar<T> sb;
  prim_bar_zero(sb);
  T Hb = T(0);
  {
    const T dp0b = gdT * s.inv_rho;
    sb.theta += -gdT * d0[0] * s.inv_rho;
    sb.inv += gdT * (dp0 - s.theta * d0[0]);
    sb.U += dp0b * g.gm1 * (s.U * d0[0] - d0[1]);
    sb.V += dp0b * g.gm1 * (s.V * d0[0] - d0[2]);
    sb.W += dp0b * g.gm1 * (s.W * d0[0] - d0[3]);
    temperature_slope_vjp(s, g, gdT, cot.dq[0]);
  }
  sb.p += -wpr * tau * dT;
  T mub = T(0);
  ns_viscous_flux_rev(s, st0.dq, g, s.p, T(1), Fvb, sb, mub);
  sb.p += mub;
  ns_viscous_vjp(s, g, s.p, T(1), Fvb, cot.dq);
  euler_jvp_rev_state<0>(s, H, Qt, g, V2b, sb, Hb);
  T Qtb[5] = {0, 0, 0, 0, 0};
  euler_jvp_rev_dq<0>(s, H, g, V2b, Qtb);
  // Q_t = -(J_0 dq_0 + J_1 dq_1 + J_2 dq_2)
  T nQtb[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) nQtb[i] = -Qtb[i];
  euler_jvp_rev_state<0>(s, H, st0.dq[0], g, nQtb, sb, Hb);
  euler_jvp_rev_state<1>(s, H, st0.dq[1], g, nQtb, sb, Hb);
  euler_jvp_rev_state<2>(s, H, st0.dq[2], g, nQtb, sb, Hb);
  euler_jvp_rev_dq<0>(s, H, g, nQtb, cot.dq[0]);
  euler_jvp_rev_dq<1>(s, H, g, nQtb, cot.dq[1]);
  euler_jvp_rev_dq<2>(s, H, g, nQtb, cot.dq[2]);
  euler_flux_dev_rev(s, q, g, gV0, sb, cot.q);
  // H = h_r + q4 + dp
  cot.q[4] += Hb;
  sb.dp += Hb;
  prim_of_rev(q, s, g, sb, cot.q);
  return phi;
}

// Adds to qb the cotangent of the values q through the pressure (gp) and the
// viscosity (gmu) of their state.
template <class T>
HGKS_HD void pressure_viscosity_rev(const T q[5], const Gas<T>& g, T gp, T gmu, T qb[5]) {
  const Prim<T> s = prim_of(q, g);
  PrimBar<T> sb;
  prim_bar_zero(sb);
  sb.p += gp;
  if (g.visc_law == 1) sb.theta += gmu * viscosity(s, g) * g.visc_exp / s.theta;
  prim_of_rev(q, s, g, sb, qb);
}

// Cotangents of the three states (st[0] = l, st[1] = r, st[2] = the
// compatibility state; values and slopes) of the full flux (flux_full) given
// the cotangents gF of F and gdF of dF; added to cot.  The fit weights
// Fq_k, dFq_k of Eq. (7) are formed as dual numbers in tau; each part runs
// one reverse pass with the cotangents gF Fq_k + gdF dFq_k of its moment
// vectors and returns its share of phi = gF . dF/dtau + gdF . d(dF)/dtau;
// phi then reaches the states through tau = mu0/p0 + C |p_l - p_r|/(p_l +
// p_r) dt.
template <class T>
HGKS_HD void flux_full_vjp(const PointState<T>* st, const Gas<T>& g, T dt, const T gF[5], const T gdF[5],
                           PointState<T>* cot) {
  T mu0, p0, pl, pr;
  {
    const Prim<T> s0 = prim_of(st[2].q, g);
    mu0 = viscosity(s0, g);
    p0 = s0.p;
    pl = prim_of(st[0].q, g).p;
    pr = prim_of(st[1].q, g).p;
  }
  const T tau = collision_time_full(mu0, p0, pl, pr, g, dt);
  Dual<T> Fq[6], dFq[6];
  fit_coefficients(Dual<T>(tau, T(1)), Dual<T>(dt), Fq, dFq);
  const T wpr = gF[4] * g.pr_fix * (T(0.5) * (g.K + T(5)));
  T phi = flux_full_eq_rev(st[2], g, gF, gdF, Fq, dFq, wpr, tau, cot[2]);
  // V_3 is the half-space sum minus the reference Euler flux (p_r in component 1).
  phi -= (gF[1] * Fq[3].d + gdF[1] * dFq[3].d) * g.p_r;
  // One copy of the half-space code for both sides: the side's state in and
  // its cotangent out through selects.
#pragma unroll 1
  for (int side = 0; side < 2; ++side) {
    const PointState<T> x = side == 0 ? st[0] : st[1];
    PointState<T> c;
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      c.q[i] = T(0);
#pragma unroll
      for (int d = 0; d < 3; ++d) c.dq[d][i] = T(0);
    }
    phi += flux_full_side_rev(x, g, side, gF, gdF, Fq + 3, dFq + 3, c);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      if (side == 0) cot[0].q[i] += c.q[i];
      else cot[1].q[i] += c.q[i];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        if (side == 0) cot[0].dq[d][i] += c.dq[d][i];
        else cot[1].dq[d][i] += c.dq[d][i];
      }
    }
  }
  const Gas<Dual<T>> gd = dual_gas(g);
  const T dtau_dpl =
      collision_time_full(Dual<T>(mu0), Dual<T>(p0), Dual<T>(pl, T(1)), Dual<T>(pr), gd, Dual<T>(dt)).d;
  const T dtau_dpr =
      collision_time_full(Dual<T>(mu0), Dual<T>(p0), Dual<T>(pl), Dual<T>(pr, T(1)), gd, Dual<T>(dt)).d;
  pressure_viscosity_rev(st[2].q, g, -phi * mu0 / (p0 * p0), phi / p0, cot[2].q);
  pressure_viscosity_rev(st[0].q, g, phi * dtau_dpl, T(0), cot[0].q);
  pressure_viscosity_rev(st[1].q, g, phi * dtau_dpr, T(0), cot[1].q);
}

}  // namespace hgks
