// Reconstruction of the high-order gas-kinetic scheme (Cao, Pan & Xu,
// arXiv:2005.08736, Sec. 2.1, Remark 1), templated on the floating type T.
//
// Normal direction: fifth-order WENO values at both ends of a cell from the
// cell averages q_{i-2..i+2}; linear weights (smooth flows) or WENO-JS /
// WENO-Z nonlinear weights.  Tangential directions: from five face averages,
// values and derivatives at the two Gauss abscissae s = +-1/(2 sqrt 3) of the
// centre face (cell units) -- the quartic through the five averages for
// linear weights, the quadratic through the WENO end values and the average
// otherwise.
#pragma once

#include "physics.cuh"

#include <cstring>
#include <type_traits>

namespace hgks {

enum Recon { RECON_LINEAR = 0, RECON_WENO_JS = 1, RECON_WENO_Z = 2 };
enum FluxKind { FLUX_SMOOTH = 0, FLUX_FULL = 1 };

// Kernel template MODE: the Recon value, or Recon + 2 for the WENO modes
// applied to characteristic variables (charvars.cuh): 3 = WENO-JS, 4 = WENO-Z.
// The scalar reconstructions below see the underlying Recon.
template <int MODE> __host__ __device__ constexpr int recon_of() { return MODE >= 3 ? MODE - 2 : MODE; }
template <int MODE> __host__ __device__ constexpr bool is_char_mode() { return MODE >= 3; }

// The high word of a double, and the double with it replaced.
HGKS_HD int high_word(double x) {
#if defined(__CUDA_ARCH__)
  return __double2hiint(x);
#else
  long long b;
  std::memcpy(&b, &x, sizeof b);
  return int(b >> 32);
#endif
}
HGKS_HD double with_high_word(double x, int hi) {
#if defined(__CUDA_ARCH__)
  return __hiloint2double(hi, __double2loint(x));
#else
  long long b;
  std::memcpy(&b, &x, sizeof b);
  b = ((long long)hi << 32) | (b & 0xffffffffLL);
  std::memcpy(&x, &b, sizeof x);
  return x;
#endif
}

// Divides the FP64 smoothness indicators, positive, by the power of two that
// brings the largest to [1, 2); what would fall below 2^-240 stays there (its
// candidate has all the weight as it is).  The weights depend on the ratios
// alone, so their products then fit FP64 for any data whose squares do.  Ten
// integer operations on the exponents, none on the FP64 pipe that bounds the
// callers; a test with a branch instead cost 4 % of the whole step (FP64
// WENO-Z + full flux 64^3).  Returns the exponent field of that power.
HGKS_HD int normalise_indicators(double& B0, double& B1, double& B2) {
  const int h0 = high_word(B0), h1 = high_word(B1), h2 = high_word(B2), one = 1023 << 20, least = (1023 - 240) << 20;
  int e = h0 > h1 ? h0 : h1;
  e = ((e > h2 ? e : h2) & 0x7ff00000) - one;
  B0 = with_high_word(B0, h0 - e > least ? h0 - e : least);
  B1 = with_high_word(B1, h1 - e > least ? h1 - e : least);
  B2 = with_high_word(B2, h2 - e > least ? h2 - e : least);
  return e;
}

// Nonlinear WENO5 end values of the centre cell, as six times their
// deviation from its average: rL = 6 (q(x_{i-1/2}) - q2), rR = 6 (q(x_{i+1/2}) - q2).
// Candidate quadratics on {i-2,i-1,i}, {i-1,i,i+1}, {i,i+1,i+2} with optimal
// weights (1/10, 6/10, 3/10) for the right end; the left end uses the mirrored
// stencils, whose smoothness indicators are the same three in reverse order.
// WENO-JS: alpha = d/(1e-6 + beta)^2.  WENO-Z: alpha = d (1 + |beta0 - beta2|/(beta + 1e-20)).
//
// Everything is formed from the differences D_k = q_k - q_{k-1} and their
// differences s_k: the candidates' deviations then take one addition each
// and the indicators three operations (12/13 beta = s^2 + 3/13 t^2, the factor
// moved into the epsilons), 54 operations per tangential reconstruction
// against 81 from the averages themselves.  The kernels that call this spend
// most of their time here and are bound by instruction issue (FP32) or the
// FP64 pipe.
// Measured with the flux's primitive form (physics.cuh), GB300: WENO-JS +
// smooth flux FP32 100x83x77, two steps 2.88 -> 2.42 ms; WENO-Z + full flux
// FP32 256^3 83.5 -> 71.4 ms a step, FP64 64^3 127 -> 78 ms.
// FP64: a division costs as much as ten multiplications there, so the
// weights are multiplied through by the product of the denominators (WENO-Z:
// B0 B1 B2; WENO-JS: its square), which leaves one (WENO-Z) or two divisions
// of the five; normalise_indicators keeps the products in range.  FP32's range
// does not allow them.
template <int MODE, class T>
HGKS_HD void weno5_dev(T q0, T q1, T q2, T q3, T q4, T& rL, T& rR) {
  static_assert(MODE == RECON_WENO_JS || MODE == RECON_WENO_Z, "nonlinear weights");
  const T D1 = q1 - q0, D2 = q2 - q1, D3 = q3 - q2, D4 = q4 - q3;
  const T s0 = D2 - D1, s1 = D3 - D2, s2 = D4 - D3;
  const T t0 = T(2) * D2 + s0, t1 = D2 + D3, t2 = T(2) * D3 - s2;
  // candidates: right c0, c1, z (stencils 0, 1, 2); left -e0, -e1, -w (stencils 2, 1, 0)
  const T w = t0 + D2, z = t2 + D3;
  const T c0 = w + s0, c1 = t1 + D3, e0 = z - s2, e1 = t1 + D2;
  const T k = T(3) / T(13);
  const T b0 = k * t0 * t0 + s0 * s0;
  const T b1 = k * t1 * t1 + s1 * s1;
  const T b2 = k * t2 * t2 + s2 * s2;
  T f0, f1, f2;  // weight factors of beta0, beta1, beta2 (up to a common factor)
  if (MODE == RECON_WENO_JS) {
    const T e = T(12e-6 / 13);
    T B0 = b0 + e, B1 = b1 + e, B2 = b2 + e;
    if constexpr (std::is_same<T, double>::value) {
      normalise_indicators(B0, B1, B2);
      const T p12 = B1 * B2, p02 = B0 * B2, p01 = B0 * B1;
      f0 = p12 * p12;
      f1 = p02 * p02;
      f2 = p01 * p01;
    } else {
      f0 = T(1) / (B0 * B0);
      f1 = T(1) / (B1 * B1);
      f2 = T(1) / (B2 * B2);
    }
  } else {
    const T e = T(12e-20 / 13);
    T B0 = b0 + e, B1 = b1 + e, B2 = b2 + e;
    if constexpr (std::is_same<T, double>::value) {
      normalise_indicators(B0, B1, B2);
      const T tau5 = tabs(B0 - B2);
      f0 = (B0 + tau5) * (B1 * B2);
      f1 = (B1 + tau5) * (B0 * B2);
      f2 = (B2 + tau5) * (B0 * B1);
    } else {
      const T tau5 = tabs(b0 - b2);
      f0 = tau5 * (T(1) / B0) + T(1);
      f1 = tau5 * (T(1) / B1) + T(1);
      f2 = tau5 * (T(1) / B2) + T(1);
    }
  }
  const T g0 = T(3) * f0, g1 = T(6) * f1, g2 = T(3) * f2;
  const T nR = f0 * c0 + g1 * c1 + g2 * z, SR = f0 + g1 + g2;
  const T nL = f2 * e0 + g1 * e1 + g0 * w, SL = f2 + g1 + g0;
  if constexpr (std::is_same<T, double>::value && MODE == RECON_WENO_Z) {
    const T inv = T(1) / (SR * SL);
    rR = nR * (SL * inv);
    rL = -(nL * (SR * inv));
  } else {
    rR = nR * (T(1) / SR);
    rL = -(nL * (T(1) / SL));
  }
}

// Both end values of the centre cell: qL at x_{i-1/2}, qR at x_{i+1/2}.
template <int MODE_, class T>
HGKS_HD void weno5_pair(T q0, T q1, T q2, T q3, T q4, T& qL, T& qR) {
  constexpr int MODE = recon_of<MODE_>();
  if constexpr (MODE == RECON_LINEAR) {
    // The optimal-weight combination of the three candidates is the
    // fifth-degree reconstruction (2, -13, 47, 27, -3)/60 of the five averages.
    const T c60 = T(1) / T(60);
    qR = (T(2) * q0 - T(13) * q1 + T(47) * q2 + T(27) * q3 - T(3) * q4) * c60;
    qL = (T(2) * q4 - T(13) * q3 + T(47) * q2 + T(27) * q1 - T(3) * q0) * c60;
  } else {
    T rL, rR;
    weno5_dev<MODE>(q0, q1, q2, q3, q4, rL, rR);
    const T c6 = T(1) / T(6);
    qR = rR * c6 + q2;
    qL = rL * c6 + q2;
  }
}

// Tangential reconstruction: values v[m] and derivatives d[m] (per unit of
// cell length) at s_0 = -1/(2 sqrt 3), s_1 = +1/(2 sqrt 3).
// Linear weights: the quartic with the five averages, written as
//   P(+-g)  = E +- O,  E = 719/720 f2 + (f1+f3)/1080 - (f0+f4)/4320,
//                      O = sqrt3 (7/432 (f0-f4) + 25/216 (f3-f1)),
//   P'(+-g) = A +- B,  A = (f0-f4)/12 + 2(f3-f1)/3,
//                      B = sqrt3/54 (-f0 + 13 f1 - 24 f2 + 13 f3 - f4).
// WENO modes: p(s) = a + b s + c s^2 with b = qR - qL, c = 3(qL+qR) - 6 f2,
// a = f2 - c/12, so p(+-g) = f2 +- b g and p'(+-g) = b +- 2 c g.
template <int MODE_, class T>
HGKS_HD void tangential(T f0, T f1, T f2, T f3, T f4, T v[2], T d[2]) {
  constexpr int MODE = recon_of<MODE_>();
  const T sq3 = T(1.7320508075688772);
  if constexpr (MODE == RECON_LINEAR) {
    const T E = T(719) / T(720) * f2 + (f1 + f3) * (T(1) / T(1080)) - (f0 + f4) * (T(1) / T(4320));
    const T O = sq3 * (T(7) / T(432) * (f0 - f4) + T(25) / T(216) * (f3 - f1));
    const T A = (f0 - f4) * (T(1) / T(12)) + T(2) / T(3) * (f3 - f1);
    const T B = sq3 / T(54) * (-f0 + T(13) * f1 - T(24) * f2 + T(13) * f3 - f4);
    v[0] = E - O;
    v[1] = E + O;
    d[0] = A - B;
    d[1] = A + B;
  } else {
    // b = (rR - rL)/6, c = (rL + rR)/2
    T rL, rR;
    weno5_dev<MODE>(f0, f1, f2, f3, f4, rL, rR);
    const T b = rR - rL, r = rL + rR;
    const T gs = T(0.5) / sq3, c6 = T(1) / T(6);
    v[0] = f2 - b * (gs * c6);
    v[1] = f2 + b * (gs * c6);
    const T cs = r * gs;
    d[0] = b * c6 - cs;
    d[1] = b * c6 + cs;
  }
}

// Values only (for fields whose tangential derivative is not needed).
template <int MODE, class T>
HGKS_HD void tangential_val(T f0, T f1, T f2, T f3, T f4, T v[2]) {
  T d[2];
  tangential<MODE>(f0, f1, f2, f3, f4, v, d);
}

}  // namespace hgks
