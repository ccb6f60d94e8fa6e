// Host check of the FP64 nonlinear reconstructions and their transposes
// (csrc/recon.cuh, csrc/adjoint.cuh) over the whole range of data whose
// smoothness indicators FP64 can hold: seeded stencils times powers of ten,
// stencils with a constant part and stencils whose two ends differ by many
// orders of magnitude, against the candidates and weights written from the
// averages in long double (whose exponents do not overflow here), the
// transposes against directional derivatives of the same in dual numbers.
// Prints the largest relative differences of values and transposes.
// Test support: built and run by tests/test_weno_range.py; not part of the
// library.
#include <cmath>
#include <cstdio>
#include <random>

#include "adjoint.cuh"

using namespace hgks;

namespace {

typedef long double R;
struct D {
  R v, d;
};
D operator+(D a, D b) { return {a.v + b.v, a.d + b.d}; }
D operator-(D a, D b) { return {a.v - b.v, a.d - b.d}; }
D operator*(D a, D b) { return {a.v * b.v, a.v * b.d + a.d * b.v}; }
D operator/(D a, D b) { return {a.v / b.v, (a.d - a.v / b.v * b.d) / b.v}; }
D operator*(R a, D b) { return {a * b.v, a * b.d}; }
D absolute(D a) { return a.v > 0 ? a : (a.v < 0 ? D{-a.v, -a.d} : D{0, 0}); }

// End value of the centre cell: right for q in order, left for q reversed.
D end_value(int mode, const D q[5]) {
  const R s6 = R(1) / 6;
  const D p[3] = {s6 * (R(2) * q[0] - R(7) * q[1] + R(11) * q[2]), s6 * (R(5) * q[2] - q[1] + R(2) * q[3]),
                  s6 * (R(2) * q[2] + R(5) * q[3] - q[4])};
  const D s[3] = {q[0] - R(2) * q[1] + q[2], q[1] - R(2) * q[2] + q[3], q[2] - R(2) * q[3] + q[4]};
  const D t[3] = {q[0] - R(4) * q[1] + R(3) * q[2], q[1] - q[3], R(3) * q[2] - R(4) * q[3] + q[4]};
  const R lin[3] = {R(1) / 10, R(6) / 10, R(3) / 10};
  D b[3], num{0, 0}, den{0, 0};
  for (int k = 0; k < 3; ++k) b[k] = R(13) / 12 * (s[k] * s[k]) + R(1) / 4 * (t[k] * t[k]);
  const D tau = absolute(b[0] - b[2]);
  for (int k = 0; k < 3; ++k) {
    const D e = b[k] + D{mode == RECON_WENO_JS ? R(1e-6) : R(1e-20), 0};
    const D a = lin[k] * (mode == RECON_WENO_JS ? D{1, 0} / (e * e) : D{1, 0} + tau / e);
    num = num + a * p[k];
    den = den + a;
  }
  return num / den;
}

double worst[2] = {0.0, 0.0};
void record(int part, double got, R want, R scale) {
  const double e = double(std::fabs(R(got) - want) / scale);
  if (!(e <= worst[part])) worst[part] = std::isfinite(e) ? e : 1e30;
}

template <int MODE>
void check(const double q[5], double gL, double gR) {
  double L, Rt, cot[5] = {0, 0, 0, 0, 0};
  R scale = 0;
  for (int k = 0; k < 5; ++k) scale = std::fmax(scale, std::fabs(R(q[k])));
  weno5_pair<MODE>(q[0], q[1], q[2], q[3], q[4], L, Rt);
  weno5_pair_vjp<MODE>(q, gL, gR, cot);
  D r[5], l[5];
  R want[5], top = 1;
  for (int j = 0; j < 5; ++j) {
    for (int k = 0; k < 5; ++k) r[k] = l[4 - k] = {R(q[k]), R(k == j)};
    const D vr = end_value(MODE, r), vl = end_value(MODE, l);
    if (j == 0) {
      record(0, L, vl.v, scale);
      record(0, Rt, vr.v, scale);
    }
    want[j] = R(gL) * vl.d + R(gR) * vr.d;
    top = std::fmax(top, std::fabs(want[j]));
  }
  for (int j = 0; j < 5; ++j) record(1, cot[j], want[j], top);
}

}  // namespace

int main() {
  std::mt19937_64 rng(77);
  std::uniform_real_distribution<double> u(-1.0, 1.0);
  const double scales[] = {1e-3, 1.0, 1e10, 1e18, 1e20, 1e24, 1e26, 1e34, 1e38, 1e45, 1e60, 1e75, 1e100, 1e130, 1e152};
  for (int trial = 0; trial < 60; ++trial) {
    double b[5];
    for (int k = 0; k < 5; ++k) b[k] = u(rng);
    if (trial % 6 == 4) b[0] = b[1] = b[2];
    if (trial % 6 == 5) b[2] = b[3] = b[4];
    const double gL = u(rng), gR = u(rng);
    for (double s : scales) {
      double q[5], c[5];
      for (int k = 0; k < 5; ++k) {
        q[k] = s * b[k];
        c[k] = k == 4 ? s * b[k] : b[k];  // one end of another magnitude
      }
      check<RECON_WENO_JS>(q, gL, gR);
      check<RECON_WENO_Z>(q, gL, gR);
      if (s <= 1e18) {
        check<RECON_WENO_JS>(c, gL, gR);
        check<RECON_WENO_Z>(c, gL, gR);
      }
    }
  }
  std::printf("%.3e %.3e\n", worst[0], worst[1]);
  return 0;
}
