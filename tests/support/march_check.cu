// Host check of the pair arithmetic of k_march against the scalar functions:
// tangential_linear_scaled_x2, tangential_linear_val_x2 and tangential_linear_x2
// against tangential, the compatibility state's midpoint rule compat_jump_x2
// (where it applies and where it must not) against the direct form in FP64,
// and face_fields_smooth_linear_x2 against face_fields_cells in FP64 -- smooth
// data, rough data and one of each in the two halves, which decide their rule
// together.  On the host a pair operation is the two scalar operations it
// stands for.  Prints the largest scaled differences of the three parts, and
// how many pairs took the rule, refused it and were of mixed kind.
// Test support: built and run by tests/test_march_pairs.py; not part of the
// library.
#include <cmath>
#include <cstdio>
#include <random>

#include "march.cuh"

using namespace hgks;

namespace {

std::mt19937_64 rng(31);
double uni(double a = -1.0, double b = 1.0) { return std::uniform_real_distribution<double>(a, b)(rng); }

double worst[3] = {0, 0, 0};
void record(int part, double got, double want, double scale) {
  const double e = std::fabs(got - want) / scale;
  if (!(e <= worst[part])) worst[part] = std::isfinite(e) ? e : 1e30;
}

template <class T>
Gas<T> gas() {
  Gas<T> g{};
  g.gamma = T(1.4);
  g.gm1 = T(0.4);
  g.K = T(2);
  g.pr_fix = T(1.0 / 0.72 - 1.0);
  g.mu_ref = T(1.0 / 1600);
  g.T_ref_inv = T(1);
  g.visc_exp = T(0.76);
  g.rho_r = T(1);
  g.p_r = T(100 / 1.4);
  g.h_r = T(1.4 / 0.4 * 100 / 1.4);
  return g;
}
// Sizes of the conservative variables: density, density times sound speed, pressure.
const double kSize[5] = {1.0, 10.0, 10.0, 10.0, 100 / 1.4};

void tangentials() {
  float2 f[5];
  float a[5], b[5], top = 0;
  for (int k = 0; k < 5; ++k) {
    f[k] = make_float2(a[k] = float(uni()), b[k] = float(uni()));
    top = std::fmax(top, std::fmax(std::fabs(a[k]), std::fabs(b[k])));
  }
  const float w = float(std::exp(uni(-3, 3)));
  float va[2], da[2], vb[2], db[2];
  tangential<RECON_LINEAR>(a[0], a[1], a[2], a[3], a[4], va, da);
  tangential<RECON_LINEAR>(b[0], b[1], b[2], b[3], b[4], vb, db);
  float2 v[2], d[2], u[2], x[2], y[2];
  tangential_linear_scaled_x2(f[0], f[1], f[2], f[3], f[4], DerivCoef(w), v, d);
  tangential_linear_val_x2(f[0], f[1], f[2], f[3], f[4], u);
  tangential_linear_x2(f[0], f[1], f[2], f[3], f[4], x, y);
  for (int m = 0; m < 2; ++m) {
    for (const float2 r : {v[m], u[m], x[m]}) {
      record(0, r.x, va[m], top);
      record(0, r.y, vb[m], top);
    }
    record(0, d[m].x * w, da[m], top);
    record(0, d[m].y * w, db[m], top);
    record(0, y[m].x, da[m], top);
    record(0, y[m].y, db[m], top);
  }
}

// A state near the reference and a jump of relative size r (compat.cuh's measure).
void state_and_jump(double r, float dm[5], float dd[5]) {
  const double rho = 1 + 0.1 * uni();
  const double u[3] = {uni(), uni(), uni()};
  const double p = 100 / 1.4 * (1 + 0.1 * uni());
  const double E = p / 0.4 + 0.5 * rho * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
  const double q[5] = {rho - 1, rho * u[0], rho * u[1], rho * u[2], E - 100 / 1.4 / 0.4};
  double j[5];
  for (int i = 0; i < 5; ++i) {
    dm[i] = float(q[i]);
    j[i] = uni() * kSize[i];
  }
  const double size = std::fabs(j[0]) / rho + (std::fabs(j[1]) + std::fabs(j[2]) + std::fabs(j[3])) / std::sqrt(rho * p) +
                      0.4 * std::fabs(j[4]) / p;
  for (int i = 0; i < 5; ++i) dd[i] = float(j[i] * r / size);
}

int taken = 0, refused = 0, mixed = 0;

void compat() {
  float dm[2][5], dd[2][5];
  const double r[2] = {std::exp(uni(std::log(1e-5), std::log(1e-1))), std::exp(uni(std::log(1e-5), std::log(1e-1)))};
  for (int h = 0; h < 2; ++h) state_and_jump(r[h], dm[h], dd[h]);
  float2 m[5], j[5], Q0[5];
  for (int i = 0; i < 5; ++i) {
    m[i] = make_float2(dm[0][i], dm[1][i]);
    j[i] = make_float2(dd[0][i], dd[1][i]);
  }
  const bool rule = compat_jump_x2(m, j, gas<float>(), Q0);
  bool small[2];
  for (int h = 0; h < 2; ++h) small[h] = compat_small_jump(dm[h], dd[h], gas<float>());
  if (std::fabs(r[0] / 2e-3 - 1) > 1e-4 && std::fabs(r[1] / 2e-3 - 1) > 1e-4 && rule != (small[0] && small[1]))
    worst[1] = 1e30;
  (rule ? taken : refused) += 1;
  if (!rule) return;
  for (int h = 0; h < 2; ++h) {
    double ql[5], qr[5], q0[5];
    for (int i = 0; i < 5; ++i) {
      ql[i] = double(dm[h][i]) + 0.5 * dd[h][i];
      qr[i] = double(dm[h][i]) - 0.5 * dd[h][i];
    }
    compat_dev(ql, qr, gas<double>(), q0);
    for (int i = 0; i < 5; ++i) record(1, h ? Q0[i].y : Q0[i].x, q0[i], kSize[i]);
  }
}

void face_fields(int kind) {  // bit h: half h is rough
  float2 q[5][6];
  double qd[2][5][6];
  for (int h = 0; h < 2; ++h) {
    float dm[5], dd[5];
    state_and_jump(1.0, dm, dd);
    const double noise = (kind >> h & 1) ? 0.1 : 2e-4;
    for (int i = 0; i < 5; ++i) {
      const double slope = 2e-3 * uni() * kSize[i];
      for (int k = 0; k < 6; ++k) {
        const float x = float(dm[i] + slope * k + noise * uni() * kSize[i]);
        qd[h][i][k] = x;
        if (h) q[i][k].y = x;
        else q[i][k].x = x;
      }
    }
  }
  const double hl[2] = {std::exp(uni()), std::exp(uni())}, hr[2] = {std::exp(uni()), std::exp(uni())};
  const float2 r6 = make_float2(float(1 / (6 * (hl[0] + hr[0]))), float(1 / (6 * (hl[1] + hr[1]))));
  float2 Q0[5], D0[5];
  face_fields_smooth_linear_x2(q, r6, gas<float>(), Q0, D0);
  for (int h = 0; h < 2; ++h) {
    double ff[10];
    face_fields_cells<double, RECON_LINEAR, FLUX_SMOOTH, 1>(qd[h], hl[h], hr[h], gas<double>(), 0, ff);
    for (int i = 0; i < 5; ++i) {
      record(2, h ? Q0[i].y : Q0[i].x, ff[i], kSize[i]);
      record(2, h ? D0[i].y : D0[i].x, ff[5 + i], kSize[i] * 30 * (h ? r6.y : r6.x));
    }
  }
  if (kind == 1 || kind == 2) ++mixed;
}

}  // namespace

int main() {
  for (int trial = 0; trial < 4000; ++trial) {
    tangentials();
    compat();
    face_fields(trial % 4);
  }
  std::printf("%.3e %.3e %.3e %d %d %d\n", worst[0], worst[1], worst[2], taken, refused, mixed);
  return 0;
}
