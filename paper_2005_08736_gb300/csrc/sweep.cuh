// Pieces of the fused sweep kernels (sweep_tile.cuh, march.cuh, adjoint.cuh):
// launch arguments, tile geometry, face fields and the tangential passes.
#pragma once

#include "charvars.cuh"
#include "compat.cuh"
#include "kernels.cuh"
#include "packed.cuh"

#include <type_traits>

namespace hgks {

template <class T>
struct SweepArgs {
  const T* q;                  // padded state (deviation)
  T* __restrict__ fd;          // face fluxes [10][fbox]: F then dF, global frame
  const T* __restrict__ wn;    // widths along d (offset kGhost)
  const T* __restrict__ wt1;   // widths along t1
  const T* __restrict__ wt2;   // widths along t2
  const double* __restrict__ scal;
  GridDev g;
  int d;
  int chunk;
  int layers;
  int xt;  // d = x and q is the copy with x slowest ([5][x][z][y], k_pad)
  Gas<T> gas;
};

// The three sweeps of a stage in one launch: block b belongs to direction d
// with start[d] <= b < start[d + 1].  The sweeps are independent of each
// other, so one grid fills the chip on grids where one direction cannot
// (32^3: 8 tiles of k_sweep, 4 of k_march a direction) and has one tail
// instead of three.
template <class T>
struct SweepArgs3 {
  const T* q;          // padded state
  const T* qx;         // its copy with x slowest (or null: the x sweep reads q)
  T* fd[3];
  const T* w[3];
  const double* scal;
  GridDev g;
  int gx[3], gy[3], chunk[3], start[4];  // k_march: chunk is whether P and S are exchanged,
                                         // start counts rows
  int share;           // k_march: rows per block
  int layers[3];       // face layers to compute: n + 1, or n where face n is face 0
  Gas<T> gas;
};

// Arguments of direction d.
template <class T>
__device__ __forceinline__ SweepArgs<T> sweep_of(const SweepArgs3<T>& s, int d) {
  auto pick = [&](auto x0, auto x1, auto x2) { return d == 0 ? x0 : (d == 1 ? x1 : x2); };
  SweepArgs<T> a;
  a.d = d;
  a.xt = d == 0 && s.qx != nullptr;
  a.q = a.xt ? s.qx : s.q;
  a.fd = pick(s.fd[0], s.fd[1], s.fd[2]);
  a.wn = pick(s.w[0], s.w[1], s.w[2]);
  a.wt1 = pick(s.w[1], s.w[2], s.w[0]);
  a.wt2 = pick(s.w[2], s.w[0], s.w[1]);
  a.scal = s.scal;
  a.g = s.g;
  a.chunk = pick(s.chunk[0], s.chunk[1], s.chunk[2]);
  a.layers = pick(s.layers[0], s.layers[1], s.layers[2]);
  a.gas = s.gas;
  return a;
}

// Direction and block coordinates of block b, and its direction's arguments.
template <class T>
__device__ __forceinline__ SweepArgs<T> sweep_of_block(const SweepArgs3<T>& s, int b, int& bx, int& by, int& bz) {
  const int d = b >= s.start[2] ? 2 : (b >= s.start[1] ? 1 : 0);
  auto pick = [&](int x0, int x1, int x2) { return d == 0 ? x0 : (d == 1 ? x1 : x2); };
  const int gx = pick(s.gx[0], s.gx[1], s.gx[2]), gy = pick(s.gy[0], s.gy[1], s.gy[2]);
  const int r = b - pick(0, s.start[1], s.start[2]);
  bx = r % gx;
  by = (r / gx) % gy;
  bz = r / (gx * gy);
  return sweep_of(s, d);
}

template <int FLUX, int MODE = 0>
struct SweepLayout {
  static constexpr int NV = FLUX == FLUX_FULL ? 15 : 5;  // state field components
  static constexpr int QM = 2 * NV;                      // characteristic modes: Qm
  static constexpr int NFF = 2 * NV + (is_char_mode<MODE>() ? 5 : 0);  // + normal slopes (+ Qm)
  static constexpr int NT1 = 4 * NV + 2 * NV;            // t1 pass outputs
};

// tangential() with the sums and differences of the linear weights shared and
// their constants folded: 18 operations against 22 (11 against 12 for values
// only), which FP64 pays for one by one.
template <int MODE, class T>
__device__ __forceinline__ void tangential_fast(T f0, T f1, T f2, T f3, T f4, T v[2], T d[2]) {
  if constexpr (recon_of<MODE>() == RECON_LINEAR) {
    const T sq3 = T(1.7320508075688772);
    const T s13 = f1 + f3, s04 = f0 + f4, d04 = f0 - f4, d31 = f3 - f1;
    const T E = T(719) / T(720) * f2 + (s13 * (T(1) / T(1080)) - s04 * (T(1) / T(4320)));
    const T O = d04 * (sq3 * T(7) / T(432)) + d31 * (sq3 * T(25) / T(216));
    const T A = d04 * (T(1) / T(12)) + d31 * (T(2) / T(3));
    const T B = s13 * (sq3 * T(13) / T(54)) - (f2 * (sq3 * T(24) / T(54)) + s04 * (sq3 / T(54)));
    v[0] = E - O;
    v[1] = E + O;
    d[0] = A - B;
    d[1] = A + B;
  } else {
    tangential<MODE>(f0, f1, f2, f3, f4, v, d);
  }
}

// Tangential reconstruction of a 5-vector field (components at src + i*sc,
// face averages at offsets -2..2 times sr): values v and derivatives d at the
// two Gauss abscissae, in the characteristic variables of b (the projection
// of every average, the scalar reconstruction per characteristic component,
// the map back).
template <int MODE, class T>
__device__ __forceinline__ void tangential_char(const T* src, int sc, int sr, const CharBasis<T>& b,
                                                T v[2][5], T d[2][5]) {
  T w[5][5];
#pragma unroll
  for (int r = 0; r < 5; ++r) {
    T qv[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) qv[i] = src[i * sc + (r - 2) * sr];
    to_char(b, qv, w[r]);
  }
  T cv[2][5], cd[2][5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    T vv[2], dd[2];
    tangential<MODE>(w[0][i], w[1][i], w[2][i], w[3][i], w[4][i], vv, dd);
    cv[0][i] = vv[0];
    cv[1][i] = vv[1];
    cd[0][i] = dd[0];
    cd[1][i] = dd[1];
  }
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    from_char(b, cv[m], v[m]);
    from_char(b, cd[m], d[m]);
  }
}

// t2 pass of the state group s (fields 5s..5s+4 of the t1-pass output) at t1
// abscissa m1 for the face at at3: value, t2-derivative (per cell length),
// t1-derivative field and normal-slope field at both t2 abscissae.
template <class T, int MODE, int NV, int NH>
__device__ __forceinline__ void t2_group(const T* tb, int s, int m1, int at3, int st2,
                                         const CharBasis<T>& b, T val[2][5], T dt2[2][5],
                                         T dt1[2][5], T dn[2][5]) {
  const T* sv = tb + (4 * (5 * s) + m1) * NH + at3;
  const T* sdv = tb + (4 * (5 * s) + 2 + m1) * NH + at3;
  const T* ss = tb + (4 * NV + 2 * (5 * s) + m1) * NH + at3;
  if constexpr (is_char_mode<MODE>()) {
    T scratch[2][5];
    tangential_char<MODE>(sv, 4 * NH, st2, b, val, dt2);
    tangential_char<MODE>(sdv, 4 * NH, st2, b, dt1, scratch);
    tangential_char<MODE>(ss, 2 * NH, st2, b, dn, scratch);
  } else {
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const T* a = sv + 4 * i * NH;
      const T* c = sdv + 4 * i * NH;
      const T* e = ss + 2 * i * NH;
      T v[2], dd[2], vd[2], vs[2], unused[2];
      tangential_fast<MODE>(a[-2 * st2], a[-st2], a[0], a[st2], a[2 * st2], v, dd);
      tangential_fast<MODE>(c[-2 * st2], c[-st2], c[0], c[st2], c[2 * st2], vd, unused);
      tangential_fast<MODE>(e[-2 * st2], e[-st2], e[0], e[st2], e[2 * st2], vs, unused);
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        val[m][i] = v[m];
        dt2[m][i] = dd[m];
        dt1[m][i] = vd[m];
        dn[m][i] = vs[m];
      }
    }
  }
}

// Geometry of one sweep: normal axis d, transverse axes P (faster in memory)
// and S, and the first tangential axis t1 = d+1.
struct SweepAxes {
  int d, P, S;
  bool t1P;        // t1 is P (d = x, z) or S (d = y)
  long long sd;    // stride of the padded state along d
  int gv[5];       // global variable of each local-frame component
  bool xt;         // the state is the copy with x slowest (x sweep)
  // Padded index of cell (x, y, z) in the state the sweep reads.
  __device__ __forceinline__ long long index(const GridDev& g, int x, int y, int z) const {
    return xt ? ((long long)(x + kGhost) * g.p[2] + (z + kGhost)) * g.p[1] + (y + kGhost)
              : pad_index(g, x, y, z);
  }
};
__device__ __forceinline__ SweepAxes sweep_axes(int d, const GridDev& g, bool xt = false) {
  SweepAxes a;
  a.d = d;
  a.P = d == 0 ? 1 : 0;
  a.S = d == 2 ? 1 : 2;
  a.t1P = ((d + 1) % 3) == a.P;
  a.xt = xt && d == 0;
  a.sd = a.xt ? (long long)g.p[1] * g.p[2]
              : (d == 0 ? 1LL : (d == 1 ? (long long)g.p[0] : (long long)g.p[0] * g.p[1]));
#pragma unroll
  for (int i = 0; i < 5; ++i) a.gv[i] = global_var(d, i);
  return a;
}

// Face fields (conservative-variable reconstruction) of one face point from
// the six cells f-3..f+2 along the normal, qa[i][k] = variable i of cell
// f-3+k (local frame), and the widths hl, hr of cells f-1 and f: the WENO5
// end values, the normal slopes, the compatibility state Q0 and its normal
// slope, into ff[k * NH + h].
template <class T, int MODE, int FLUX, int NH>
HGKS_HD void face_fields_cells(const T qa[5][6], T hl, T hr, const Gas<T>& gas,
                                                  int h, T* ff) {
  const T rhl = T(1) / hl, rhr = T(1) / hr, r6 = T(1) / (T(6) * (hl + hr));
  T Ql[5], Qr[5], Dl[5], Dr[5], D0[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const T q0 = qa[i][0], q1 = qa[i][1], q2 = qa[i][2], q3 = qa[i][3], q4 = qa[i][4], q5 = qa[i][5];
    T Li, Ri, Lr, Rr;
    bool packed = false;
#if defined(__CUDA_ARCH__)
    if constexpr (std::is_same<T, float>::value && recon_of<MODE>() != RECON_LINEAR) {
      // Both cells' WENO5 pairs in the halves of packed FP32 pairs.
      float2 L2, R2;
      weno5_pair_x2<recon_of<MODE>()>(make_float2(q0, q1), make_float2(q1, q2), make_float2(q2, q3),
                                      make_float2(q3, q4), make_float2(q4, q5), L2, R2);
      Li = L2.x;
      Ri = R2.x;
      Lr = L2.y;
      Rr = R2.y;
      packed = true;
    }
#endif
    if (!packed) {
      weno5_pair<MODE>(q0, q1, q2, q3, q4, Li, Ri);
      weno5_pair<MODE>(q1, q2, q3, q4, q5, Lr, Rr);
    }
    Ql[i] = Ri;
    Qr[i] = Lr;
    Dl[i] = (T(4) * Ri + T(2) * Li - T(6) * q2) * rhl;
    Dr[i] = -(T(4) * Lr + T(2) * Rr - T(6) * q3) * rhr;
    D0[i] = (q1 - T(15) * q2 + T(15) * q3 - q4) * r6;
  }
  T Q0[5];
  compat_state(Ql, Qr, gas, Q0);
  if constexpr (FLUX == FLUX_SMOOTH) {
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      ff[i * NH + h] = Q0[i];
      ff[(5 + i) * NH + h] = D0[i];
    }
  } else {
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      ff[i * NH + h] = Ql[i];
      ff[(5 + i) * NH + h] = Qr[i];
      ff[(10 + i) * NH + h] = Q0[i];
      ff[(15 + i) * NH + h] = Dl[i];
      ff[(20 + i) * NH + h] = Dr[i];
      ff[(25 + i) * NH + h] = D0[i];
    }
  }
}

// Face fields of face layer f at transverse point (Pc, Sc) into ff[k * NH + h]:
// WENO5 end values of cells f-1 and f, their normal slopes, the compatibility
// state Q0 and its normal slope (local frame).  Smooth flux: fields Q0, dQ0/dn;
// full flux: Q_l, Q_r, Q0, dQ_l/dn, dQ_r/dn, dQ0/dn.
template <class T, int MODE, int FLUX, int NH>
__device__ __forceinline__ void face_fields_item(const T* __restrict__ q, const GridDev& g,
                                                 const SweepAxes& ax, const T* __restrict__ wn,
                                                 const Gas<T>& gas, int f, int Pc, int Sc, int h,
                                                 T* ff) {
  int c[3];
  c[ax.d] = f - 3;
  c[ax.P] = Pc;
  c[ax.S] = Sc;
  const long long cb = ax.index(g, c[0], c[1], c[2]);
  const long long sd = ax.sd;
  const T hl = wn[f - 1 + kGhost], hr = wn[f + kGhost];
  if constexpr (!is_char_mode<MODE>()) {
    T qa[5][6];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const T* qv = q + ax.gv[i] * g.P + cb;
#pragma unroll
      for (int k = 0; k < 6; ++k) qa[i][k] = __ldg(qv + k * sd);
    }
    face_fields_cells<T, MODE, FLUX, NH>(qa, hl, hr, gas, h, ff);
  } else {
    // Characteristic variables of Qm, the mean of the two cells beside the face.
    const T rhl = T(1) / hl, rhr = T(1) / hr, r6 = T(1) / (T(6) * (hl + hr));
    T Ql[5], Qr[5], Dl[5], Dr[5], D0[5];
    T qa[6][5], qm[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const T* qv = q + ax.gv[i] * g.P + cb;
#pragma unroll
      for (int k = 0; k < 6; ++k) qa[k][i] = __ldg(qv + k * sd);
      qm[i] = T(0.5) * (qa[2][i] + qa[3][i]);
    }
    const CharBasis<T> b = char_basis(qm, gas);
    T w[6][5];
#pragma unroll
    for (int k = 0; k < 6; ++k) to_char(b, qa[k], w[k]);
    T e[4][5];  // Q at x_{i+1/2} and x_{i-1/2} from cell i, at x_{i+1/2} and x_{i+3/2} from cell i+1
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      weno5_pair<MODE>(w[0][i], w[1][i], w[2][i], w[3][i], w[4][i], e[1][i], e[0][i]);
      weno5_pair<MODE>(w[1][i], w[2][i], w[3][i], w[4][i], w[5][i], e[2][i], e[3][i]);
    }
    T E[4][5];
#pragma unroll
    for (int k = 0; k < 4; ++k) from_char(b, e[k], E[k]);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      Ql[i] = E[0][i];
      Qr[i] = E[2][i];
      Dl[i] = (T(4) * E[0][i] + T(2) * E[1][i] - T(6) * qa[2][i]) * rhl;
      Dr[i] = -(T(4) * E[2][i] + T(2) * E[3][i] - T(6) * qa[3][i]) * rhr;
      D0[i] = (qa[1][i] - T(15) * qa[2][i] + T(15) * qa[3][i] - qa[4][i]) * r6;
      ff[(SweepLayout<FLUX, MODE>::QM + i) * NH + h] = qm[i];
    }
    T Q0[5];
    compat_state(Ql, Qr, gas, Q0);
    if constexpr (FLUX == FLUX_SMOOTH) {
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        ff[i * NH + h] = Q0[i];
        ff[(5 + i) * NH + h] = D0[i];
      }
    } else {
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        ff[i * NH + h] = Ql[i];
        ff[(5 + i) * NH + h] = Qr[i];
        ff[(10 + i) * NH + h] = Q0[i];
        ff[(15 + i) * NH + h] = Dl[i];
        ff[(20 + i) * NH + h] = Dr[i];
        ff[(25 + i) * NH + h] = D0[i];
      }
    }
  }
}

// One group of five fields of the t1 pass at point `at`: group g < NV/5 is
// state group g (values at both t1 abscissae and t1-derivatives), else the
// normal slopes of state group g - NV/5 (values only).
template <class T, int MODE, int NV, int NH>
HGKS_HD void t1_pass_group(const T* ff, T* tb, int at, int st1, int grp) {
  if (grp < NV / 5) {
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const int k = 5 * grp + i;
      const T* src = ff + k * NH + at;
      T v[2], dd[2];
      tangential<MODE>(src[-2 * st1], src[-st1], src[0], src[st1], src[2 * st1], v, dd);
      tb[(4 * k + 0) * NH + at] = v[0];
      tb[(4 * k + 1) * NH + at] = v[1];
      tb[(4 * k + 2) * NH + at] = dd[0];
      tb[(4 * k + 3) * NH + at] = dd[1];
    }
  } else {
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const int j = 5 * (grp - NV / 5) + i;  // state field whose normal slope this is
      const T* src = ff + (NV + j) * NH + at;
      T v[2];
      tangential_val<MODE>(src[-2 * st1], src[-st1], src[0], src[st1], src[2 * st1], v);
      tb[(4 * NV + 2 * j + 0) * NH + at] = v[0];
      tb[(4 * NV + 2 * j + 1) * NH + at] = v[1];
    }
  }
}

// t1_pass_group in FP32 with nonlinear weights: the five fields of the
// group two at a time in packed FP32 pairs (fields 0 and 1, 2 and 3), the
// fifth alone; the same outputs and layout.
template <int MODE, int NV, int NH>
__device__ __forceinline__ void t1_pass_group_wx2(const float* ff, float* tb, int at, int st1, int grp) {
  const bool state = grp < NV / 5;
  // first field of the group in ff
  const int kf = state ? 5 * grp : NV + 5 * (grp - NV / 5);
#pragma unroll
  for (int i = 0; i < 4; i += 2) {
    const float* sa = ff + (kf + i) * NH + at;
    const float* sb = sa + NH;
    float2 f[5], v[2], dd[2];
#pragma unroll
    for (int j = 0; j < 5; ++j) f[j] = make_float2(sa[(j - 2) * st1], sb[(j - 2) * st1]);
    tangential_weno_x2<MODE>(f[0], f[1], f[2], f[3], f[4], v, dd);
    if (state) {
      const int k = kf + i;
      tb[(4 * k + 0) * NH + at] = v[0].x;
      tb[(4 * k + 1) * NH + at] = v[1].x;
      tb[(4 * k + 2) * NH + at] = dd[0].x;
      tb[(4 * k + 3) * NH + at] = dd[1].x;
      tb[(4 * k + 4) * NH + at] = v[0].y;
      tb[(4 * k + 5) * NH + at] = v[1].y;
      tb[(4 * k + 6) * NH + at] = dd[0].y;
      tb[(4 * k + 7) * NH + at] = dd[1].y;
    } else {
      const int j = kf - NV + i;  // state field whose normal slope this is
      tb[(4 * NV + 2 * j + 0) * NH + at] = v[0].x;
      tb[(4 * NV + 2 * j + 1) * NH + at] = v[1].x;
      tb[(4 * NV + 2 * j + 2) * NH + at] = v[0].y;
      tb[(4 * NV + 2 * j + 3) * NH + at] = v[1].y;
    }
  }
  {
    const float* src = ff + (kf + 4) * NH + at;
    float v[2], dd[2];
    tangential<MODE>(src[-2 * st1], src[-st1], src[0], src[st1], src[2 * st1], v, dd);
    if (state) {
      const int k = kf + 4;
      tb[(4 * k + 0) * NH + at] = v[0];
      tb[(4 * k + 1) * NH + at] = v[1];
      tb[(4 * k + 2) * NH + at] = dd[0];
      tb[(4 * k + 3) * NH + at] = dd[1];
    } else {
      const int j = kf - NV + 4;
      tb[(4 * NV + 2 * j + 0) * NH + at] = v[0];
      tb[(4 * NV + 2 * j + 1) * NH + at] = v[1];
    }
  }
}

}  // namespace hgks
