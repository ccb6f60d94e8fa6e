// Fused sweep kernel: for one S2O4 stage, the face fields, the tangential
// reconstruction to the 2x2 Gauss points and the BGK flux there, for a TP x TS
// tile of faces (P the faster-varying transverse axis in memory, S the slower
// one) marching through a chunk of face layers along the normal (face f lies
// between cells f-1 and f).  (FP32 with linear weights and the smooth flux:
// march.cuh.)
//
// Per face layer:
//   phase 1  one thread per point of the tile plus a halo of 2: the six cells
//            f-3..f+2 along d, WENO5 end values of cells f-1 and f, the normal
//            slopes, the compatibility state Q0 and its normal slope;
//   then for each STATE GROUP s of five fields and five slopes (smooth flux:
//   Q_0; full flux: Q_l, Q_r, Q_0 one after the other):
//   phase 2  the pass along t1 = d+1 (30 values per point, halo 2 along t2);
//   phase 3  two threads per face, thread m1 for the t1 abscissa m1: the pass
//            along t2 = d+2 gives both t2 abscissae; Q_l, Q_r add their
//            half-space moments to the Gauss points' sums, Q_0 closes the flux.
// A group's values of the second t2 abscissa and the half-space sums wait in
// the thread's own slots of shared memory.
//
// Why by groups: the full flux's three at once need 90 planes of t1-pass values
// and three point states in registers (FP32: 210 KB and 246 registers, 8 warps
// per SM, FMA pipe 54 % active).  One group needs 30 planes and one point
// state: 111 KB and 128 registers (16 bytes of spills at most), 16 warps per SM
// in two CTAs whose phases overlap.  In FP64 the tile grows from 8 x 8 to 16 x 8 (face
// fields at 1.9 points per face instead of 2.25), and every reconstruction of
// the pass along t2 serves both abscissae.
// Measured (GB300, one step): FP32 WENO-Z + full flux 256^3 73.4 -> 59.9 ms
// (56.3 with the strides as constants and shorter marches); in characteristic
// variables 90x75x67 2.59 -> 2.24 ms; eight boxes of 32^3 to 96^3 11.4 -> 8.92
// ms; FP64 WENO-Z + full flux 64^3 71.1 -> 46.0 ms.
// Bound by the FMA pipe and instruction issue (FP32), the FP64 pipe (FP64).
#pragma once

#include "sweep.cuh"

namespace hgks {

template <class T, int MODE, int FLUX, int TP, int TS>
struct SweepShape {
  static constexpr int HP = TP + 4, HS = TS + 4, NH = HP * HS;
  static constexpr int NV = FLUX == FLUX_FULL ? 15 : 5, NFF = SweepLayout<FLUX, MODE>::NFF, NT1 = 30;
  static constexpr int THREADS = 2 * TP * TS;
  // Slots per thread: the point state of the second t2 abscissa, then (full
  // flux) per t2 abscissa the half-space sums (15) and the pressure term of tau.
  static constexpr int ST = 20, SUMS = FLUX == FLUX_FULL ? 16 : 0, SLOTS = ST + 2 * SUMS;
  static constexpr size_t SMEM = sizeof(T) * ((NFF + NT1) * NH + SLOTS * THREADS);
  static constexpr int MIN_BLOCKS = sizeof(T) == 8 ? 1 : (FLUX == FLUX_FULL || is_char_mode<MODE>() ? 2 : 3);
  static_assert(TP == 16, "a warp holds one row of 16 faces and both t1 abscissae");
};

// Unit u of the t1 pass of group s at point `at`, two of its ten fields
// (states 0..4, slopes 5..9): (0,1), (2,3), (4,9), (5,6), (7,8).  States give
// values and t1-derivatives at both abscissae, slopes values.  FP32 with
// nonlinear weights evaluates the two in packed pairs.
template <class T, int MODE, int NV, int NH>
__device__ __forceinline__ void t1_pass_unit(const T* ff, T* tb, int s, int at, int st1, int u) {
  const int ja = u < 2 ? 2 * u : (u == 2 ? 4 : 2 * u - 1), jb = u == 2 ? 9 : ja + 1;
  auto from = [&](int j) { return ff + (5 * s + (j < 5 ? j : NV + j - 5)) * NH + at; };
  auto to = [&](int j) { return tb + (j < 5 ? 4 * j : 10 + 2 * j) * NH + at; };
  const T *sa = from(ja), *sb = from(jb);
  T *oa = to(ja), *ob = to(jb);
  T va[2], da[2], vb[2], db[2];
  if constexpr (std::is_same<T, float>::value && recon_of<MODE>() != RECON_LINEAR) {
    float2 f[5], v[2], d[2];
#pragma unroll
    for (int j = 0; j < 5; ++j) f[j] = make_float2(sa[(j - 2) * st1], sb[(j - 2) * st1]);
    tangential_weno_x2<recon_of<MODE>()>(f[0], f[1], f[2], f[3], f[4], v, d);
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      va[m] = v[m].x;
      vb[m] = v[m].y;
      da[m] = d[m].x;
      db[m] = d[m].y;
    }
  } else {
    tangential_fast<MODE>(sa[-2 * st1], sa[-st1], sa[0], sa[st1], sa[2 * st1], va, da);
    tangential_fast<MODE>(sb[-2 * st1], sb[-st1], sb[0], sb[st1], sb[2 * st1], vb, db);
  }
  oa[0] = va[0];
  oa[NH] = va[1];
  ob[0] = vb[0];
  ob[NH] = vb[1];
  if (u <= 2) {
    oa[2 * NH] = da[0];
    oa[3 * NH] = da[1];
  }
  if (u < 2) {
    ob[2 * NH] = db[0];
    ob[3 * NH] = db[1];
  }
}

// The pass along t1 of group s at point `at` in characteristic variables of
// Qm there: its states (slopes = false) or its normal slopes.
template <class T, int MODE, int NV, int NH>
__device__ __forceinline__ void t1_pass_char(const T* ff, T* tb, int s, bool slopes, int at, int st1,
                                             const Gas<T>& gas) {
  T qm[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) qm[i] = ff[(2 * NV + i) * NH + at];
  const CharBasis<T> b = char_basis(qm, gas);
  T v[2][5], d[2][5];
  tangential_char<MODE>(ff + (5 * s + (slopes ? NV : 0)) * NH + at, NH, st1, b, v, d);
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    T* o = tb + (slopes ? 20 + 2 * i : 4 * i) * NH + at;
    o[0] = v[0][i];
    o[NH] = v[1][i];
    if (!slopes) {
      o[2 * NH] = d[0][i];
      o[3 * NH] = d[1][i];
    }
  }
}

// The pass along t2 at t1 abscissa m1 of one face: the point state of the
// first t2 abscissa in g0, that of the second in the slots (component c of
// value, n, t1, t2 derivative: slot 5 c + i).
template <class T, int MODE, int NH, int NT>
__device__ __forceinline__ void t2_pass(const T* tb, int m1, int at, int st2, const CharBasis<T>& cbs, T rh1,
                                             T rh2, PointState<T>& g0, T* slot) {
  if constexpr (std::is_same<T, float>::value && recon_of<MODE>() != RECON_LINEAR && !is_char_mode<MODE>()) {
    // Two reconstructions per packed evaluation: each component's
    // t1-derivative and normal-slope fields together, the value fields of
    // components (0, 1) and (2, 3) together, component 4's alone.
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const T* sdv = tb + (4 * i + 2 + m1) * NH + at;
      const T* ss = tb + (20 + 2 * i + m1) * NH + at;
      float2 f[5], w[2], unused[2];
#pragma unroll
      for (int j = 0; j < 5; ++j) f[j] = make_float2(sdv[(j - 2) * st2], ss[(j - 2) * st2]);
      tangential_weno_x2<recon_of<MODE>()>(f[0], f[1], f[2], f[3], f[4], w, unused);
      g0.dq[0][i] = w[0].y;
      g0.dq[1][i] = w[0].x * rh1;
      slot[(5 + i) * NT] = w[1].y;
      slot[(10 + i) * NT] = w[1].x * rh1;
    }
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      const T* sa = tb + (4 * i + m1) * NH + at;
      const T* sb = sa + 4 * NH;
      float2 f[5], v[2], dd[2];
#pragma unroll
      for (int j = 0; j < 5; ++j) f[j] = make_float2(sa[(j - 2) * st2], sb[(j - 2) * st2]);
      tangential_weno_x2<recon_of<MODE>()>(f[0], f[1], f[2], f[3], f[4], v, dd);
      g0.q[i] = v[0].x;
      g0.q[i + 1] = v[0].y;
      g0.dq[2][i] = dd[0].x * rh2;
      g0.dq[2][i + 1] = dd[0].y * rh2;
      slot[i * NT] = v[1].x;
      slot[(i + 1) * NT] = v[1].y;
      slot[(15 + i) * NT] = dd[1].x * rh2;
      slot[(16 + i) * NT] = dd[1].y * rh2;
    }
    const T* sv = tb + (16 + m1) * NH + at;
    T v[2], dd[2];
    tangential<MODE>(sv[-2 * st2], sv[-st2], sv[0], sv[st2], sv[2 * st2], v, dd);
    g0.q[4] = v[0];
    g0.dq[2][4] = dd[0] * rh2;
    slot[4 * NT] = v[1];
    slot[19 * NT] = dd[1] * rh2;
  } else {
    T val[2][5], d2[2][5], d1[2][5], dn[2][5];
    t2_group<T, MODE, 5, NH>(tb, 0, m1, at, st2, cbs, val, d2, d1, dn);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      g0.q[i] = val[0][i];
      g0.dq[0][i] = dn[0][i];
      g0.dq[1][i] = d1[0][i] * rh1;
      g0.dq[2][i] = d2[0][i] * rh2;
      slot[i * NT] = val[1][i];
      slot[(5 + i) * NT] = dn[1][i];
      slot[(10 + i) * NT] = d1[1][i] * rh1;
      slot[(15 + i) * NT] = d2[1][i] * rh2;
    }
  }
}

// One tile's chunk.  t1 runs along P (the x and z sweeps) or along S, as a
// compile-time choice: the strides of both passes are then constants.
template <class T, int MODE, int FLUX, int STAGE, int TP, int TS, bool T1P>
__device__ __forceinline__ void sweep_tile(const SweepArgs<T>& a, int bx, int by, int bz) {
  using L = SweepShape<T, MODE, FLUX, TP, TS>;
  constexpr int HP = L::HP, HS = L::HS, NH = L::NH, NV = L::NV, NT = L::THREADS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* ff = reinterpret_cast<T*>(smem_raw);  // [NFF][NH]
  T* tb = ff + L::NFF * NH;                // [NT1][NH]
  T* slot = tb + L::NT1 * NH + threadIdx.x;  // [SLOTS][NT], this thread's column

  const int d = a.d;
  const SweepAxes ax = sweep_axes(d, a.g, a.xt != 0);
  const int P = ax.P, S = ax.S;
  const int nP = a.g.n[P], nS = a.g.n[S], nd = a.g.n[d];
  const int p0 = bx * TP, s0 = by * TS;
  const int f0 = bz * a.chunk, f1 = min(f0 + a.chunk, a.layers);
  const int tid = threadIdx.x;

  // Phase-3 role: face (ip, is) and t1 abscissa m1; the abscissae sit in the
  // halves of a warp, which exchange their sums so that one half stores F and
  // the other dF.
  const int m1 = (tid >> 4) & 1, ip = tid & 15, is = tid >> 5;
  const bool live = s0 + is < nS;  // the warp's row exists
  const bool face = live && p0 + ip < nP;
  const int cP = min(p0 + ip, nP - 1), cS = min(s0 + is, nS - 1);
  const T rh1 = T(1) / a.wt1[(T1P ? cP : cS) + kGhost], rh2 = T(1) / a.wt2[(T1P ? cS : cP) + kGhost];
  const int at3 = (is + 2) * HP + (ip + 2);
  constexpr int st1 = T1P ? 1 : HP, st2 = T1P ? HP : 1;
  const T dt = T(a.scal[0]);
  const long long FS = (long long)(a.g.n[0] + (d == 0)) * (a.g.n[1] + (d == 1)) * (a.g.n[2] + (d == 2));
  // Face-flux layout: x fastest for the y and z faces; y fastest ([z][x][y])
  // for the x faces (k_update reads them through a shared-memory transpose).
  long long fout, fstep;
  if (d == 0) {
    fout = (long long)cS * (a.g.n[0] + 1) * a.g.n[1] + cP;
    fstep = a.g.n[1];
  } else if (d == 1) {
    fout = (long long)cS * (a.g.n[1] + 1) * a.g.n[0] + cP;
    fstep = a.g.n[0];
  } else {
    fout = (long long)cS * a.g.n[0] + cP;
    fstep = (long long)a.g.n[0] * a.g.n[1];
  }

#pragma unroll 1
  for (int f = f0; f < f1; ++f) {
    // ---------------- phase 1: face fields ----------------
#pragma unroll 1
    for (int h = tid; h < NH; h += NT) {
      const int Pc = p0 - 2 + h % HP, Sc = s0 - 2 + h / HP;
      if (Pc <= nP + 1 && Sc <= nS + 1) {
        face_fields_item<T, MODE, FLUX, NH>(a.q, a.g, ax, a.wn, a.gas, f, Pc, Sc, h, ff);
      } else {
#pragma unroll 1
        for (int k = 0; k < L::NFF; ++k) ff[k * NH + h] = T(0);
      }
    }
    __syncthreads();

#pragma unroll 1
    for (int s = 0; s < NV / 5; ++s) {
      // ---------------- phase 2: pass along t1 of group s ----------------
      // Points of the tile with a halo of 2 along t2.
      constexpr int items = T1P ? TP * HS : HP * TS;
      constexpr int UNITS = is_char_mode<MODE>() ? 2 : 5;
#pragma unroll 1
      for (int it = tid; it < UNITS * items; it += NT) {
        const int u = it / items, pt = it - u * items;
        const int at = T1P ? (pt / TP) * HP + 2 + pt % TP : 2 * HP + pt;
        if constexpr (is_char_mode<MODE>()) t1_pass_char<T, MODE, NV, NH>(ff, tb, s, u == 1, at, st1, a.gas);
        else t1_pass_unit<T, MODE, NV, NH>(ff, tb, s, at, st1, u);
      }
      __syncthreads();

      // ---------------- phase 3: pass along t2 and the group's flux part ----------------
      if (live) {
        CharBasis<T> cbs{};
        if constexpr (is_char_mode<MODE>()) {
          T qm[5];
#pragma unroll
          for (int i = 0; i < 5; ++i) qm[i] = ff[(2 * NV + i) * NH + at3];
          cbs = char_basis(qm, a.gas);
        }
        PointState<T> st;
        t2_pass<T, MODE, NH, NT>(tb, m1, at3, st2, cbs, rh1, rh2, st, slot);
        T Fs[10];
#pragma unroll
        for (int i = 0; i < 10; ++i) Fs[i] = T(0);
#pragma unroll 1
        for (int m2 = 0; m2 < 2; ++m2) {
          if (m2 == 1) {
#pragma unroll
            for (int i = 0; i < 5; ++i) {
              st.q[i] = slot[i * NT];
              st.dq[0][i] = slot[(5 + i) * NT];
              st.dq[1][i] = slot[(10 + i) * NT];
              st.dq[2][i] = slot[(15 + i) * NT];
            }
          }
          T* sum = slot + (L::ST + m2 * L::SUMS) * NT;
          if constexpr (FLUX == FLUX_SMOOTH) {
            T F[5], dF[5];
            flux_smooth(st, a.gas, STAGE == 1, F, dF);
#pragma unroll
            for (int i = 0; i < 5; ++i) {
              if (STAGE == 1) Fs[i] += F[i];
              Fs[5 + i] += dF[i];
            }
          } else if (s < 2) {
            FullSide<T> h;
            flux_full_side(st, a.gas, s, h);
            if (s == 0) {
#pragma unroll
              for (int k = 0; k < 15; ++k) sum[k * NT] = h.V[k / 5][k % 5];
              sum[15 * NT] = h.p;
            } else {
#pragma unroll
              for (int k = 0; k < 15; ++k) sum[k * NT] += h.V[k / 5][k % 5];
              sum[15 * NT] = pressure_jump(sum[15 * NT], h.p);
            }
          } else {
            FullEq<T> e;
            flux_full_eq(st, a.gas, e);
            T Vs[3][5], F[5], dF[5];
#pragma unroll
            for (int k = 0; k < 15; ++k) Vs[k / 5][k % 5] = sum[k * NT];
            flux_full_close(e, Vs, sum[15 * NT], a.gas, dt, F, dF);
#pragma unroll
            for (int i = 0; i < 5; ++i) {
              if (STAGE == 1) Fs[i] += F[i];
              Fs[5 + i] += dF[i];
            }
          }
        }
        if (s == NV / 5 - 1) {
          const long long o = fout + (long long)f * fstep;
#pragma unroll
          for (int i = 0; i < 5; ++i) {
            const T sent = __shfl_xor_sync(0xffffffffu, m1 ? Fs[i] : Fs[5 + i], 16);
            const T total = (m1 ? Fs[5 + i] : Fs[i]) + sent;
            // The second stage needs dF only (Eq. (6)); its F planes are not written.
            if (face && (STAGE == 1 || m1)) {
              T* out = a.fd + (5 * m1 + ax.gv[i]) * FS + o;
              *out = T(0.25) * total;
              if (f == 0 && a.layers == nd) out[nd * fstep] = T(0.25) * total;  // periodic: face n is face 0
            }
          }
        }
      }
      // The next group's t1 pass overwrites tb; the next layer's face fields
      // overwrite ff, whose Qm planes phase 3 reads in the characteristic modes.
      if (s < NV / 5 - 1 || is_char_mode<MODE>()) __syncthreads();
    }
  }
}

// Body of one block: `sweeps` the arguments, b the block.
template <class T, int MODE, int FLUX, int STAGE, int TP, int TS>
__device__ __forceinline__ void sweep_block(const SweepArgs3<T>& sweeps, int b) {
  int bx, by, bz;
  const SweepArgs<T> a = sweep_of_block(sweeps, b, bx, by, bz);
  if (a.d == 1) sweep_tile<T, MODE, FLUX, STAGE, TP, TS, false>(a, bx, by, bz);
  else sweep_tile<T, MODE, FLUX, STAGE, TP, TS, true>(a, bx, by, bz);
}

template <class T, int MODE, int FLUX, int STAGE, int TP, int TS>
__global__ void __launch_bounds__(SweepShape<T, MODE, FLUX, TP, TS>::THREADS, (SweepShape<T, MODE, FLUX, TP, TS>::MIN_BLOCKS))
    k_sweep(const __grid_constant__ SweepArgs3<T> sweeps) {
  sweep_block<T, MODE, FLUX, STAGE, TP, TS>(sweeps, blockIdx.x);
}

}  // namespace hgks
