// Kernel sequences of one S2O4 stage and of the reductions, per floating
// type.  Included once by kernels_f32.cu and once by kernels_f64.cu.
#pragma once

#include "engine.h"
#include "kernels.cuh"
#include "sweep.cuh"
#include "march.cuh"
#include "sweep_tile.cuh"
#include "adjoint.cuh"
#include "turbulence.cuh"
#include "batch.cuh"

#include <algorithm>
#include <type_traits>
#include <vector>

namespace hgks {

inline GridDev grid_of(const Engine& e) {
  GridDev g;
  for (int c = 0; c < 3; ++c) {
    g.n[c] = e.n[c];
    g.p[c] = e.p[c];
  }
  g.P = e.P;
  g.N = e.N;
  return g;
}

template <class T>
Gas<T> gas_of(const hgks_config& c) {
  Gas<T> g;
  g.gamma = T(c.gamma);
  g.gm1 = T(c.gamma - 1.0);
  g.K = T((5.0 - 3.0 * c.gamma) / (c.gamma - 1.0));
  g.pr_fix = T(1.0 / c.prandtl - 1.0);
  g.visc_law = c.visc;
  g.mu_ref = T(c.mu_ref);
  g.T_ref_inv = T(1.0 / c.T_ref);
  g.visc_exp = T(c.visc_exp);
  g.tau_num_C = c.flux == HGKS_FLUX_FULL ? T(c.tau_num_C) : T(0);
  g.rho_r = T(c.rho_ref);
  g.p_r = T(c.p_ref);
  g.h_r = T(c.gamma / (c.gamma - 1.0) * c.p_ref);
  return g;
}

// Kernel MODE of a configuration: the reconstruction, + 2 for WENO in
// characteristic variables (with linear weights the projection changes
// nothing, so it is skipped).
inline int sweep_mode(const hgks_config& c) {
  return c.recon + (c.recon_vars == 1 && c.recon != HGKS_RECON_LINEAR ? 2 : 0);
}

inline unsigned blocks_for(long long n, int threads) {
  return unsigned((n + threads - 1) / threads);
}

// Ghost fill of q; with `copy` also the copy with x slowest for the x sweep.
template <class T>
PadArgs<T> pad_args(const Engine& e, void* q, bool copy) {
  return {static_cast<T*>(q), copy ? static_cast<T*>(e.qx) : nullptr, grid_of(e),
          e.cfg.bc_y == HGKS_BC_WALL_ISOTHERMAL ? 1 : 0, gas_of<T>(e.cfg), T(e.cfg.T_wall)};
}

template <class T>
cudaError_t enqueue_ghosts(const Engine& e, void* qbuf, bool copy, Probe* probe) {
  if (probe) probe->begin(e.stream, KC_GHOST);
  k_pad<T><<<dim3((e.p[0] + 31) / 32, (e.p[1] + 31) / 32, e.p[2]), 256, 0, e.stream>>>(pad_args<T>(e, qbuf, copy));
  if (probe) probe->end(e.stream);
  return cudaGetLastError();
}

// Tile of k_sweep, TP x TS faces.  FP64 is bound by its pipe, not by latency:
// with the smooth flux one CTA of 512 threads has 1.56 points of face fields
// per face where two of 16 x 8 faces have 1.88 (a step on 16 x 8 / 16 x 16:
// linear 128^3 44.3 / 40.5 ms; WENO-Z 64^3 16.4 / 15.4, in characteristic
// variables, whose 128 registers spill up to 712 bytes, 20.8 / 19.3; on grids
// of little more than a tile the smaller one would do, 12 x 10 x 9 0.45 / 0.58
// and 0.55 / 0.72, 40 x 36 x 20 with walls 2.54 / 2.82).  FP32 needs the second
// CTA's other phase: the full flux on 16 x 16 tiles, one CTA, takes 58.1 ms at
// 256^3, on 16 x 8 56.3.
template <class T, int FLUX> struct SweepTile {
  static constexpr int TP = 16, TS = sizeof(T) == 8 && FLUX == FLUX_SMOOTH ? 16 : 8;
};

// What the three sweeps of a stage on the padded state q share.
template <class T>
SweepArgs3<T> sweep_common(const Engine& e, const T* q) {
  SweepArgs3<T> a;
  a.q = q;
  // The x sweep reads the copy of the state with x slowest (k_pad).
  a.qx = static_cast<const T*>(e.qx);
  for (int d = 0; d < 3; ++d) {
    a.fd[d] = static_cast<T*>(e.fd[d]);
    a.w[d] = static_cast<const T*>(e.w[d]);
    // Face n of a periodic direction is face 0.
    a.layers[d] = e.n[d] + (d == 1 && e.cfg.bc_y != HGKS_BC_PERIODIC ? 1 : 0);
  }
  a.scal = e.scal;
  a.g = grid_of(e);
  a.gas = gas_of<T>(e.cfg);
  a.start[0] = 0;
  return a;
}

// Layers of direction d that each CTA of k_sweep or k_sweep_adj marches
// through.  The march along the normal carries nothing from one layer to the
// next, so its length only sets the number of CTAs: 24 per SM for the three
// directions, down to one layer each on small grids (24 / 48 / 96 per SM, one
// step: FP32 WENO-Z + full flux 256^3 55.2 / 54.2 / 54.0 ms and 96^3 2.92 / 2.93 /
// 2.95, WENO-JS + smooth 100x83x77 0.946 / 0.944 / 0.964, FP64 linear 128^3 40.4 /
// 40.7 / 40.8; hgks_autotune finds what suits a grid).  No march is longer than a
// tenth of an SM's share of all layers: in a direction of few tiles and many
// layers it would finish long after the others (long boxes, one step: FP64
// WENO-Z + full flux 6 x 6 x 512 21.7 -> 9.2 ms, FP32 16 x 16 x 200 269 -> 207
// us).  An even split of all layers instead costs flat boxes, whose long
// marches start first, 2 to 4 % (128 x 128 x 6 and x 16); cubes are not
// concerned.
inline int march_length(const int tiles[3], const int layers[3], int d, int sms) {
  const long long most = 24LL * sms, all = tiles[0] + tiles[1] + tiles[2];
  long long work = 0;
  for (int c = 0; c < 3; ++c) work += (long long)tiles[c] * layers[c];
  const long long chunks = (most + all - 1) / all, tenth = (work + 10LL * sms - 1) / (10LL * sms);
  return int(std::min((layers[d] + chunks - 1) / chunks, tenth));
}

// k_sweep with a TP x TS tile.
template <class T, int TP, int TS>
SweepArgs3<T> sweep_args(const Engine& e, const T* q) {
  SweepArgs3<T> a = sweep_common(e, q);
  int tiles[3];
  for (int d = 0; d < 3; ++d) {
    const int P = d == 0 ? 1 : 0, S = d == 2 ? 1 : 2;
    a.gx[d] = (e.n[P] + TP - 1) / TP;
    a.gy[d] = (e.n[S] + TS - 1) / TS;
    tiles[d] = a.gx[d] * a.gy[d];
  }
  for (int d = 0; d < 3; ++d) {
    a.chunk[d] = e.sweep_chunk > 0 ? std::min(e.sweep_chunk, a.layers[d]) : march_length(tiles, a.layers, d, e.sms);
    a.start[d + 1] = a.start[d] + tiles[d] * ((a.layers[d] + a.chunk[d] - 1) / a.chunk[d]);
  }
  return a;
}

// Rows per block of k_march for grids of so many rows that run at the same
// time: every block takes the same number of rows of the sequence of all
// tiles' rows (march_block), and the blocks are no more than the SMs, one each,
// so that they finish together; at least two rows, since each stretch repeats
// four rows of face fields (a quarter of a row's work each).  This is the only
// launch shape: shorter stretches repeat more and longer ones leave SMs idle
// (256^3: 8.55 ms a step, 8.56 to 8.88 with 526 to 64 rows a block instead of
// 1,051, 10.2 with 8; 128 x 128 x 96 with walls 0.93, 1.00 with 16; 32^3 77 us,
// 97 with 8).
inline int march_share_of(const std::vector<long long>& rows, int sms) {
  long long all = 0;
  for (const long long r : rows) all += r;
  const auto blocks = [&](long long share) {
    long long n = 0;
    for (const long long r : rows) n += (r + share - 1) / share;
    return n;
  };
  long long share = std::max(2LL, (all + sms - 1) / sms);
  while (share < all && blocks(share) > sms) ++share;
  return int(share);
}

// P is the transverse axis that is contiguous in memory, unless the grid is so
// thin along it that the other one gives at most two fifths of the rows: a row
// costs the same whatever part of its 32 faces exists.  Between two fifths and
// two thirds the strided loads cost what the fewer rows save (one step, P
// contiguous / exchanged: 6 x 128 x 128 294 / 169 us, 8 x 200 x 50 207 / 148,
// 12 x 64 x 64 112 / 96; but 16 x 128 x 128 292 / 287, 128 x 16 x 128 243 / 259,
// 20 x 100 x 160 332 / 382, 16 x 24 x 64 78 / 104).
inline SweepArgs3<float> march_args(const Engine& e, const float* q) {
  SweepArgs3<float> a = sweep_common(e, q);
  for (int d = 0; d < 3; ++d) {
    const int P = d == 0 ? 1 : 0, S = d == 2 ? 1 : 2;
    const auto tiles = [&](int p) { return (e.n[p] + March::TP - 1) / March::TP; };
    const bool exchange = 5LL * tiles(S) * e.n[P] <= 2LL * tiles(P) * e.n[S];
    a.gx[d] = tiles(exchange ? S : P);
    a.gy[d] = (a.layers[d] + March::LAYERS - 1) / March::LAYERS;
    a.chunk[d] = exchange ? 1 : 0;
    a.start[d + 1] = a.start[d] + a.gx[d] * a.gy[d] * e.n[exchange ? P : S];
  }
  a.share = e.march_share > 0 ? e.march_share : march_share_of({a.start[3]}, e.sms);
  return a;
}
inline int march_blocks(const SweepArgs3<float>& a) { return (a.start[3] + a.share - 1) / a.share; }

template <class T, int MODE, int FLUX, int STAGE>
cudaError_t launch_sweep(const Engine& e, const T* q) {
  if constexpr (std::is_same<T, float>::value && MODE == RECON_LINEAR && FLUX == FLUX_SMOOTH) {
    const SweepArgs3<float> a = march_args(e, q);
    const cudaError_t err = cudaFuncSetAttribute(k_march<STAGE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)March::SMEM);
    if (err != cudaSuccess) return err;
    k_march<STAGE><<<march_blocks(a), March::THREADS, March::SMEM, e.stream>>>(a);
    return cudaGetLastError();
  } else {
    constexpr int TP = SweepTile<T, FLUX>::TP, TS = SweepTile<T, FLUX>::TS;
    using L = SweepShape<T, MODE, FLUX, TP, TS>;
    const SweepArgs3<T> a = sweep_args<T, TP, TS>(e, q);
    auto kern = k_sweep<T, MODE, FLUX, STAGE, TP, TS>;
    const cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::SMEM);
    if (err != cudaSuccess) return err;
    kern<<<a.start[3], L::THREADS, L::SMEM, e.stream>>>(a);
    return cudaGetLastError();
  }
}

// The three sweeps of a stage.
template <class T, int MODE, int FLUX>
cudaError_t launch_all_directions(const Engine& e, const T* q, int stage, Probe* probe) {
  if (probe) probe->begin(e.stream, stage == 1 ? KC_FLUX1 : KC_FLUX2);
  const cudaError_t err = stage == 1 ? launch_sweep<T, MODE, FLUX, 1>(e, q)
                                     : launch_sweep<T, MODE, FLUX, 2>(e, q);
  if (probe) probe->end(e.stream);
  return err;
}

// Arguments of the update kernel on the context's current buffers.
template <class T>
UpdateArgs<T> update_args(const Engine& e) {
  UpdateArgs<T> ua;
  ua.q = static_cast<T*>(e.q);
  ua.qs = static_cast<T*>(e.qs);
  ua.inc = static_cast<T*>(e.inc);
  ua.comp = static_cast<T*>(e.comp);
  ua.comp_out = static_cast<T*>(e.comp2);
  ua.flag = e.guard ? e.flag : nullptr;
  ua.fx = static_cast<const T*>(e.fd[0]);
  ua.fy = static_cast<const T*>(e.fd[1]);
  ua.fz = static_cast<const T*>(e.fd[2]);
  ua.wx = static_cast<const T*>(e.w[0]);
  ua.wy = static_cast<const T*>(e.w[1]);
  ua.wz = static_cast<const T*>(e.w[2]);
  ua.scal = e.scal;
  ua.time = e.scal;
  ua.g = grid_of(e);
  const bool mass_flux = e.cfg.force_mode == HGKS_FORCE_MASS_FLUX;
  ua.force_x = mass_flux ? T(0) : T(e.cfg.force_x);
  ua.rho_r = T(e.cfg.rho_ref);
  return ua;
}

template <class T>
cudaError_t enqueue_rhs_and_update(const Engine& e, int stage, Probe* probe) {
  T* qin = static_cast<T*>(stage == 1 ? e.q : e.qs);
  cudaError_t err = enqueue_ghosts<T>(e, qin, e.qx != nullptr, probe);
  if (err != cudaSuccess) return err;
  const int mode = sweep_mode(e.cfg), flux = e.cfg.flux;
#define HGKS_DISPATCH(M, F) \
  if (mode == M && flux == F) err = launch_all_directions<T, M, F>(e, qin, stage, probe);
  HGKS_DISPATCH(0, 0) HGKS_DISPATCH(1, 0) HGKS_DISPATCH(2, 0) HGKS_DISPATCH(3, 0) HGKS_DISPATCH(4, 0)
  HGKS_DISPATCH(0, 1) HGKS_DISPATCH(1, 1) HGKS_DISPATCH(2, 1) HGKS_DISPATCH(3, 1) HGKS_DISPATCH(4, 1)
#undef HGKS_DISPATCH
  if (err != cudaSuccess) return err;
  const UpdateArgs<T> ua = update_args<T>(e);
  const bool mass_flux = e.cfg.force_mode == HGKS_FORCE_MASS_FLUX;
  if (probe) probe->begin(e.stream, KC_UPDATE);
  const dim3 ugrid((e.n[0] + kUpdTX - 1) / kUpdTX, (e.n[1] + kUpdTY - 1) / kUpdTY, e.n[2]);
  if (stage == 1)
    k_update<T, 1><<<ugrid, kUpdTX * kUpdTY, 0, e.stream>>>(ua);
  else
    k_update<T, 2><<<ugrid, kUpdTX * kUpdTY, 0, e.stream>>>(ua);
  if (mass_flux && stage == 2) {
    // Sec. 3.3: the force that keeps the volume integral of rho U at its
    // target, on Q~^{n+1} (in qs, compensation in comp2), with rho^n and
    // (rho U)^n read from Q^n (q).
    const GridDev g = grid_of(e);
    k_massflux_sums<T><<<e.diag_blocks, 256, 0, e.stream>>>(
        ua.qs, ua.q, ua.comp_out, g, ua.wx, ua.wy, ua.wz, e.cfg.rho_ref, e.part, ua.flag);
    k_massflux_force<<<1, 256, 0, e.stream>>>(e.part, e.diag_blocks, e.cfg.mass_flux, e.scal, ua.flag);
    k_force_apply<T><<<blocks_for(e.N, 256), 256, 0, e.stream>>>(ua.qs, ua.q, ua.comp_out, g,
                                                                 e.cfg.rho_ref, e.scal, ua.flag);
  }
  if (probe) probe->end(e.stream);
  return cudaGetLastError();
}

template <class T>
cudaError_t enqueue_sweep_only(const Engine& e) {
  const T* q = static_cast<const T*>(e.q);
  const int mode = sweep_mode(e.cfg), flux = e.cfg.flux;
#define HGKS_SW(M, F) \
  if (mode == M && flux == F) return launch_sweep<T, M, F, 1>(e, q);
  HGKS_SW(0, 0) HGKS_SW(1, 0) HGKS_SW(2, 0) HGKS_SW(3, 0) HGKS_SW(4, 0)
  HGKS_SW(0, 1) HGKS_SW(1, 1) HGKS_SW(2, 1) HGKS_SW(3, 1) HGKS_SW(4, 1)
#undef HGKS_SW
  return cudaErrorInvalidValue;
}

// CFL reduction and check of the state in qbuf; with_dt also sets the step's
// dt (dt_fixed > 0 overrides the CFL step).
template <class T>
CflArgs<T> cfl_args(const Engine& e, const void* qbuf, bool with_dt, double dt_fixed) {
  return {static_cast<const T*>(qbuf), grid_of(e), static_cast<const T*>(e.w[0]),
          static_cast<const T*>(e.w[1]), static_cast<const T*>(e.w[2]), e.cfg.rho_ref, e.cfg.p_ref,
          e.cfg.gamma, e.dtmin, e.flag, reinterpret_cast<unsigned*>(e.flag + 1),
          with_dt ? e.scal : nullptr, e.cfg.cfl, dt_fixed, e.guard ? 1 : 0};
}

template <class T>
cudaError_t enqueue_cfl(const Engine& e, const void* qbuf, bool with_dt, double dt_fixed) {
  k_cfl<T><<<e.cfl_blocks, 256, 0, e.stream>>>(cfl_args<T>(e, qbuf, with_dt, dt_fixed));
  return cudaGetLastError();
}

template <class T>
cudaError_t enqueue_diag(const Engine& e) {
  k_diag<T><<<e.diag_blocks, 256, 0, e.stream>>>(
      static_cast<const T*>(e.q), grid_of(e), static_cast<const T*>(e.w[0]),
      static_cast<const T*>(e.w[1]), static_cast<const T*>(e.w[2]), e.cfg.rho_ref, e.cfg.p_ref,
      e.cfg.gamma, e.part);
  k_diag_final<<<1, 256, 0, e.stream>>>(e.part, e.diag_blocks, e.diag_out);
  return cudaGetLastError();
}

inline TurbArgs turb_args(const hgks_config& c, const int n[3]) {
  TurbArgs a;
  const double L[3] = {c.lx, c.ly, c.lz};
  double vol = 1.0;
  for (int d = 0; d < 3; ++d) {
    const double h = L[d] / n[d];
    a.inv60h[d] = 1.0 / (60.0 * h);
    vol *= h;
  }
  a.vol = vol;
  a.rho_r = c.rho_ref;
  a.E_r = c.p_ref / (c.gamma - 1.0);
  a.gm1 = c.gamma - 1.0;
  a.visc_law = c.visc;
  a.mu_ref = c.mu_ref;
  a.T_ref_inv = 1.0 / c.T_ref;
  a.visc_exp = c.visc_exp;
  const double K = (5.0 - 3.0 * c.gamma) / (c.gamma - 1.0);
  a.mub_ratio = 2.0 * K / (3.0 * (K + 3.0));
  return a;
}

// Turbulence statistics of Q^n: per-block FP64 sums, final sum into
// e.turb_out (kTurbSums doubles).
template <class T>
cudaError_t enqueue_turbulence(const Engine& e) {
  const HistGate gate{e.scal, nullptr, 0};
  k_turb<T><<<e.diag_blocks, 256, 0, e.stream>>>(static_cast<const T*>(e.q), grid_of(e),
                                                 turb_args(e.cfg, e.n), e.turb_part, gate);
  const TurbSink sink{e.turb_out, nullptr, nullptr, 0};
  k_turb_final<<<1, 256, 0, e.stream>>>(e.turb_part, e.diag_blocks, sink, gate);
  return cudaGetLastError();
}

// A record of the statistics history from the state in qbuf.
template <class T>
cudaError_t enqueue_history_record(const Engine& e, const void* qbuf, bool gated) {
  const HistGate gate{e.scal, e.flag, gated ? e.hist_every : 0};
  k_turb<T><<<e.diag_blocks, 256, 0, e.stream>>>(static_cast<const T*>(qbuf), grid_of(e),
                                                 turb_args(e.cfg, e.n), e.turb_part, gate);
  const TurbSink sink{nullptr, e.hist, e.hist_count, e.hist_cap};
  k_turb_final<<<1, 256, 0, e.stream>>>(e.turb_part, e.diag_blocks, sink, gate);
  return cudaGetLastError();
}

// Channel plane averages: kChanSums FP64 sums per y row into e.chan_out.
template <class T>
cudaError_t enqueue_channel_rows(const Engine& e) {
  const hgks_config& c = e.cfg;
  k_channel_rows<T><<<e.n[1], 256, 0, e.stream>>>(static_cast<const T*>(e.q), grid_of(e), c.rho_ref,
                                                  c.p_ref, c.gamma - 1.0, e.chan_out);
  return cudaGetLastError();
}

template <class T>
cudaError_t enqueue_from_fp64(const Engine& e, const double* src, int conservative) {
  const GridDev g = grid_of(e);
  const dim3 grid((g.n[0] + 255) / 256, g.n[1], g.n[2]);
  const double inv_gm1 = 1.0 / (e.cfg.gamma - 1.0);
  k_from_prim<T><<<grid, 256, 0, e.stream>>>(src, static_cast<T*>(e.q), g, e.cfg.rho_ref,
                                              e.cfg.p_ref / (e.cfg.gamma - 1.0), inv_gm1, conservative);
  return cudaGetLastError();
}

template <class T>
cudaError_t enqueue_to_fp64(const Engine& e, double* dst) {
  const GridDev g = grid_of(e);
  const dim3 grid((g.n[0] + 255) / 256, g.n[1], g.n[2]);
  k_to_cons<T><<<grid, 256, 0, e.stream>>>(static_cast<const T*>(e.q), dst, g, e.cfg.rho_ref,
                                            e.cfg.p_ref / (e.cfg.gamma - 1.0));
  return cudaGetLastError();
}

// Tiles of the adjoint sweep: four shared-memory planes (face fields, t1 pass
// and their cotangents) must fit one CTA.  Twelve rows instead of eight where
// that fits: fewer halo points per face (FP64 smooth 1.67 instead of 1.88) and
// 12 warps instead of 8 (168 registers): FP64 40x36x33 window 63.1 -> 60.8 ms,
// FP32 full flux 64^3 6.30 -> 6.09 ms (16 rows, 128 registers: 6.03).
template <class T, int FLUX> struct AdjTile { static constexpr int TP = 16, TS = sizeof(T) == 8 ? 12 : 8, NT = 32 * TS; };
template <> struct AdjTile<float, FLUX_FULL> { static constexpr int TP = 8, TS = 12, NT = 384; };
template <> struct AdjTile<double, FLUX_FULL> { static constexpr int TP = 8, TS = 4, NT = 128; };

template <class T, int MODE, int FLUX>
cudaError_t launch_adjoint_sweeps(const Engine& e, const T* q, const T* wL, const T* wdL) {
  constexpr int TP = AdjTile<T, FLUX>::TP, TS = AdjTile<T, FLUX>::TS, NT = AdjTile<T, FLUX>::NT;
  const GridDev g = grid_of(e);
  constexpr size_t smem = adj_smem_bytes<T, FLUX, TP, TS>();
  auto kern = k_sweep_adj<T, MODE, FLUX, TP, TS, NT>;
  cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  AdjArgs<T> a;
  a.q = q;
  a.wL = wL;
  a.wdL = wdL;
  a.acc = static_cast<T*>(e.adj_acc);
  a.scal = e.scal;
  a.g = g;
  a.gas = gas_of<T>(e.cfg);
  a.start[0] = 0;
  int tiles[3];
  for (int d = 0; d < 3; ++d) {
    const int P = d == 0 ? 1 : 0, S = d == 2 ? 1 : 2;
    a.w[d] = static_cast<const T*>(e.w[d]);
    a.gx[d] = (g.n[P] + TP - 1) / TP;
    a.gy[d] = (g.n[S] + TS - 1) / TS;
    tiles[d] = a.gx[d] * a.gy[d];
  }
  // A layer takes tens of microseconds and shares nothing with the next:
  // march_length's 24 CTAs per SM keep the tail under a few per cent.
  for (int d = 0; d < 3; ++d) {
    a.chunk[d] = march_length(tiles, g.n, d, e.sms);
    a.start[d + 1] = a.start[d] + tiles[d] * ((g.n[d] + a.chunk[d] - 1) / a.chunk[d]);
  }
  kern<<<a.start[3], NT, smem, e.stream>>>(a);
  err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  T* acc = static_cast<T*>(e.adj_acc);
  k_fold_ghosts_z<T><<<blocks_for(6LL * g.p[0] * g.p[1], 256), 256, 0, e.stream>>>(acc, g);
  k_fold_ghosts_y<T><<<blocks_for(6LL * g.p[0] * g.n[2], 256), 256, 0, e.stream>>>(acc, g);
  k_fold_ghosts_x<T><<<blocks_for(6LL * g.n[1] * g.n[2], 256), 256, 0, e.stream>>>(acc, g);
  return cudaGetLastError();
}

template <class T>
cudaError_t dispatch_adjoint_sweeps(const Engine& e, const T* q, const T* wL, const T* wdL) {
  const int mode = e.cfg.recon, flux = e.cfg.flux;
#define HGKS_ADJ(M, F) \
  if (mode == M && flux == F) return launch_adjoint_sweeps<T, M, F>(e, q, wL, wdL);
  HGKS_ADJ(0, 0) HGKS_ADJ(1, 0) HGKS_ADJ(2, 0)
  HGKS_ADJ(0, 1) HGKS_ADJ(1, 1) HGKS_ADJ(2, 1)
#undef HGKS_ADJ
  return cudaErrorInvalidValue;
}

template <class T>
cudaError_t enqueue_adjoint_step(const Engine& e, const double* adj_in, double* adj_out) {
  const GridDev g = grid_of(e);
  T* acc = static_cast<T*>(e.adj_acc);
  T* mu = static_cast<T*>(e.adj_mu);
  T* wL = static_cast<T*>(e.adj_wL);
  T* wdL = static_cast<T*>(e.adj_wdL);
  const size_t accb = 5 * (size_t)e.P * sizeof(T);
  // Q* = Q^n + dt/2 L + dt^2/8 dL (also fills the ghost cells of Q^n); the
  // step's non-physical guard does not apply here.
  Engine ea = e;
  ea.guard = false;
  cudaError_t err = enqueue_rhs_and_update<T>(ea, 1);
  if (err != cudaSuccess) return err;
  err = enqueue_ghosts<T>(e, e.qs, false);
  if (err != cudaSuccess) return err;
  // mu* = (d dL(Q*)/dQ*)^T (dt^2/3 lam).
  err = cudaMemsetAsync(acc, 0, accb, e.stream);
  if (err != cudaSuccess) return err;
  k_adj_combine<T><<<blocks_for(e.N, 256), 256, 0, e.stream>>>(0, adj_in, acc, mu, wL, wdL, nullptr,
                                                               e.scal, g);
  err = dispatch_adjoint_sweeps<T>(e, static_cast<const T*>(e.qs), nullptr, wdL);
  if (err != cudaSuccess) return err;
  // Cotangents of L(Q^n) and dL(Q^n), then their VJP at Q^n.
  k_adj_combine<T><<<blocks_for(e.N, 256), 256, 0, e.stream>>>(1, adj_in, acc, mu, wL, wdL, nullptr,
                                                               e.scal, g);
  err = cudaMemsetAsync(acc, 0, accb, e.stream);
  if (err != cudaSuccess) return err;
  err = dispatch_adjoint_sweeps<T>(e, static_cast<const T*>(e.q), wL, wdL);
  if (err != cudaSuccess) return err;
  k_adj_combine<T><<<blocks_for(e.N, 256), 256, 0, e.stream>>>(2, adj_in, acc, mu, wL, wdL, adj_out,
                                                               e.scal, g);
  return cudaGetLastError();
}

// ---------------------------------------------------------- batched step ---
// One S2O4 step of every member (same precision, reconstruction and flux;
// constant or no body force) with one batched launch per phase
// (batch.cuh) on stream s.  Each member's arguments are those of its own
// launches: its buffers, grid, chunking and non-physical guard.

// Launch Job over the members (in groups of kBatchMax): job i runs blocks[i] blocks.
template <class Job>
cudaError_t launch_batched(const std::vector<Job>& jobs, const std::vector<int>& blocks, size_t smem,
                           cudaStream_t s) {
  auto kern = k_batched<Job>;
  if (smem > 0) {
    const cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
  }
  for (size_t i0 = 0; i0 < jobs.size(); i0 += kBatchMax) {
    BatchTable<Job> t;
    t.n = (int)std::min<size_t>(kBatchMax, jobs.size() - i0);
    int acc = 0;
    for (int m = 0; m < t.n; ++m) {
      t.start[m] = acc;
      t.job[m] = jobs[i0 + m];
      acc += blocks[i0 + m];
    }
    t.start[t.n] = acc;
    if (acc == 0) continue;
    kern<<<acc, Job::kThreads, smem, s>>>(t);
    const cudaError_t err = cudaGetLastError();
    if (err != cudaSuccess) return err;
  }
  return cudaSuccess;
}

template <class T, int MODE, int FLUX, int STAGE>
cudaError_t batched_sweeps(const std::vector<Engine*>& ms, int stage, cudaStream_t s) {
  std::vector<int> blocks;
  if constexpr (std::is_same<T, float>::value && MODE == RECON_LINEAR && FLUX == FLUX_SMOOTH) {
    std::vector<MarchJob<STAGE>> jobs;
    for (Engine* e : ms) {
      jobs.push_back({march_args(*e, static_cast<const T*>(stage == 1 ? e->q : e->qs))});
      blocks.push_back(march_blocks(jobs.back().a));
    }
    return launch_batched(jobs, blocks, March::SMEM, s);
  } else {
    constexpr int TP = SweepTile<T, FLUX>::TP, TS = SweepTile<T, FLUX>::TS;
    std::vector<SweepJob<T, MODE, FLUX, STAGE, TP, TS>> jobs;
    for (Engine* e : ms) {
      jobs.push_back({sweep_args<T, TP, TS>(*e, static_cast<const T*>(stage == 1 ? e->q : e->qs))});
      blocks.push_back(jobs.back().a.start[3]);
    }
    return launch_batched(jobs, blocks, SweepShape<T, MODE, FLUX, TP, TS>::SMEM, s);
  }
}

template <class T>
cudaError_t enqueue_batched_step(const std::vector<Engine*>& ms, double dt_fixed, cudaStream_t s) {
  cudaError_t err;
  {
    std::vector<CflJob<T>> jobs;
    std::vector<int> blocks;
    for (Engine* e : ms) {
      jobs.push_back({cfl_args<T>(*e, e->q, true, dt_fixed), e->cfl_blocks});
      blocks.push_back(e->cfl_blocks);
    }
    if ((err = launch_batched(jobs, blocks, 0, s)) != cudaSuccess) return err;
  }
  const int mode = sweep_mode(ms[0]->cfg), flux = ms[0]->cfg.flux;
  for (int stage = 1; stage <= 2; ++stage) {
    std::vector<PadJob<T>> pj;
    std::vector<int> pb;
    for (Engine* e : ms) {
      const int gx = (e->p[0] + 31) / 32, gy = (e->p[1] + 31) / 32;
      pj.push_back({pad_args<T>(*e, stage == 1 ? e->q : e->qs, e->qx != nullptr), gx, gy});
      pb.push_back(gx * gy * e->p[2]);
    }
    if ((err = launch_batched(pj, pb, 0, s)) != cudaSuccess) return err;
    err = cudaErrorInvalidValue;
#define HGKS_BSW(M, F)                                                                           \
    if (mode == M && flux == F)                                                                  \
      err = stage == 1 ? batched_sweeps<T, M, F, 1>(ms, stage, s)                        \
                       : batched_sweeps<T, M, F, 2>(ms, stage, s);
    HGKS_BSW(0, 0) HGKS_BSW(1, 0) HGKS_BSW(2, 0) HGKS_BSW(3, 0) HGKS_BSW(4, 0)
    HGKS_BSW(0, 1) HGKS_BSW(1, 1) HGKS_BSW(2, 1) HGKS_BSW(3, 1) HGKS_BSW(4, 1)
#undef HGKS_BSW
    if (err != cudaSuccess) return err;
    std::vector<int> ub;
    if (stage == 1) {
      std::vector<UpdateJob<T, 1>> uj;
      for (Engine* e : ms) {
        const int gx = (e->n[0] + kUpdTX - 1) / kUpdTX, gy = (e->n[1] + kUpdTY - 1) / kUpdTY;
        uj.push_back({update_args<T>(*e), gx, gy});
        ub.push_back(gx * gy * e->n[2]);
      }
      err = launch_batched(uj, ub, 0, s);
    } else {
      std::vector<UpdateJob<T, 2>> uj;
      for (Engine* e : ms) {
        const int gx = (e->n[0] + kUpdTX - 1) / kUpdTX, gy = (e->n[1] + kUpdTY - 1) / kUpdTY;
        uj.push_back({update_args<T>(*e), gx, gy});
        ub.push_back(gx * gy * e->n[2]);
      }
      err = launch_batched(uj, ub, 0, s);
    }
    if (err != cudaSuccess) return err;
  }
  return cudaSuccess;
}

#define HGKS_INSTANTIATE(T)                                                  \
  template cudaError_t enqueue_ghosts<T>(const Engine&, void*, bool, Probe*); \
  template cudaError_t enqueue_rhs_and_update<T>(const Engine&, int, Probe*); \
  template cudaError_t enqueue_cfl<T>(const Engine&, const void*, bool, double); \
  template cudaError_t enqueue_sweep_only<T>(const Engine&);                 \
  template cudaError_t enqueue_diag<T>(const Engine&);                       \
  template cudaError_t enqueue_turbulence<T>(const Engine&);                 \
  template cudaError_t enqueue_history_record<T>(const Engine&, const void*, bool); \
  template cudaError_t enqueue_channel_rows<T>(const Engine&);               \
  template cudaError_t enqueue_from_fp64<T>(const Engine&, const double*, int); \
  template cudaError_t enqueue_to_fp64<T>(const Engine&, double*);           \
  template cudaError_t enqueue_adjoint_step<T>(const Engine&, const double*, double*); \
  template cudaError_t enqueue_batched_step<T>(const std::vector<Engine*>&, double, cudaStream_t);

}  // namespace hgks
