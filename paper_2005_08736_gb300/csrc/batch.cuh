// Batched launches of an ensemble step: ONE grid per phase of the S2O4 step
// (CFL reduction and dt; ghost fill with the transposed copy, the three sweeps
// and the update of each stage) covering every instance of the ensemble.  The
// instance table is a kernel parameter (__grid_constant__: it stays in the
// constant bank, no copy): instance m owns the blocks [start[m], start[m+1])
// of the grid, and each block runs the same body as the single-instance kernel
// (kernels.cuh, sweep_tile.cuh, march.cuh) on its instance's arguments and its
// local block coordinates.  No block waits on another: the phases are ordered
// by the stream (and the captured graph) only.
#pragma once

#include "engine.h"
#include "kernels.cuh"
#include "march.cuh"
#include "sweep_tile.cuh"

namespace hgks {

template <class Job>
struct BatchTable {
  int n;                      // instances
  int start[kBatchMax + 1];   // first block of each instance; start[n] = grid size
  Job job[kBatchMax];
};

// The instance that owns block b: the last m with start[m] <= b.
template <class Job>
__device__ __forceinline__ int batch_instance(const BatchTable<Job>& t, int b) {
  int lo = 0, hi = t.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (t.start[mid] <= b) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

template <class Job>
__global__ void __launch_bounds__(Job::kThreads, Job::kMinBlocks)
    k_batched(const __grid_constant__ BatchTable<Job> t) {
  const int b = blockIdx.x;
  const int m = batch_instance(t, b);
  t.job[m].run(b - t.start[m]);
}

// ------------------------------------------------------------------ jobs ---

template <class T>
struct CflJob {
  static constexpr int kThreads = 256, kMinBlocks = 1;
  CflArgs<T> a;
  int nblocks;
  __device__ __forceinline__ void run(int b) const { cfl_block(a, b, nblocks); }
};

template <class T>
struct PadJob {
  static constexpr int kThreads = 256, kMinBlocks = 1;
  PadArgs<T> a;
  int gx, gy;
  __device__ __forceinline__ void run(int b) const { pad_block(a, b % gx, (b / gx) % gy, b / (gx * gy)); }
};

template <class T, int MODE, int FLUX, int STAGE, int TP, int TS>
struct SweepJob {
  static constexpr int kThreads = SweepShape<T, MODE, FLUX, TP, TS>::THREADS;
  static constexpr int kMinBlocks = SweepShape<T, MODE, FLUX, TP, TS>::MIN_BLOCKS;
  SweepArgs3<T> a;
  __device__ __forceinline__ void run(int b) const { sweep_block<T, MODE, FLUX, STAGE, TP, TS>(a, b); }
};

template <int STAGE>
struct MarchJob {
  static constexpr int kThreads = March::THREADS, kMinBlocks = 1;
  SweepArgs3<float> a;
  __device__ __forceinline__ void run(int b) const { march_block<STAGE>(a, b); }
};

template <class T, int STAGE>
struct UpdateJob {
  static constexpr int kThreads = kUpdTX * kUpdTY, kMinBlocks = sizeof(T) == 4 ? 8 : 1;
  UpdateArgs<T> a;
  int gx, gy;
  __device__ __forceinline__ void run(int b) const {
    __shared__ T sfx[STAGE == 1 ? 10 : 5][kUpdTX + 1][kUpdTY + 1];
#define HGKS_UPD_BX (b % gx)
#define HGKS_UPD_BY ((b / gx) % gy)
#define HGKS_UPD_BZ (b / (gx * gy))
#include "update_body.inc"
#undef HGKS_UPD_BX
#undef HGKS_UPD_BY
#undef HGKS_UPD_BZ
  }
};

}  // namespace hgks
