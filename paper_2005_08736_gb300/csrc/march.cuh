// Sweeps of the FP32 scheme with linear weights and the smooth flux: the
// three directions of one S2O4 stage in one launch, marching along a
// TRANSVERSE axis.
//
// A CTA owns 10 face layers along the normal n and 32 faces along P (the
// transverse axis that is contiguous in memory, but for very thin grids,
// march_args) and marches row by row along S, the other transverse axis.  Per row s:
//   A  face fields (WENO5 end values, compatibility state Q0, normal slope)
//      of row s + 2 at 32 + 4 points of P, from the row's cells, which were
//      copied to shared memory asynchronously a row ahead;
//   B  the tangential pass along S for row s, from the fields of rows
//      s-2 .. s+2: four rows in a thread-private ring in shared memory, the
//      newest in registers; 15 values at the two S abscissae to shared memory;
//   C  the tangential pass along P and the flux at the four Gauss points.
// Two adjacent face layers are the halves of packed FP32 pairs (packed.cuh)
// from the cells to the flux, so no pair is ever regrouped and no alignment
// of the grid is needed.  Six warps make A and B of a row while ten warps do
// C of the row before (two buffers between them, one barrier a row): about
// 700 and 600 instructions each, so both halves finish together and the FMA
// pipe sees all sixteen warps all the time.
//
// Why this split: marching along the normal instead (the tiles of sweep_tile.cuh)
// recomputes the face fields of a halo of two on all four sides (1.69x for a
// 32 x 8 tile) and the first tangential pass on two (1.31x), and its passes
// alternate over the CTA with five barriers per two layers; there the face
// fields and the first pass took 63 % of the time for 40 % of the work.  Here
// the halo is 36/32 in P and four rows per march in S.  The linear passes
// along S and P commute, so S may come first in every direction; the frame is
// (n, P, S) and the flux is symmetric in the two tangential axes.
// 512 threads, 165.6 KB of shared memory: one CTA per SM.
// Measured (GB300, three sweeps of stage 1 / 2): 256^3 4.03 / 3.70 ms with
// the tiles (32 x 8, packed pairs, tuned march), 3.17 / 2.87 ms here; 32^3 95 /
// 86 us (three launches of the default tile), 26 / 26 us.  FMA pipe 54 %
// active, 49 % of the issue slots (128^3, ncu); what is left is issue and
// shared-memory bandwidth (52 % of its peak).  Tried: one role at a time in
// 192- or 256-thread CTAs, two per SM: 3.63 and 3.51 ms (warps waited at the
// barriers while a third of them made A and B).
#pragma once

#include "compat.cuh"
#include "sweep.cuh"

namespace hgks {

struct March {
  static constexpr int TP = 32, LP = 5, LAYERS = 2 * LP;  // faces along P, layer pairs
  static constexpr int HP = TP + 4, NPT = LP * HP;        // point pairs
  static constexpr int MAKERS = 192;                      // threads of A and B (one per point pair)
  static constexpr int THREADS = MAKERS + 2 * LP * TP;    // and of C (two per face pair)
  static constexpr int RING = 4, NFF = 10, NOUT = 30;
  static constexpr int PLANES = LAYERS + 5;               // cells along n of the layers' stencils
  static constexpr int CELLS = 5 * PLANES * HP;
  static constexpr size_t SMEM = sizeof(float2) * NPT * (RING * NFF + 2 * NOUT) + sizeof(float) * 2 * CELLS;
  static_assert(MAKERS >= NPT && MAKERS >= 5 * HP && MAKERS % 32 == 0, "a maker per point pair and staged column");
};

// Coefficients of the linear tangential reconstruction's derivative for cells
// of width w: P'(+-g) = a (f0 - f4 + 8 (f3 - f1)) +- b (13 (f1 + f3) - 24 f2 -
// (f0 + f4)), a = 1/(12 w), b = sqrt3/(54 w).  The integers are exact and a is
// formed like the normal slope's 1/(6 (hl + hr)), so on a uniform grid the
// derivatives along all three axes carry the same rounding: what balances in
// rho u.grad u + grad p stays balanced (the density fluctuations of a
// low-Mach flow are what is left over).
struct DerivCoef {
  float2 a, b;
  HGKS_HD explicit DerivCoef(float w) {
    a = bc2(1.f / (6.f * (w + w)));
    b = bc2((1.7320508075688772f / 54.f) / w);
  }
};

// tangential_linear_x2 with the derivatives per unit length.
HGKS_HD void tangential_linear_scaled_x2(float2 f0, float2 f1, float2 f2, float2 f3, float2 f4, const DerivCoef& c,
                                         float2 v[2], float2 d[2]) {
  const float sq3 = 1.7320508075688772f;
  const float2 s13 = add2(f1, f3), s04 = add2(f0, f4);
  const float2 d04 = sub2(f0, f4), d31 = sub2(f3, f1);
  const float2 E = add2(f2, fma2(f2, bc2(-1.f / 720.f), fma2(s13, bc2(1.f / 1080.f), mul2(s04, bc2(-1.f / 4320.f)))));
  const float2 O = fma2(d04, bc2(sq3 * 7.f / 432.f), mul2(d31, bc2(sq3 * 25.f / 216.f)));
  const float2 A = fma2(d31, bc2(8.f), d04);
  const float2 B = mul2(c.b, fma2(s13, bc2(-13.f), fma2(f2, bc2(24.f), s04)));
  v[0] = sub2(E, O);
  v[1] = add2(E, O);
  d[0] = fma2(c.a, A, B);
  d[1] = sub2(mul2(c.a, A), B);
}

// Rows row, row + 1, ... (at most `most`) of one tile; returns their number.
template <int STAGE>
__device__ __forceinline__ int march_rows(const SweepArgs3<float>& sweeps, int row, int most) {
  constexpr int HP = March::HP, NPT = March::NPT, NFF = March::NFF;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* ring = reinterpret_cast<float2*>(smem_raw);  // [RING][NFF][NPT]
  float2* outb = ring + March::RING * NFF * NPT;       // [2][NOUT][NPT], rows s in turn
  float* cells = reinterpret_cast<float*>(outb + 2 * March::NOUT * NPT);  // [2][5][PLANES][HP], rows in turn
  const SweepArgs<float> a = sweep_of(sweeps, row >= sweeps.start[2] ? 2 : (row >= sweeps.start[1] ? 1 : 0));
  const GridDev& g = a.g;
  const int d = a.d;
  const int P = a.chunk ? (d == 2 ? 1 : 2) : (d == 0 ? 1 : 0), S = 3 - d - P;
  const int nd = sweeps.g.n[d], nP = sweeps.g.n[P], nS = sweeps.g.n[S];
  const int layers = sweeps.layers[d];
  const int rel = row - sweeps.start[d], tile = rel / nS, tiles = sweeps.gx[d];
  const int p0 = (tile % tiles) * March::TP, f0 = (tile / tiles) * March::LAYERS;
  const int s0 = rel % nS, s1 = min(s0 + most, nS);
  const int tid = threadIdx.x;
  // Strides of the state the sweep reads, per axis, and of its variables.
  const long long sx = a.xt ? (long long)g.p[2] * g.p[1] : 1LL, sy = a.xt ? 1LL : (long long)g.p[0],
                  sz = a.xt ? (long long)g.p[1] : (long long)g.p[0] * g.p[1];
  const auto stride = [&](int axis) { return axis == 0 ? sx : (axis == 1 ? sy : sz); };
  const long long sn = stride(d), sp = stride(P), ss = stride(S);
  const int gv[5] = {0, 1 + d, 1 + P, 1 + S, 4};
  const bool t1P = P == (d + 1) % 3;
  const float *wP = t1P ? a.wt1 : a.wt2, *wS = t1P ? a.wt2 : a.wt1;

  if (tid < March::MAKERS) {
    // A, B: point pair (layers f, f + 1; column hp).  Columns past the grid's
    // halo repeat the last one (their results are not used).
    const int v = tid / HP, hp = tid % HP, f = f0 + 2 * v;
    const bool live = tid < NPT && f < layers;
    float2 r6;
    {
      const int fa = min(f, nd), fb = min(f + 1, nd);
      r6 = make_float2(1.f / (6.f * (a.wn[fa - 1 + kGhost] + a.wn[fa + kGhost])),
                       1.f / (6.f * (a.wn[fb - 1 + kGhost] + a.wn[fb + kGhost])));
    }
    // Cells f0-3 .. f0+LAYERS+1 along n of the CTA's columns, one row ahead:
    // thread (variable v, column hp) copies its cells asynchronously, all that
    // the pairs with a layer that exists read.  The plane past the ghost cells
    // (walls, an even number of cells) repeats the last one: only a layer that
    // does not exist reads it, but that layer shares its pair with face n, and
    // the two choose their compatibility rule together.
    const int gvv = v == 0 ? 0 : (v == 1 ? 1 + d : (v == 2 ? 1 + P : (v == 3 ? 1 + S : 4)));
    const float* src = a.q + gvv * g.P + (long long)f0 * sn + (min(p0 - 2 + hp, nP + 1) + kGhost) * sp +
                       (long long)kGhost * ss;
    const unsigned dst = (unsigned)__cvta_generic_to_shared(cells + v * (March::PLANES * HP) + hp);
    const int planes = v < 5 ? min(March::PLANES, (layers - f0 + 1) / 2 * 2 + 5) : 0, last = nd + 5 - f0;
    auto stage = [&](int row) {
      const float* q = src + (long long)row * ss;
      const unsigned to = dst + (row & 1) * (March::CELLS * 4);
      auto copy = [&](int j) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to + j * (HP * 4)), "l"(q) : "memory");
      };
      if (planes == March::PLANES && last >= March::PLANES - 1) {
#pragma unroll
        for (int j = 0; j < March::PLANES; ++j, q += sn) copy(j);
      } else {
#pragma unroll
        for (int j = 0; j < March::PLANES; ++j) {
          if (j < planes) copy(j);
          if (j < last) q += sn;
        }
      }
    };
    stage(s0 - 2);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const float* mine = cells + 2 * v * HP + hp;  // cell f - 3 of column hp, variable 0
#pragma unroll 1
    for (int r = s0 - 2; r < s1 + 2; ++r) {
      if (r + 1 < s1 + 2) stage(r + 1);
      const int slot = (r - s0 + 2) & 3;
      if (live) {
        // ---------------- A: face fields of row r ----------------
        float2 Q0[5], D0[5];
        {
          const float* c = mine + (r & 1) * March::CELLS;
          float2 w[5][6];
#pragma unroll
          for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int k = 0; k < 6; ++k)
              w[i][k] = make_float2(c[(i * March::PLANES + k) * HP], c[(i * March::PLANES + k + 1) * HP]);
          face_fields_smooth_linear_x2(w, r6, a.gas, Q0, D0);
        }
        if (r >= s0 + 2) {
          // ---------------- B: pass along S for row r - 2 ----------------
          const DerivCoef cS(wS[r - 2 + kGhost]);
          const float2* r0 = ring + slot * (NFF * NPT) + tid;              // row r - 4
          const float2* r1 = ring + ((slot + 1) & 3) * (NFF * NPT) + tid;  // r - 3
          const float2* r2 = ring + ((slot + 2) & 3) * (NFF * NPT) + tid;
          const float2* r3 = ring + ((slot + 3) & 3) * (NFF * NPT) + tid;
          float2* o = outb + (r & 1) * (March::NOUT * NPT) + tid;
#pragma unroll
          for (int i = 0; i < 5; ++i) {
            float2 val[2], dv[2], n[2];
            tangential_linear_scaled_x2(r0[i * NPT], r1[i * NPT], r2[i * NPT], r3[i * NPT], Q0[i], cS, val, dv);
            tangential_linear_val_x2(r0[(5 + i) * NPT], r1[(5 + i) * NPT], r2[(5 + i) * NPT], r3[(5 + i) * NPT],
                                     D0[i], n);
#pragma unroll
            for (int m = 0; m < 2; ++m) {
              o[(15 * m + i) * NPT] = val[m];
              o[(15 * m + 5 + i) * NPT] = dv[m];
              o[(15 * m + 10 + i) * NPT] = n[m];
            }
          }
        }
        float2* rn = ring + slot * (NFF * NPT) + tid;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
          rn[i * NPT] = Q0[i];
          rn[(5 + i) * NPT] = D0[i];
        }
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();  // row r's pass along S and row r + 1's cells are there
    }
    __syncthreads();
  } else {
    // C: face pair (layers fo, fo + 1; column ip) at the S abscissa m; the two
    // abscissae sit in the halves of a warp, which exchange their sums so that
    // each stores one layer.
    const int ct = tid - March::MAKERS, lane = ct & 31, m = lane >> 4;
    const int lp = ct / (2 * March::TP), ip = ((ct >> 5) & 1) * 16 + (lane & 15);
    const int fo = f0 + 2 * lp;
    const int at = lp * HP + ip + 2;
    const bool live = p0 + ((ct >> 5) & 1) * 16 < nP && fo < layers;  // some face of the warp exists
    const bool face = p0 + ip < nP && fo + m < layers;
    const DerivCoef cP(wP[min(p0 + ip, nP - 1) + kGhost]);
    const long long FS = (long long)(g.n[0] + (d == 0)) * (g.n[1] + (d == 1)) * (g.n[2] + (d == 2));
    // Face-flux layout: x fastest for the y and z faces, y fastest ([z][x][y])
    // for the x faces.
    const long long ox = d == 0 ? (long long)g.n[1] : 1LL, oy = d == 0 ? 1LL : (long long)g.n[0],
                    oz = (long long)(g.n[0] + (d == 0)) * (g.n[1] + (d == 1));
    const auto ostride = [&](int axis) { return axis == 0 ? ox : (axis == 1 ? oy : oz); };
    const long long fstep = ostride(d), rstep = ostride(S);
    long long fi = (long long)s0 * rstep + (long long)(fo + m) * fstep + (p0 + ip) * ostride(P);
    __syncthreads();
#pragma unroll 1
    for (int r = s0 - 2; r <= s1 + 2; ++r) {
      const int s = r - 3;  // the row whose pass along S the previous step made
      if (s >= s0 && live) {
        // ---------------- C: pass along P and flux of row s ----------------
        float2 Fs[10];
#pragma unroll
        for (int i = 0; i < 10; ++i) Fs[i] = make_float2(0.f, 0.f);
        const float2* o = outb + (s & 1) * (March::NOUT * NPT) + 15 * m * NPT + at;
        PointStateX2 pt[2];
#pragma unroll
        for (int i = 0; i < 5; ++i) {
          const float2* sv = o + i * NPT;
          const float2* sd = o + (5 + i) * NPT;
          const float2* sl = o + (10 + i) * NPT;
          float2 v[2], dv[2], ds[2], dn[2];
          tangential_linear_scaled_x2(sv[-2], sv[-1], sv[0], sv[1], sv[2], cP, v, dv);
          tangential_linear_val_x2(sd[-2], sd[-1], sd[0], sd[1], sd[2], ds);
          tangential_linear_val_x2(sl[-2], sl[-1], sl[0], sl[1], sl[2], dn);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            pt[k].q[i] = v[k];
            pt[k].dq[0][i] = dn[k];
            pt[k].dq[1][i] = dv[k];
            pt[k].dq[2][i] = ds[k];
          }
        }
        flux_smooth_x2<STAGE == 1>(pt[0], a.gas, Fs);
        flux_smooth_x2<STAGE == 1>(pt[1], a.gas, Fs);
#pragma unroll
        for (int k = STAGE == 1 ? 0 : 1; k < 2; ++k) {
          // The second stage needs dF only (Eq. (6)); its F planes are not written.
#pragma unroll
          for (int i = 0; i < 5; ++i) {
            const float2 x = Fs[5 * k + i];
            const float sum = 0.25f * ((m ? x.y : x.x) + __shfl_xor_sync(0xffffffffu, m ? x.x : x.y, 16));
            float* out = a.fd + (5 * k + gv[i]) * FS + fi;
            if (face) *out = sum;
            if (face && fo + m == 0 && layers == nd) out[nd * fstep] = sum;  // periodic: face n is face 0
          }
        }
        fi += rstep;
      }
      __syncthreads();
    }
  }
  return s1 - s0;
}

// Body of one block: `sweeps` the arguments, b the block.  The rows of all
// tiles of the three directions form one sequence (gx tiles along P, gy layer
// groups along n, nS rows each; direction d starts at row start[d]) and every
// block takes `share` consecutive rows of it, through as many tiles as they
// span: the blocks finish together whatever the grid.
template <int STAGE>
__device__ __forceinline__ void march_block(const SweepArgs3<float>& sweeps, int b) {
  int row = b * sweeps.share;
  const int end = min(row + sweeps.share, sweeps.start[3]);
#pragma unroll 1
  while (row < end) row += march_rows<STAGE>(sweeps, row, end - row);
}


template <int STAGE>
__global__ void __launch_bounds__(March::THREADS, 1)
    k_march(const __grid_constant__ SweepArgs3<float> sweeps) {
  march_block<STAGE>(sweeps, blockIdx.x);
}

}  // namespace hgks
