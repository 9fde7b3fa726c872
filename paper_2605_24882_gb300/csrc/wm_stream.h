// Streaming stencil kernels: the operator-type steps of the float solves on
// levels with a stencil form.
//
// A block owns a strip of kBU columns of one patch's local DOF grid, a chunk of
// its rows and up to TPB tiles of 32 systems (lane = system); warp = column.
// It streams down the window rows of the extended grid (halo cells from the
// neighbouring patch, or wrapped): cp.async copies keep the next kD rows on
// their way into a shared-memory ring, with all that the row's step needs (ids
// further ahead), so that no step waits for a load from global memory; each
// value of a row, read once per column that needs it, is added to the 2p+1
// output rows it belongs to, whose running sums stay in registers.  The
// coefficients of a window row (for every output it feeds, pairs (S, M)) lie
// next to each other in a table made for this order; a load of a coefficient
// serves the block's tiles.
//
// NSH = 0: the lanes of a tile may have any shifts.  S z and M z are summed as
// one packed pair (FFMA2: one instruction per tap, tile and output, the
// coefficient pair as it lies in memory); the shift enters once per output.
// NSH = 1: the tiles of the block have one shift.  The warp combines
// A = S + sigma M of its column one row ahead and one packed instruction serves
// two tiles.
//
// What bounds it: the shared-memory pipe (72% busy; per output and tile 5 window
// reads, 13 / 4 coefficient reads of two wavefronts each, the inputs' copies and
// reads) and latency at 16 warps per SM, which the 128 registers of the running
// sums of four tiles allow.  The tile-at-a-time kernel it replaces read every
// window value 2p+1 times and the coefficients once per tile (26 load wavefronts
// and 105 instructions per output against 16 and 60).  Chebyshev step, level 0 of
// the 64 x 64 sphere (p = 2), 568 tiles in runs of eight of one shift: 1.83 -> 1.47 ms
// (3.2 -> 4.0 TB/s); 256 x 256 torus (p = 3), 72 tiles in such runs 1.09 -> 0.66 ms.
// Mixed shifts, rate of the level-0 smoothing: 213 systems on the 256 x 256 sphere
// 1.2 -> 3.1 TB/s, 1136 on the 128 x 128 bicubic one 1.05 -> 1.95.
// Loads straight to registers a row ahead were slower (2.6 ms): the six load
// scoreboards of a warp make the first use of any value wait for all of them.
#pragma once

#include <algorithm>
#include <vector>

#include "wm_solver.h"
#include "wm_stencil.h"

namespace {

constexpr int kBU = 8;      // columns of a block, one warp each
constexpr int kD = 3;       // window rows on their way (two: 1-3% slower)
constexpr int kNST = kD + 1;
// Rows whose products a dot sums in float before it goes on in double.  The chunks of
// the kernels that form dots are multiples of it, so that a system's float sums do not
// depend on the launch's shape, that is, on how many tiles share the batch.
constexpr int kGrp = 8;
constexpr int kBlocks = 2, kBlocks1 = 4;  // blocks per SM of four tiles and of one (register budgets 128 and 64)

// what a window row holds for one column: the coefficients (S, M) of every
// output it feeds by cell, then output row; diagonal and row (32 x DOF, or -1)
// of the output that this window row completes
template <int P>
struct __align__(16) ColRow {
  static constexpr int SW = 2 * P + 1, S2 = SW * SW;
  static_assert(S2 % 2 == 1, "the diagonal lies beside the last coefficient");
  float2 coef[S2];
  float2 diag;
  int own;
  int pad[(S2 * 8 + 12) % 16 == 0 ? 4 : (16 - (S2 * 8 + 12) % 16) / 4];
};

struct StreamGeo {
  int N, nlv, ELV, EU, ncol, nbu, nvc, VH, items;
  const int32_t* ext;   // [np][ELV][EU]  32 x cell ids (0: no cell), row stride padded to whole blocks
  const int32_t* done;  // [np][ELV][EU]  by window row: 32 x the row (0: none) that it completes in this column
  const float2* dext;   // [np][ELV][EU]  (dS, dM) of the cells
  const void* cols;     // [np][ELV][ncol] ColRow
};

// cp.async of 4, 8 and 16 bytes
__device__ __forceinline__ void cp8(unsigned smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(smem), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp4(unsigned smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp16(unsigned smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// dot accumulator: a few products in float, then added in double
struct FAcc {
  double d = 0.0;
  float f = 0.f;
  __device__ __forceinline__ void add(float v) { f += v; }
  __device__ __forceinline__ void flush() {
    d += (double)f;
    f = 0.f;
  }
};

// 1 / d: the hardware's approximation improved by one Newton step
// x (2 - d x), which leaves it within an ulp (d > 0, a diagonal of S + sigma M)
__device__ __forceinline__ float recip(float d) {
  float x;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(d));
  return fmaf(x, fmaf(-d, x, 1.f), x);
}

// rows of an output that the epilogue reads besides the window
template <int MODE>
struct StIn {
  static constexpr int value = MODE == ST_CHEBDOT ? 3 : MODE == ST_CHEB ? 2 : MODE == ST_RESID ? 1 : 0;
};
// shared memory: kNST stages (a window row and what its step needs, byte
// offsets within a stage), combined rows, ids
template <int P, int MODE, int NSH, int TPB>
struct StreamLayout {
  static constexpr int CW = kBU + 2 * P;                 // cells of a window row
  static constexpr int NCELL = (CW + kBU - 1) / kBU;     // cells a warp copies
  static constexpr int CELL = TPB * 32 * (int)sizeof(float);  // bytes of a cell
  static constexpr int NIN = StIn<MODE>::value;
  static constexpr int ORW = CW * CELL;                  // inputs of the output rows, by warp
  static constexpr int COL = ORW + NIN * kBU * CELL;     // ColRow of the columns
  static constexpr int DCL = COL + kBU * (int)sizeof(ColRow<P>);  // ST_CHEB1: diagonals of the cells
  static constexpr int STAGE = DCL + (MODE == ST_CHEB1 ? kBU * NCELL * (int)sizeof(float2) : 0);
  static constexpr int NID = 8;                          // rows of ids (at least 2 kD + 1, a power of two)
  static_assert(NID >= 2 * kD + 1, "ring of ids");
  static constexpr int CU = ColRow<P>::S2 + 1;           // combined row: A of every tap, Chebyshev weight
  static constexpr int COMB = kNST * STAGE;
  static constexpr int CHALF = NSH * kBU * CU * (int)sizeof(float2);  // one of two
  static constexpr int IDS = COMB + 2 * CHALF;           // [NID][kBU] int4
  static constexpr size_t total = (size_t)IDS + (size_t)NID * kBU * 4 * sizeof(int);
  static_assert(STAGE % 16 == 0 && CHALF % 16 == 0 && COL % 16 == 0 && DCL % 16 == 0, "aligned regions");
};
template <int P, int MODE, int NSH, int TPB>
__global__ void __launch_bounds__(kBU * 32, TPB == 1 ? kBlocks1 : kBlocks)
    k_stream(const StreamGeo G, const double* __restrict__ sigma, const float2* __restrict__ ctab,
             const int* __restrict__ sid, int kstep, const float* __restrict__ z, const float* __restrict__ r,
             const float* prev, const float* __restrict__ q, float* out, float* __restrict__ out1,
             const int2* __restrict__ groups, int g0, const int* __restrict__ tile_active, double* __restrict__ part,
             double* __restrict__ part2) {
  wm_wait_previous();
  using LY = StreamLayout<P, MODE, NSH, TPB>;
  using CR = ColRow<P>;
  constexpr int SW = CR::SW, S2 = CR::S2, CW = LY::CW, NIN = LY::NIN, STAGE = LY::STAGE, CELL = LY::CELL;
  constexpr bool CHEB = MODE == ST_CHEB || MODE == ST_CHEBDOT;
  constexpr bool CENTRE = MODE != ST_RESID;       // the input at the output row is needed
  constexpr bool DOT = MODE == ST_APPLY || MODE == ST_CHEBDOT;
  constexpr int NCELL = LY::NCELL, NID = LY::NID, CU = LY::CU;
  constexpr int NS = NSH == 0 ? TPB : 1;       // shifts that a lane keeps
  static_assert((TPB == 4 || (TPB == 1 && NSH == 0)) && NCELL == 2, "the copies and the ids per row and warp below");
  extern __shared__ __align__(16) unsigned char smraw[];
  const int lane = threadIdx.x, w = __shfl_sync(0xffffffffu, (int)threadIdx.y, 0);
  const int item = blockIdx.x;
  const int bu = item % G.nbu;
  const int vc = (item / G.nbu) % G.nvc, m = item / (G.nbu * G.nvc);
  const int2 grp = TPB == 1 ? make_int2(g0 + blockIdx.y, 1) : groups[g0 + blockIdx.y];  // (first tile, count)
  const int t0 = grp.x;
  // src: a tile that is not to be computed stands in for one that is: the same
  // inputs, shift and stores
  int src[TPB];
  {
    unsigned act = 0;
#pragma unroll
    for (int k = 0; k < TPB; ++k)
      if (k < grp.y && tile_active[t0 + k]) act |= 1u << k;
    if (act == 0) return;
    const int first = __ffs(act) - 1;
#pragma unroll
    for (int k = 0; k < TPB; ++k) src[k] = act >> k & 1 ? k : first;
  }
  const int v0 = vc * G.VH;
  const int steps = min(G.nlv - v0, G.VH) + 2 * P;  // window rows
  const int col = bu * kBU + w;
  const bool mine = col < G.ncol;                   // this warp's column exists
  // shift of lane and tile (NSH = 0) or of the block
  float sg[NS], c1[NS], c2[NS], c0[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const int g = (t0 + src[k]) * 32 + lane;
    sg[k] = (float)sigma[g];
    c1[k] = c2[k] = c0[k] = 0.f;
    if constexpr (CHEB) {
      const float2 c = ctab[sid[g] * WM_MAX_CHEB + kstep];
      c1[k] = kstep == 0 ? 0.f : c.x;
      c2[k] = c.y;
    }
    if constexpr (MODE == ST_CHEB1) {
      // steps 0 and 1 from z = 0: with z1 = c20 Dinv r the second step is
      // z1 (1 + c1 + c2 / c20) - c2 Dinv A z1
      c0[k] = ctab[sid[g] * WM_MAX_CHEB].y;
      const float2 c = ctab[sid[g] * WM_MAX_CHEB + 1];
      c1[k] = 1.f + c.x + c.y / c0[k];
      c2[k] = c.y;
    }
  }
  auto sh = [](int k) { return NSH == 0 ? k : 0; };  // shift of tile k
  // running pointers: ids of the row to copy next (4 bytes by each of four
  // lanes: the warp's cells w, w + kBU, .. < CW, others repeating the first, and
  // the row that the window row completes), the column's ColRow, the cells' diagonals
  const size_t strip = ((size_t)m * G.ELV + v0) * G.EU + bu * kBU + w;
  const int32_t* ip = (lane < 3 ? G.ext + (w + lane * kBU < CW ? lane * kBU : 0) : G.done) + strip;
  const float2* dp = G.dext + strip + (w + lane * kBU < CW ? lane * kBU : 0);
  const char* cp = reinterpret_cast<const char*>(reinterpret_cast<const CR*>(G.cols) +
                                                 ((size_t)m * G.ELV + v0) * G.ncol + col) + lane * 16;
  const unsigned cstep = (unsigned)G.ncol * (unsigned)sizeof(CR);
  const size_t tb = (size_t)t0 * G.N * 32;
  const unsigned ts = (unsigned)G.N * 32u;  // tile stride
  // this lane's part of a row of 32 systems: 16-byte chunk lane % 8; with four
  // tiles of tile lane / 8, with one of the cells (0, 1), r (2) and prev (3)
  size_t cofs = tb + (size_t)((lane % 8) * 4);
  const int lq = lane / 8;
  if constexpr (TPB == 4) {
#pragma unroll
    for (int k = 0; k < TPB; ++k)
      if (lq == k) cofs += (unsigned)src[k] * ts;
  }
  z += cofs;
  if constexpr (NIN > 0) r += cofs;
  if constexpr (NIN > 1) prev += cofs;
  if constexpr (NIN > 2) q += cofs;
  const float* one = lq < 2 || NIN == 0 ? z : lq == 2 || NIN == 1 ? r : prev;  // TPB = 1: this lane's source
  const bool one_on = lq == 0 || (lq == 1 && w + kBU < CW) || (lq == 2 && NIN > 0 && mine) || (lq == 3 && NIN > 1 && mine);
  const unsigned one_to = lq < 2 ? (w + lq * kBU) * CELL : LY::ORW + (w * NIN + lq - 2) * CELL;
  float *ot[TPB], *ot1[TPB];
#pragma unroll
  for (int k = 0; k < TPB; ++k) {
    ot[k] = out + tb + (unsigned)src[k] * ts + lane;
    ot1[k] = MODE == ST_CHEB1 ? out1 + tb + (unsigned)src[k] * ts + lane : nullptr;
  }
  const unsigned sbase = (unsigned)__cvta_generic_to_shared(smraw);
  const unsigned sid_ = sbase + LY::IDS + w * 16;

  // ids of row s
  auto copy_ids = [&](int s) {
    if (s < steps && lane < 4) cp4(sid_ + (s & (NID - 1)) * (kBU * 16) + lane * 4, ip);
    ip += G.EU;
  };
  // window row s (its ids have arrived) into the stage at byte so, and the ids of row s + kD
  auto copy_row = [&](int s, unsigned so) {
    if (s < steps) {
      const uint4 id = *reinterpret_cast<const uint4*>(smraw + LY::IDS + ((s & (NID - 1)) * kBU + w) * 16);
      if constexpr (TPB == 4) {
        const unsigned st = sbase + so + lane * 16;
        cp16(st + w * CELL, z + id.x);
        if (w + kBU < CW) cp16(st + (w + kBU) * CELL, z + id.y);
        if (mine) {
          if constexpr (NIN > 0) cp16(st + LY::ORW + w * (NIN * CELL), r + id.w);
          if constexpr (NIN > 1) cp16(st + LY::ORW + w * (NIN * CELL) + CELL, prev + id.w);
          if constexpr (NIN > 2) cp16(st + LY::ORW + w * (NIN * CELL) + 2 * CELL, q + id.w);
        }
      } else {
        const unsigned st = sbase + so + (lane % 8) * 16;
        if (one_on) cp16(st + one_to, one + (lq == 0 ? id.x : lq == 1 ? id.y : id.w));
        if constexpr (NIN > 2)
          if (lane < 8 && mine) cp16(st + LY::ORW + (w * NIN + 2) * CELL, q + id.w);
      }
      if (mine) {
        const unsigned st = sbase + so + lane * 16;
        if (lane < (int)(sizeof(CR) / 16)) cp16(st + LY::COL + w * (int)sizeof(CR), cp);
      }
      if constexpr (MODE == ST_CHEB1) {
        if (lane < NCELL) cp8(sbase + so + LY::DCL + (w * NCELL + lane) * 8, dp);
        dp += G.EU;
      }
      cp += cstep;
    }
    copy_ids(s + kD);
    cp_commit();
  };
  // A = S + sigma M of this warp's column in the stage at so, and the Chebyshev weight
  auto combine = [&](unsigned so, int half) {
    if constexpr (NSH > 0) {
#pragma unroll
      for (int e0 = 0; e0 < CU; e0 += 32) {
        const int e = e0 + lane;
        if (e < CU) {
          // (entry S2: the diagonal)
          const float2 v = reinterpret_cast<const float2*>(smraw + so + LY::COL + w * (int)sizeof(CR))[e];
          float a = v.x + sg[0] * v.y;
          if ((CHEB || MODE == ST_CHEB1) && e == S2) a = c2[0] * recip(a);
          reinterpret_cast<float2*>(smraw + LY::COMB + half * LY::CHALF)[w * CU + e] = make_float2(a, a);
        }
      }
    }
  };
#pragma unroll
  for (int s = 0; s < kD; ++s) copy_ids(s);
  cp_commit();
  cp_wait<0>();
  __syncwarp();
#pragma unroll
  for (int s = 0; s < kD; ++s) copy_row(s, s * STAGE);
  if constexpr (NSH > 0) {
    cp_wait<kD - 1>();
    __syncwarp();
    if (mine) combine(0, 0);
  }

  // running sums: (S z, M z) per tile, or two tiles' A z
  float2 acc[SW][NSH == 0 ? TPB : TPB / 2];
  float zr[SW][TPB];  // the input at the column, a window row per slot
  FAcc dot[TPB], dot2[TPB];
  unsigned so = 0, sprev = kD * STAGE;  // stages of rows s and s - 1
  auto flush = [&]() {
#pragma unroll
    for (int k = 0; k < TPB; ++k) {
      dot[k].flush();
      if constexpr (MODE == ST_CHEBDOT) dot2[k].flush();
    }
  };

  for (int sb = 0; sb < steps; sb += SW) {
#pragma unroll
    for (int u = 0; u < SW; ++u) {
      const int s = sb + u;
      if (s >= steps) break;
      // this thread's copies of row s (NSH > 0: and of row s + 1), ids of row s + kD
      cp_wait<NSH == 0 ? kD - 1 : kD - 2>();
      if constexpr (MODE == ST_CHEB1) {  // r of this warp's cells becomes z1 = c20 Dinv r
        __syncwarp();
#pragma unroll
        for (int i = 0; i < NCELL; ++i)
          if (w + i * kBU < CW) {
            const float2 d = *reinterpret_cast<const float2*>(smraw + so + LY::DCL + (w * NCELL + i) * 8);
            float f[NS];
#pragma unroll
            for (int k = 0; k < NS; ++k) f[k] = c0[k] * recip(d.x + sg[k] * d.y);
            float* p = reinterpret_cast<float*>(smraw + so + (w + i * kBU) * CELL) + lane;
#pragma unroll
            for (int k = 0; k < TPB; ++k) p[k * 32] *= f[sh(k)];
          }
      }
      __syncthreads();  // row s is there, row s - 1 is no longer read
      copy_row(s + kD, sprev);
      const unsigned sc_ = so;
      sprev = so;
      so = so == kD * STAGE ? 0 : so + STAGE;
      if (!mine) continue;
      if (DOT && s > 2 * P && (s - 2 * P) % kGrp == 0) flush();  // the last kGrp output rows' products
      if (NSH > 0 && s + 1 < steps) combine(so, (s + 1) & 1);
      const float* zw = reinterpret_cast<const float*>(smraw + sc_ + w * CELL) + lane;
      const CR& R = *reinterpret_cast<const CR*>(smraw + sc_ + LY::COL + w * (int)sizeof(CR));
      const float4* cf = NSH == 0 ? reinterpret_cast<const float4*>(R.coef)
                                  : reinterpret_cast<const float4*>(smraw + LY::COMB + (s & 1) * LY::CHALF) +
                                        w * (CU / 2);
      float4 c4 = make_float4(0.f, 0.f, 0.f, 0.f);  // the last one holds the diagonal or the weight too
#pragma unroll
      for (int du = 0; du < SW; ++du) {
        float zv[TPB];
#pragma unroll
        for (int k = 0; k < TPB; ++k) {
          zv[k] = zw[(du * TPB + k) * 32];
          if (CENTRE && du == P) zr[u][k] = zv[k];
        }
#pragma unroll
        for (int dv = 0; dv < SW; ++dv) {
          const int sl = (u - dv + SW) % SW;  // slot of output row s - dv
          const int e = du * SW + dv;
          if (e % 2 == 0) c4 = cf[e / 2];
          const float2 a = e % 2 == 0 ? make_float2(c4.x, c4.y) : make_float2(c4.z, c4.w);
          if constexpr (NSH == 0) {
#pragma unroll
            for (int k = 0; k < TPB; ++k) {
              const float2 zz = make_float2(zv[k], zv[k]);
              acc[sl][k] = e == 0 ? __fmul2_rn(a, zz) : __ffma2_rn(a, zz, acc[sl][k]);
            }
          } else {
#pragma unroll
            for (int k = 0; k < TPB / 2; ++k) {
              const float2 zz = make_float2(zv[2 * k], zv[2 * k + 1]);
              acc[sl][k] = e == 0 ? __fmul2_rn(a, zz) : __ffma2_rn(a, zz, acc[sl][k]);
            }
          }
        }
      }
      const int own = s >= 2 * P ? R.own : -1;  // the output row that row s completes
      if (own < 0) continue;
      const int sl = (u + 1) % SW;              // output row s - 2p
      const int sc = (u - P + SW) % SW;         // its centre row
      const float* orr = reinterpret_cast<const float*>(smraw + sc_ + LY::ORW + w * (NIN * CELL)) + lane;
#pragma unroll
      for (int k = 0; k < TPB; ++k) {
        float az, wt;  // A z and c2 / diagonal
        if constexpr (NSH == 0) {
          az = acc[sl][k].x + sg[k] * acc[sl][k].y;
          wt = CHEB || MODE == ST_CHEB1 ? c2[k] * recip(c4.z + sg[k] * c4.w) : 0.f;
        } else {
          az = k % 2 == 0 ? acc[sl][k / 2].x : acc[sl][k / 2].y;
          wt = c4.z;
        }
        const float rv = NIN > 0 ? orr[k * 32] : 0.f;
        float res;
        if constexpr (CHEB) {
          const float zc = zr[sc][k];
          const float pv = orr[(TPB + k) * 32];
          res = zc + c1[sh(k)] * (zc - pv) + wt * (rv - az);
          if constexpr (MODE == ST_CHEBDOT) {
            dot[k].add(rv * res);
            dot2[k].add(res * orr[(2 * TPB + k) * 32]);
          }
        } else if constexpr (MODE == ST_CHEB1) {
          const float z1 = zr[sc][k];
          ot1[k][(unsigned)own] = z1;
          res = c1[sh(k)] * z1 - wt * az;
        } else if constexpr (MODE == ST_RESID) {
          res = rv - az;
        } else {
          res = az;
          dot[k].add(zr[sc][k] * az);
        }
        ot[k][(unsigned)own] = res;
      }
    }
  }
  if constexpr (DOT) {  // the block's partial sums, warps in order
    flush();
    double* red = reinterpret_cast<double*>(smraw);  // [TPB][kBU][32]
    static_assert(LY::total >= sizeof(double) * TPB * kBU * 32, "reduction buffer");
    cp_wait<0>();
    for (int h = 0; h < (MODE == ST_CHEBDOT ? 2 : 1); ++h) {
      __syncthreads();
#pragma unroll
      for (int k = 0; k < TPB; ++k) red[(k * kBU + w) * 32 + lane] = h == 0 ? dot[k].d : dot2[k].d;
      __syncthreads();
      for (int k = w; k < TPB; k += kBU) {
        if (!(k < grp.y && tile_active[t0 + k])) continue;
        double a = 0.0;
#pragma unroll
        for (int y = 0; y < kBU; ++y) a += red[(k * kBU + y) * 32 + lane];
        (h == 0 ? part : part2)[((size_t)(t0 + k) * G.items + item) * 32 + lane] = a;
      }
    }
  }
}

// Shape of a launch.  Where the strips x groups of four tiles give every SM a block,
// blocks of four tiles (every coefficient read once for the four) and chunks for two
// waves of blocks (one wave of longer chunks: 3% slower on the 128 x 128 bicubic sphere).
// Below that a block of one tile, which does each step (a window row) in a fraction of
// the time, may be faster, and shorter chunks, at 2p more rows each: the shape of least
// time by a model in which an SM takes its share of the blocks and a step lasts the
// block's latency or, with several blocks on the SM, their work (cycles, measured on the
// 64 x 64 sphere; 71 systems there: 8.4 -> 8.0 ms a call against two waves throughout).
constexpr int kSMs = 152;
struct StCost {
  int resident;         // blocks that an SM holds
  double lat, work;     // cycles of a step: alone on its SM, and of SM time
};
constexpr StCost kCost[2][2] = {{{kBlocks, 900.0, 1000.0}, {kBlocks1, 400.0, 400.0}},    // p = 2: four tiles, one
                                {{kBlocks, 1700.0, 1900.0}, {kBlocks1, 700.0, 900.0}}};  // p = 3
constexpr int kWantBlocks = 2 * kSMs * kBlocks;
constexpr int kMinRows = 6, kMinRows1 = 3;  // rows of a chunk at least: many strips, few
// cycles of nvc chunks of VH rows on `base` strips
inline double st_cost(const StCost& c, int64_t base, int nvc, int VH, int p) {
  const int64_t n = (base * nvc + kSMs - 1) / kSMs;  // blocks per SM
  return (VH + 2 * p + 4) * std::max(c.lat * (double)((n + c.resident - 1) / c.resident), c.work * (double)n);
}

inline int strips(const wm_level& L) { return (L.nlu + kBU - 1) / kBU; }

StreamGeo stream_geo(const wm_level& L, int np, int p, const StreamTiles& st, bool dot, bool* one) {
  StreamGeo G;
  G.N = L.N;
  G.nlv = L.nlv;
  G.ELV = L.nlv + 2 * p;
  G.ncol = L.nlu;
  G.nbu = strips(L);
  G.EU = G.nbu * kBU + 2 * p;
  const int64_t strip = (int64_t)np * G.nbu, base4 = strip * std::max(1, st.n[0] + st.n[1]);
  *one = false;
  auto split = [&](int chunks) {
    G.VH = (L.nlv + chunks - 1) / chunks;
    if (dot) G.VH = (G.VH + kGrp - 1) / kGrp * kGrp;
    G.nvc = (L.nlv + G.VH - 1) / G.VH;
  };
  if (base4 >= kSMs) {
    const int64_t want = (kWantBlocks + base4 - 1) / base4;
    split((int)std::min<int64_t>(std::max(1, L.nlv / kMinRows), std::max<int64_t>(1, want)));
  } else {
    double best = 0.0;
    int chunks = 1;
    for (int k = 0; k < 2; ++k)
      for (int c = 1; c <= std::max(1, L.nlv / kMinRows1); ++c) {
        split(c);
        const double t = st_cost(kCost[p == 2 ? 0 : 1][k], k == 0 ? base4 : strip * std::max(1, st.tiles), G.nvc, G.VH, p);
        if (best == 0.0 || t < best) {
          best = t;
          *one = k == 1;
          chunks = c;
        }
      }
    split(chunks);
  }
  G.items = np * G.nbu * G.nvc;
  G.ext = L.d_st_ext.p;
  G.done = L.d_st_done.p;
  G.dext = L.d_st_dext.p;
  G.cols = L.d_st_cols.p;
  return G;
}

template <int P, int MODE, int NSH, int TPB>
int launch_stream_n(const StreamArgs& a, const StreamGeo& G, const int2* groups, int n) {
  if (n <= 0) return WM_OK;
  constexpr size_t sm = StreamLayout<P, MODE, NSH, TPB>::total;
  static bool configured = false;
  if (!configured) {
    WM_CUDA(cudaFuncSetAttribute(k_stream<P, MODE, NSH, TPB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    configured = true;
  }
  for (int g0 = 0; g0 < n; g0 += 65535) {  // grid.y limit
    WM_TRY(wm_launch_next(a.cat, (k_stream<P, MODE, NSH, TPB>), dim3(G.items, std::min(65535, n - g0)), dim3(32,
        kBU), sm, a.s, G, a.sigma, a.ctab, a.sid, a.kstep, a.z, a.r, a.prev, a.q, a.out, a.out1, groups, g0,
        a.tile_active, a.part, a.part2));
    WM_CUDA(cudaGetLastError());
  }
  return WM_OK;
}
template <int P, int MODE>
int launch_stream(const StreamArgs& a) {
  const int* n = a.st.n;
  bool one = false;
  const StreamGeo G = stream_geo(*a.L, a.np, P, a.st, MODE == ST_APPLY || MODE == ST_CHEBDOT, &one);
  if (one) return launch_stream_n<P, MODE, 0, 1>(a, G, nullptr, a.st.tiles);
  WM_TRY((launch_stream_n<P, MODE, 1, kStreamTiles>(a, G, a.st.groups, n[1])));
  return launch_stream_n<P, MODE, 0, kStreamTiles>(a, G, a.st.groups + n[1], n[0]);
}

}  // namespace

template <int P>
int wm_stream_run(int mode, const StreamArgs& a) {
  switch (mode) {
    case ST_CHEB: return launch_stream<P, ST_CHEB>(a);
    case ST_RESID: return launch_stream<P, ST_RESID>(a);
    case ST_APPLY: return launch_stream<P, ST_APPLY>(a);
    case ST_CHEBDOT: return launch_stream<P, ST_CHEBDOT>(a);
    case ST_CHEB1: return launch_stream<P, ST_CHEB1>(a);
  }
  return WM_ERR_INVALID_ARG;
}
