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
// A tile's arithmetic depends on its shifts alone, not on the kernel, the block or the
// tiles beside it: a solve stops at thresholds, and sums formed another way move a
// system across one (a field of a batch by 1e-9 of its norm).  A tile of one shift has
// its rows combined, A = S + sigma M, one sum per output and one weight c2 / diagonal; a
// tile of several shifts sums S z and M z and divides c2 (r - A z) by the diagonal.  Taps
// are added window row by window row, left to right.
// NSH = 2: two pairs of tiles, each of one shift.  The warp combines its column's rows for
// both shifts one row ahead; a packed instruction (FFMA2) per tap serves a tile of each.
// NSH = 0: any tiles.  Several shifts: one FFMA2 per tap, tile and output on the pair
// (S, M) as it lies in memory.  One shift each (`ones`): one FFMA2 for the rows of two
// tiles, in registers, and one for their sums.
//
// What bounds it: the shared-memory pipe (per output and tile 5 window reads, 13 / 4
// coefficient reads of two wavefronts each, the inputs' copies and reads: 16 wavefronts
// and 67 instructions where the tile-at-a-time kernel it replaces took 26 and 105) and
// latency at 16 warps per SM, which the 128 registers of the running sums of four tiles
// allow.  Chebyshev step (16 bytes per DOF and system; in brackets that kernel's time):
// level 0 of the 64 x 64 sphere (p = 2), 568 tiles in runs of eight of one shift 1.52 ms
// (1.86), 4.9 TB/s; 71 tiles of a shift each 0.26 ms (0.41); 256 x 256 torus (p = 3), 72
// tiles in runs of two 0.63 ms (1.10), 3.8 TB/s.  Several shifts in a tile: 213 systems
// on the 256 x 256 sphere 0.44 ms, 3.0 TB/s; 1152 on the 128 x 128 bicubic sphere
// 0.73 ms, 2.6 TB/s.
// Loads straight to registers a row ahead were slower (2.6 ms): the six load
// scoreboards of a warp make the first use of any value wait for all of them.
#pragma once

#include <algorithm>
#include <type_traits>
#include <vector>

#include "wm_quotient.h"
#include "wm_solver.h"
#include "wm_stencil.h"

namespace {

constexpr int kBU = 8;      // columns of a block, one warp each
constexpr int kD = 3;       // window rows on their way (two: 1-3% slower)
constexpr int kNST = kD + 1;
// Rows whose products a dot sums in float before it goes on in double: the row blocks of
// wm_stencil.cu.  The chunks of the kernels that form dots are multiples of it, so that a
// system's float sums do not depend on the launch's shape, that is, on how many tiles
// share the batch.
template <int P>
struct StGrp {
  static constexpr int value = P == 2 ? 6 : 8;
};
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
  __device__ __forceinline__ void add(float a, float b) { f = fmaf(a, b, f); }
  __device__ __forceinline__ void flush() {
    d += (double)f;
    f = 0.f;
  }
};

// rows of an output that the epilogue reads besides the window
template <int MODE, int NSH>
struct StIn {
  static constexpr int value =
      MODE == ST_CHEBDOT ? 3 : MODE == ST_CHEB ? 2 : MODE == ST_RESID || (MODE == ST_CHEB1 && NSH == 0) ? 1 : 0;
};
// shared memory: kNST stages (a window row and what its step needs, byte
// offsets within a stage), combined rows, ids
template <int P, int MODE, int NSH, int TPB>
struct StreamLayout {
  static constexpr int CW = kBU + 2 * P;                 // cells of a window row
  static constexpr int NCELL = (CW + kBU - 1) / kBU;     // cells a warp copies
  static constexpr int CELL = TPB * 32 * (int)sizeof(float);  // bytes of a cell
  static constexpr int NIN = StIn<MODE, NSH>::value;
  static constexpr int ORW = CW * CELL;                  // inputs of the output rows, by warp
  static constexpr int COL = ORW + NIN * kBU * CELL;     // ColRow of the columns
  static constexpr int DCL = COL + kBU * (int)sizeof(ColRow<P>);  // ST_CHEB1: diagonals of the cells
  static constexpr int STAGE = DCL + (MODE == ST_CHEB1 ? kBU * NCELL * (int)sizeof(float2) : 0);
  static constexpr int NID = 8;                          // rows of ids (at least 2 kD + 1, a power of two)
  static_assert(NID >= 2 * kD + 1, "ring of ids");
  // combined row: A of every tap, then two weights of the completed output, each for NSH shifts
  static constexpr int CU = (ColRow<P>::S2 + 2 + 3) / 4 * 4;
  static constexpr int COMB = kNST * STAGE;
  static constexpr int CHALF = NSH * kBU * CU * (int)sizeof(float);  // one of two
  static constexpr int FACT = COMB + 2 * CHALF;  // ST_CHEB1, NSH = 0: [2][kBU * NCELL][TPB] c2_0 / the cells' diagonals
  static constexpr int FHALF = MODE == ST_CHEB1 && NSH == 0 ? kBU * NCELL * TPB * (int)sizeof(float) : 0;
  // shifts and Chebyshev coefficients by tile and lane, where there are no registers for them
  static constexpr bool SPAR = P == 3 && TPB == 4 && NSH == 0;
  static constexpr int PAR = FACT + 2 * FHALF;
  // and the double sums of the dot products by tile, warp and lane
  static constexpr bool SDOT = SPAR && MODE == ST_APPLY;
  static constexpr int DOTS = PAR + (SPAR ? TPB * 32 * (int)sizeof(float4) : 0);
  static constexpr int IDS = DOTS + (SDOT ? TPB * kBU * 32 * (int)sizeof(double) : 0);  // [NID][kBU] int4
  static constexpr size_t total = (size_t)IDS + (size_t)NID * kBU * 4 * sizeof(int);
  static_assert(STAGE % 16 == 0 && CHALF % 16 == 0 && FHALF % 16 == 0 && COL % 16 == 0 && DCL % 16 == 0,
                "aligned regions");
};

// what a launch takes besides the level's tables
struct StreamIo {
  const double* sigma;
  const float2* ctab;
  const int *sid, *tile_active;
  const float *z, *r, *prev, *q;
  float *out, *out1;
  double *part, *part2;
  const int4* groups;
  const int* order;
  int n_one;  // groups [0, n_one) (TPB = 1: tiles) have one shift per tile
  int g0, kstep, pstride;
};

// the tiles of group y (-1: none)
template <int TPB>
__device__ __forceinline__ void stream_tiles_of(const StreamIo& io, int y, int (&tile)[TPB]) {
  if constexpr (TPB == 1) {
    tile[0] = io.order[y];
  } else {
    const int4 g = io.groups[y];
    tile[0] = g.x;
    tile[1] = g.y;
    tile[2] = g.z;
    tile[3] = g.w;
  }
}

// A block's work: one spatial chunk of group y.  ones (NSH = 0): the tiles have one shift each.
template <int P, int MODE, int NSH, int TPB>
__device__ __forceinline__ void stream_block(const StreamGeo& G, const StreamIo& io, int y, bool ones) {
  using LY = StreamLayout<P, MODE, NSH, TPB>;
  using CR = ColRow<P>;
  constexpr int SW = CR::SW, S2 = CR::S2, CW = LY::CW, NIN = LY::NIN, STAGE = LY::STAGE, CELL = LY::CELL;
  constexpr bool CHEB = MODE == ST_CHEB || MODE == ST_CHEBDOT;
  constexpr bool CENTRE = MODE != ST_RESID;       // the input at the output row is needed
  constexpr bool DOT = MODE == ST_APPLY || MODE == ST_CHEBDOT;
  constexpr int NCELL = LY::NCELL, NID = LY::NID, CU = LY::CU, GRP = StGrp<P>::value;
  constexpr int NS = NSH == 0 ? TPB : NSH;        // shifts that a lane keeps
  static_assert((TPB == 4 || (TPB == 1 && NSH == 0)) && (NSH == 0 || NSH == 2) && NCELL == 2,
                "the copies and the ids per row and warp below");
  extern __shared__ __align__(16) unsigned char smraw[];
  const int lane = threadIdx.x, w = __shfl_sync(0xffffffffu, (int)threadIdx.y, 0);
  const int item = blockIdx.x;
  const int bu = item % G.nbu;
  const int vc = (item / G.nbu) % G.nvc, m = item / (G.nbu * G.nvc);
  // src: a tile that is not to be computed stands in for one that is: the same
  // inputs, shift and stores (NSH = 2: for the other one of its shift first)
  int src[TPB], tile[TPB];
  stream_tiles_of(io, y, tile);
  unsigned act = 0;
#pragma unroll
  for (int k = 0; k < TPB; ++k)
    if (tile[k] >= 0 && io.tile_active[tile[k]]) act |= 1u << k;
  if (act == 0) return;
  {
    int first = tile[0];
#pragma unroll
    for (int k = TPB - 1; k >= 0; --k)
      if (act >> k & 1) first = tile[k];
#pragma unroll
    for (int k = 0; k < TPB; ++k)
      src[k] = act >> k & 1 ? tile[k] : NSH == 2 && (act >> (k ^ 1) & 1) ? tile[(k ^ 1) % TPB] : first;
  }
  const int v0 = vc * G.VH;
  const int steps = min(G.nlv - v0, G.VH) + 2 * P;  // window rows
  const int col = bu * kBU + w;
  const bool mine = col < G.ncol;                   // this warp's column exists
  // the shift of tile k: its lane's (NSH = 0) or one of the block's
  auto sh = [](int k) { return NSH == 2 ? k / 2 : k; };
  float sg[NS], c1[NS], c2[NS], c0[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const int g = src[NSH == 2 ? (2 * k) % TPB : k] * 32 + (NSH == 0 ? lane : 0);
    sg[k] = (float)io.sigma[g];
    c1[k] = c2[k] = c0[k] = 0.f;
    if constexpr (CHEB) {
      const float2 c = io.ctab[io.sid[g] * WM_MAX_CHEB + io.kstep];
      c1[k] = io.kstep == 0 ? 0.f : c.x;
      c2[k] = c.y;
    }
    if constexpr (MODE == ST_CHEB1) {  // steps 0 and 1
      c0[k] = io.ctab[io.sid[g] * WM_MAX_CHEB].y;
      const float2 c = io.ctab[io.sid[g] * WM_MAX_CHEB + 1];
      c1[k] = c.x;
      c2[k] = c.y;
    }
  }
  // the parameters of tile k
  float4* const spar = reinterpret_cast<float4*>(smraw + LY::PAR) + lane;  // SPAR: {sg, c1, c2, c0}
  if constexpr (LY::SPAR) {
    if (w == 0)
#pragma unroll
      for (int k = 0; k < TPB; ++k) spar[k * 32] = make_float4(sg[k], c1[k], c2[k], c0[k]);
    __syncthreads();
  }
  auto par = [&](int k) {
    if constexpr (LY::SPAR)
      return spar[k * 32];
    else
      return make_float4(sg[sh(k)], c1[sh(k)], c2[sh(k)], c0[sh(k)]);
  };
  // running pointers: ids of the row to copy next (4 bytes by each of four
  // lanes: the warp's cells w, w + kBU, .. < CW, others repeating the first, and
  // the row that the window row completes), the column's ColRow, the cells' diagonals
  const size_t strip = ((size_t)m * G.ELV + v0) * G.EU + bu * kBU + w;
  const int32_t* ip = (lane < 3 ? G.ext + (w + lane * kBU < CW ? lane * kBU : 0) : G.done) + strip;
  const float2* dp = G.dext + strip + (w + lane * kBU < CW ? lane * kBU : 0);
  const char* cp = reinterpret_cast<const char*>(reinterpret_cast<const CR*>(G.cols) +
                                                 ((size_t)m * G.ELV + v0) * G.ncol + col) + lane * 16;
  const unsigned cstep = (unsigned)G.ncol * (unsigned)sizeof(CR);
  const size_t ts = (size_t)G.N * 32;  // tile stride
  // this lane's part of a row of 32 systems: 16-byte chunk lane % 8; with four
  // tiles of tile lane / 8, with one of the cells (0, 1), r (2) and prev (3)
  const int lq = lane / 8;
  size_t cofs = (size_t)src[0] * ts;
  if constexpr (TPB == 4) {
#pragma unroll
    for (int k = 1; k < TPB; ++k)
      if (lq == k) cofs = (size_t)src[k] * ts;
  }
  cofs += (lane % 8) * 4;
  const float* const one =  // TPB = 1: this lane's source
      (lq < 2 || NIN == 0 ? io.z : lq == 2 || NIN == 1 ? io.r : io.prev) + cofs;
  const bool one_on = lq == 0 || (lq == 1 && w + kBU < CW) || (lq == 2 && NIN > 0 && mine) || (lq == 3 && NIN > 1 && mine);
  const unsigned one_to = lq < 2 ? (w + lq * kBU) * CELL : LY::ORW + (w * NIN + lq - 2) * CELL;
  unsigned row0[TPB];  // first row of 32 systems of the tile stored to
#pragma unroll
  for (int k = 0; k < TPB; ++k) row0[k] = (unsigned)src[k] * (unsigned)G.N;
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
        cp16(st + w * CELL, io.z + (cofs + id.x));
        if (w + kBU < CW) cp16(st + (w + kBU) * CELL, io.z + (cofs + id.y));
        if (mine) {
          if constexpr (NIN > 0) cp16(st + LY::ORW + w * (NIN * CELL), io.r + (cofs + id.w));
          if constexpr (NIN > 1) cp16(st + LY::ORW + w * (NIN * CELL) + CELL, io.prev + (cofs + id.w));
          if constexpr (NIN > 2) cp16(st + LY::ORW + w * (NIN * CELL) + 2 * CELL, io.q + (cofs + id.w));
        }
      } else {
        const unsigned st = sbase + so + (lane % 8) * 16;
        if (one_on) cp16(st + one_to, one + (lq == 0 ? id.x : lq == 1 ? id.y : id.w));
        if constexpr (NIN > 2)
          if (lane < 8 && mine) cp16(st + LY::ORW + (w * NIN + 2) * CELL, io.q + (cofs + id.w));
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
  auto of_shift = [](const float (&v)[NS], int k) {
    float a = v[0];
#pragma unroll
    for (int j = 1; j < NS; ++j)
      if (k == j) a = v[j];
    return a;
  };
  // NSH = 2: A = S + sigma M of this warp's column in the stage at so for both shifts
  // of the block, and the weights of the output that the row completes: c2 / diagonal
  // (ST_CHEB1: c2_0 / diagonal and c2 / diagonal; A times c2_0 / the cell's diagonal).
  // A lane does one division at most.
  auto combine = [&](unsigned so, int half) {
    if constexpr (NSH > 0) {
      float* const tab = reinterpret_cast<float*>(smraw + LY::COMB + half * LY::CHALF) + w * (CU * NSH);
      const float2* const cd = reinterpret_cast<const float2*>(smraw + so + LY::COL + w * (int)sizeof(CR));
      float f0 = 0.f, f1 = 0.f;  // ST_CHEB1: by lane cell (SW: the output) x shift
      if constexpr (MODE == ST_CHEB1) {
        static_assert((SW + 1) * NSH <= 32, "lanes");
        const int i = min(lane / NSH, SW), k = lane % NSH, c = w + i;
        const float2 d = i < SW ? reinterpret_cast<const float2*>(smraw + so + LY::DCL)[(c % kBU) * NCELL + c / kBU]
                                : cd[S2];
        const float dinv = wm_quotient(1.f, fmaf(of_shift(sg, k), d.y, d.x));
        f0 = of_shift(c0, k) * dinv;
        f1 = of_shift(c2, k) * dinv;
      }
#pragma unroll
      for (int e0 = 0; e0 < S2; e0 += 32) {
        const int e = e0 + lane;
        const float2 v = cd[min(e, S2 - 1)];
        float a[NS];
#pragma unroll
        for (int k = 0; k < NSH; ++k) {
          a[k] = fmaf(sg[k], v.y, v.x);
          if constexpr (MODE == ST_CHEB1) a[k] *= __shfl_sync(0xffffffffu, f0, min(e, S2 - 1) / SW * NSH + k);
        }
        if (e < S2) reinterpret_cast<float2*>(tab)[e] = make_float2(a[0], a[NS - 1]);
      }
      if constexpr (CHEB) {
        const int k = lane - (32 - NSH);  // the last lanes have no entry (p = 3: of the second pass)
        if (k >= 0) {
          const float2 d = cd[S2];
          tab[S2 * NSH + k] = wm_quotient(of_shift(c2, k), fmaf(of_shift(sg, k), d.y, d.x));
        }
      }
      if constexpr (MODE == ST_CHEB1) {
        const int k = lane - SW * NSH;
        if (k >= 0 && k < NSH) {
          tab[S2 * NSH + k] = f0;
          tab[(S2 + 1) * NSH + k] = f1;
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
    if constexpr (MODE == ST_CHEB1)
      __syncthreads();  // (diagonals of other warps' cells)
    else
      __syncwarp();
    if (mine) combine(0, 0);
  }

  // running sums: (S z, M z) per tile, or A z of two tiles (NSH = 2: k and k + 2; ones:
  // 2k and 2k + 1) or one
  float2 acc[SW][NSH == 0 ? TPB : 2];
  float zr[SW][TPB];  // the input at the column, a window row per slot
  FAcc dot[TPB], dot2[TPB];
  unsigned so = 0, sprev = kD * STAGE;  // stages of rows s and s - 1
  double* const sdot = reinterpret_cast<double*>(smraw + LY::DOTS) + w * 32 + lane;
  if constexpr (LY::SDOT) {
#pragma unroll
    for (int k = 0; k < TPB; ++k) sdot[k * (kBU * 32)] = 0.0;
  }
  auto flush = [&]() {
#pragma unroll
    for (int k = 0; k < TPB; ++k) {
      if constexpr (LY::SDOT) {
        sdot[k * (kBU * 32)] += (double)dot[k].f;
        dot[k].f = 0.f;
      } else {
        dot[k].flush();
      }
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
      if constexpr (MODE == ST_CHEB1 && NSH == 0) {
        __syncwarp();
        const float2* const dcl = reinterpret_cast<const float2*>(smraw + so + LY::DCL) + w * NCELL;
        if (ones) {  // c2_0 / diagonal of this warp's cells
          if (lane < NCELL * TPB) {
            const int k = lane % TPB;
            const float2 d = dcl[lane / TPB];
            float4 pk = par(0);
            if constexpr (LY::SPAR) {
              pk = par(k);
            } else {
#pragma unroll
              for (int j = 1; j < TPB; ++j)
                if (k == j) pk = par(j);
            }
            reinterpret_cast<float*>(smraw + LY::FACT + (s & 1) * LY::FHALF)[w * (NCELL * TPB) + lane] =
                pk.w * wm_quotient(1.f, fmaf(pk.x, d.y, d.x));
          }
        } else {  // their r becomes z1 = c2_0 r / diagonal
#pragma unroll
          for (int i = 0; i < NCELL; ++i)
            if (w + i * kBU < CW) {
              const float2 d = dcl[i];
              float* p = reinterpret_cast<float*>(smraw + so + (w + i * kBU) * CELL) + lane;
#pragma unroll
              for (int k = 0; k < TPB; ++k) {
                const float4 pk = par(k);
                p[k * 32] = wm_quotient(pk.w * p[k * 32], fmaf(pk.x, d.y, d.x));
              }
            }
        }
      }
      __syncthreads();  // row s is there, row s - 1 is no longer read
      copy_row(s + kD, sprev);
      const unsigned sc_ = so;
      sprev = so;
      so = so == kD * STAGE ? 0 : so + STAGE;
      if (!mine) continue;
      if (DOT && s > 2 * P && (s - 2 * P) % GRP == 0) flush();  // the last GRP output rows' products
      if (NSH > 0 && s + 1 < steps) combine(so, (s + 1) & 1);
      const float* zw = reinterpret_cast<const float*>(smraw + sc_ + w * CELL) + lane;
      const CR& R = *reinterpret_cast<const CR*>(smraw + sc_ + LY::COL + w * (int)sizeof(CR));
      const float4* cf = NSH == 0 ? reinterpret_cast<const float4*>(R.coef)
                                  : reinterpret_cast<const float4*>(smraw + LY::COMB + (s & 1) * LY::CHALF) +
                                        w * (CU * NSH / 4);
      float4 c4 = make_float4(0.f, 0.f, 0.f, 0.f);  // the last one holds the diagonal or the weight too
      // e: tap, k: sum, a z + sum
      auto add2 = [&](int e, int sl, int k, float2 a, float2 zz) {
        acc[sl][k] = e == 0 ? __fmul2_rn(a, zz) : __ffma2_rn(a, zz, acc[sl][k]);
      };
      auto taps = [&](auto one) {
        constexpr bool ONE = decltype(one)::value;
        float sgt[TPB];  // ONE: the tiles' shifts
        if constexpr (ONE) {
#pragma unroll
          for (int k = 0; k < TPB; ++k) sgt[k] = par(k).x;
        }
#pragma unroll
        for (int du = 0; du < SW; ++du) {
          float zv[TPB], f[TPB];
#pragma unroll
          for (int k = 0; k < TPB; ++k) {
            zv[k] = zw[(du * TPB + k) * 32];
            if (CENTRE && du == P) zr[u][k] = zv[k];
          }
          if constexpr (ONE && MODE == ST_CHEB1) {
            const int c = w + du;
            const float* const fc = reinterpret_cast<const float*>(smraw + LY::FACT + (s & 1) * LY::FHALF) +
                                    ((c % kBU) * NCELL + c / kBU) * TPB;
#pragma unroll
            for (int k = 0; k < TPB; ++k) f[k] = fc[k];
          }
#pragma unroll
          for (int dv = 0; dv < SW; ++dv) {
            const int sl = (u - dv + SW) % SW;  // slot of output row s - dv
            const int e = du * SW + dv;
            if (e % 2 == 0) c4 = cf[e / 2];
            const float2 a = e % 2 == 0 ? make_float2(c4.x, c4.y) : make_float2(c4.z, c4.w);
            if constexpr (NSH == 2) {
              add2(e, sl, 0, a, make_float2(zv[0], zv[2 % TPB]));
              add2(e, sl, 1, a, make_float2(zv[1 % TPB], zv[3 % TPB]));
            } else if constexpr (!ONE) {
#pragma unroll
              for (int k = 0; k < TPB; ++k) add2(e, sl, k, a, make_float2(zv[k], zv[k]));
            } else if constexpr (TPB == 1) {
              float A = fmaf(sgt[0], a.y, a.x);
              if constexpr (MODE == ST_CHEB1) A *= f[0];
              acc[sl][0].x = e == 0 ? A * zv[0] : fmaf(A, zv[0], acc[sl][0].x);
            } else {
#pragma unroll
              for (int k = 0; k < TPB / 2; ++k) {
                float2 A = __ffma2_rn(make_float2(sgt[2 * k], sgt[2 * k + 1]), make_float2(a.y, a.y),
                                      make_float2(a.x, a.x));
                if constexpr (MODE == ST_CHEB1) A = __fmul2_rn(A, make_float2(f[2 * k], f[2 * k + 1]));
                add2(e, sl, k, A, make_float2(zv[2 * k], zv[2 * k + 1]));
              }
            }
          }
        }
      };
      if constexpr (NSH == 0) {
        if (ones)
          taps(std::true_type{});
        else
          taps(std::false_type{});
      } else {
        taps(std::false_type{});
      }
      const int own = s >= 2 * P ? R.own : -1;  // the output row that row s completes
      if (own < 0) continue;
      const int sl = (u + 1) % SW;              // output row s - 2p
      const int sc = (u - P + SW) % SW;         // its centre row
      const float* orr = reinterpret_cast<const float*>(smraw + sc_ + LY::ORW + w * (NIN * CELL)) + lane;
      float2 w2 = make_float2(0.f, 0.f);  // NSH = 2, ST_CHEB1: the second weights
      if constexpr (NSH == 2 && MODE == ST_CHEB1) w2 = reinterpret_cast<const float2*>(cf)[S2 + 1];
#pragma unroll
      for (int k = 0; k < TPB; ++k) {
        const float4 pk = par(k);  // sg, c1, c2, c0
        float az;
        if constexpr (NSH == 2) {
          az = k < 2 ? acc[sl][k % 2].x : acc[sl][k % 2].y;
        } else {
          const float one = TPB == 1 ? acc[sl][0].x : k % 2 == 0 ? acc[sl][k / 2].x : acc[sl][k / 2].y;
          az = ones ? one : fmaf(pk.x, acc[sl][k].y, acc[sl][k].x);
        }
        const float diag = NSH == 0 ? fmaf(pk.x, c4.w, c4.z) : 1.f;
        const float rv = NIN > 0 ? orr[k * 32] : 0.f;
        float res;
        if constexpr (CHEB) {
          const float zc = zr[sc][k];
          const float mom = fmaf(pk.y, zc - orr[(TPB + k) * 32], zc);
          const float d = rv - az;
          if constexpr (NSH == 0)  // ones: (c2 / diagonal) d, else (c2 d) / diagonal
            res = fmaf(wm_quotient(pk.z * (ones ? 1.f : d), diag), ones ? d : 1.f, mom);
          else
            res = fmaf(k < 2 ? c4.z : c4.w, d, mom);
          if constexpr (MODE == ST_CHEBDOT) {
            dot[k].add(rv, res);
            dot2[k].add(res, orr[(2 * TPB + k) * 32]);
          }
        } else if constexpr (MODE == ST_CHEB1) {
          const float zc = zr[sc][k];  // NSH = 2, ones: r, else z1
          float z1, wt;
          if constexpr (NSH == 2) {
            z1 = (k < 2 ? c4.z : c4.w) * zc;
            wt = k < 2 ? w2.x : w2.y;
          } else {
            const float q = wm_quotient(ones ? 1.f : pk.z * (rv - az), diag);
            z1 = ones ? pk.w * q * zc : zc;
            wt = ones ? pk.z * q : q;
          }
          io.out1[(size_t)(row0[k] + own) * 32 + lane] = z1;
          res = fmaf(wt, NSH == 2 || ones ? zc - az : 1.f, fmaf(pk.y, z1, z1));
        } else if constexpr (MODE == ST_RESID) {
          res = rv - az;
        } else {
          res = az;
          dot[k].add(zr[sc][k], az);
        }
        io.out[(size_t)(row0[k] + own) * 32 + lane] = res;
      }
    }
  }
  if constexpr (DOT) {  // the block's partial sums, warps in order
    flush();
    double* red = reinterpret_cast<double*>(smraw);  // [TPB][kBU][32]
    static_assert(LY::total >= sizeof(double) * TPB * kBU * 32, "reduction buffer");
    cp_wait<0>();
    stream_tiles_of(io, y, tile);  // (again: the registers are short in the loop)
    for (int h = 0; h < (MODE == ST_CHEBDOT ? 2 : 1); ++h) {
      __syncthreads();
#pragma unroll
      for (int k = 0; k < TPB; ++k)
        red[(k * kBU + w) * 32 + lane] = LY::SDOT ? sdot[k * (kBU * 32)] : h == 0 ? dot[k].d : dot2[k].d;
      __syncthreads();
#pragma unroll
      for (int k = 0; k < TPB; ++k) {
        if (w != k || tile[k] < 0 || !io.tile_active[tile[k]]) continue;
        double a = 0.0;
#pragma unroll
        for (int y = 0; y < kBU; ++y) a += red[(k * kBU + y) * 32 + lane];
        (h == 0 ? io.part : io.part2)[((size_t)tile[k] * io.pstride + item) * 32 + lane] = a;
      }
    }
  }
}

// The groups of a launch: pairs of tiles of one shift, two to a block (NSH = 2), or
// (NSH = 0) tiles of one shift each, then tiles of any shifts, four or one to a block.
// The dot products at a V-cycle's end of the tiles of NSH = 0 are other kernels'
// (wm_sten_dots, k_dots_rz_zq).
template <int P, int MODE, int NSH, int TPB>
__global__ void __launch_bounds__(kBU * 32, TPB == 1 ? kBlocks1 : kBlocks)
    k_stream(const __grid_constant__ StreamGeo G, const __grid_constant__ StreamIo io) {
  wm_wait_previous();
  const int y = io.g0 + blockIdx.y;
  stream_block<P, MODE, NSH, TPB>(G, io, y, y < io.n_one);
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
  const int64_t strip = (int64_t)np * G.nbu, base4 = strip * std::max(1, st.n[0] + st.n[1] + st.n[2]);
  const int grp = p == 2 ? StGrp<2>::value : StGrp<3>::value;
  *one = false;
  auto split = [&](int chunks) {
    G.VH = (L.nlv + chunks - 1) / chunks;
    if (dot) G.VH = (G.VH + grp - 1) / grp * grp;
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

// Whether the pairs of tiles of one shift have a launch of their own: always without
// other tiles, else where it has four waves of blocks (a launch waits for its longest block:
// 100 samples on the 128 x 64 bicubic torus 101 ms a call, with a launch at any number of
// blocks 117; on the 128 x 128 sphere 229 ms, never with one 244)
bool stream_pairs(const StreamGeo& G, const StreamTiles& st) {
  return st.n[0] > 0 && (st.n[1] + st.n[2] == 0 || (int64_t)st.n[0] * G.items >= 4 * kSMs * kBlocks);
}

// groups [g0, g0 + n)
template <int P, int MODE, int NSH, int TPB>
int launch_stream_n(const StreamArgs& a, const StreamGeo& G, StreamIo io, int g0, int n) {
  if (n <= 0) return WM_OK;
  constexpr size_t sm = StreamLayout<P, MODE, NSH, TPB>::total;
  static bool configured = false;
  if (!configured) {
    WM_CUDA(cudaFuncSetAttribute(k_stream<P, MODE, NSH, TPB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    configured = true;
  }
  for (int k = 0; k < n; k += 65535) {  // grid.y limit
    io.g0 = g0 + k;
    WM_TRY(wm_launch_next(a.cat, (k_stream<P, MODE, NSH, TPB>), dim3(G.items, std::min(65535, n - k)), dim3(32, kBU), sm,
                          a.s, G, io));
    WM_CUDA(cudaGetLastError());
  }
  return WM_OK;
}
template <int P, int MODE>
int launch_stream(const StreamArgs& a) {
  bool one = false;
  const StreamGeo G = stream_geo(*a.L, a.np, P, a.st, MODE == ST_APPLY || MODE == ST_CHEBDOT, &one);
  StreamIo io;
  io.sigma = a.sigma;
  io.ctab = a.ctab;
  io.sid = a.sid;
  io.tile_active = a.tile_active;
  io.z = a.z;
  io.r = a.r;
  io.prev = a.prev;
  io.q = a.q;
  io.out = a.out;
  io.out1 = a.out1;
  io.part = a.part;
  io.part2 = a.part2;
  io.groups = a.st.groups;
  io.order = a.st.order;
  io.g0 = 0;
  io.kstep = a.kstep;
  io.pstride = a.pstride > 0 ? a.pstride : G.items;
  constexpr int REST = MODE == ST_CHEBDOT ? ST_CHEB : MODE;
  const int* n = a.st.n;
  io.n_one = one ? a.st.n_uni : n[0] + n[1];
  if (one) return launch_stream_n<P, REST, 0, 1>(a, G, io, 0, a.st.tiles);
  const int pairs = stream_pairs(G, a.st) ? n[0] : 0;  // in a launch of their own
  WM_TRY((launch_stream_n<P, MODE, 2, kStreamTiles>(a, G, io, 0, pairs)));
  return launch_stream_n<P, REST, 0, kStreamTiles>(a, G, io, pairs, n[0] + n[1] + n[2] - pairs);
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
