// Shared-memory stencil kernels: the operator-type steps of the float64 solves and
// the true residuals of both precisions (the float solves' steps are the
// streaming kernels of wm_stream.h).
//
// A block owns a BU x BV tile of one patch's local DOF grid for one system
// tile.  It stages the (BU + 2p) x (BV + 2p) window of the input vector
// (through the extended grid map: halo cells come from the neighbouring
// patch, or wrap on the torus) into shared memory, once per block, and every
// warp then sweeps one column of BV outputs with a (2p+1)-row register window,
// so each staged value is read from shared memory 2p+1 times instead of each
// neighbour being fetched from L1/L2 (2p+1)^2 times.  Lane = system, so every
// staged row is one coalesced 256-byte transaction and the row's stencil
// coefficients (S, M) are warp-uniform loads shared by the 32 systems.
// Only the owner patch of a shared DOF computes its row.
#include <algorithm>

#include "wm_solver.h"
#include "wm_stencil.h"

namespace {

constexpr int BU = 8;   // outputs per block along u (one warp each)
// outputs per warp along v: for p = 2 the patches have 2^l + 2 local DOFs per
// side, which a height of 6 covers with less waste than 8 (66 and 18 exactly)
#ifndef WM_BV_P2
#define WM_BV_P2 6
#endif
template <int P>
struct BvOf {
  static constexpr int value = P == 2 ? WM_BV_P2 : 8;
  static_assert(value % 2 == 0 && value >= 2, "row pairs of the double-float residual");
};

struct StenGeo {
  int nlu, nlv, ELU, ELV, nbu, nbv, N;
  const int32_t* ext;
  const int32_t* own;
};

// per-thread dot accumulator (blocks of 16 products)
struct DAcc {
  double d = 0.0;
  double f = 0;
  int n = 0;
  __device__ __forceinline__ void add(double v) {
    f += v;
    if (++n == 16) {
      d += f;
      f = 0;
      n = 0;
    }
  }
  __device__ __forceinline__ double get() const { return d + f; }
};

// the block's partial sum of tile t
__device__ __forceinline__ void block_reduce(double acc, double* part, int t) {
  __shared__ double red[BU][32];
  red[threadIdx.y][threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.y == 0) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < BU; ++w) s += red[w][threadIdx.x];
    part[((size_t)t * gridDim.x + blockIdx.x) * 32 + threadIdx.x] = s;
  }
}

// ---------------------------------------------------------------- epilogues
// Chebyshev step in three-term form (tiles with per-lane shifts):
// z_next = z + c1 (z - z_prev) + c2 D^{-1} (r - A z), with c1 = 0 at step 0
// and z_prev = 0 where there is none; out may alias z_prev
struct ChebEpi {
  static constexpr bool PARTIALS = false;
  static constexpr int NIN = 2;  // r and z_prev of the output rows are staged
  const double* in[2];           // in[1] = nullptr: z_prev = 0
  int N, kstep;
  const double *dS, *dM;
  double* out;
  const double* sigma;
  const double2* ctab;  // (c1, c2) per [shift][step] of this level
  const int* sid;
  double sg, c1, c2;
  __device__ __forceinline__ void init(int t) {
    const int g = t * 32 + threadIdx.x;
    const double2 c = ctab[sid[g] * WM_MAX_CHEB + kstep];
    c1 = kstep == 0 ? 0.0 : c.x;
    c2 = c.y;
    sg = sigma[g];
  }
  // staged[a]: input a at this output row and lane
  __device__ __forceinline__ void row(int t, int i, double aS, double aM, double zc, const double* staged) {
    const double res = staged[0] - (aS + sg * aM);
    const double zp = in[1] ? staged[1] : 0.0;
    out[((size_t)t * N + i) * 32 + threadIdx.x] = zc + c1 * (zc - zp) + c2 * res / (dS[i] + sg * dM[i]);
  }
  __device__ __forceinline__ void finish(int) {}
};

// residual: res = r - A z
struct ResidEpi {
  static constexpr bool PARTIALS = false;
  static constexpr int NIN = 1;  // r staged
  const double* in[1];
  int N;
  double* res;
  const double* sigma;
  double sg;
  __device__ __forceinline__ void init(int t) { sg = sigma[t * 32 + threadIdx.x]; }
  __device__ __forceinline__ void row(int t, int i, double aS, double aM, double, const double* staged) {
    res[((size_t)t * N + i) * 32 + threadIdx.x] = staged[0] - (aS + sg * aM);
  }
  __device__ __forceinline__ void finish(int) {}
};

// outer apply: q = A p, partial (p, q)
struct ApplyEpi {
  static constexpr bool PARTIALS = true;
  static constexpr int NIN = 0;
  const double* in[1];
  int N;
  double* q;
  const double* sigma;
  double* part;
  double sg;
  DAcc acc;
  __device__ __forceinline__ void init(int t) { sg = sigma[t * 32 + threadIdx.x]; }
  __device__ __forceinline__ void row(int t, int i, double aS, double aM, double zc, const double*) {
    const double qv = aS + sg * aM;
    q[((size_t)t * N + i) * 32 + threadIdx.x] = qv;
    acc.add(zc * qv);
  }
  __device__ __forceinline__ void finish(int t) { block_reduce(acc.get(), part, t); }
};

// float64 true residual of flagged systems: r = b - A x, partial ||r||^2
template <typename Tr>
struct TrueResEpi {
  static constexpr bool PARTIALS = true;
  static constexpr int NIN = 0;
  const double* in[1];
  int N;
  const double* rhs;
  const int *src_of, *rep;
  Tr* r;
  const double* sigma;
  double* part;
  double sg;
  int src;
  bool mine;
  double acc;
  __device__ __forceinline__ void init(int t) {
    const int g = t * 32 + threadIdx.x;
    sg = sigma[g];
    src = src_of[g];
    mine = rep[g] != 0;
    acc = 0.0;
  }
  __device__ __forceinline__ void row(int t, int i, double aS, double aM, double, const double*) {
    if (!mine) return;
    const double b = src >= 0 ? rhs[((size_t)(src / 32) * N + i) * 32 + (src % 32)] : 0.0;
    const double rt = b - (aS + sg * aM);
    r[((size_t)t * N + i) * 32 + threadIdx.x] = (Tr)rt;
    acc += rt * rt;
  }
  __device__ __forceinline__ void finish(int t) { block_reduce(acc, part, t); }
};

// ---------------------------------------------------------------- the kernel
// 16-byte asynchronous global->shared copy; src_bytes = 0 writes zeros
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, int src_bytes) {
  unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sa), "l"(gmem), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

template <int P, int BVT, int NIN>
struct SmemLayout {
  static constexpr int BV = BVT;
  static constexpr int CU = BU + 2 * P, CV = BV + 2 * P, NC = CU * CV, S2 = (2 * P + 1) * (2 * P + 1);
  static constexpr size_t win = (size_t)NC * 32 * sizeof(double);
  static constexpr size_t coef = (size_t)BU * BV * S2 * sizeof(double2);
  static constexpr size_t rows = (size_t)NIN * BU * BV * 32 * sizeof(double);
  static constexpr size_t ids = (size_t)(NC + BU * BV) * sizeof(int);
  static constexpr size_t total = win + coef + rows + ids;
};

// BVT: outputs of a warp.  The float64 unit of an SM does one warp FMA in 17 cycles, so a
// block of 8 x 6 outputs (2,400 of them) takes 20 us however many SMs are idle: launches
// of fewer blocks than SMs take blocks two rows high.  One sample on the 8 x 8 sphere
// (51 systems, 48 blocks): a Chebyshev step 34 -> 16 us (event-timed).
template <int P, int BVT, typename Epi>
__global__ void __launch_bounds__(BU * 32, 1) k_sten(StenGeo G, const double2* __restrict__ csm,
                                                     const double* __restrict__ src, int tiles,
                                                     const int* __restrict__ tile_active, const Epi epi_arg,
                                                     const int* __restrict__ skip_uni) {
  wm_wait_previous();
  using LY = SmemLayout<P, BVT, Epi::NIN>;
  constexpr int BV = LY::BV, NIN = Epi::NIN, SW = 2 * P + 1, CU = LY::CU, NC = LY::NC, S2 = LY::S2;
  constexpr int ROWCH = 32 * sizeof(double) / 16;  // 16-byte chunks per staged row
  Epi epi = epi_arg;  // per-thread copy (its per-tile fields live in registers)
  extern __shared__ __align__(16) unsigned char smraw[];
  double* sm = reinterpret_cast<double*>(smraw);
  double2* scf = reinterpret_cast<double2*>(smraw + LY::win);
  double* srw = reinterpret_cast<double*>(smraw + LY::win + LY::coef);       // [NIN][BU*BV][32] epilogue inputs
  int* sid = reinterpret_cast<int*>(smraw + LY::win + LY::coef + LY::rows);  // [NC] cells, then [BU*BV] rows
  int* srow = sid + NC;
  const int lane = threadIdx.x, w = threadIdx.y;
  const int tid = w * 32 + lane;
  int b = blockIdx.x;
  const int bu = b % G.nbu;
  b /= G.nbu;
  const int bv = b % G.nbv;
  const int m = b / G.nbv;
  const int t = blockIdx.y;
  // skip_uni: tiles with a single shift are done by k_sten_uni
  if (t >= tiles || !tile_active[t] || (skip_uni && skip_uni[t])) return;
  epi.init(t);
  // phase 0: global DOF of every window cell and every output row of the block
  const int32_t* E = G.ext + (size_t)m * G.ELV * G.ELU;
  const int32_t* OWN = G.own + (size_t)m * G.nlv * G.nlu;
  for (int c = tid; c < NC + BU * BV; c += BU * 32) {
    int v = -1;
    if (c < NC) {
      int eu = bu * BU + c % CU, ev = bv * BV + c / CU;
      if (eu < G.ELU && ev < G.ELV) v = E[(size_t)ev * G.ELU + eu];
    } else {
      int o = c - NC;
      int iu = bu * BU + o % BU, iv = bv * BV + o / BU;
      if (iu < G.nlu && iv < G.nlv) v = OWN[(size_t)iv * G.nlu + iu];
    }
    sid[c] = v;
  }
  __syncthreads();
  // phase 1: asynchronous copies of the window rows, the coefficient rows and the outputs' inputs
  for (int c = tid; c < NC * ROWCH; c += BU * 32) {
    const int part = c % ROWCH, gi = sid[c / ROWCH];
    cp_async16(sm + (size_t)c * 2, gi >= 0 ? src + ((size_t)t * G.N + gi) * 32 + part * 2 : src, gi >= 0 ? 16 : 0);
  }
  for (int c = tid; c < BU * BV * S2; c += BU * 32) {
    const int gi = srow[c / S2];
    cp_async16(scf + c, gi >= 0 ? csm + (size_t)gi * S2 + c % S2 : csm, gi >= 0 ? 16 : 0);
  }
#pragma unroll
  for (int a = 0; a < NIN; ++a) {  // compile-time input index keeps epi in registers
    const double* base = epi.in[a];
    if (!base) continue;
    for (int c = tid; c < BU * BV * ROWCH; c += BU * 32) {
      const int part = c % ROWCH, o = c / ROWCH, gi = srow[o];
      cp_async16(srw + ((size_t)a * BU * BV + o) * 32 + part * 2,
                 gi >= 0 ? base + ((size_t)t * G.N + gi) * 32 + part * 2 : src, gi >= 0 ? 16 : 0);
    }
  }
  cp_async_wait_all();
  __syncthreads();
  // phase 2: each warp sweeps the column iu with a ring of SW staged rows
  const int iu = bu * BU + w;
  if (iu < G.nlu) {
    double win[SW][SW];
#pragma unroll
    for (int r = 0; r < SW - 1; ++r)
#pragma unroll
      for (int du = 0; du < SW; ++du) win[r][du] = sm[((size_t)r * CU + w + du) * 32 + lane];
#pragma unroll
    for (int j = 0; j < BV; ++j) {
      const int rn = j + SW - 1;  // staged row entering the window
#pragma unroll
      for (int du = 0; du < SW; ++du) win[rn % SW][du] = sm[((size_t)rn * CU + w + du) * 32 + lane];
      const int i = srow[j * BU + w];
      if (i >= 0) {
        const double2* cf = scf + (size_t)(j * BU + w) * S2;
        double aS = 0, aM = 0;
#pragma unroll
        for (int dv = 0; dv < SW; ++dv)
#pragma unroll
          for (int du = 0; du < SW; ++du) {
            const double2 c = cf[dv * SW + du];
            const double z = win[(j + dv) % SW][du];
            aS += c.x * z;
            aM += c.y * z;
          }
        double stg[NIN > 0 ? NIN : 1];
#pragma unroll
        for (int a = 0; a < NIN; ++a) stg[a] = srw[((size_t)a * BU * BV + j * BU + w) * 32 + lane];
        epi.row(t, i, aS, aM, win[(j + P) % SW][P], stg);
      }
    }
  }
  epi.finish(t);
}

// ------------------------------------------- operator steps, one shift per tile
// Operator-type steps for runs of consecutive tiles whose 32 systems share one
// shift sigma (sample-major packing puts the 32 samples of one sinc node in a
// tile, and the ns / 32 tiles of a node next to each other):
//   UNI_CHEB     three-term Chebyshev step  out = z + c1 (z - z_prev) + w (r - A z)
//   UNI_RESID    residual                   out = r - A z
//   UNI_APPLY    outer apply                out = A z, per-block partial (z, A z)
//   UNI_CHEBDOT  the Chebyshev step that ends a V-cycle, also forming the
//                per-block partials (r, z_new) and (z_new, q) of the outer CG
//                (q staged as a third row)
//   UNI_CHEB1    the first two pre-smoothing steps from z = 0 in one pass:
//                z1 = c2_0 Dinv r (written to out1), out = z1 + c1 z1 + c2 Dinv (r - A z1),
//                A z1 formed from the window of r with c2_0 Dinv folded into the rows
// A block owns one spatial block of one patch and a group of at most
// kUniGroup consecutive tiles of one shift (a host-built list of (first tile,
// count); `split` blocks share a group when the grid would be too small).
// Everything that depends only on the spatial block and the shift is done
// once for the group: the DOF ids of the window and of the output rows and the
// combined rows
// A = S + sigma M (with the Chebyshev weights w = c2 / (dS + sigma dM)), so an
// output costs one float64 FMA per stencil entry (the unit that bounds this
// kernel) and no division.
enum { UNI_CHEB = 0, UNI_RESID = 1, UNI_APPLY = 2, UNI_CHEBDOT = 3, UNI_CHEB1 = 4 };
template <int MODE>
struct UniCheb {
  static constexpr bool value = MODE == UNI_CHEB || MODE == UNI_CHEBDOT;
};
template <int MODE>
struct UniRows {  // staged 32-system rows per output row
  static constexpr int value = MODE == UNI_CHEBDOT ? 3 : (MODE == UNI_CHEB ? 2 : (MODE == UNI_RESID ? 1 : 0));
};
template <int P, int MODE>
struct UniLayout {
  static constexpr int BV = BvOf<P>::value;
  static constexpr int CU = BU + 2 * P, CV = BV + 2 * P, NC = CU * CV, S2 = (2 * P + 1) * (2 * P + 1);
  static constexpr int S2P = (S2 + 1) / 2 * 2;                // padded combined row length
  static constexpr int NR = UniRows<MODE>::value;
  static constexpr int ND = UniCheb<MODE>::value ? 2 : 0;     // staged diagonals dS, dM
  static constexpr size_t win = (size_t)NC * 32 * sizeof(double);  // window of the input vector
  static constexpr size_t stage = win + (size_t)NR * BU * BV * 32 * sizeof(double);  // and rows of the outputs
  // raw (S, M) rows, needed at set-up only: they sit in the stage buffer
  static constexpr size_t raw = (size_t)BU * BV * S2 * sizeof(double2);
  static constexpr size_t stages = stage > raw ? stage : raw;
  static constexpr size_t coef = (size_t)BU * BV * S2P * sizeof(double);  // combined rows
  static constexpr size_t diag = MODE == UNI_CHEB1 ? (size_t)3 * NC * sizeof(double)  // dS, dM, Dinv of the cells
                                                   : (size_t)(ND + 1) * BU * BV * sizeof(double);  // dS, dM, w
  static constexpr size_t diag16 = (diag + 15) / 16 * 16;
  static constexpr size_t ids = (size_t)(NC + BU * BV) * sizeof(int);
  static constexpr size_t total = stages + coef + diag16 + ids;
  // 16-byte copies of one staged tile: window chunks and row chunks, and per thread
  static constexpr int ROWCH = 32 * sizeof(double) / 16;
  static constexpr int WCH = NC * ROWCH, RCH = BU * BV * ROWCH;
  static constexpr int WPT = (WCH + BU * 32 - 1) / (BU * 32), RPT = (RCH + BU * 32 - 1) / (BU * 32);
  static_assert(stage % 16 == 0 && raw % 16 == 0 && coef % 16 == 0, "16-byte aligned regions");
};
// blocks per SM that the shared memory allows (with the 2 KB of the partial-sum
// reduction and the 1 KB the runtime reserves per block), at most two (the copy
// offsets and the window need the registers); this is also the register budget
template <int P, int MODE>
struct UniMinBlocks {
  static constexpr size_t per = UniLayout<P, MODE>::total + 3 * 1024;
  static constexpr int fit = (int)((228 * 1024) / per);
  static constexpr int value = fit >= 2 ? 2 : 1;
};
// 8-byte asynchronous copy through L1 (diagonal entries)
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem, int src_bytes) {
  unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(sa), "l"(gmem), "r"(src_bytes) : "memory");
}

template <int P, int MODE>
__global__ void __launch_bounds__(BU * 32, (UniMinBlocks<P, MODE>::value))
    k_sten_uni(StenGeo G, const double2* __restrict__ csm, const double* __restrict__ dS,
               const double* __restrict__ dM, const double* __restrict__ sigma, const double2* __restrict__ ctab,
               const int* __restrict__ sid, int kstep, const double* __restrict__ z, const double* __restrict__ r,
               const double* prev, double* out, int tiles, const int* __restrict__ tile_active,
               const int2* __restrict__ groups, int split, double* __restrict__ part, const double* __restrict__ qd,
               double* __restrict__ part2, double* __restrict__ out1) {
  wm_wait_previous();
  using LY = UniLayout<P, MODE>;
  constexpr bool CHEB = UniCheb<MODE>::value;
  constexpr int BV = LY::BV, SW = 2 * P + 1, CU = LY::CU, NC = LY::NC, S2 = LY::S2, S2P = LY::S2P;
  constexpr int NR = LY::NR, ROWCH = LY::ROWCH;
  constexpr int NT = BU * 32;  // threads per block
  extern __shared__ __align__(16) unsigned char smraw[];
  double* const stg = reinterpret_cast<double*>(smraw);    // [NC][32] window, [NR][BU*BV][32] rows
  double2* const sraw = reinterpret_cast<double2*>(smraw);  // [BU*BV][S2], set-up only
  double* const scf = reinterpret_cast<double*>(smraw + LY::stages);             // [BU*BV][S2P]
  double* const sdg = reinterpret_cast<double*>(smraw + LY::stages + LY::coef);  // [ND][BU*BV], then w
  double* const swt = sdg + LY::ND * BU * BV;
  int* const sid_ = reinterpret_cast<int*>(smraw + LY::stages + LY::coef + LY::diag16);
  int* const srow = sid_ + NC;
  const int lane = threadIdx.x, w = threadIdx.y;
  const int tid = w * 32 + lane;
  int b = blockIdx.x;
  const int bu = b % G.nbu;
  b /= G.nbu;
  const int bv = b % G.nbv;
  const int m = b / G.nbv;
  // this block's tiles [ta, tb): part `sp` of group blockIdx.y / split
  const int2 gr = groups[blockIdx.y / split];
  const int sp = blockIdx.y % split;
  const int per = (gr.y + split - 1) / split;
  const int ta = gr.x + sp * per;
  const int tb = min(min(gr.x + gr.y, ta + per), tiles);
  unsigned todo = 0;  // active tiles of the range, bit t - ta (at most kUniGroup bits)
  for (int t = ta; t < tb; ++t)
    if (tile_active[t]) todo |= 1u << (t - ta);
  if (todo == 0) return;
  double sg, c1 = 0, c2 = 0, c20 = 0;
  {
    const int g = gr.x * 32;  // every system of the group has this shift
    if constexpr (CHEB) {
      const double2 c = ctab[sid[g] * WM_MAX_CHEB + kstep];
      c1 = kstep == 0 ? 0.0 : c.x;
      c2 = c.y;
    }
    if constexpr (MODE == UNI_CHEB1) {  // steps 0 and 1
      const double2 c0 = ctab[sid[g] * WM_MAX_CHEB], c = ctab[sid[g] * WM_MAX_CHEB + 1];
      c20 = c0.y;
      c1 = c.x;
      c2 = c.y;
    }
    sg = sigma[g];
  }
  // set-up 1: global DOF of every window cell and every output row
  const int32_t* E = G.ext + (size_t)m * G.ELV * G.ELU;
  const int32_t* OWN = G.own + (size_t)m * G.nlv * G.nlu;
  for (int c = tid; c < NC + BU * BV; c += NT) {
    int v = -1;
    if (c < NC) {
      int eu = bu * BU + c % CU, ev = bv * BV + c / CU;
      if (eu < G.ELU && ev < G.ELV) v = E[ev * G.ELU + eu];
    } else {
      int o = c - NC;
      int iu = bu * BU + o % BU, iv = bv * BV + o / BU;
      if (iu < G.nlu && iv < G.nlv) v = OWN[iv * G.nlu + iu];
    }
    sid_[c] = v;
  }
  __syncthreads();
  // set-up 2: (S, M) rows and diagonals, copy offsets
  for (int c = tid; c < BU * BV * S2; c += NT) {
    const int gi = srow[c / S2];
    cp_async16(sraw + c, gi >= 0 ? csm + (size_t)gi * S2 + c % S2 : csm, gi >= 0 ? 16 : 0);
  }
  if constexpr (MODE == UNI_CHEB1) {  // diagonals of every window cell
    for (int c = tid; c < 2 * NC; c += NT) {
      const int gi = sid_[c % NC];
      const double* base = c < NC ? dS : dM;
      cp_async8(sdg + c, gi >= 0 ? base + gi : dS, gi >= 0 ? 8 : 0);
    }
  }
  if constexpr (CHEB) {
    for (int c = tid; c < 2 * BU * BV; c += NT) {
      const int gi = srow[c % (BU * BV)];
      const double* base = c < BU * BV ? dS : dM;
      cp_async8(sdg + c, gi >= 0 ? base + gi : dS, gi >= 0 ? 8 : 0);
    }
  }
  // each thread's source offsets (within a tile) of its window and row
  // chunks: -1 zero-fills a cell outside the surface, -2 marks no chunk
  int woff[LY::WPT];
#pragma unroll
  for (int k = 0; k < LY::WPT; ++k) {
    const int c = tid + k * NT;
    int o = -2;
    if (c < LY::WCH) {
      const int gi = sid_[c / ROWCH];
      o = gi >= 0 ? gi * 32 + (c % ROWCH) * 2 : -1;
    }
    woff[k] = o;
  }
  int roff[NR > 0 ? LY::RPT : 1];
#pragma unroll
  for (int k = 0; k < (NR > 0 ? LY::RPT : 1); ++k) {
    const int c = tid + k * NT;
    int o = -2;
    if (NR > 0 && c < LY::RCH) {
      const int gi = srow[c / ROWCH];
      o = gi >= 0 ? gi * 32 + (c % ROWCH) * 2 : -1;
    }
    roff[k] = o;
  }
  // the 16-byte copies of tile t into the stage buffer; absent inputs (z_prev, q) are not copied
  auto issue = [&](int t) {
    const size_t to = (size_t)t * G.N * 32;
#pragma unroll
    for (int k = 0; k < LY::WPT; ++k) {
      const int o = woff[k];
      if (o != -2) cp_async16(stg + (tid + k * NT) * 2, o >= 0 ? z + to + o : z, o >= 0 ? 16 : 0);
    }
#pragma unroll
    for (int a = 0; a < NR; ++a) {
      const double* base = a == 0 ? r : (a == 1 ? prev : qd);
      if (base == nullptr) continue;
#pragma unroll
      for (int k = 0; k < LY::RPT; ++k) {
        const int o = roff[k];
        if (o != -2)
          cp_async16(stg + NC * 32 + a * BU * BV * 32 + (tid + k * NT) * 2, o >= 0 ? base + to + o : base,
                     o >= 0 ? 16 : 0);
      }
    }
  };
  cp_async_wait_all();
  __syncthreads();
  double* sdc = sdg + 2 * NC;  // UNI_CHEB1: Dinv of every window cell
  if constexpr (MODE == UNI_CHEB1) {
    for (int c = tid; c < NC; c += NT) sdc[c] = sid_[c] >= 0 ? 1.0 / (sdg[c] + sg * sdg[NC + c]) : 0.0;
    __syncthreads();
  }
  // set-up 3: combined rows and the Chebyshev diagonal weights
  for (int c = tid; c < BU * BV * S2P; c += NT) {
    const int o = c / S2P, sl = c - o * S2P;
    double a = 0;
    if (sl < S2) {
      const double2 q = sraw[o * S2 + sl];
      a = q.x + sg * q.y;
      if constexpr (MODE == UNI_CHEB1)  // times c2_0 Dinv of the neighbour's cell: A z1 from r
        a *= c20 * sdc[((o / BU) + sl / SW) * CU + (o % BU) + sl % SW];
    }
    scf[c] = a;
  }
  if constexpr (CHEB)
    for (int c = tid; c < BU * BV; c += NT) swt[c] = srow[c] >= 0 ? c2 / (sdg[c] + sg * sdg[BU * BV + c]) : 0.0;
  __syncthreads();  // the raw rows are dead from here on
  const int iu = bu * BU + w;
  while (todo) {
    const int t = ta + __ffs(todo) - 1;
    todo &= todo - 1;
    issue(t);
    cp_async_wait_all();
    __syncthreads();
    // each warp sweeps the column iu with a ring of SW rows in registers
    const double* const srw = stg + NC * 32;
    DAcc dot;   // UNI_APPLY: (z, A z); UNI_CHEBDOT: (r, z_new) over this thread's outputs
    DAcc dot2;  // UNI_CHEBDOT: (z_new, q)
    if (iu < G.nlu) {
      double win[SW][SW];
#pragma unroll
      for (int rr = 0; rr < SW - 1; ++rr)
#pragma unroll
        for (int du = 0; du < SW; ++du) win[rr][du] = stg[(rr * CU + w + du) * 32 + lane];
#pragma unroll
      for (int j = 0; j < BV; ++j) {
        const int rn = j + SW - 1;  // staged row entering the window
#pragma unroll
        for (int du = 0; du < SW; ++du) win[rn % SW][du] = stg[(rn * CU + w + du) * 32 + lane];
        const int o = j * BU + w;
        const int i = srow[o];
        if (i < 0) continue;  // past the patch's edge or another patch's row
        double az = 0;
#pragma unroll
        for (int q = 0; q < S2P / 2; ++q) {
          const double2 a = reinterpret_cast<const double2*>(scf + (j * BU + w) * S2P)[q];
          az = fma(a.x, win[(j + (2 * q) / SW) % SW][(2 * q) % SW], az);
          if (2 * q + 1 < S2) az = fma(a.y, win[(j + (2 * q + 1) / SW) % SW][(2 * q + 1) % SW], az);
        }
        const double zc = win[(j + P) % SW][P];
        double res;
        if constexpr (CHEB) {
          const double rv = srw[o * 32 + lane];
          const double zp = prev ? srw[(BU * BV + o) * 32 + lane] : 0.0;
          res = zc + c1 * (zc - zp) + swt[o] * (rv - az);
          if constexpr (MODE == UNI_CHEBDOT) {
            dot.add(rv * res);
            if (qd) dot2.add(res * srw[(2 * BU * BV + o) * 32 + lane]);
          }
        } else if constexpr (MODE == UNI_CHEB1) {
          const double dc = sdc[(j + P) * CU + w + P];  // Dinv of the output row
          const double z1 = c20 * dc * zc;              // zc is r here
          out1[((size_t)t * G.N + i) * 32 + lane] = z1;
          res = z1 + c1 * z1 + c2 * dc * (zc - az);
        } else if constexpr (MODE == UNI_RESID) {
          res = srw[o * 32 + lane] - az;
        } else {
          res = az;
          dot.add(zc * az);
        }
        out[((size_t)t * G.N + i) * 32 + lane] = res;
      }
    }
    if constexpr (MODE == UNI_APPLY || MODE == UNI_CHEBDOT) {
      block_reduce(dot.get(), part, t);
      if (MODE == UNI_CHEBDOT && qd) {
        __syncthreads();
        block_reduce(dot2.get(), part2, t);
      }
    }
    __syncthreads();  // the stage buffer (and the reduction buffer) may be refilled
  }
}

StenGeo geo_of(const wm_level& L) {
  StenGeo G;
  G.nlu = L.nlu;
  G.nlv = L.nlv;
  G.ELU = L.ELU;
  G.ELV = L.ELV;
  G.nbu = L.nbu;
  G.nbv = L.nbv;
  G.N = L.N;
  G.ext = L.d_ext.p;
  G.own = L.d_own.p;
  return G;
}

template <int P, int BVT, typename Epi>
int launch_bv(const wm_level& L, int np, int tiles, const double* src, const int* tile_active, const Epi& epi, int cat,
              cudaStream_t s, const int* skip_uni) {
  constexpr size_t sm = SmemLayout<P, BVT, Epi::NIN>::total;
  static bool configured = false;
  if (!configured) {
    WM_CUDA(cudaFuncSetAttribute(k_sten<P, BVT, Epi>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    configured = true;
  }
  StenGeo G = geo_of(L);
  G.nbv = (L.nlv + BVT - 1) / BVT;
  dim3 grid(np * G.nbu * G.nbv, tiles);
  WM_TRY(wm_launch_next(cat, (k_sten<P, BVT, Epi>), grid, dim3(32, BU), sm, s, G, L.d_csm64.p, src, tiles,
      tile_active, epi, skip_uni));
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}
// (steps that leave per-block partial sums keep the standard height: the caller
// counts its blocks)
template <int P, typename Epi>
int launch(const wm_level& L, int np, int tiles, const double* src, const int* tile_active, const Epi& epi, int cat,
           cudaStream_t s, const int* skip_uni = nullptr) {
  if (Epi::PARTIALS || (int64_t)np * L.nbu * L.nbv * tiles >= 152)
    return launch_bv<P, BvOf<P>::value>(L, np, tiles, src, tile_active, epi, cat, s, skip_uni);
  return launch_bv<P, 2>(L, np, tiles, src, tile_active, epi, cat, s, skip_uni);
}

// dot products of float vectors by the row blocks of the kernels above: products of a
// column's rows in float, then double
template <int P>
__global__ void __launch_bounds__(BU * 32)
    k_sten_dots(StenGeo G, const int* __restrict__ list, const float* __restrict__ r, const float* __restrict__ z,
                const float* __restrict__ q, const int* __restrict__ tile_active, double* __restrict__ part_rz,
                double* __restrict__ part_zq, int stride) {
  wm_wait_previous();
  constexpr int BV = BvOf<P>::value;
  const int t = list[blockIdx.y], lane = threadIdx.x, w = threadIdx.y;
  if (!tile_active[t]) return;
  int b = blockIdx.x;
  const int bu = b % G.nbu;
  b /= G.nbu;
  const int bv = b % G.nbv, m = b / G.nbv;
  const int iu = bu * BU + w;
  float rz = 0.f, zq = 0.f;
  if (iu < G.nlu) {
    const int32_t* own = G.own + ((size_t)m * G.nlv + bv * BV) * G.nlu + iu;
    int id[BV];
    float rv[BV], zv[BV], qv[BV];
#pragma unroll
    for (int j = 0; j < BV; ++j) id[j] = bv * BV + j < G.nlv ? own[(size_t)j * G.nlu] : -1;
#pragma unroll
    for (int j = 0; j < BV; ++j) {
      const size_t o = ((size_t)t * G.N + max(id[j], 0)) * 32 + lane;
      rv[j] = id[j] >= 0 ? r[o] : 0.f;
      zv[j] = id[j] >= 0 ? z[o] : 0.f;
      qv[j] = id[j] >= 0 ? q[o] : 0.f;
    }
#pragma unroll
    for (int j = 0; j < BV; ++j)
      if (id[j] >= 0) {
        rz = fmaf(rv[j], zv[j], rz);
        zq = fmaf(zv[j], qv[j], zq);
      }
  }
  __shared__ double red[2][BU][32];
  red[0][w][lane] = rz;
  red[1][w][lane] = zq;
  __syncthreads();
  if (w < 2) {
    double a = 0.0;
#pragma unroll
    for (int y = 0; y < BU; ++y) a += red[w][y][lane];
    (w == 0 ? part_rz : part_zq)[((size_t)t * stride + blockIdx.x) * 32 + lane] = a;
  }
}

// ------------------------------------------- double-float true residual
// r = b - (S x + sigma M x) of the systems flagged for residual replacement,
// with every operation on the FP32 pipes: the FP64 rate of this part is
// about 1/60 of its FP32 rate (conversions to and from float64 run there
// too), so the kernel never touches a float64 register in its loops.
//  * float64 inputs (x, b, sigma) are split into float pairs hi + lo with
//    integer operations on their bits (relative error at most 2^-47);
//  * each product a*x is the rounded hi*hi plus its exact rounding error
//    (FMA) plus the two cross terms; the rounded products are summed with
//    Knuth's two-sum and all errors gathered in a float tail (about 48
//    significant bits for the stencil sum);
//  * where the 32 shifts of a tile are equal (sample-major packing;
//    k_sten_trueres_df_uni) each coefficient row is combined once per block
//    into A = S + sigma M in the same arithmetic and one sum is formed, two
//    output rows at a time on the packed FP32 instructions (FMUL2/FFMA2/FADD2,
//    rounding per component as the scalar ones); otherwise (k_sten_trueres_df)
//    S x and M x are the two packed sums and are combined per output.
// Each output also accumulates B_i = sum_j |a_ij x_j| (float, from the rounded
// hi products, within a factor 1 + 2^-22 of the exact sum): the entry's
// rounding error stays below 2^-42 B_i (operand splits 2^-47 and 2^-48,
// dropped lo*lo and cross-term roundings 2^-47, float tail 25 x 2^-47), and the
// caller checks 2^-42 ||B|| against the convergence tolerance before it
// trusts the residuals, recomputing them in float64 otherwise (also when a
// value of the system is below 2^-102, where float pairs lose precision).
// The squared norms are accumulated in float over the 8 outputs of a thread
// (entries of r below about 1e-22 in magnitude lose their contribution).

// v = hi + lo with hi = v rounded to 24 significant bits and lo the rest
// rounded to float: |v - hi - lo| <= 2^-47 |v| (2^-48 while lo is a normal
// float), using integer operations on
// the bits of v and one int->float conversion.  Non-finite v or |v| >= 2^128
// gives hi = +-inf; 0 < |v| < 2^-102 (lo would be subnormal) sets `tiny` and
// returns (+-0, 0).
__device__ __forceinline__ float2 split_bits(double v, bool& tiny) {
  // 32-bit halves only (no 64-bit integer or float64 instructions)
  const unsigned hi32 = (unsigned)__double2hiint(v), lo32 = (unsigned)__double2loint(v);
  const unsigned sign = hi32 & 0x80000000u;
  const int e = (int)((hi32 >> 20) & 0x7FFu);
  if (e < 921) {
    tiny |= ((hi32 & 0x7FFFFFFFu) | lo32) != 0u;
    return make_float2(__int_as_float((int)sign), 0.f);
  }
  if (e >= 1151) return make_float2(__int_as_float((int)(sign | 0x7F800000u)), 0.f);
  // round the magnitude to the nearest multiple of 2^29 units (24 significant
  // bits; a carry into the exponent is the correct rounding)
  const unsigned lr = lo32 + 0x10000000u;
  const unsigned hr = (hi32 & 0x7FFFFFFFu) + (lr < lo32 ? 1u : 0u);
  const unsigned hl = lr & 0xE0000000u;
  const int rem = (int)(lo32 - hl);  // |rem| <= 2^28 units of 2^(e-1075)
  const int efh = (int)(hr >> 20) - 896;
  if (efh >= 255) return make_float2(__int_as_float((int)(sign | 0x7F800000u)), 0.f);
  const float h = __int_as_float((int)(sign | ((unsigned)efh << 23) | ((hr & 0xFFFFFu) << 3) | (hl >> 29)));
  const float l = __fmul_rn(__fmul_rn(__int2float_rn(rem), 3.7252902984619141e-09f /* 2^-28 */),
                            __int_as_float((e - 920) << 23) /* 2^(e-1047) */);
  return make_float2(h, sign ? -l : l);
}
// error-free sum: a + b = s + e exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}
// (ah + al) + (gh + gl) * (mh + ml) as a renormalised pair
__device__ __forceinline__ float2 df_axpy(float ah, float al, float gh, float gl, float mh, float ml) {
  const float p = __fmul_rn(gh, mh);
  float e = fmaf(gh, mh, -p);
  e = fmaf(gh, ml, fmaf(gl, mh, e));
  float t, err;
  two_sum(ah, p, t, err);
  const float lo = __fadd_rn(al, __fadd_rn(e, err));
  float h, l;
  two_sum(t, lo, h, l);
  return make_float2(h, l);
}

// (s, c) += (ah + al) * (xh + xl), dropping al * xl; b += |ah xh|: two sums at once on
// the packed FP32 pipe (FMUL2 / FFMA2 / FADD2: each component rounds as the scalar form)
__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }
__device__ __forceinline__ void df_acc2(float2& s, float2& c, float& b0, float& b1, float2 ah, float2 al, float2 xh,
                                        float2 xl) {
  const float2 p = __fmul2_rn(ah, xh);
  b0 = __fadd_rn(b0, fabsf(p.x));
  b1 = __fadd_rn(b1, fabsf(p.y));
  float2 e = __ffma2_rn(ah, xh, neg2(p));
  e = __ffma2_rn(ah, xl, __ffma2_rn(al, xh, e));
  const float2 t = __fadd2_rn(s, p);
  const float2 bp = __fadd2_rn(t, neg2(s));
  const float2 err = __fadd2_rn(__fadd2_rn(s, neg2(__fadd2_rn(t, neg2(bp)))), __fadd2_rn(p, neg2(bp)));
  s = t;
  c = __fadd2_rn(c, __fadd2_rn(err, e));
}

template <int P>
struct DfLayout {
  static constexpr int BV = BvOf<P>::value;
  static constexpr int CU = BU + 2 * P, CV = BV + 2 * P, NC = CU * CV, S2 = (2 * P + 1) * (2 * P + 1);
  static constexpr size_t win = (size_t)NC * 32 * sizeof(double);
  static constexpr size_t coef = (size_t)BU * BV * S2 * sizeof(float4);
  static constexpr size_t ids = (size_t)(NC + BU * BV) * sizeof(int);
  static constexpr size_t total = win + coef + ids;
};

template <int P>
__global__ void __launch_bounds__(BU * 32, 2)
    k_sten_trueres_df(StenGeo G, const float4* __restrict__ cdf, const double* __restrict__ x, int tiles,
                      const int* __restrict__ tile_rep, const double* __restrict__ sigma,
                      const double* __restrict__ rhs, const int* __restrict__ src_of, const int* __restrict__ rep,
                      float* __restrict__ r, double* __restrict__ part, double* __restrict__ part_bound,
                      const int* __restrict__ skip_uni) {
  wm_wait_previous();
  constexpr int BV = BvOf<P>::value;
  using LY = DfLayout<P>;
  constexpr int SW = 2 * P + 1, CU = LY::CU, NC = LY::NC, S2 = LY::S2;
  extern __shared__ __align__(16) unsigned char smraw[];
  double* smd = reinterpret_cast<double*>(smraw);
  float2* smf = reinterpret_cast<float2*>(smraw);  // the same cells after the split
  float4* scf = reinterpret_cast<float4*>(smraw + LY::win);
  int* sid = reinterpret_cast<int*>(smraw + LY::win + LY::coef);
  int* srow = sid + NC;
  const int lane = threadIdx.x, w = threadIdx.y;
  const int tid = w * 32 + lane;
  int b = blockIdx.x;
  const int bu = b % G.nbu;
  b /= G.nbu;
  const int bv = b % G.nbv;
  const int m = b / G.nbv;
  const int t = blockIdx.y;
  if (t >= tiles || !tile_rep[t] || skip_uni[t]) return;  // tiles of one shift: the group kernel's
  const int g = t * 32 + lane;
  const double sg = sigma[g];
  bool tiny = false;  // a value of this system too small for float pairs
  const float2 sgp = split_bits(sg, tiny);
  tiny = false;       // (a tiny shift only loses its own negligible part)
  const bool mine = rep[g] != 0;
  const int src = src_of[g];
  // phase 0: global DOF of every window cell and every output row
  const int32_t* E = G.ext + (size_t)m * G.ELV * G.ELU;
  const int32_t* OWN = G.own + (size_t)m * G.nlv * G.nlu;
  for (int c = tid; c < NC + BU * BV; c += BU * 32) {
    int v = -1;
    if (c < NC) {
      int eu = bu * BU + c % CU, ev = bv * BV + c / CU;
      if (eu < G.ELU && ev < G.ELV) v = E[(size_t)ev * G.ELU + eu];
    } else {
      int o = c - NC;
      int iu = bu * BU + o % BU, iv = bv * BV + o / BU;
      if (iu < G.nlu && iv < G.nlv) v = OWN[(size_t)iv * G.nlu + iu];
    }
    sid[c] = v;
  }
  __syncthreads();
  // phase 1: window rows of x (16 chunks of 16 bytes each) and coefficient rows
  for (int c = tid; c < NC * 16; c += BU * 32) {
    int part16 = c % 16, cell = c / 16;
    int gi = sid[cell];
    const double* gp = gi >= 0 ? x + ((size_t)t * G.N + gi) * 32 + part16 * 2 : x;
    cp_async16(smd + (size_t)cell * 32 + part16 * 2, gp, gi >= 0 ? 16 : 0);
  }
  for (int c = tid; c < BU * BV * S2; c += BU * 32) {
    int o = c / S2, k = c % S2;
    int gi = srow[o];
    const float4* gp = gi >= 0 ? cdf + (size_t)gi * S2 + k : cdf;
    cp_async16(scf + c, gp, gi >= 0 ? 16 : 0);
  }
  cp_async_wait_all();
  __syncthreads();
  // split x in place
  __shared__ int s_tiny[BU][32];
  for (int c = tid; c < NC * 32; c += BU * 32) smf[c] = split_bits(smd[c], tiny);  // lane c % 32 == lane
  s_tiny[w][lane] = tiny;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < BU; ++k) tiny |= s_tiny[k][lane] != 0;
  float acc = 0.f, accb = 0.f;
  const int iu = bu * BU + w;
  auto emit = [&](int i, float s, float c, float bnd) {
    if (!mine) return;
    const float2 bp = split_bits(src >= 0 ? rhs[((size_t)(src / 32) * G.N + i) * 32 + (src % 32)] : 0.0, tiny);
    float d, de;
    two_sum(bp.x, -s, d, de);
    const float rt = __fadd_rn(d, __fadd_rn(de, __fsub_rn(bp.y, c)));
    r[((size_t)t * G.N + i) * 32 + lane] = rt;
    acc = fmaf(rt, rt, acc);
    accb = fmaf(bnd, bnd, accb);
  };
  if (iu < G.nlu) {
#pragma unroll 1
    for (int j = 0; j < BV; ++j) {
      const int i = srow[j * BU + w];
      if (i < 0) continue;
      const float4* cf = scf + (size_t)(j * BU + w) * S2;
      const float2* zw = smf + ((size_t)j * CU + w) * 32 + lane;
      // S x and M x side by side on the packed instructions
      float2 sp = make_float2(0.f, 0.f), cp = make_float2(0.f, 0.f);
      float b1 = 0.f, b2 = 0.f;
#pragma unroll 4  // (residuals of the 128 x 128 bicubic sphere, 1136 systems: 727 us a launch, unroll 1: 797)
      for (int dv = 0; dv < SW; ++dv)
#pragma unroll
        for (int du = 0; du < SW; ++du) {
          float4 q = cf[dv * SW + du];
          float2 z = zw[(dv * CU + du) * 32];
          df_acc2(sp, cp, b1, b2, make_float2(q.x, q.z), make_float2(q.y, q.w), make_float2(z.x, z.x),
                  make_float2(z.y, z.y));
        }
      if (i >= 0) {
        float2 a = df_axpy(sp.x, cp.x, sgp.x, sgp.y, sp.y, cp.y);  // S x + sigma M x
        emit(i, a.x, a.y, fmaf(sgp.x, b2, b1));
      }
    }
  }
  block_reduce((double)acc, part, t);
  __syncthreads();
  block_reduce(tiny && mine ? HUGE_VAL : (double)accb, part_bound, t);  // +inf fails the caller's error check
}

// The same residual for groups of one-shift tiles (the list of the one-shift
// kernel): a block computes its window's DOF ids and the combined double-float
// rows A = S + sigma M of its shift once, then streams the x windows of the
// group's flagged tiles through shared memory.
template <int P>
struct DfUniLayout {
  static constexpr int BV = BvOf<P>::value;
  static constexpr int CU = BU + 2 * P, CV = BV + 2 * P, NC = CU * CV, S2 = (2 * P + 1) * (2 * P + 1);
  static constexpr size_t win = (size_t)NC * 32 * sizeof(double);          // x window (raw rows at set-up)
  static constexpr size_t raw = (size_t)BU * BV * S2 * sizeof(float4);      // (S_hi, S_lo, M_hi, M_lo) rows
  static constexpr size_t pairs = (size_t)BU * (BV / 2) * S2 * sizeof(float4);  // combined row pairs
  static constexpr size_t ids = (size_t)(NC + BU * BV) * sizeof(int);
  static constexpr size_t total = win + pairs + ids;
  static_assert(raw <= win, "the raw rows are staged in the window area");
};

template <int P>
__global__ void __launch_bounds__(BU * 32, 3)
    k_sten_trueres_df_uni(StenGeo G, const float4* __restrict__ cdf, const double* __restrict__ x, int tiles,
                          const int* __restrict__ tile_rep, const int2* __restrict__ groups, int split,
                          const double* __restrict__ sigma, const double* __restrict__ rhs,
                          const int* __restrict__ src_of, const int* __restrict__ rep, float* __restrict__ r,
                          double* __restrict__ part, double* __restrict__ part_bound) {
  wm_wait_previous();
  constexpr int BV = BvOf<P>::value;
  using LY = DfUniLayout<P>;
  constexpr int SW = 2 * P + 1, CU = LY::CU, NC = LY::NC, S2 = LY::S2;
  constexpr int NT = BU * 32;
  extern __shared__ __align__(16) unsigned char smraw[];
  double* smd = reinterpret_cast<double*>(smraw);
  float2* smf = reinterpret_cast<float2*>(smraw);  // the same cells after the split
  float4* sraw = reinterpret_cast<float4*>(smraw);  // set-up only
  float4* scf = reinterpret_cast<float4*>(smraw + LY::win);
  int* sid = reinterpret_cast<int*>(smraw + LY::win + LY::pairs);
  int* srow = sid + NC;
  __shared__ int s_tiny[BU][32];
  const int lane = threadIdx.x, w = threadIdx.y;
  const int tid = w * 32 + lane;
  int b = blockIdx.x;
  const int bu = b % G.nbu;
  b /= G.nbu;
  const int bv = b % G.nbv;
  const int m = b / G.nbv;
  const int2 gr = groups[blockIdx.y / split];
  const int sp = blockIdx.y % split;
  const int per = (gr.y + split - 1) / split;
  const int ta = gr.x + sp * per;
  const int tb = min(min(gr.x + gr.y, ta + per), tiles);
  unsigned todo = 0;  // flagged tiles of the range, bit t - ta
  for (int t = ta; t < tb; ++t)
    if (tile_rep[t]) todo |= 1u << (t - ta);
  if (todo == 0) return;
  bool tiny = false;
  const float2 sgp = split_bits(sigma[gr.x * 32], tiny);  // the group's shift (a tiny shift only loses itself)
  // set-up: global DOF of every window cell and every output row
  const int32_t* E = G.ext + (size_t)m * G.ELV * G.ELU;
  const int32_t* OWN = G.own + (size_t)m * G.nlv * G.nlu;
  for (int c = tid; c < NC + BU * BV; c += NT) {
    int v = -1;
    if (c < NC) {
      int eu = bu * BU + c % CU, ev = bv * BV + c / CU;
      if (eu < G.ELU && ev < G.ELV) v = E[(size_t)ev * G.ELU + eu];
    } else {
      int o = c - NC;
      int iu = bu * BU + o % BU, iv = bv * BV + o / BU;
      if (iu < G.nlu && iv < G.nlv) v = OWN[(size_t)iv * G.nlu + iu];
    }
    sid[c] = v;
  }
  __syncthreads();
  for (int c = tid; c < BU * BV * S2; c += NT) {
    const int o = c / S2, k = c % S2;
    const int gi = srow[o];
    cp_async16(sraw + c, gi >= 0 ? cdf + (size_t)gi * S2 + k : cdf, gi >= 0 ? 16 : 0);
  }
  cp_async_wait_all();
  __syncthreads();
  // combined rows A = S + sigma M as row pairs: entry (pair jj*BU + w, slot) =
  // (A_hi of rows 2jj and 2jj+1, A_lo of both), the operands of the packed loop
  for (int c = tid; c < BU * (BV / 2) * S2; c += NT) {
    const int pi = c / S2, sl = c - pi * S2;
    const int o0 = (pi / BU) * 2 * BU + pi % BU;  // rows 2jj and 2jj+1 of column w
    const float4 q0 = sraw[o0 * S2 + sl], q1 = sraw[(o0 + BU) * S2 + sl];
    const float2 a0 = df_axpy(q0.x, q0.y, sgp.x, sgp.y, q0.z, q0.w);
    const float2 a1 = df_axpy(q1.x, q1.y, sgp.x, sgp.y, q1.z, q1.w);
    scf[c] = make_float4(a0.x, a1.x, a0.y, a1.y);
  }
  __syncthreads();  // the raw rows are dead: the window area is free
  const int iu = bu * BU + w;
  while (todo) {
    const int t = ta + __ffs(todo) - 1;
    todo &= todo - 1;
    const int g = t * 32 + lane;
    const bool mine = rep[g] != 0;
    const int src = src_of[g];
    for (int c = tid; c < NC * 16; c += NT) {  // x window: 16 chunks of 16 bytes per cell
      const int part16 = c % 16, cell = c / 16;
      const int gi = sid[cell];
      cp_async16(smd + (size_t)cell * 32 + part16 * 2, gi >= 0 ? x + ((size_t)t * G.N + gi) * 32 + part16 * 2 : x,
                 gi >= 0 ? 16 : 0);
    }
    cp_async_wait_all();
    __syncthreads();
    tiny = false;
    for (int c = tid; c < NC * 32; c += NT) smf[c] = split_bits(smd[c], tiny);  // lane c % 32 == lane
    s_tiny[w][lane] = tiny;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < BU; ++k) tiny |= s_tiny[k][lane] != 0;
    float acc = 0.f, accb = 0.f;
    auto emit = [&](int i, float s, float c, float bnd) {
      if (!mine) return;
      const float2 bp = split_bits(src >= 0 ? rhs[((size_t)(src / 32) * G.N + i) * 32 + (src % 32)] : 0.0, tiny);
      float d, de;
      two_sum(bp.x, -s, d, de);
      const float rt = __fadd_rn(d, __fadd_rn(de, __fsub_rn(bp.y, c)));
      r[((size_t)t * G.N + i) * 32 + lane] = rt;
      acc = fmaf(rt, rt, acc);
      accb = fmaf(bnd, bnd, accb);
    };
    if (iu < G.nlu) {
#pragma unroll 1
      for (int j = 0; j < BV; j += 2) {
        const int i0 = srow[j * BU + w], i1 = srow[(j + 1) * BU + w];
        if (i0 < 0 && i1 < 0) continue;  // rows past the patch edge or owned by another patch
        const float4* cf = scf + (size_t)((j / 2) * BU + w) * S2;  // row pair (j, j+1)
        const float2* zw = smf + ((size_t)j * CU + w) * 32 + lane;
        float2 spp = make_float2(0.f, 0.f), cpp = make_float2(0.f, 0.f);
        float b0 = 0.f, b1 = 0.f;
#pragma unroll
        for (int dv = 0; dv < SW; ++dv)
#pragma unroll
          for (int du = 0; du < SW; ++du) {
            const float4 q = cf[dv * SW + du];
            const float2 z0 = zw[(dv * CU + du) * 32], z1 = zw[((dv + 1) * CU + du) * 32];
            df_acc2(spp, cpp, b0, b1, make_float2(q.x, q.y), make_float2(q.z, q.w), make_float2(z0.x, z1.x),
                    make_float2(z0.y, z1.y));
          }
        if (i0 >= 0) emit(i0, spp.x, cpp.x, b0);
        if (i1 >= 0) emit(i1, spp.y, cpp.y, b1);
      }
    }
    block_reduce((double)acc, part, t);
    __syncthreads();
    block_reduce(tiny && mine ? HUGE_VAL : (double)accb, part_bound, t);  // +inf fails the caller's error check
    __syncthreads();  // the window and the reduction buffer may be refilled
  }
}

__global__ void k_build_csm(int N, int W, int S2, const int16_t* __restrict__ slot, const double* __restrict__ S,
                            const double* __restrict__ M, double2* __restrict__ c64, float4* __restrict__ cdf) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= (int64_t)N * W) return;
  int sl = slot[t];
  if (sl < 0) return;
  int i = (int)(t / W);
  c64[(size_t)i * S2 + sl] = make_double2(S[t], M[t]);
  float sh = (float)S[t], mh = (float)M[t];
  cdf[(size_t)i * S2 + sl] = make_float4(sh, (float)(S[t] - (double)sh), mh, (float)(M[t] - (double)mh));
}

}  // namespace

// ====================================================================== host
// levels whose patches have fewer local DOFs per side keep the row kernels (with the
// tile-at-a-time kernels, moving the 10- and 18-wide levels of the sphere to the row
// kernels was slower: 174.5 and 184.0 against 172.5 ms per bench step)
#ifndef WM_STEN_MIN_NL
#define WM_STEN_MIN_NL 8
#endif

int wm_sten_build(const wm_geom_desc& g, int np, wm_level& L, cudaStream_t s) {
  L.sten = false;
  if (g.degree < 2 || g.degree > 3 || L.nlu < WM_STEN_MIN_NL || L.nlv < WM_STEN_MIN_NL) return WM_OK;
  std::vector<int32_t> ext, own;
  std::vector<int16_t> slot;
  if (wm_host_stencil(g, np, L, ext, own, slot) != WM_OK) return WM_OK;  // row kernels only
  const int p = g.degree, S2 = (2 * p + 1) * (2 * p + 1);
  L.ELU = L.nlu + 2 * p;
  L.ELV = L.nlv + 2 * p;
  L.nbu = (L.nlu + BU - 1) / BU;
  const int bv = p == 2 ? BvOf<2>::value : BvOf<3>::value;
  L.nbv = (L.nlv + bv - 1) / bv;
  WM_TRY(L.d_ext.upload(ext, s));
  WM_TRY(L.d_own.upload(own, s));
  DevBuf<int16_t> d_slot;
  WM_TRY(d_slot.upload(slot, s));
  WM_TRY(L.d_csm64.alloc((size_t)L.N * S2));
  WM_TRY(L.d_csmdf.alloc((size_t)L.N * S2));
  WM_CUDA(cudaMemsetAsync(L.d_csm64.p, 0, sizeof(double2) * (size_t)L.N * S2, s));
  WM_CUDA(cudaMemsetAsync(L.d_csmdf.p, 0, sizeof(float4) * (size_t)L.N * S2, s));
  int64_t n = (int64_t)L.N * L.W;
  WM_LAUNCH(WM_PC_ASSEMBLY, s, k_build_csm<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(
                                   L.N, L.W, S2, d_slot.p, L.d_S64.p, L.d_M64.p, L.d_csm64.p, L.d_csmdf.p));
  WM_CUDA(cudaGetLastError());
  WM_CUDA(cudaStreamSynchronize(s));
  d_slot.release();
  WM_TRY(wm_stream_build(np, p, L, ext, s));
  L.sten = true;
  return WM_OK;
}

int wm_sten_chunks(const wm_level& L, int np) { return L.sten ? np * L.nbu * L.nbv : 0; }

#define WM_DISPATCH_P(P_, ...)                     \
  switch (P_) {                                    \
    case 2: {                                      \
      constexpr int PP = 2;                        \
      __VA_ARGS__;                                 \
    } break;                                       \
    case 3: {                                      \
      constexpr int PP = 3;                        \
      __VA_ARGS__;                                 \
    } break;                                       \
    default: return WM_ERR_UNSUPPORTED;            \
  }

// SMs of the current device (grid sizing of the one-shift kernel)
static int device_sms() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    return 152;
  }
  return n > 0 ? n : 152;
}

template <int P, int MODE>
static int launch_uni(const wm_level& L, int np, int tiles, const UniTiles& ut, int kstep, const double* sigma,
                      const double2* ctab, const int* sid, const double* r, const double* z, const double* prev,
                      double* out, const int* tile_active, double* part, int cat, cudaStream_t s,
                      const double* qd = nullptr, double* part2 = nullptr, double* out1 = nullptr) {
  constexpr size_t sm = UniLayout<P, MODE>::total;
  static bool configured = false;
  if (!configured) {
    WM_CUDA(cudaFuncSetAttribute(k_sten_uni<P, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    configured = true;
  }
  if (ut.n_groups <= 0) return WM_OK;
  static const int sms = device_sms();
  const int bx = np * L.nbu * L.nbv;
  // blocks that share a group: enough blocks for ut.waves waves
  const int64_t want = (int64_t)ut.waves * sms * UniMinBlocks<P, MODE>::value;
  int split = 1;
  while (split < kUniGroup && (int64_t)bx * ut.n_groups * split < want) split *= 2;
  const int gmax = 65535 / split;  // grid.y limit
  for (int g0 = 0; g0 < ut.n_groups; g0 += gmax) {
    const int ng = std::min(gmax, ut.n_groups - g0);
    dim3 grid(bx, ng * split);
    WM_TRY(wm_launch_next(cat, (k_sten_uni<P, MODE>), grid, dim3(32, BU), sm, s, geo_of(L), L.d_csm64.p, L.d_dS64.p,
        L.d_dM64.p, sigma, ctab, sid, kstep, z, r, prev, out, tiles, tile_active, ut.groups + g0, split, part, qd,
        part2, out1));
    WM_CUDA(cudaGetLastError());
  }
  return WM_OK;
}

int wm_sten_cheb_step(const wm_level& L, int np, int p, int tiles, int kstep, const double* sigma,
                      const double2* ctab, const int* sid, const double* r, const double* z, const double* prev,
                      double* out, const int* tile_active, const UniTiles& ut, int cat, cudaStream_t s,
                      const double* q, double* part_rz, double* part_zq, bool generic_only) {
  if (generic_only) {
    // the one-shift tiles were done elsewhere: generic kernel for the others only
  } else if (ut.n > 0 && part_rz) {
    WM_DISPATCH_P(p, { WM_TRY((launch_uni<PP, UNI_CHEBDOT>(L, np, tiles, ut, kstep, sigma, ctab, sid, r, z, prev,
                                                           out, tile_active, part_rz, cat, s, q, part_zq))); });
  } else if (ut.n > 0) {
    WM_DISPATCH_P(p, { WM_TRY((launch_uni<PP, UNI_CHEB>(L, np, tiles, ut, kstep, sigma, ctab, sid, r, z, prev, out,
                                                        tile_active, nullptr, cat, s))); });
  }
  if (ut.n >= tiles) return WM_OK;
  ChebEpi e;
  e.N = L.N;
  e.kstep = kstep;
  e.dS = L.d_dS64.p;
  e.dM = L.d_dM64.p;
  e.out = out;
  e.sigma = sigma;
  e.ctab = ctab;
  e.sid = sid;
  e.in[0] = r;
  e.in[1] = prev;
  const int* skip = ut.n > 0 ? ut.flag : nullptr;
  WM_DISPATCH_P(p, return launch<PP>(L, np, tiles, z, tile_active, e, cat, s, skip));
  return WM_OK;
}

int wm_sten_cheb_first2(const wm_level& L, int np, int p, int tiles, const double* sigma, const double2* ctab,
                        const int* sid, const double* r, double* z1, double* z2, const int* tile_active,
                        const UniTiles& ut, int cat, cudaStream_t s) {
  WM_DISPATCH_P(p, { WM_TRY((launch_uni<PP, UNI_CHEB1>(L, np, tiles, ut, 1, sigma, ctab, sid, nullptr, r, nullptr, z2,
                                                       tile_active, nullptr, cat, s, nullptr, nullptr, z1))); });
  return WM_OK;
}

int wm_sten_residual(const wm_level& L, int np, int p, int tiles, const double* sigma, const double* r,
                     const double* z, double* res, const int* tile_active, const UniTiles& ut, int cat,
                     cudaStream_t s) {
  if (ut.n > 0) {
    WM_DISPATCH_P(p, { WM_TRY((launch_uni<PP, UNI_RESID>(L, np, tiles, ut, 0, sigma, nullptr, nullptr, r, z, nullptr,
                                                         res, tile_active, nullptr, cat, s))); });
    if (ut.n >= tiles) return WM_OK;
  }
  ResidEpi e;
  e.N = L.N;
  e.res = res;
  e.sigma = sigma;
  e.in[0] = r;
  const int* skip = ut.n > 0 ? ut.flag : nullptr;
  WM_DISPATCH_P(p, return launch<PP>(L, np, tiles, z, tile_active, e, cat, s, skip));
  return WM_OK;
}

int wm_sten_apply_pq(const wm_level& L, int np, int p, int tiles, const double* sigma, const double* pv, double* q,
                     const int* tile_active, const UniTiles& ut, double* part, cudaStream_t s) {
  if (ut.n > 0) {
    WM_DISPATCH_P(p, { WM_TRY((launch_uni<PP, UNI_APPLY>(L, np, tiles, ut, 0, sigma, nullptr, nullptr, nullptr, pv,
                                                         nullptr, q, tile_active, part, WM_PC_APPLY64, s))); });
    if (ut.n >= tiles) return WM_OK;
  }
  ApplyEpi e;
  e.N = L.N;
  e.q = q;
  e.sigma = sigma;
  e.part = part;
  const int* skip = ut.n > 0 ? ut.flag : nullptr;
  WM_DISPATCH_P(p, return launch<PP>(L, np, tiles, pv, tile_active, e, WM_PC_APPLY64, s, skip));
  return WM_OK;
}

template <typename Tr>
int wm_sten_true_residual(const wm_level& L, int np, int p, int tiles, const double* sigma, const double* x,
                          const double* rhs, const int* src_of, const int* rep, const int* tile_rep, Tr* r,
                          double* part, cudaStream_t s) {
  TrueResEpi<Tr> e;
  e.N = L.N;
  e.rhs = rhs;
  e.src_of = src_of;
  e.rep = rep;
  e.r = r;
  e.sigma = sigma;
  e.part = part;
  WM_DISPATCH_P(p, return launch<PP>(L, np, tiles, x, tile_rep, e, WM_PC_TRUERES, s));
  return WM_OK;
}

int wm_sten_dots(const wm_level& L, int np, int p, const int* list, int n, const float* r, const float* z,
                 const float* q, const int* tile_active, double* part_rz, double* part_zq, int stride,
                 cudaStream_t s) {
  for (int k = 0; k < n; k += 65535)  // grid.y limit
    WM_DISPATCH_P(p, {
      WM_TRY(wm_launch_next(WM_PC_CGVEC, k_sten_dots<PP>, dim3(np * L.nbu * L.nbv, std::min(65535, n - k)), dim3(32, BU),
                            0, s, geo_of(L), list + k, r, z, q, tile_active, part_rz, part_zq, stride));
    });
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

template <int P>
static int launch_df(const wm_level& L, int np, int tiles, const UniTiles& ut, const double* sigma, const double* x,
                     const double* rhs, const int* src_of, const int* rep, const int* tile_rep, float* r, double* part,
                     double* part_bound, cudaStream_t s) {
  constexpr size_t sm = DfLayout<P>::total;
  constexpr size_t smu = DfUniLayout<P>::total;
  static bool configured = false;
  if (!configured) {
    WM_CUDA(cudaFuncSetAttribute(k_sten_trueres_df<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    WM_CUDA(cudaFuncSetAttribute(k_sten_trueres_df_uni<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smu));
    configured = true;
  }
  const int bx = np * L.nbu * L.nbv;
  if (ut.n_groups > 0) {
    static const int sms = device_sms();
    const int64_t want = (int64_t)ut.waves * sms * 3;
    int split = 1;
    while (split < kUniGroup && (int64_t)bx * ut.n_groups * split < want) split *= 2;
    const int gmax = 65535 / split;
    for (int g0 = 0; g0 < ut.n_groups; g0 += gmax) {
      const int ng = std::min(gmax, ut.n_groups - g0);
      WM_TRY(wm_launch_next(WM_PC_TRUERES, k_sten_trueres_df_uni<P>, dim3(bx, ng * split), dim3(32, BU), smu, s,
          geo_of(L), L.d_csmdf.p, x, tiles, tile_rep, ut.groups + g0, split, sigma, rhs, src_of, rep, r, part,
          part_bound));
      WM_CUDA(cudaGetLastError());
    }
  }
  if (ut.n < tiles) {
    WM_TRY(wm_launch_next(WM_PC_TRUERES, k_sten_trueres_df<P>, dim3(bx, tiles), dim3(32, BU), sm, s, geo_of(L), L.d_csmdf.p, x,
        tiles, tile_rep, sigma, rhs, src_of, rep, r, part, part_bound, ut.flag));
    WM_CUDA(cudaGetLastError());
  }
  return WM_OK;
}

int wm_sten_true_residual_df(const wm_level& L, int np, int p, int tiles, const UniTiles& ut, const double* sigma,
                             const double* x, const double* rhs, const int* src_of, const int* rep,
                             const int* tile_rep, float* r, double* part, double* part_bound, cudaStream_t s) {
  WM_DISPATCH_P(p, {
    return launch_df<PP>(L, np, tiles, ut, sigma, x, rhs, src_of, rep, tile_rep, r, part, part_bound, s);
  });
  return WM_OK;
}

template int wm_sten_true_residual<float>(const wm_level&, int, int, int, const double*, const double*, const double*,
                                          const int*, const int*, const int*, float*, double*, cudaStream_t);
template int wm_sten_true_residual<double>(const wm_level&, int, int, int, const double*, const double*,
                                           const double*, const int*, const int*, const int*, double*, double*,
                                           cudaStream_t);
