// Shared-memory stencil kernels (wm_stencil.cu) for levels with a stencil form.
#pragma once

#include "wm_internal.h"

#ifndef WM_MAX_CHEB
#define WM_MAX_CHEB 8
#endif

// Tiles whose 32 systems share one shift (sample-major packing: the 32 samples
// of one sinc node), for the combined-coefficient kernel: a per-tile flag (the
// generic kernel skips those tiles) and groups of at most kUniGroup
// consecutive such tiles with the same shift index, each (first tile, count).
// A block of the one-shift kernel serves one group (or part of one).
constexpr int kUniGroup = 8;
struct UniTiles {
  const int* flag = nullptr;     // [tiles] 1 where the 32 shifts of the tile are equal
  int n = 0;                     // number of such tiles
  const int2* groups = nullptr;  // [n_groups] (first tile, count), count in 1..kUniGroup
  int n_groups = 0;
  int waves = 4;                 // grid target: runs are split until the grid has this many waves
};

// Builds the stencil form of a level (extended grids, owner map, coefficient
// slots) after its rows are assembled; leaves L.sten = false when the level
// keeps the row kernels (degree outside 2..3, patches narrower than 8).
int wm_sten_build(const wm_geom_desc& g, int np, wm_level& L, cudaStream_t s);
// number of spatial blocks of a stencil launch on the level (partial-sum chunks)
int wm_sten_chunks(const wm_level& L, int np);

// Float64 steps.  Three-term Chebyshev step
// out = z + c1 (z - prev) + c2 D^{-1} (r - A z)
// (c1 = 0 at kstep 0, prev = nullptr for z_prev = 0; out may alias prev).
// ctab: (c1, c2) per [shift][step] of the level (WM_MAX_CHEB steps per shift).
// The one-shift tiles of `ut` go to the combined-coefficient kernel, the
// others to the generic one.
int wm_sten_cheb_step(const wm_level& L, int np, int p, int tiles, int kstep, const double* sigma,
                      const double2* ctab, const int* sid, const double* r, const double* z, const double* prev,
                      double* out, const int* tile_active, const UniTiles& ut, int cat, cudaStream_t s,
                      const double* q = nullptr, double* part_rz = nullptr, double* part_zq = nullptr,
                      bool generic_only = false);
// With part_rz set, the one-shift tiles of the step also leave per-block partial
// sums (r, out) in part_rz and, with q set, (out, q) in part_zq ([tile][chunk][32],
// chunk = spatial block); the other tiles get none (the caller forms them).
// generic_only: the one-shift tiles are left alone (done by another launch).
// The first two pre-smoothing steps from z = 0 for the one-shift tiles only:
// z1 = c2_0 D^{-1} r and z2 = z1 + c1_1 z1 + c2_1 D^{-1} (r - A z1) in one pass
// over the window of r (the other tiles take the row-form first step and
// wm_sten_cheb_step with generic_only).
int wm_sten_cheb_first2(const wm_level& L, int np, int p, int tiles, const double* sigma, const double2* ctab,
                        const int* sid, const double* r, double* z1, double* z2, const int* tile_active,
                        const UniTiles& ut, int cat, cudaStream_t s);
// residual res = r - A z and outer apply q = A p with per-block partial sums
// (p, q) in `part` ([tile][chunk][32], chunk = spatial block); the one-shift
// tiles of `ut` take the combined-coefficient kernel
int wm_sten_residual(const wm_level& L, int np, int p, int tiles, const double* sigma, const double* r,
                     const double* z, double* res, const int* tile_active, const UniTiles& ut, int cat,
                     cudaStream_t s);
int wm_sten_apply_pq(const wm_level& L, int np, int p, int tiles, const double* sigma, const double* pv, double* q,
                     const int* tile_active, const UniTiles& ut, double* part, cudaStream_t s);
// partial sums (r, z) and (z, q) of the n tiles in `list` by the row blocks of the steps
// above ([tile][stride][32], chunk = spatial block), with their float sums
int wm_sten_dots(const wm_level& L, int np, int p, const int* list, int n, const float* r, const float* z,
                 const float* q, const int* tile_active, double* part_rz, double* part_zq, int stride,
                 cudaStream_t s);
template <typename Tr>
int wm_sten_true_residual(const wm_level& L, int np, int p, int tiles, const double* sigma, const double* x,
                          const double* rhs, const int* src_of, const int* rep, const int* tile_rep, Tr* r,
                          double* part, cudaStream_t s);
// the same residual (float output) with the stencil sums in double-float
// arithmetic on the FP32 pipes; part_bound receives the per-block partial
// sums of ||B||^2 with B_i = sum_j |a_ij| |x_j| (the rounding error of entry i
// is below 2^-42 B_i), or +inf for a system with a value below 2^-102
// (one-shift tiles of `ut` by groups, the others one tile per block)
int wm_sten_true_residual_df(const wm_level& L, int np, int p, int tiles, const UniTiles& ut,
                             const double* sigma, const double* x, const double* rhs, const int* src_of, const int* rep,
                             const int* tile_rep, float* r, double* part, double* part_bound, cudaStream_t s);

// ---- streaming kernels of the float solves (wm_stream.h): every tile, any shifts
constexpr int kStreamTiles = 4;  // tiles of a block
// The batch's tiles in groups of up to kStreamTiles (tile ids, -1: none): n[0] groups of
// two pairs of tiles, each pair of one shift, n[1] of tiles of one shift each, then n[2]
// of tiles of any shifts; `order`: the tiles one by one in the same order, the first n_pair
// of the pairs, the first n_uni of one shift.
struct StreamTiles {
  const int4* groups = nullptr;
  const int* order = nullptr;
  int n[3] = {0, 0, 0};
  int tiles = 0, n_pair = 0, n_uni = 0;
};
// the grouping: `uni` flags the tiles of one shift, `shift` is its index
void wm_stream_groups(const std::vector<int>& uni, const std::vector<int>& shift, std::vector<int4>& groups,
                      std::vector<int>& order, StreamTiles* st);
// ST_CHEB     three-term Chebyshev step out = z + c1 (z - prev) + c2 D^{-1} (r - A z)
//             (c1 = 0 at kstep 0; prev = nullptr there; out may alias prev)
// ST_CHEBDOT  the same, with the partial sums (r, out) in part and (out, q) in part2 for
//             the tiles that wm_stream_items counts
// ST_CHEB1    the first two steps from z = 0 in one pass over z (which is r here):
//             out1 = z1 = c2_0 D^{-1} r, out = z1 + c1_1 z1 + c2_1 D^{-1} (r - A z1)
// ST_RESID    out = r - A z
// ST_APPLY    out = A z, with the partial sums (z, out) in part
// Partial sums: [tile][item][32], wm_stream_items() items (rows of pstride items).
enum { ST_CHEB = 0, ST_RESID = 1, ST_APPLY = 2, ST_CHEBDOT = 3, ST_CHEB1 = 4 };
struct StreamArgs {
  const wm_level* L = nullptr;
  int np = 0;
  StreamTiles st;
  int kstep = 0;
  const double* sigma = nullptr;
  const float2* ctab = nullptr;  // the level's (c1, c2) per [shift][step]
  const int* sid = nullptr;
  const int* tile_active = nullptr;
  const float *z = nullptr, *r = nullptr, *prev = nullptr, *q = nullptr;
  float *out = nullptr, *out1 = nullptr;
  double *part = nullptr, *part2 = nullptr;
  int pstride = 0;  // items of a tile's row of part (0: wm_stream_items())
  int cat = 0;
  cudaStream_t s = nullptr;
};
int wm_stream(int p, int mode, const StreamArgs& a);
int wm_stream_build(int np, int p, wm_level& L, const std::vector<int32_t>& ext, cudaStream_t s);
// whether a diagonal of S + sigma M on the level is beyond the kernels' quotients (wm_quotient.h):
// the row kernels then do the float steps
bool wm_stream_far(const wm_level& L, double sigma);
// partial sums per tile and system of the kernels that form dot products (`fused`: of
// how many of the first tiles of st.order ST_CHEBDOT forms them), and the most that a solve of up to `tiles` tiles leaves over all its tiles
int wm_stream_items(const wm_level& L, int np, int p, const StreamTiles& st, int* fused = nullptr);
size_t wm_stream_part_max(const wm_level& L, int np, int tiles);
