// Tables and launches of the streaming stencil kernels (wm_stream.h).
#include "wm_stream.h"

extern template int wm_stream_run<2>(int, const StreamArgs&);
extern template int wm_stream_run<3>(int, const StreamArgs&);

namespace {

// the ColRow table: zero coefficients for outputs that are not computed here
template <int P>
__global__ void k_stream_cols(int64_t n, int nlu, int nlv, int ELV, const int32_t* __restrict__ own,
                              const double2* __restrict__ csm, const float* __restrict__ dS,
                              const float* __restrict__ dM, ColRow<P>* __restrict__ out) {
  constexpr int SW = 2 * P + 1, S2 = SW * SW;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int e = (int)(t % S2);
  const int64_t b = t / S2;
  const int u = (int)(b % nlu), s = (int)((b / nlu) % ELV), m = (int)(b / ((int64_t)nlu * ELV));
  const int du = e / SW, dv = e % SW, j = s - dv;
  auto row = [&](int jj) { return jj >= 0 && jj < nlv ? own[((size_t)m * nlv + jj) * nlu + u] : -1; };
  float2 v = make_float2(0.f, 0.f);
  const int i = row(j);
  if (i >= 0) {
    const double2 a = csm[(size_t)i * S2 + dv * SW + du];
    v = make_float2((float)a.x, (float)a.y);
  }
  out[b].coef[e] = v;
  if (e == 0) {
    const int o = row(s - 2 * P);
    out[b].own = o;
    out[b].diag = o >= 0 ? make_float2(dS[o], dM[o]) : make_float2(1.f, 0.f);
  }
}

// diagonals (dS, dM) of the cells ((1, 0) where there is none); ids become 32 x id, 0 for none
__global__ void k_stream_diag(int64_t n, int32_t* __restrict__ ids, const float* __restrict__ dS,
                              const float* __restrict__ dM, float2* __restrict__ d) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int i = ids[t];
  d[t] = i >= 0 ? make_float2(dS[i], dM[i]) : make_float2(1.f, 0.f);
  ids[t] = i >= 0 ? 32 * i : 0;  // (no cell: DOF 0 is read, with a coefficient of zero)
}

// by window row and column: 32 x the row that the window row completes (0: none)
__global__ void k_stream_done(int64_t n, int nlu, int nlv, int ELV, int EU, const int32_t* __restrict__ own,
                              int32_t* __restrict__ done) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const int u = (int)(t % EU), s = (int)((t / EU) % ELV), m = (int)(t / ((int64_t)EU * ELV));
  const int j = s - (ELV - nlv);
  const int i = u < nlu && j >= 0 ? own[((size_t)m * nlv + j) * nlu + u] : -1;
  done[t] = i >= 0 ? 32 * i : 0;
}

// largest entry of each of two arrays of positive numbers (as their bits)
__global__ void k_stream_max(int n, const float* __restrict__ a, const float* __restrict__ b, int* __restrict__ most) {
  int ma = 0, mb = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    ma = max(ma, __float_as_int(a[i]));
    mb = max(mb, __float_as_int(b[i]));
  }
  atomicMax(most, __reduce_max_sync(0xffffffffu, ma));
  atomicMax(most + 1, __reduce_max_sync(0xffffffffu, mb));
}

template <int P>
int build(int np, wm_level& L, const std::vector<int32_t>& ext, cudaStream_t s) {
  const int EU = strips(L) * kBU + 2 * P, ELV = L.nlv + 2 * P, ELU = L.nlu + 2 * P;
  std::vector<int32_t> e((size_t)np * ELV * EU, -1);
  for (int64_t row = 0; row < (int64_t)np * ELV; ++row)
    std::copy_n(ext.begin() + row * ELU, ELU, e.begin() + row * EU);
  const int64_t ne = (int64_t)e.size(), nc = (int64_t)np * ELV * L.nlu * ColRow<P>::S2;
  auto nb = [](int64_t n) { return (unsigned)((n + 255) / 256); };
  WM_TRY(L.d_st_ext.upload(e, s));
  WM_TRY(L.d_st_dext.alloc(e.size()));
  WM_TRY(L.d_st_done.alloc(e.size()));
  WM_TRY(L.d_st_cols.alloc((size_t)np * ELV * L.nlu * sizeof(ColRow<P>)));
  WM_LAUNCH(WM_PC_ASSEMBLY, s, k_stream_done<<<nb(ne), 256, 0, s>>>(ne, L.nlu, L.nlv, ELV, EU, L.d_own.p,
                                                                    L.d_st_done.p));
  WM_LAUNCH(WM_PC_ASSEMBLY, s, k_stream_cols<P><<<nb(nc), 256, 0, s>>>(
                                   nc, L.nlu, L.nlv, ELV, L.d_own.p, L.d_csm64.p, L.d_dS32.p, L.d_dM32.p,
                                   reinterpret_cast<ColRow<P>*>(L.d_st_cols.p)));
  WM_LAUNCH(WM_PC_ASSEMBLY, s, k_stream_diag<<<nb(ne), 256, 0, s>>>(ne, L.d_st_ext.p, L.d_dS32.p, L.d_dM32.p,
                                                                    L.d_st_dext.p));
  DevBuf<int> most;
  WM_TRY(most.alloc(2));
  WM_CUDA(cudaMemsetAsync(most.p, 0, 2 * sizeof(int), s));
  WM_LAUNCH(WM_PC_ASSEMBLY, s, k_stream_max<<<std::min(nb(L.N), 1024u), 256, 0, s>>>(L.N, L.d_dS32.p, L.d_dM32.p, most.p));
  WM_CUDA(cudaGetLastError());
  WM_CUDA(cudaMemcpyAsync(L.diag_max, most.p, sizeof(L.diag_max), cudaMemcpyDeviceToHost, s));
  WM_CUDA(cudaStreamSynchronize(s));  // (the host table goes out of scope)
  most.release();
  return WM_OK;
}

}  // namespace

int wm_stream_build(int np, int p, wm_level& L, const std::vector<int32_t>& ext, cudaStream_t s) {
  return p == 2 ? build<2>(np, L, ext, s) : build<3>(np, L, ext, s);
}

bool wm_stream_far(const wm_level& L, double sigma) {
  return L.sten && !(sigma * L.diag_max[1] + L.diag_max[0] < 0x1p120);
}

int wm_stream_items(const wm_level& L, int np, int p, const StreamTiles& st, int* fused) {
  bool one = false;
  const StreamGeo G = stream_geo(L, np, p, st, true, &one);
  if (fused) *fused = !one && stream_pairs(G, st) ? st.n_pair : 0;
  return G.items;
}

size_t wm_stream_part_max(const wm_level& L, int np, int tiles) {
  // with base4 = strips x groups blocks: at least kSMs of them, items x tiles stay under
  // (strips + kWantBlocks / groups) tiles, groups >= tiles / 4; fewer, strips x chunks x tiles
  // with strips x tiles < 4 kSMs
  if (!L.sten) return 0;
  return (size_t)np * strips(L) * tiles + (size_t)kStreamTiles * kWantBlocks +
         (size_t)kStreamTiles * kSMs * std::max(1, L.nlv / kMinRows1);
}

int wm_stream(int p, int mode, const StreamArgs& a) {
  StreamArgs b = a;
  if (!b.prev) {  // no z_prev: step 0 (c1 = 0) reads z in its place
    if (mode == ST_CHEB || mode == ST_CHEBDOT)
      if (b.kstep != 0) return WM_ERR_INVALID_ARG;
    b.prev = b.z;
  }
  if (p == 2) return wm_stream_run<2>(mode, b);
  if (p == 3) return wm_stream_run<3>(mode, b);
  return WM_ERR_UNSUPPORTED;
}

void wm_stream_groups(const std::vector<int>& uni, const std::vector<int>& shift, std::vector<int4>& groups,
                      std::vector<int>& order, StreamTiles* st) {
  const int tiles = (int)uni.size();
  std::vector<int> one, kinds[3];  // kinds[0]: pairs, two entries each
  for (int t = 0; t < tiles; ++t) (uni[t] ? one : kinds[2]).push_back(t);
  for (size_t k = 0; k < one.size(); ++k) {
    const bool pair = k + 1 < one.size() && shift[one[k]] == shift[one[k + 1]];
    kinds[pair ? 0 : 1].push_back(one[k]);
    if (pair) kinds[0].push_back(one[++k]);
  }
  groups.clear();
  order.clear();
  for (int c = 0; c < 3; ++c) {
    const std::vector<int>& v = kinds[c];
    order.insert(order.end(), v.begin(), v.end());
    st->n[c] = 0;
    for (size_t k = 0; k < v.size(); k += kStreamTiles, ++st->n[c]) {
      auto at = [&](size_t j) { return j < v.size() ? v[j] : -1; };
      groups.push_back(make_int4(at(k), at(k + 1), at(k + 2), at(k + 3)));
    }
  }
  st->tiles = tiles;
  st->n_uni = (int)one.size();
  st->n_pair = (int)kinds[0].size();
}
