// White-noise loads from Philox4x32-10 normals at the Gauss points (Sec. 3.3).
//
// The discrete white noise b_s must have covariance M.  It is drawn at the
// Gauss points: b_s,i = sum_q sqrt(w_q a_q) xi_{s,q} phi_i(x_q), so that
// Cov(b_s) = B B^T is exactly the mass matrix of the same Gauss rule.
//
// Philox4x32-10 is written from its published definition (Salmon, Moraes,
// Dror, Shaw, SC'11): ten rounds of two 32x32->64 multiplications by
// 0xD2511F53 and 0xCD9E8D57 with the key bumped by (0x9E3779B9, 0xBB67AE85).
#include "wm_internal.h"
#include "wm_normal_tables.h"

namespace {

struct U4 {
  uint32_t x, y, z, w;
};

__device__ __forceinline__ U4 philox10(U4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    U4 n;
    n.x = hi1 ^ c.y ^ k0;
    n.y = lo1;
    n.z = hi0 ^ c.w ^ k1;
    n.w = lo0;
    c = n;
  }
  return c;
}

// the 53-bit uniform (n 2^-53) of two words, n in [1, 2^53]
__device__ __forceinline__ uint64_t uniform53(uint32_t hi, uint32_t lo) {
  return ((uint64_t)(hi >> 5) << 26) + (uint64_t)(lo >> 6) + 1ull;
}

// log(n 2^-53) for n in [1, 2^53]: table-driven reduction (P. T. P. Tang, "Table-driven
// implementation of the logarithm function in IEEE floating-point arithmetic", 1990) to
// log 2^e + log c + log1p(r) with |r| <= 2^-7 and the Taylor series of log1p, the
// leading sums kept exact.  Sixteen float64 operations, error below an ulp.
__device__ __forceinline__ double log_u53(uint64_t n) {
  const int sh = __clzll((long long)n) - 11;  // -1 for 2^53
  const uint64_t mant = (sh >= 0 ? n << sh : n >> 1) & 0xFFFFFFFFFFFFFull;
  const int j = (int)(mant >> 45);
  const int half = j >= 53;  // m/2 in [0.707, 1): log u near 0 has no cancellation
  const double m = __longlong_as_double((long long)(((uint64_t)(1023 - half) << 52) | mant));
  // e = half - 1 - sh as a double by its bits (-53 .. 0)
  const double e = __hiloint2double(0x43300000, 1024 + half - 1 - sh) - 4503599627371520.0;  // 2^52 + 1024
  const LogEntry t = kLogTab[j];
  const double r = fma(m, t.ic, -1.0);
  const double h = fma(e, kLn2Hi, t.hi);  // exact
  const double s = h + r;
  const double lo = ((h - s) + r) + fma(e, kLn2Lo, t.lo);
  const double r2 = r * r;
  double q = -1.0 / 8.0;
  q = fma(q, r, 1.0 / 7.0);
  q = fma(q, r, -1.0 / 6.0);
  q = fma(q, r, 1.0 / 5.0);
  q = fma(q, r, -1.0 / 4.0);
  q = fma(q, r, 1.0 / 3.0);
  q = fma(q, r, -1.0 / 2.0);
  return s + fma(r2, q, lo);
}

// cos and sin of 2 pi n 2^-53, n in [1, 2^53]: the nearest 64th of a turn from the table
// and the Taylor series of the rest (at most pi / 64)
__device__ __forceinline__ void sincos_u53(uint64_t n, double* sn, double* cs) {
  const int j = (int)((n + (1ull << 46)) >> 47);
  // the rest d = n - j 2^47 (|d| <= 2^46) as a double by its bits
  const long long d = (long long)(n - ((uint64_t)j << 47));
  const double x = (__longlong_as_double(0x4330000000000000ll + (d + (1ll << 47))) - 4644337115725824.0) * kTurn53;
  const double2 t = kTurn[j & 63];
  const double x2 = x * x;
  double a = fma(x2, 1.0 / 362880.0, -1.0 / 5040.0);
  a = fma(a, x2, 1.0 / 120.0);
  a = fma(a, x2, -1.0 / 6.0);
  const double sx = fma(a, x2 * x, x);
  double b = fma(x2, 1.0 / 40320.0, -1.0 / 720.0);
  b = fma(b, x2, 1.0 / 24.0);
  b = fma(b, x2, -1.0 / 2.0);
  const double cm = b * x2;  // cos x - 1
  *cs = t.x + fma(t.x, cm, -(t.y * sx));
  *sn = t.y + fma(t.y, cm, t.x * sx);
}

// The Box–Muller pair of normals with pair index `pair` of (seed, sample, stream).
__device__ __forceinline__ void normal_pair(uint64_t seed, int sample, int stream, int64_t pair, double* z0,
                                            double* z1) {
  U4 c;
  c.x = (uint32_t)(pair & 0xFFFFFFFFll);
  c.y = (uint32_t)sample;
  c.z = (uint32_t)stream;
  c.w = (uint32_t)(pair >> 32);
  U4 o = philox10(c, (uint32_t)(seed & 0xFFFFFFFFull), (uint32_t)(seed >> 32));
  double rad = sqrt(-2.0 * log_u53(uniform53(o.x, o.y)));
  double s, co;
  sincos_u53(uniform53(o.z, o.w), &s, &co);
  *z0 = rad * co;
  *z1 = rad * s;
}

__global__ void k_philox(const uint32_t* __restrict__ ctr, uint32_t k0, uint32_t k1, uint32_t* __restrict__ out,
                         int64_t n) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  U4 c = {ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]};
  U4 o = philox10(c, k0, k1);
  out[4 * i] = o.x;
  out[4 * i + 1] = o.y;
  out[4 * i + 2] = o.z;
  out[4 * i + 3] = o.w;
}

__global__ void k_normals(uint64_t seed, int sample, int stream, int64_t q0, int64_t n, double* __restrict__ out) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  int64_t q = q0 + i;
  double z0, z1;
  normal_pair(seed, sample, stream, q >> 1, &z0, &z1);
  out[i] = (q & 1) ? z1 : z0;
}

// normals 0..N-1 of samples s0 + (tile, lane) into [tiles][N][32], zero from sample
// s0 + ns on; lane = sample, a thread does the two normals of a pair
__global__ void k_normals_tiled(uint64_t seed, int s0, int ns, int stream, int N, double* __restrict__ out) {
  const int t = blockIdx.y, s = t * WM_LANES + threadIdx.x;
  const int64_t pair = (int64_t)blockIdx.x * blockDim.y + threadIdx.y;
  const int64_t i = 2 * pair;
  if (i >= N) return;
  double z0 = 0.0, z1 = 0.0;
  if (s < ns) normal_pair(seed, s0 + s, stream, pair, &z0, &z1);
  double* const o = out + ((size_t)t * N + i) * WM_LANES + threadIdx.x;
  o[0] = z0;
  if (i + 1 < N) o[WM_LANES] = z1;
}

// sqrt(w_q a_q) of every Gauss point, [E][nq^2] (the factor k_noise_local
// forms per sample, with the same operations)
template <int P>
__global__ void k_noise_weights(int E, int nu, int nv, const double* __restrict__ metric,
                                const double* __restrict__ gw, double* __restrict__ w) {
  constexpr int NQ = P + 1, NQ2 = NQ * NQ;
  const int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (q >= (int64_t)E * NQ2) return;
  const int j = (int)(q % NQ2);
  const int gv = j / NQ, gu = j % NQ;
  const double elw = 1.0 / ((double)nu * nv);
  w[q] = sqrt(gw[gu] * gw[gv] * elw * metric[4 * q]);
}

// One thread per (EPT elements, sample s0+sl): the (p+1)^2 local load
// contributions sum_q sqrt(w_q a_q) xi_q phi_k(x_q) of each element, xi the
// Philox normals of sample s0 + sl.  bl layout [E][nk][ns].  WT: the factors
// sqrt(w_q a_q) from the table of k_noise_weights instead of per sample.
// Bound by the float64 unit (595 G operations a second): about 62 a normal pair with the
// logarithm, sine and cosine above (90 with the general ones of 2 pi u and the
// conversions) and 13 for the contraction.  EPT = 2 where (p+1)^2 is odd and there are
// threads enough: two elements share their middle pair, nine pairs instead of ten.
// 256 samples of the 64 x 64 sphere, with the gather: 4.87 -> 3.23 ms.
template <int P, bool WT, int EPT>
__global__ void k_noise_local(int E, int nu, int nv, int ns, int s0, uint64_t seed,
                              const double* __restrict__ metric, const double* __restrict__ gw,
                              const double* __restrict__ bu, const double* __restrict__ bv, double* __restrict__ bl,
                              const double* __restrict__ wtab) {
  constexpr int NQ = P + 1, NK = (P + 1) * (P + 1), NQ2 = NQ * NQ, NP = EPT * NQ2;
  int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t e0 = tid / ns * EPT;
  if (e0 >= E) return;
  int sl = (int)(tid % ns);
  double xi[NP + 1];
  const int64_t q0 = e0 * NQ2;
  // points of the thread, in pairs of the sample's sequence; an odd first point is the
  // second of its pair
  if constexpr (NP % 2 == 0) {  // q0 is even
#pragma unroll
    for (int h = 0; h < NP / 2; ++h) normal_pair(seed, s0 + sl, 0, (q0 >> 1) + h, &xi[2 * h], &xi[2 * h + 1]);
  } else {
    int64_t pr0 = q0 >> 1, pr1 = (q0 + NP - 1) >> 1;
    for (int64_t pr = pr0; pr <= pr1; ++pr) {
      double z0, z1;
      normal_pair(seed, s0 + sl, 0, pr, &z0, &z1);
      int j0 = (int)(2 * pr - q0);
      if (j0 >= 0) xi[j0] = z0;
      if (j0 + 1 < NP) xi[j0 + 1] = z1;
    }
  }
#pragma unroll
  for (int h = 0; h < EPT; ++h) {
    const int64_t e = e0 + h;
    if (e >= E) break;
    const int eu = (int)(e % nu), ev = (int)((e / nu) % nv);
    double wq[NQ2];
    if constexpr (WT) {
#pragma unroll
      for (int j = 0; j < NQ2; ++j) wq[j] = wtab[e * NQ2 + j] * xi[h * NQ2 + j];
    } else {
      double elw = 1.0 / ((double)nu * nv);
#pragma unroll
      for (int j = 0; j < NQ2; ++j) {
        int gv = j / NQ, gu = j % NQ;
        wq[j] = sqrt(gw[gu] * gw[gv] * elw * metric[4 * (e * NQ2 + j)]) * xi[h * NQ2 + j];
      }
    }
    const double* BU = bu + (size_t)eu * (P + 1) * NQ;
    const double* BV = bv + (size_t)ev * (P + 1) * NQ;
#pragma unroll
    for (int kv = 0; kv <= P; ++kv)
#pragma unroll
      for (int ku = 0; ku <= P; ++ku) {
        double acc = 0.0;
#pragma unroll
        for (int gv = 0; gv < NQ; ++gv) {
          double t = 0.0;
#pragma unroll
          for (int gu = 0; gu < NQ; ++gu) t += BU[ku * NQ + gu] * wq[gv * NQ + gu];
          acc += BV[kv * NQ + gv] * t;
        }
        bl[((size_t)e * NK + kv * (P + 1) + ku) * ns + sl] = acc;
      }
  }
}

// One thread per (DOF i, row s0+sl): b[tile][i][lane] = sum over the element
// functions containing i of their local contributions, in element order.
__global__ void k_noise_gather(int N, int ns, int s0, const int32_t* __restrict__ ptr,
                               const int32_t* __restrict__ idx, const double* __restrict__ bl,
                               double* __restrict__ b) {
  int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (tid >= (int64_t)N * ns) return;
  int i = (int)(tid / ns);
  int sl = (int)(tid - (int64_t)i * ns);
  double acc = 0.0;
  for (int t = ptr[i]; t < ptr[i + 1]; ++t) acc += bl[(size_t)idx[t] * ns + sl];
  int s = s0 + sl;
  b[((size_t)(s / WM_LANES) * N + i) * WM_LANES + (s % WM_LANES)] = acc;
}

}  // namespace

int wm_k_philox(const uint32_t* ctr, uint64_t key, uint32_t* out, int64_t n, cudaStream_t s) {
  if (n <= 0) return WM_OK;
  WM_LAUNCH(WM_PC_NOISE, s, k_philox<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(ctr, (uint32_t)(key & 0xFFFFFFFFull),
                                                       (uint32_t)(key >> 32), out, n));
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

int wm_k_normals(uint64_t seed, int sample, int stream_id, int64_t q0, int64_t n, double* out, cudaStream_t s) {
  if (n <= 0) return WM_OK;
  WM_LAUNCH(WM_PC_NOISE, s, k_normals<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(seed, sample, stream_id, q0, n, out));
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

int wm_k_normals_tiled(uint64_t seed, int s0, int ns, int stream_id, int N, double* out, int tiles,
                       cudaStream_t s) {
  if (tiles <= 0 || N <= 0) return WM_OK;
  const unsigned pairs = (unsigned)((N + 1) / 2);
  WM_LAUNCH(WM_PC_NOISE, s, k_normals_tiled<<<dim3((pairs + 7) / 8, tiles), dim3(WM_LANES, 8), 0, s>>>(
                                seed, s0, ns, stream_id, N, out));
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

int wm_k_noise_tiled(const wm_hier* h, uint64_t seed, int sample_first, int row0, int ns, double* b_tiled,
                     double* bl, cudaStream_t s) {
  const wm_level& L = h->lv[0];
  const int64_t n1 = (int64_t)L.E * ns;
  // two elements per thread from 1,024 threads per SM on
  const bool two = n1 >= 2ll * 152 * 1024;
#define WM_NLE(PP, WT_, EPT_)                                                                                     \
  k_noise_local<PP, WT_, EPT_><<<(unsigned)(((L.E + EPT_ - 1) / EPT_ * (int64_t)ns + 127) / 128), 128, 0, s>>>(     \
      L.E, L.nu, L.nv, ns, sample_first, seed, L.d_metric.p, h->d_gw.p, L.d_bu.p, L.d_bv.p, bl, L.d_noise_w.p)
#define WM_NL(PP)                                            \
  if (L.d_noise_w.p) {                                       \
    if (PP % 2 == 0 && two)                                  \
      WM_NLE(PP, true, (PP % 2 == 0 ? 2 : 1));               \
    else                                                     \
      WM_NLE(PP, true, 1);                                   \
  } else                                                     \
    WM_NLE(PP, false, 1)
  wm_prof_begin(WM_PC_NOISE, s);
  switch (h->p) {
    case 1: WM_NL(1); break;
    case 2: WM_NL(2); break;
    case 3: WM_NL(3); break;
    case 4: WM_NL(4); break;
    default: return WM_ERR_UNSUPPORTED;
  }
#undef WM_NL
#undef WM_NLE
  wm_prof_end(WM_PC_NOISE, s);
  WM_CUDA(cudaGetLastError());
  int64_t n2 = (int64_t)L.N * ns;
  WM_LAUNCH(WM_PC_NOISE, s, k_noise_gather<<<(unsigned)((n2 + 255) / 256), 256, 0, s>>>(L.N, ns, row0, L.d_ng_ptr.p, L.d_ng_idx.p, bl,
                                                              b_tiled));
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

int wm_k_noise_weights(const wm_hier* h, wm_level& L, cudaStream_t s) {
  const int nq2 = h->nq * h->nq;
  WM_TRY(L.d_noise_w.alloc((size_t)L.E * nq2));
  const int64_t n = (int64_t)L.E * nq2;
  const unsigned g = (unsigned)((n + 255) / 256);
  switch (h->p) {
    case 1: WM_LAUNCH(WM_PC_ASSEMBLY, s, (k_noise_weights<1><<<g, 256, 0, s>>>(L.E, L.nu, L.nv, L.d_metric.p, h->d_gw.p, L.d_noise_w.p))); break;
    case 2: WM_LAUNCH(WM_PC_ASSEMBLY, s, (k_noise_weights<2><<<g, 256, 0, s>>>(L.E, L.nu, L.nv, L.d_metric.p, h->d_gw.p, L.d_noise_w.p))); break;
    case 3: WM_LAUNCH(WM_PC_ASSEMBLY, s, (k_noise_weights<3><<<g, 256, 0, s>>>(L.E, L.nu, L.nv, L.d_metric.p, h->d_gw.p, L.d_noise_w.p))); break;
    case 4: WM_LAUNCH(WM_PC_ASSEMBLY, s, (k_noise_weights<4><<<g, 256, 0, s>>>(L.E, L.nu, L.nv, L.d_metric.p, h->d_gw.p, L.d_noise_w.p))); break;
    default: return WM_ERR_UNSUPPORTED;
  }
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}

// ---------------------------------------------------------------- no-alloc entry
// White-noise loads for callers that cannot allocate device memory: a host
// framework whose caching allocator owns the device memory, or code that may
// not call cudaMalloc because it synchronises the device.  The element-local
// contributions go to a fixed file-scope device array instead of workspace
// memory; the loads are gathered straight into the caller's [n][N] output.
#include <mutex>

#define WM_NOALLOC_SCRATCH_DOUBLES (1 << 22) /* 32 MiB, resident on every device that loads the library */

static __device__ __align__(256) double g_noalloc_scratch[WM_NOALLOC_SCRATCH_DOUBLES];

namespace {

// b[s][i] = sum over the element functions containing i of their contributions
__global__ void k_noise_gather_rows(int N, int ns, const int32_t* __restrict__ ptr, const int32_t* __restrict__ idx,
                                    const double* __restrict__ bl, double* __restrict__ b) {
  int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (tid >= (int64_t)N * ns) return;
  int s = (int)(tid / N);
  int i = (int)(tid - (int64_t)s * N);
  double acc = 0.0;
  for (int t = ptr[i]; t < ptr[i + 1]; ++t) acc += bl[(size_t)idx[t] * ns + s];
  b[(size_t)s * N + i] = acc;
}

// Device address of the scratch array, looked up once per device with that
// device current (a host-side name of a __device__ array is not its address).
int noalloc_scratch(int dev, double** out) {
  static std::mutex mu;
  static double* addr[256] = {};
  if (dev < 0 || dev >= 256) return WM_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> g(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    WM_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    addr[dev] = static_cast<double*>(p);
  }
  *out = addr[dev];
  return WM_OK;
}

// device (or managed) memory the kernels may write
bool device_writable(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" int wm_noise_loads_noalloc(wm_hier_t h, uint64_t seed, int n_samples, double* b, void* stream) {
  if (!h || n_samples < 0 || (n_samples > 0 && !b)) return WM_ERR_INVALID_ARG;
  if (n_samples == 0) return WM_OK;
  int dev = 0;
  WM_CUDA(cudaGetDevice(&dev));
  if (dev != h->device) {
    wm_set_error("wm_noise_loads_noalloc: the hierarchy lives on device %d but device %d is current", h->device, dev);
    return WM_ERR_INVALID_ARG;
  }
  if (!device_writable(b)) {
    wm_set_error("wm_noise_loads_noalloc: b must be device memory");
    return WM_ERR_INVALID_ARG;
  }
  const wm_level& L = h->lv[0];
  int64_t need = (int64_t)L.E * L.nk * n_samples;
  if (need > (int64_t)WM_NOALLOC_SCRATCH_DOUBLES) {
    wm_set_error("wm_noise_loads_noalloc: elements x (p+1)^2 x samples = %lld exceeds the fixed scratch of %d "
                 "doubles; use fewer samples per call",
                 (long long)need, WM_NOALLOC_SCRATCH_DOUBLES);
    return WM_ERR_INVALID_ARG;
  }
  double* bl = nullptr;
  WM_TRY(noalloc_scratch(dev, &bl));
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int64_t n1 = (int64_t)L.E * n_samples;
  unsigned g1 = (unsigned)((n1 + 127) / 128);
  switch (h->p) {
    case 1: WM_LAUNCH(WM_PC_NOISE, s, (k_noise_local<1, false, 1><<<g1, 128, 0, s>>>(L.E, L.nu, L.nv, n_samples, 0, seed, L.d_metric.p, h->d_gw.p, L.d_bu.p, L.d_bv.p, bl, nullptr))); break;
    case 2: WM_LAUNCH(WM_PC_NOISE, s, (k_noise_local<2, false, 1><<<g1, 128, 0, s>>>(L.E, L.nu, L.nv, n_samples, 0, seed, L.d_metric.p, h->d_gw.p, L.d_bu.p, L.d_bv.p, bl, nullptr))); break;
    case 3: WM_LAUNCH(WM_PC_NOISE, s, (k_noise_local<3, false, 1><<<g1, 128, 0, s>>>(L.E, L.nu, L.nv, n_samples, 0, seed, L.d_metric.p, h->d_gw.p, L.d_bu.p, L.d_bv.p, bl, nullptr))); break;
    case 4: WM_LAUNCH(WM_PC_NOISE, s, (k_noise_local<4, false, 1><<<g1, 128, 0, s>>>(L.E, L.nu, L.nv, n_samples, 0, seed, L.d_metric.p, h->d_gw.p, L.d_bu.p, L.d_bv.p, bl, nullptr))); break;
    default: return WM_ERR_UNSUPPORTED;
  }
  WM_CUDA(cudaGetLastError());
  int64_t n2 = (int64_t)L.N * n_samples;
  WM_LAUNCH(WM_PC_NOISE, s, k_noise_gather_rows<<<(unsigned)((n2 + 255) / 256), 256, 0, s>>>(
                                L.N, n_samples, L.d_ng_ptr.p, L.d_ng_idx.p, bl, b));
  WM_CUDA(cudaGetLastError());
  return WM_OK;
}
