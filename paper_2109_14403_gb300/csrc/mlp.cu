// mlp.cu -- the warm-start network of include/dmn_mlp.h: tensor maps, the choice
// and launch of the tcgen05 GEMMs of the forward and backward passes (the bias
// gradients and the loss ride with them), and the memory-bound kernels around
// them (features, normalisation, AMSGrad with the weight packing).
#include <cudaTypedefs.h>
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <vector>

#include "../../include/dmn.h"
#include "../../include/dmn_mlp.h"
#include "dmn_internal.h"
#include "mlp_gemm.cuh"

using namespace dmn;
using namespace dmn::mlp;
typedef __nv_bfloat16 bf16;

namespace {

// ------------------------------------------------------------------ TMA maps
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

cudaError_t get_encode() {
  if (g_encode) return cudaSuccess;
  cudaDriverEntryPointQueryResult q;
  void *fn = nullptr;
  cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                   cudaEnableDefault, &q);
  if (e != cudaSuccess) return e;
  if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
  g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  return cudaSuccess;
}

// bf16 row-major [rows x cols] read in box_rows x 64-column boxes, 128 B swizzle
bool make_map(CUtensorMap *map, const void *ptr, uint64_t rows, uint64_t cols, uint32_t box_rows = 128) {
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols * 2};
  const cuuint32_t box[2] = {64, box_rows};
  const cuuint32_t es[2] = {1, 1};
  return g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides,
                  box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int g_gemm_configured_dev = -1;
int g_gemm_sms = 0;

cudaError_t gemm_setup() {
  cudaError_t e = get_encode();
  if (e != cudaSuccess) return e;
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if (g_gemm_configured_dev == dev) return cudaSuccess;
  const auto smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
  e = cudaFuncSetAttribute(gemm_bf16_tile<false, false, BN, STAGES>, smem, GEMM_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_bf16_tile<false, true, BN, STAGES>, smem, GEMM_SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_bf16_tile<false, false, WG_BN, WG_ST>, smem, tile_smem(WG_BN, WG_ST));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_bf16_tile<false, true, WG_BN, WG_ST>, smem, tile_smem(WG_BN, WG_ST));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_bf16_wgrad, smem, tile_smem(WG_BN, WG_ST));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_bf16_tn_wide<false>, smem, wide_smem(false));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_bf16_tn_wide<true>, smem, wide_smem(true));
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g_gemm_sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) g_gemm_configured_dev = dev;
  return e;
}
bool gemm_args_ok(const void *A, const void *B, int M, int N, int K) {
  return M % BM == 0 && N % BN == 0 && K % BK == 0 && M > 0 && N > 0 && K > 0 && M / BM <= 65535 &&
         N / BN <= 65535 &&  // grid limits
         !((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15);
}

// a product whose tiles are all resident at once is short: its launch overlaps
// the one before it (pdl.cuh)
bool overlaps(int M, int N) { return (M / BM) * (N / BN) <= 2 * g_gemm_sms; }

// ... with at most one 128 x 128 tile an SM: tiles of 64 columns, up to two CTAs
// an SM.  Such a product lasts as long as one tile, and half of the columns are
// half of its epilogue (a step of 4,096 pairs 180 -> 172 us, of 64 142 -> 126;
// inference of 64 to 4,096 rows 47..57 -> 42..52).  The hidden layers and their
// input gradients; the same chain of MMAs for every output.
bool narrow(int M, int N, const EpiArgs &ep) {
  return (M / BM) * (N / BN) <= g_gemm_sms && (ep.mode == EPI_BIAS_SILU || ep.mode == EPI_DSILU);
}

// C = A . B^T with the fused epilogue ep; A [M x K], B [N x K] bf16; rows of A
// from a_rows on read as zero.  N a multiple of 256 and enough 128 x 256 tiles: the
// persistent wide form (one CTA per SM), else (and with z_out or the loss, the
// training step's) the tile form, whose 128 x 128 tiles spread a product over
// twice the SMs (4,096 rows, a hidden layer: 18 -> 12 us).  Enough is a tile for
// every SM, or for plain FP32 output for more than half of them: with fewer the tile
// form has an SM for every half tile (64 tiles, K = 512 to 4,096: 0.85 to 0.9 of the
// wide form's time; 128 tiles, K = 4,096: 1.10).
cudaError_t gemm(cudaStream_t s, const void *A, const void *B, int M, int N, int K, EpiArgs ep, int64_t a_rows) {
  if (!gemm_args_ok(A, B, M, N, K)) return cudaErrorInvalidValue;
  cudaError_t e = gemm_setup();
  if (e != cudaSuccess) return e;
  CUtensorMap ma, mb;
  if (!make_map(&ma, A, a_rows, K)) return cudaErrorInvalidValue;
  const bool plain = ep.mode == EPI_F32;
  const int64_t tiles = int64_t(M / BM) * (N / WBN);
  if (N % WBN == 0 && tiles * (plain ? 2 : 1) >= g_gemm_sms + (plain ? 1 : 0) && !ep.z_out && ep.mode != EPI_LOSS) {
    CUtensorMap mh = ma;  // unused unless the activation leaves by TMA
    if (!make_map(&mb, B, N, K, WBN) || (ep.mode == EPI_BIAS_SILU && !make_map(&mh, ep.h_out, M, N, 32)))
      return cudaErrorInvalidValue;
    const int ctas = int(tiles < g_gemm_sms ? tiles : g_gemm_sms);
    const bool lng = plain || K >= 2048;
    (lng ? gemm_bf16_tn_wide<true> : gemm_bf16_tn_wide<false>)<<<ctas, wide_threads(lng), wide_smem(lng), s>>>(
        ma, mb, mh, M, N, K, ep);
    return cudaGetLastError();
  }
  if (narrow(M, N, ep)) {
    if (!make_map(&mb, B, N, K, WG_BN)) return cudaErrorInvalidValue;
    return launch_chained(true, gemm_bf16_tile<false, false, WG_BN, WG_ST>, dim3(N / WG_BN, M / BM), dim3(128),
                          tile_smem(WG_BN, WG_ST), s, ma, mb, K, ep);
  }
  if (!make_map(&mb, B, N, K)) return cudaErrorInvalidValue;
  return launch_chained(overlaps(M, N), gemm_bf16_tile<false, false, BN, STAGES>, dim3(N / BN, M / BM), dim3(128),
                        GEMM_SMEM, s, ma, mb, K, ep);
}
// input gradient: C [M x N] = A . B, A [M x K], B [K x N] as stored
cudaError_t gemm_dgrad(cudaStream_t s, const void *A, const void *B, int M, int N, int K, EpiArgs ep) {
  if (!gemm_args_ok(A, B, M, N, K)) return cudaErrorInvalidValue;
  cudaError_t e = gemm_setup();
  if (e != cudaSuccess) return e;
  CUtensorMap ma, mb;
  if (!make_map(&ma, A, M, K) || !make_map(&mb, B, K, N, BK)) return cudaErrorInvalidValue;
  if (narrow(M, N, ep))
    return launch_chained(true, gemm_bf16_tile<false, true, WG_BN, WG_ST>, dim3(N / WG_BN, M / BM), dim3(128),
                          tile_smem(WG_BN, WG_ST), s, ma, mb, K, ep);
  return launch_chained(overlaps(M, N), gemm_bf16_tile<false, true, BN, STAGES>, dim3(N / BN, M / BM), dim3(128),
                        GEMM_SMEM, s, ma, mb, K, ep);
}
// adds layer l's weight gradient to a launch: C [M x N] (fp32) = A^T . B, A [K x
// M], B [K x N] (rows from b_rows on read as zero)
bool wgrad_add(WgradArgs &W, const void *A, const void *B, int M, int N, int K, float *C, int64_t b_rows) {
  const int l = W.layers;
  if (l >= kMaxLayers || !gemm_args_ok(A, B, M, N, K) || !make_map(&W.a[l], A, K, M, BK) ||
      !make_map(&W.b[l], B, b_rows, N, BK))
    return false;
  W.nx[l] = N / WG_BN;
  W.ldc[l] = N;
  W.out[l] = C;
  W.blk0[l + 1] = W.blk0[l] + W.nx[l] * (M / BM);
  W.layers = l + 1;
  return true;
}

int64_t rup(int64_t x, int64_t m) { return (x + m - 1) / m * m; }
unsigned blocks_for(int64_t n, int t = 256) {
  int64_t b = (n + t - 1) / t;
  return unsigned(b < 1 ? 1 : (b > 65535 * 8 ? 65535 * 8 : b));
}

// ------------------------------------------------------------------ kernels
// A double rounded to the nearest float (ties to even) by integer
// operations: the FP64 pipe of this GPU runs at 1/64 of the FP32 rate, and
// the network input converts 768 words per row.  Magnitudes outside the
// normal float range (and NaN) take the FP64 conversion; zero and double
// subnormals give a signed zero.
// (the conversion as a call: otherwise every lane issues it under a false
// predicate, which kept the FP64 pipe 55 % busy)
__device__ __noinline__ float f32_rn_call(double d) { return __double2float_rn(d); }
__device__ __forceinline__ float f32_rn(double d) {
  const unsigned hi = unsigned(__double2hiint(d)), lo = unsigned(__double2loint(d));
  const unsigned t = hi & 0x7fffffffu, sign = hi & 0x80000000u;
  if (t - (897u << 20) >= (254u << 20)) return t < (1u << 20) ? __uint_as_float(sign) : f32_rn_call(d);
  unsigned r = __funnelshift_l(lo, t - (896u << 20), 3);        // exponent and 23 bits, truncated
  r += (lo & 0x1fffffffu) + (r & 1u) > 0x10000000u ? 1u : 0u;  // to nearest, ties to even; a carry moves into the exponent
  return __uint_as_float(sign | r);
}
// The same result without a call and by branches, for the rows read word by word:
// bound by their half-sector loads, they lose more to the call's registers than to
// the FP64 pipe (65,536 rows at K = 8, states 8 bytes off: 208 us, 225 with the call)
__device__ __forceinline__ float f32_rn_inline(double d) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(d));
  const unsigned E = unsigned(b >> 52) & 0x7ffu, sign = unsigned(b >> 32) & 0x80000000u;
  if (E == 0u) return __uint_as_float(sign);
  if (E < 897u || E > 1150u) return __double2float_rn(d);
  const unsigned long long mant = b & ((1ull << 52) - 1);
  unsigned r = sign | ((E - 896u) << 23) | unsigned(mant >> 29);
  const unsigned rem = unsigned(mant & ((1ull << 29) - 1)), half = 1u << 28;
  if (rem > half || (rem == half && (r & 1u))) r += 1u;  // a carry moves into the exponent
  return __uint_as_float(r);
}

// feature c of a row: deps (6), theta^{n+1}, theta^{n+1} - theta^n,
// a^n - a^{n-1} (n3) as the difference of the two words rounded to float;
// a = the state block at t^n, ap = at t^{n-1} or NULL (its columns 0)
constexpr int kExtraFeatures = 0;
template <float (*RN)(double) = f32_rn>
__device__ __forceinline__ float feature(int c, int n3, const double *dep, double th, const double *a,
                                         const double *ap) {
  (void)n3;
  if (c < 6) return RN(dep[c]);
  if (c == 6) return RN(th);
  if (c == 7) return float(th - a[6]);
  return ap ? RN(a[c]) - RN(ap[c]) : 0.0f;  // a^n - a^{n-1}: state words 8..
}

__global__ void k_features(int64_t n, int n3, int sw, const double *deps, const double *theta,
                           const double *sin, const double *sprev, float *feat) {
  const int nin = 8 + n3 + kExtraFeatures;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n * nin;
       i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = i / nin;
    const int c = int(i - r * nin);
    feat[i] = feature(c, n3, deps + r * 6, theta[r], sin + r * sw, sprev ? sprev + r * sw : nullptr);
  }
}

// features of k_features, normalised and rounded to bf16 in one pass: one
// warp per row, each lane two adjacent columns per step (one bf16x2 store;
// ld = kin is a multiple of 128, so the pairs stay 4-byte aligned).  Bound by the
// two states' jumps it reads (12 KB a row at K = 8).  Three instances, chosen by
// the call: 16-byte loads of a lane's pair of jumps, two steps in flight (states
// 16-byte aligned, an even number of words; 65,536 rows 166 us, one step 173, four
// 178, seven 193); word by word (aligned 180, 8 bytes off 208); no previous state
// (65,536 rows at K = 8 a call 76 us, 86 inside the instance for two states, whose
// registers keep half of the warps out).
enum { ROWS_FIRST, ROWS_WORDS, ROWS_VEC };  // no previous state; word by word; 16-byte loads
template <int MODE>
__global__ void __launch_bounds__(256)
    k_features_norm(int64_t n, int n3, int sw, int ld, const double *deps, const double *theta, const double *sin,
                    const double *sprev, const float *mean, const float *inv, bf16 *x) {
  const int nin = 8 + n3 + kExtraFeatures;
  const int lane = threadIdx.x & 31;
  const int64_t nwarp = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5; r < n; r += nwarp) {
    const double *a = sin + r * sw;
    const double *ap = MODE == ROWS_FIRST ? nullptr : sprev + r * sw;
    __nv_bfloat162 *xr = reinterpret_cast<__nv_bfloat162 *>(x + r * ld);
    auto put = [&](int c0, float f0, float f1) {  // features of columns c0, c0 + 1
      float v0 = 0.0f, v1 = 0.0f;
      if (c0 < nin) v0 = (f0 - __ldg(mean + c0)) * __ldg(inv + c0);
      if (c0 + 1 < nin) v1 = (f1 - __ldg(mean + c0 + 1)) * __ldg(inv + c0 + 1);
      xr[c0 >> 1] = __floats2bfloat162_rn(v0, v1);
    };
    if constexpr (MODE == ROWS_VEC) {
      constexpr int U = 2;
      for (int c0 = 2 * lane; c0 < ld; c0 += 64 * U) {
        double2 q[U], p[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int c = c0 + 64 * u;
          const bool in = c >= 8 && c + 1 < sw && c < nin;  // c + 1 == nin: the word after the jumps
          q[u] = in ? *reinterpret_cast<const double2 *>(a + c) : make_double2(0.0, 0.0);
          p[u] = in ? *reinterpret_cast<const double2 *>(ap + c) : make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int c = c0 + 64 * u;
          if (c >= ld) break;
          if (c < 8 || c + 1 >= sw) {  // the load's features; a state that ends with the jumps
            float f[2];
#pragma unroll
            for (int w = 0; w < 2; ++w)
              f[w] = c + w < nin ? feature(c + w, n3, deps + r * 6, theta[r], a, ap) : 0.0f;
            put(c, f[0], f[1]);
          } else {
            put(c, f32_rn(q[u].x) - f32_rn(p[u].x), f32_rn(q[u].y) - f32_rn(p[u].y));
          }
        }
      }
    } else if constexpr (MODE == ROWS_WORDS) {
      for (int c0 = 2 * lane; c0 < ld; c0 += 64) {
        float v[2] = {0.0f, 0.0f};
#pragma unroll
        for (int u = 0; u < 2; ++u)
          if (c0 + u < nin)
            v[u] = (feature<f32_rn_inline>(c0 + u, n3, deps + r * 6, theta[r], a, ap) - mean[c0 + u]) * inv[c0 + u];
        xr[c0 >> 1] = __floats2bfloat162_rn(v[0], v[1]);
      }
    } else {
      for (int c0 = 2 * lane; c0 < ld; c0 += 64) {
        float f[2];
#pragma unroll
        for (int u = 0; u < 2; ++u)
          f[u] = c0 + u < nin ? feature(c0 + u, n3, deps + r * 6, theta[r], a, ap) : 0.0f;
        put(c0, f[0], f[1]);
      }
    }
  }
}

__global__ void k_targets(int64_t n, int n3, int sw, const double *sin, const double *sout,
                          float *tgt) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n * n3;
       i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = i / n3;
    const int j = int(i - r * n3);
    tgt[i] = float(sout[r * sw + 8 + j] - sin[r * sw + 8 + j]);
  }
}

// partial column sums (sum, sum of squares) over a slab of rows; 32 columns
// per block in x, 8 row lanes in y; FP64 accumulation
__global__ void k_colstats(int64_t n, int cols, const float *x, double *acc) {
  __shared__ double s1[8][32], s2[8][32];
  const int c = blockIdx.x * 32 + threadIdx.x;
  double a = 0.0, b = 0.0;
  if (c < cols) {
    for (int64_t r = blockIdx.y * 8 + threadIdx.y; r < n; r += int64_t(gridDim.y) * 8) {
      const double v = x[r * cols + c];
      a += v;
      b += v * v;
    }
  }
  s1[threadIdx.y][threadIdx.x] = a;
  s2[threadIdx.y][threadIdx.x] = b;
  __syncthreads();
  if (threadIdx.y == 0 && c < cols) {
    for (int k = 1; k < 8; ++k) {
      a += s1[k][threadIdx.x];
      b += s2[k][threadIdx.x];
    }
    atomicAdd(&acc[2 * c], a);
    atomicAdd(&acc[2 * c + 1], b);
  }
}

__global__ void k_colstats_final(int64_t n, int cols, const double *acc, float *mean, float *inv,
                                 float *stdv) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  const double mu = acc[2 * c] / double(n);
  double var = acc[2 * c + 1] / double(n) - mu * mu;
  if (var < 0.0) var = 0.0;
  const double sd = sqrt(var);
  // spread below 1e-9 of the column's scale: treat the column as constant
  const bool flat = !(sd > 1e-9 * fabs(mu)) || sd == 0.0;
  mean[c] = float(mu);
  if (inv) inv[c] = flat ? 0.0f : float(1.0 / sd);
  if (stdv) stdv[c] = flat ? 0.0f : float(sd);
}

__global__ void k_norm_x(int64_t n, int nin, int ld, const float *feat, const float *mean,
                         const float *inv, bf16 *x) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n * ld;
       i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = i / ld;
    const int c = int(i - r * ld);
    x[i] = __float2bfloat16(c < nin ? (feat[r * nin + c] - mean[c]) * inv[c] : 0.0f);
  }
}

__global__ void k_norm_t(int64_t n, int nout, int ld, const float *tgt, const float *mean,
                         const float *inv, float *t) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n * ld;
       i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t r = i / ld;
    const int c = int(i - r * ld);
    t[i] = c < nout ? (tgt[r * nout + c] - mean[c]) * inv[c] : 0.0f;
  }
}

// AMSGrad with bias correction (Reddi, Kale, Kumar 2018; the maximum of the
// second-moment estimates replaces it in the step size)
struct AmsArgs {
  float lr, b1, b2, eps, bc1, bc2;
};
__device__ __forceinline__ void amsgrad_elem(float &w, float gi, float &m, float &v, float &vmax, const AmsArgs &a) {
  const float mi = a.b1 * m + (1.0f - a.b1) * gi;
  const float vi = a.b2 * v + (1.0f - a.b2) * gi * gi;
  const float vm = fmaxf(vmax, vi);
  m = mi;
  v = vi;
  vmax = vm;
  w -= a.lr * (mi / a.bc1) / (sqrtf(vm / a.bc2) + a.eps);
}
__global__ void k_amsgrad(int64_t count, float *w, const float *g, float *m, float *v, float *vmax, AmsArgs a) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < count;
       i += int64_t(gridDim.x) * blockDim.x)
    amsgrad_elem(w[i], g[i], m[i], v[i], vmax[i], a);
}
// The same for the network's parameters, four a thread, with the bf16 weights
// of the next pass (every layer's count and offset are multiples of four)
struct PackArgs {
  int layers;
  int64_t ow[kMaxLayers], ob[kMaxLayers];  // weights of layer l: [ow, ob)
  bf16 *w[kMaxLayers];
};
__global__ void __launch_bounds__(256)
    k_amsgrad_pack(int64_t count4, float4 *w, const float4 *g, float4 *m, float4 *v, float4 *vmax, AmsArgs a,
                   const PackArgs P) {
  const int64_t i = blockIdx.x * int64_t(256) + threadIdx.x;
  chain_begin();
  if (i >= count4) return;
  const float4 gi = g[i];
  float4 wi = w[i], mi = m[i], vi = v[i], xi = vmax[i];
  amsgrad_elem(wi.x, gi.x, mi.x, vi.x, xi.x, a);
  amsgrad_elem(wi.y, gi.y, mi.y, vi.y, xi.y, a);
  amsgrad_elem(wi.z, gi.z, mi.z, vi.z, xi.z, a);
  amsgrad_elem(wi.w, gi.w, mi.w, vi.w, xi.w, a);
  w[i] = wi;
  m[i] = mi;
  v[i] = vi;
  vmax[i] = xi;
  int l = 0;
  while (l + 1 < P.layers && 4 * i >= P.ow[l + 1]) ++l;
  if (4 * i < P.ob[l]) {
    __nv_bfloat162 *o = reinterpret_cast<__nv_bfloat162 *>(P.w[l] + (4 * i - P.ow[l]));
    o[0] = __floats2bfloat162_rn(wi.x, wi.y);
    o[1] = __floats2bfloat162_rn(wi.z, wi.w);
  }
}

// optimiser constants of the training step (AMSGrad defaults)
constexpr float kBeta1 = 0.9f, kBeta2 = 0.999f, kEps = 1e-8f;

// One AMSGrad step at iteration step >= 1.  The bias corrections 1 - b^t are
// formed in FP64 from the FP32 betas and rounded once: in FP32, 1 - powf(b2, t)
// for b2 near 1 would lose about 5 of its 24 bits to cancellation.
AmsArgs ams_args(float lr, float b1, float b2, float eps, int64_t step) {
  return {lr, b1, b2, eps, float(1.0 - pow(double(b1), double(step))), float(1.0 - pow(double(b2), double(step)))};
}

// bf16 weights from the fp32 master copy
__global__ void k_pack(int64_t n, const float *w32, bf16 *w) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    w[i] = __float2bfloat16(w32[i]);
}

uint64_t splitmix(uint64_t &s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

}  // namespace

struct dmn_mlp_s {
  int K, n3, nin, kin, H, nh, nout_pad, L;
  int64_t bmax;
  std::vector<int> din, dout;
  std::vector<int64_t> ow, ob;
  int64_t nparam;
  float *params, *grads, *m, *v, *vmax;
  std::vector<bf16 *> w;
  float *fmean, *finv, *tmean, *tstd, *tinv;
  bf16 *x;
  std::vector<bf16 *> z, h, dz;
  float *t, *lpart;
  double *acc;
  int *err;
  int step;
};

namespace {
dmn_status fail(dmn_status s, const char *fmt, ...) {
  char msg[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(msg, sizeof(msg), fmt, ap);
  va_end(ap);
  set_error_message(msg);
  return s;
}
dmn_status cuda_fail(cudaError_t e, const char *what) {
  return fail(e == cudaErrorMemoryAllocation ? DMN_ERR_OOM : DMN_ERR_CUDA, "%s: %s", what,
              cudaGetErrorString(e));
}
void free_mlp(dmn_mlp p) {
  if (!p) return;
  void *bufs[] = {p->params, p->grads, p->m, p->v, p->vmax, p->fmean, p->finv, p->tmean, p->tstd,
                  p->tinv, p->x, p->t, p->lpart, p->acc, p->err};
  for (void *b : bufs) cudaFree(b);
  for (auto *b : p->w) cudaFree(b);
  for (auto *b : p->z) cudaFree(b);
  for (auto *b : p->h) cudaFree(b);
  for (auto *b : p->dz) cudaFree(b);
  delete p;
}
template <typename T>
cudaError_t dalloc(T **p, size_t count) {
  return cudaMalloc(reinterpret_cast<void **>(p), sizeof(T) * (count ? count : 1));
}
cudaError_t pack_all(dmn_mlp p, cudaStream_t s) {
  for (int l = 0; l < p->L; ++l) {
    const int64_t n = int64_t(p->dout[l]) * p->din[l];
    k_pack<<<blocks_for(n), 256, 0, s>>>(n, p->params + p->ow[l], p->w[l]);
  }
  return cudaGetLastError();
}
// the batch's rows, copied into the workspace only if TMA cannot read them
// where they are (16-byte alignment); rows from n on are read as zero
cudaError_t stage_x(dmn_mlp p, cudaStream_t s, int64_t n, const void *x, const bf16 **in) {
  *in = static_cast<const bf16 *>(x);
  if (!(reinterpret_cast<uintptr_t>(x) & 15)) return cudaSuccess;
  *in = p->x;
  return cudaMemcpyAsync(p->x, x, sizeof(bf16) * p->kin * n, cudaMemcpyDeviceToDevice, s);
}
// forward pass; t: training, the loss against these targets into dz of the last
// layer (and pre-activations kept), else the prediction into da
cudaError_t forward(dmn_mlp p, cudaStream_t s, int64_t n, int64_t npad, const float *t, float *da,
                    const bf16 *x_in) {
  cudaError_t e = cudaSuccess;
  const bf16 *in = x_in;
  int64_t rows = n;
  for (int l = 0; l < p->L; ++l) {
    EpiArgs ep;
    memset(&ep, 0, sizeof(ep));
    ep.err = p->err;
    ep.bias = p->params + p->ob[l];
    ep.ldc = p->dout[l];
    if (l < p->L - 1) {
      ep.mode = EPI_BIAS_SILU;
      ep.z_out = t ? p->z[l] : nullptr;  // pre-activations only for the backward pass
      ep.h_out = p->h[l];
    } else {
      ep.m_valid = int(n);
      ep.n_valid = p->n3;
      if (t) {
        ep.mode = EPI_LOSS;
        ep.target = t;
        ep.gscale = 1.0f / (float(n) * float(p->n3));
        ep.loss_part = p->lpart;
        ep.h_out = p->dz[l];
      } else {
        ep.mode = EPI_BIAS_F32;
        ep.f_out = da;
        ep.scale = p->tstd;
        ep.shift = p->tmean;
        ep.ld_f = p->n3;
      }
    }
    e = gemm(s, in, p->w[l], int(npad), p->dout[l], p->din[l], ep, rows);
    if (e != cudaSuccess) return e;
    if (l < p->L - 1) in = p->h[l];
    rows = npad;
  }
  return e;
}
}  // namespace

extern "C" dmn_status dmn_mlp_create(dmn_mlp *out, int32_t K, int32_t hidden, int32_t n_hidden,
                                     int64_t max_batch, uint64_t seed) {
  set_error_message("");
  if (!out) return fail(DMN_ERR_ARG, "dmn_mlp_create: out is NULL");
  *out = nullptr;
  if (K < 1 || K > 9) return fail(DMN_ERR_ARG, "dmn_mlp_create: K=%d outside 1..9", K);
  if (hidden < 128 || hidden % 128 || hidden > 4096)
    return fail(DMN_ERR_ARG, "dmn_mlp_create: hidden=%d not a multiple of 128 in 128..4096", hidden);
  if (n_hidden < 1 || n_hidden > 8) return fail(DMN_ERR_ARG, "dmn_mlp_create: n_hidden=%d", n_hidden);
  if (max_batch < 1 || max_batch > (1 << 22))
    return fail(DMN_ERR_ARG, "dmn_mlp_create: max_batch=%lld", (long long)max_batch);
  cudaError_t e = get_encode();
  if (e != cudaSuccess) return cuda_fail(e, "cuTensorMapEncodeTiled entry point");
  dmn_mlp p = new dmn_mlp_s();
  p->K = K;
  p->n3 = 3 * ((1 << K) - 1);
  p->nin = 8 + p->n3 + kExtraFeatures;
  p->kin = int(rup(p->nin, 128));
  p->H = hidden;
  p->nh = n_hidden;
  p->nout_pad = int(rup(p->n3, 128));
  p->L = n_hidden + 1;
  p->bmax = rup(max_batch, 128);
  p->nparam = 0;
  for (int l = 0; l < p->L; ++l) {
    p->din.push_back(l == 0 ? p->kin : hidden);
    p->dout.push_back(l == p->L - 1 ? p->nout_pad : hidden);
    p->ow.push_back(p->nparam);
    p->nparam += int64_t(p->din[l]) * p->dout[l];
    p->ob.push_back(p->nparam);
    p->nparam += p->dout[l];
  }
  p->step = 0;
  p->params = p->grads = p->m = p->v = p->vmax = nullptr;
  p->fmean = p->finv = p->tmean = p->tstd = p->tinv = nullptr;
  p->x = nullptr;
  p->t = p->lpart = nullptr;
  p->acc = nullptr;
  p->err = nullptr;
  p->w.assign(p->L, nullptr);
  p->z.assign(p->nh, nullptr);
  p->h.assign(p->nh, nullptr);
  p->dz.assign(p->L, nullptr);
  const int64_t B = p->bmax;
  bool ok = dalloc(&p->params, p->nparam) == cudaSuccess && dalloc(&p->grads, p->nparam) == cudaSuccess &&
            dalloc(&p->m, p->nparam) == cudaSuccess && dalloc(&p->v, p->nparam) == cudaSuccess &&
            dalloc(&p->vmax, p->nparam) == cudaSuccess && dalloc(&p->fmean, p->kin) == cudaSuccess &&
            dalloc(&p->finv, p->kin) == cudaSuccess && dalloc(&p->tmean, p->nout_pad) == cudaSuccess &&
            dalloc(&p->tstd, p->nout_pad) == cudaSuccess && dalloc(&p->tinv, p->nout_pad) == cudaSuccess &&
            dalloc(&p->x, B * p->kin) == cudaSuccess && dalloc(&p->t, B * p->nout_pad) == cudaSuccess &&
            dalloc(&p->lpart, (B / BM) * (p->nout_pad / BN) * 4) == cudaSuccess &&
            dalloc(&p->acc, 2 * int64_t(p->kin > p->nout_pad ? p->kin : p->nout_pad)) == cudaSuccess &&
            dalloc(&p->err, 1) == cudaSuccess;
  for (int l = 0; ok && l < p->L; ++l)
    ok = dalloc(&p->w[l], int64_t(p->din[l]) * p->dout[l]) == cudaSuccess &&
         dalloc(&p->dz[l], B * p->dout[l]) == cudaSuccess;
  for (int l = 0; ok && l < p->nh; ++l)
    ok = dalloc(&p->z[l], B * hidden) == cudaSuccess && dalloc(&p->h[l], B * hidden) == cudaSuccess;
  if (!ok) {
    free_mlp(p);
    return fail(DMN_ERR_OOM, "dmn_mlp_create: device allocation failed");
  }
  // seeded initialisation on the host
  std::vector<float> hp(p->nparam, 0.0f);
  uint64_t st = seed * 0x2545F4914F6CDD1Dull + 0x1234567ull;
  for (int l = 0; l < p->L; ++l) {
    const int fan_in = l == 0 ? p->nin : hidden;
    const int rows = l == p->L - 1 ? p->n3 : hidden;
    const float a = 1.0f / sqrtf(float(fan_in));
    for (int r = 0; r < rows; ++r)
      for (int c = 0; c < fan_in; ++c) {
        const double u = double(splitmix(st) >> 11) * (1.0 / 9007199254740992.0);
        hp[p->ow[l] + int64_t(r) * p->din[l] + c] = float((2.0 * u - 1.0) * a);
      }
  }
  const int cmax = p->kin > p->nout_pad ? p->kin : p->nout_pad;
  std::vector<float> ones(cmax, 1.0f);
  if ((e = cudaMemcpy(p->params, hp.data(), sizeof(float) * p->nparam, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemset(p->m, 0, sizeof(float) * p->nparam)) != cudaSuccess ||
      (e = cudaMemset(p->v, 0, sizeof(float) * p->nparam)) != cudaSuccess ||
      (e = cudaMemset(p->vmax, 0, sizeof(float) * p->nparam)) != cudaSuccess ||
      (e = cudaMemset(p->grads, 0, sizeof(float) * p->nparam)) != cudaSuccess ||
      (e = cudaMemset(p->fmean, 0, sizeof(float) * p->kin)) != cudaSuccess ||
      (e = cudaMemcpy(p->finv, ones.data(), sizeof(float) * p->kin, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemset(p->tmean, 0, sizeof(float) * p->nout_pad)) != cudaSuccess ||
      (e = cudaMemcpy(p->tstd, ones.data(), sizeof(float) * p->nout_pad, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemcpy(p->tinv, ones.data(), sizeof(float) * p->nout_pad, cudaMemcpyHostToDevice)) != cudaSuccess ||
      (e = cudaMemset(p->err, 0, sizeof(int))) != cudaSuccess || (e = pack_all(p, 0)) != cudaSuccess ||
      (e = cudaDeviceSynchronize()) != cudaSuccess) {
    free_mlp(p);
    return cuda_fail(e, "dmn_mlp_create");
  }
  *out = p;
  return DMN_OK;
}

extern "C" dmn_status dmn_mlp_destroy(dmn_mlp m) {
  set_error_message("");
  if (!m) return fail(DMN_ERR_ARG, "dmn_mlp_destroy: NULL");
  free_mlp(m);
  return DMN_OK;
}

extern "C" dmn_status dmn_mlp_dims(dmn_mlp m, int32_t *n_in, int32_t *n_in_pad, int32_t *n_out,
                                   int32_t *n_out_pad) {
  if (!m) return fail(DMN_ERR_ARG, "dmn_mlp_dims: NULL");
  if (n_in) *n_in = m->nin;
  if (n_in_pad) *n_in_pad = m->kin;
  if (n_out) *n_out = m->n3;
  if (n_out_pad) *n_out_pad = m->nout_pad;
  return DMN_OK;
}

extern "C" dmn_status dmn_mlp_features(dmn_mlp m, dmn_stream stream, int64_t n, const double *d_deps,
                                       const double *d_theta, const double *d_state_in,
                                       const double *d_state_prev, int64_t state_words,
                                       float *d_feat) {
  set_error_message("");
  if (!m || n < 0 || !d_deps || !d_theta || !d_state_in || !d_feat || state_words < 8 + m->n3)
    return fail(DMN_ERR_ARG, "dmn_mlp_features: invalid argument");
  if (n == 0) return DMN_OK;
  k_features<<<blocks_for(n * m->nin), 256, 0, (cudaStream_t)stream>>>(
      n, m->n3, int(state_words), d_deps, d_theta, d_state_in, d_state_prev, d_feat);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_features");
}

extern "C" dmn_status dmn_mlp_input(dmn_mlp m, dmn_stream stream, int64_t n, const double *d_deps,
                                    const double *d_theta, const double *d_state_in,
                                    const double *d_state_prev, int64_t state_words,
                                    void *d_x_bf16) {
  set_error_message("");
  if (!m || n < 0 || !d_deps || !d_theta || !d_state_in || !d_x_bf16 || state_words < 8 + m->n3)
    return fail(DMN_ERR_ARG, "dmn_mlp_input: invalid argument");
  if (n == 0) return DMN_OK;
  const bool vec = ((reinterpret_cast<uintptr_t>(d_state_in) | reinterpret_cast<uintptr_t>(d_state_prev)) & 15) == 0 &&
                   (state_words & 1) == 0;
  const auto f = !d_state_prev ? k_features_norm<ROWS_FIRST>
                               : (vec ? k_features_norm<ROWS_VEC> : k_features_norm<ROWS_WORDS>);
  f<<<blocks_for(n * 32), 256, 0, (cudaStream_t)stream>>>(
      n, m->n3, int(state_words), m->kin, d_deps, d_theta, d_state_in, d_state_prev, m->fmean,
      m->finv, static_cast<bf16 *>(d_x_bf16));
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_input");
}

extern "C" dmn_status dmn_mlp_targets(dmn_mlp m, dmn_stream stream, int64_t n,
                                      const double *d_state_in, const double *d_state_out,
                                      int64_t state_words, float *d_tgt) {
  set_error_message("");
  if (!m || n < 0 || !d_state_in || !d_state_out || !d_tgt || state_words < 8 + m->n3)
    return fail(DMN_ERR_ARG, "dmn_mlp_targets: invalid argument");
  if (n == 0) return DMN_OK;
  k_targets<<<blocks_for(n * m->n3), 256, 0, (cudaStream_t)stream>>>(
      n, m->n3, int(state_words), d_state_in, d_state_out, d_tgt);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_targets");
}

extern "C" dmn_status dmn_mlp_fit_normalization(dmn_mlp m, dmn_stream stream, int64_t n,
                                                const float *d_feat, const float *d_tgt) {
  set_error_message("");
  if (!m || n < 2 || !d_feat || !d_tgt) return fail(DMN_ERR_ARG, "dmn_mlp_fit_normalization: invalid argument");
  cudaStream_t s = (cudaStream_t)stream;
  const int cmax = m->kin > m->nout_pad ? m->kin : m->nout_pad;
  cudaError_t e = cudaMemsetAsync(m->acc, 0, sizeof(double) * 2 * cmax, s);
  if (e != cudaSuccess) return cuda_fail(e, "memset");
  const unsigned gy = unsigned(n / 8 < 256 ? (n / 8 > 0 ? n / 8 : 1) : 256);
  k_colstats<<<dim3((m->nin + 31) / 32, gy), dim3(32, 8), 0, s>>>(n, m->nin, d_feat, m->acc);
  k_colstats_final<<<(m->nin + 127) / 128, 128, 0, s>>>(n, m->nin, m->acc, m->fmean, m->finv, nullptr);
  e = cudaMemsetAsync(m->acc, 0, sizeof(double) * 2 * cmax, s);
  if (e != cudaSuccess) return cuda_fail(e, "memset");
  k_colstats<<<dim3((m->n3 + 31) / 32, gy), dim3(32, 8), 0, s>>>(n, m->n3, d_tgt, m->acc);
  k_colstats_final<<<(m->n3 + 127) / 128, 128, 0, s>>>(n, m->n3, m->acc, m->tmean, m->tinv, m->tstd);
  e = cudaGetLastError();
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_fit_normalization");
}

extern "C" dmn_status dmn_mlp_normalize_features(dmn_mlp m, dmn_stream stream, int64_t n,
                                                 const float *d_feat, void *d_x_bf16) {
  set_error_message("");
  if (!m || n < 0 || !d_feat || !d_x_bf16) return fail(DMN_ERR_ARG, "dmn_mlp_normalize_features: invalid argument");
  if (n == 0) return DMN_OK;
  k_norm_x<<<blocks_for(n * m->kin), 256, 0, (cudaStream_t)stream>>>(
      n, m->nin, m->kin, d_feat, m->fmean, m->finv, static_cast<bf16 *>(d_x_bf16));
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_normalize_features");
}

extern "C" dmn_status dmn_mlp_normalize_targets(dmn_mlp m, dmn_stream stream, int64_t n,
                                                const float *d_tgt, float *d_t) {
  set_error_message("");
  if (!m || n < 0 || !d_tgt || !d_t) return fail(DMN_ERR_ARG, "dmn_mlp_normalize_targets: invalid argument");
  if (n == 0) return DMN_OK;
  k_norm_t<<<blocks_for(n * m->nout_pad), 256, 0, (cudaStream_t)stream>>>(
      n, m->n3, m->nout_pad, d_tgt, m->tmean, m->tinv, d_t);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_normalize_targets");
}

extern "C" dmn_status dmn_mlp_train_step(dmn_mlp m, dmn_stream stream, int64_t n,
                                         const void *d_x_bf16, const float *d_t, float lr,
                                         float *d_loss) {
  set_error_message("");
  if (!m || n < 1 || n > m->bmax || !d_x_bf16 || !d_t || !(lr >= 0.0f))
    return fail(DMN_ERR_ARG, "dmn_mlp_train_step: invalid argument");
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t npad = rup(n, 128);
  const bf16 *x = nullptr;
  const float *t = d_t;
  cudaError_t e = stage_x(m, s, n, d_x_bf16, &x);
  if (e == cudaSuccess && (reinterpret_cast<uintptr_t>(d_t) & 15)) {
    t = m->t;
    e = cudaMemcpyAsync(m->t, d_t, sizeof(float) * m->nout_pad * n, cudaMemcpyDeviceToDevice, s);
  }
  if (e != cudaSuccess) return cuda_fail(e, "dmn_mlp_train_step staging");
  if ((e = forward(m, s, n, npad, t, nullptr, x)) != cudaSuccess) return cuda_fail(e, "forward");
  for (int l = m->L - 1; l > 0; --l) {  // input gradient through W_l and silu' of the layer below
    EpiArgs ed;
    memset(&ed, 0, sizeof(ed));
    ed.err = m->err;
    ed.mode = EPI_DSILU;
    ed.z_in = m->z[l - 1];
    ed.h_out = m->dz[l - 1];
    ed.ldc = m->H;
    if ((e = gemm_dgrad(s, m->dz[l], m->w[l], int(npad), m->din[l], m->dout[l], ed)) != cudaSuccess)
      return cuda_fail(e, "dgrad");
  }
  WgradArgs wg = {};  // weight gradients dW_l = dZ_l^T . input_l (reduction over the batch)
  wg.err = m->err;
  for (int l = 0; l < m->L; ++l)
    if (!wgrad_add(wg, m->dz[l], l == 0 ? x : m->h[l - 1], m->dout[l], m->din[l], int(npad), m->grads + m->ow[l],
                   l == 0 ? n : npad))
      return cuda_fail(cudaErrorInvalidValue, "wgrad");
  PackArgs P = {};
  P.layers = m->L;
  for (int l = 0; l < m->L; ++l) {
    wg.dz[l] = m->dz[l];
    wg.db[l] = m->grads + m->ob[l];
    wg.cols[l] = m->dout[l];
    wg.cblk0[l + 1] = wg.cblk0[l] + m->dout[l] / CS_COLS;
    P.ow[l] = m->ow[l];
    P.ob[l] = m->ob[l];
    P.w[l] = m->w[l];
  }
  wg.nloss = int(npad / BM) * (m->nout_pad / BN) * 4;
  wg.loss_part = m->lpart;
  wg.loss = d_loss;
  wg.lscale = 1.0f / (float(n) * float(m->n3));
  const bool small = overlaps(int(npad), m->H);
  if ((e = launch_chained(small, gemm_bf16_wgrad, dim3(wg.blk0[m->L] + wg.cblk0[m->L] + (d_loss ? 1 : 0)), dim3(128),
                          tile_smem(WG_BN, WG_ST), s, wg, int(npad))) != cudaSuccess)
    return cuda_fail(e, "wgrad");
  m->step += 1;
  const int64_t n4 = m->nparam / 4;
  e = launch_chained(
      small, k_amsgrad_pack, dim3(unsigned((n4 + 255) / 256)), dim3(256), 0, s, n4, reinterpret_cast<float4 *>(m->params), reinterpret_cast<const float4 *>(m->grads),
      reinterpret_cast<float4 *>(m->m), reinterpret_cast<float4 *>(m->v), reinterpret_cast<float4 *>(m->vmax),
      ams_args(lr, kBeta1, kBeta2, kEps, m->step), P);
  if (e != cudaSuccess) return cuda_fail(e, "dmn_mlp_train_step");
  return DMN_OK;
}

extern "C" dmn_status dmn_mlp_amsgrad(dmn_stream stream, int64_t n, float *d_w, const float *d_g,
                                      float *d_m, float *d_v, float *d_vmax, float lr, float beta1,
                                      float beta2, float eps, int64_t step) {
  set_error_message("");
  if (n < 0 || step < 1) return fail(DMN_ERR_ARG, "dmn_mlp_amsgrad: n >= 0 and step >= 1 required");
  if (n == 0) return DMN_OK;
  if (!d_w || !d_g || !d_m || !d_v || !d_vmax) return fail(DMN_ERR_ARG, "dmn_mlp_amsgrad: NULL pointer");
  if (!(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps > 0.0f) ||
      !isfinite(lr))
    return fail(DMN_ERR_ARG, "dmn_mlp_amsgrad: 0 <= beta < 1, eps > 0 required");
  k_amsgrad<<<blocks_for(n), 256, 0, (cudaStream_t)stream>>>(n, d_w, d_g, d_m, d_v, d_vmax,
                                                             ams_args(lr, beta1, beta2, eps, step));
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_amsgrad");
}

extern "C" dmn_status dmn_mlp_get_moments(dmn_mlp m, float *h_m, float *h_v, float *h_vmax) {
  if (!m) return fail(DMN_ERR_ARG, "dmn_mlp_get_moments: NULL");
  cudaError_t e = cudaSuccess;
  if (h_m && e == cudaSuccess) e = cudaMemcpy(h_m, m->m, sizeof(float) * m->nparam, cudaMemcpyDeviceToHost);
  if (h_v && e == cudaSuccess) e = cudaMemcpy(h_v, m->v, sizeof(float) * m->nparam, cudaMemcpyDeviceToHost);
  if (h_vmax && e == cudaSuccess)
    e = cudaMemcpy(h_vmax, m->vmax, sizeof(float) * m->nparam, cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_get_moments");
}

extern "C" dmn_status dmn_mlp_predict(dmn_mlp m, dmn_stream stream, int64_t n, const void *d_x_bf16,
                                      float *d_da) {
  set_error_message("");
  if (!m || n < 0 || n > m->bmax || !d_x_bf16 || !d_da) return fail(DMN_ERR_ARG, "dmn_mlp_predict: invalid argument");
  if (n == 0) return DMN_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t npad = rup(n, 128);
  const bf16 *x = nullptr;
  cudaError_t e = stage_x(m, s, n, d_x_bf16, &x);
  if (e == cudaSuccess) e = forward(m, s, n, npad, nullptr, d_da, x);
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_predict");
}

extern "C" int64_t dmn_mlp_param_count(dmn_mlp m) { return m ? m->nparam : -1; }

extern "C" dmn_status dmn_mlp_get_params(dmn_mlp m, float *h) {
  if (!m || !h) return fail(DMN_ERR_ARG, "dmn_mlp_get_params: invalid argument");
  cudaError_t e = cudaMemcpy(h, m->params, sizeof(float) * m->nparam, cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_get_params");
}

extern "C" dmn_status dmn_mlp_set_params(dmn_mlp m, const float *h) {
  if (!m || !h) return fail(DMN_ERR_ARG, "dmn_mlp_set_params: invalid argument");
  cudaError_t e = cudaMemcpy(m->params, h, sizeof(float) * m->nparam, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = pack_all(m, 0);
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_set_params");
}

extern "C" dmn_status dmn_mlp_get_grads(dmn_mlp m, float *h) {
  if (!m || !h) return fail(DMN_ERR_ARG, "dmn_mlp_get_grads: invalid argument");
  cudaError_t e = cudaMemcpy(h, m->grads, sizeof(float) * m->nparam, cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_get_grads");
}

extern "C" dmn_status dmn_mlp_get_normalization(dmn_mlp m, float *fmean, float *finv, float *tmean,
                                                float *tstd) {
  if (!m) return fail(DMN_ERR_ARG, "dmn_mlp_get_normalization: NULL");
  cudaError_t e = cudaSuccess;
  if (fmean && e == cudaSuccess) e = cudaMemcpy(fmean, m->fmean, sizeof(float) * m->nin, cudaMemcpyDeviceToHost);
  if (finv && e == cudaSuccess) e = cudaMemcpy(finv, m->finv, sizeof(float) * m->nin, cudaMemcpyDeviceToHost);
  if (tmean && e == cudaSuccess) e = cudaMemcpy(tmean, m->tmean, sizeof(float) * m->n3, cudaMemcpyDeviceToHost);
  if (tstd && e == cudaSuccess) e = cudaMemcpy(tstd, m->tstd, sizeof(float) * m->n3, cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_mlp_get_normalization");
}

extern "C" dmn_status dmn_gemm_bf16_tn(dmn_stream stream, int32_t M, int32_t N, int32_t K,
                                       const void *d_a, const void *d_b, float *d_c) {
  set_error_message("");
  if (!d_a || !d_b || !d_c || M <= 0 || N <= 0 || K <= 0 || M % 128 || N % 128 || K % 64)
    return fail(DMN_ERR_ARG, "dmn_gemm_bf16_tn: M, N must be multiples of 128 and K of 64");
  if (reinterpret_cast<uintptr_t>(d_c) & 15)  // rows leave as 16- or 32-byte stores
    return fail(DMN_ERR_ARG, "dmn_gemm_bf16_tn: d_c must be 16-byte aligned");
  EpiArgs ep;
  memset(&ep, 0, sizeof(ep));
  ep.mode = EPI_F32;
  ep.f_out = d_c;
  ep.ldc = N;
  cudaError_t e = gemm((cudaStream_t)stream, d_a, d_b, M, N, K, ep, M);
  return e == cudaSuccess ? DMN_OK : cuda_fail(e, "dmn_gemm_bf16_tn");
}
