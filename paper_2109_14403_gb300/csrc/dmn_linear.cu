// dmn_linear.cu -- the DMN's linear elastic homogenization function DMN^L and
// the reverse-mode gradient of the offline-training loss (arXiv 2109.14403,
// Sec. 3.2), for a batch of stiffness samples.  Declared in
// include/dmn_linear.h.
//
// dmn_linear_forward: one CTA of G = 2^(K-1) threads per sample, persistent
// over the batch; the laminates of a level run one per thread, the levels one
// after another with a barrier, the node stiffnesses in shared memory.
// dmn_linear_loss_grad: level-synchronous over the whole batch, one launch
// per level (FP32: two levels) and direction, every (sample, node) pair a
// thread, the node stiffnesses and their adjoints in the caller's workspace;
// the backward pass walks the tree top-down: per node it turns the adjoint G of
// its stiffness into the adjoints of its two children and into dJ/dn and
// dJ/dc1, which each block sums over its samples before one FP64 atomic add.
// A laminate is computed in condensed form: with D = C_L - C_R, M = c2 C_L +
// c1 C_R, U = D B, K = B^T M B,
//   C = c1 C_L + c2 C_R - c1 c2 U K^-1 U^T,
// and its reverse mode, with W = U K^-1, A = G W, Q = W^T G W:
//   G_L = c1 G - 2 c1 c2 sym(A B^T) + c1 c2^2 B Q B^T
//   G_R = c2 G + 2 c1 c2 sym(A B^T) + c1^2 c2 B Q B^T
//   dJ/dc1 = <G, D> - (c2 - c1) <U, A> - c1 c2 <Q, B^T U>
//   dJ/dB = -2 c1 c2 (D A - M B Q)
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "../../include/dmn_linear.h"
#include "dmn_internal.h"
#include "pdl.cuh"

namespace dmn {
namespace {

constexpr int kLinMaxK = 8;

// B a = sym(a (x) n): 6x3, nine of its entries zero
__host__ __device__ constexpr bool bnz(int a, int f) { return a < 3 ? a == f : f != a - 3; }
template <typename T>
__device__ __forceinline__ void bmat(const T n[3], T B[6][3]) {
  const T r = T(kRsq2);
#pragma unroll
  for (int a = 0; a < 6; ++a)
#pragma unroll
    for (int f = 0; f < 3; ++f) B[a][f] = T(0);
  B[0][0] = n[0];
  B[1][1] = n[1];
  B[2][2] = n[2];
  B[3][1] = r * n[2];
  B[3][2] = r * n[1];
  B[4][0] = r * n[2];
  B[4][2] = r * n[0];
  B[5][0] = r * n[1];
  B[5][1] = r * n[0];
}

__device__ __forceinline__ float mad(float x, float y, float z) { return fmaf(x, y, z); }
__device__ __forceinline__ double mad(double x, double y, double z) { return fma(x, y, z); }
// x y + z w, every operation rounded (no fused multiply-add)
__device__ __forceinline__ float sum_rn(float x, float y, float z, float w) {
  return __fadd_rn(__fmul_rn(x, y), __fmul_rn(z, w));
}
__device__ __forceinline__ double sum_rn(double x, double y, double z, double w) {
  return __dadd_rn(__dmul_rn(x, y), __dmul_rn(z, w));
}

// The sums over B skip its zeros: IEEE arithmetic does not let the compiler
// drop a product with a zero it knows (the other factor could be infinite).
// Operations counted in the source (a fused multiply-add as one): a laminate's
// forward 459, with the zeros 810; its reverse mode with the children's adjoints
// 1,147 and 1,803 (65,536 samples, K = 8: the step 1837 -> 1720 us).  What is left keeps the order and the roundings of the full sums (fused
// multiply-adds from the first product on), so gradients keep their bits.
// sum_b x[b] B[b][f]
template <typename T>
__device__ __forceinline__ T row_b(const T x[6], const T B[6][3], int f) {
  T s = T(0);
#pragma unroll
  for (int b = 0; b < 6; ++b)
    if (bnz(b, f)) s = mad(x[b], B[b][f], s);
  return s;
}
// sum_f x[f] B[a][f], the first two products joined as x0 B0 + (x1 B1)
template <typename T>
__device__ __forceinline__ T row_bt(const T x[3], const T B[6][3], int a) {
  if (a < 3) return x[a] * B[a][a];
  if (a == 3) return mad(x[2], B[3][2], x[1] * B[3][1]);
  if (a == 4) return mad(x[2], B[4][2], x[0] * B[4][0]);
  return mad(x[0], B[5][0], x[1] * B[5][1]);
}

// U = D B, MB = M B, K^-1 (symmetric), W = U K^-1
template <typename T>
__device__ __forceinline__ void lam_core(const T *CL, const T *CR, const T B[6][3], T c1, T U[6][3],
                                         T MB[6][3], T Ki[3][3], T W[6][3]) {
  const T c2 = T(1) - c1;
#pragma unroll
  for (int a = 0; a < 6; ++a) {
    T d[6], m[6];
#pragma unroll
    for (int b = 0; b < 6; ++b) {
      const T l = sget(CL, a, b), r = sget(CR, a, b);
      d[b] = l - r;
      m[b] = c2 * l + c1 * r;
    }
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      U[a][f] = row_b(d, B, f);
      MB[a][f] = row_b(m, B, f);
    }
  }
  T Kk[3][3];
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    const T col[6] = {MB[0][f], MB[1][f], MB[2][f], MB[3][f], MB[4][f], MB[5][f]};
#pragma unroll
    for (int e = 0; e < 3; ++e) Kk[e][f] = row_b(col, B, e);
  }
  const T k00 = Kk[0][0], k11 = Kk[1][1], k22 = Kk[2][2];
  const T k01 = T(0.5) * (Kk[0][1] + Kk[1][0]), k02 = T(0.5) * (Kk[0][2] + Kk[2][0]);
  const T k12 = T(0.5) * (Kk[1][2] + Kk[2][1]);
  const T a00 = k11 * k22 - k12 * k12, a01 = k02 * k12 - k01 * k22, a02 = k01 * k12 - k02 * k11;
  const T a11 = k00 * k22 - k02 * k02, a12 = k01 * k02 - k00 * k12, a22 = k00 * k11 - k01 * k01;
  const T id = T(1) / (k00 * a00 + k01 * a01 + k02 * a02);
  Ki[0][0] = a00 * id;
  Ki[0][1] = Ki[1][0] = a01 * id;
  Ki[0][2] = Ki[2][0] = a02 * id;
  Ki[1][1] = a11 * id;
  Ki[1][2] = Ki[2][1] = a12 * id;
  Ki[2][2] = a22 * id;
#pragma unroll
  for (int a = 0; a < 6; ++a)
#pragma unroll
    for (int f = 0; f < 3; ++f) W[a][f] = U[a][0] * Ki[0][f] + U[a][1] * Ki[1][f] + U[a][2] * Ki[2][f];
}

template <typename T>
__device__ __forceinline__ void lam_forward(const T *CL, const T *CR, const T n[3], T c1, T *out) {
  T B[6][3], U[6][3], MB[6][3], Ki[3][3], W[6][3];
  bmat(n, B);
  lam_core(CL, CR, B, c1, U, MB, Ki, W);
  const T c2 = T(1) - c1, cc = c1 * c2;
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = i; j < 6; ++j) {
      const int q = sidx(i, j);
      out[q] = c1 * CL[q] + c2 * CR[q] - cc * (W[i][0] * U[j][0] + W[i][1] * U[j][1] + W[i][2] * U[j][2]);
    }
}

// reverse mode of one laminate; the children's adjoints GL, GR are formed if
// `kids` (leaf children have none)
template <bool kids, typename T>
__device__ __forceinline__ void lam_backward(const T *CL, const T *CR, const T n[3], T c1, const T *G, T *GL, T *GR,
                                             T gn[3], T &gc1) {
  T B[6][3], U[6][3], MB[6][3], Ki[3][3], W[6][3];
  bmat(n, B);
  lam_core(CL, CR, B, c1, U, MB, Ki, W);
  const T c2 = T(1) - c1, cc = c1 * c2;
  T A[6][3];
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      T s = T(0);
#pragma unroll
      for (int j = 0; j < 6; ++j) s += sget(G, i, j) * W[j][f];
      A[i][f] = s;
    }
  T Q[3][3];
#pragma unroll
  for (int e = 0; e < 3; ++e)
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      T s = T(0);
#pragma unroll
      for (int i = 0; i < 6; ++i) s += W[i][e] * A[i][f];
      Q[e][f] = s;
    }
#pragma unroll
  for (int e = 0; e < 3; ++e)
#pragma unroll
    for (int f = e + 1; f < 3; ++f) Q[e][f] = Q[f][e] = T(0.5) * (Q[e][f] + Q[f][e]);
  // <G, D>, <U, A>, <Q, B^T U>
  T GD = T(0);
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = i; j < 6; ++j) {
      const int q = sidx(i, j);
      GD += (i == j ? T(1) : T(2)) * G[q] * (CL[q] - CR[q]);
    }
  T UA = T(0), QBU = T(0);
#pragma unroll
  for (int a = 0; a < 6; ++a)
#pragma unroll
    for (int f = 0; f < 3; ++f) UA += U[a][f] * A[a][f];
#pragma unroll
  for (int e = 0; e < 3; ++e)
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      const T col[6] = {U[0][f], U[1][f], U[2][f], U[3][f], U[4][f], U[5][f]};
      QBU += Q[e][f] * row_b(col, B, e);
    }
  gc1 = GD - (c2 - c1) * UA - cc * QBU;
  // dJ/dB = -2 c1 c2 (D A - M B Q), then dJ/dn through B(n)
  T gB[6][3];
#pragma unroll
  for (int a = 0; a < 6; ++a)
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      if (!bnz(a, f)) continue;
      T da = T(0);
#pragma unroll
      for (int b = 0; b < 6; ++b) da += (sget(CL, a, b) - sget(CR, a, b)) * A[b][f];
      const T mbq = MB[a][0] * Q[0][f] + MB[a][1] * Q[1][f] + MB[a][2] * Q[2][f];
      gB[a][f] = T(-2) * cc * (da - mbq);
    }
  const T r = T(kRsq2);
  gn[0] = gB[0][0] + r * (gB[4][2] + gB[5][1]);
  gn[1] = gB[1][1] + r * (gB[3][2] + gB[5][0]);
  gn[2] = gB[2][2] + r * (gB[3][1] + gB[4][0]);
  if constexpr (kids) {
    T BQ[6][3];
#pragma unroll
    for (int a = 0; a < 6; ++a)
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const T col[3] = {Q[0][f], Q[1][f], Q[2][f]};
        // BQ[4][1]: two rounded products, each of which another entry has too (Q
        // is symmetric: r n2 Q[0][1] in BQ[3][0], r n0 Q[1][2] in BQ[5][2])
        BQ[a][f] = a == 4 && f == 1 ? sum_rn(col[0], B[4][0], col[2], B[4][2]) : row_bt(col, B, a);
      }
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
      for (int j = i; j < 6; ++j) {
        const int q = sidx(i, j);
        T ab = row_bt(A[i], B, j);
#pragma unroll
        for (int f = 0; f < 3; ++f)
          if (bnz(i, f)) ab = mad(A[j][f], B[i][f], ab);
        ab = T(0.5) * ab;
        const T bqb = row_bt(BQ[i], B, j);
        GL[q] = c1 * G[q] - T(2) * cc * ab + cc * c2 * bqb;
        GR[q] = c2 * G[q] + T(2) * cc * ab + cc * c1 * bqb;
      }
  }
}

// shared-memory carving of dmn_linear_forward (T words): normals 3N, c1 N,
// phases 42, nodes 21N
struct LinLayout {
  int nh, c1, ph, ns, words;
};
__host__ __device__ inline LinLayout lin_layout(int K) {
  const int N = (1 << K) - 1;
  LinLayout L;
  L.nh = 0;
  L.c1 = L.nh + 3 * N;
  L.ph = L.c1 + N;
  L.ns = L.ph + 42;
  L.words = L.ns + 21 * N;
  return L;
}

// per-CTA constants: normalised normals, c1 from the weight propagation
// (Sec. 3.1, bottom level first; c1 = W_1 / (W_1 + W_2)).  The subtree
// weights use the node array as scratch (it is free before the first sample);
// ends with a barrier.
template <typename T>
__device__ void lin_constants(int K, const double *normals, const double *v, T *nh, T *c1s, T *scratch) {
  const int N = (1 << K) - 1, L = 1 << K, t = threadIdx.x;
  for (int p = t; p < N; p += blockDim.x) {
    const double x = normals[3 * p], y = normals[3 * p + 1], z = normals[3 * p + 2];
    const double il = 1.0 / sqrt(x * x + y * y + z * z);
    nh[3 * p] = T(x * il);
    nh[3 * p + 1] = T(y * il);
    nh[3 * p + 2] = T(z * il);
  }
  T *Wt = scratch;  // leaves [0, L), nodes [L, L + N)
  for (int j = t; j < L; j += blockDim.x) Wt[j] = T(v[j] > 0.0 ? v[j] : 0.0);
  __syncthreads();
  for (int k = K; k >= 1; --k) {
    for (int i = t; i < (1 << (k - 1)); i += blockDim.x) {
      const int p = (1 << K) - (1 << k) + i;
      const int pc = (1 << K) - (1 << (k + 1)) + 2 * i;
      const T a = k == K ? Wt[2 * i] : Wt[L + pc], b = k == K ? Wt[2 * i + 1] : Wt[L + pc + 1];
      const T W = a + b;
      Wt[L + p] = W;
      c1s[p] = W > T(0) ? a / W : T(0.5);
    }
    __syncthreads();
  }
}

template <typename T>
__device__ void load_phases(const double *C1, const double *C2, T *ph) {
  for (int q = threadIdx.x; q < 42; q += blockDim.x) {
    const double *C = q < 21 ? C1 : C2;
    const int r = q < 21 ? q : q - 21;
    int i = 0, j = 0;
    for (int a = 0, k = 0; a < 6; ++a)
      for (int b = a; b < 6; ++b, ++k)
        if (k == r) {
          i = a;
          j = b;
        }
    ph[q] = T(0.5 * (C[6 * i + j] + C[6 * j + i]));
  }
}

// bottom-up pass of one sample into the node array
template <typename T>
__device__ void lin_sweep_up(int K, const T *nh, const T *c1s, const T *ph, T *ns) {
  for (int k = K; k >= 1; --k) {
    const int cnt = 1 << (k - 1);
    for (int j = threadIdx.x; j < cnt; j += blockDim.x) {
      const int p = (1 << K) - (1 << k) + j;
      const T *CL, *CR;
      if (k == K) {
        CL = ph;
        CR = ph + 21;
      } else {
        const int pc = (1 << K) - (1 << (k + 1)) + 2 * j;
        CL = ns + 21 * pc;
        CR = ns + 21 * (pc + 1);
      }
      lam_forward(CL, CR, nh + 3 * p, c1s[p], ns + 21 * p);
    }
    __syncthreads();
  }
}

// x^p and x^(1/p) for x >= 0, MODE 1: p = 1, 2: p = 2, 0: any p.  The first two
// take no pow(): with 72 to 93 powers a sample on the FP64 pipe the error and
// seed kernels took 956 and 1540 us of a 6890 us training step (p = 1, K = 8,
// 65,536 samples).  The mode is a template argument of the sums: a test of p in
// every term is an FP64 comparison each.
__host__ __device__ inline int pow_mode(double p) { return p == 1.0 ? 1 : (p == 2.0 ? 2 : 0); }
template <int MODE>
__device__ __forceinline__ double pow_p(double x, double p) {
  return MODE == 1 ? x : (MODE == 2 ? x * x : pow(x, p));
}
template <int MODE>
__device__ __forceinline__ double root_p(double x, double p) {
  return MODE == 1 ? x : (MODE == 2 ? sqrt(x) : pow(x, 1.0 / p));
}

// x^q for x >= 0; a whole q up to 16 by repeated squaring: the relative error
// of x^k is at most (k - 1) 2^-53 however the products are paired (seen: 11 2^-53 at
// q = 16; 45 at 64, so larger q take pow()).  One FP64 pow() is a serial chain of some 8 us here,
// and a 32-sample step had six of them in a row.
constexpr double kSquaringMaxQ = 16.0;
__device__ __forceinline__ double pow_q(double x, double q) {
  if (!(q >= 0.0 && q <= kSquaringMaxQ) || q != floor(q)) return pow(x, q);
  double r = 1.0;
  for (int k = int(q); k; k >>= 1, x *= x)
    if (k & 1) r *= x;
  return r;
}

// S^(1/q): a whole q up to 16 from the FP32 root by two Newton steps (a relative
// error e becomes (q - 1) / 2 e^2: 1e-6 -> 7.5e-12 at most -> rounding, 1/q of pow_q's
// error among it), a fifth of the FP64 pow()'s chain
__device__ __forceinline__ double root_q(double S, double q) {
  if (!(q >= 1.0 && q <= kSquaringMaxQ) || q != floor(q) || !(S > 1e-30 && S < 1e30)) return pow(S, 1.0 / q);
  double x = double(powf(float(S), float(1.0 / q)));
#pragma unroll 1
  for (int k = 0; k < 2; ++k) {
    const double y = pow_q(x, q - 1.0);
    x -= (x * y - S) / (q * y);
  }
  return x;
}

// |x|_p of the 36 components f(i, j), six partial sums
template <int MODE, typename F>
__device__ __forceinline__ double lin_norm(double p, F f) {
  double col[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll(MODE ? 6 : 1)
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < 6; ++j) col[j] += pow_p<MODE>(fabs(f(i, j)), p);
  return root_p<MODE>(((col[0] + col[1]) + (col[2] + col[3])) + (col[4] + col[5]), p);
}

// The error and seed kernels take a sample on LP = 1 thread, or on eight lanes,
// one row of the six each, where the batch is too small to fill the SMs (an
// FP64 instruction holds a warp's sub-partition for 64 cycles, so what counts
// there is the length of a lane's chain, not the number of lanes).
template <int LP>
__device__ __forceinline__ double lane_sum(double x) {
#pragma unroll
  for (int o = LP / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
// p-norm over the 36 components f(i, j) of a sample, row i on lane i
template <int MODE, int LP, typename F>
__device__ __forceinline__ double sample_norm(double p, int row, F f) {
  if (LP == 1) return lin_norm<MODE>(p, f);
  double a = 0.0, b = 0.0;
  if (row < 6) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      a += pow_p<MODE>(fabs(f(row, j)), p);
      b += pow_p<MODE>(fabs(f(row, j + 3)), p);
    }
  }
  return root_p<MODE>(lane_sum<LP>(a + b), p);
}

template <typename T>
__global__ void k_lin_forward(int K, int64_t n, const double *C1, const double *C2, const double *normals,
                              const double *v, double *Cbar) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T *sm = reinterpret_cast<T *>(smem_raw);
  const LinLayout L = lin_layout(K);
  const int N = (1 << K) - 1, root = N - 1;
  lin_constants<T>(K, normals, v, sm + L.nh, sm + L.c1, sm + L.ns);
  for (int64_t s = blockIdx.x; s < n; s += gridDim.x) {
    load_phases<T>(C1 + 36 * s, C2 + 36 * s, sm + L.ph);
    __syncthreads();
    lin_sweep_up<T>(K, sm + L.nh, sm + L.c1, sm + L.ph, sm + L.ns);
    const T *D = sm + L.ns + 21 * root;
    for (int q = threadIdx.x; q < 36; q += blockDim.x) Cbar[36 * s + q] = double(sget(D, q / 6, q % 6));
    __syncthreads();
  }
}

// Batch reduction of the errors, by the blocks that form them: block b leaves
// its largest error m_b and S_b = sum (e / m_b)^q in part[2b], part[2b + 1];
// the block that comes last (ticket) joins them in block order, so the result
// does not depend on the order of arrival:
//   scal[0] = m = max e, scal[1] = S^(1/q - 1) / n with S = sum (m_b / m)^q S_b,
//   scal[2] = the loss's data term.  A block whose errors are all zero (or
// NaN) has m_b = 0 and hands on their plain sum.  (One CTA over all errors, two
// general powers a sample in a row, took 1815 us at 65,536 samples; the step
// as a whole went from 6890 to 1837 us with this, the exact powers and the
// parallel chain through the weights, and from 1637 to 173 us at 32 samples.)
// All threads of all blocks call it; blockDim.x = kLvlThreads.
constexpr int kLvlThreads = 128;
__device__ __forceinline__ double block_max(double x, double *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  x = red[0];
  for (int w = 1; w < kLvlThreads / 32; ++w) x = fmax(x, red[w]);
  return x;
}
__device__ __forceinline__ double block_sum(double x, double *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  x = red[0];
  for (int w = 1; w < kLvlThreads / 32; ++w) x += red[w];
  return x;
}
__device__ void lin_reduce(int64_t n, double e, double q, double *part, double *scal) {
  __shared__ double red[kLvlThreads / 32];
  __shared__ bool last;
  const int t = threadIdx.x;
  const double mb = block_max(e, red);
  const double Sb = block_sum(mb > 0.0 ? pow_q(e / mb, q) : e, red);
  if (t == 0) {
    part[2 * blockIdx.x] = mb;
    part[2 * blockIdx.x + 1] = Sb;
    __threadfence();
    last = atomicAdd(reinterpret_cast<unsigned *>(scal + 4), 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double m = 0.0;
  for (unsigned b = t; b < gridDim.x; b += kLvlThreads) m = fmax(m, part[2 * b]);
  m = block_max(m, red);
  double acc = 0.0;
  if (m > 0.0)
    for (unsigned b = t; b < gridDim.x; b += kLvlThreads) {
      const double mm = part[2 * b];
      acc += mm > 0.0 ? pow_q(mm / m, q) * part[2 * b + 1] : part[2 * b + 1];
    }
  const double S = block_sum(acc, red);
  if (t == 0) {
    const double root = m > 0.0 ? root_q(S, q) / double(n) : 0.0;
    scal[0] = m;
    scal[1] = m > 0.0 ? root / S : 0.0;
    scal[2] = m * root;
  }
}

// ---- level-synchronous training pass over the whole batch.  Node values
// live in the caller's workspace as [node][21][sample] (samples fastest, so a
// warp's loads of one component are contiguous); one launch per level and
// direction, a 2-D grid of (sample blocks, nodes of the level), so every
// block serves one node and reduces its gradient terms before one atomic add.

template <typename T>
__device__ __forceinline__ void lvl_load(const T *X, int p, int64_t n, int64_t s, T out[21]) {
#pragma unroll
  for (int q = 0; q < 21; ++q) out[q] = X[(int64_t(p) * 21 + q) * n + s];
}
template <typename T>
__device__ __forceinline__ void lvl_store(T *X, int p, int64_t n, int64_t s, const T v[21]) {
#pragma unroll
  for (int q = 0; q < 21; ++q) X[(int64_t(p) * 21 + q) * n + s] = v[q];
}
template <typename T>
__device__ __forceinline__ void phase_packed(const double *C, T out[21]) {
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = i; j < 6; ++j) out[sidx(i, j)] = T(0.5 * (C[6 * i + j] + C[6 * j + i]));
}

// Slot of node pp's (level k) first child in an array of the leaves [0, L) and
// the nodes [L, L + N); its second child follows
__device__ __forceinline__ int child_slot(int K, int k, int pp) {
  const int i = pp - ((1 << K) - (1 << k));
  return k == K ? 2 * i : (2 << K) - (1 << (k + 1)) + 2 * i;
}
// level of node pp
__device__ __forceinline__ int node_level(int K, int pp) { return 32 - __clz((1 << K) - pp - 1); }
// the nodes' weights from the leaves' (slots as above); all threads of the
// block, at least 2^(K-1) of them; a barrier before and after each level
__device__ __forceinline__ void tree_weights(int K, int t, double *Wt) {
  for (int k = K; k >= 1; --k) {
    if (t < (1 << (k - 1))) {
      const int pp = (1 << K) - (1 << k) + t, ch = child_slot(K, k, pp);
      Wt[(1 << K) + pp] = Wt[ch] + Wt[ch + 1];
    }
    __syncthreads();
  }
}

// Set-up of a training pass, one launch:
//  block 0   c1 of every node in the laminate precision (first half of the
//            threads: the weights level by level, then all quotients at once)
//            and the normalised normals (second half);
//  block 1   zeroes the gradient sums and the scalars (nz doubles from acc);
//  others    the phase stiffnesses of every sample, packed, in the laminate
//            precision: PH[phase][21][sample] (converted once instead of by
//            every bottom laminate).
// Bound by the latency of FP64 division and square root: neither is in the
// level loop.
constexpr int kSetupThreads = 2 << kLinMaxK;
template <typename T>
__global__ void __launch_bounds__(kSetupThreads)
    k_lvl_setup(int K, int64_t n, const double *normals, const double *v, const double *C1, const double *C2, T *nh,
                T *c1s, T *PH, double *acc, int nz) {
  __shared__ double Wt[2 * (1 << kLinMaxK)];
  const int N = (1 << K) - 1, L = 1 << K, t = threadIdx.x;
  constexpr int H = kSetupThreads / 2;
  chain_begin();
  if (blockIdx.x > 1) {
    const int64_t i = int64_t(blockIdx.x - 2) * H + (t & (H - 1)), ph = t / H;  // one phase a thread
    if (i >= n) return;
    T a[21];
    phase_packed((ph ? C2 : C1) + 36 * i, a);
    lvl_store(PH, int(ph), n, i, a);
    return;
  }
  if (blockIdx.x == 1) {
    for (int i = t; i < nz; i += kSetupThreads) acc[i] = 0.0;
    return;
  }
  if (t < L) Wt[t] = v[t] > 0.0 ? v[t] : 0.0;
  if (t >= H && t - H < N) {
    const int pp = t - H;
    const double x = normals[3 * pp], y = normals[3 * pp + 1], z = normals[3 * pp + 2];
    const double il = 1.0 / sqrt(x * x + y * y + z * z);
    nh[3 * pp] = T(x * il);
    nh[3 * pp + 1] = T(y * il);
    nh[3 * pp + 2] = T(z * il);
  }
  __syncthreads();
  tree_weights(K, t, Wt);
  if (t < N) {
    const double a = Wt[child_slot(K, node_level(K, t), t)], W = Wt[L + t];
    c1s[t] = T(W > 0.0 ? a / W : 0.5);
  }
}

template <typename T>
__global__ void __launch_bounds__(kLvlThreads) k_lvl_fwd(int K, int k, int64_t n, const T *PH, const T *nh,
                                                         const T *c1s, T *NS) {
  chain_begin();
  const int64_t s = int64_t(blockIdx.x) * kLvlThreads + threadIdx.x;
  if (s >= n) return;
  const int j = blockIdx.y, pp = (1 << K) - (1 << k) + j;
  T CL[21], CR[21], out[21];
  if (k == K) {
    lvl_load(PH, 0, n, s, CL);
    lvl_load(PH, 1, n, s, CR);
  } else {
    const int pc = (1 << K) - (1 << (k + 1)) + 2 * j;
    lvl_load(NS, pc, n, s, CL);
    lvl_load(NS, pc + 1, n, s, CR);
  }
  const T nn[3] = {nh[3 * pp], nh[3 * pp + 1], nh[3 * pp + 2]};
  lam_forward(CL, CR, nn, c1s[pp], out);
  lvl_store(NS, pp, n, s, out);
}

// per-sample error e_s = |T - D|_p / |T|_p from the root column (FP64), and the
// batch reduction
template <int MODE, int LP, typename T>
__global__ void __launch_bounds__(kLvlThreads) k_lvl_err(int K, int64_t n, const T *NS, const double *Ct, double p,
                                                         double q, double *err, double *part, double *scal) {
  const int64_t s = (int64_t(blockIdx.x) * kLvlThreads + threadIdx.x) / LP;
  const int row = LP == 1 ? 0 : threadIdx.x % LP;
  chain_begin();
  double e = 0.0;
  const int64_t sc = s < n ? s : n - 1;  // lanes past the batch repeat its last sample
  const double *Tg = Ct + 36 * sc;
  const T *R = NS + (int64_t((1 << K) - 2) * 21) * n + sc;  // component q of the root: R[q n]
  T D[21];
  if (LP == 1) lvl_load(NS, (1 << K) - 2, n, sc, D);
  const double nx = sample_norm<MODE, LP>(p, row, [&](int i, int j) {
    return Tg[6 * i + j] - double(LP == 1 ? sget(D, i, j) : R[(i <= j ? sidx(i, j) : sidx(j, i)) * n]);
  });
  e = nx / sample_norm<MODE, LP>(p, row, [&](int i, int j) { return Tg[6 * i + j]; });
  if (s >= n || row != 0) e = 0.0;
  else err[s] = e;
  lin_reduce(n, e, q, part, scal);
}

// dJ/dD at the root: (1/N) S^(1/q-1) (e_s/m)^(q-1) de_s/dD, with |T - D|_p =
// e_s |T|_p; for p = 1 every component's is +-1 / |T|_1
template <int MODE, int LP, typename T>
__device__ __forceinline__ void lin_seed(int64_t n, int row, const double *Tg, const T *R, double p, double q,
                                         double e, const double *scal, bool st, T *G) {
  const double m = scal[0];
  const double coef = (m > 0.0 && e > 0.0) ? scal[1] * pow_q(e / m, q - 1.0) : 0.0;
  const double nt = sample_norm<MODE, LP>(p, row, [&](int i, int j) { return Tg[6 * i + j]; });
  const double f = MODE == 1 ? 1.0 / nt : (MODE == 2 ? 1.0 / (e * nt) : pow(e * nt, 1.0 - p)) / nt;
  auto put = [&](int i, int j) {
    const int c = sidx(i, j);
    const double x = Tg[6 * i + j] - double(R[c * n]);
    const double sg = x > 0.0 ? 1.0 : (x < 0.0 ? -1.0 : 0.0);
    const double xp = MODE == 1 ? 1.0 : (MODE == 2 ? fabs(x) : pow(fabs(x), p - 1.0));
    const double de = e > 0.0 ? -sg * xp * f : 0.0;
    if (st) G[c * n] = T(coef * de);
  };
  if (LP == 1) {
#pragma unroll
    for (int i = 0; i < 6; ++i)
#pragma unroll
      for (int j = i; j < 6; ++j) put(i, j);
  } else {
#pragma unroll
    for (int j = 0; j < 6; ++j)
      if (row <= j) put(row, j);
  }
}
// Also, in the last block, the weights' sum in leaf order (into scal[5]: one
// thread, 9 us at K = 8 beside the other blocks; the weights sum to about 1 and
// 1 is taken off, so its order shows) and the loss (J, data term, penalty).
template <int MODE, int LP, typename T>
__global__ void __launch_bounds__(kLvlThreads) k_lvl_seed(int K, int64_t n, const T *NS, const double *Ct, double p,
                                                          double q, const double *err, const double *v,
                                                          double penalty, double *scal, double *loss, T *GA) {
  __shared__ double wl[1 << kLinMaxK];
  chain_begin();
  if (blockIdx.x == gridDim.x - 1) {
    for (int j = threadIdx.x; j < (1 << K); j += kLvlThreads) wl[j] = v[j] > 0.0 ? v[j] : 0.0;
    __syncthreads();
    if (threadIdx.x == 0) {
      double w = 0.0;
#pragma unroll 8
      for (int j = 0; j < (1 << K); ++j) w += wl[j];
      const double data = scal[2], pen = penalty * (w - 1.0) * (w - 1.0);
      scal[5] = w;
      loss[0] = data + pen;
      loss[1] = data;
      loss[2] = pen;
    }
    return;
  }
  const int64_t s = (int64_t(blockIdx.x) * kLvlThreads + threadIdx.x) / LP;
  const int row = LP == 1 ? 0 : threadIdx.x % LP;
  const int64_t sc = s < n ? s : n - 1, root = int64_t((1 << K) - 2) * 21 * n + sc;
  lin_seed<MODE, LP>(n, row, Ct + 36 * sc, NS + root, p, q, err[sc], scal, s < n, GA + root);
}

template <typename T>
__global__ void __launch_bounds__(kLvlThreads) k_lvl_bwd(int K, int k, int64_t n, const T *PH, const T *nh,
                                                         const T *c1s, const T *NS, T *GA, double *gnh,
                                                         double *gc1) {
  chain_begin();
  __shared__ T red[4][kLvlThreads / 32];
  const int64_t s = int64_t(blockIdx.x) * kLvlThreads + threadIdx.x;
  const int j = blockIdx.y, pp = (1 << K) - (1 << k) + j;
  T gn[3] = {T(0), T(0), T(0)}, g1 = T(0);
  if (s < n) {
    T CL[21], CR[21], G[21], GL[21], GR[21];
    const int pc = (1 << K) - (1 << (k + 1)) + 2 * j;
    if (k == K) {
      lvl_load(PH, 0, n, s, CL);
      lvl_load(PH, 1, n, s, CR);
    } else {
      lvl_load(NS, pc, n, s, CL);
      lvl_load(NS, pc + 1, n, s, CR);
    }
    lvl_load(GA, pp, n, s, G);
    const T nn[3] = {nh[3 * pp], nh[3 * pp + 1], nh[3 * pp + 2]};
    if (k == K) {
      lam_backward<false>(CL, CR, nn, c1s[pp], G, GL, GR, gn, g1);
    } else {
      lam_backward<true>(CL, CR, nn, c1s[pp], G, GL, GR, gn, g1);
      lvl_store(GA, pc, n, s, GL);
      lvl_store(GA, pc + 1, n, s, GR);
    }
  }
  // block sums of dJ/dn and dJ/dc1 of this node (laminate precision), one
  // FP64 atomic add each
  T r[4] = {gn[0], gn[1], gn[2], g1};
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r[c] += __shfl_down_sync(0xffffffffu, r[c], o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0)
#pragma unroll
    for (int c = 0; c < 4; ++c) red[c][warp] = r[c];
  __syncthreads();
  if (threadIdx.x < 4) {
    T acc = T(0);
    for (int w = 0; w < kLvlThreads / 32; ++w) acc += red[threadIdx.x][w];
    atomicAdd(threadIdx.x < 3 ? gnh + 3 * pp + threadIdx.x : gc1 + pp, double(acc));
  }
}

// Two levels in one pass, FP32 laminates: a thread takes node j of level k and
// its two children (level k + 1) of one sample, so that the children's
// stiffnesses go to the parent, and the parent's adjoints to the children, in
// registers.  LEAF: the children are bottom laminates (their children the
// phases).  Of the 12 words of 21 a parent and its children move in two
// launches (forward: 4 in, 2 in again, 3 out) the pass keeps 7; of the reverse
// mode's 19 (9 + 2 x 5, no adjoints below the bottom) 15.  K = 8, 65,536
// samples: the step 1714 -> 1493 us; 32 samples (half the launches): 172 ->
// 155 us.
template <bool LEAF, typename T>
__global__ void __launch_bounds__(kLvlThreads, LEAF ? 3 : 4) k_lvl_fwd2(int K, int k, int64_t n, const T *PH, const T *nh,
                                                          const T *c1s, T *NS) {
  chain_begin();
  const int64_t s = int64_t(blockIdx.x) * kLvlThreads + threadIdx.x;
  if (s >= n) return;
  const int j = blockIdx.y, pp = (1 << K) - (1 << k) + j, pc = (1 << K) - (1 << (k + 1)) + 2 * j;
  const int pg = (1 << K) - (1 << (k + 2)) + 4 * j;  // grandchildren
  T X[21], Y[21];
  {
    T CL[21], CR[21];
    lvl_load(LEAF ? PH : NS, LEAF ? 0 : pg, n, s, CL);
    lvl_load(LEAF ? PH : NS, LEAF ? 1 : pg + 1, n, s, CR);
    const T nn[3] = {nh[3 * pc], nh[3 * pc + 1], nh[3 * pc + 2]};
    lam_forward(CL, CR, nn, c1s[pc], X);
    lvl_store(NS, pc, n, s, X);
  }
  {
    T CL[21], CR[21];
    lvl_load(LEAF ? PH : NS, LEAF ? 0 : pg + 2, n, s, CL);
    lvl_load(LEAF ? PH : NS, LEAF ? 1 : pg + 3, n, s, CR);
    const T nn[3] = {nh[3 * pc + 3], nh[3 * pc + 4], nh[3 * pc + 5]};
    lam_forward(CL, CR, nn, c1s[pc + 1], Y);
    lvl_store(NS, pc + 1, n, s, Y);
  }
  T out[21];
  const T nn[3] = {nh[3 * pp], nh[3 * pp + 1], nh[3 * pp + 2]};
  lam_forward(X, Y, nn, c1s[pp], out);
  lvl_store(NS, pp, n, s, out);
}

template <bool LEAF, typename T>
__global__ void __launch_bounds__(kLvlThreads, 3) k_lvl_bwd2(int K, int k, int64_t n, const T *PH, const T *nh,
                                                          const T *c1s, const T *NS, T *GA, double *gnh,
                                                          double *gc1) {
  chain_begin();
  __shared__ T red[3][4][kLvlThreads / 32];
  const int64_t s = int64_t(blockIdx.x) * kLvlThreads + threadIdx.x;
  const int j = blockIdx.y, pp = (1 << K) - (1 << k) + j, pc = (1 << K) - (1 << (k + 1)) + 2 * j;
  const int pg = (1 << K) - (1 << (k + 2)) + 4 * j;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // sums of dJ/dn and dJ/dc1 over the warp's samples
  auto warp_sums = [&](int node, const T gn[3], T g1) {
    T r[4] = {gn[0], gn[1], gn[2], g1};
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) r[c] += __shfl_down_sync(0xffffffffu, r[c], o);
    if (lane == 0)
#pragma unroll
      for (int c = 0; c < 4; ++c) red[node][c][warp] = r[c];
  };
  T G[21], GR[21];
  {
    T gn[3] = {T(0), T(0), T(0)}, g1 = T(0);
    if (s < n) {
      T CL[21], CR[21], GL[21];
      lvl_load(NS, pc, n, s, CL);
      lvl_load(NS, pc + 1, n, s, CR);
      lvl_load(GA, pp, n, s, G);
      const T nn[3] = {nh[3 * pp], nh[3 * pp + 1], nh[3 * pp + 2]};
      lam_backward<true>(CL, CR, nn, c1s[pp], G, GL, GR, gn, g1);
#pragma unroll
      for (int q = 0; q < 21; ++q) G[q] = GL[q];
    }
    warp_sums(0, gn, g1);
  }
#pragma unroll 1
  for (int c = 0; c < 2; ++c) {
    T gn[3] = {T(0), T(0), T(0)}, g1 = T(0);
    if (s < n) {
      T CL[21], CR[21];
      lvl_load(LEAF ? PH : NS, LEAF ? 0 : pg + 2 * c, n, s, CL);
      lvl_load(LEAF ? PH : NS, LEAF ? 1 : pg + 2 * c + 1, n, s, CR);
      const int p = pc + c;
      const T nn[3] = {nh[3 * p], nh[3 * p + 1], nh[3 * p + 2]};
      if (LEAF) {
        T *none = nullptr;
        lam_backward<false>(CL, CR, nn, c1s[p], G, none, none, gn, g1);
      } else {
        T HL[21], HR[21];
        lam_backward<true>(CL, CR, nn, c1s[p], G, HL, HR, gn, g1);
        lvl_store(GA, pg + 2 * c, n, s, HL);
        lvl_store(GA, pg + 2 * c + 1, n, s, HR);
      }
#pragma unroll
      for (int q = 0; q < 21; ++q) G[q] = GR[q];
    }
    warp_sums(1 + c, gn, g1);
  }
  __syncthreads();
  if (threadIdx.x < 12) {
    const int node = threadIdx.x >> 2, c = threadIdx.x & 3, p = node == 0 ? pp : pc + node - 1;
    T acc = T(0);
    for (int w = 0; w < kLvlThreads / 32; ++w) acc += red[node][c][w];
    atomicAdd(c < 3 ? gnh + 3 * p + c : gc1 + p, double(acc));
  }
}

// The same for a small batch, where a launch is as long as one thread's chain:
// the two children on two threads (warps w and w + 4 of 8), so a chain of two
// laminates, not three.  Forward: the second child's stiffness to the first's
// thread through shared memory.  Reverse: both threads take the parent, each its
// own child.  (K = 8, 32 samples: 93 -> 84 us.)
template <bool LEAF, typename T>
__global__ void __launch_bounds__(2 * kLvlThreads, 1)
    k_lvl_fwd2s(int K, int k, int64_t n, const T *PH, const T *nh, const T *c1s, T *NS) {
  __shared__ T ys[21][kLvlThreads];
  chain_begin();
  const int t = threadIdx.x % kLvlThreads, c = threadIdx.x / kLvlThreads;
  const int64_t s = int64_t(blockIdx.x) * kLvlThreads + t;
  const int j = blockIdx.y, pp = (1 << K) - (1 << k) + j, pc = (1 << K) - (1 << (k + 1)) + 2 * j + c;
  const int pg = (1 << K) - (1 << (k + 2)) + 4 * j + 2 * c;  // grandchildren of this child
  T X[21];
  if (s < n) {
    T CL[21], CR[21];
    lvl_load(LEAF ? PH : NS, LEAF ? 0 : pg, n, s, CL);
    lvl_load(LEAF ? PH : NS, LEAF ? 1 : pg + 1, n, s, CR);
    const T nn[3] = {nh[3 * pc], nh[3 * pc + 1], nh[3 * pc + 2]};
    lam_forward(CL, CR, nn, c1s[pc], X);
    if (c == 1)
#pragma unroll
      for (int q = 0; q < 21; ++q) ys[q][t] = X[q];
    lvl_store(NS, pc, n, s, X);
  }
  __syncthreads();
  if (c == 0 && s < n) {
    T Y[21], out[21];
#pragma unroll
    for (int q = 0; q < 21; ++q) Y[q] = ys[q][t];
    const T nn[3] = {nh[3 * pp], nh[3 * pp + 1], nh[3 * pp + 2]};
    lam_forward(X, Y, nn, c1s[pp], out);
    lvl_store(NS, pp, n, s, out);
  }
}

template <bool LEAF, typename T>
__global__ void __launch_bounds__(2 * kLvlThreads, 1)
    k_lvl_bwd2s(int K, int k, int64_t n, const T *PH, const T *nh, const T *c1s, const T *NS, T *GA, double *gnh,
                double *gc1) {
  __shared__ T red[3][4][kLvlThreads / 32];
  chain_begin();
  const int t = threadIdx.x % kLvlThreads, c = threadIdx.x / kLvlThreads;
  const int64_t s = int64_t(blockIdx.x) * kLvlThreads + t;
  const int j = blockIdx.y, pp = (1 << K) - (1 << k) + j, pc = (1 << K) - (1 << (k + 1)) + 2 * j;
  const int pg = (1 << K) - (1 << (k + 2)) + 4 * j + 2 * c;
  const int lane = t & 31, warp = t >> 5;
  auto warp_sums = [&](int node, const T gn[3], T g1) {
    T r[4] = {gn[0], gn[1], gn[2], g1};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) r[i] += __shfl_down_sync(0xffffffffu, r[i], o);
    if (lane == 0)
#pragma unroll
      for (int i = 0; i < 4; ++i) red[node][i][warp] = r[i];
  };
  T G[21];
  {
    T gn[3] = {T(0), T(0), T(0)}, g1 = T(0);
    if (s < n) {
      T CL[21], CR[21], GL[21], GR[21];
      lvl_load(NS, pc, n, s, CL);
      lvl_load(NS, pc + 1, n, s, CR);
      lvl_load(GA, pp, n, s, G);
      const T nn[3] = {nh[3 * pp], nh[3 * pp + 1], nh[3 * pp + 2]};
      lam_backward<true>(CL, CR, nn, c1s[pp], G, GL, GR, gn, g1);
#pragma unroll
      for (int q = 0; q < 21; ++q) G[q] = c ? GR[q] : GL[q];
    }
    if (c == 0) warp_sums(0, gn, g1);
  }
  {
    T gn[3] = {T(0), T(0), T(0)}, g1 = T(0);
    if (s < n) {
      T CL[21], CR[21];
      lvl_load(LEAF ? PH : NS, LEAF ? 0 : pg, n, s, CL);
      lvl_load(LEAF ? PH : NS, LEAF ? 1 : pg + 1, n, s, CR);
      const int p = pc + c;
      const T nn[3] = {nh[3 * p], nh[3 * p + 1], nh[3 * p + 2]};
      if (LEAF) {
        T *none = nullptr;
        lam_backward<false>(CL, CR, nn, c1s[p], G, none, none, gn, g1);
      } else {
        T HL[21], HR[21];
        lam_backward<true>(CL, CR, nn, c1s[p], G, HL, HR, gn, g1);
        lvl_store(GA, pg, n, s, HL);
        lvl_store(GA, pg + 1, n, s, HR);
      }
    }
    warp_sums(1 + c, gn, g1);
  }
  __syncthreads();
  if (threadIdx.x < 12) {
    const int node = threadIdx.x >> 2, i = threadIdx.x & 3, p = node == 0 ? pp : pc + node - 1;
    T acc = T(0);
    for (int w = 0; w < kLvlThreads / 32; ++w) acc += red[node][i][w];
    atomicAdd(i < 3 ? gnh + 3 * p + i : gc1 + p, double(acc));
  }
}

// The chain through the weights (c1 = W_1 / W, w = <v>_+, penalty) and the
// normalisation of the normals: one CTA.  Its second half takes the normals;
// the first the weights level by level, then every node's two quotients at
// once, then the adjoints of the subtree weights from the root down, so that
// the level loops hold additions only.  (One thread with the weights in local
// memory took 928 us at K = 8; divisions in the level loop, 19.)
__global__ void __launch_bounds__(kSetupThreads)
    k_lin_finish(int K, const double *normals, const double *v, double penalty, const double *gnh,
                 const double *gc1, const double *scal, double *grad_n, double *grad_v) {
  chain_begin();
  __shared__ double Wt[2 << kLinMaxK], gW[2 << kLinMaxK];  // leaves [0, L), nodes [L, L + N)
  const int N = (1 << K) - 1, L = 1 << K, t = threadIdx.x;
  constexpr int H = kSetupThreads / 2;
  if (t < L) Wt[t] = v[t] > 0.0 ? v[t] : 0.0;
  if (t >= H && t - H < N) {
    const int pp = t - H;
    const double x = normals[3 * pp], y = normals[3 * pp + 1], z = normals[3 * pp + 2];
    const double il = 1.0 / sqrt(x * x + y * y + z * z);
    const double nh[3] = {x * il, y * il, z * il};
    const double g[3] = {gnh[3 * pp], gnh[3 * pp + 1], gnh[3 * pp + 2]};
    const double gd = g[0] * nh[0] + g[1] * nh[1] + g[2] * nh[2];
    for (int c = 0; c < 3; ++c) grad_n[3 * pp + c] = (g[c] - gd * nh[c]) * il;
  }
  __syncthreads();
  tree_weights(K, t, Wt);
  if (t < N) {  // into the children's slots: what c1's derivative adds to the node's own adjoint
    const int ch = child_slot(K, node_level(K, t), t);
    const double W = Wt[L + t], a = Wt[ch], b = Wt[ch + 1], g = gc1[t];
    gW[ch] = W > 0.0 ? g * b / (W * W) : 0.0;       // d c1 / d W_1 = W_2 / W^2
    gW[ch + 1] = W > 0.0 ? -g * a / (W * W) : 0.0;  // d c1 / d W_2 = -W_1 / W^2
  }
  if (t == 0) gW[L + N - 1] = 2.0 * penalty * (scal[5] - 1.0);
  __syncthreads();
  for (int k = 1; k <= K; ++k) {
    if (t < (1 << (k - 1))) {
      const int pp = (1 << K) - (1 << k) + t, ch = child_slot(K, k, pp);
      gW[ch] = gW[L + pp] + gW[ch];
      gW[ch + 1] = gW[L + pp] + gW[ch + 1];
    }
    __syncthreads();
  }
  if (t < L) grad_v[t] = Wt[t] > 0.0 ? gW[t] : 0.0;
}

__global__ void k_amsgrad(int64_t n, double *x, const double *g, double *m, double *s, double *smax, double lr,
                          double b1, double b2, double eps, double c1, double c2) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    m[i] = b1 * m[i] + (1.0 - b1) * g[i];
    s[i] = b2 * s[i] + (1.0 - b2) * g[i] * g[i];
    smax[i] = fmax(smax[i], s[i]);
    x[i] -= lr * (m[i] / c1) / (sqrt(smax[i] / c2) + eps);
  }
}

dmn_status lin_fail(const char *msg) {
  set_error_message(msg);
  return DMN_ERR_ARG;
}

dmn_status lin_cuda(cudaError_t e, const char *what) {
  char msg[256];
  snprintf(msg, sizeof(msg), "%s: %s", what, cudaGetErrorString(e));
  set_error_message(msg);
  return DMN_ERR_CUDA;
}

// grid of a persistent launch: resident CTAs on every SM, at most n
template <typename Kern>
cudaError_t lin_grid(Kern f, int threads, size_t smem, int64_t n, int *grid) {
  int dev = 0, sms = 0, per = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem))) != cudaSuccess)
    return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f, threads, smem)) != cudaSuccess) return e;
  if (per < 1) return cudaErrorInvalidConfiguration;
  const int64_t g = std::min<int64_t>(int64_t(sms) * per, n);
  *grid = int(std::max<int64_t>(g, 1));
  return cudaSuccess;
}

const char *lin_check(int32_t K, int64_t n, const double *C1, const double *C2, const double *normals,
                      const double *v, int32_t precision) {
  if (K < 1 || K > kLinMaxK) return "K must be 1..8";
  if (n < 0) return "n_samples < 0";
  if (n > 0 && (!C1 || !C2 || !normals || !v)) return "NULL pointer";
  if (precision != DMN_LIN_FP64 && precision != DMN_LIN_FP32) return "unknown precision";
  return nullptr;
}

template <typename T>
dmn_status lin_forward(cudaStream_t st, int K, int64_t n, const double *C1, const double *C2,
                       const double *normals, const double *v, double *Cbar) {
  const size_t smem = sizeof(T) * lin_layout(K).words;
  const int threads = 1 << (K - 1);
  int grid = 0;
  cudaError_t e = lin_grid(k_lin_forward<T>, threads, smem, n, &grid);
  if (e != cudaSuccess) return lin_cuda(e, "dmn_linear: launch configuration");
  k_lin_forward<T><<<grid, threads, smem, st>>>(K, n, C1, C2, normals, v, Cbar);
  if ((e = cudaGetLastError()) != cudaSuccess) return lin_cuda(e, "dmn_linear: forward launch");
  return DMN_OK;
}

// the training pass: forward by levels, errors, batch reduction, seed,
// backward by levels; NS and GA in the workspace
template <typename T>
dmn_status lin_train_pass(cudaStream_t st, int K, int64_t n, const double *C1, const double *C2,
                          const double *Ct, const double *normals, const double *v, double p, double q,
                          double penalty, double *err, double *scal, double *loss, T *consts, T *PH, T *NS, T *GA,
                          double *gnh, double *gc1, double *grad_n, double *grad_v) {
  const unsigned nb = unsigned((n + kLvlThreads - 1) / kLvlThreads);
  if (nb > 2147483647u) return lin_fail("dmn_linear_loss_grad: batch too large");
  const int N = (1 << K) - 1;
  T *nh = consts, *c1s = consts + 3 * N;
  const unsigned ns = unsigned((n + kSetupThreads / 2 - 1) / (kSetupThreads / 2));
  cudaError_t e = cudaSuccess;
  // Up to 2,048 samples the error and seed kernels take eight lanes a sample
  // (general powers, K = 5, 2,048 samples: 205 us a step, 560 with one), and a small
  // batch's launches overlap: its kernels last little longer than their launch (with
  // the lanes 107 -> 93 us at K = 8, 32 samples).  Where a batch fills the chip, early
  // CTAs of the next launch keep out those of the one that runs.  Steps that overlap
  // against steps that do not, us:
  //   FP32, p = 1, 2: 512 samples at K = 3, 5, 8 84, 107, 131 to 105, 119, 142; 2,048
  //     95, 114, 165 to 106, 123, 167; 4,096 101, 135, 205 to 105, 122, 204
  //   FP64: 512 at K = 3, 5 209, 316 to 223, 332, 64 at K = 8 438 to 462; but 1,024 at K = 5
  //     394 to 331, 512 at K = 6 416 to 384, 256 at K = 8 613 to 539
  //   general powers, FP32: 768 at K = 3 181 to 191, 512 at K = 5 201 to 207, 64 at K = 8
  //     197 to 206; but 2,048 at K = 3 273 to 191, 256 and 2,048 at K = 8 314 to 228, 616 to 251
  // So by the bottom laminates (256 warps of them), and for exact powers in FP32 up
  // to 2,048 samples whatever the depth.
  const bool lanes8 = n <= 2048;
  const int mode = pow_mode(p);
  const bool few = (n << (K - 1)) <= 8192;
  const bool overlap = mode == 0 ? few && n < 1024 : (sizeof(T) == 4 ? n <= 2048 : few && n <= 2048);
  const bool split = n <= kLvlThreads;  // a block of samples: at most 2^(K-2) CTAs a launch
  auto go = [&](auto f, dim3 grid, unsigned threads, auto... args) {
    if (e == cudaSuccess) e = launch_chained(overlap, f, grid, dim3(threads), 0, st, args...);
  };
  go(k_lvl_setup<T>, dim3(2 + ns), kSetupThreads, K, n, normals, v, C1, C2, nh, c1s, PH, gnh, 4 * N + 5);
  // FP32: pairs of levels from the bottom (FP64 laminates: 251 registers for one
  // level, and bound by the FP64 pipe, so one level a launch)
  int k = K;
  if constexpr (sizeof(T) == 4)
    for (; k >= 2; k -= 2) {
      const auto f = split ? (k == K ? k_lvl_fwd2s<true, T> : k_lvl_fwd2s<false, T>)
                           : (k == K ? k_lvl_fwd2<true, T> : k_lvl_fwd2<false, T>);
      go(f, dim3(nb, 1u << (k - 2)), split ? 2 * kLvlThreads : kLvlThreads, K, k - 1, n, PH, nh, c1s, NS);
    }
  for (; k >= 1; --k) go(k_lvl_fwd<T>, dim3(nb, 1u << (k - 1)), kLvlThreads, K, k, n, PH, nh, c1s, NS);
  // the blocks' partial sums: in the adjoints' array, free until the seed, from an 8-byte boundary
  double *part = reinterpret_cast<double *>((reinterpret_cast<uintptr_t>(GA) + 7) & ~uintptr_t(7));
  if (lanes8) {  // at most 128 CTAs
    const unsigned nb8 = unsigned((8 * n + kLvlThreads - 1) / kLvlThreads);
    go(mode == 1 ? k_lvl_err<1, 8, T> : mode == 2 ? k_lvl_err<2, 8, T> : k_lvl_err<0, 8, T>, dim3(nb8), kLvlThreads,
       K, n, NS, Ct, p, q, err, part, scal);
    go(mode == 1 ? k_lvl_seed<1, 8, T> : mode == 2 ? k_lvl_seed<2, 8, T> : k_lvl_seed<0, 8, T>, dim3(nb8 + 1),
       kLvlThreads, K, n, NS, Ct, p, q, err, v, penalty, scal, loss, GA);
  } else {
    go(mode == 1 ? k_lvl_err<1, 1, T> : mode == 2 ? k_lvl_err<2, 1, T> : k_lvl_err<0, 1, T>, dim3(nb), kLvlThreads,
       K, n, NS, Ct, p, q, err, part, scal);
    go(mode == 1 ? k_lvl_seed<1, 1, T> : mode == 2 ? k_lvl_seed<2, 1, T> : k_lvl_seed<0, 1, T>, dim3(nb + 1),
       kLvlThreads, K, n, NS, Ct, p, q, err, v, penalty, scal, loss, GA);
  }
  // the same pairs, root first
  k = 1;
  if constexpr (sizeof(T) == 4) {
    if (K & 1) {
      go(k_lvl_bwd<T>, dim3(nb, 1), kLvlThreads, K, 1, n, PH, nh, c1s, NS, GA, gnh, gc1);
      k = 2;
    }
    for (; k < K; k += 2) {
      const auto f = split ? (k + 1 == K ? k_lvl_bwd2s<true, T> : k_lvl_bwd2s<false, T>)
                           : (k + 1 == K ? k_lvl_bwd2<true, T> : k_lvl_bwd2<false, T>);
      go(f, dim3(nb, 1u << (k - 1)), split ? 2 * kLvlThreads : kLvlThreads, K, k, n, PH, nh, c1s, NS, GA, gnh, gc1);
    }
  }
  for (; k <= K; ++k) go(k_lvl_bwd<T>, dim3(nb, 1u << (k - 1)), kLvlThreads, K, k, n, PH, nh, c1s, NS, GA, gnh, gc1);
  go(k_lin_finish, dim3(1), kSetupThreads, K, normals, v, penalty, gnh, gc1, scal, grad_n, grad_v);
  if (e != cudaSuccess) return lin_cuda(e, "dmn_linear_loss_grad: launch");
  return DMN_OK;
}

}  // namespace
}  // namespace dmn

using namespace dmn;

extern "C" dmn_status dmn_linear_forward(dmn_stream stream, int32_t K, int64_t n_samples, const double *d_C1,
                                         const double *d_C2, const double *d_normals, const double *d_v,
                                         double *d_Cbar, int32_t precision) {
  set_error_message("");
  if (const char *why = lin_check(K, n_samples, d_C1, d_C2, d_normals, d_v, precision)) return lin_fail(why);
  if (n_samples > 0 && !d_Cbar) return lin_fail("dmn_linear_forward: NULL output");
  if (n_samples == 0) return DMN_OK;
  cudaStream_t st = (cudaStream_t)stream;
  return precision == DMN_LIN_FP64
             ? lin_forward<double>(st, K, n_samples, d_C1, d_C2, d_normals, d_v, d_Cbar)
             : lin_forward<float>(st, K, n_samples, d_C1, d_C2, d_normals, d_v, d_Cbar);
}

extern "C" dmn_status dmn_linear_loss_grad(dmn_stream stream, int32_t K, int64_t n_samples, const double *d_C1,
                                           const double *d_C2, const double *d_Ctarget, const double *d_normals,
                                           const double *d_v, double p, double q, double penalty,
                                           double *d_loss, double *d_grad_n, double *d_grad_v, double *d_work,
                                           int32_t precision) {
  set_error_message("");
  if (const char *why = lin_check(K, n_samples, d_C1, d_C2, d_normals, d_v, precision)) return lin_fail(why);
  if (n_samples < 1) return lin_fail("dmn_linear_loss_grad: needs at least one sample");
  if (!d_Ctarget || !d_loss || !d_grad_n || !d_grad_v || !d_work)
    return lin_fail("dmn_linear_loss_grad: NULL pointer");
  if (!(p >= 1.0) || !(q >= 1.0) || !std::isfinite(p) || !std::isfinite(q) || !(penalty >= 0.0) ||
      !std::isfinite(penalty))
    return lin_fail("dmn_linear_loss_grad: p, q >= 1 and penalty >= 0 required");
  cudaStream_t st = (cudaStream_t)stream;
  const int N = (1 << K) - 1;
  double *err = d_work, *gnh = d_work + n_samples, *gc1 = gnh + 3 * N, *scal = gc1 + N;
  double *consts = scal + 8, *nodes = consts + 4 * N;
  const int64_t cells = int64_t(21) * N * n_samples, ph = int64_t(42) * n_samples;
  if (precision == DMN_LIN_FP64)
    return lin_train_pass<double>(st, K, n_samples, d_C1, d_C2, d_Ctarget, d_normals, d_v, p, q, penalty, err, scal,
                                  d_loss, consts, nodes, nodes + ph, nodes + ph + cells, gnh, gc1, d_grad_n,
                                  d_grad_v);
  float *f = reinterpret_cast<float *>(nodes);
  return lin_train_pass<float>(st, K, n_samples, d_C1, d_C2, d_Ctarget, d_normals, d_v, p, q, penalty, err, scal,
                               d_loss, reinterpret_cast<float *>(consts), f, f + ph, f + ph + cells, gnh, gc1,
                               d_grad_n, d_grad_v);
}

extern "C" dmn_status dmn_linear_amsgrad(dmn_stream stream, int64_t n_params, double *d_params,
                                         const double *d_grad, double *d_m, double *d_s, double *d_smax, double lr,
                                         double beta1, double beta2, double eps, int64_t step) {
  set_error_message("");
  if (n_params < 0 || step < 1) return lin_fail("dmn_linear_amsgrad: n_params >= 0 and step >= 1 required");
  if (n_params == 0) return DMN_OK;
  if (!d_params || !d_grad || !d_m || !d_s || !d_smax) return lin_fail("dmn_linear_amsgrad: NULL pointer");
  if (!(beta1 >= 0.0 && beta1 < 1.0) || !(beta2 >= 0.0 && beta2 < 1.0) || !(eps > 0.0) || !std::isfinite(lr))
    return lin_fail("dmn_linear_amsgrad: 0 <= beta < 1, eps > 0 required");
  const double c1 = 1.0 - std::pow(beta1, double(step)), c2 = 1.0 - std::pow(beta2, double(step));
  const int blocks = int(std::min<int64_t>((n_params + 255) / 256, 1024));
  k_amsgrad<<<blocks, 256, 0, (cudaStream_t)stream>>>(n_params, d_params, d_grad, d_m, d_s, d_smax, lr, beta1,
                                                      beta2, eps, c1, c2);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return lin_cuda(e, "dmn_linear_amsgrad launch");
  return DMN_OK;
}
