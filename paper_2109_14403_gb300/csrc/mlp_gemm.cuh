// mlp_gemm.cuh -- BF16 tensor-core GEMMs for the warm-start MLP on sm_103a: FP32
// accumulation in tensor memory, a fused epilogue.  C[M x N] = A[M x K] . B[N x K]^T
// with K contiguous; the tile form also takes an operand with M or N contiguous
// (the backward pass's, as stored).
//
// Two forms, chosen by gemm() in mlp.cu.  The persistent wide form (below,
// gemm_bf16_tn_wide: 128 x 256 tiles) serves inference and plain products of N a
// multiple of 256 with tiles enough for the SMs; the tile form serves everything
// else: other N (a multiple of 128), small products, and all of a training step.
// Tile form: one CTA of 128 threads computes a tile of 128 rows and 128 columns from
// a ring of three stages, or of 64 columns from four (short products and the
// weight gradients); grid: column tiles fastest; two CTAs share an SM, so one's
// epilogue overlaps the other's MMAs:
//   warp 0, lane 0  loads A and B tiles (64 wide in K) with TMA bulk tensor
//                   copies into the ring of 128-byte-swizzled shared memory,
//                   signalled by mbarriers with transaction counts;
//   warp 1          allocates a TMEM column per tile column; its lane 0 issues
//                   tcgen05.mma (kind::f16, BF16 x BF16 -> F32, M = 128, the
//                   tile's N, K = 16 per instruction) and releases each stage with
//                   tcgen05.commit on that stage's "empty" mbarrier;
//   all 4 warps     wait for the final commit, read the accumulator with
//                   tcgen05.ld (warp w owns TMEM lanes 32w..32w+31 = tile rows)
//                   and run the epilogue.  The de-normalised FP32 prediction
//                   (rows of an odd length) goes through the then idle
//                   operand ring: each warp stages its 32 rows and writes
//                   them row by row, the lanes on consecutive columns.
// Every wait is bounded (about two seconds of SM clock): on a timeout the CTA
// records an error code, stops issuing work, frees its TMEM and returns.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pdl.cuh"

namespace dmn {
namespace mlp {

constexpr int BM = 128, BN = 128, BK = 64, STAGES = 3;
constexpr int TILE_A = BM * BK * 2, TILE_B = BN * BK * 2;  // bytes per stage
constexpr int GEMM_SMEM = STAGES * (TILE_A + TILE_B) + 1024 + 256;
constexpr long long kWaitCycles = 4000000000ll;  // ~2 s at 2 GHz

enum Epi {
  EPI_BIAS_SILU = 0,  // z = acc + bias -> Z (bf16, optional), H = silu(z) (bf16)
  EPI_BIAS_F32 = 1,   // (acc + bias) * scale + shift -> fp32 on valid rows and columns
  EPI_DSILU = 2,      // dz = acc * silu'(z_in) -> dZ (bf16)
  EPI_F32 = 3,        // plain fp32 store
  EPI_LOSS = 4        // d = acc + bias - target on valid rows and columns, 0 elsewhere:
                      // dZ = 2 d gscale (bf16), sum d^2 of each warp -> loss_part (tile form)
};

struct EpiArgs {
  int mode;
  int ldc;                     // leading dimension of row-major outputs (= N)
  const float *bias;           // [N]
  __nv_bfloat16 *z_out;        // [M x ldc]
  __nv_bfloat16 *h_out;        // [M x ldc]
  const __nv_bfloat16 *z_in;   // [M x ldc] pre-activation for silu'
  float *f_out;                // [M x ldc] fp32 output
  const float *scale, *shift;  // [N] de-normalisation (EPI_BIAS_F32, optional)
  const float *target;         // [m_valid x ldc] (EPI_LOSS), 16-byte aligned
  float gscale;                // EPI_LOSS: 1 / (rows x columns of the mean)
  float *loss_part;            // EPI_LOSS: one per warp of every tile
  int m_valid, n_valid;        // valid rows / columns (EPI_BIAS_F32, EPI_LOSS)
  int ld_f;                    // leading dimension of f_out
  int *err;                    // error code (0 = fine)
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait on an mbarrier phase
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try(bar, parity))
    if (clock64() - t0 > kWaitCycles) return false;
  return true;
}
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar,
                                            int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}
// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (tcgen05 descriptor version 1)
__device__ __forceinline__ uint64_t sdesc_sw128(const void *tile) {
  const uint64_t a = smem_u32(tile);
  return ((a & 0x3FFFFull) >> 4) | (1ull << 16) | (uint64_t(1024 >> 4) << 32) | (1ull << 46) |
         (2ull << 61);
}
// instruction descriptor: D f32, A and B bf16, both K-major, N and M
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(N >> 3) << 17) | (uint32_t(M >> 4) << 24);
}
__device__ __forceinline__ void umma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc,
                                     uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// the logistic function; the quotient with the fast reciprocal (a few FP32
// ulp), which the bf16 rounding of every result that uses it hides
__device__ __forceinline__ float sigmoidf_(float z) { return __fdividef(1.0f, 1.0f + __expf(-z)); }

// two 16-column accumulator loads in flight, one wait
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float v[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]),
        "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
        "=r"(r[30]), "=r"(r[31])
      : "r"(taddr + 16u));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// The epilogue of 16 accumulator columns n..n+15 of output row r, every mode
// but the staged de-normalised prediction (EPI_BIAS_F32 with scale)
__device__ __forceinline__ void epi_chunk16(const EpiArgs &ep, int r, int n, const float v[16]) {
  if (ep.mode == EPI_BIAS_SILU) {
    __align__(16) __nv_bfloat16 zb[16], hb[16];
    __align__(16) float bb[16];  // the chunk's biases, four vector loads (n is a multiple of 16)
#pragma unroll
    for (int q = 0; q < 4; ++q) reinterpret_cast<float4 *>(bb)[q] = reinterpret_cast<const float4 *>(ep.bias + n)[q];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float z = v[i] + bb[i];
      zb[i] = __float2bfloat16(z);
      hb[i] = __float2bfloat16(z * sigmoidf_(z));
    }
    if (ep.z_out) {
      uint4 *zo = reinterpret_cast<uint4 *>(ep.z_out + size_t(r) * ep.ldc + n);
      zo[0] = reinterpret_cast<uint4 *>(zb)[0];
      zo[1] = reinterpret_cast<uint4 *>(zb)[1];
    }
    uint4 *ho = reinterpret_cast<uint4 *>(ep.h_out + size_t(r) * ep.ldc + n);
    ho[0] = reinterpret_cast<uint4 *>(hb)[0];
    ho[1] = reinterpret_cast<uint4 *>(hb)[1];
  } else if (ep.mode == EPI_DSILU) {
    __align__(16) __nv_bfloat16 db[16], zi[16];
    const uint4 *zp = reinterpret_cast<const uint4 *>(ep.z_in + size_t(r) * ep.ldc + n);
    reinterpret_cast<uint4 *>(zi)[0] = zp[0];
    reinterpret_cast<uint4 *>(zi)[1] = zp[1];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float z = __bfloat162float(zi[i]);
      const float sg = sigmoidf_(z);
      db[i] = __float2bfloat16(v[i] * sg * (1.0f + z * (1.0f - sg)));
    }
    uint4 *dout = reinterpret_cast<uint4 *>(ep.h_out + size_t(r) * ep.ldc + n);
    dout[0] = reinterpret_cast<uint4 *>(db)[0];
    dout[1] = reinterpret_cast<uint4 *>(db)[1];
  } else {  // EPI_F32
    float4 *fo = reinterpret_cast<float4 *>(ep.f_out + size_t(r) * ep.ldc + n);
#pragma unroll
    for (int q = 0; q < 4; ++q) fo[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  }
}

// EPI_LOSS of 16 columns of row r; returns the sum of squares
__device__ __forceinline__ float epi_loss16(const EpiArgs &ep, int r, int n, const float v[16]) {
  __align__(16) __nv_bfloat16 g[16];
  __align__(16) float tg[16], bb[16];
  const bool rv = r < ep.m_valid;
  float part = 0.0f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    reinterpret_cast<float4 *>(bb)[q] = reinterpret_cast<const float4 *>(ep.bias + n)[q];
    reinterpret_cast<float4 *>(tg)[q] =
        rv ? __ldcs(reinterpret_cast<const float4 *>(ep.target + size_t(r) * ep.ldc + n) + q) : float4{};
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float d = rv && n + i < ep.n_valid ? v[i] + bb[i] - tg[i] : 0.0f;
    part += d * d;
    g[i] = __float2bfloat16(2.0f * d * ep.gscale);
  }
  uint4 *o = reinterpret_cast<uint4 *>(ep.h_out + size_t(r) * ep.ldc + n);
  o[0] = reinterpret_cast<uint4 *>(g)[0];
  o[1] = reinterpret_cast<uint4 *>(g)[1];
  return part;
}

// Shared-memory descriptor of an operand whose M or N index is contiguous in
// memory (MN-major, 128-byte swizzle): blocks of 64 of that index (128 bytes)
// by the step's K rows; eight rows are a 1024-byte swizzle atom (stride
// offset), the next 64 of the index follow BK rows later (leading offset).
__device__ __forceinline__ uint64_t sdesc_mn_sw128(const void *tile) {
  const uint64_t a = smem_u32(tile);
  return ((a & 0x3FFFFull) >> 4) | (uint64_t((BK * 128) >> 4) << 16) | (uint64_t(1024 >> 4) << 32) | (1ull << 46) |
         (2ull << 61);
}

// Tile form.  AMN / BMN: the operand is given with M (N) contiguous, [K x M]
// ([K x N]); the tensor core takes it that way, so that the backward pass
// needs no transposed copies: dW = dZ^T . X with both operands as the batch's
// rows, dX = dZ . W with W as stored.  BNT columns and NST stages: 128 and 3, or 64
// and 4 for short products and the weight gradients (gemm_bf16_wgrad), two CTAs
// per SM.
constexpr int WG_BN = 64, WG_ST = 4;  // the narrow tile
__host__ __device__ constexpr int tile_smem(int bnt, int nst) { return nst * (TILE_A + bnt * BK * 2) + 1024 + 256; }
static_assert(tile_smem(BN, STAGES) == GEMM_SMEM && 2 * (tile_smem(WG_BN, WG_ST) + 1024) <= 228 * 1024, "shared memory");
template <bool AMN, bool BMN, int BNT, int NST>
__device__ __forceinline__ void gemm_tile_body(const CUtensorMap &map_a, const CUtensorMap &map_b, int K,
                                               const EpiArgs &ep, int bx, int by) {
  extern __shared__ __align__(1024) unsigned char gsm[];
  unsigned char *base = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(gsm) + 1023) & ~uintptr_t(1023));
  unsigned char *sa = base;                         // NST x TILE_A
  constexpr int TB = BNT * BK * 2;
  unsigned char *sb = base + NST * TILE_A;          // NST x TB
  uint64_t *full = reinterpret_cast<uint64_t *>(sb + NST * TB);
  uint64_t *empty = full + NST;
  uint64_t *done = empty + NST;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
  int *fail = reinterpret_cast<int *>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // column tiles fastest: the CTAs that share an A panel run together and
  // read it from L2 (the A panel of a 65,536-row batch is larger than L2)
  const int m0 = by * BM, n0 = bx * BNT;
  const int nk = K / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    *fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(uint32_t(BNT)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {  // ---- TMA producer ----
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % NST;
      if (kb >= NST && !mbar_wait(&empty[s], ((kb / NST) - 1) & 1)) {
        atomicExch(fail, 1);
        break;
      }
      if (*(volatile int *)fail) break;
      mbar_expect_tx(&full[s], TILE_A + TB);
      const int k0 = kb * BK;
      if (AMN) {  // blocks of 64 along M (N)
        tma_load_2d(sa + s * TILE_A, &map_a, &full[s], m0, k0);
        tma_load_2d(sa + s * TILE_A + BK * 128, &map_a, &full[s], m0 + 64, k0);
      } else {
        tma_load_2d(sa + s * TILE_A, &map_a, &full[s], k0, m0);
      }
      if (BMN) {
#pragma unroll
        for (int b = 0; b < BNT / 64; ++b)
          tma_load_2d(sb + s * TB + b * BK * 128, &map_b, &full[s], n0 + 64 * b, k0);
      } else {
        tma_load_2d(sb + s * TB, &map_b, &full[s], k0, n0);
      }
    }
  } else if (warp == 1 && lane == 0) {  // ---- MMA issuer ----
    const uint32_t idesc = idesc_bf16(BM, BNT) | (AMN ? 1u << 15 : 0u) | (BMN ? 1u << 16 : 0u);
    int kb = 0;
    for (; kb < nk; ++kb) {
      const int s = kb % NST;
      if (!mbar_wait(&full[s], (kb / NST) & 1)) {
        atomicExch(fail, 1);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint64_t ad = AMN ? sdesc_mn_sw128(sa + s * TILE_A) : sdesc_sw128(sa + s * TILE_A);
      const uint64_t bd = BMN ? sdesc_mn_sw128(sb + s * TB) : sdesc_sw128(sb + s * TB);
      // 16 of K per step: 32 bytes inside the swizzle atom, or 16 rows of 128 bytes
#pragma unroll
      for (int k = 0; k < BK / 16; ++k)
        umma(tmem, ad + (AMN ? 128 : 2) * k, bd + (BMN ? 128 : 2) * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
      umma_commit(&empty[s]);
    }
    umma_commit(done);  // arrives once all issued MMAs have completed
  }
  __syncwarp();
  // ---- epilogue: all 4 warps ----
  bool ok = mbar_wait(done, 0);
  // the epilogue's tcgen05.ld is warp-synchronous: decide CTA-wide
  ok = __syncthreads_and(ok && *(volatile int *)fail == 0);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!ok && threadIdx.x == 0 && ep.err) atomicExch(ep.err, 1);
  if (ok) {
    const int r = m0 + warp * 32 + lane;  // tile row owned by this thread
    const uint32_t trow = tmem + (uint32_t(warp * 32) << 16);
    float part = 0.0f;
    for (int c0 = 0; c0 < BNT; c0 += 16) {
      float v[16];
      tmem_ld16(trow + c0, v);
      const int n = n0 + c0;
      if (ep.mode == EPI_BIAS_F32) {  // staged: the ring holds no operands once `done` has fired
        float *srow = reinterpret_cast<float *>(base) + (warp * 32 + lane) * (BNT + 1);
#pragma unroll
        for (int i = 0; i < 16; ++i) srow[c0 + i] = v[i];
      } else if (ep.mode == EPI_LOSS) {
        part += epi_loss16(ep, r, n, v);
      } else {
        epi_chunk16(ep, r, n, v);
      }
    }
    if (ep.mode == EPI_LOSS) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
      if (lane == 0) ep.loss_part[(by * int(gridDim.x) + bx) * 4 + warp] = part;
    }
    if (ep.mode == EPI_BIAS_F32) {
      // de-normalised prediction on valid rows and columns: the warp writes
      // its 32 staged rows, lane l on columns l, l + 32, ..
      static_assert(BM * (BNT + 1) * 4 <= NST * (TILE_A + TB), "staged FP32 tile fits the ring");
      constexpr int NC = BNT / 32;
      __syncwarp();
      const float *tile = reinterpret_cast<const float *>(base);
      float bb[NC], sc[NC], sh[NC];
      bool cv[NC];
#pragma unroll
      for (int q = 0; q < NC; ++q) {
        const int n = n0 + lane + 32 * q;
        cv[q] = n < ep.n_valid;
        bb[q] = cv[q] ? ep.bias[n] : 0.0f;
        sc[q] = cv[q] ? ep.scale[n] : 0.0f;
        sh[q] = cv[q] ? ep.shift[n] : 0.0f;
      }
      for (int rr = 0; rr < 32; ++rr) {
        const int row = warp * 32 + rr, rg = m0 + row;
        if (rg >= ep.m_valid) break;
        float *dst = ep.f_out + size_t(rg) * ep.ld_f + n0 + lane;
#pragma unroll
        for (int q = 0; q < NC; ++q)
          if (cv[q]) dst[32 * q] = (tile[row * (BNT + 1) + lane + 32 * q] + bb[q]) * sc[q] + sh[q];
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(uint32_t(BNT)));
  }
}

template <bool AMN, bool BMN, int BNT, int NST>
__global__ void __launch_bounds__(128, 2)
    gemm_bf16_tile(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                   int K, const EpiArgs ep) {
  chain_begin();
  gemm_tile_body<AMN, BMN, BNT, NST>(map_a, map_b, K, ep, blockIdx.x, blockIdx.y);
}

// The weight gradients of every layer, dW_l = dZ_l^T . X_l, in one launch: each
// is a few tiles that run through the whole batch (16 to 28 of 128 x 128 at 512
// hidden units: 30 us a layer on that many SMs), together (128 x 64: 168 tiles)
// they fill the chip.  Each output stays one chain of MMAs over the batch, the
// order of its roundings.
// The bias gradients (column sums of dZ_l) and the loss read what these tiles
// read, so they are blocks of the same launch, behind the tiles in the slots
// that 168 tiles leave free on 152 SMs (as a kernel of their own after them: a step
// of 4,096 rows 191.6 us, now 180.2).
constexpr int kMaxLayers = 9;
struct WgradArgs {
  CUtensorMap a[kMaxLayers], b[kMaxLayers];  // dZ_l [K x M_l], X_l [K x N_l]
  int layers, blk0[kMaxLayers + 1], nx[kMaxLayers], ldc[kMaxLayers];
  float *out[kMaxLayers];
  int *err;
  int cblk0[kMaxLayers + 1], cols[kMaxLayers];  // column sums: first block (after the tiles) and columns of each layer
  const __nv_bfloat16 *dz[kMaxLayers];
  float *db[kMaxLayers];
  int nloss;  // the loss: partial sums, their number and scale (loss NULL: no block)
  const float *loss_part;
  float *loss, lscale;
};
static_assert(sizeof(WgradArgs) <= 4000, "kernel parameters");

// Column sums of dz [rows x C] (rows a multiple of 32), 32 columns from c0 on:
// 16 lanes of two columns, each thread four of 32 row classes (rows r mod 32,
// one chain each), then the classes pairwise.
constexpr int CS_COLS = 32;
__device__ __forceinline__ void colsum_body(const __nv_bfloat16 *dz, int C, int rows, int c0, float *db,
                                            float2 (*red)[16]) {
  const int x = threadIdx.x & 15, g = threadIdx.x >> 4;
  const __nv_bfloat16 *p = dz + c0 + 2 * x;
  float2 s[4] = {};
#pragma unroll 8
  for (int r = g; r < rows; r += 32)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 v =
          __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p + size_t(r + 8 * k) * C));
      s[k].x += v.x;
      s[k].y += v.y;
    }
#pragma unroll
  for (int k = 0; k < 4; ++k) red[g + 8 * k][x] = s[k];
  __syncthreads();
  for (int o = 16; o > 0; o >>= 1) {
    for (int q = g; q < o; q += 8) {
      red[q][x].x += red[q + o][x].x;
      red[q][x].y += red[q + o][x].y;
    }
    __syncthreads();
  }
  if (g == 0) *reinterpret_cast<float2 *>(db + c0 + 2 * x) = red[0][x];
}
// The loss: the sum of the tiles' partial sums in FP64, 32 rows of 32 lanes in a
// fixed order
__device__ __forceinline__ void loss_body(const float *part, int n, float scale, float *loss, double *rl) {
  const int lane = threadIdx.x & 31;
  for (int w = threadIdx.x >> 5; w < 32; w += 4) {
    double s = 0.0;
    for (int i = 32 * w + lane; i < n; i += 1024) s += double(part[i]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) rl[w] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = rl[0];
    for (int w = 1; w < 32; ++w) s += rl[w];
    *loss = float(s * double(scale));
  }
}
__global__ void __launch_bounds__(128, 2) gemm_bf16_wgrad(const __grid_constant__ WgradArgs A, int K) {
  extern __shared__ __align__(1024) unsigned char gsm[];
  chain_begin();
  int l = 0, q = int(blockIdx.x);
  if (q >= A.blk0[A.layers]) {
    q -= A.blk0[A.layers];
    if (q >= A.cblk0[A.layers]) {
      loss_body(A.loss_part, A.nloss, A.lscale, A.loss, reinterpret_cast<double *>(gsm));
      return;
    }
    while (q >= A.cblk0[l + 1]) ++l;
    colsum_body(A.dz[l], A.cols[l], K, (q - A.cblk0[l]) * CS_COLS, A.db[l], reinterpret_cast<float2(*)[16]>(gsm));
    return;
  }
  while (q >= A.blk0[l + 1]) ++l;
  q -= A.blk0[l];
  EpiArgs ep = {};
  ep.mode = EPI_F32;
  ep.f_out = A.out[l];
  ep.ldc = A.ldc[l];
  ep.err = A.err;
  gemm_tile_body<true, true, WG_BN, WG_ST>(A.a[l], A.b[l], K, ep, q % A.nx[l], q / A.nx[l]);
}

// ---------------------------------------------------------------- wide form
// Persistent form for N a multiple of 256 (inference: the network's layers have N
// = 512 or 768): one CTA per SM loops over 128 x 256 tiles (column tiles
// fastest, so the CTAs sharing an A panel run together and read it from L2).
// Warps with fixed roles:
//   warp 0, lane 0  TMA producer: A (128 x 64) and B (256 x 64) of each K step
//                   into a 3-stage ring (48 KB per stage);
//   warp 1          allocates all 512 TMEM columns (two 256-column FP32
//                   accumulators); its lane 0 issues tcgen05.mma (M = 128,
//                   N = 256, K = 16) and commits each stage to its "empty"
//                   barrier and each finished tile to its accumulator's
//                   "full" barrier;
//   warps 2..17     the epilogue, four warps per TMEM lane quarter: warp w
//                   reads lanes 32 (w % 4).. (tile rows) of one quarter of the
//                   columns with tcgen05.ld, the next 32 columns in flight
//                   while it works on 32, releases the accumulator ("empty",
//                   one arrival per warp) as soon as its last columns are in
//                   registers, so the MMAs of the next tile run into the other
//                   accumulator meanwhile, and applies the fused epilogue.
// The epilogue bounds the hidden layers: SiLU takes two special-function
// operations an element, 4096 cycles of a 128 x 256 tile, as long as its MMAs at
// K = 512, so it needs warps enough to keep them busy (eight warps: 50 us a
// layer of 65,536 rows, mostly waiting for TMEM and for its own row-strided
// stores; now 38, the output layer 94 -> 76) and stores that cost nothing: bf16 rows go through shared memory (32
// rows x 64 columns a warp, 128-byte swizzle) and out by TMA.  The de-normalised
// FP32 prediction (rows of an odd length: no TMA) is staged as 32 rows x 32
// columns and written a row at a time, the lanes on consecutive columns.  Every
// wait is bounded as in the form above.
// LONG, for long reductions (K >= 2048: a tile's MMAs take four times its
// epilogue) and plain FP32 output: the staging's memory is a fourth stage instead,
// and eight warps of 128 columns store directly (the prediction through 32 x 17
// floats a warp, two rows at a time).  8,192^3: 876 -> 772 us; inference of 65,536
// rows with 4,096 hidden units 3,449 -> 3,285 (1,024 units, which stay: 470, 460 this
// way; 16,384 rows of them 157, 166).  FP32 rows leave as whole 32-byte sectors: half
// a sector an instruction, merged or not as the warps happen to run, took 217 to
// 247 us at 65,536 x 2,048 x 512; now 190.
constexpr int WBN = 256;
constexpr int WTILE_B = WBN * BK * 2;
constexpr int WSTAGE = TILE_A + WTILE_B;  // 48 KB, a multiple of 1024
__host__ __device__ constexpr int wide_stages(bool lng) { return lng ? 4 : 3; }
__host__ __device__ constexpr int wide_epi(bool lng) { return lng ? 8 : 16; }  // epilogue warps
__host__ __device__ constexpr int wide_threads(bool lng) { return 64 + 32 * wide_epi(lng); }
// staging per epilogue warp: 32 rows of 128 bytes, or of 17 floats
__host__ __device__ constexpr int wide_stage_epi(bool lng) { return wide_epi(lng) * (lng ? 32 * 17 * 4 : 4096); }
__host__ __device__ constexpr int wide_smem(bool lng) {
  return wide_stages(lng) * WSTAGE + wide_stage_epi(lng) + 1024 + 256;
}
static_assert(wide_smem(false) <= 232448 && wide_smem(true) <= 232448, "opt-in shared memory per CTA");

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// 32 accumulator columns in flight; tmem_wait makes them readable
__device__ __forceinline__ void tmem_issue32(uint32_t taddr, uint32_t r[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,"
      "%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]),
        "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
        "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait(uint32_t r[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                 "+r"(r[29])
               :
               : "memory");
  asm volatile("" : "+r"(r[30]), "+r"(r[31])::"memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, const void *src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(src)), "r"(x), "r"(y)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// eight floats to a 32-byte boundary: one whole sector a lane
__device__ __forceinline__ void st_sector(float *p, const float v[8]) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}

// Modes EPI_BIAS_SILU without z_out (map_h: its bf16 output, [M x N], boxes of
// 32 rows x 64 columns; unused in the others) and EPI_BIAS_F32; LONG: the same and
// EPI_F32, map_h unused.
template <bool LONG>
__global__ void __launch_bounds__(wide_threads(LONG), 1)
    gemm_bf16_tn_wide(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                      const __grid_constant__ CUtensorMap map_h, int M, int N, int K, const EpiArgs ep) {
  extern __shared__ __align__(1024) unsigned char gsm[];
  unsigned char *base = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(gsm) + 1023) & ~uintptr_t(1023));
  constexpr int WST = wide_stages(LONG), WEPI = wide_epi(LONG);
  unsigned char *stage_epi = base + WST * WSTAGE;
  uint64_t *full = reinterpret_cast<uint64_t *>(stage_epi + wide_stage_epi(LONG));
  uint64_t *empty = full + WST;
  uint64_t *accf = empty + WST;  // 2: accumulator full (MMA -> epilogue)
  uint64_t *acce = accf + 2;     // 2: accumulator empty (epilogue -> MMA)
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acce + 2);
  int *fail = reinterpret_cast<int *>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ntn = N / WBN, ntiles = (M / BM) * ntn, nk = K / BK;

  if (threadIdx.x == 0) {
    for (int st = 0; st < WST; ++st) {
      mbar_init(&full[st], 1);
      mbar_init(&empty[st], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], WEPI);
    }
    *fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {  // ---- TMA producer ----
      int it = 0;
      for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int m0 = (t / ntn) * BM, n0 = (t % ntn) * WBN;
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int st = it % WST;
          if (it >= WST && !mbar_wait(&empty[st], ((it / WST) - 1) & 1)) {
            atomicExch(fail, 1);
            break;
          }
          if (*(volatile int *)fail) break;
          mbar_expect_tx(&full[st], WSTAGE);
          tma_load_2d(base + st * WSTAGE, &map_a, &full[st], kb * BK, m0);
          tma_load_2d(base + st * WSTAGE + TILE_A, &map_b, &full[st], kb * BK, n0);
        }
        if (*(volatile int *)fail) break;
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ---- MMA issuer ----
      const uint32_t idesc = idesc_bf16(BM, WBN);
      int it = 0, j = 0;
      for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++j) {
        const int b = j & 1;
        if (j >= 2 && !mbar_wait(&acce[b], ((j >> 1) - 1) & 1)) {
          atomicExch(fail, 1);
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc = tmem + uint32_t(b * WBN);
        bool bad = false;
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int st = it % WST;
          if (!mbar_wait(&full[st], (it / WST) & 1)) {
            atomicExch(fail, 1);
            bad = true;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t ad = sdesc_sw128(base + st * WSTAGE), bd = sdesc_sw128(base + st * WSTAGE + TILE_A);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k)
            umma(acc, ad + 2 * k, bd + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
          umma_commit(&empty[st]);
        }
        if (bad) break;
        umma_commit(&accf[b]);  // arrives once this tile's MMAs have completed
      }
    }
  } else if constexpr (LONG) {  // ---- epilogue: warps 2..9 ----
    const int qd = warp & 3;  // TMEM lane quarter = tile rows 32 qd ..
    constexpr int CW = WBN / (WEPI / 4);  // this warp's columns ch0 .. ch0 + CW - 1
    const int ch0 = ((warp - 2) >> 2) * CW;
    float *stg = reinterpret_cast<float *>(stage_epi) + (warp - 2) * 32 * 17;
    const bool row32 = !(reinterpret_cast<uintptr_t>(ep.f_out) & 31);
    int j = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++j) {
      const int b = j & 1;
      const bool ok = mbar_wait(&accf[b], (j >> 1) & 1);
      if (!__all_sync(0xffffffffu, ok) || *(volatile int *)fail) {
        if (lane == 0) atomicExch(fail, 1);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int m0 = (t / ntn) * BM + qd * 32, n0 = (t % ntn) * WBN;
      const uint32_t trow = tmem + (uint32_t(qd * 32) << 16) + uint32_t(b * WBN);
      if (ep.mode == EPI_F32 && row32) {
        float *fo = ep.f_out + size_t(m0 + lane) * ep.ldc + n0 + ch0;
#pragma unroll
        for (int h = 0; h < CW; h += 16) {
          float v[16];
          tmem_ld16(trow + ch0 + h, v);
#pragma unroll
          for (int q = 0; q < 2; ++q) st_sector(fo + h + 8 * q, v + 8 * q);
        }
      } else if (ep.mode == EPI_BIAS_F32) {
        for (int c0 = ch0; c0 < ch0 + CW; c0 += 16) {
          float v[16];
          tmem_ld16(trow + c0, v);
#pragma unroll
          for (int i = 0; i < 16; ++i) stg[lane * 17 + i] = v[i];
          __syncwarp();
          // lanes 0..15 on row rr, 16..31 on row rr + 1, consecutive columns
          const int cl = lane & 15, n = n0 + c0 + cl;
          const bool cv = n < ep.n_valid;
          const float bb = cv ? ep.bias[n] : 0.0f, sc = cv ? ep.scale[n] : 0.0f, sh = cv ? ep.shift[n] : 0.0f;
          for (int rr = lane >> 4; rr < 32; rr += 2)
            if (cv && m0 + rr < ep.m_valid)
              ep.f_out[size_t(m0 + rr) * ep.ld_f + n] = (stg[rr * 17 + cl] + bb) * sc + sh;
          __syncwarp();
        }
      } else {
        for (int c0 = ch0; c0 < ch0 + CW; c0 += 32) {
          float v[32];
          tmem_ld32(trow + c0, v);
          epi_chunk16(ep, m0 + lane, n0 + c0, v);
          epi_chunk16(ep, m0 + lane, n0 + c0 + 16, v + 16);
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&acce[b]);
    }
  } else {  // ---- epilogue: warps 2..17 ----
    const int qd = warp & 3;
    constexpr int CW = WBN / (WEPI / 4);
    static_assert(CW == 64, "two 32-column chunks, one 128-byte row of bf16");
    const int ch0 = ((warp - 2) >> 2) * CW;
    unsigned char *stg = stage_epi + (warp - 2) * 4096;
    float *stf = reinterpret_cast<float *>(stg);
    const bool act = ep.mode == EPI_BIAS_SILU;  // else EPI_BIAS_F32
    int j = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++j) {
      const int b = j & 1;
      const bool ok = mbar_wait(&accf[b], (j >> 1) & 1);
      if (!__all_sync(0xffffffffu, ok) || *(volatile int *)fail) {
        if (lane == 0) atomicExch(fail, 1);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int m0 = (t / ntn) * BM + qd * 32, n0 = (t % ntn) * WBN + ch0;
      const uint32_t trow = tmem + (uint32_t(qd * 32) << 16) + uint32_t(b * WBN + ch0);
      uint32_t acc[2][32];
      tmem_issue32(trow, acc[0]);
      tmem_wait(acc[0]);
      tmem_issue32(trow + 32u, acc[1]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h == 1) {
          tmem_wait(acc[1]);
          // the accumulator is read: hand it back before working on it
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&acce[b]);
        }
        float v[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(acc[h][i]);
        const int n = n0 + 32 * h;
        if (act) {
          if (h == 0) {  // the last tile's rows have left the staging buffer
            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {  // 8 columns: one 16-byte unit of the swizzled row
            const float4 b0 = __ldg(reinterpret_cast<const float4 *>(ep.bias + n) + 2 * q);
            const float4 b1 = __ldg(reinterpret_cast<const float4 *>(ep.bias + n) + 2 * q + 1);
            const float bb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
            __align__(16) __nv_bfloat162 hb[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float z0 = v[8 * q + 2 * i] + bb[2 * i], z1 = v[8 * q + 2 * i + 1] + bb[2 * i + 1];
              hb[i] = __floats2bfloat162_rn(z0 * sigmoidf_(z0), z1 * sigmoidf_(z1));
            }
            *reinterpret_cast<uint4 *>(stg + lane * 128 + (((4 * h + q) ^ (lane & 7)) << 4)) =
                *reinterpret_cast<uint4 *>(hb);
          }
        } else {
          // de-normalised prediction on valid rows and columns; column c of row
          // r in slot c ^ r of the row
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 32; ++i) stf[lane * 32 + (i ^ lane)] = v[i];
          __syncwarp();
          const int nc = n + lane;
          const bool cv = nc < ep.n_valid;
          const float bb = cv ? ep.bias[nc] : 0.0f, sc = cv ? ep.scale[nc] : 0.0f, sh = cv ? ep.shift[nc] : 0.0f;
          float *dst = ep.f_out + size_t(m0) * ep.ld_f + nc;
          const int rows = ep.m_valid - m0 < 32 ? ep.m_valid - m0 : 32;
          if (rows == 32 && cv) {
#pragma unroll 8
            for (int rr = 0; rr < 32; ++rr) dst[size_t(rr) * ep.ld_f] = (stf[rr * 32 + (lane ^ rr)] + bb) * sc + sh;
          } else if (cv) {
            for (int rr = 0; rr < rows; ++rr) dst[size_t(rr) * ep.ld_f] = (stf[rr * 32 + (lane ^ rr)] + bb) * sc + sh;
          }
        }
      }
      if (act) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) tma_store_2d(&map_h, stg, n0, m0);
      }
    }
    if (act && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
  }
  __syncwarp();  // lanes 1..31 of the producer and MMA warps wait for lane 0 here
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && *(volatile int *)fail && ep.err) atomicExch(ep.err, 1);
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
  }
}

}  // namespace mlp
}  // namespace dmn
