// dmn_drive.cu -- device side of dmn_eval_mixed (include/dmn.h): prescribed
// strain components, and the per-point outer Newton update of the unknown
// strain increments and temperature from the algorithmic tangents that
// Algorithm 1 returns (arXiv 2109.14403, eqs. ddsdde, ddsddt, drplde, drpldt).
#include "dmn_internal.h"

namespace dmn {
namespace {

constexpr int kUpdThreads = 32, kWorkThreads = 128;

// LU with partial pivoting on a 7 x 7 system, in registers (every index is a
// constant after unrolling; rows are exchanged by selects); false when a pivot
// vanishes.  Pivots by the leading 32 bits of the magnitudes (integer
// comparisons; an FP64 instruction takes 64 cycles of a warp here), one
// reciprocal per column: 161 operations and seven divisions a point.  (With the
// system in local memory and a division per row the 4,096-point predictor took
// 44 us.)
template <int k>
__device__ __forceinline__ void lu_column(double A[7][7], double b[7], double inv[7], bool &ok) {
  unsigned best = unsigned(__double2hiint(A[k][k])) & 0x7fffffffu;
  int piv = k;
#pragma unroll
  for (int r = k + 1; r < 7; ++r) {
    const unsigned m = unsigned(__double2hiint(A[r][k])) & 0x7fffffffu;
    piv = m > best ? r : piv;
    best = m > best ? m : best;
  }
#pragma unroll
  for (int r = k + 1; r < 7; ++r) {
    const bool sw = piv == r;
#pragma unroll
    for (int c = k; c < 7; ++c) {
      const double x = A[k][c], y = A[r][c];
      A[k][c] = sw ? y : x;
      A[r][c] = sw ? x : y;
    }
    const double x = b[k], y = b[r];
    b[k] = sw ? y : x;
    b[r] = sw ? x : y;
  }
  ok = ok && best != 0u;
  inv[k] = 1.0 / A[k][k];
#pragma unroll
  for (int r = k + 1; r < 7; ++r) {
    const double f = A[r][k] * inv[k];
#pragma unroll
    for (int c = k + 1; c < 7; ++c) A[r][c] = fma(-f, A[k][c], A[r][c]);
    b[r] = fma(-f, b[k], b[r]);
  }
}
__device__ __forceinline__ bool solve7(double A[7][7], double b[7]) {
  double inv[7];
  bool ok = true;
  lu_column<0>(A, b, inv, ok);
  lu_column<1>(A, b, inv, ok);
  lu_column<2>(A, b, inv, ok);
  lu_column<3>(A, b, inv, ok);
  lu_column<4>(A, b, inv, ok);
  lu_column<5>(A, b, inv, ok);
  lu_column<6>(A, b, inv, ok);
#pragma unroll
  for (int k = 6; k >= 0; --k) {
#pragma unroll
    for (int c = 6; c > 0; --c)
      if (c > k) b[k] = fma(-A[k][c], b[c], b[k]);
    b[k] *= inv[k];
  }
  return ok;
}

// One Newton step on a point's unknowns under mask m: the stress-prescribed
// strain increments (bits 0..5) and theta when adiabatic (bit 6); the others'
// rows and columns are the identity's.  r holds the residuals of the unknowns'
// equations (stress rows, then the heat balance c (theta - theta^n)/dt -
// D_bar), o the outputs whose tangents form the Jacobian.  Adds the step to
// deps / theta; false when the system is singular (nothing changed).
__device__ __forceinline__ bool newton_step(unsigned m, const double *o, double c_heat, double dt,
                                            const double r[7], double *deps, double *theta) {
  double A[7][7], b[7];
#pragma unroll
  for (int a = 0; a < 7; ++a) {
    const bool ua = (m >> a) & 1u;
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      const bool u = ua && ((m >> q) & 1u);
      double v = a == q ? 1.0 : 0.0;
      if (u) {
        if (a < 6) v = q < 6 ? o[6 + 6 * a + q] : o[42 + a];  // d sigma / d eps, d sigma / d theta
        else v = q < 6 ? -o[49 + q] : c_heat / dt - o[55];    // heat balance
      }
      A[a][q] = v;
    }
    b[a] = ua ? -r[a] : 0.0;
  }
  if (!solve7(A, b)) return false;
  bool fin = true;
#pragma unroll
  for (int a = 0; a < 7; ++a) fin = fin && isfinite(b[a]);
  if (!fin) return false;
#pragma unroll
  for (int a = 0; a < 6; ++a)
    if ((m >> a) & 1u) deps[a] += b[a];
  if ((m >> 6) & 1u) *theta += b[6];
  return true;
}

// Prescribed strain components and outer = 0.  With predict, the outputs in
// out are those of the increment that ended in state_in (stress and tangents
// at theta^n); the start is the solution of the linear model they give,
//   sigma ~ sigma^n + C deps + C_theta (theta - theta^n),
//   D ~ D_eps . deps + D_theta (theta - theta^n),
// for the prescribed stresses and the heat balance.
__global__ void __launch_bounds__(kUpdThreads) k_mixed_prepare(int64_t n, int sw, const uint8_t *mask, const double *target,
                                double *deps, double *theta, double dt, double c_heat,
                                const double *sin, const double *out, int predict, int32_t *outer) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x) {
    const unsigned m = mask[i];
    double *e = deps + i * 6;
    const double *tg = target + i * 6;
    for (int c = 0; c < 6; ++c)
      if (!((m >> c) & 1u)) e[c] = tg[c];
    outer[i] = 0;
    if (!predict || (m & 0x7fu) == 0u) continue;
    const double *o = out + i * 57;
    const double thn = sin[i * sw + 6];
    const bool adiabatic = (m >> 6) & 1u;
    double x[6], th = adiabatic ? thn : theta[i];
    for (int c = 0; c < 6; ++c) x[c] = ((m >> c) & 1u) ? 0.0 : tg[c];
    double r[7];
#pragma unroll
    for (int c = 0; c < 7; ++c) {
      double v = 0.0;
      if (c < 6) {
        if ((m >> c) & 1u) {
          v = o[c] - tg[c] + o[42 + c] * (th - thn);
#pragma unroll
          for (int q = 0; q < 6; ++q) v += o[6 + 6 * c + q] * x[q];
        }
      } else if (adiabatic) {
        v = (c_heat / dt - o[55]) * (th - thn);
#pragma unroll
        for (int q = 0; q < 6; ++q) v -= o[49 + q] * x[q];
      }
      r[c] = v;
    }
    if (newton_step(m, o, c_heat, dt, r, x, &th)) {
      for (int c = 0; c < 6; ++c) e[c] = x[c];
      theta[i] = th;
    }
  }
}

// Residuals of the prescribed stresses and of the heat balance at the last
// evaluation; a point that meets them is done (outer = +evaluations), one that
// cannot go on is given up (outer = -evaluations), any other takes one Newton
// step on (unknown deps components, theta) and is counted in *open.  One point
// a thread: a serial FP64 chain, in CTAs of one warp so that a small batch
// spreads over the SMs.
__global__ void __launch_bounds__(kUpdThreads)
    k_mixed_update(int64_t n, int sw, const uint8_t *mask, const double *target, double *deps, double *theta,
                   double dt, double c_heat, double tol, const double *sin, const double *out,
                   const int32_t *status, int32_t *outer, int it, int last, unsigned long long *open) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x) {
    if (outer[i] != 0) continue;  // settled in an earlier evaluation
    const unsigned m = mask[i];
    const double *o = out + i * 57;
    if (status[i] & (DMN_PT_NOT_CONVERGED | DMN_PT_NONFINITE)) {  // Algorithm 1 failed
      outer[i] = -(it + 1);
      continue;
    }
    double smax = 1.0;
    for (int c = 0; c < 6; ++c) smax = fmax(smax, fabs(o[c]));
    double r[7];
    bool ok = true;
#pragma unroll
    for (int c = 0; c < 7; ++c) {
      r[c] = 0.0;
      if (!((m >> c) & 1u)) continue;
      if (c < 6) {
        r[c] = o[c] - target[i * 6 + c];
        if (!(fabs(r[c]) <= tol * smax)) ok = false;
      } else {
        r[c] = c_heat * (theta[i] - sin[i * sw + 6]) / dt - o[48];
        if (!(fabs(r[c]) <= tol * c_heat / dt)) ok = false;
      }
    }
    if (ok) {
      outer[i] = it + 1;
      continue;
    }
    if (last) {
      outer[i] = -(it + 1);
      continue;
    }
    if (!newton_step(m, o, c_heat, dt, r, deps + i * 6, theta + i)) {
      outer[i] = -(it + 1);
      continue;
    }
    atomicAdd(open, 1ull);
  }
}

// The next evaluation's warm-start increment a - a^n of the points still open
// (the solve skips the others), one warp a point, lanes along the jumps: bound
// by its 20 bytes per jump.  (Inside k_mixed_update a thread walked its own
// point's 765 jumps: 360 us at K = 8, 4,096 points, most of them settled.)
__global__ void __launch_bounds__(kWorkThreads)
    k_mixed_work(int64_t n, int sw, int n3, const double *sin, const double *sout, const int32_t *outer,
                 float *work) {
  const int lane = threadIdx.x & 31;
  const int64_t nwarp = (int64_t(gridDim.x) * kWorkThreads) >> 5;
  for (int64_t i = (blockIdx.x * int64_t(kWorkThreads) + threadIdx.x) >> 5; i < n; i += nwarp) {
    if (outer[i] != 0) continue;
    const double *a = sin + i * sw + 8, *b = sout + i * sw + 8;
#pragma unroll 4
    for (int j = lane; j < n3; j += 32) work[i * n3 + j] = float(b[j] - a[j]);
  }
}

// the status bit of the given-up points; outer becomes the evaluation count
__global__ void k_mixed_finish(int64_t n, int32_t *status, int32_t *outer) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x)
    if (outer[i] < 0) {
      status[i] |= DMN_PT_OUTER_NOT_CONVERGED;
      outer[i] = -outer[i];
    }
}

int blocks_for(int64_t n, int threads = 128) {
  int64_t b = (n + threads - 1) / threads;
  return int(b > 65535 ? 65535 : (b < 1 ? 1 : b));
}

}  // namespace

cudaError_t mixed_prepare(cudaStream_t s, int64_t n, int sw, const uint8_t *mask,
                          const double *target, double *deps, double *theta, double dt,
                          double c_heat, const double *sin, const double *out, bool predict,
                          int32_t *outer) {
  k_mixed_prepare<<<blocks_for(n, kUpdThreads), kUpdThreads, 0, s>>>(n, sw, mask, target, deps, theta, dt, c_heat, sin,
                                                out, predict ? 1 : 0, outer);
  return cudaGetLastError();
}

cudaError_t mixed_update(cudaStream_t s, int64_t n, int sw, int n3, const uint8_t *mask,
                         const double *target, double *deps, double *theta, double dt, double c_heat,
                         double tol, const double *sin, const double *sout, const double *out,
                         const int32_t *status, int32_t *outer, int it, bool last, float *work,
                         unsigned long long *open) {
  k_mixed_update<<<blocks_for(n, kUpdThreads), kUpdThreads, 0, s>>>(n, sw, mask, target, deps, theta, dt, c_heat,
                                                                    tol, sin, out, status, outer, it, last ? 1 : 0,
                                                                    open);
  if (work)
    k_mixed_work<<<blocks_for(n * 32, kWorkThreads), kWorkThreads, 0, s>>>(n, sw, n3, sin, sout, outer, work);
  return cudaGetLastError();
}

cudaError_t mixed_finish(cudaStream_t s, int64_t n, int32_t *status, int32_t *outer) {
  k_mixed_finish<<<blocks_for(n), 128, 0, s>>>(n, status, outer);
  return cudaGetLastError();
}

}  // namespace dmn
