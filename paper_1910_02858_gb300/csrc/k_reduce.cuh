// Global FP64 reductions (Sec. 5.3: the global time step is the only
// all-to-all operation of the method): conserved totals, kinetic energy and its
// rate, and the CFL/DFL rates of Eqs. CFLCondition/DFLCondition evaluated per
// reference direction through the metrics.  Per-block partials (deterministic
// order), summed on the host in FP64.
#pragma once
#include "dg_common.cuh"
#include "launch.h"

namespace flexi {

constexpr int RED_T = 256;
constexpr int RED_Q = 9;  // 5 totals, KE, dKE/dt, max conv rate, max visc rate
constexpr int RED_M = 4;  // nodes per thread between two updates of a block's largest rates

// sum (ops q < 7) or maximum of the threads' values, in a fixed order; result in red[q][0]
__device__ __forceinline__ void reduce_block(double (*red)[RED_T]) {
  for (int s = RED_T / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
#pragma unroll
      for (int q = 0; q < 7; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + s];
      red[7][threadIdx.x] = fmax(red[7][threadIdx.x], red[7][threadIdx.x + s]);
      red[8][threadIdx.x] = fmax(red[8][threadIdx.x], red[8][threadIdx.x + s]);
    }
    __syncthreads();
  }
}

// x truncated to FP32 on the integer pipe (a conversion holds the FP64 pipe for 18 clocks, and
// a node has 17 of them); 0 below and infinity above the FP32 range, NaN stays NaN or infinite
__device__ __forceinline__ float trunc_f32(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = (int)((hi >> 20) & 0x7ff) - 896;
  unsigned m = (hi << 3) | (lo >> 29);  // exponent's low bits and the 23 leading fraction bits
  m = (m & 0x7fffffu) | ((unsigned)e << 23);
  m = e <= 0 ? 0u : (e >= 255 ? ((hi & 0x7fffffffu) > 0x7ff00000u ? 0x7fc00000u : 0x7f800000u) : m);
  return __uint_as_float(m | (hi & 0x80000000u));
}

// The sums need every node in FP64 (about 35 operations); the two rates need only the node
// where they are largest.  They are bounded from both sides in FP32 first (three square
// roots and 30 products), and only nodes whose upper bound reaches the block's largest lower
// bound so far are evaluated in FP64 (100 operations): the maximum is the same value.  The
// last block adds up the blocks' results in block order and puts the status word behind
// them, so that one copy of 10 values reaches the host.  16^3, N = 7, the call: 429 -> 240 us
// with conversions to FP32, 167 us with trunc_f32 (HBM: 53 us).
template <typename real>
__global__ void __launch_bounds__(RED_T, 4) k_reduce(const real* __restrict__ U, const real* __restrict__ Ut,
                                                 const double* __restrict__ wJ, const double* __restrict__ Ja64,
                                                 const double* __restrict__ sJ64, double* __restrict__ partial,
                                                 long long nodes, int n3, Phys<real> ph, double kv_coef,
                                                 const unsigned* __restrict__ status, unsigned* __restrict__ arrived) {
  __shared__ double red[RED_Q][RED_T];
  __shared__ float sLow[2][RED_T / 32];
  __shared__ bool sLast;
  double acc[RED_Q];
#pragma unroll
  for (int q = 0; q < RED_Q; ++q) acc[q] = 0.0;
  const double g = (double)ph.gamma;
  const float kvf = (float)kv_coef;
  // truncation of the inputs (2^-23 each) and rounding of the sums below: each term is within
  // 2^-18 of its magnitude bound
  constexpr float eps = 1.0f / (1 << 18);
  float lowC = 0.0f, lowV = 0.0f;  // largest lower bounds seen by the block
  const long long step = (long long)gridDim.x * RED_T;
  for (long long base = (long long)blockIdx.x * RED_T; base < nodes; base += RED_M * step) {
    float upC[RED_M], upV[RED_M], loC = 0.0f, loV = 0.0f;
#pragma unroll
    for (int m = 0; m < RED_M; ++m) {
      const long long idx = base + m * step + threadIdx.x;
      upC[m] = upV[m] = -1.0f;
      if (idx >= nodes) continue;
      const long long e = idx / n3;
      const int node = (int)(idx - e * n3);
      double u[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) u[v] = (double)U[(e * NV + v) * n3 + node];
      const double w = wJ[idx];
#pragma unroll
      for (int v = 0; v < NV; ++v) acc[v] = dg_fma(w, u[v], acc[v]);
      const double ir = dg_rcp(u[0]);
      const double vel[3] = {u[1] * ir, u[2] * ir, u[3] * ir};
      const double q2 = vel[0] * vel[0] + vel[1] * vel[1] + vel[2] * vel[2];
      const double hq2 = 0.5 * q2;
      acc[5] = dg_fma(w * u[0], hq2, acc[5]);
      if (Ut != nullptr) {
        const real* ut = Ut + e * NV * n3 + node;
        acc[6] = dg_fma(w, vel[0] * (double)ut[n3] + vel[1] * (double)ut[2 * n3] + vel[2] * (double)ut[3 * n3] -
                               hq2 * (double)ut[0], acc[6]);
      }
      const float p = trunc_f32((g - 1.0) * (u[4] - u[0] * hq2));
      const float irf = trunc_f32(ir), vx = trunc_f32(vel[0]), vy = trunc_f32(vel[1]), vz = trunc_f32(vel[2]);
      const float c = sqrtf((float)g * p * irf), va = fabsf(vx) + fabsf(vy) + fabsf(vz) + c;
      const float sj = trunc_f32(sJ64[idx]);
      float lc = 0.0f, lv = 0.0f, big = 0.0f, low = c * c;
      const double* a = Ja64 + e * 9 * n3 + node;
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        const float a0 = trunc_f32(a[(3 * l) * n3]), a1 = trunc_f32(a[(3 * l + 1) * n3]), a2 = trunc_f32(a[(3 * l + 2) * n3]);
        const float s = a0 * a0 + a1 * a1 + a2 * a2, nrm = sqrtf(s);
        low = fminf(low, s);
        lc += fabsf(a0 * vx + a1 * vy + a2 * vz) + c * nrm;
        big += nrm * va;
        lv += (nrm * sj) * (nrm * sj);
      }
      lc *= sj;
      big *= sj * eps;
      lv *= kvf * irf;
      upC[m] = lc + big;
      upV[m] = lv * (1.0f + eps);
      // a bound, or a square in it, that is not well inside the range (or NaN) decides nothing:
      // evaluate the node
      if (!(low > 1e-30f && lc > 1e-30f && upC[m] < 1e30f)) upC[m] = INFINITY;
      else loC = fmaxf(loC, lc - big);
      if (!(low > 1e-30f && lv > 1e-30f && upV[m] < 1e30f)) upV[m] = INFINITY;
      else loV = fmaxf(loV, lv * (1.0f - eps));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      loC = fmaxf(loC, __shfl_xor_sync(0xffffffffu, loC, o));
      loV = fmaxf(loV, __shfl_xor_sync(0xffffffffu, loV, o));
    }
    __syncthreads();  // the previous round's values are read
    if ((threadIdx.x & 31) == 0) {
      sLow[0][threadIdx.x >> 5] = loC;
      sLow[1][threadIdx.x >> 5] = loV;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < RED_T / 32; ++k) {
      lowC = fmaxf(lowC, sLow[0][k]);
      lowV = fmaxf(lowV, sLow[1][k]);
    }
#pragma unroll
    for (int m = 0; m < RED_M; ++m) {
      if (upC[m] < 0.0f || (upC[m] < lowC && upV[m] < lowV)) continue;
      const long long idx = base + m * step + threadIdx.x;
      const long long e = idx / n3;
      const int node = (int)(idx - e * n3);
      double u[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) u[v] = (double)U[(e * NV + v) * n3 + node];
      const double ir = dg_rcp(u[0]), sj = sJ64[idx];
      const double vel[3] = {u[1] * ir, u[2] * ir, u[3] * ir};
      const double* a = Ja64 + e * 9 * n3 + node;
      if (!(upC[m] < lowC)) {
        const double q2 = vel[0] * vel[0] + vel[1] * vel[1] + vel[2] * vel[2];
        const double c = dg_sqrt(g * ((g - 1.0) * (u[4] - 0.5 * u[0] * q2)) * ir);
        double lc = 0.0;
#pragma unroll 1
        for (int l = 0; l < 3; ++l) {
          const double a0 = a[(3 * l) * n3], a1 = a[(3 * l + 1) * n3], a2 = a[(3 * l + 2) * n3];
          lc += fabs(a0 * vel[0] + a1 * vel[1] + a2 * vel[2]) + c * dg_sqrt(a0 * a0 + a1 * a1 + a2 * a2);
        }
        acc[7] = fmax(acc[7], lc * sj);
      }
      if (!(upV[m] < lowV)) {
        double s = 0.0;  // sum of |Ja^l|^2
#pragma unroll 1
        for (int k = 0; k < 9; ++k) s = dg_fma(a[k * n3], a[k * n3], s);
        acc[8] = fmax(acc[8], s * sj * sj * (kv_coef * ir));
      }
    }
  }
#pragma unroll
  for (int q = 0; q < RED_Q; ++q) red[q][threadIdx.x] = acc[q];
  __syncthreads();
  reduce_block(red);
  if (threadIdx.x < RED_Q) partial[(size_t)(1 + blockIdx.x) * RED_Q + 1 + threadIdx.x] = red[threadIdx.x][0];
  __threadfence();
  __syncthreads();
  // the count wraps, so it is 0 again after every launch's blocks, whatever runs beside them
  if (threadIdx.x == 0) sLast = atomicInc(arrived, gridDim.x - 1) == gridDim.x - 1;
  __syncthreads();
  if (!sLast) return;
  __threadfence();
#pragma unroll
  for (int q = 0; q < RED_Q; ++q) {
    double x = 0.0;
    for (int b = threadIdx.x; b < gridDim.x; b += RED_T) {
      const double y = __ldcg(partial + (size_t)(1 + b) * RED_Q + 1 + q);
      x = q < 7 ? x + y : fmax(x, y);
    }
    red[q][threadIdx.x] = x;
  }
  __syncthreads();
  reduce_block(red);
  if (threadIdx.x < RED_Q) partial[threadIdx.x] = red[threadIdx.x][0];
  if (threadIdx.x == 0) partial[RED_Q] = (double)*status;
}

template <typename real>
cudaError_t launch_reduce(const real* U, const real* Ut, const double* wJ, const double* Ja64, const double* sJ64,
                          long long nodes, int n3, const Phys<real>& ph, double kv_coef, double* partial,
                          int nblocks, const unsigned* status, unsigned* arrived, cudaStream_t st) {
  k_reduce<real><<<nblocks, RED_T, 0, st>>>(U, Ut, wJ, Ja64, sJ64, partial, nodes, n3, ph, kv_coef, status, arrived);
  return cudaGetLastError();
}

}  // namespace flexi
