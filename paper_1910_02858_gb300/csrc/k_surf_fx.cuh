// Prolongation and surface/RK kernels of the FP64 form with their contractions in block
// fixed point (fx.cuh).
//
// k_surf spends 60 of its 87 FP64 instructions per node (n = 8, Gauss) on the l_hat
// products of the surface integral and the l(+-1) products of the next face states; at 64
// clocks per FP64 warp instruction that is 3.5 times the kernel's memory time.  Here they
// take three integer multiply-adds each; the FP64 pipe keeps the RK update and the
// primitive face states.  16^3 elements, N = 7: k_surf 297 -> 181 us (268 B per node:
// 84 us at the measured copy rate), k_prolong 158 -> 83 us.  Elements with values outside the
// fixed-point range use the FP64 expressions of k_surf.
#pragma once
#include "fx.cuh"

namespace flexi {

// Face states of U for the CTA's elements from sU[el][5][n3p] (FP64, padded lines): values of
// both ends of every line in fixed point into sFace[el][6][5][n2], then W(U_face) to the side
// arrays.  Block-wide; sU and sFace are overwritten; sMag: [NE][NV] slots, zero on entry.
template <int n, bool LGL>
__device__ __forceinline__ void faces_from_volume_fx(double* sU, double* sFace, int* sMag, const Ops<double>& ops,
                                                     const FxOps& fx, const int* sES, int e0, int K, int S,
                                                     double* __restrict__ Wf, const Phys<double>& ph,
                                                     unsigned* __restrict__ status, int tid, unsigned wmask) {
  using C = Cfg<n>;
  constexpr int n2 = C::n2, n3 = C::n3, n3p = C::n3p, P = C::P, NE = C::NE, T = C::T;
  const int el = tid / n3, node = tid - el * n3;
  double* own = sU + el * NV * n3p + pidx<n>(node % n, (node / n) % n, node / n2);
  bool fixed = false;
  if constexpr (!LGL) {
    fx_max<NE == 1, NV>(sMag + el * NV, wmask, [&](int v) { return fx_mag(own[v * n3p]); });
    __syncthreads();
    int bad = 0;
    for (int t = tid; t < NE * NV; t += T) bad |= (sMag[t] >> 20) > 1022 + 900;
    fixed = !__syncthreads_or(bad);
    if (fixed) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
        own[v * n3p] = __longlong_as_double(fx_shr(fx_from<60>(own[v * n3p], sMag[el * NV + v] >> 20), 1));
    }
  }
  __syncthreads();
  // ends of the lines of field f = element * 5 + v along l
#pragma unroll 1
  for (int it = tid; it < NE * 15 * n2; it += T) {
    const int f = it / (3 * n2), r = it - f * 3 * n2;
    const int l = r / n2, line = r - l * n2;
    const int a0 = line % n, a1 = line / n;
    const int stride = l == 0 ? 1 : (l == 1 ? P : P * n);
    const double* b = sU + f * n3p + (l == 0 ? P * line : (l == 1 ? a0 + P * n * a1 : a0 + P * a1));
    double um = 0.0, up = 0.0;
    if constexpr (LGL) {
      um = b[0];
      up = b[(n - 1) * stride];
    } else if (fixed) {
      fx64 ym, yp;
      fx_ends<n>(reinterpret_cast<const fx64*>(b), stride, fx, ym, yp);
      const int t = (sMag[f] >> 20) - 1022 - 59 + 64 - fx.kp;
      um = fx_to(ym, t);
      up = fx_to(yp, t);
    } else {
#pragma unroll 1
      for (int a = 0; a < n; ++a) {
        um = dg_fma(ops.lm[a], b[a * stride], um);
        up = dg_fma(ops.lp[a], b[a * stride], up);
      }
    }
    const int el2 = NE == 1 ? 0 : f / NV;
    const int v = f - el2 * NV;
    double* d = sFace + ((el2 * 6 + 2 * l) * NV + v) * n2 + line;
    d[0] = um;
    d[NV * n2] = up;
  }
  __syncthreads();
  for (int it = tid; it < NE * 6 * n2; it += T) {
    const int f = it / n2, pq = it - f * n2;
    if (e0 + f / 6 >= K) continue;
    double Uf[NV], W[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) Uf[v] = sFace[(f * NV + v) * n2 + pq];
    cons_to_prim(Uf, W, ph);
    if (!(W[0] > 0.0) || !(W[4] > 0.0)) atomicOr(status, 1u);
    const int es = sES[f];
    double* dst = Wf + ((size_t)(es_slave(es) * S + es_side(es)) * NV) * n2 + orient_pq(es_orient(es), n - 1, pq % n, pq / n);
#pragma unroll
    for (int v = 0; v < NV; ++v) dst[v * n2] = W[v];
  }
}

template <int n, bool LGL>
__global__ void __launch_bounds__(Cfg<n>::T, n >= 7 ? 2 : 4) k_prolong_fx(
    const double* __restrict__ U, const int* __restrict__ elemSide, double* __restrict__ Wf, int K, int S,
    const __grid_constant__ Ops<double> ops, const __grid_constant__ FxOps fx, const __grid_constant__ Phys<double> ph,
    unsigned* __restrict__ status) {
  using C = Cfg<n>;
  constexpr int n2 = C::n2, n3 = C::n3, NE = C::NE, T = C::T;
  __shared__ double sU[NE * NV * C::n3p];
  __shared__ double sFace[NE * 6 * NV * n2];
  __shared__ int sES[NE * 6], sMag[NE * NV];
  const int tid = threadIdx.x;
  const int el = tid / n3, node = tid - el * n3;
  const int e0 = blockIdx.x * NE;
  const unsigned wmask = (tid | 31) < T ? 0xffffffffu : (1u << (T & 31)) - 1u;
  for (int t = tid; t < NE * 6; t += T) sES[t] = (e0 + t / 6 < K) ? elemSide[(size_t)e0 * 6 + t] : 0;
  for (int t = tid; t < NE * NV; t += T) sMag[t] = 0;
  double* own = sU + el * NV * C::n3p + pidx<n>(node % n, (node / n) % n, node / n2);
#pragma unroll
  for (int v = 0; v < NV; ++v)
    own[v * C::n3p] = e0 + el < K ? U[((size_t)(e0 + el) * NV + v) * n3 + node] : 1.0;
  __syncthreads();
  faces_from_volume_fx<n, LGL>(sU, sFace, sMag, ops, fx, sES, e0, K, S, Wf, ph, status, tid, wmask);
}

// surface integral, -1/J, RK stage update (MODE 1; MODE 0: U_t) and the face states of the new U.
// Registers are capped for 1024-1536 resident threads: 24^3 curved elements with a source,
// N = 7, 3 CTAs against 2: 865 -> 835 us (696 with the source constants formed on the host)
template <int n, int MODE, bool LGL>
__global__ void __launch_bounds__(Cfg<n>::T, n == 8 ? 3 : (n == 7 ? 4 : (n == 6 ? 6 : 8))) k_surf_fx(
    const double* __restrict__ Ff, const int* __restrict__ elemSide, const double* __restrict__ sJ,
    const double* __restrict__ Utv, double* __restrict__ U, double* __restrict__ dU, double* __restrict__ Ut,
    double* __restrict__ Wf, const double* __restrict__ phase, const RkStage<double> rk, const SourceParams src, int K, int S,
    const __grid_constant__ Ops<double> ops, const __grid_constant__ FxOps fx, const __grid_constant__ Phys<double> ph,
    unsigned* __restrict__ status) {
  using C = Cfg<n>;
  constexpr int n2 = C::n2, n3 = C::n3, NE = C::NE, T = C::T, n3p = C::n3p;
  __shared__ double sF[NE * 6 * NV * n2];
  __shared__ double sU[(MODE == 1) ? NE * NV * n3p : 1];
  __shared__ int sES[NE * 6], sMag[NE * 2 * NV];
  __shared__ int4 sL[n];  // l_hat_i(-1), l_hat_i(+1) in fixed point
  const int tid = threadIdx.x;
  const int el = tid / n3, node = tid - el * n3;
  const int e0 = blockIdx.x * NE, e = e0 + el;
  const bool valid = e < K;
  const int i = node % n, j = (node / n) % n, k = node / n2;
  const unsigned wmask = (tid | 31) < T ? 0xffffffffu : (1u << (T & 31)) - 1u;
  // the node's own values are requested first, so that their latency overlaps the gather
  double vtv[NV], vU[NV], vdU[NV], sj = 0.0;
  if (valid) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const size_t g = ((size_t)e * NV + v) * n3 + node;
      vtv[v] = Utv[g];
      if (MODE == 1) {
        vU[v] = U[g];
        vdU[v] = dU[g];
      }
    }
    sj = sJ[(size_t)e * n3 + node];
  }
  for (int t = tid; t < n; t += T) sL[t] = make_int4(fx.lh[n - 1 - t], fx.ll[n - 1 - t], fx.lh[t], fx.ll[t]);
  for (int t = tid; t < NE * 6; t += T) sES[t] = (e0 + t / 6 < K) ? elemSide[(size_t)e0 * 6 + t] : 0;
  for (int t = tid; t < NE * 2 * NV; t += T) sMag[t] = 0;
  __syncthreads();
  int mx[NV] = {0, 0, 0, 0, 0};
  for (int it = tid; it < NE * 6 * n2; it += T) {
    const int f = it / n2, pq = it - f * n2;
    const bool live = e0 + f / 6 < K;
    const int es = sES[f];
    const double* src_f = Ff + ((size_t)es_side(es) * NV) * n2 + orient_pq(es_orient(es), n - 1, pq % n, pq / n);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double x = live ? dg_neg_if(src_f[v * n2], es_slave(es)) : 0.0;  // the slave side takes -f* s_hat
      sF[(f * NV + v) * n2 + pq] = x;
      if constexpr (NE == 1)
        mx[v] = max(mx[v], fx_mag(x));
      else
        atomicMax(sMag + (f / 6) * 2 * NV + v, fx_mag(x));
    }
  }
  if constexpr (NE == 1) fx_max<true, NV>(sMag, wmask, [&](int v) { return mx[v]; });
  __syncthreads();
  int bad = 0;
  for (int t = tid; t < NE * 2 * NV; t += T) bad |= (sMag[t] >> 20) > 1022 + 900;
  const bool fixed = !__syncthreads_or(bad);
  if (fixed) {
    for (int it = tid; it < NE * 6 * n2; it += T) {  // the thread's own entries, as above
      const int f = it / n2, pq = it - f * n2;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        double* x = sF + (f * NV + v) * n2 + pq;
        *x = __longlong_as_double(fx_from<61>(*x, sMag[(f / 6) * 2 * NV + v] >> 20));
      }
    }
  }
  __syncthreads();
  // ut = U_t (MODE 0) or dt U_t (MODE 1: dt folded into the -1/J factor)
  double ut[NV];
  const int pq0 = j + n * k, pq1 = i + n * k, pq2 = i + n * j;
  const double* Fe = sF + el * 6 * NV * n2;
  const double scale = MODE == 1 ? -(rk.dt * sj) : -sj;
  if (fixed) {
    const int4 L0 = sL[i], L1 = sL[j], L2 = sL[k];
    const fx64* Fx = reinterpret_cast<const fx64*>(Fe);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      fx64 sum = 0;  // two products per accumulator: 62-bit factors leave no room for more
      auto dir = [&](int d, int at, int pq, int4 L) {
        if (LGL && at > 0 && at < n - 1) return;  // Gauss-Lobatto: only nodes on a face receive its flux
        FxAcc a;
        if (!LGL || at == 0) a.add(fx_split(Fx[(2 * d * NV + v) * n2 + pq]), L.x, L.y);
        if (!LGL || at == n - 1) a.add(fx_split(Fx[((2 * d + 1) * NV + v) * n2 + pq]), L.z, L.w);
        sum += a.get();
      };
      dir(0, i, pq0, L0);
      dir(1, j, pq1, L1);
      dir(2, k, pq2, L2);
      ut[v] = (vtv[v] + fx_to(sum, (sMag[el * 2 * NV + v] >> 20) - 1022 + 3 - fx.kl)) * scale;
    }
  } else {
    const double c0 = ops.lhm[i], c1 = ops.lhp[i], c2 = ops.lhm[j], c3 = ops.lhp[j], c4 = ops.lhm[k], c5 = ops.lhp[k];
#pragma unroll 1
    for (int v = 0; v < NV; ++v) {
      double s = v == 0 ? vtv[0] : (v == 1 ? vtv[1] : (v == 2 ? vtv[2] : (v == 3 ? vtv[3] : vtv[4])));
      if (!LGL || i == 0) s = dg_fma(c0, Fe[(0 * NV + v) * n2 + pq0], s);
      if (!LGL || i == n - 1) s = dg_fma(c1, Fe[(1 * NV + v) * n2 + pq0], s);
      if (!LGL || j == 0) s = dg_fma(c2, Fe[(2 * NV + v) * n2 + pq1], s);
      if (!LGL || j == n - 1) s = dg_fma(c3, Fe[(3 * NV + v) * n2 + pq1], s);
      if (!LGL || k == 0) s = dg_fma(c4, Fe[(4 * NV + v) * n2 + pq2], s);
      if (!LGL || k == n - 1) s = dg_fma(c5, Fe[(5 * NV + v) * n2 + pq2], s);
      s *= scale;
#pragma unroll
      for (int w = 0; w < NV; ++w) ut[w] = w == v ? s : ut[w];
    }
  }
  if (src.on && valid) {
    const double* p = phase + (size_t)e * 2 * n3 + node;
    double Sv[NV];
    manufactured_source(p[0], p[n3], src, Sv);
#pragma unroll
    for (int v = 0; v < NV; ++v) ut[v] = dg_fma(MODE == 1 ? rk.dt : 1.0, Sv[v], ut[v]);
  }
  if constexpr (MODE == 0) {
    if (valid) {
#pragma unroll
      for (int v = 0; v < NV; ++v) Ut[((size_t)e * NV + v) * n3 + node] = ut[v];
    }
  } else {
    double* own = sU + el * NV * n3p + pidx<n>(i, j, k);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      double un = 1.0;
      if (valid) {
        const size_t g = ((size_t)e * NV + v) * n3 + node;
        const double du = dg_fma(rk.A, vdU[v], ut[v]);  // A dU + dt U_t
        un = dg_fma(rk.B, du, vU[v]);
        dU[g] = du;
        U[g] = un;
      }
      own[v * n3p] = un;
    }
    if (rk.prolong) {
      __syncthreads();  // the face fluxes are read: sF takes the face values
      for (int t = tid; t < NE * NV; t += T) sMag[t] = 0;
      __syncthreads();
      faces_from_volume_fx<n, LGL>(sU, sF, sMag, ops, fx, sES, e0, K, S, Wf, ph, status, tid, wmask);
    }
  }
}

}  // namespace flexi
