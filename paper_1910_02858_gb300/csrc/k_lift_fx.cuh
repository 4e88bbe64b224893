// Lifting and volume integral of the FP64 form with the line contractions in block
// fixed point (fx.cuh).  Standard volume integral, BR1.
//
// The FP64 body (lift_vol_body) is bound by the FP64 pipe: of its 850 FP64 instructions
// per node (n = 8, Gauss) 480 are D_hat multiply-adds, 90 lifting face terms, 90 gradient
// prolongation and 90 metric products.  All of those are sums of products under one scale
// and run here on the integer pipes; the FP64 pipe keeps the primitive variables, the
// surface terms' means and the pointwise fluxes.  16^3 elements, N = 7: 3.06 -> 1.37 ms;
// curved 24^3: 10.4 -> 4.55 ms.  Elements whose values leave the fixed-point range
// (above 2^200, infinities, NaN) take the FP64 body.
#pragma once
#include "fx.cuh"

namespace flexi {

// slots of an element's magnitude table
enum { FX_W = 0, FX_J = 5, FX_S = 8, FX_Q = 9, FX_F = 24, FX_SLOTS = 32 };
// largest exponent field that the fixed-point kernel takes: the products of four such
// values stay inside the FP64 range; larger values, infinities and NaN go to the FP64 body
constexpr int FX_MAX_EXP = 1022 + 200;

// the FP64 body as a function of its own, for elements outside the fixed-point range
template <int n, bool LGL>
__device__ __noinline__ void lift_vol_fp64(const double* U, const double* Ja, const double* sJ, const double* Wf,
                                           const double* fgeo, const int* elemSide, double* Gf, double* Utv,
                                           double* Gvol, int K, int S, int bigBase, const double* QB,
                                           const Ops<double>& ops, const Phys<double>& ph) {
  lift_vol_body<double, n, 0, LGL, 0, false>(U, Ja, sJ, Wf, fgeo, elemSide, Gf, Utv, Gvol, K, S, bigBase, QB, ops, ph);
}

template <int n>
constexpr size_t lift_fx_smem() {
  using C = Cfg<n>;
  return 8 * (C::NE * 30 * C::n3p + C::NE * 90 * C::n2) + sizeof(int) * C::NE * (12 + 6 * C::n2 + FX_SLOTS + 16);
}

// CTAs per SM asked of the register allocator: what the shared memory allows (n = 8, 7: one)
template <int n>
constexpr int lift_fx_min_blocks() { return n >= 7 ? 1 : (n == 6 ? 2 : (n == 5 ? 4 : 6)); }

template <int n, bool LGL>
__global__ void __launch_bounds__(Cfg<n>::T, lift_fx_min_blocks<n>()) k_lift_vol_fx(
    const double* __restrict__ U, const double* __restrict__ Ja, const double* __restrict__ sJ,
    const double* __restrict__ Wf, const double* __restrict__ fgeo, const int* __restrict__ elemSide,
    double* __restrict__ Gf, double* __restrict__ Utv, double* __restrict__ Gvol, int K, int S, int bigBase,
    const double* __restrict__ QB, const __grid_constant__ Ops<double> ops, const __grid_constant__ FxOps fx,
    const __grid_constant__ Phys<double> ph) {
  using C = Cfg<n>;
  constexpr int n2 = C::n2, n3 = C::n3, NE = C::NE, T = C::T, n3p = C::n3p, P = C::P;
  constexpr bool kWarp = NE == 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fx64* sA = reinterpret_cast<fx64*>(smem_raw);  // [NE][15][n3p] staged fields
  fx64* sB = sA + NE * 15 * n3p;                 // [NE][15][n3p] contraction results
  fx64* sQ = sB + NE * 15 * n3p;                 // [NE][6][15][n2] lifting surface terms (v*3+d)
  int* sES = reinterpret_cast<int*>(sQ + NE * 90 * n2);
  int* sSlot = sES + NE * 6;
  int* sMpq = sSlot + NE * 6;            // [NE][6][n2]
  int* sMag = sMpq + NE * 6 * n2;        // [NE][FX_SLOTS] largest magnitude words
  int* sExp = sMag + NE * FX_SLOTS;      // [NE][16] exponent bound of lifting field v*3+d
  const int tid = threadIdx.x;
  const int el = tid / n3, node = tid - el * n3;
  const int e0 = blockIdx.x * NE, e = e0 + el;
  const bool valid = e < K;
  const int i = node % n, j = (node / n) % n, k = node / n2;
  const int pn = pidx<n>(i, j, k);
  const unsigned wmask = (tid | 31) < T ? 0xffffffffu : (1u << (T & 31)) - 1u;

  for (int t = tid; t < NE * FX_SLOTS; t += T) sMag[t] = 0;
  for (int t = tid; t < NE * 6; t += T) {
    const int es = (e0 + t / 6 < K) ? elemSide[(size_t)e0 * 6 + t] : 0;
    sES[t] = es;
    sSlot[t] = es_slave(es) * S + es_side(es);
  }
  double W[NV], jac[9], sj;
  {
    double Uo[NV] = {1.0, 0.0, 0.0, 0.0, 1.0};
    if (valid) {
#pragma unroll
      for (int v = 0; v < NV; ++v) Uo[v] = U[((size_t)e * NV + v) * n3 + node];
    }
#pragma unroll
    for (int c = 0; c < 9; ++c) jac[c] = valid ? Ja[((size_t)e * 9 + c) * n3 + node] : 0.0;
    sj = valid ? sJ[(size_t)e * n3 + node] : 0.0;
    cons_to_prim(Uo, W, ph);
  }
  __syncthreads();
  int* mag = sMag + el * FX_SLOTS;
#pragma unroll
  for (int v = 0; v < NV; ++v) fx_max<kWarp>(mag + FX_W + v, fx_mag(W[v]), wmask);
#pragma unroll
  for (int d = 0; d < 3; ++d)
    fx_max<kWarp>(mag + FX_J + d, max(fx_mag(jac[d]), max(fx_mag(jac[3 + d]), fx_mag(jac[6 + d]))), wmask);
  fx_max<kWarp>(mag + FX_S, fx_mag(sj), wmask);
  // a2: BR1 surface terms Q = U* n_d s_hat (br1_surface_terms) with their largest magnitudes
  {
    double* Qd = reinterpret_cast<double*>(sQ);
    int mx[15];
#pragma unroll
    for (int c = 0; c < 15; ++c) mx[c] = 0;
    for (int it = tid; it < NE * 6 * n2; it += T) {
      const int el2 = it / (6 * n2);
      const int r = it - el2 * 6 * n2;
      const int s = r / n2, pq = r - s * n2;
      double q[15];
      if (e0 + el2 < K) {
        const int es = sES[el2 * 6 + s];
        const int side = es_side(es);
        const int mpq = orient_pq(es_orient(es), n - 1, pq % n, pq / n);
        sMpq[it] = mpq;
        const double* w0 = Wf + ((size_t)side * NV) * n2 + mpq;
        const double* w1 = Wf + ((size_t)(S + side) * NV) * n2 + mpq;
        const double* g = fgeo + ((size_t)side * 4) * n2 + mpq;
        if (side >= bigBase) {
          const double* qb = QB + ((size_t)(side - bigBase) * 15) * n2 + mpq;
#pragma unroll
          for (int c = 0; c < 15; ++c) q[c] = qb[c * n2];
        } else {
          const double sc = dg_neg_if(0.5 * g[3 * n2], es_slave(es));
          const double nd[3] = {g[0] * sc, g[n2] * sc, g[2 * n2] * sc};
#pragma unroll
          for (int v = 0; v < NV; ++v) {
            const double ws = w0[v * n2] + w1[v * n2];
#pragma unroll
            for (int d = 0; d < 3; ++d) q[v * 3 + d] = ws * nd[d];
          }
        }
      } else {
#pragma unroll
        for (int c = 0; c < 15; ++c) q[c] = 0.0;
      }
#pragma unroll
      for (int c = 0; c < 15; ++c) {
        Qd[((el2 * 6 + s) * 15 + c) * n2 + pq] = q[c];
        if constexpr (kWarp)
          mx[c] = max(mx[c], fx_mag(q[c]));
        else
          atomicMax(sMag + el2 * FX_SLOTS + FX_Q + c, fx_mag(q[c]));
      }
    }
    if constexpr (kWarp) {
#pragma unroll
      for (int c = 0; c < 15; ++c) fx_max<true>(mag + FX_Q + c, mx[c], wmask);
    }
  }
  __syncthreads();
  {
    int bad = 0;
    for (int t = tid; t < NE * FX_SLOTS; t += T) bad |= (sMag[t] >> 20) > FX_MAX_EXP;
    for (int t = tid; t < NE * 15; t += T) {
      const int el2 = t / 15, c = t - el2 * 15;
      const int* m = sMag + el2 * FX_SLOTS;
      sExp[el2 * 16 + c] = max((m[FX_W + c / 3] >> 20) + (m[FX_J + c % 3] >> 20) - 2044, (m[FX_Q + c] >> 20) - 1022);
    }
    if (__syncthreads_or(bad)) {
      lift_vol_fp64<n, LGL>(U, Ja, sJ, Wf, fgeo, elemSide, Gf, Utv, Gvol, K, S, bigBase, QB, ops, ph);
      return;
    }
  }
  // surface terms, metric terms, 1/J and the primitive variables to fixed point
  for (int it = tid; it < NE * 90 * n2; it += T) {
    const int el2 = NE == 1 ? 0 : it / (90 * n2);
    const int c = (it / n2) % 15;
    sQ[it] = fx_shr(fx_from(__longlong_as_double(sQ[it]), sExp[el2 * 16 + c] + 1022), 3);
  }
  FxSplit wi[NV], ji[9];
#pragma unroll
  for (int v = 0; v < NV; ++v) wi[v] = fx_split(fx_from(W[v], mag[FX_W + v] >> 20));
#pragma unroll
  for (int c = 0; c < 9; ++c) ji[c] = fx_split(fx_from(jac[c], mag[FX_J + c % 3] >> 20));

  // a3: per reference direction l, Ja^l_d W_v staged as field d*5 + v and contracted along l
  const int* ex = sExp + el * 16;
#pragma unroll
  for (int l = 0; l < 3; ++l) {
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int sh = 3 + ex[v * 3 + d] - ((mag[FX_W + v] >> 20) + (mag[FX_J + d] >> 20) - 2044);
        sA[(el * 15 + d * NV + v) * n3p + pn] = fx_shr(fx_mul(ji[l * 3 + d], wi[v]), min(sh, 62));
      }
    __syncthreads();
    constexpr int L = NE * 15 * n2;
    const int stride = l == 0 ? 1 : (l == 1 ? P : P * n);
#pragma unroll 1
    for (int it = tid; it < L; it += T) {
      const int f = it / n2, line = it - f * n2;  // f = element * 15 + d * 5 + v
      const int el2 = NE == 1 ? 0 : f / 15;
      const int c = f - el2 * 15, d = c / NV, v = c - d * NV;
      const int a0 = line % n, a1 = line / n;
      const int base = f * n3p + (l == 0 ? P * line : (l == 1 ? a0 + P * n * a1 : a0 + P * a1));
      fx64 x[n];
#pragma unroll
      for (int a = 0; a < n; ++a) x[a] = sA[base + a * stride];
      const fx64* q = sQ + ((el2 * 6 + 2 * l) * 15 + v * 3 + d) * n2 + line;
      fx_line<n, LGL, true>(x, q[0], q[15 * n2], fx, [&](int ii, fx64 y) {
        fx64* dst = sB + base + ii * stride;
        *dst = l == 0 ? y : *dst + y;
      });
    }
    __syncthreads();
  }
  // dW_v/dx_d = (sum) / J
  const int ES = mag[FX_S] >> 20;
  double G[15];
  {
    const FxSplit si = fx_split(fx_from(sj, ES));
#pragma unroll
    for (int c = 0; c < 15; ++c) {
      const fx64 g = fx_mul(fx_split(sB[(el * 15 + c) * n3p + pn] >> fx.rsh), si);
      G[c] = fx_to(g, ex[(c % NV) * 3 + c / NV] - 57 + fx.cE + fx.rsh + ES - 1022);
      sA[(el * 15 + c) * n3p + pn] = LGL ? __double_as_longlong(G[c]) : fx_shr(g, 1);
    }
  }
  if (Gvol != nullptr && valid) {
#pragma unroll
    for (int c = 0; c < 15; ++c) Gvol[((size_t)e * 15 + c) * n3 + node] = G[c];
  }
  __syncthreads();
  // a4: gradients to the faces, both ends of every line
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    const int stride = l == 0 ? 1 : (l == 1 ? P : P * n);
#pragma unroll 1
    for (int it = tid; it < NE * 15 * n2; it += T) {
      const int f = it / n2, line = it - f * n2;
      const int el2 = NE == 1 ? 0 : f / 15;
      const int c = f - el2 * 15;
      if (e0 + el2 >= K) continue;
      const int a0 = line % n, a1 = line / n;
      const fx64* b = sA + f * n3p + (l == 0 ? P * line : (l == 1 ? a0 + P * n * a1 : a0 + P * a1));
      double gm, gp;
      if constexpr (LGL) {
        gm = __longlong_as_double(b[0]);
        gp = __longlong_as_double(b[(n - 1) * stride]);
      } else {
        fx64 x[n], ym, yp;
#pragma unroll
        for (int a = 0; a < n; ++a) x[a] = b[a * stride];
        fx_ends<n>(x, fx, ym, yp);
        const int t = sExp[el2 * 16 + (c % NV) * 3 + c / NV] - 57 + fx.cE + fx.rsh + (sMag[el2 * FX_SLOTS + FX_S] >> 20) -
                      1022 + 1 + fx.pE + 2;
        gm = fx_to(ym, t);
        gp = fx_to(yp, t);
      }
      const int fc = el2 * 6 + 2 * l;
      Gf[((size_t)sSlot[fc] * 15 + c) * n2 + sMpq[fc * n2 + line]] = gm;
      Gf[((size_t)sSlot[fc + 1] * 15 + c) * n2 + sMpq[(fc + 1) * n2 + line]] = gp;
    }
  }
  // a6: physical fluxes in FP64, contravariant fluxes in fixed point
  double* sF = reinterpret_cast<double*>(sB) + el * 15 * n3p + pn;  // the thread's own entries
  {
    double Uo[NV] = {1.0, 0.0, 0.0, 0.0, 1.0};
    if (valid) {
#pragma unroll
      for (int v = 0; v < NV; ++v) Uo[v] = U[((size_t)e * NV + v) * n3 + node];
    }
    int mx[NV] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      double F[NV];
      flux_total(Uo, W, G, d, ph, F);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        sF[(d * NV + v) * n3p] = F[v];
        mx[v] = max(mx[v], fx_mag(F[v]));
      }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) fx_max<kWarp>(mag + FX_F + v, mx[v], wmask);
  }
  __syncthreads();
  {
    int bad = 0;
    for (int t = tid; t < NE * NV; t += T) bad |= (sMag[(t / NV) * FX_SLOTS + FX_F + t % NV] >> 20) > 1022 + 600;
    if (__syncthreads_or(bad)) {
      lift_vol_fp64<n, LGL>(U, Ja, sJ, Wf, fgeo, elemSide, Gf, Utv, Gvol, K, S, bigBase, QB, ops, ph);
      return;
    }
  }
  const int EJ[3] = {mag[FX_J] >> 20, mag[FX_J + 1] >> 20, mag[FX_J + 2] >> 20};
  const int EJm = max(EJ[0], max(EJ[1], EJ[2]));
  {
    FxSplit F[15];
#pragma unroll
    for (int c = 0; c < 15; ++c) F[c] = fx_split(fx_from(sF[c * n3p], mag[FX_F + c % NV] >> 20));
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      FxSplit a[3];
#pragma unroll
      for (int d = 0; d < 3; ++d)
        a[d] = fx_split((((fx64)ji[l * 3 + d].h << 30) + ji[l * 3 + d].l) >> min(EJm - EJ[d], 63));
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        fx64 hh = 0, mid = (1ll << 29) + 3 * (1ll << 28);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          hh += (fx64)a[d].h * F[d * NV + v].h;
          mid += (fx64)a[d].h * F[d * NV + v].l;
          mid += (fx64)a[d].l * F[d * NV + v].h;
        }
        sA[(el * 15 + l * NV + v) * n3p + pn] = fx_shr(hh + (mid >> 30), 4);
      }
    }
  }
  __syncthreads();
  // a7: volume integral, the three directions into separate results
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    const int stride = l == 0 ? 1 : (l == 1 ? P : P * n);
#pragma unroll 1
    for (int it = tid; it < NE * NV * n2; it += T) {
      const int el2 = NE == 1 ? 0 : it / (NV * n2);
      const int r = it - el2 * NV * n2;
      const int v = r / n2, line = r - v * n2;
      const int a0 = line % n, a1 = line / n;
      const int base = (el2 * 15 + l * NV + v) * n3p + (l == 0 ? P * line : (l == 1 ? a0 + P * n * a1 : a0 + P * a1));
      fx64 x[n];
#pragma unroll
      for (int a = 0; a < n; ++a) x[a] = sA[base + a * stride];
      fx_line<n, LGL, false>(x, 0, 0, fx, [&](int ii, fx64 y) { sB[base + ii * stride] = y; });
    }
  }
  __syncthreads();
  if (valid) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const fx64* r = sB + (el * 15 + v) * n3p + pn;
      Utv[((size_t)e * NV + v) * n3 + node] = fx_to(r[0] + r[NV * n3p] + r[2 * NV * n3p],
                                                    (mag[FX_F + v] >> 20) + EJm - 2044 - 56 + fx.cE);
    }
  }
}

}  // namespace flexi
