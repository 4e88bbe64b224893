// Reverse of the lifting and the volume integral (k_adj_vol) of the FP64 form with its
// contractions in block fixed point (fx.cuh).  Standard volume integral, BR1.
//
// k_adj_vol holds about 900 FP64 instructions per node (n = 6): 60 D_hat^T products, the
// prolongation's and the metric terms' transposes; at 64 clocks each they set its time.  Those sums
// run on the integer pipes here, the pointwise flux derivatives stay in FP64.  Affine
// elements fold the metric constants in before the lifting's transpose (15 line contractions
// instead of 45).  8^3 elements, N = 5: 215 -> 80 us; curved 7 x 9 x 8, N = 6: 349 -> 144 us.
#pragma once
#include "fx.cuh"

namespace flexi {

// slots: lam/J by variable, metric terms by physical direction (nodes and faces), lam_lift and
// face gradient adjoints at d*5+v.  As in volume_fx, a variable's three lam_lift components are
// scaled by direction so that their products with Ja_d meet at the largest of them.
enum { FXA_L = 0, FXA_J = 5, FXA_X = 8, FXA_B = 23, FXA_SLOTS = 38 };

// the FP64 kernel as a function, for elements outside the fixed-point range
template <int n>
__device__ __noinline__ void adj_vol_fp64(const double* U, const double* Ja, const double* sJ, const double* Gvol,
                                          const double* fgeo, const int* elemSide, const double* lam, const double* LGf,
                                          double* LWs, double* LWf, double* muv, int K, int S, int bigBase, double* LQB,
                                          const Ops<double>& ops, const Phys<double>& ph, int grp) {
  __syncthreads();
  adj_vol_body<double, n, false, 0>(U, Ja, sJ, Gvol, fgeo, elemSide, lam, LGf, LWs, LWf, muv, K, S, bigBase, LQB, ops, ph, grp);
}

template <int n>
constexpr size_t adj_fx_smem() {
  using C = Cfg<n>;
  const size_t own = 8 * C::NE * (15 * C::n3p + 90 * C::n2 + 18 * C::n2) + sizeof(int) * C::NE * (6 + 6 * C::n2 + FXA_SLOTS);
  const size_t body = adj_vol_smem<double, n>(false, false);
  return own > body ? own : body;
}

// affine: the metric terms are aff[e][10]; else Ja, fgeo.  n = 7: two CTAs of 343 threads at 80
// registers (160 B spilled) against one at 168: reverse of one right-hand side, 16^3 curved
// elements, 2539 -> 2209 us (2200 with scales by direction)
template <int n, bool AFF>
__global__ void __launch_bounds__(Cfg<n>::T, n == 8 ? 1 : (n == 7 ? 2 : (n == 6 ? 3 : 4))) k_adj_vol_fx(
    const double* __restrict__ U, const double* __restrict__ Ja, const double* __restrict__ aff,
    const double* __restrict__ sJ, const double* __restrict__ Gvol, const double* __restrict__ fgeo,
    const int* __restrict__ elemSide, const double* __restrict__ lam, const double* __restrict__ LGf,
    double* __restrict__ LWs, double* __restrict__ LWf, double* __restrict__ muv, int K, int S, int bigBase,
    double* __restrict__ LQB, const int* __restrict__ order, const __grid_constant__ Ops<double> ops,
    const __grid_constant__ FxOps fx, const __grid_constant__ Phys<double> ph) {
  using C = Cfg<n>;
  constexpr int n2 = C::n2, n3 = C::n3, NE = C::NE, T = C::T, n3p = C::n3p;
  constexpr bool kWarp = NE == 1;
  const int grp = order != nullptr ? order[blockIdx.x] : blockIdx.x;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fx64* sA = reinterpret_cast<fx64*>(smem_raw);  // [NE][15][n3p] line fields l*5 + v
  fx64* sF = sA + NE * 15 * n3p;                 // [NE][6][15][n2] face gradient adjoints; then [NE][6][5][n2] adjoints of U*
  fx64* sN = sF + NE * 90 * n2;                  // [NE][6][3][n2] outward n_d s_hat
  int* sES = reinterpret_cast<int*>(sN + NE * 18 * n2);
  int* sMpq = sES + NE * 6;        // [NE][6][n2]
  int* sMag = sMpq + NE * 6 * n2;  // [NE][FXA_SLOTS]
  const int tid = threadIdx.x;
  const int el = tid / n3, node = tid - el * n3;
  const int e0 = grp * NE, e = e0 + el;
  const bool valid = e < K;
  const int i = node % n, j = (node / n) % n, k = node / n2;
  const unsigned wmask = (tid | 31) < T ? 0xffffffffu : (1u << (T & 31)) - 1u;
  fx64* own = sA + el * 15 * n3p + pidx<n>(i, j, k);
  int* mag = sMag + el * FXA_SLOTS;
  auto fp64 = [&]() {
    adj_vol_fp64<n>(U, Ja, sJ, Gvol, fgeo, elemSide, lam, LGf, LWs, LWf, muv, K, S, bigBase, LQB, ops, ph, grp);
  };
  for (int t = tid; t < NE * FXA_SLOTS; t += T) sMag[t] = 0;
  for (int t = tid; t < NE * 6; t += T) sES[t] = (e0 + t / 6 < K) ? elemSide[(size_t)e0 * 6 + t] : 0;
  const double sj = valid ? sJ[(size_t)e * n3 + node] : 0.0;
  // metric term l*3 + d of the node (read again where it is needed: registers are short)
  auto metric = [&](int c) {
    return !valid ? 0.0 : (AFF ? aff[(size_t)e * 10 + c] : Ja[((size_t)e * 9 + c) * n3 + node]);
  };
  __syncthreads();
  // lam_vol = -lam / J, the metric terms' and the face data's magnitudes
  {
    double lv[NV];
    int mJ[3] = {0, 0, 0};
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      lv[v] = valid ? -lam[((size_t)e * NV + v) * n3 + node] * sj : 0.0;
      own[v * n3p] = __double_as_longlong(lv[v]);
    }
#pragma unroll
    for (int c = 0; c < 9; ++c) mJ[c % 3] = max(mJ[c % 3], fx_mag(metric(c)));
    for (int it = tid; it < NE * 6 * n2; it += T) {
      const int f = it / n2, pq = it - f * n2;
      if (e0 + f / 6 >= K) continue;
      const int es = sES[f], side = es_side(es);
      const int mpq = orient_pq(es_orient(es), n - 1, pq % n, pq / n);
      sMpq[it] = mpq;
      const double* src = LGf + ((size_t)(es_slave(es) * S + side) * 15) * n2 + mpq;
      int* m = sMag + (f / 6) * FXA_SLOTS;
#pragma unroll
      for (int c = 0; c < 15; ++c) {
        const double x = src[c * n2];
        sF[(f * 15 + c) * n2 + pq] = __double_as_longlong(x);
        atomicMax(m + FXA_B + c, fx_mag(x));
      }
      if constexpr (!AFF) {
        const double* g = fgeo + ((size_t)side * 4) * n2 + mpq;
        const double sc = dg_neg_if(g[3 * n2], es_slave(es));
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const double x = side < bigBase ? g[d * n2] * sc : 0.0;
          sN[(f * 3 + d) * n2 + pq] = __double_as_longlong(x);
          mJ[d] = kWarp ? max(mJ[d], fx_mag(x)) : mJ[d];
          if constexpr (!kWarp) atomicMax(m + FXA_J + d, fx_mag(x));
        }
      }
    }
    fx_max<kWarp, 8>(mag, wmask, [&](int s) { return s < 5 ? fx_mag(lv[s < 5 ? s : 0]) : mJ[s < 5 ? 0 : s - 5]; });
  }
  __syncthreads();
  {
    int bad = 0;
    for (int t = tid; t < NE * FXA_SLOTS; t += T) bad |= (sMag[t] >> 20) > 1022 + 200;
    if (__syncthreads_or(bad)) {
      fp64();
      return;
    }
  }
  const int* EJ = mag + FXA_J;  // exponent of direction d: EJ[d] >> 20
  for (int it = tid; it < NE * 6 * n2; it += T) {  // the thread's own entries, as above
    const int f = it / n2, pq = it - f * n2;
    if (e0 + f / 6 >= K) continue;
    const int* m = sMag + (f / 6) * FXA_SLOTS;
#pragma unroll
    for (int c = 0; c < 15; ++c) {
      fx64* x = sF + (f * 15 + c) * n2 + pq;
      *x = fx_from<61>(__longlong_as_double(*x), m[FXA_B + c] >> 20);
    }
    if constexpr (!AFF) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        fx64* x = sN + (f * 3 + d) * n2 + pq;
        *x = fx_from<62>(__longlong_as_double(*x), m[FXA_J + d] >> 20);
      }
    }
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const fx64 x = fx_from<59>(__longlong_as_double(own[v * n3p]), mag[FXA_L + v] >> 20);
#pragma unroll
    for (int l = 0; l < 3; ++l) own[(l * NV + v) * n3p] = x;
  }
  __syncthreads();
  // reverse of a7: D_hat^T along l of lam_vol
#pragma unroll 1
  for (int it = tid; it < NE * 15 * n2; it += T) {
    const int f = it / n2, line = it - f * n2;
    int stride;
    const int at = fx_line_at<n>((f % 15) / NV, line, stride);
    fx_line<n, false, false>(sA + f * n3p + at, stride, 0, 0, fx);
  }
  __syncthreads();
  // reverse of a6: lam_d = sum_l Ja^l_d lamF^l, then the pointwise fluxes
  double lamU[NV] = {0, 0, 0, 0, 0}, lamW[NV] = {0, 0, 0, 0, 0}, W[NV];
  {
    double Uo[NV] = {1.0, 0.0, 0.0, 0.0, 1.0}, lvisc[3][NV];
    if (valid) {
#pragma unroll
      for (int v = 0; v < NV; ++v) Uo[v] = U[((size_t)e * NV + v) * n3 + node];
    }
    cons_to_prim(Uo, W, ph);
    {
      FxSplit ji[9];
#pragma unroll
      for (int c = 0; c < 9; ++c) ji[c] = fx_split(fx_from<62>(metric(c), EJ[c % 3] >> 20));
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        FxSplit t[3];
#pragma unroll
        for (int l = 0; l < 3; ++l) t[l] = fx_split(own[(l * NV + v) * n3p] << 2);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          FxAcc s;
#pragma unroll
          for (int l = 0; l < 3; ++l) s.add(ji[l * 3 + d], t[l]);
          lvisc[d][v] = -fx_to(s.get(), (EJ[d] >> 20) + (mag[FXA_L + v] >> 20) - 2044 + 5 - fx.kc);
        }
      }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      double ld[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) ld[v] = -lvisc[d][v];
      conv_vjp(Uo, W, d, ld, lamU, lamW);
    }
    double G[15], lamG[15];
#pragma unroll
    for (int c = 0; c < 15; ++c) {
      G[c] = valid ? Gvol[((size_t)e * 15 + c) * n3 + node] : 0.0;
      lamG[c] = 0.0;
    }
    visc_vjp(W, G, lvisc, ph, lamW, lamG);
    // reverse of a4: the faces' gradient adjoints spread with l(+-1); lam_lift = lamG / J
    const int pq0 = j + n * k, pq1 = i + n * k, pq2 = i + n * j;
    const fx64* Fe = sF + el * 90 * n2;
    auto spread = [&](int f, int pq, int at, int c) {
      FxAcc a;  // two products per accumulator, as the factors have 61 and 62 bits
      a.add(fx_split(Fe[(2 * f * 15 + c) * n2 + pq]), fx.lh[n - 1 - at], fx.ll[n - 1 - at]);
      a.add(fx_split(Fe[((2 * f + 1) * 15 + c) * n2 + pq]), fx.lh[at], fx.ll[at]);
      return a.get();
    };
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      int mx[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const int c = d * NV + v;
        const fx64 b = spread(0, pq0, i, c) + spread(1, pq1, j, c) + spread(2, pq2, k, c);
        const double x = (lamG[c] + fx_to(b, (mag[FXA_B + c] >> 20) - 1022 + 3 - fx.kl)) * sj;
        mx[v] = fx_mag(x);
        own[c * n3p] = __double_as_longlong(x);  // the thread's entries: field d*5 + v
      }
      fx_max<kWarp, NV>(mag + FXA_X + d * NV, wmask, [&](int s) { return mx[s]; });
    }
  }
  __syncthreads();
  {  // magnitude words -> the exponents under which lam_lift_d,v is converted (flux_exponents, k_lift_fx.cuh)
    int bad = 0;
    for (int t = tid; t < NE * NV; t += T) {
      int* m = sMag + (t / NV) * FXA_SLOTS;
      int* f = m + FXA_X + t % NV;
      int x = 0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        bad |= (f[d * NV] >> 20) > 1022 + 600;
        x = max(x, (f[d * NV] >> 20) + (m[FXA_J + d] >> 20));
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) f[d * NV] = x - (m[FXA_J + d] >> 20);
    }
    if (__syncthreads_or(bad)) {
      fp64();
      return;
    }
  }
  // reverse of a3: W receives sum_l sum_d Ja^l_d D_hat^T_l lam_lift^d; the face means of W the ends
  fx64* sS = sF;  // [NE][6][5][n2]
  if constexpr (AFF) {
    {
      FxSplit ji[9];
#pragma unroll
      for (int c = 0; c < 9; ++c) ji[c] = fx_split(fx_from<62>(metric(c), EJ[c % 3] >> 20));
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        FxSplit x[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) x[d] = fx_split(fx_from<60>(__longlong_as_double(own[(d * NV + v) * n3p]), mag[FXA_X + d * NV + v]));
#pragma unroll
        for (int l = 0; l < 3; ++l) {
          FxAcc s;
#pragma unroll
          for (int d = 0; d < 3; ++d) s.add(ji[l * 3 + d], x[d]);
          own[(l * NV + v) * n3p] = s.get();
        }
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int it = tid; it < NE * 15 * n2; it += T) {
      const int f = it / n2, line = it - f * n2;
      const int el2 = f / 15, c = f - el2 * 15, l = c / NV, v = c - l * NV;
      int stride;
      const int at = fx_line_at<n>(l, line, stride);
      fx64 ym, yp;
      fx_line_ends<n>(sA + f * n3p + at, stride, fx, ym, yp);
      fx64* q = sS + ((el2 * 6 + 2 * l) * NV + v) * n2 + line;
      q[0] = -ym;
      q[NV * n2] = yp;
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < NV; ++v)
      lamW[v] += fx_to(own[v * n3p] + own[(NV + v) * n3p] + own[(2 * NV + v) * n3p],
                       (EJ[0] >> 20) + mag[FXA_X + v] - 2044 + 6 - fx.kc);
  } else {
    fx64 acc[NV] = {0, 0, 0, 0, 0};
    fx64 x[15];
#pragma unroll
    for (int c = 0; c < 15; ++c) x[c] = fx_from<59>(__longlong_as_double(own[c * n3p]), mag[FXA_X + c]);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int l = 0; l < 3; ++l) own[(l * NV + v) * n3p] = x[d * NV + v];
      __syncthreads();
#pragma unroll 1
      for (int it = tid; it < NE * 15 * n2; it += T) {
        const int f = it / n2, line = it - f * n2;
        const int el2 = f / 15, c = f - el2 * 15, l = c / NV, v = c - l * NV;
        int stride;
        const int at = fx_line_at<n>(l, line, stride);
        fx64 y[2];
        fx_line_ends<n>(sA + f * n3p + at, stride, fx, y[0], y[1]);
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const int fc = el2 * 6 + 2 * l + m;
          const fx64 z = fx_mul(fx_split(y[m] << 2), fx_split(sN[(fc * 3 + d) * n2 + line]));
          fx64* q = sS + (fc * NV + v) * n2 + line;
          *q = d == 0 ? z : *q + z;
          const int side = es_side(sES[fc]);
          if (side >= bigBase && e0 + el2 < K)  // adjoint of the projected lifting flux QB
            LQB[((size_t)(side - bigBase) * 15 + v * 3 + d) * n2 + sMpq[fc * n2 + line]] =
                fx_to(y[m], sMag[el2 * FXA_SLOTS + FXA_X + d * NV + v] - 1022 + 5 - fx.kp);
        }
      }
      __syncthreads();
      FxSplit a[3];
#pragma unroll
      for (int l = 0; l < 3; ++l) a[l] = fx_split(fx_from<62>(metric(l * 3 + d), EJ[d] >> 20));
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        FxAcc s;
#pragma unroll
        for (int l = 0; l < 3; ++l) s.add(a[l], fx_split(own[(l * NV + v) * n3p] << 2));
        acc[v] += s.get();
      }
      // a thread stages only its own entries, read by line tasks before the barrier above
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) lamW[v] += fx_to(acc[v], (EJ[0] >> 20) + mag[FXA_X + v] - 2044 + 5 - fx.kc);
  }
  // adjoints of the face means of W to the side arrays
  for (int it = tid; it < NE * 6 * n2; it += T) {
    const int f = it / n2, pq = it - f * n2;
    if (e0 + f / 6 >= K) continue;
    const int es = sES[f], side = es_side(es);
    const int* m = sMag + (f / 6) * FXA_SLOTS;
    double* dst = LWs + ((size_t)(es_slave(es) * S + side) * NV) * n2 + sMpq[it];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const int t = (m[FXA_J] >> 20) + m[FXA_X + v] - 2044 + (AFF ? 6 : 5) - fx.kp;
      dst[v * n2] = side >= bigBase ? 0.0 : fx_to(sS[(f * NV + v) * n2 + pq], t);
    }
  }
  prim_vjp(W, lamW, ph, lamU);
  if (valid) {
#pragma unroll
    for (int v = 0; v < NV; ++v) muv[((size_t)e * NV + v) * n3 + node] = lamU[v];
  }
}

template <int n>
static cudaError_t launch_adj_vol_fx(const DevMesh& m, const double* U, const double* lam, const double* LGf, double* LWs,
                                     double* LWf, double* muv, double* LQB, const Ops<double>& ops, const Phys<double>& ph,
                                     cudaStream_t st) {
  using C = Cfg<n>;
  constexpr size_t smem = adj_fx_smem<n>();
  const int groups = (m.K + C::NE - 1) / C::NE;
  static std::atomic<unsigned long long> attr[2];
  cudaError_t err;
#define FLEXI_ADJ_FX(AFF, GRID, ORDER)                                                                                \
  do {                                                                                                                \
    if ((err = ensure_dynamic_smem(&k_adj_vol_fx<n, AFF>, smem, attr[AFF])) != cudaSuccess) return err;              \
    k_adj_vol_fx<n, AFF><<<GRID, C::T, smem, st>>>(U, (const double*)m.Ja, (const double*)m.affine, (const double*)m.sJ,           \
                                                   (const double*)m.Gvol, (const double*)m.fgeo, m.elemSide, lam,    \
                                                   LGf, LWs, LWf, muv, m.K, m.S, m.Sface, LQB, ORDER, ops, m.fxT, ph); \
    if ((err = cudaGetLastError()) != cudaSuccess) return err;                                                        \
  } while (0)
  if (m.nAffine > 0) FLEXI_ADJ_FX(true, m.nAffine, (m.nAffine < groups ? m.order : nullptr));
  if (m.nAffine < groups) FLEXI_ADJ_FX(false, groups - m.nAffine, (m.nAffine > 0 ? m.order + m.nAffine : nullptr));
#undef FLEXI_ADJ_FX
  return cudaSuccess;
}

}  // namespace flexi
