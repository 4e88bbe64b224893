// Lifting and volume integral of the FP64 form with the line contractions in block
// fixed point (fx.cuh).  Standard and kinetic-energy-preserving volume integral, BR1.
//
// With FP64 sweeps the kernel is bound by the FP64 pipe: of its 850 FP64 instructions
// per node (n = 8, Gauss) 480 are D_hat multiply-adds, 90 lifting face terms, 90 gradient
// prolongation and 90 metric products.  All of those are sums of products under one scale
// and run here on the integer pipes; the FP64 pipe keeps the primitive variables, the
// surface means and the pointwise fluxes.  Elements whose values leave the fixed-point
// range (above 2^200, infinities, NaN) take the FP64 schedule of lift_vol_fp64.  16^3 elements,
// N = 7: 3061 -> 750 us (curved), 559 us (affine; 77 FP64 and 3,775 integer instructions per
// node); 638 MB (470 affine) are 95 (70) us at the measured copy rate.  No pipe is the bound on its
// own: FP64, ALU and FMA-heavy pipe and the issue slots are each busy 43 to 47 % of the time, as
// the phases that use the one or the others follow each other with barriers between.
#pragma once
#include "fx.cuh"

namespace flexi {

// slots of an element's magnitude table: primitive variables (nodes and face means), metric
// terms by physical direction (nodes and faces; affine elements J^l_d / J), 1/J (affine
// elements J^l_d by direction), fluxes at d*5+v, projected lifting fluxes of mortar sides (v*3+d)
enum { FX_W = 0, FX_J = 5, FX_S = 8, FX_F = 11, FX_Q = 26, FX_SLOTS = 42 };
// largest exponent fields that the fixed-point kernel takes: products of four such values
// stay inside the FP64 range
constexpr int FX_MAX_EXP = 1022 + 200, FX_MAX_FLUX = 1022 + 600;

// one line of a D_hat contraction in place with its face terms, in FP64
template <int n, bool LGL, bool FACE>
__device__ __forceinline__ void fp64_line(double* __restrict__ p, int stride, double qm, double qp, const Ops<double>& o) {
  double x[n];
#pragma unroll
  for (int a = 0; a < n; ++a) x[a] = p[a * stride];
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    double y = 0.0;
    if (FACE && (!LGL || i == 0)) y = dg_fma(o.lhm[i], qm, y);
    if (FACE && (!LGL || i == n - 1)) y = dg_fma(o.lhp[i], qp, y);
#pragma unroll
    for (int a = 0; a < n; ++a) y = dg_fma(o.DhatT[a * n + i], x[a], y);
    p[i * stride] = y;
  }
}

// The kernel below for elements outside the fixed-point range: the same schedule over the
// same shared memory in FP64 (speed does not matter here, the footprint does: the general
// FP64 body's would cost the resident second CTA).
template <int n, bool LGL, bool KEP>
__device__ __noinline__ void lift_vol_fp64(const double* U, const double* Ja, const double* sJ, const double* Wf,
                                           const double* fgeo, double* Gf, double* Utv, double* Gvol, int K, int S,
                                           int bigBase, const double* QB, const Ops<double>& ops, const Phys<double>& ph,
                                           double* sA, double* sW, const int* sES, const int* sMpq, int grp) {
  using C = Cfg<n>;
  constexpr int n2 = C::n2, n3 = C::n3, NE = C::NE, T = C::T, n3p = C::n3p, P = C::P;
  const int tid = threadIdx.x;
  const int el = tid / n3, node = tid - el * n3;
  const int e0 = grp * NE, e = e0 + el;
  const bool valid = e < K;
  double* own = sA + el * 15 * n3p + pidx<n>(node % n, (node / n) % n, node / n2);
  double Uo[NV] = {1.0, 0.0, 0.0, 0.0, 1.0}, W[NV], jac[9], G[15];
  if (valid) {
#pragma unroll
    for (int v = 0; v < NV; ++v) Uo[v] = U[((size_t)e * NV + v) * n3 + node];
  }
#pragma unroll
  for (int c = 0; c < 9; ++c) jac[c] = valid ? Ja[((size_t)e * 9 + c) * n3 + node] : 0.0;
  const double sj = valid ? sJ[(size_t)e * n3 + node] : 0.0;
  cons_to_prim(Uo, W, ph);
  __syncthreads();
  for (int it = tid; it < NE * 6 * n2; it += T) {
    const int f = it / n2, pq = it - f * n2;
    const int es = sES[f], side = es_side(es), mpq = sMpq[it];
    if (e0 + f / 6 >= K || side >= bigBase) continue;
    const double* g = fgeo + ((size_t)side * 4) * n2 + mpq;
    const double sc = dg_neg_if(0.5 * g[3 * n2], es_slave(es));
    for (int v = 0; v < NV; ++v)
      sW[(f * 8 + v) * n2 + pq] = Wf[((size_t)side * NV + v) * n2 + mpq] + Wf[((size_t)(S + side) * NV + v) * n2 + mpq];
    for (int d = 0; d < 3; ++d) sW[(f * 8 + 5 + d) * n2 + pq] = g[d * n2] * sc;
  }
  auto lines = [&](auto face, int d) {
    for (int it = tid; it < NE * 15 * n2; it += T) {
      const int f = it / n2, line = it - f * n2;
      const int el2 = f / 15, c = f - el2 * 15, l = c / NV, v = c - l * NV;
      double q[2] = {0.0, 0.0};
      if constexpr (decltype(face)::value) {
        for (int m = 0; m < 2; ++m) {
          const int fc = el2 * 6 + 2 * l + m, side = es_side(sES[fc]);
          const double* w = sW + fc * 8 * n2 + line;
          if (e0 + el2 < K)
            q[m] = side < bigBase ? w[v * n2] * w[(5 + d) * n2]
                                  : QB[((size_t)(side - bigBase) * 15 + v * 3 + d) * n2 + sMpq[fc * n2 + line]];
        }
      }
      const int a0 = line % n, a1 = line / n;
      fp64_line<n, LGL, decltype(face)::value>(
          sA + f * n3p + (l == 0 ? P * line : (l == 1 ? a0 + P * n * a1 : a0 + P * a1)),
          l == 0 ? 1 : (l == 1 ? P : P * n), q[0], q[1], ops);
    }
  };
  for (int d = 0; d < 3; ++d) {
    for (int l = 0; l < 3; ++l)
      for (int v = 0; v < NV; ++v) own[(l * NV + v) * n3p] = jac[l * 3 + d] * W[v];
    __syncthreads();
    lines(std::true_type{}, d);
    __syncthreads();
    for (int v = 0; v < NV; ++v) {
      const double g = (own[v * n3p] + own[(NV + v) * n3p] + own[(2 * NV + v) * n3p]) * sj;
      G[d * NV + v] = own[v * n3p] = g;
      if (Gvol != nullptr && valid) Gvol[((size_t)e * 15 + d * NV + v) * n3 + node] = g;
    }
    __syncthreads();
    for (int it = tid; it < NE * 30 * n2; it += T) {  // one (face, variable, face node) per task
      const int f = it / n2, pq = it - f * n2;
      const int el2 = f / 30, c = f - el2 * 30, s = c / NV, v = c - s * NV, l = s >> 1;
      if (e0 + el2 >= K) continue;
      const double* b = sA + (el2 * 15 + v) * n3p;
      double val = 0.0;
      if constexpr (LGL) {
        val = b[pvol_index<n>(l, (s & 1) ? n - 1 : 0, pq % n, pq / n)];
      } else {
        for (int a = 0; a < n; ++a)
          val = dg_fma((s & 1) ? ops.lp[a] : ops.lm[a], b[pvol_index<n>(l, a, pq % n, pq / n)], val);
      }
      const int es = sES[el2 * 6 + s];
      Gf[((size_t)(es_slave(es) * S + es_side(es)) * 15 + d * NV + v) * n2 + sMpq[(el2 * 6 + s) * n2 + pq]] = val;
    }
    __syncthreads();
  }
  if (Utv == nullptr) return;
  double F[3][NV];
  for (int d = 0; d < 3; ++d) {
    if constexpr (KEP) {
      flux_viscous(W, dg_rcp(W[0]), G, d, ph, F[d]);
      for (int v = 0; v < NV; ++v) F[d][v] = -F[d][v];
    } else {
      flux_total(Uo, W, G, d, ph, F[d]);
    }
  }
  for (int l = 0; l < 3; ++l)
    for (int v = 0; v < NV; ++v)
      own[(l * NV + v) * n3p] = jac[l * 3] * F[0][v] + jac[l * 3 + 1] * F[1][v] + jac[l * 3 + 2] * F[2][v];
  __syncthreads();
  lines(std::false_type{}, 0);
  __syncthreads();
  double acc[NV];
  for (int v = 0; v < NV; ++v) acc[v] = own[v * n3p] + own[(NV + v) * n3p] + own[(2 * NV + v) * n3p];
  if constexpr (KEP) {  // as split_volume_fx
    const double H = dg_div(Uo[4] + W[4], W[0]);
    for (int v = 0; v < NV; ++v) own[v * n3p] = W[v];
    own[5 * n3p] = H;
    for (int c = 0; c < 9; ++c) own[(6 + c) * n3p] = jac[c];
    __syncthreads();
    for (int l = 0; l < 3; ++l) {
      const int il = l == 0 ? node % n : (l == 1 ? (node / n) % n : node / n2), stride = l == 0 ? 1 : (l == 1 ? P : P * n);
      for (int a = 0; a < n; ++a) {
        if (a == il) continue;
        const double* f = own + (a - il) * stride;
        const double j0 = jac[l * 3] + f[(6 + 3 * l) * n3p], j1 = jac[l * 3 + 1] + f[(7 + 3 * l) * n3p],
                     j2 = jac[l * 3 + 2] + f[(8 + 3 * l) * n3p];
        const double us = W[1] + f[n3p], vs = W[2] + f[2 * n3p], ws = W[3] + f[3 * n3p];
        const double m = 0.125 * (W[0] + f[0]) * (us * j0 + vs * j1 + ws * j2), hp = 0.5 * (W[4] + f[4 * n3p]);
        const double d = ops.DT[a * n + il];
        acc[0] += d * (2.0 * m);
        acc[1] += d * (m * us + hp * j0);
        acc[2] += d * (m * vs + hp * j1);
        acc[3] += d * (m * ws + hp * j2);
        acc[4] += d * (m * (H + f[5 * n3p]));
      }
    }
  }
  if (valid)
    for (int v = 0; v < NV; ++v) Utv[((size_t)e * NV + v) * n3 + node] = acc[v];
}

template <int n>
constexpr size_t lift_fx_smem() {
  using C = Cfg<n>;
  return 8 * C::NE * (15 * C::n3p + 48 * C::n2) + 8 * C::n2 + sizeof(int) * C::NE * (12 + 6 * C::n2 + FX_SLOTS + 32);
}

// CTAs per SM asked of the register allocator (n = 8: two of 512 threads at 64 registers;
// n = 7: three of 343 at 56 against two at 80, 16^3: 657 -> 601 us, affine 453 -> 398 (now 608, 388); the
// pairs of the split form want the registers: 14^3 curved, N = 6, 647 -> 627 us with two, 18^3
// curved, N = 4, 367 -> 343 us with six of 125 threads instead of seven)
template <int n, bool KEP>
constexpr int lift_fx_min_blocks() {
  return n == 8 ? 2 : (n == 7 ? (KEP ? 2 : 3) : (n == 6 ? 4 : (n == 5 ? (KEP ? 6 : 7) : (n == 4 ? 12 : 6))));
}

// free indices and stride of line `line` along l; offset of its first entry in a field
template <int n>
__device__ __forceinline__ int fx_line_at(int l, int line, int& stride) {
  constexpr int P = Cfg<n>::P;
  const int a0 = line % n, a1 = line / n;
  stride = l == 0 ? 1 : (l == 1 ? P : P * n);
  return l == 0 ? P * line : (l == 1 ? a0 + P * n * a1 : a0 + P * a1);
}

// Scale of the fluxes of variables v >= V0: their largest magnitude words at FX_F + d*5+v
// become the exponents under which F_d,v is converted, x_v - E(Ja_d), where x_v is the largest
// of E(F_d,v) + E(Ja_d).  False when a flux leaves the fixed-point range.  Block-wide; synced.
template <int NE, int T, int V0>
__device__ __forceinline__ bool flux_exponents(int* sMag, int JS) {
  int bad = 0;
  for (int t = threadIdx.x; t < NE * (NV - V0); t += T) {
    int* m = sMag + (t / (NV - V0)) * FX_SLOTS;
    int* f = m + FX_F + V0 + t % (NV - V0);
    int x = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      bad |= (f[d * NV] >> 20) > FX_MAX_FLUX;
      x = max(x, (f[d * NV] >> 20) + (m[JS + d] >> 20));
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) f[d * NV] = x - (m[JS + d] >> 20);
  }
  return !__syncthreads_or(bad);
}

// a6, a7: physical fluxes in FP64, contravariant fluxes and the volume integral in fixed
// point.  metric(ji): the node's nine metric terms, direction d under the exponent of slot
// JS + d.  A variable's three fluxes are scaled by direction: in a flat element the flux
// through the large area may be far smaller than the others and still decide the sum, so
// F_d is taken to the scale at which its product with the largest |Ja^l_d| meets the largest
// such product of the three directions (one exponent for all three lost a digit of U_t per
// factor ten of aspect ratio against FP64).  False, with nothing written, when a flux leaves
// the fixed-point range.  Block-wide.
template <int n, bool LGL, int JS, typename Metric>
__device__ __forceinline__ bool volume_fx(const double* __restrict__ U, double* __restrict__ Utv, const double (&W)[NV],
                                          const double (&G)[15], int K, int grp, unsigned wmask, fx64* sA, int* sMag,
                                          const FxOps& fx, const Phys<double>& ph, Metric metric) {
  using C = Cfg<n>;
  constexpr int n2 = C::n2, n3 = C::n3, NE = C::NE, T = C::T, n3p = C::n3p;
  const int tid = threadIdx.x;
  const int el = tid / n3, node = tid - el * n3;
  const int e = grp * NE + el;
  const bool valid = e < K;
  int* mag = sMag + el * FX_SLOTS;
  fx64* own = sA + el * 15 * n3p + pidx<n>(node % n, (node / n) % n, node / n2);  // the thread's entries
  {
    double Uo[NV] = {1.0, 0.0, 0.0, 0.0, 1.0};
    if (valid) {
#pragma unroll
      for (int v = 0; v < NV; ++v) Uo[v] = U[((size_t)e * NV + v) * n3 + node];
    }
    const double ir = 1.0 / Uo[0];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      double F[NV];
      flux_total(Uo, W, ir, G, d, ph, F);
#pragma unroll
      for (int v = 0; v < NV; ++v) own[(d * NV + v) * n3p] = __double_as_longlong(F[v]);
      fx_max<NE == 1, NV>(mag + FX_F + d * NV, wmask, [&](int s) { return fx_mag(F[s]); });
    }
  }
  __syncthreads();
  if (!flux_exponents<NE, T, 0>(sMag, JS)) return false;
  {
    FxSplit ji[9];
    metric(ji);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      FxSplit F[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) F[d] = fx_split(fx_from<60>(__longlong_as_double(own[(d * NV + v) * n3p]), mag[FX_F + d * NV + v]));
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        FxAcc s;
#pragma unroll
        for (int d = 0; d < 3; ++d) s.add(ji[l * 3 + d], F[d]);
        own[(l * NV + v) * n3p] = s.get();
      }
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int it = tid; it < NE * 15 * n2; it += T) {
    const int f = it / n2, line = it - f * n2;
    int stride;
    const int at = fx_line_at<n>((NE == 1 ? f : f % 15) / NV, line, stride);
    fx_line<n, LGL, false>(sA + f * n3p + at, stride, 0, 0, fx);
  }
  __syncthreads();
  if (valid) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const fx64* r = own + v * n3p;
      Utv[((size_t)e * NV + v) * n3 + node] =
          fx_to(r[0] + r[NV * n3p] + r[2 * NV * n3p], mag[FX_F + v] + (mag[JS] >> 20) - 2044 + 6 - fx_up(n, LGL) - fx.kc);
    }
  }
  return true;
}

// Split form (kinetic-energy preserving, Gauss-Lobatto): the viscous flux as in volume_fx; the
// advective part 2 sum_a D_ia F#(i, a) with one thread per node over its 3 (n - 1) pairs, in
// fixed point: pair sums and their products replace 21 FP64 multiply-adds per pair.  The
// diagonal terms 2 D_ii F(U_i) and the strong form's face terms -(+-1) l_hat(+-1) F(U_i) cancel
// (2 w_i D_ii = +-1 at the ends, 0 inside), so neither is formed.  Scales: rho, p, H and, by
// direction, the velocity and Ja each under a power of two of their own.  Their products meet
// at the largest of them: the mass flux at 2^bC, the largest of |u_d| |Ja_d|, momentum d at the
// larger of mass flux times u_d and p Ja_d (shifts sc, sm, sp of the smaller operands).
// 990 elements, N = 7: 1130 -> 240 us with the lifting (232 with one scale for all directions and
// for all rows of D, at up to 190 times the rounding noise of FP64 sums).
template <int n, bool AFF, int JS, typename Metric>
__device__ __forceinline__ bool split_volume_fx(const double* __restrict__ U, double* __restrict__ Utv, const double (&W)[NV],
                                                const double (&G)[15], int K, int grp, unsigned wmask, fx64* sA, int* sMag,
                                                int2* sD, const FxOps& fx, const FxStrong& fd, const Phys<double>& ph,
                                                Metric metric) {
  using C = Cfg<n>;
  constexpr int n2 = C::n2, n3 = C::n3, NE = C::NE, T = C::T, n3p = C::n3p, P = C::P;
  const int tid = threadIdx.x;
  const int el = tid / n3, node = tid - el * n3;
  const int e = grp * NE + el;
  const bool valid = e < K;
  int* mag = sMag + el * FX_SLOTS;
  fx64* own = sA + el * 15 * n3p + pidx<n>(node % n, (node / n) % n, node / n2);
  double H;
  {
    double E = 1.0;
    if (valid) E = U[((size_t)e * NV + 4) * n3 + node];
    const double ir = 1.0 / W[0];
    H = (E + W[4]) * ir;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      double F[NV];
      flux_viscous(W, ir, G, d, ph, F);
      F[0] = H;  // slots of the first variable: H
#pragma unroll
      for (int v = 1; v < NV; ++v) own[(d * NV + v) * n3p] = __double_as_longlong(-F[v]);
      fx_max<NE == 1, NV>(mag + FX_F + d * NV, wmask, [&](int s) { return fx_mag(F[s]); });
    }
  }
  for (int t = tid; t < n2; t += T) sD[t] = make_int2(fd.h[t], fd.l[t]);
  __syncthreads();
  {
    int bad = 0;
    for (int t = tid; t < NE; t += T) bad |= (sMag[t * FX_SLOTS + FX_F] >> 20) > FX_MAX_EXP + 200;
    if (__syncthreads_or(bad)) return false;
  }
  if (!flux_exponents<NE, T, 1>(sMag, JS)) return false;
  double vis[NV];
  {
    FxSplit ji[9];
    metric(ji);
#pragma unroll
    for (int v = 1; v < NV; ++v) {
      FxSplit F[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) F[d] = fx_split(fx_from<60>(__longlong_as_double(own[(d * NV + v) * n3p]), mag[FX_F + d * NV + v]));
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        FxAcc s;
#pragma unroll
        for (int d = 0; d < 3; ++d) s.add(ji[l * 3 + d], F[d]);
        own[(l * NV + v) * n3p] = s.get();
      }
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int it = tid; it < NE * 12 * n2; it += T) {
    const int q = it / n2, line = it - q * n2;
    const int el2 = q / 12, c = q - el2 * 12, l = c >> 2, f = el2 * 15 + l * NV + 1 + (c & 3);
    int stride;
    const int at = fx_line_at<n>(l, line, stride);
    fx_line<n, true, false>(sA + f * n3p + at, stride, 0, 0, fx);
  }
  __syncthreads();
  vis[0] = 0.0;
#pragma unroll
  for (int v = 1; v < NV; ++v)
    vis[v] = fx_to(own[v * n3p] + own[(NV + v) * n3p] + own[(2 * NV + v) * n3p],
                   mag[FX_F + v] + (mag[JS] >> 20) - 2044 + 6 - fx_up(n, true) - fx.kc);
  // advective part: bounds b of rho, H, p, mass flux and momentum flux as powers of two
  const int bR = (mag[FX_W] >> 20) - 1022, bH = (mag[FX_F] >> 20) - 1022, bP = (mag[FX_W + 4] >> 20) - 1022;
  int bC = -4096;
#pragma unroll
  for (int d = 0; d < 3; ++d) bC = max(bC, (mag[FX_W + 1 + d] >> 20) + (mag[JS + d] >> 20) - 2044);
  int sc[3], sm[3], sp[3], bM[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int bU = (mag[FX_W + 1 + d] >> 20) - 1022, bJ = (mag[JS + d] >> 20) - 1022;
    bM[d] = max(bP + bJ, bR + bC + bU + 2);
    sc[d] = min(bC - bU - bJ, 62);
    sm[d] = min(bM[d] - (bR + bC + bU + 2), 62);
    sp[d] = min(bM[d] - (bP + bJ), 62);
  }
  const bool shift_p = (sp[0] | sp[1] | sp[2]) != 0;
  fx64 q[6];
  q[0] = fx_from<61>(W[0], bR + 1022);
#pragma unroll
  for (int d = 0; d < 3; ++d) q[1 + d] = fx_from<60>(W[1 + d], mag[FX_W + 1 + d] >> 20);
  q[4] = fx_from<60>(W[4], bP + 1022);
  q[5] = fx_from<61>(H, bH + 1022);
#pragma unroll
  for (int c = 0; c < 6; ++c) own[c * n3p] = q[c];
  {
    FxSplit ji[9];
    metric(ji);
    if constexpr (!AFF) {
#pragma unroll
      for (int c = 0; c < 9; ++c) own[(6 + c) * n3p] = fx_shr(((fx64)ji[c].h << 32) + ji[c].l, 2);
    } else {  // J^l_d is the pair's mean: its sum in the same units
#pragma unroll
      for (int c = 0; c < 9; ++c) own[(6 + c) * n3p] = fx_shr(((fx64)ji[c].h << 32) + ji[c].l, 1);
    }
  }
  __syncthreads();
  fx64 sum[NV] = {0, 0, 0, 0, 0};
#pragma unroll 1
  for (int l = 0; l < 3; ++l) {
    const int il = l == 0 ? node % n : (l == 1 ? (node / n) % n : node / n2), stride = l == 0 ? 1 : (l == 1 ? P : P * n);
    const fx64* jo = own + (6 + 3 * l) * n3p;
    const fx64 J0 = jo[0], J1 = jo[n3p], J2 = jo[2 * n3p];
    const bool end = il == 0 || il == n - 1;
    FxAcc s[NV];
    int a = il;
#pragma unroll 1
    for (int k = 1; k < n; ++k) {
      a = a + 1 == n ? 0 : a + 1;
      const fx64* f = own + (a - il) * stride;
      const FxSplit u = fx_split(q[1] + f[n3p]), v = fx_split(q[2] + f[2 * n3p]), w = fx_split(q[3] + f[3 * n3p]);
      fx64 j0 = J0, j1 = J1, j2 = J2;
      if constexpr (!AFF) {
        const fx64* jp = f + (6 + 3 * l) * n3p;
        j0 += jp[0];
        j1 += jp[n3p];
        j2 += jp[2 * n3p];
      }
      FxAcc c;
      c.add(u, fx_split(j0 >> sc[0]));
      c.add(v, fx_split(j1 >> sc[1]));
      c.add(w, fx_split(j2 >> sc[2]));
      // 8 {rho}{u . Ja}; the operands of D are shifted up, below 2^60.6 for the sums over a row
      const fx64 m4 = fx_mul(fx_split(q[0] + f[0]), fx_split(c.get() << 2)) << 1;
      const FxSplit ms = fx_split(m4);
      if (shift_p) {  // a momentum flux beyond the pressure's
        j0 >>= sp[0];
        j1 >>= sp[1];
        j2 >>= sp[2];
      }
      const FxSplit p = fx_split(q[4] + f[4 * n3p]);
      const int2 D = sD[a * n + il];
      const FxSplit d{D.x, D.y};
      s[0].add(ms, d);
      FxAcc x;
      x.add(fx_split(m4 >> sm[0]), u);
      x.add(p, fx_split(j0));
      s[1].add(fx_split(x.get() << 1), d);
      x = FxAcc();
      x.add(fx_split(m4 >> sm[1]), v);
      x.add(p, fx_split(j1));
      s[2].add(fx_split(x.get() << 1), d);
      x = FxAcc();
      x.add(fx_split(m4 >> sm[2]), w);
      x.add(p, fx_split(j2));
      s[3].add(fx_split(x.get() << 1), d);
      s[4].add(fx_split(fx_mul(ms, fx_split(q[5] + f[5 * n3p])) << 2), d);
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) sum[v] += s[v].get() << (end ? 2 : 0);  // scale of the rows of D
  }
  if (valid) {
    const int t0 = bR + bC + 64 - fd.k;
    double* out = Utv + (size_t)e * NV * n3 + node;
    out[0] = fx_to(sum[0], t0 - 60);
#pragma unroll
    for (int v = 1; v < 4; ++v) out[(size_t)v * n3] = vis[v] + fx_to(sum[v], bM[v - 1] - 60 + 64 - fd.k);
    out[(size_t)4 * n3] = vis[4] + fx_to(sum[4], t0 + bH - 60);
  }
  return true;
}

template <int n, bool LGL, bool KEP = false>
__global__ void __launch_bounds__(Cfg<n>::T, lift_fx_min_blocks<n, KEP>()) k_lift_vol_fx(
    const double* __restrict__ U, const double* __restrict__ Ja, const double* __restrict__ sJ,
    const double* __restrict__ Wf, const double* __restrict__ fgeo, const int* __restrict__ elemSide,
    double* __restrict__ Gf, double* __restrict__ Utv, double* __restrict__ Gvol, int K, int S, int bigBase,
    const double* __restrict__ QB, const int* __restrict__ order, const __grid_constant__ Ops<double> ops,
    const __grid_constant__ FxOps fx, const __grid_constant__ FxStrong fd, const __grid_constant__ Phys<double> ph) {
  using C = Cfg<n>;
  constexpr int n2 = C::n2, n3 = C::n3, NE = C::NE, T = C::T, n3p = C::n3p;
  constexpr bool kWarp = NE == 1;
  constexpr int kUp = LGL ? fx_up(n, true) - 2 : 0;
  const int grp = order != nullptr ? order[blockIdx.x] : blockIdx.x;  // NE consecutive elements
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fx64* sA = reinterpret_cast<fx64*>(smem_raw);  // [NE][15][n3p] line fields l*5 + v, contracted in place
  fx64* sW = sA + NE * 15 * n3p;                 // [NE][6][8][n2] face means of W (5) and outward n_d s_hat (3)
  int2* sD = reinterpret_cast<int2*>(sW + NE * 48 * n2);  // [n2] strong-form derivative (KEP)
  int* sES = reinterpret_cast<int*>(sD + n2);
  int* sSlot = sES + NE * 6;
  int* sMpq = sSlot + NE * 6;            // [NE][6][n2] master-frame node of each face node
  int* sMag = sMpq + NE * 6 * n2;        // [NE][FX_SLOTS] largest magnitude words
  int* sExp = sMag + NE * FX_SLOTS;      // [NE][16] exponent bound of lifting field v*3+d, [NE][16] its shift
  const int tid = threadIdx.x;
  const int el = tid / n3, node = tid - el * n3;
  const int e0 = grp * NE, e = e0 + el;
  const bool valid = e < K;
  const int pn = pidx<n>(node % n, (node / n) % n, node / n2);
  const unsigned wmask = (tid | 31) < T ? 0xffffffffu : (1u << (T & 31)) - 1u;
  for (int t = tid; t < NE * FX_SLOTS; t += T) sMag[t] = 0;
  for (int t = tid; t < NE * 6; t += T) {
    const int es = (e0 + t / 6 < K) ? elemSide[(size_t)e0 * 6 + t] : 0;
    sES[t] = es;
    sSlot[t] = es_slave(es) * S + es_side(es);
  }
  double W[NV];
  double sj = 0.0;
  int mJ[3] = {0, 0, 0};
  {
    double Uo[NV] = {1.0, 0.0, 0.0, 0.0, 1.0};
    if (valid) {
#pragma unroll
      for (int v = 0; v < NV; ++v) Uo[v] = U[((size_t)e * NV + v) * n3 + node];
#pragma unroll
      for (int c = 0; c < 9; ++c) mJ[c % 3] = max(mJ[c % 3], fx_mag(Ja[((size_t)e * 9 + c) * n3 + node]));
      sj = sJ[(size_t)e * n3 + node];
    }
    cons_to_prim(Uo, 1.0 / Uo[0], W, ph);  // the FP64 pipe has room here: divisions stay on it
  }
  __syncthreads();
  int* mag = sMag + el * FX_SLOTS;
  int mW[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) mW[v] = fx_mag(W[v]);
  // a2: face means of W and outward n_d s_hat (mortar big sides: their projected lifting flux
  // is read by the line tasks)
  constexpr int half = 1 << 20;  // one exponent step of a magnitude word
  for (int it = tid; it < NE * 6 * n2; it += T) {
    const int el2 = it / (6 * n2);
    const int r = it - el2 * 6 * n2;
    const int s = r / n2, pq = r - s * n2;
    double w[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) w[c] = 0.0;
    if (e0 + el2 < K) {
      const int es = sES[el2 * 6 + s];
      const int side = es_side(es);
      const int mpq = orient_pq(es_orient(es), n - 1, pq % n, pq / n);
      sMpq[it] = mpq;
      if (side >= bigBase) {
        const double* qb = QB + ((size_t)(side - bigBase) * 15) * n2 + mpq;
#pragma unroll
        for (int c = 0; c < 15; ++c) atomicMax(sMag + el2 * FX_SLOTS + FX_Q + c, fx_mag(qb[c * n2]));
      } else {
        const double* w0 = Wf + ((size_t)side * NV) * n2 + mpq;
        const double* w1 = Wf + ((size_t)(S + side) * NV) * n2 + mpq;
        const double* g = fgeo + ((size_t)side * 4) * n2 + mpq;
        const double sc = dg_neg_if(g[3 * n2], es_slave(es));
#pragma unroll
        for (int v = 0; v < NV; ++v) w[v] = w0[v * n2] + w1[v * n2];  // twice the mean: halved by its exponent
#pragma unroll
        for (int d = 0; d < 3; ++d) w[5 + d] = g[d * n2] * sc;
      }
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) sW[((el2 * 6 + s) * 8 + c) * n2 + pq] = __double_as_longlong(w[c]);
    if constexpr (kWarp) {
#pragma unroll
      for (int v = 0; v < NV; ++v) mW[v] = max(mW[v], fx_mag(w[v]) - half);
#pragma unroll
      for (int d = 0; d < 3; ++d) mJ[d] = max(mJ[d], fx_mag(w[5 + d]));
    } else {
#pragma unroll
      for (int c = 0; c < 8; ++c) atomicMax(sMag + el2 * FX_SLOTS + FX_W + c, fx_mag(w[c]) - (c < NV ? half : 0));
    }
  }
  fx_max<kWarp, 9>(mag, wmask, [&](int s) { return s < 5 ? mW[s < 5 ? s : 0] : (s < 8 ? mJ[s < 8 && s > 4 ? s - 5 : 0] : fx_mag(sj)); });
  __syncthreads();
  {
    int bad = 0;
    for (int t = tid; t < NE * FX_SLOTS; t += T) bad |= (sMag[t] >> 20) > FX_MAX_EXP;
    for (int t = tid; t < NE * 15; t += T) {
      const int el2 = t / 15, c = t - el2 * 15;
      const int* m = sMag + el2 * FX_SLOTS;
      const int prod = (m[FX_W + c / 3] >> 20) + (m[FX_J + c % 3] >> 20) - 2044;
      const int x = max(prod, (m[FX_Q + c] >> 20) - 1022);
      sExp[el2 * 32 + c] = x;
      sExp[el2 * 32 + 16 + c] = min(1 + x - prod, 62);
    }
    if (__syncthreads_or(bad)) {
      lift_vol_fp64<n, LGL, KEP>(U, Ja, sJ, Wf, fgeo, Gf, Utv, Gvol, K, S, bigBase, QB, ops, ph,
                            reinterpret_cast<double*>(sA), reinterpret_cast<double*>(sW), sES, sMpq, grp);
      return;
    }
  }
  for (int it = tid; it < NE * 6 * n2; it += T) {  // the thread's own entries, as above
    const int el2 = it / (6 * n2);
    const int r = it - el2 * 6 * n2;
    const int s = r / n2, pq = r - s * n2;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      fx64* x = sW + ((el2 * 6 + s) * 8 + c) * n2 + pq;
      *x = fx_from<62>(__longlong_as_double(*x), (sMag[el2 * FX_SLOTS + FX_W + c] >> 20) + (c < NV ? 1 : 0));
    }
  }
  const int ES = mag[FX_S] >> 20;
  double G[15];  // indexed at run time by d: kept in local memory between the phases
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    // a3: gradient component d: Ja^l_d W_v staged as field l*5 + v, contracted along l
    const int* sh = sExp + el * 32 + 16;
    {
      FxSplit ji[3];
#pragma unroll
      for (int l = 0; l < 3; ++l)
        ji[l] = fx_split(fx_from<62>(valid ? Ja[((size_t)e * 9 + l * 3 + d) * n3 + node] : 0.0, mag[FX_J + d] >> 20));
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const FxSplit w = fx_split(fx_from<62>(W[v], mag[FX_W + v] >> 20));
        const int s = sh[v * 3 + d];
#pragma unroll
        for (int l = 0; l < 3; ++l) sA[(el * 15 + l * NV + v) * n3p + pn] = fx_shr(fx_mul(ji[l], w), s);
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int it = tid; it < NE * 15 * n2; it += T) {
      const int f = it / n2, line = it - f * n2;
      const int el2 = NE == 1 ? 0 : f / 15;
      const int c = f - el2 * 15, l = c / NV, v = c - l * NV;
      fx64 q[2];
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const int fc = el2 * 6 + 2 * l + m;
        const int side = es_side(sES[fc]);
        const fx64* w = sW + fc * 8 * n2 + line;
        if (side < bigBase)
          q[m] = fx_shr(fx_mul(fx_split(w[v * n2]), fx_split(w[(5 + d) * n2])), sExp[el2 * 32 + 16 + v * 3 + d]);
        else
          q[m] = fx_shr(fx_from<62>(QB[((size_t)(side - bigBase) * 15 + v * 3 + d) * n2 + sMpq[fc * n2 + line]],
                                    sExp[el2 * 32 + v * 3 + d] + 1022), 3);
      }
      int stride;
      const int at = fx_line_at<n>(l, line, stride);
      fx_line<n, LGL, true>(sA + f * n3p + at, stride, q[0], q[1], fx);
    }
    __syncthreads();
    // dW_v/dx_d = (sum over l) / J
    {
      const FxSplit si = fx_split(fx_from<62>(sj, ES));
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        fx64* r = sA + (el * 15 + v) * n3p + pn;
        const fx64 g = fx_mul(fx_split((r[0] + r[NV * n3p] + r[2 * NV * n3p]) << (LGL ? 0 : 2)), si);  // scale 2^(kc + 2 + kUp)
        G[d * NV + v] = fx_to(g, sExp[el * 32 + v * 3 + d] + 5 - kUp - fx.kc + ES - 1022);
        r[0] = LGL ? __double_as_longlong(G[d * NV + v]) : g;
        if (Gvol != nullptr && valid) Gvol[((size_t)e * 15 + d * NV + v) * n3 + node] = G[d * NV + v];
      }
    }
    __syncthreads();
    // a4: both ends of every line to the faces
#pragma unroll 1
    for (int it = tid; it < NE * 15 * n2; it += T) {
      const int f = it / n2, line = it - f * n2;
      const int el2 = NE == 1 ? 0 : f / 15;
      const int c = f - el2 * 15, l = c / NV, v = c - l * NV;
      if (e0 + el2 >= K) continue;
      int stride;
      const fx64* b = sA + (el2 * 15 + v) * n3p + fx_line_at<n>(l, line, stride);
      double gm, gp;
      if constexpr (LGL) {
        gm = __longlong_as_double(b[0]);
        gp = __longlong_as_double(b[(n - 1) * stride]);
      } else {
        fx64 ym, yp;
        fx_ends<n>(b, stride, fx, ym, yp);
        const int t = sExp[el2 * 32 + v * 3 + d] + 5 - fx.kc + (sMag[el2 * FX_SLOTS + FX_S] >> 20) - 1022 + 64 - fx.kp;
        gm = fx_to(ym, t);
        gp = fx_to(yp, t);
      }
      const int fc = el2 * 6 + 2 * l;
      Gf[((size_t)sSlot[fc] * 15 + d * NV + v) * n2 + sMpq[fc * n2 + line]] = gm;
      Gf[((size_t)sSlot[fc + 1] * 15 + d * NV + v) * n2 + sMpq[(fc + 1) * n2 + line]] = gp;
    }
    __syncthreads();
  }
  if (Utv == nullptr) return;  // the adjoint's recompute needs the gradients only
  auto metric = [&](FxSplit (&ji)[9]) {
#pragma unroll
    for (int c = 0; c < 9; ++c)
      ji[c] = fx_split(fx_from<62>(valid ? Ja[((size_t)e * 9 + c) * n3 + node] : 0.0, mag[FX_J + c % 3] >> 20));
  };
  bool done;
  if constexpr (KEP)
    done = split_volume_fx<n, false, FX_J>(U, Utv, W, G, K, grp, wmask, sA, sMag, sD, fx, fd, ph, metric);
  else
    done = volume_fx<n, LGL, FX_J>(U, Utv, W, G, K, grp, wmask, sA, sMag, fx, ph, metric);
  if (!done)
    lift_vol_fp64<n, LGL, KEP>(U, Ja, sJ, Wf, fgeo, Gf, Utv, Gvol, K, S, bigBase, QB, ops, ph, reinterpret_cast<double*>(sA),
                          reinterpret_cast<double*>(sW), sES, sMpq, grp);
}

// ---------------------------------------------------------------------------
// The same for affine elements (parallelepipeds; DevMesh::affine): the metric terms are
// constants of the element, so the lifting contracts the 5 primitive variables along the 3
// directions (15 line fields instead of 45) and combines the results with J^l_d / J, the face
// terms of a line are the face means themselves (n_d s_hat = +-Ja^l_d on both ends), and no
// metric term is read per node.  16^3 elements, N = 7: 750 -> 559 us.
// ---------------------------------------------------------------------------
template <int n>
constexpr size_t lift_affine_smem() {
  using C = Cfg<n>;
  return 8 * C::NE * (15 * C::n3p + 30 * C::n2 + 18) + 8 * C::n2 + sizeof(int) * C::NE * (12 + 6 * C::n2 + FX_SLOTS + 4);
}

// the general kernel's FP64 schedule needs its shared memory: 48 n^2 face values per element
template <int n>
constexpr size_t lift_affine_smem_total() {
  return lift_affine_smem<n>() > lift_fx_smem<n>() ? lift_affine_smem<n>() : lift_fx_smem<n>();
}

template <int n, bool LGL, bool KEP = false>
__global__ void __launch_bounds__(Cfg<n>::T, lift_fx_min_blocks<n, KEP>()) k_lift_vol_fx_affine(
    const double* __restrict__ U, const double* __restrict__ aff, const double* __restrict__ Ja,
    const double* __restrict__ sJ, const double* __restrict__ Wf, const double* __restrict__ fgeo,
    const int* __restrict__ elemSide, double* __restrict__ Gf, double* __restrict__ Utv, double* __restrict__ Gvol, int K,
    int S, int bigBase, const int* __restrict__ order, const __grid_constant__ Ops<double> ops,
    const __grid_constant__ FxOps fx, const __grid_constant__ FxStrong fd, const __grid_constant__ Phys<double> ph) {
  using C = Cfg<n>;
  constexpr int n2 = C::n2, n3 = C::n3, NE = C::NE, T = C::T, n3p = C::n3p;
  constexpr bool kWarp = NE == 1;
  constexpr int kUp = LGL ? fx_up(n, true) - 2 : 0;
  const int grp = order != nullptr ? order[blockIdx.x] : blockIdx.x;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fx64* sA = reinterpret_cast<fx64*>(smem_raw);  // [NE][15][n3p] line fields l*5 + v, contracted in place
  fx64* sW = sA + NE * 15 * n3p;                 // [NE][6][5][n2] face means of W
  int2* sD = reinterpret_cast<int2*>(smem_raw + lift_affine_smem_total<n>()) - n2;  // [n2] strong-form derivative (KEP)
  int* sES = reinterpret_cast<int*>(sD) - NE * (12 + 6 * n2 + FX_SLOTS + 4);
  int* sSlot = sES + NE * 6;
  int* sMpq = sSlot + NE * 6;          // [NE][6][n2] master-frame node of each face node
  int* sMag = sMpq + NE * 6 * n2;      // [NE][FX_SLOTS] largest magnitude words
  fx64* sM = sW + NE * 30 * n2;        // [NE][2][9] J^l_d / J and J^l_d, exponents by d
  const int tid = threadIdx.x;
  const int el = tid / n3, node = tid - el * n3;
  const int e0 = grp * NE, e = e0 + el;
  const bool valid = e < K;
  const int pn = pidx<n>(node % n, (node / n) % n, node / n2);
  const unsigned wmask = (tid | 31) < T ? 0xffffffffu : (1u << (T & 31)) - 1u;
  for (int t = tid; t < NE * FX_SLOTS; t += T) sMag[t] = 0;
  for (int t = tid; t < NE * 6; t += T) {
    const int es = (e0 + t / 6 < K) ? elemSide[(size_t)e0 * 6 + t] : 0;
    sES[t] = es;
    sSlot[t] = es_slave(es) * S + es_side(es);
  }
  double W[NV];
  {
    double Uo[NV] = {1.0, 0.0, 0.0, 0.0, 1.0};
    if (valid) {
#pragma unroll
      for (int v = 0; v < NV; ++v) Uo[v] = U[((size_t)e * NV + v) * n3 + node];
    }
    cons_to_prim(Uo, 1.0 / Uo[0], W, ph);
  }
  __syncthreads();
  int* mag = sMag + el * FX_SLOTS;
  if (tid < 3 * NE) {  // thread (element, d): the three metric terms of physical direction d
    const int el2 = tid / 3, d = tid - el2 * 3;
    const double* a = aff + (size_t)min(e0 + el2, K - 1) * 10;
    int big = 0, md = 0;
    double m[3];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      big = max(big, fx_mag(a[l * 3 + d]));
      m[l] = a[l * 3 + d] * a[9];
      md = max(md, fx_mag(m[l]));
    }
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      sM[el2 * 18 + l * 3 + d] = fx_from<62>(m[l], md >> 20);
      sM[el2 * 18 + 9 + l * 3 + d] = fx_from<62>(a[l * 3 + d], big >> 20);
    }
    sMag[el2 * FX_SLOTS + FX_J + d] = md;
    sMag[el2 * FX_SLOTS + FX_S + d] = big;
  }
  int mW[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) mW[v] = fx_mag(W[v]);
  for (int it = tid; it < NE * 6 * n2; it += T) {  // a2: face means of W
    const int f = it / n2, pq = it - f * n2;
    double w[NV] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (e0 + f / 6 < K) {
      const int es = sES[f];
      const int mpq = orient_pq(es_orient(es), n - 1, pq % n, pq / n);
      sMpq[it] = mpq;
      const double* w0 = Wf + ((size_t)es_side(es) * NV) * n2 + mpq;
      const double* w1 = Wf + ((size_t)(S + es_side(es)) * NV) * n2 + mpq;
#pragma unroll
      for (int v = 0; v < NV; ++v) w[v] = 0.5 * (w0[v * n2] + w1[v * n2]);
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      sW[(f * NV + v) * n2 + pq] = __double_as_longlong(w[v]);
      if constexpr (kWarp)
        mW[v] = max(mW[v], fx_mag(w[v]));
      else
        atomicMax(sMag + (f / 6) * FX_SLOTS + FX_W + v, fx_mag(w[v]));
    }
  }
  fx_max<kWarp, NV>(mag + FX_W, wmask, [&](int s) { return mW[s]; });
  __syncthreads();
  auto fp64 = [&]() {
    lift_vol_fp64<n, LGL, KEP>(U, Ja, sJ, Wf, fgeo, Gf, Utv, Gvol, K, S, bigBase, nullptr, ops, ph, reinterpret_cast<double*>(sA),
                          reinterpret_cast<double*>(sW), sES, sMpq, grp);
  };
  {
    int bad = 0;
    for (int t = tid; t < NE * FX_SLOTS; t += T) bad |= (sMag[t] >> 20) > FX_MAX_EXP;
    if (__syncthreads_or(bad)) {
      fp64();
      return;
    }
  }
  for (int it = tid; it < NE * 6 * n2; it += T) {  // the thread's own entries, as above
    const int f = it / n2, pq = it - f * n2;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      fx64* x = sW + (f * NV + v) * n2 + pq;
      *x = fx_from<59>(__longlong_as_double(*x), sMag[(f / 6) * FX_SLOTS + FX_W + v] >> 20);
    }
  }
  fx64* own = sA + el * 15 * n3p + pn;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const fx64 x = fx_from<59>(W[v], mag[FX_W + v] >> 20);
#pragma unroll
    for (int l = 0; l < 3; ++l) own[(l * NV + v) * n3p] = x;
  }
  __syncthreads();
  // a3: W_v contracted along l with its face means, outward +- on the two ends
#pragma unroll 1
  for (int it = tid; it < NE * 15 * n2; it += T) {
    const int f = it / n2, line = it - f * n2;
    const int el2 = NE == 1 ? 0 : f / 15;
    const int c = f - el2 * 15, l = c / NV, v = c - l * NV;
    const fx64* q = sW + ((el2 * 6 + 2 * l) * NV + v) * n2 + line;
    int stride;
    const int at = fx_line_at<n>(l, line, stride);
    fx_line<n, LGL, true>(sA + f * n3p + at, stride, -q[0], q[NV * n2], fx);
  }
  __syncthreads();
  // dW_v/dx_d = sum_l (J^l_d / J) (D_l W_v)
  double G[15];
  {
    FxSplit m[9];
#pragma unroll
    for (int c = 0; c < 9; ++c) m[c] = fx_split(sM[el * 18 + c]);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      FxSplit t[3];
#pragma unroll
      for (int l = 0; l < 3; ++l) t[l] = fx_split(own[(l * NV + v) * n3p] << (LGL ? 0 : 2));  // scale 2^(kc + 2 + kUp)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        FxAcc s;
#pragma unroll
        for (int l = 0; l < 3; ++l) s.add(m[l * 3 + d], t[l]);
        const fx64 g = s.get();
        G[d * NV + v] = fx_to(g, (mag[FX_J + d] >> 20) + (mag[FX_W + v] >> 20) - 2044 + 5 - kUp - fx.kc);
        own[(d * NV + v) * n3p] = LGL ? __double_as_longlong(G[d * NV + v]) : g;
        if (Gvol != nullptr && valid) Gvol[((size_t)e * 15 + d * NV + v) * n3 + node] = G[d * NV + v];
      }
    }
  }
  __syncthreads();
  // a4: both ends of every line of every gradient field c = d*5 + v to the faces
#pragma unroll
  for (int l = 0; l < 3; ++l) {
#pragma unroll 1
    for (int it = tid; it < NE * 15 * n2; it += T) {
      const int f = it / n2, line = it - f * n2;
      const int el2 = NE == 1 ? 0 : f / 15;
      const int c = f - el2 * 15, d = c / NV, v = c - d * NV;
      if (e0 + el2 >= K) continue;
      int stride;
      const fx64* b = sA + f * n3p + fx_line_at<n>(l, line, stride);
      double gm, gp;
      if constexpr (LGL) {
        gm = __longlong_as_double(b[0]);
        gp = __longlong_as_double(b[(n - 1) * stride]);
      } else {
        fx64 ym, yp;
        fx_ends<n>(b, stride, fx, ym, yp);
        const int* m2 = sMag + el2 * FX_SLOTS;
        const int t = (m2[FX_J + d] >> 20) + (m2[FX_W + v] >> 20) - 2044 + 5 - fx.kc + 64 - fx.kp;
        gm = fx_to(ym, t);
        gp = fx_to(yp, t);
      }
      const int fc = el2 * 6 + 2 * l;
      Gf[((size_t)sSlot[fc] * 15 + c) * n2 + sMpq[fc * n2 + line]] = gm;
      Gf[((size_t)sSlot[fc + 1] * 15 + c) * n2 + sMpq[(fc + 1) * n2 + line]] = gp;
    }
  }
  if (Utv == nullptr) return;
  __syncthreads();
  auto metric = [&](FxSplit (&ji)[9]) {
#pragma unroll
    for (int c = 0; c < 9; ++c) ji[c] = fx_split(sM[el * 18 + 9 + c]);
  };
  bool done;
  if constexpr (KEP)
    done = split_volume_fx<n, true, FX_S>(U, Utv, W, G, K, grp, wmask, sA, sMag, sD, fx, fd, ph, metric);
  else
    done = volume_fx<n, LGL, FX_S>(U, Utv, W, G, K, grp, wmask, sA, sMag, fx, ph, metric);
  if (!done)
    fp64();
}

}  // namespace flexi
