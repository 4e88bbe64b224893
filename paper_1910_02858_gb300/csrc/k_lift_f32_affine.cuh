// Lifting and volume integral of the FP32 forms on affine elements (parallelepipeds;
// DevMesh::affine).  Standard volume integral, BR1.
//
// lift_vol_body's FP32 form is bound by instruction issue (1,935 per node at n = 8): 45 of its
// 60 line contractions are the lifting of Ja^l_d W.  With constant metric terms the lifting
// contracts the five primitive variables along the three directions (15 line fields, face
// terms = the face means themselves) and combines them with J^l_d / J; the ten metric values
// per node are not read; and every contraction is done in one pass over all 15 line fields
// with the even-odd split of the operators (half the products), into separate results per
// direction.  SW 1 / 2: the contractions on tensor cores in three-term TF32 / BF16 splits
// (k_tc.cuh), one pass instead of nine, the face terms in the idle columns of the product for n <= 6.
// 16^3 elements, N = 7: 163 -> 102 us (FP32); 32^3, N = 5: 540 -> 330 us (FP32); TF32 19 x 23 x 17, N = 5:
// 283 -> 166 us.
#pragma once
#include "k_tc.cuh"
#include "launch.h"

namespace flexi {

// one line from src to dst by the even-odd split (EvenOdd, launch.h)
template <int n, bool LGL, bool FACE>
__device__ __forceinline__ void eo_line(const float* src, float* dst, int stride, float qm,
                                        float qp, const EvenOdd& o) {
  constexpr int h = n / 2, c = (n + 1) / 2, N = n - 1;
  float e[c], d[h];
#pragma unroll
  for (int a = 0; a < h; ++a) {
    const float x = src[a * stride], y = src[(N - a) * stride];
    e[a] = x + y;
    d[a] = x - y;
  }
  if constexpr (n & 1) e[c - 1] = src[(c - 1) * stride];
  const float qs = qp + qm, qd = qp - qm;
#pragma unroll
  for (int i = 0; i < c; ++i) {
    const bool face = FACE && (!LGL || i == 0);
    float O = face ? o.s[i] * qs : 0.0f;
#pragma unroll
    for (int a = 0; a < h; ++a) O = fmaf(o.o[i][a], d[a], O);
    if (i < h) {
      float E = face ? o.t[i] * qd : 0.0f;
#pragma unroll
      for (int a = 0; a < c; ++a) E = fmaf(o.e[i][a], e[a], E);
      dst[i * stride] = O + E;
      dst[(N - i) * stride] = O - E;
    } else {
      dst[i * stride] = O;
    }
  }
}

// Tensor-core contraction of the 15 line fields of every element along their directions, in
// place: a warp's 16 lines are read, multiplied and written back.  AUG (n <= 6): columns n and
// n + 1 of a line hold its face values -q(-l), q(+l) against l_hat in the operator (else zeros).
// Ends synced.
template <int n, int NE, int SW, bool AUG>
__device__ __forceinline__ void tc_lines(float* __restrict__ buf, const float* __restrict__ sQ, const BFrag<SW>& bf, int tid,
                                         int T) {
  constexpr int n2 = n * n, n3p = Cfg<n>::n3p, P = Cfg<n>::P;
  constexpr int L = NE * 15 * n2, tiles = (L + 15) / 16;
  const int warp = tid >> 5, lane = tid & 31, nwarps = T >> 5;
  const int gid = lane >> 2, tig = lane & 3;
  if (warp < nwarps) {
#pragma unroll 1
    for (int tile = warp; tile < tiles; tile += nwarps) {
      int base[2], stride[2], face[2];
      bool ok[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int g = tile * 16 + gid + 8 * h;
        ok[h] = g < L;
        const int gg = ok[h] ? g : 0;
        const int f = gg / n2, line = gg - f * n2;
        const int el = f / 15, c = f - el * 15, l = c / NV, v = c - l * NV;
        const int a0 = line % n, a1 = line / n;
        stride[h] = l == 0 ? 1 : (l == 1 ? P : P * n);
        base[h] = f * n3p + (l == 0 ? P * line : (l == 1 ? a0 + P * n * a1 : a0 + P * a1));
        face[h] = ((el * 6 + 2 * l) * NV + v) * n2 + line;
      }
      auto Aval = [&](int h, int a) -> float {
        if (!ok[h]) return 0.f;
        if (a < n) return buf[base[h] + stride[h] * a];
        if (AUG && a == n) return -sQ[face[h]];
        if (AUG && a == n + 1) return sQ[face[h] + NV * n2];
        return 0.f;
      };
      float c[4] = {0.f, 0.f, 0.f, 0.f};
      tc_product<SW>(Aval, bf, tig, c);
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int cc = 0; cc < 2; ++cc)
          if (ok[h] && 2 * tig + cc < n) buf[base[h] + stride[h] * (2 * tig + cc)] = c[2 * h + cc];
    }
  }
  __syncthreads();
}

template <int n, int SW>
constexpr size_t lift_f32_affine_smem() {
  using C = Cfg<n>;
  return sizeof(float) * (C::NE * ((SW == 0 ? 20 : 15) * C::n3p + 30 * C::n2) + (SW ? C::n2 + 4 * n : 0)) +
         sizeof(int) * (C::NE * (12 + 6 * C::n2));
}

template <int n, int SW>
constexpr int lift_f32_affine_min_blocks() { return n == 8 ? 2 : (n == 7 ? 3 : (n == 6 ? 5 : 6)); }

template <int n, int SW, bool LGL>
__global__ void __launch_bounds__(Cfg<n>::T, lift_f32_affine_min_blocks<n, SW>()) k_lift_vol_f32_affine(
    const float* __restrict__ U, const float* __restrict__ aff, const float* __restrict__ Wf,
    const int* __restrict__ elemSide, float* __restrict__ Gf, float* __restrict__ Utv, float* __restrict__ Gvol, int K, int S,
    const int* __restrict__ order, const __grid_constant__ Ops<float> ops, const __grid_constant__ EvenOdd eo,
    const __grid_constant__ Phys<float> ph) {
  using C = Cfg<n>;
  constexpr int n2 = C::n2, n3 = C::n3, NE = C::NE, T = C::T, n3p = C::n3p, P = C::P;
  constexpr bool kAug = SW != 0 && n <= 6;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* sT = reinterpret_cast<float*>(smem_raw);  // [NE][15][n3p] line fields l*5 + v; gradients d*5 + v; fluxes
  float* sQ = sT + NE * 15 * n3p;                  // [NE][6][5][n2] face means of W
  float* sWv = sQ + NE * 30 * n2;                  // SW 0: [NE][5][n3p] W
  float* sOp = sWv;                                // SW: DhatT, lm, lp, lhm, lhp
  int* sSlot = reinterpret_cast<int*>(sWv + (SW == 0 ? NE * NV * n3p : n2 + 4 * n));
  int* sES = sSlot + NE * 6;
  int* sMpq = sES + NE * 6;  // [NE][6][n2]
  const int tid = threadIdx.x;
  const int grp = order != nullptr ? order[blockIdx.x] : blockIdx.x;
  const int el = tid / n3, node = tid - el * n3;
  const int e0 = grp * NE, e = e0 + el;
  const bool valid = e < K;
  const int i = node % n, j = (node / n) % n, k = node / n2;
  const int pn = pidx<n>(i, j, k);
  float* own = sT + el * 15 * n3p + pn;
  if constexpr (SW != 0) load_ops<float, n>(sOp, ops, tid, T);
  for (int t = tid; t < NE * 6; t += T) {
    const int es = (e0 + t / 6 < K) ? elemSide[(size_t)e0 * 6 + t] : 0;
    sES[t] = es;
    sSlot[t] = es_slave(es) * S + es_side(es);
  }
  float Uo[NV] = {1.f, 0.f, 0.f, 0.f, 1.f}, W[NV];
  if (valid) {
#pragma unroll
    for (int v = 0; v < NV; ++v) Uo[v] = U[((size_t)e * NV + v) * n3 + node];
  }
  const float ir = 1.0f / Uo[0];
  cons_to_prim(Uo, ir, W, ph);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    if constexpr (SW == 0) {
      sWv[(el * NV + v) * n3p + pn] = W[v];
    } else {
#pragma unroll
      for (int l = 0; l < 3; ++l) own[(l * NV + v) * n3p] = W[v];
    }
  }
  __syncthreads();
  for (int it = tid; it < NE * 6 * n2; it += T) {  // a2: face means of W
    const int f = it / n2, pq = it - f * n2;
    if (e0 + f / 6 >= K) continue;
    const int es = sES[f];
    const int mpq = orient_pq(es_orient(es), n - 1, pq % n, pq / n);
    sMpq[it] = mpq;
    const float* w0 = Wf + ((size_t)es_side(es) * NV) * n2 + mpq;
    const float* w1 = Wf + ((size_t)(S + es_side(es)) * NV) * n2 + mpq;
#pragma unroll
    for (int v = 0; v < NV; ++v) sQ[(f * NV + v) * n2 + pq] = 0.5f * (w0[v * n2] + w1[v * n2]);
  }
  float m[9], sj;
  {
    const float* a = aff + (size_t)min(e, K - 1) * 10;
    sj = a[9];
#pragma unroll
    for (int c = 0; c < 9; ++c) m[c] = a[c];
  }
  __syncthreads();
  // a3: W_v contracted along l with its face means
  BFrag<SW> bfr;
  if constexpr (SW == 0) {
#pragma unroll 1
    for (int it = tid; it < NE * 15 * n2; it += T) {
      const int f = it / n2, line = it - f * n2;
      const int el2 = NE == 1 ? 0 : f / 15;
      const int c = f - el2 * 15, l = c / NV, v = c - l * NV;
      const int a0 = line % n, a1 = line / n;
      const int stride = l == 0 ? 1 : (l == 1 ? P : P * n);
      const int base = l == 0 ? P * line : (l == 1 ? a0 + P * n * a1 : a0 + P * a1);
      const float* q = sQ + ((el2 * 6 + 2 * l) * NV + v) * n2 + line;
      eo_line<n, LGL, true>(sWv + (el2 * NV + v) * n3p + base, sT + f * n3p + base, stride, -q[0], q[NV * n2], eo);
    }
    __syncthreads();
  } else {
    bfr = make_bfrag<n, SW, kAug>(sOp, tid & 31);
    tc_lines<n, NE, SW, kAug>(sT, sQ, bfr, tid, T);
  }
  // dW_v/dx_d = sum_l (J^l_d / J) (D_l W_v)
  float G[15];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    float t[3];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      t[l] = own[(l * NV + v) * n3p];
      if constexpr (SW != 0 && !kAug) {  // face terms
        const int x = l == 0 ? i : (l == 1 ? j : k), pq = l == 0 ? j + n * k : (l == 1 ? i + n * k : i + n * j);
        const float* q = sQ + ((el * 6 + 2 * l) * NV + v) * n2 + pq;
        const float* lh = sOp + n2 + 2 * n;
        t[l] = fmaf(lh[n + x], q[NV * n2], fmaf(-lh[x], q[0], t[l]));
      }
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) G[d * NV + v] = (m[d] * t[0] + m[3 + d] * t[1] + m[6 + d] * t[2]) * sj;
#pragma unroll
    for (int d = 0; d < 3; ++d) own[(d * NV + v) * n3p] = G[d * NV + v];
  }
  if (Gvol != nullptr && valid) {
#pragma unroll
    for (int c = 0; c < 15; ++c) Gvol[((size_t)e * 15 + c) * n3 + node] = G[c];
  }
  __syncthreads();
  // a4: both ends of every line of every gradient field to the faces
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    constexpr int step = NE == 1 ? T / n2 : 1;
    const int stride = l == 0 ? 1 : (l == 1 ? P : P * n);
    auto ends = [&](const float* b, float& gm, float& gp) {
      if constexpr (LGL) {
        gm = b[0];
        gp = b[(n - 1) * stride];
      } else {
        float e = 0.f, o = 0.f;
        constexpr int h = n / 2;
#pragma unroll
        for (int a = 0; a < h; ++a) {
          const float x = b[a * stride], y = b[(n - 1 - a) * stride];
          e = fmaf(eo.pe[a], x + y, e);
          o = fmaf(eo.po[a], x - y, o);
        }
        if constexpr (n & 1) e = fmaf(eo.pe[h], b[h * stride], e);
        gm = e - o;
        gp = e + o;
      }
    };
    if constexpr (NE == 1) {  // a thread's tasks share their line: slots and face nodes read once
      const int line = tid % n2;
      const int a0 = line % n, a1 = line / n;
      const int base = l == 0 ? P * line : (l == 1 ? a0 + P * n * a1 : a0 + P * a1);
      float* gm_out = Gf + (size_t)sSlot[2 * l] * 15 * n2 + sMpq[(2 * l) * n2 + line];
      float* gp_out = Gf + (size_t)sSlot[2 * l + 1] * 15 * n2 + sMpq[(2 * l + 1) * n2 + line];
#pragma unroll 1
      for (int c = tid / n2; c < 15; c += step) {
        float gm, gp;
        ends(sT + c * n3p + base, gm, gp);
        gm_out[c * n2] = gm;
        gp_out[c * n2] = gp;
      }
    } else {
#pragma unroll 1
      for (int it = tid; it < NE * 15 * n2; it += T) {
        const int f = it / n2, line = it - f * n2;
        const int el2 = f / 15, c = f - el2 * 15;
        if (e0 + el2 >= K) continue;
        const int a0 = line % n, a1 = line / n;
        float gm, gp;
        ends(sT + f * n3p + (l == 0 ? P * line : (l == 1 ? a0 + P * n * a1 : a0 + P * a1)), gm, gp);
        const int fc = el2 * 6 + 2 * l;
        Gf[((size_t)sSlot[fc] * 15 + c) * n2 + sMpq[fc * n2 + line]] = gm;
        Gf[((size_t)sSlot[fc + 1] * 15 + c) * n2 + sMpq[(fc + 1) * n2 + line]] = gp;
      }
    }
  }
  // a6: contravariant fluxes
  float F[3][NV];
#pragma unroll
  for (int d = 0; d < 3; ++d) flux_total(Uo, W, ir, G, d, ph, F[d]);
  __syncthreads();
#pragma unroll
  for (int l = 0; l < 3; ++l)
#pragma unroll
    for (int v = 0; v < NV; ++v)
      own[(l * NV + v) * n3p] = m[l * 3] * F[0][v] + m[l * 3 + 1] * F[1][v] + m[l * 3 + 2] * F[2][v];
  __syncthreads();
  // a7: volume integral, in place per direction
  if constexpr (SW == 0) {
#pragma unroll 1
    for (int it = tid; it < NE * 15 * n2; it += T) {
      const int f = it / n2, line = it - f * n2;
      const int l = (NE == 1 ? f : f % 15) / NV;
      const int a0 = line % n, a1 = line / n;
      float* b = sT + f * n3p + (l == 0 ? P * line : (l == 1 ? a0 + P * n * a1 : a0 + P * a1));
      eo_line<n, LGL, false>(b, b, l == 0 ? 1 : (l == 1 ? P : P * n), 0.f, 0.f, eo);
    }
    __syncthreads();
  } else {
    tc_lines<n, NE, SW, false>(sT, sQ, bfr, tid, T);
  }
  if (valid) {
#pragma unroll
    for (int v = 0; v < NV; ++v)
      Utv[((size_t)e * NV + v) * n3 + node] = own[v * n3p] + own[(NV + v) * n3p] + own[(2 * NV + v) * n3p];
  }
}

}  // namespace flexi
