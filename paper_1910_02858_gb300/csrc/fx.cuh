// Block fixed-point arithmetic of the FP64 form's line contractions.
//
// On this chip an FP64 warp instruction holds its SM sub-partition for 64 clocks
// (measured: 64.4 DFMA, 76 DADD), a 32 x 32 -> 64 bit integer multiply-add
// (IMAD.WIDE) for 2.2 and the other integer instructions for 1-2.  The D_hat and
// l_hat contractions and the metric products are sums of products whose terms
// share a scale, so they run on the integer pipes: the values of a field of one
// element become 58-61 bit integers under one power of two (the field's largest
// magnitude), the operators 58-60 bit integers, every product keeps its leading
// 60 bits from three 32 x 32 multiply-adds (the product of the two low halves is
// below the last kept bit), and sums are exact.  The quantum is 2^-57 of the
// field's largest value or less, against the 2^-53 to which FP64 rounds every
// partial sum.  Terms of one sum that differ by more than their shared scale allows
// (fluxes and metric terms of flat elements, rows of D_hat on Gauss-Lobatto nodes,
// gradients of a shear layer) have exponents of their own and meet at the largest
// product: the rounding noise of a right-hand side is 0.1 to 1.02 times that with
// FP64 sums, over N = 2..7, both node sets, curved elements and aspect ratios to 4096.
// The error is relative to the element's largest value of a field: lines on which
// the field is everywhere below 2^-6 of that keep fewer digits than FP64 would.
#pragma once
#include <cmath>
#include <cstring>

#include "dg_common.cuh"

namespace flexi {

constexpr int FXH = MAXN / 2;

// One-dimensional operators in fixed point, split by the symmetry of the node sets
// (Dhat[N-i][N-a] = -Dhat[i][a], l_hat_i(-1) = l_hat_{N-i}(+1)): with e_a = x_a + x_{N-a},
// o_a = x_a - x_{N-a} (e_h = x_h at the middle node), q_s = q(+1) + q(-1) and
// q_d = q(+1) - q(-1),
//   y_i = E_i + O_i, y_{N-i} = O_i - E_i,
//   E_i = sum_a DE_ia e_a + t_i q_d,  O_i = sum_a DO_ia o_a + s_i q_s,
// which halves the multiply-adds.  An entry c is stored as round(c 2^kc) = h 2^32 + l,
// |l| <= 2^31, with kc the largest for which every row's sum of magnitudes stays below 2^62.
// Gauss-Lobatto: the rows of the inner nodes are 5.3 to 9.8 times smaller than the first one, so
// their scale is 2^(kc + fx_up), and fx_line<LGL> brings the ends' results to it.
constexpr int fx_up(int n, bool lgl) {
  return !lgl ? 0 : (n == 6 || n == 8 ? 3 : 2);  // the most for which the sums over three lines stay in range
}

struct FxOps {
  int eh[FXH][FXH], el[FXH][FXH];  // DE[i][a], i < n/2, a < (n+1)/2
  int oh[FXH][FXH], ol[FXH][FXH];  // DO[i][a], i < (n+1)/2, a < n/2
  int sh[FXH], sl[FXH], th[FXH], tl[FXH];
  int peh[FXH], pel[FXH], poh[FXH], pol[FXH];  // prolongation to the line's ends, scale 2^kp
  int lh[MAXN], ll[MAXN];  // l_hat_i(+1), scale 2^kl (l_hat_i(-1) is the entry of N - i)
  int kc, kp, kl;
};

// Strong-form derivative D[i][a], a != i, of the Lobatto nodes at a*n + i (split forms): scale 2^k in
// the end rows, the largest for which their sums of magnitudes stay below 2^62, and 2^(k + 2) in the
// others (sums below 2^62.21: with operands below 2^60.6 both accumulators of FxAcc hold n - 1 products)
struct FxStrong {
  int h[MAXN * MAXN], l[MAXN * MAXN];
  int k;
};
inline FxStrong make_fx_strong(const Ops<double>& o, int n) {
  FxStrong f;
  std::memset(&f, 0, sizeof(f));
  double row = 0;
  for (int i = 0; i < n; i += n - 1) {
    double s = 0;
    for (int a = 0; a < n; ++a) s += a == i ? 0.0 : std::fabs(o.DT[a * n + i]);
    row = std::fmax(row, s);
  }
  int x;
  std::frexp(row * (1 + 1e-12), &x);
  f.k = 62 - x;
  for (int t = 0; t < n * n; ++t) {
    const bool end = t % n == 0 || t % n == n - 1;
    const long long v = std::llrint(std::ldexp(o.DT[t], f.k + (end ? 0 : 2)));
    f.l[t] = (int)(unsigned)(v & 0xffffffffll);
    f.h[t] = (int)((v - f.l[t]) / (1ll << 32));
  }
  return f;
}

// host construction from the FP64 operators (integer rounding of scaled doubles: the
// same on every machine)
inline FxOps make_fx_ops(const Ops<double>& o, int n, bool lgl) {
  FxOps f;
  std::memset(&f, 0, sizeof(f));
  const int N = n - 1, h = n / 2, c = (n + 1) / 2, up = fx_up(n, lgl);
  double row = 0, prow = 0, pe = 0, po = 0;
  for (int i = 0; i < n; ++i) {
    double e = 0.5 * std::fabs(o.lhp[i] - o.lhm[i]), d = 0.5 * std::fabs(o.lhp[i] + o.lhm[i]);
    for (int a = 0; a < c; ++a) {
      const double x = o.DhatT[a * n + i], y = 2 * a == N ? x : o.DhatT[(N - a) * n + i];
      e += 0.5 * std::fabs(x + y);
      d += 0.5 * std::fabs(x - y);
    }
    row = std::fmax(row, std::fmax(e, d));
  }
  for (int a = 0; a < c; ++a) {
    pe += 2 * a == N ? std::fabs(o.lp[a]) : 0.5 * std::fabs(o.lp[a] + o.lm[a]);
    po += 0.5 * std::fabs(o.lp[a] - o.lm[a]);
  }
  prow = std::fmax(pe, po);
  int x;
  std::frexp(row * (1 + 1e-12), &x);
  f.kc = 62 - x;
  std::frexp(prow * (1 + 1e-12), &x);
  f.kp = 62 - x;
  auto split = [](long long v, int& hi, int& lo) {
    lo = (int)(unsigned)(v & 0xffffffffll);
    hi = (int)((v - lo) / (1ll << 32));
  };
  // the operators' symmetric means: A = 2^(kc - 1) times twice the entry, halved below
  auto A = [&](int i, int a) {
    const int k = f.kc - 2 + (i > 0 && i < N ? up : 0);
    return std::llrint(std::ldexp(o.DhatT[a * n + i], k)) - std::llrint(std::ldexp(o.DhatT[(N - a) * n + N - i], k));
  };
  auto Q = [&](int i) {
    const int k = f.kc - 2 + (i > 0 && i < N ? up : 0);
    return std::llrint(std::ldexp(o.lhp[i], k)) + std::llrint(std::ldexp(o.lhm[N - i], k));
  };
  auto L = [&](int a) {
    return std::llrint(std::ldexp(o.lp[a], f.kp - 2)) + std::llrint(std::ldexp(o.lm[N - a], f.kp - 2));
  };
  for (int i = 0; i < h; ++i) {
    for (int a = 0; a < c; ++a) split(2 * a == N ? 2 * A(i, a) : A(i, a) + A(i, N - a), f.eh[i][a], f.el[i][a]);
    split(Q(i) - Q(N - i), f.th[i], f.tl[i]);
  }
  for (int i = 0; i < c; ++i) {
    for (int a = 0; a < h; ++a) split(A(i, a) - A(i, N - a), f.oh[i][a], f.ol[i][a]);
    split(Q(i) + Q(N - i), f.sh[i], f.sl[i]);
  }
  double lmax = 0;
  for (int i = 0; i < n; ++i) lmax = std::fmax(lmax, std::fmax(std::fabs(o.lhp[i]), std::fabs(o.lhm[i])));
  std::frexp(lmax * (1 + 1e-12), &x);
  f.kl = 62 - x;
  for (int i = 0; i < n; ++i)
    split(std::llrint(std::ldexp(o.lhp[i], f.kl - 1)) + std::llrint(std::ldexp(o.lhm[N - i], f.kl - 1)), f.lh[i], f.ll[i]);
  for (int a = 0; a < c; ++a) split(2 * a == N ? 2 * L(a) : L(a) + L(N - a), f.peh[a], f.pel[a]);
  for (int a = 0; a < h; ++a) split(L(a) - L(N - a), f.poh[a], f.pol[a]);
  return f;
}

// the transposed operators: Dhat^T as the line contraction, l_hat(+-1) as the end values and
// l(+-1) as the values spread from the ends (lh, ll)
inline FxOps make_fx_ops_transposed(const Ops<double>& o, int n) {
  Ops<double> t = o;
  for (int i = 0; i < n; ++i) {
    for (int a = 0; a < n; ++a) t.DhatT[a * n + i] = o.DhatT[i * n + a];
    t.lm[i] = o.lhm[i];
    t.lp[i] = o.lhp[i];
    t.lhm[i] = o.lm[i];
    t.lhp[i] = o.lp[i];
  }
  return make_fx_ops(t, n, false);
}

// ---------------------------------------------------------------------------
// device primitives
// ---------------------------------------------------------------------------
using fx64 = long long;

// c + a b with 32-bit signed a, b (IMAD.WIDE; written out because the compiler otherwise
// sign-extends operands from the constant bank and multiplies 64 x 64 bits)
__device__ __forceinline__ fx64 fx_mad(int a, int b, fx64 c) {
  fx64 r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// magnitude word: ordered like |x|, its exponent field is x's (NaN and infinities 2047)
__device__ __forceinline__ int fx_mag(double x) { return __double2hiint(x) & 0x7fffffff; }

// x 2^(B - (E - 1022)) for |x| < 2^(E - 1022), E a biased exponent field, B >= 53; truncated
template <int B>
__device__ __forceinline__ fx64 fx_from(double x, int E) {
  const int hi = __double2hiint(x);
  const int ex = (hi >> 20) & 0x7ff;
  const unsigned mh = (unsigned)(hi & 0xfffff) | 0x100000u;
  unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)__double2loint(x)) << (B - 53);
  m = ex == 0 ? 0 : m >> min(E - ex, 63);  // subnormal values count as zero
  const long long s = (long long)(hi >> 31);
  return ((fx64)m ^ s) - s;
}

// r 2^t, rounded to nearest; below the normal range a value under 2^-1021
__device__ __forceinline__ double fx_to(fx64 r, int t) {
  const long long s = r >> 63;
  const unsigned long long a = (unsigned long long)((r ^ s) - s);
  const unsigned ahi = (unsigned)(a >> 32), alo = (unsigned)a;
  const int lz = __clz(ahi ? ahi : alo) + (ahi ? 0 : 32);  // >= 1; 64 for zero
  const unsigned long long m = ((a << (lz - 1)) + 0x200) >> 10;
  // the exponent field joins the high word only; the leading bit of m adds one to it
  const int e = lz == 64 ? 0 : max(1085 + t - lz, 0);
  const int hi = ((int)(m >> 32) + (e << 20)) | ((int)s & (int)0x80000000);
  return __hiloint2double(hi, (int)(unsigned)m);
}

// a value as v = h 2^32 + l with the low half signed, |l| <= 2^31 (|v| < 2^62)
struct FxSplit {
  int h, l;
};
__device__ __forceinline__ FxSplit fx_split(fx64 v) {
  return {(int)(v >> 32) + (int)((unsigned)v >> 31), (int)(unsigned)v};
}

// Sum of products / 2^64: the high products and the two kinds of cross products are
// accumulated apart (the low products lie below the result's last bit, and signed low
// halves have mean zero).  The cross sum carries an offset of 2^63, so that its high word
// joins the high sum without a sign extension, and half a unit of the result.
struct FxAcc {
  fx64 hh = -(1ll << 31), mid = (fx64)0x8000000080000000ull;
  __device__ __forceinline__ void add(FxSplit a, FxSplit b) { add(a, b.h, b.l); }
  __device__ __forceinline__ void add(FxSplit a, int h, int l) {
    hh = fx_mad(a.h, h, hh);
    mid = fx_mad(a.h, l, mid);
    mid = fx_mad(a.l, h, mid);
  }
  __device__ __forceinline__ fx64 get() const { return hh + (fx64)((unsigned long long)mid >> 32); }
};

__device__ __forceinline__ fx64 fx_mul(FxSplit a, FxSplit b) {
  FxAcc s;
  s.add(a, b);
  return s.get();
}

// rounded right shift, sh >= 1
__device__ __forceinline__ fx64 fx_shr(fx64 v, int sh) { return (v + (1ll << (sh - 1))) >> sh; }

// One line of a D_hat contraction in place: x[0], x[stride], ... (|x| < 2^59.6) become the
// contraction (< 2^58.6; LGL: 2^fx_up times that, see FxOps); FACE: plus the face terms
// l_hat_i(-1) qm + l_hat_i(+1) qp (Gauss-Lobatto: only at the line's ends)
template <int n, bool LGL, bool FACE>
__device__ __forceinline__ void fx_line(fx64* __restrict__ p, int stride, fx64 qm, fx64 qp, const FxOps& o) {
  constexpr int h = n / 2, c = (n + 1) / 2, N = n - 1;
  FxSplit e[c], d[h];
#pragma unroll
  for (int a = 0; a < h; ++a) {
    const fx64 x = p[a * stride], y = p[(N - a) * stride];
    e[a] = fx_split(x + y);
    d[a] = fx_split(x - y);
  }
  if constexpr (n & 1) e[c - 1] = fx_split(p[(c - 1) * stride]);
  FxSplit qs{0, 0}, qd{0, 0};
  if constexpr (FACE) {
    qs = fx_split(qp + qm);
    qd = fx_split(qp - qm);
  }
#pragma unroll
  for (int i = 0; i < c; ++i) {
    const bool face = FACE && (!LGL || i == 0);
    FxAcc so;
#pragma unroll
    for (int a = 0; a < h; ++a) so.add(d[a], o.oh[i][a], o.ol[i][a]);
    if (face) so.add(qs, o.sh[i], o.sl[i]);
    const fx64 O = so.get() << (i == 0 ? fx_up(n, LGL) : 0);
    if (i < h) {
      FxAcc se;
#pragma unroll
      for (int a = 0; a < c; ++a) se.add(e[a], o.eh[i][a], o.el[i][a]);
      if (face) se.add(qd, o.th[i], o.tl[i]);
      const fx64 E = se.get() << (i == 0 ? fx_up(n, LGL) : 0);
      p[i * stride] = O + E;
      p[(N - i) * stride] = O - E;
    } else {
      p[i * stride] = O;
    }
  }
}

// both end values of a line, sum_a l_a(-1) x_a and sum_a l_a(+1) x_a
template <int n>
__device__ __forceinline__ void fx_ends(const fx64* __restrict__ p, int stride, const FxOps& o, fx64& ym, fx64& yp) {
  constexpr int h = n / 2, c = (n + 1) / 2, N = n - 1;
  FxAcc e, d;
#pragma unroll
  for (int a = 0; a < c; ++a) {
    const fx64 x = p[a * stride];
    if (2 * a == N) {
      e.add(fx_split(x), o.peh[a], o.pel[a]);
    } else {
      const fx64 y = p[(N - a) * stride];
      e.add(fx_split(x + y), o.peh[a], o.pel[a]);
      if (a < h) d.add(fx_split(x - y), o.poh[a], o.pol[a]);
    }
  }
  const fx64 E = e.get(), D = d.get();
  yp = E + D;
  ym = E - D;
}

// Normal of a face in fixed point for fx_visc_normal: n_d and -2/3 n_d (60 bits) under the
// exponent e_d of n_d
struct FxNormal {
  FxSplit n[3], m[3];
  int e[3];
};
__device__ __forceinline__ FxNormal fx_normal(const double n[3]) {
  FxNormal q;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    q.e[d] = fx_mag(n[d]) >> 20;
    q.n[d] = fx_split(fx_from<60>(n[d], q.e[d]));
    q.m[d] = fx_split(fx_from<60>(-(2.0 / 3.0) * n[d], q.e[d]));
  }
  return q;
}

// visc_normal with the stress sums tn_c = sum_d (G_dc + G_cd) n_d - 2/3 div n_c in fixed point
// (26 of its 45 FP64 instructions; HLLC k_face at 16^3, N = 7: 275 -> 226 us).  The diagonal, each
// pair of off-diagonal gradients and each component of n have their own exponent and the products
// of a sum meet at its largest: a shear layer's gradient, large against all others, leaves the sums
// that it does not enter as accurate as in FP64.  Gradients outside the range take the FP64 sums.
__device__ __forceinline__ void fx_visc_normal(const double W[NV], const double ir, const double G[15], const double n[3],
                                               const FxNormal& q, const Phys<double>& ph, double f[NV]) {
  int ed = 0, eo[3];  // diagonal; off-diagonal pair k: the two directions other than k
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int i = (k + 1) % 3, j = (k + 2) % 3;
    ed = max(ed, fx_mag(G[k * 5 + 1 + k]) >> 20);
    eo[k] = max(fx_mag(G[i * 5 + 1 + j]), fx_mag(G[j * 5 + 1 + i])) >> 20;
  }
  if (max(max(ed, eo[0]), max(eo[1], eo[2])) > 1900) {
    visc_normal(W, ir, G, n, ph, f);
    return;
  }
  fx64 g[3], a[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int i = (k + 1) % 3, j = (k + 2) % 3;
    g[k] = fx_from<60>(G[k * 5 + 1 + k], ed);
    a[k] = fx_from<60>(G[i * 5 + 1 + j], eo[k]) + fx_from<60>(G[j * 5 + 1 + i], eo[k]);
  }
  const fx64 div = g[0] + g[1] + g[2];
  double tn[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int i = (c + 1) % 3, j = (c + 2) % 3;  // a[i] meets n_j, a[j] meets n_i
    const int xd = ed + q.e[c], xi = eo[i] + q.e[j], xj = eo[j] + q.e[i], x = max(xd, max(xi, xj));
    const int sd = min(x - xd, 62);
    FxAcc s;
    s.add(fx_split((2 * g[c]) >> sd), q.n[c]);
    s.add(fx_split(div >> sd), q.m[c]);
    s.add(fx_split(a[i] >> min(x - xi, 62)), q.n[j]);
    s.add(fx_split(a[j] >> min(x - xj, 62)), q.n[i]);
    tn[c] = ph.mu * fx_to(s.get(), x - 2044 + 64 - 120);
  }
  const double pir = W[4] * ir;
  double dTn = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) dTn = dg_fma(dg_fma(-pir, G[d * 5 + 0], G[d * 5 + 4]), n[d], dTn);
  f[0] = 0.0;
  f[1] = tn[0];
  f[2] = tn[1];
  f[3] = tn[2];
  f[4] = tn[0] * W[1] + tn[1] * W[2] + tn[2] * W[3] + ph.lam_th * dTn * ir;
}

// fx_line without face terms, and the line's end values as fx_ends
template <int n>
__device__ __forceinline__ void fx_line_ends(fx64* __restrict__ p, int stride, const FxOps& o, fx64& ym, fx64& yp) {
  constexpr int h = n / 2, c = (n + 1) / 2, N = n - 1;
  FxSplit e[c], d[h];
#pragma unroll
  for (int a = 0; a < h; ++a) {
    const fx64 x = p[a * stride], y = p[(N - a) * stride];
    e[a] = fx_split(x + y);
    d[a] = fx_split(x - y);
  }
  if constexpr (n & 1) e[c - 1] = fx_split(p[(c - 1) * stride]);
  {
    FxAcc se, sd;
#pragma unroll
    for (int a = 0; a < c; ++a) se.add(e[a], o.peh[a], o.pel[a]);
#pragma unroll
    for (int a = 0; a < h; ++a) sd.add(d[a], o.poh[a], o.pol[a]);
    const fx64 E = se.get(), D = sd.get();
    yp = E + D;
    ym = E - D;
  }
#pragma unroll
  for (int i = 0; i < c; ++i) {
    FxAcc so;
#pragma unroll
    for (int a = 0; a < h; ++a) so.add(d[a], o.oh[i][a], o.ol[i][a]);
    const fx64 O = so.get();
    if (i < h) {
      FxAcc se;
#pragma unroll
      for (int a = 0; a < c; ++a) se.add(e[a], o.eh[i][a], o.el[i][a]);
      const fx64 E = se.get();
      p[i * stride] = O + E;
      p[(N - i) * stride] = O - E;
    } else {
      p[i * stride] = O;
    }
  }
}

// Largest magnitude words of n fields over the threads of an element: get(s) is the
// thread's word for slot s.  One warp reduction per slot, lane s keeps the s-th, one shared
// atomic per warp where a CTA holds one element (every thread of mask calls it, and every
// warp has at least COUNT of them); else one atomic per thread and slot.
template <bool WARP, int COUNT, typename Get>
__device__ __forceinline__ void fx_max(int* slots, unsigned mask, Get get) {
  if constexpr (WARP) {
    const int lane = threadIdx.x & 31;
    int mine = 0;
#pragma unroll
    for (int s = 0; s < COUNT; ++s) {
      const int r = __reduce_max_sync(mask, get(s));
      mine = lane == s ? r : mine;
    }
    if (lane < COUNT) atomicMax(slots + lane, mine);
  } else {
#pragma unroll
    for (int s = 0; s < COUNT; ++s) atomicMax(slots + s, get(s));
  }
}

}  // namespace flexi
