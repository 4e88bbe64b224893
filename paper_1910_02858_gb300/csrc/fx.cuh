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
// partial sum.
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
// which halves the multiply-adds.  An entry c is stored as round(c 2^(60 - cE)) =
// h 2^30 + l with |l| <= 2^29; m* hold the rounding constant of the middle sum and the
// mean of the omitted low-by-low products.
struct FxOps {
  int eh[FXH][FXH], el[FXH][FXH];  // DE[i][a], i < n/2, a < (n+1)/2
  int oh[FXH][FXH], ol[FXH][FXH];  // DO[i][a], i < (n+1)/2, a < n/2
  int sh[FXH], sl[FXH], th[FXH], tl[FXH];
  int peh[FXH], pel[FXH], poh[FXH], pol[FXH];  // prolongation: l(+-1), 58 bits under 2^pE
  long long meq[FXH], moq[FXH];  // middle sums of E and O with face terms
  long long me[FXH], mo[FXH];    // and without
  long long mpe, mpo;
  int cE, pE;
  int rsh;  // the lifting's three-direction sums shifted right by rsh stay below 2^60
  int ok;   // 0: the operators do not fit the format (not reached for n <= 8)
};

// host construction from the FP64 operators (integer rounding of scaled doubles: the
// same on every machine)
inline FxOps make_fx_ops(const Ops<double>& o, int n) {
  FxOps f;
  std::memset(&f, 0, sizeof(f));
  const int N = n - 1, h = n / 2, c = (n + 1) / 2;
  double big = 0, row = 0, pbig = 0;
  for (int i = 0; i < n; ++i) {
    double s = std::fabs(o.lhm[i]) + std::fabs(o.lhp[i]);
    big = std::fmax(big, std::fmax(std::fabs(o.lhm[i]), std::fabs(o.lhp[i])));
    pbig = std::fmax(pbig, std::fabs(o.lp[i]));
    for (int a = 0; a < n; ++a) {
      s += std::fabs(o.DhatT[a * n + i]);
      big = std::fmax(big, std::fabs(o.DhatT[a * n + i]));
    }
    row = std::fmax(row, s);
  }
  std::frexp(big, &f.cE);
  std::frexp(pbig, &f.pE);
  int re;
  std::frexp(3.0 * row, &re);
  const int bits = 57 + re - f.cE;  // |sum over three directions| < 2^bits
  f.rsh = bits > 60 ? bits - 60 : 0;
  f.ok = bits <= 62 ? 1 : 0;
  auto split = [](long long v, int& hi, int& lo) {
    const long long q = (v + (1ll << 29)) >> 30;
    hi = (int)q;
    lo = (int)(v - q * (1ll << 30));
  };
  // the operators' symmetric means: A = 2^(59 - cE) times the entry
  auto A = [&](int i, int a) {
    return std::llrint(std::ldexp(o.DhatT[a * n + i], 58 - f.cE)) -
           std::llrint(std::ldexp(o.DhatT[(N - a) * n + N - i], 58 - f.cE));
  };
  auto Q = [&](int i) {
    return std::llrint(std::ldexp(o.lhp[i], 58 - f.cE)) + std::llrint(std::ldexp(o.lhm[N - i], 58 - f.cE));
  };
  for (int i = 0; i < h; ++i) {
    long long m = 0;
    for (int a = 0; a < c; ++a) {
      split(2 * a == N ? 2 * A(i, a) : A(i, a) + A(i, N - a), f.eh[i][a], f.el[i][a]);
      m += f.el[i][a];
    }
    split(Q(i) - Q(N - i), f.th[i], f.tl[i]);
    f.me[i] = (1ll << 29) + m / 2;
    f.meq[i] = f.me[i] + f.tl[i] / 2;
  }
  for (int i = 0; i < c; ++i) {
    long long m = 0;
    for (int a = 0; a < h; ++a) {
      split(A(i, a) - A(i, N - a), f.oh[i][a], f.ol[i][a]);
      m += f.ol[i][a];
    }
    split(Q(i) + Q(N - i), f.sh[i], f.sl[i]);
    f.mo[i] = (1ll << 29) + m / 2;
    f.moq[i] = f.mo[i] + f.sl[i] / 2;
  }
  f.mpe = f.mpo = 1ll << 29;
  auto L = [&](int a) {  // 2^(57 - pE) l_a(+1), mean with its mirror image
    return std::llrint(std::ldexp(o.lp[a], 56 - f.pE)) + std::llrint(std::ldexp(o.lm[N - a], 56 - f.pE));
  };
  for (int a = 0; a < c; ++a) {
    split(2 * a == N ? 2 * L(a) : L(a) + L(N - a), f.peh[a], f.pel[a]);
    f.mpe += f.pel[a] / 2;
  }
  for (int a = 0; a < h; ++a) {
    split(L(a) - L(N - a), f.poh[a], f.pol[a]);
    f.mpo += f.pol[a] / 2;
  }
  return f;
}

// ---------------------------------------------------------------------------
// device primitives
// ---------------------------------------------------------------------------
using fx64 = long long;

// magnitude word: ordered like |x|, its exponent field is x's (NaN and infinities 2047)
__device__ __forceinline__ int fx_mag(double x) { return __double2hiint(x) & 0x7fffffff; }

// x 2^(60 - (E - 1022)) for |x| < 2^(E - 1022), E a biased exponent field; truncated
__device__ __forceinline__ fx64 fx_from(double x, int E) {
  const int hi = __double2hiint(x);
  const int ex = (hi >> 20) & 0x7ff;
  const unsigned mh = (unsigned)(hi & 0xfffff) | 0x100000u;
  unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)__double2loint(x)) << 7;
  m = ex == 0 ? 0 : m >> min(E - ex, 63);  // subnormal values count as zero
  const long long s = (long long)(hi >> 31);
  return ((fx64)m ^ s) - s;
}

// r 2^t, rounded to nearest; 0 below the normal range
__device__ __forceinline__ double fx_to(fx64 r, int t) {
  const long long s = r >> 63;
  const unsigned long long a = (unsigned long long)((r ^ s) - s);
  const unsigned ahi = (unsigned)(a >> 32), alo = (unsigned)a;
  const int lz = __clz(ahi ? ahi : alo) + (ahi ? 0 : 32);  // >= 1 for a != 0
  const unsigned long long m = ((a << (lz - 1)) + 0x200) >> 10;
  const int e = 1086 + t - lz;
  const unsigned long long b = ((unsigned long long)(unsigned)(e - 1) << 52) + m;
  return __longlong_as_double((a == 0 || e < 1) ? 0ll : (long long)(b | (unsigned long long)(s & (1ll << 63))));
}

// a value split into 30-bit halves, v = h 2^30 + l, 0 <= l < 2^30 (|v| < 2^61)
struct FxSplit {
  int h, l;
};
__device__ __forceinline__ FxSplit fx_split(fx64 v) { return {(int)(v >> 30), (int)v & 0x3fffffff}; }

// a b / 2^60 (the mean of the omitted low-by-low product is in the rounding constant)
__device__ __forceinline__ fx64 fx_mul(FxSplit a, FxSplit b) {
  const fx64 mid = (fx64)a.h * b.l + ((fx64)a.l * b.h + ((1ll << 29) + (1ll << 28)));
  return (fx64)a.h * b.h + (mid >> 30);
}

// rounded right shift, sh >= 1
__device__ __forceinline__ fx64 fx_shr(fx64 v, int sh) { return (v + (1ll << (sh - 1))) >> sh; }

// One line of a D_hat contraction: x[0..n) -> y(i, value) for every output node i; FACE: plus
// the face terms l_hat_i(-1) qm + l_hat_i(+1) qp (Gauss-Lobatto: only at the line's ends)
template <int n, bool LGL, bool FACE, typename Put>
__device__ __forceinline__ void fx_line(const fx64 (&x)[n], fx64 qm, fx64 qp, const FxOps& o, Put put) {
  constexpr int h = n / 2, c = (n + 1) / 2, N = n - 1;
  FxSplit e[c], d[h];
#pragma unroll
  for (int a = 0; a < h; ++a) {
    e[a] = fx_split(x[a] + x[N - a]);
    d[a] = fx_split(x[a] - x[N - a]);
  }
  if constexpr (n & 1) e[c - 1] = fx_split(x[c - 1]);
  FxSplit qs{0, 0}, qd{0, 0};
  if constexpr (FACE) {
    qs = fx_split(qp + qm);
    qd = fx_split(qp - qm);
  }
#pragma unroll
  for (int i = 0; i < c; ++i) {
    const bool face = FACE && (!LGL || i == 0);
    fx64 hh = 0, mid = face ? o.moq[i] : o.mo[i];
#pragma unroll
    for (int a = 0; a < h; ++a) {
      hh += (fx64)d[a].h * o.oh[i][a];
      mid += (fx64)d[a].h * o.ol[i][a];
      mid += (fx64)d[a].l * o.oh[i][a];
    }
    if (face) {
      hh += (fx64)qs.h * o.sh[i];
      mid += (fx64)qs.h * o.sl[i];
      mid += (fx64)qs.l * o.sh[i];
    }
    const fx64 O = hh + (mid >> 30);
    if (i < h) {
      hh = 0;
      mid = face ? o.meq[i] : o.me[i];
#pragma unroll
      for (int a = 0; a < c; ++a) {
        hh += (fx64)e[a].h * o.eh[i][a];
        mid += (fx64)e[a].h * o.el[i][a];
        mid += (fx64)e[a].l * o.eh[i][a];
      }
      if (face) {
        hh += (fx64)qd.h * o.th[i];
        mid += (fx64)qd.h * o.tl[i];
        mid += (fx64)qd.l * o.th[i];
      }
      const fx64 E = hh + (mid >> 30);
      put(i, O + E);
      put(N - i, O - E);
    } else {
      put(i, O);
    }
  }
}

// both end values of a line, sum_a l_a(-1) x_a and sum_a l_a(+1) x_a
template <int n>
__device__ __forceinline__ void fx_ends(const fx64 (&x)[n], const FxOps& o, fx64& ym, fx64& yp) {
  constexpr int h = n / 2, c = (n + 1) / 2, N = n - 1;
  fx64 he = 0, me = o.mpe, ho = 0, mo = o.mpo;
#pragma unroll
  for (int a = 0; a < c; ++a) {
    const FxSplit e = fx_split(2 * a == N ? x[a] : x[a] + x[N - a]);
    he += (fx64)e.h * o.peh[a];
    me += (fx64)e.h * o.pel[a];
    me += (fx64)e.l * o.peh[a];
    if (a < h) {
      const FxSplit d = fx_split(x[a] - x[N - a]);
      ho += (fx64)d.h * o.poh[a];
      mo += (fx64)d.h * o.pol[a];
      mo += (fx64)d.l * o.poh[a];
    }
  }
  const fx64 e = he + (me >> 30), d = ho + (mo >> 30);
  yp = e + d;
  ym = e - d;
}

// largest magnitude word over the threads of an element into a shared slot: one
// reduction and one shared atomic per warp where a CTA holds one element (WARP; every
// thread of mask calls it), else one atomic per thread
template <bool WARP>
__device__ __forceinline__ void fx_max(int* slot, int mag, unsigned mask) {
  if constexpr (WARP) {
    mag = __reduce_max_sync(mask, mag);
    if ((threadIdx.x & 31) == 0) atomicMax(slot, mag);
  } else {
    atomicMax(slot, mag);
  }
}

}  // namespace flexi
