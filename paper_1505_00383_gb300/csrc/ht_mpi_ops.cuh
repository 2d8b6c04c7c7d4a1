// General arithmetic on the floating limb strings of ht_mpi.cuh for the
// tracker's linear algebra: signed sums of a few terms through one fixed-point
// frame, renormalisation, conjugation, conversion of reals, and 1/sqrt by
// Newton's iteration.  Host+device, like ht_mpi.cuh.
#pragma once
#include <cmath>

#include "ht_mpi.cuh"

namespace ht {
namespace mpi {

// ------------------------------------------------------------ general sums
// Smallest E with |re|, |im| < 2^E (from the top limb; lower limbs add less
// than one unit of it).  Zero gives a very small E.
template <int W>
HT_HD int bound_exp(const fz<W>& z) {
  for (int k = W - 1; k >= 0; --k) {
    const int32_t ar = z.r[k] < 0 ? -z.r[k] : z.r[k], ai = z.i[k] < 0 ? -z.i[k] : z.i[k];
    const int32_t mx = ar > ai ? ar : ai;
    if (mx != 0) {
      return z.f + RB * k + bitlen32((uint32_t)mx) + 1;  // (mx + 1) 2^(29 k + f) bounds the lower limbs too
    }
  }
  return -30000;
}

// The window of W limbs of carried fixed-point strings (limbs 0..WA-2 in
// [0, 2^29), the top signed, frame F) from the highest significant limb of
// |re| and |im| down, the sign folded into its top limb; N components
// (2: re and im; 1: a real).  The strings move up limb by limb while their top
// limb only repeats the sign (mostly not at all, or once), so every index is
// static.  A value -2^(29 k) needs limb k, although that limb is all sign.
template <int WA, int W, int N>
HT_HD void top_window(int32_t (*d)[WA], int& F) {
  int up = 0;
  while (up < WA - 1) {
    bool only_sign = true;
#pragma unroll
    for (int c = 0; c < N; ++c) {
      const int32_t sg = d[c][WA - 1] >> 31;
      int32_t low = 0;
#pragma unroll
      for (int k = 0; k < WA - 1; ++k) low |= d[c][k];
      only_sign = only_sign && d[c][WA - 1] == sg && (sg == 0 || low != 0);
    }
    if (!only_sign) break;
    ++up;
#pragma unroll
    for (int c = 0; c < N; ++c) {
      const int32_t sg = d[c][WA - 1] >> 31;
#pragma unroll
      for (int k = WA - 1; k >= 1; --k) d[c][k] = d[c][k - 1];
      d[c][0] = 0;
      d[c][WA - 1] += (int32_t)((uint32_t)sg << RB);
    }
  }
  F += RB * (WA - W - up);
}

// Fixed-point complex (WA limbs each, frame F) to a floating fz<W>: the W
// limbs from the highest significant one down (the sign folded into the top).
template <int WA, int W>
HT_HD fz<W> fixed_to_fz(const int32_t* ar_in, const int32_t* ai_in, int F) {
  static_assert(WA >= W, "the window lies inside the string");
  int32_t d[2][WA];
#pragma unroll
  for (int k = 0; k < WA; ++k) {
    d[0][k] = ar_in[k];
    d[1][k] = ai_in[k];
  }
  carry32<WA>(d[0]);
  carry32<WA>(d[1]);
  fz<W> z;
  z.f = F;
  top_window<WA, W, 2>(d, z.f);
#pragma unroll
  for (int k = 0; k < W; ++k) {
    z.r[k] = d[0][WA - W + k];
    z.i[k] = d[1][WA - W + k];
  }
  normalize_top<W>(z);
  return z;
}

// s times a fixed-point complex (WA limbs each, frame F), s a double, to
// fz<W>: the product is formed exactly in WA + 2 limbs per component (s's
// significand in a 24-bit and a 29-bit part) and cut to W limbs as
// fixed_to_fz does.
template <int WA, int W>
HT_HD fz<W> fixed_scaled_to_fz(const int32_t* ar, const int32_t* ai, int F, double s) {
  int64_t ms;
  int es;
  decompose(s, ms, es);  // s = ms 2^es, |ms| < 2^53
  const bool neg = ms < 0;
  const uint64_t u = (uint64_t)(neg ? -ms : ms);
  const int64_t lo = (int64_t)(u & (uint64_t)MASK), hi = (int64_t)(u >> RB);
  int64_t cr[WA + 2], ci[WA + 2];
  for (int k = 0; k < WA + 2; ++k) cr[k] = ci[k] = 0;
  for (int k = 0; k < WA; ++k) {  // |a_k lo| < 2^58, |a_k hi| < 2^53
    cr[k] += (int64_t)ar[k] * lo;
    cr[k + 1] += (int64_t)ar[k] * hi;
    ci[k] += (int64_t)ai[k] * lo;
    ci[k + 1] += (int64_t)ai[k] * hi;
  }
  if (neg)
    for (int k = 0; k < WA + 2; ++k) {
      cr[k] = -cr[k];
      ci[k] = -ci[k];
    }
  carry<WA + 2>(cr);
  carry<WA + 2>(ci);
  int32_t br[WA + 2], bi[WA + 2];  // top limbs below 2^24 in magnitude
  for (int k = 0; k < WA + 2; ++k) {
    br[k] = (int32_t)cr[k];
    bi[k] = (int32_t)ci[k];
  }
  return fixed_to_fz<WA + 2, W>(br, bi, F + es);
}

template <int W>
HT_HD bool is_zero(const fz<W>& z) {
  int32_t o = 0;
  for (int k = 0; k < W; ++k) o |= z.r[k] | z.i[k];
  return o == 0;
}

// sum_k e_k z_k (e_k small signed integers, n <= N terms), rounded to fz<W>.
// One fixed frame F of WA = W + 1 limbs: its top holds the largest bound plus
// headroom for the n terms, and F lies at most 28 bits below every nonzero
// term's limb 0 (the shift rule of acc_add_fast).  A nonzero term's top limb
// is nonzero, so F is at least 29 (W - 1) + 28 bits below the largest term's
// magnitude: each term's truncation is below 2^(1 - 29 W) times the largest.
template <int W, int N>
HT_HD fz<W> sum(const fz<W>* z, const int* e, int n) {
  constexpr int WA = W + 1;
  int E = -30000, fmax = -30000;
  for (int k = 0; k < n; ++k) {
    if (e[k] == 0 || is_zero<W>(z[k])) continue;
    const int ek = e[k] < 0 ? -e[k] : e[k];
    const int b = bound_exp<W>(z[k]) + bitlen32((uint32_t)(ek - 1));  // + ceil(log2 |e_k|)
    E = b > E ? b : E;
    fmax = z[k].f > fmax ? z[k].f : fmax;
  }
  int32_t ar[WA], ai[WA];
  for (int k = 0; k < WA; ++k) ar[k] = ai[k] = 0;
  if (fmax == -30000) {
    fz<W> zero;
    zero.f = 0;
    for (int k = 0; k < W; ++k) zero.r[k] = zero.i[k] = 0;
    return zero;
  }
  const int head = bitlen32((uint32_t)n) > 1 ? bitlen32((uint32_t)n) : 1;  // 2^head >= n + 1
  int F = E + head - (RB * (WA - 1) + 28);
  F = F > fmax - (RB - 1) ? F : fmax - (RB - 1);
  for (int k = 0; k < n; ++k)
    if (e[k] != 0 && !is_zero<W>(z[k])) acc_add_fast<W, WA>(ar, ai, z[k], e[k], F);
  return fixed_to_fz<WA, W>(ar, ai, F);
}
// a + b or a - b: sum's frame and rounding for two terms.
template <int W, bool SUB>
HT_HD fz<W> add_sub(const fz<W>& a, const fz<W>& b) {
  constexpr int WA = W + 1;
  const int ea = bound_exp<W>(a), eb = bound_exp<W>(b);  // -30000: zero
  const int E = ea > eb ? ea : eb;
  const int fa = ea > -30000 ? a.f : -30000, fb = eb > -30000 ? b.f : -30000;
  const int fmax = fa > fb ? fa : fb;
  fz<W> z;
  if (fmax == -30000) {
    z.f = 0;
#pragma unroll
    for (int k = 0; k < W; ++k) z.r[k] = z.i[k] = 0;
    return z;
  }
  int F = E + 2 - (RB * (WA - 1) + 28);
  F = F > fmax - (RB - 1) ? F : fmax - (RB - 1);
  int32_t ar[WA], ai[WA], dr[WA], di[WA];
#pragma unroll
  for (int k = 0; k < WA; ++k) ar[k] = ai[k] = dr[k] = di[k] = 0;
  const int pa = F - a.f + RB, pb = F - b.f + RB;
  if (ea > -30000 && pa < RB * (W + 1)) {
    shifted_digits<W, WA>(a.r, pa / RB, pa % RB, ar);
    shifted_digits<W, WA>(a.i, pa / RB, pa % RB, ai);
  }
  if (eb > -30000 && pb < RB * (W + 1)) {
    shifted_digits<W, WA>(b.r, pb / RB, pb % RB, dr);
    shifted_digits<W, WA>(b.i, pb / RB, pb % RB, di);
  }
#pragma unroll
  for (int k = 0; k < WA; ++k) {
    ar[k] = SUB ? ar[k] - dr[k] : ar[k] + dr[k];
    ai[k] = SUB ? ai[k] - di[k] : ai[k] + di[k];
  }
  return fixed_to_fz<WA, W>(ar, ai, F);
}
template <int W>
HT_HD fz<W> add(const fz<W>& a, const fz<W>& b) {
  return add_sub<W, false>(a, b);
}
template <int W>
HT_HD fz<W> sub(const fz<W>& a, const fz<W>& b) {
  return add_sub<W, true>(a, b);
}
template <int W>
HT_HD fz<W> conj(fz<W> a) {
  for (int k = 0; k < W; ++k) a.i[k] = -a.i[k];
  return a;
}
template <int W>
HT_HD fz<W> from_real(double d) {
  const double zero = 0.0;
  return from_doubles<W, 1>(&d, &zero);
}
// Value of the real part rounded to double (for norms, seeds and decisions).
template <int W>
HT_HD double real_to_double(const fz<W>& z) {
  double acc = 0.0;
  for (int k = W - 1; k >= 0; --k) {
    double lim = (double)z.r[k];
    int ex = z.f + RB * k;
    while (ex > 600) {
      lim *= bitsd((int64_t)(1023 + 600) << 52);
      ex -= 600;
    }
    while (ex < -600) {
      lim *= bitsd((int64_t)(1023 - 600) << 52);
      ex += 600;
    }
    acc += lim * bitsd((int64_t)(1023 + ex) << 52);
  }
  return acc;
}
// Real limb strings (the re part of an fz<W> whose im is zero), for 1/sqrt:
// the product and the difference take a third of the complex ones' work and
// give the same limbs.
template <int W>
struct rz {
  int32_t f;
  int32_t r[W];
};
template <int W>
HT_HD void normalize_top(rz<W>& z) {
  const int32_t t = z.r[W - 1] < 0 ? -z.r[W - 1] : z.r[W - 1];
  const int s = t >= (1 << 29) ? 2 : (t >= (1 << 28) ? 1 : 0);
  if (s == 0) return;
#pragma unroll
  for (int k = 0; k < W - 1; ++k)
    z.r[k] = (int32_t)((((uint32_t)z.r[k] >> s) | ((uint32_t)z.r[k + 1] << (RB - s))) & (uint32_t)MASK);
  z.r[W - 1] >>= s;
  z.f += s;
}
template <int W>
HT_HD rz<W> mul(const rz<W>& a, const rz<W>& b) {
  constexpr int C0 = W - 2 > 0 ? W - 2 : 0, NC = 2 * W - C0;
  int32_t d[NC];
  int64_t c = 0;
#pragma unroll
  for (int k = 0; k < NC - 1; ++k) {
#pragma unroll
    for (int x = 0; x < W; ++x) {
      const int y = k + C0 - x;
      if (y < 0 || y >= W) continue;
      c += (int64_t)a.r[x] * b.r[y];
    }
    d[k] = (int32_t)c & MASK;
    c >>= RB;
  }
  d[NC - 1] = (int32_t)c;
  const int32_t t = d[NC - 1];
  const bool high = !(t == 0 || t == -1);
  rz<W> z;
  z.f = a.f + b.f + (high ? RB * W : RB * (W - 1));
#pragma unroll
  for (int k = 0; k < W; ++k) {
    const int32_t lo = k == W - 1 ? d[k + W - 1 - C0] + (int32_t)((uint32_t)t << RB) : d[k + W - 1 - C0];
    z.r[k] = high ? d[k + W - C0] : lo;
  }
  normalize_top<W>(z);
  return z;
}
// a - b for nonzero a (b may be zero)
template <int W>
HT_HD rz<W> sub(const rz<W>& a, const rz<W>& b) {
  constexpr int WA = W + 1;
  auto bound = [](const rz<W>& z) {
    for (int k = W - 1; k >= 0; --k) {
      const int32_t m = z.r[k] < 0 ? -z.r[k] : z.r[k];
      if (m != 0) return z.f + RB * k + bitlen32((uint32_t)m) + 1;
    }
    return -30000;
  };
  const int ea = bound(a), eb = bound(b);
  const int E = ea > eb ? ea : eb, fb = eb > -30000 ? b.f : -30000, fmax = a.f > fb ? a.f : fb;
  int F = E + 2 - (RB * (WA - 1) + 28);
  F = F > fmax - (RB - 1) ? F : fmax - (RB - 1);
  int32_t d[1][WA], t[WA];
#pragma unroll
  for (int k = 0; k < WA; ++k) d[0][k] = t[k] = 0;
  const int pa = F - a.f + RB, pb = F - b.f + RB;
  if (pa < RB * (W + 1)) shifted_digits<W, WA>(a.r, pa / RB, pa % RB, d[0]);
  if (eb > -30000 && pb < RB * (W + 1)) shifted_digits<W, WA>(b.r, pb / RB, pb % RB, t);
#pragma unroll
  for (int k = 0; k < WA; ++k) d[0][k] -= t[k];
  carry32<WA>(d[0]);
  rz<W> z;
  z.f = F;
  top_window<WA, W, 1>(d, z.f);
#pragma unroll
  for (int k = 0; k < W; ++k) z.r[k] = d[0][WA - W + k];
  normalize_top<W>(z);
  return z;
}

// The real part as a real string, and back (im zero).
template <int W>
HT_HD rz<W> real_of(const fz<W>& z) {
  rz<W> y;
  y.f = z.f;
#pragma unroll
  for (int k = 0; k < W; ++k) y.r[k] = z.r[k];
  return y;
}
template <int W>
HT_HD fz<W> complex_of(const rz<W>& y) {
  fz<W> z;
  z.f = y.f;
#pragma unroll
  for (int k = 0; k < W; ++k) {
    z.r[k] = y.r[k];
    z.i[k] = 0;
  }
  return z;
}

// 1 / sqrt(v) for a positive real v (im = 0): Newton's iteration
// y <- y (3 - v y^2) / 2 from the double seed; each step doubles the bits.
template <int W>
HT_HD fz<W> inv_sqrt(const fz<W>& v, int steps) {
  const double vd = real_to_double<W>(v);
  rz<W> y = real_of<W>(from_real<W>(1.0 / std::sqrt(vd)));
  const rz<W> x = real_of<W>(v), c3 = real_of<W>(from_real<W>(3.0));
#pragma unroll 1
  for (int it = 0; it < steps; ++it) {
    y = mul<W>(y, sub<W>(c3, mul<W>(x, mul<W>(y, y))));
    y.f -= 1;  // halve
  }
  return complex_of<W>(y);
}

// a / b for reals, b nonzero: Newton's iteration y <- y (2 - b y) for 1 / b
// from the double seed (each step doubles the bits), then a y.
template <int W>
HT_HD rz<W> quotient(const rz<W>& a, const rz<W>& b, double b_lead) {
  rz<W> y = real_of<W>(from_real<W>(1.0 / b_lead));
  const rz<W> two = real_of<W>(from_real<W>(2.0));
#pragma unroll 1
  for (int it = 0; it < 3; ++it) y = mul<W>(y, sub<W>(two, mul<W>(b, y)));
  return mul<W>(a, y);
}
// Weights of cubic Hermite interpolation at u (past 1 when it extrapolates) of an interval of
// length d: of the values and slopes at 0 and at 1, w[0..3] = 2 u^3 - 3 u^2 +
// 1, (u^3 - 2 u^2 + u) d, 3 u^2 - 2 u^3, (u^3 - u^2) d.
template <int W>
HT_HD void hermite_weights(const rz<W>& u, const rz<W>& d, rz<W>* w) {
  const rz<W> u2 = mul<W>(u, u), u3 = mul<W>(u2, u);
  const fz<W> t[4] = {complex_of<W>(u3), complex_of<W>(u2), complex_of<W>(u), from_real<W>(1.0)};
  const int e[4][4] = {{2, -3, 0, 1}, {1, -2, 1, 0}, {-2, 3, 0, 0}, {1, -1, 0, 0}};
#pragma unroll 1
  for (int k = 0; k < 4; ++k) {
    w[k] = real_of<W>(sum<W, 4>(t, e[k], 4));
    if (k & 1) w[k] = mul<W>(w[k], d);
  }
}

// ------------------------------------------------------------ least squares
// Building blocks of modified Gram-Schmidt on columns of limb strings (the
// tracker's corrector, Section 2): every dot product and norm is one exact
// fixed-point sum of its products, rounded once.
template <int W>
HT_HD int inv_sqrt_steps() {
  return W >= 8 ? 3 : 2;  // from a 53-bit seed: 2 steps give 212 bits, 3 give 424
}
// sum_i conj(q_i) a_i over i < rows (rows <= N; scratch holds rows entries)
template <int W, int N>
HT_HD fz<W> dot_conj(const fz<W>* q, const fz<W>* a, int rows, fz<W>* scratch) {
  int e[N];
  for (int i = 0; i < rows; ++i) {
    scratch[i] = mul<W>(conj<W>(q[i]), a[i]);
    e[i] = 1;
  }
  return sum<W, N>(scratch, e, rows);
}
// sum_i |a_i|^2 (imaginary part exactly zero: the cross columns cancel)
template <int W, int N>
HT_HD fz<W> norm2(const fz<W>* a, int rows, fz<W>* scratch) {
  int e[N];
  for (int i = 0; i < rows; ++i) {
    scratch[i] = mul<W>(a[i], conj<W>(a[i]));
    e[i] = 1;
  }
  return sum<W, N>(scratch, e, rows);
}
// a_i -= r q_i
template <int W>
HT_HD void sub_scaled(fz<W>* a, const fz<W>& r, const fz<W>* q, int rows) {
  for (int i = 0; i < rows; ++i) a[i] = sub<W>(a[i], mul<W>(r, q[i]));
}
// sum_k e_k z_k with e = (1, -1, -1, ...): b - sum_j r_j x_j for the back
// substitution (terms[0] = b, terms[1..n] = the products)
template <int W, int N>
HT_HD fz<W> first_minus_rest(const fz<W>* terms, int n) {
  int e[N];
  for (int k = 0; k < n; ++k) e[k] = k == 0 ? 1 : -1;
  return sum<W, N>(terms, e, n);
}
// Limb string to L doubles per component (the fixed-point reading of the
// limbs: limbs 0..W-2 in [0, 2^29), top signed, frame f).
template <int W, int L>
HT_HD void to_doubles(const fz<W>& z, double* re, double* im) {
  fixed_to_doubles<W, L>(z.r, z.f, re);
  fixed_to_doubles<W, L>(z.i, z.f, im);
}

}  // namespace mpi
}  // namespace ht
