// One polynomial and its gradient at one point in the integer format of
// ht_mpi.cuh (host+device: the evaluation kernel runs it per lane, the host
// tests run it as is).  The reverse-mode sweep is the one of ht_eval.cuh.
#pragma once
#include <cmath>
#include <cstdint>
#include <vector>

#include "ht_mpi.cuh"

namespace ht {
namespace mpi {

template <int L>
struct IntW;
// W limbs of a product, WA of an accumulator.  A sum of n terms loses up to
// n units of its frame's last place, 2^(3 + 2 log2 n - (29 WA - 1)) of the
// largest term: in double two limbs would leave 2^-38 for 246 terms, so it
// takes three (2^-67, and 18.9 ms instead of 20.2 at n = 32, 65,536 points: the
// frame lies near the terms' last limb, so few digits move); DD 2^-96, QD 2^-212.
template <>
struct IntW<1> {
  static constexpr int W = 3, WA = 3;
};
template <>
struct IntW<2> {
  static constexpr int W = 5, WA = 4;
};
template <>
struct IntW<4> {
  static constexpr int W = 8, WA = 8;
};

// log2 |z| from the leading limbs (-1000 for zero)
HT_HD float log2_mod(double re, double im) {
  if (re == 0.0 && im == 0.0) return -1000.0f;
  const int er = re == 0.0 ? -1100 : ilog2(re), ei = im == 0.0 ? -1100 : ilog2(im);
  const int e = er > ei ? er : ei;
  const double a = std::ldexp(re, -e), b = std::ldexp(im, -e);
  return (float)e + 0.5f * std::log2((float)(a * a + b * b));
}

// Accumulator frames for polynomial m0..m1 at a point, one per output: the
// returned frame for the value, Fv[i] for the derivative by x_i.  Each frame
// lies above the largest bound on that output's terms -- log2 |c| + sum a
// log2 |x| for a value term; that minus log2 |x_v| plus log2 a_v for the
// derivative by x_v -- with one bit of margin for the float bounds and
// log2(terms + 1) + 1 bits of headroom for the sums, so every output is exact
// to its own last limb relative to its own largest term.
template <int WA>
HT_HD int frame_of(float E, int cnt) {
  int head = 1;
  while ((1 << head) < cnt + 1) ++head;
  const int Eint = (int)std::ceil((E > -3.0e4f ? E : -3.0e4f) + 1.0f) + head + 1;
  return Eint - (RB * (WA - 1) + 28);
}
// The bounds themselves: the returned one for the value's terms, Ev[i] for the
// derivative's by x_i, over the monomials m0..m1.
template <class LG>
HT_HD float bounds_for_poly(const int32_t* mon_off, const uint16_t* pairs, const float* clg, int m0, int m1,
                            const LG& lg, int nv, float* Ev) {
  for (int i = 0; i < nv; ++i) Ev[i] = -3.0e4f;
  float E = -3.0e4f;
  for (int m = m0; m < m1; ++m) {
    const int beg = mon_off[m], k = mon_off[m + 1] - beg;
    float lt = clg[m];
    for (int r = 0; r < k; ++r) {
      const uint16_t q = pairs[beg + r];
      lt += (float)(q >> 8) * lg[q & 0xff];
    }
    E = E > lt ? E : lt;
    for (int r = 0; r < k; ++r) {
      const uint16_t q = pairs[beg + r];
      const int v = q & 0xff;
      const float d = lt - lg[v] + std::log2((float)(q >> 8));
      Ev[v] = Ev[v] > d ? Ev[v] : d;
    }
  }
  return E;
}
template <int WA, class LG>
HT_HD int frames_for_poly(const int32_t* mon_off, const uint16_t* pairs, const float* clg, int m0, int m1,
                          const LG& lg, int nv, int* Fv) {
  float Ev[64];
  const float E = bounds_for_poly(mon_off, pairs, clg, m0, m1, lg, nv, Ev);
  const int cnt = m1 - m0;
  for (int i = 0; i < nv; ++i) Fv[i] = frame_of<WA>(Ev[i], cnt);
  return frame_of<WA>(E, cnt);
}

// The reverse-mode sweep of one monomial c x_{v_0}^{a_0} ... x_{v_{k-1}}^{a_{k-1}}
// as a list of steps, built once per system (sweep_steps).  The state is one
// running limb string cur (the common factor, then the forward products, then
// the product S of the variables behind the derivative at hand) and the
// stored forward products P (P[0] = cf, P[r] = cf x_{v_0} .. x_{v_{r-1}}):
//   START  cur = c
//   MULX   cur <- cur x_v      common factor, forward products, S
//   TOP    cur = x_{v_{k-1}};  the derivative by it is P[k-1]
//   MULP   the derivative by x_{v_r} is P[r] cur
// A step may store its result in P, and may add it to an output: to the value,
// or a_r times to the derivative by x_{v_r}.  Every product has cur as one
// operand and a string read from memory as the other, so the product and the
// accumulation are each emitted once (the 8-limb product is several hundred
// instructions) and only cur and the result stay in registers.
namespace step {
enum : uint32_t { START = 0, MULX = 1, TOP = 2, MULP = 3 };
constexpr int VALUE = 127;  // output slot of the polynomial's value
// bits 0-1 kind, 2 store, 3 add, 4-10 variable, 11-17 index of P (stored, or
// TOP's and MULP's source), 18-24 output slot, 25-31 exponent (at most 127)
inline uint32_t make(uint32_t kind, int var, int p, bool store, bool add, int slot, int e) {
  return kind | (store ? 4u : 0u) | (add ? 8u : 0u) | (uint32_t)var << 4 | (uint32_t)p << 11 | (uint32_t)slot << 18 |
         (uint32_t)e << 25;
}
}  // namespace step

// Number of steps of a monomial with the k variables pr (variable | exponent << 8).
inline int64_t sweep_step_count(const uint16_t* pr, int k) {
  int64_t n = 1 + 2 * k + (k > 2 ? k - 2 : 0);
  for (int r = 0; r < k; ++r) n += (pr[r] >> 8) - 1;
  return n;
}
// The lists' offsets are 32-bit.
inline bool offsets_fit(int64_t entries) { return entries <= INT32_MAX; }

// Append the steps of a monomial with the k <= 64 variables pr (variable | exponent << 8).
template <class Out>
inline void sweep_steps(const uint16_t* pr, int k, Out& out) {
  int chain = 0;  // products of the common factor
  for (int r = 0; r < k; ++r) chain += (pr[r] >> 8) - 1;
  out.push_back(step::make(step::START, 0, 0, k > 0 && chain == 0, k == 0, step::VALUE, 1));
  for (int r = 0; r < k; ++r)
    for (int e = 1; e < (pr[r] >> 8); ++e) {
      --chain;
      out.push_back(step::make(step::MULX, pr[r] & 0xff, 0, chain == 0, false, 0, 1));
    }
  for (int r = 0; r < k; ++r)  // the last forward product is the value
    out.push_back(step::make(step::MULX, pr[r] & 0xff, (r + 1) & 63, r + 1 < k, r + 1 == k, step::VALUE, 1));
  for (int r = k - 1; r >= 0; --r) {
    const int v = pr[r] & 0xff, e = pr[r] >> 8;
    out.push_back(step::make(r == k - 1 ? step::TOP : step::MULP, v, r, false, true, v, e));
    if (r >= 1 && r < k - 1) out.push_back(step::make(step::MULX, v, 0, false, false, 0, 1));
  }
}

// Run the steps st..end of consecutive monomials with the coefficients cf[0..]
// at the point X (converted variables): acc.add(slot, t, e) receives every
// result that is added; P is scratch for the forward products.
template <int L, class XA, class Acc, class PS>
HT_HD void run_steps(const uint32_t* st, const uint32_t* end, const fz<IntW<L>::W>* cf, const XA& X, Acc& acc, PS* P) {
  constexpr int W = IntW<L>::W;
  using Z = fz<W>;
  Z cur;
  uint32_t next = st != end ? *st : 0;
  while (st != end) {
    const uint32_t o = next, kind = o & 3u;
    if (++st != end) next = *st;
    const int p = (int)(o >> 11) & 127;
    Z t;
    if (kind == step::START) {
      t = cur = *cf++;
    } else if (kind == step::TOP) {
      t = static_cast<Z>(P[p]);
      cur = X[(o >> 4) & 127];
    } else {
      Z b;
      if (kind == step::MULX)
        b = X[(o >> 4) & 127];
      else
        b = static_cast<Z>(P[p]);
      t = mul<W>(cur, b);
      if (kind == step::MULX) cur = t;
    }
    if (o & 4u) P[p] = t;
    if (o & 8u) acc.add((int)(o >> 18) & 127, t, (int)(o >> 25));
  }
}

#if !defined(__CUDACC__)
// Value (fixed-point vr, vi in frame F) and gradient (through acc.add(var, d,
// e, Fv[var])) of the monomials m0..m1 given by their pairs, on the host: the
// steps the device runs, built here.  X is anything indexable by variable
// that yields the converted limb string.
template <int L, class XA, class Acc, class PS>
inline void eval_poly_int(const int32_t* mon_off, const uint16_t* pairs, const fz<IntW<L>::W>* cfz, int m0, int m1,
                          const XA& X, int F, const int* Fv, Acc& acc, int32_t* vr, int32_t* vi, PS* P) {
  constexpr int W = IntW<L>::W, WA = IntW<L>::WA;
  std::vector<uint32_t> st;
  for (int m = m0; m < m1; ++m) sweep_steps(pairs + mon_off[m], mon_off[m + 1] - mon_off[m], st);
  struct {
    Acc& acc;
    const int* Fv;
    int F;
    int32_t *vr, *vi;
    void add(int slot, const fz<W>& t, int e) {
      if (slot == step::VALUE)
        acc_add_fast<W, WA>(vr, vi, t, 1, F);
      else
        acc.add(slot, t, e, Fv[slot]);
    }
  } out{acc, Fv, F, vr, vi};
  run_steps<L>(st.data(), st.data() + st.size(), cfz + m0, X, out, P);
}
#endif

}  // namespace mpi
}  // namespace ht
