// How many warps share a polynomial in the evaluation (host only, plain C++ so
// that the host tests can build it).
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>

namespace ht {

// The sizes of a system that its evaluation time depends on.
struct EvalShape {
  int nv = 0, np = 0;     // variables, polynomials
  int max_terms = 0;      // monomials of the longest polynomial
  int64_t max_steps = 0;  // sweep steps of the longest polynomial
  double mean_steps = 0;  // and of an average one
  // double: complex products of the sweep, and terms of all outputs
  int64_t max_products = 0, max_slots = 0;
  double mean_products = 0, mean_slots = 0;
};
// CTAs of G polynomials on S warps each.
struct EvalSplit {
  int S = 1, G = 1;
};

// The S of least modelled time for n_blocks blocks of 32 points on sms SMs.
// In units of one sweep step of a warp alone on its sub-partition (0.33, 0.49
// and 0.86 us in D, DD and QD) a CTA's pass costs
//   staging   1 (QD 4) for every point a warp converts, nv / T of them;
//   steps     1 each, of whole monomials, 1/S of a polynomial's;
//   outputs   1.25 for every output a warp converts, (nv + 1) / S;
//   exchange  1.5 for each of the nv + 1 outputs when S > 1: the bounds and
//             the row slots go through shared memory whatever S is.
// A warp needs at least that sum for the longest polynomial; an SM needs 0.45
// of the mean sum for every warp on its fullest sub-partition (the products
// are latency-bound until then); the 3-norm of the two joins them.  The unsplit kernels of D and DD take 4/3 of the latency (64 registers
// a thread) but hold 32 warps an SM, the others 16.  Waves of CTAs add up.
// The constants were fitted to the times of eight supports (6 to 32
// variables, 8 to 246 monomials, 35 to 2,706 steps a polynomial) at 10 to
// 16,384 points, S = 1 to 16: the pick costs 1.5 % more than the best S on
// average and 21 % at most, and no call takes longer than the kernel that
// preceded splitting.  (A fixed 1/20 of a pass for the exchange, right for 246
// monomials, took S = 4 for 12 polynomials of 16 two-variable monomials at
// 4,064 points: DD 122 us for 86 unsplit, QD 253 for 145.)
inline EvalSplit eval_split(const EvalShape& e, int limbs, int64_t n_blocks, int64_t sms) {
  const double stage = limbs == 4 ? 4.0 : 1.0, slot = 1.25, exchange = 1.5, load = 0.45;
  const int unsplit_warps = limbs == 4 ? 16 : 32;
  EvalSplit best;
  double least = 1e300;
  for (int S = 1; S <= 16 && S <= e.max_terms; ++S) {
    const int warps = S == 1 ? unsplit_warps : 16;
    const int most = std::min(e.np, warps / S), groups = (e.np + most - 1) / most, G = (e.np + groups - 1) / groups;
    const int T = S * G;
    const double share = (double)((e.max_terms + S - 1) / S) / e.max_terms;
    const double fixed = slot * (e.nv + 1) / S + (S > 1 ? exchange * (e.nv + 1) : 0.0);
    double alone = stage * ((e.nv + T - 1) / T) + e.max_steps * share + fixed;
    const double mean = stage * e.nv / T + e.mean_steps / S + fixed;
    if (S == 1 && limbs < 4) alone *= 4.0 / 3.0;
    // time of a wave that puts c CTAs on an SM
    auto wave = [&](int64_t c) {
      const double crowd = load * mean * (double)((c * T + 3) / 4);
      return std::cbrt(alone * alone * alone + crowd * crowd * crowd);
    };
    const int64_t resident = std::max(1, warps / T), items = n_blocks * groups, slots = sms * resident;
    const int64_t rest = items % slots;
    const double t = (double)(items / slots) * wave(resident) + (rest > 0 ? wave((rest + sms - 1) / sms) : 0.0);
    if (t < least * 0.98) {  // a split has to gain something
      least = t;
      best.S = S;
      best.G = G;
    }
  }
  return best;
}

// Double evaluation on the FP64 pipe: whether a CTA of `warps` warps for each of
// `units` units (a polynomial at 32 points, its terms in `chunks` chunks)
// beats one warp for each.  In units of one complex product at the pipe's full
// rate (0.17 us) a unit loads a sub-partition with its products and 0.45 for
// every term it adds; dealt over a CTA's warps, on the SM's four, with 0.55 a
// term and 3.2 for every output and chunk (searches and loads of the sums).
// Alone, one warp waits 0.8 a product and 1.8 a term; the CTA's warps 3.2 for
// each of the products of their share of whole monomials and for each chunk.
// The 3-norm joins latency and load.  The constants were fitted to eight supports at 32
// to 16,384 points; the pick costs 0.3 % more than the better of the two on
// average, 9 % at most.  (Two units a sub-partition, the line for polynomials
// of 130 monomials, lost 36 % for 12 of 16 two-variable monomials at 3,000
// points, 28.9 -> 39.2 us, and kept cyclic 10-roots at 4,064 points at 94.8
// us for 66.1.)
inline bool double_split_pays(const EvalShape& e, int64_t units, int64_t sms, int warps, int64_t chunks) {
  auto join = [](double alone, double load) { return alone * alone * alone + load * load * load; };
  auto waves = [&](int64_t slots) { return (double)((units + slots - 1) / slots); };
  const double share = (double)((e.max_terms + warps - 1) / warps) / e.max_terms;
  const double load_one = e.mean_products + 0.45 * e.mean_slots;
  const double load_split = e.mean_products + 0.55 * e.mean_slots + 3.2 * (e.nv + 1) * chunks;
  const double one = join(0.8 * e.max_products + 1.8 * e.max_slots, load_one * waves(4 * sms));
  const double split = join(3.2 * e.max_products * share + 3.2 * chunks, load_split * waves(sms) / 4.0);
  return split < 0.97 * 0.97 * 0.97 * one;
}

}  // namespace ht
