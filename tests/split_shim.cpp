// Host build of the evaluation's split rules (csrc/ht_split.h) and step lists.
#include "../paper_1505_00383_gb300/csrc/ht_mpi_eval.cuh"
#include "../paper_1505_00383_gb300/csrc/ht_split.h"

extern "C" {

int64_t split_steps(const uint16_t* pairs, int k) {
  std::vector<uint32_t> st;
  ht::mpi::sweep_steps(pairs, k, st);
  return (int64_t)st.size();
}

int64_t split_step_count(const uint16_t* pairs, int k) { return ht::mpi::sweep_step_count(pairs, k); }

int split_offsets_fit(int64_t n) { return ht::mpi::offsets_fit(n); }

int split_pick(int nv, int np, int max_terms, int64_t max_steps, double mean_steps, int limbs, int64_t n_blocks,
               int64_t sms) {
  ht::EvalShape e;
  e.nv = nv;
  e.np = np;
  e.max_terms = max_terms;
  e.max_steps = max_steps;
  e.mean_steps = mean_steps;
  const ht::EvalSplit s = ht::eval_split(e, limbs, n_blocks, sms);
  return s.S * 100 + s.G;
}

int double_pays(int nv, int max_terms, int64_t max_products, double mean_products, int64_t max_slots, double mean_slots,
                int64_t units, int64_t sms, int warps, int64_t chunks) {
  ht::EvalShape e;
  e.nv = nv;
  e.max_terms = max_terms;
  e.max_products = max_products;
  e.mean_products = mean_products;
  e.max_slots = max_slots;
  e.mean_slots = mean_slots;
  return ht::double_split_pays(e, units, sms, warps, chunks);
}
}
