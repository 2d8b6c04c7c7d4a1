// One polynomial's value and gradient row on the integer pipe, for one point
// per lane (device only): the per-output frames, the sweep's steps of
// ht_mpi_eval.cuh with the row's fixed-point accumulators in local memory, and
// the conversion of every output to L doubles.  The evaluation kernels and the
// tracker both use it.
#pragma once
#include "ht_mpi_eval.cuh"
#include "ht_mpi_ops.cuh"

namespace ht {

using mpi::IntW;
constexpr int kIntMaxVars = 64;

// The fixed-point accumulators of one polynomial's outputs at the lane's
// point: slot i the derivative by x_i, slot nv the value, each 2 WA limbs
// (re, im) in local memory, moved in 128-bit words (padded to whole ones).
template <int L>
struct RowAcc {
  static constexpr int W = IntW<L>::W, WA = IntW<L>::WA, Q = (2 * WA + 3) / 4;  // int4 words per slot
  int4* a;        // [(nv + 1) Q]
  const int* Fv;  // frames of the slots
  int nv;
  __device__ __forceinline__ int at(int v) const { return v == mpi::step::VALUE ? nv : v; }
  __device__ __forceinline__ void zero(int i) {
#pragma unroll
    for (int k = 0; k < Q; ++k) a[i * Q + k] = make_int4(0, 0, 0, 0);
  }
  __device__ __forceinline__ void load(int i, int32_t* ar, int32_t* ai) const {
    int32_t w[4 * Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      const int4 q = a[i * Q + k];
      w[4 * k] = q.x;
      w[4 * k + 1] = q.y;
      w[4 * k + 2] = q.z;
      w[4 * k + 3] = q.w;
    }
#pragma unroll
    for (int k = 0; k < WA; ++k) {
      ar[k] = w[k];
      ai[k] = w[WA + k];
    }
  }
  __device__ __forceinline__ void add(int v, const mpi::fz<W>& d, int e) {
    const int i = at(v);
    int32_t ar[WA], ai[WA];
    load(i, ar, ai);
    mpi::acc_add_fast<W, WA>(ar, ai, d, e, Fv[i]);
    int32_t w[4 * Q];
#pragma unroll
    for (int k = 0; k < WA; ++k) {
      w[k] = ar[k];
      w[WA + k] = ai[k];
    }
#pragma unroll
    for (int k = 2 * WA; k < 4 * Q; ++k) w[k] = 0;
#pragma unroll
    for (int k = 0; k < Q; ++k) a[i * Q + k] = make_int4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
  }
};

// The lane's point converted once: X[i] (limb string) and lg[i] = log2 |x_i|,
// from x in the layout [nv][2][L][n].
template <int L>
__device__ __forceinline__ void int_point(const double* __restrict__ x, int nv, int64_t n, int64_t p,
                                          mpi::fz<IntW<L>::W>* X, float* lg) {
  for (int i = 0; i < nv; ++i) {
    double re[L], im[L];
#pragma unroll
    for (int l = 0; l < L; ++l) {
      re[l] = x[((int64_t)(i * 2) * L + l) * n + p];
      im[l] = x[((int64_t)(i * 2 + 1) * L + l) * n + p];
    }
    X[i] = mpi::from_doubles<IntW<L>::W, L>(re, im);
    lg[i] = mpi::log2_mod(re[0], im[0]);
  }
}

// Monomials m0..m1 of one polynomial at the lane's point.  X and lg are
// indexable by variable (local arrays or shared-memory views); P is scratch
// for the forward products (max monomial size entries).  int_row_run leaves
// the exact sums in the row's slots (the tracker goes on from there); int_row
// rounds them into the doubles of the outputs (value vrow [2][L][n], gradient
// jrow [nv][2][L][n]).
struct IntPoly {
  const int32_t* mon_off;
  const uint16_t* pairs;
  const int32_t* step_off;  // range of each monomial in steps
  const uint32_t* steps;
  const float* clg;
};
template <int L, class XA, class LG, class PS>
__device__ __forceinline__ void int_row_run(const IntPoly& s, const mpi::fz<IntW<L>::W>* __restrict__ cfz, int m0, int m1,
                                            const XA& X, const LG& lg, int nv, RowAcc<L>& row, int* Fv, PS* P) {
  Fv[nv] = mpi::frames_for_poly<IntW<L>::WA>(s.mon_off, s.pairs, s.clg, m0, m1, lg, nv, Fv);
  for (int i = 0; i <= nv; ++i) row.zero(i);
  mpi::run_steps<L>(s.steps + s.step_off[m0], s.steps + s.step_off[m1], cfz + m0, X, row, P);
}
// Slot i of a row (limbs ar, ai in frame F) to the output's doubles.
template <int L>
__device__ __forceinline__ void store_slot(const int32_t* ar, const int32_t* ai, int F, double* q, int64_t n) {
  constexpr int WA = IntW<L>::WA;
  double o[L];
  mpi::fixed_to_doubles<WA, L>(ar, F, o);
#pragma unroll
  for (int l = 0; l < L; ++l) q[l * n] = o[l];
  mpi::fixed_to_doubles<WA, L>(ai, F, o);
#pragma unroll
  for (int l = 0; l < L; ++l) q[(L + l) * n] = o[l];
}
template <int L, class XA, class LG, class PS>
__device__ void int_row(const IntPoly& s, const mpi::fz<IntW<L>::W>* __restrict__ cfz, int m0, int m1, const XA& X,
                        const LG& lg, int nv, double* vrow, double* jrow, int64_t n, int64_t p, PS* P) {
  constexpr int WA = IntW<L>::WA;
  int Fv[kIntMaxVars + 1];
  int4 acc[(kIntMaxVars + 1) * RowAcc<L>::Q];
  RowAcc<L> row{acc, Fv, nv};
  int_row_run<L>(s, cfz, m0, m1, X, lg, nv, row, Fv, P);
  for (int i = 0; i <= nv; ++i) {
    int32_t ar[WA], ai[WA];
    row.load(i, ar, ai);
    store_slot<L>(ar, ai, Fv[i], (i == nv ? vrow : jrow + (int64_t)i * 2 * L * n) + p, n);
  }
}
// Views of a CTA's converted points in shared memory: limb strings padded to
// NW words, [var][lane][NW] (a multiple of 16 bytes, moved in 128-bit words;
// the 12- and 20-word strides of DD and QD put the eight lanes of each
// quarter-warp access in distinct banks), and log2 moduli [var][32].
template <int L>
struct SmemPoints {
  static constexpr int W = IntW<L>::W, NW = mpi::fzs<W>::NW;
  const int32_t* x;
  int lane;
  __device__ __forceinline__ mpi::fz<W> operator[](int v) const {
    return static_cast<mpi::fz<W>>(reinterpret_cast<const mpi::fzs<W>*>(x)[v * 32 + lane]);
  }
};
struct SmemLog {
  const float* g;
  int lane;
  __device__ __forceinline__ float operator[](int v) const { return g[v * 32 + lane]; }
};
template <int L>
__device__ __forceinline__ void store_point(int32_t* x, int v, int lane, const mpi::fz<IntW<L>::W>& z) {
  reinterpret_cast<mpi::fzs<IntW<L>::W>*>(x)[v * 32 + lane] = mpi::fzs<IntW<L>::W>(z);
}
// Bytes of shared memory for the points of nv variables.
template <int L>
constexpr size_t smem_points_bytes(int nv) {
  return (size_t)nv * 32 * (sizeof(mpi::fzs<IntW<L>::W>) + sizeof(float));
}

}  // namespace ht
