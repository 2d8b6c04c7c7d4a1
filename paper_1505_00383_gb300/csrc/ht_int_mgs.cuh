// Modified Gram-Schmidt least squares on limb strings with one matrix row per
// lane (device only): the corrector's solve of the DD and QD tracker and of
// ht_mgs_solve_ex variant 2.
//
// A warp has 32 / rows slots of `rows` lanes.  They hold the slots / C
// systems the warp serves, each on C slots: slot c of a system has the columns
// j = c mod C.  A lane holds its row's entry of the pivot column in registers
// and its row of its columns in local memory; a dot product over the rows is
// one exact fixed-point sum across the slot's lanes (row_sum), rounded once,
// so every lane of the slot has the result.  There is no barrier: the warps
// are independent of each other.  C = 1 does the least work (a pivot column is
// normalised on every slot of its system); with C = slots a system takes a
// C-th of the steps, which is faster while there are warps to spare (DD n =
// 12 with 5 paths an SM: 625,000 clocks a solve with C = 1, 465,000 + the back
// substitution with 2).  The results do not depend on C.
//
// Why rows and not whole systems per lane: with a system per lane the columns
// were dealt to the warps of a CTA, which met at a barrier per column, and
// the columns lived in local memory behind runtime indexes; the warps waited
// for the pivot column's owner (4.7 barrier cycles an issue, 19 % of the
// issue slots used in QD).  n = 12 DD, 4,096 paths: 945 -> 534 ms; with groups
// of active / SMs paths, C and the summed back substitution 370 ms.
//
// What bounds it now: the latency of a warp's dependent arithmetic (a column
// step of a lone DD warp: product 850 clocks, sum over the rows 2,000, product
// 1,000, difference 1,550) and, in QD, instruction fetch.
#pragma once
#include "ht_int_row.cuh"

namespace ht {

template <int L>
struct RowLanes {
  static constexpr int W = IntW<L>::W, WA = W + 1;
  static constexpr int ND = (2 * WA + 3) / 4 * 4;  // exchanged words a lane, 16-byte multiple
  using Z = mpi::fz<W>;

  int rows, i, slot, base;        // rows a system; this lane's row, its slot, that slot's first lane
  int C, sub, cs;                 // slots a system; this lane's system in the warp, its columns are cs mod C
  bool row;                       // the lane has a row of a live system
  int32_t* dig;                   // shared [32][ND]
  int64_t* sums;                  // shared [slots][2 WA]

  static __host__ __device__ int slots(int rows) { return 32 / rows; }
  // Words of shared memory of one warp: the lanes' digits, then the slots' sums.
  static __host__ __device__ int words(int rows) { return 32 * ND + slots(rows) * 2 * WA * 2; }
  // row is false for lanes past the last whole system; the caller clears it
  // for systems it does not have
  __device__ __forceinline__ RowLanes(int rows_, int C_, int32_t* xch) : rows(rows_), C(C_) {
    const int lane = threadIdx.x & 31;
    slot = lane / rows;
    i = lane - slot * rows;
    base = slot * rows;
    sub = slot / C;
    cs = slot - sub * C;
    row = sub < slots(rows) / C;
    dig = xch;
    sums = reinterpret_cast<int64_t*>(xch + 32 * ND);
  }

  // sum over the slot's rows of z, or of -z on the lanes with neg, for the
  // lanes with part (`terms` of them): the frame, digits and rounding of mpi::sum
  __device__ __forceinline__ Z row_sum(const Z& z, bool part, bool neg, int terms) const {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, hb = mpi::bitlen32((uint32_t)terms), head = hb > 1 ? hb : 1;
    const int b0 = part ? mpi::bound_exp<W>(z) : -30000;
    int E = b0, fm = b0 > -30000 ? z.f : -30000;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
      const int oe = __shfl_down_sync(full, E, off), of = __shfl_down_sync(full, fm, off);
      if (i < off && i + off < rows) {
        E = max(E, oe);
        fm = max(fm, of);
      }
    }
    E = __shfl_sync(full, E, base);
    fm = __shfl_sync(full, fm, base);
    const int F = max(E + head - (mpi::RB * (WA - 1) + 28), fm - (mpi::RB - 1));
    int32_t d[ND];
#pragma unroll
    for (int k = 0; k < ND; ++k) d[k] = 0;
    const int sp = F - z.f + mpi::RB;
    if (b0 > -30000 && sp < mpi::RB * (W + 1)) {
      mpi::shifted_digits<W, WA>(z.r, sp / mpi::RB, sp % mpi::RB, d);
      mpi::shifted_digits<W, WA>(z.i, sp / mpi::RB, sp % mpi::RB, d + WA);
    }
    if (neg) {
#pragma unroll
      for (int k = 0; k < 2 * WA; ++k) d[k] = -d[k];
    }
    int4* q = reinterpret_cast<int4*>(dig + lane * ND);
#pragma unroll
    for (int k = 0; k < ND / 4; ++k) q[k] = make_int4(d[4 * k], d[4 * k + 1], d[4 * k + 2], d[4 * k + 3]);
    __syncwarp();
    if (row)
      for (int w = i; w < 2 * WA; w += rows) {  // the slot's lanes deal the words
        int64_t s = 0;
#pragma unroll 4
        for (int k = 0; k < rows; ++k) s += dig[(base + k) * ND + w];
        sums[slot * 2 * WA + w] = s;
      }
    __syncwarp();
    int64_t c[2 * WA];
    const int s0 = row ? slot * 2 * WA : 0;
#pragma unroll
    for (int k = 0; k < 2 * WA; ++k) c[k] = sums[s0 + k];
    mpi::carry<WA>(c);
    mpi::carry<WA>(c + WA);
    int32_t ar[WA], ai[WA];
#pragma unroll
    for (int k = 0; k < WA; ++k) {
      ar[k] = (int32_t)c[k];
      ai[k] = (int32_t)c[WA + k];
    }
    Z s = mpi::fixed_to_fz<WA, W>(ar, ai, F);
    if (fm == -30000) {  // all terms zero
      s.f = 0;
#pragma unroll
      for (int k = 0; k < W; ++k) s.r[k] = s.i[k] = 0;
    }
    return s;
  }

  // z of another lane
  static __device__ __forceinline__ Z shfl(const Z& z, int src) {
    Z t;
    t.f = __shfl_sync(0xffffffffu, z.f, src);
#pragma unroll
    for (int k = 0; k < W; ++k) {
      t.r[k] = __shfl_sync(0xffffffffu, z.r[k], src);
      t.i[k] = __shfl_sync(0xffffffffu, z.i[k], src);
    }
    return t;
  }

  // Least squares of [A | b_0 .. b_{nrhs-1}], cols <= rows <= 32, cols + nrhs
  // <= MAXC.  load(j) gives this lane's row's entry of column j, once, for
  // the lane's columns and column 0; put_q(j, z) takes it in the orthogonal
  // factor (j < cols) or in a reduced right-hand side; put_r(j, z) the
  // entries j >= i of row i of R (1/r_ii at j = i; rows i < cols), which
  // get_r(i, j) returns to any lane of the system; put_x(k, z) coordinate i
  // of solution k.
  // Each output is put by one slot of the system.  All 32 lanes of the warp
  // call it.
  template <int MAXC, class Load, class PutQ, class PutR, class GetR, class PutX>
  __device__ __forceinline__ void solve(int cols, int nrhs, Load load, PutQ put_q, PutR put_r, GetR get_r,
                                        PutX put_x) const {
    const int Wc = cols + nrhs;
    mpi::fzs<W> a[MAXC];  // the lane's row of A (its columns)
    Z Q, nxt;
    Q.f = nxt.f = 0;
#pragma unroll
    for (int k = 0; k < W; ++k) Q.r[k] = Q.i[k] = nxt.r[k] = nxt.i[k] = 0;
    if (row) nxt = load(0);
    // phase q projects the columns j > q on column q, C at a time, then
    // normalises column q + 1 (step Wc; the first phase, q = -1, only
    // normalises column 0)
    for (int q = -1; q < cols; ++q)
      for (int jb = q < 0 ? Wc : (q + 1) / C * C;; jb += C) {
        const bool pivot = jb >= Wc;
        if (pivot && q + 1 == cols) break;
        const int j = pivot ? q + 1 : jb + cs;
        const bool mine = row && j > q && j < Wc;
        Z u, v;
        if (pivot) {
          if (C > 1 && q >= 0) nxt = shfl(nxt, min(base + ((q + 1) % C - cs) * rows + i, 31));
          u = v = nxt;
        } else {
          u = v = Q;
          if (mine) v = q == 0 ? load(j) : static_cast<Z>(a[j]);
        }
        Z s = row_sum(mpi::mul<W>(mpi::conj<W>(u), v), row, false, rows);
        if (pivot) s = mpi::inv_sqrt<W>(s, mpi::inv_sqrt_steps<W>());
        const Z t = mpi::mul<W>(s, u);
        if (mine && i == (pivot ? j : q) && (!pivot || cs == 0)) put_r(j, s);
        if (pivot) {
          Q = t;
          if (row && cs == 0) put_q(j, t);
          break;
        }
        v = mpi::sub<W>(v, t);
        if (mine) {
          a[j] = v;
          if (j == q + 1) nxt = v;
          if (q + 1 == cols) put_q(j, v);
        }
      }
    __syncwarp();  // R's entries are visible to the system's slots
    // Back substitution, the right-hand sides dealt to the system's slots: lane
    // l keeps x_l once it is known, and x_j is the sum over the lanes of
    // y_j (lane j) and -r_jl x_l (lanes l > j), times 1/r_jj.  (One lane adding
    // the n - j products by itself took 25,000 clocks a coordinate in QD.)
    for (int k0 = 0; k0 < nrhs; k0 += C) {
      const int k = k0 + cs;
      const bool mine = row && k < nrhs;
      Z x;
      x.f = 0;
#pragma unroll
      for (int l = 0; l < W; ++l) x.r[l] = x.i[l] = 0;
      for (int j = cols - 1; j >= 0; --j) {
        const bool part = mine && i >= j && i < cols;
        Z z = x;
        if (part) z = get_r(j, i == j ? cols + k : i);
        if (part && i > j) z = mpi::mul<W>(z, x);
        z = row_sum(z, part, i > j, cols - j);
        if (part && i == j) {
          x = mpi::mul<W>(z, get_r(j, j));
          put_x(k, x);
        }
      }
    }
  }
};

}  // namespace ht
