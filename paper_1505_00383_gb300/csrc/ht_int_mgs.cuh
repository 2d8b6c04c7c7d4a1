// Modified Gram-Schmidt least squares on limb strings with one matrix row per
// lane (device only): the corrector's solve of the DD and QD tracker and of
// ht_mgs_solve_ex variant 2.
//
// A warp serves PP = min(8, 32 / rows) systems, lane (system, row).  A lane
// holds its row's entry of the pivot column in registers and its row in local
// memory; a dot product over the rows is one exact fixed-point sum across the
// system's lanes (row_sum), rounded once, so every lane of the system has the
// result.  There is no barrier: the warps are independent of each other.
//
// Why rows and not whole systems per lane: with a system per lane the columns
// were dealt to the warps of a CTA, which met at a barrier per column, and
// the columns lived in local memory behind runtime indexes; the warps waited
// for the pivot column's owner (4.7 barrier cycles an issue, 19 % of the
// issue slots used in QD).
#pragma once
#include "ht_int_row.cuh"

namespace ht {

template <int L>
struct RowLanes {
  static constexpr int W = IntW<L>::W, WA = W + 1;
  static constexpr int ND = (2 * WA + 3) / 4 * 4;  // exchanged words a lane, 16-byte multiple
  static constexpr int PP_MAX = 8;                 // systems a warp
  // Shared memory of one warp: the lanes' digits, then the systems' sums.
  static constexpr int WORDS = 32 * ND + PP_MAX * 2 * WA * 2;
  using Z = mpi::fz<W>;

  int rows, i, sub, base, head;  // rows a system; this lane's row, its system in the warp, that system's first lane
  bool row;                      // the lane has a row of a live system
  int32_t* dig;                  // shared [32][ND]
  int64_t* sums;                 // shared [PP_MAX][2 WA]

  static __host__ __device__ int systems(int rows) {
    const int pp = 32 / rows;
    return pp > PP_MAX ? PP_MAX : pp;
  }
  __device__ __forceinline__ RowLanes(int rows_, int32_t* xch) : rows(rows_) {
    const int lane = threadIdx.x & 31;
    sub = lane / rows;
    i = lane - sub * rows;
    base = sub * rows;
    head = mpi::bitlen32((uint32_t)rows) > 1 ? mpi::bitlen32((uint32_t)rows) : 1;
    row = sub < systems(rows);
    dig = xch;
    sums = reinterpret_cast<int64_t*>(xch + 32 * ND);
  }

  // sum of z over the system's rows: the frame, digits and rounding of mpi::sum
  __device__ __forceinline__ Z row_sum(const Z& z) const {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int b0 = row ? mpi::bound_exp<W>(z) : -30000;
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
    int4* q = reinterpret_cast<int4*>(dig + lane * ND);
#pragma unroll
    for (int k = 0; k < ND / 4; ++k) q[k] = make_int4(d[4 * k], d[4 * k + 1], d[4 * k + 2], d[4 * k + 3]);
    __syncwarp();
    if (row)
      for (int w = i; w < 2 * WA; w += rows) {  // the system's lanes deal the words
        int64_t s = 0;
#pragma unroll 4
        for (int k = 0; k < rows; ++k) s += dig[(base + k) * ND + w];
        sums[sub * 2 * WA + w] = s;
      }
    __syncwarp();
    int64_t c[2 * WA];
    const int s0 = row ? sub * 2 * WA : 0;
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

  // Least squares of [A | b_0 .. b_{nrhs-1}], cols <= rows <= 32, cols + nrhs
  // <= MAXC.  load(j) gives this lane's entry of column j, put_q(j, z) takes
  // its entry of the orthogonal factor (j < cols) or of a reduced right-hand
  // side, put_r(j, z) the entries j >= i of its row of R (1/r_ii at j = i;
  // lanes i < cols), put_x(k, z) coordinate i of solution k.  All 32 lanes of
  // the warp call it.
  template <int MAXC, class Load, class PutQ, class PutR, class PutX>
  __device__ __forceinline__ void solve(int cols, int nrhs, Load load, PutQ put_q, PutR put_r, PutX put_x) const {
    const int Wc = cols + nrhs;
    mpi::fzs<W> a[MAXC], r[MAXC];  // the lane's row of A, and of R
    Z Q, nxt;
    Q.f = nxt.f = 0;
#pragma unroll
    for (int k = 0; k < W; ++k) Q.r[k] = Q.i[k] = nxt.r[k] = nxt.i[k] = 0;
    if (row) nxt = load(0);
    // phase q projects the columns j > q on column q, then normalises column
    // q + 1 (j = Wc; the first phase, q = -1, only normalises column 0)
    for (int q = -1; q < cols; ++q)
      for (int j = q < 0 ? Wc : q + 1; j <= Wc; ++j) {
        const bool pivot = j == Wc;
        if (pivot && q + 1 == cols) break;
        Z u, v;
        if (pivot) {
          u = v = nxt;
        } else {
          u = Q;
          v = Q;
          if (row) v = q == 0 ? load(j) : static_cast<Z>(a[j]);
        }
        Z s = row_sum(mpi::mul<W>(mpi::conj<W>(u), v));
        if (pivot) s = mpi::inv_sqrt<W>(s, mpi::inv_sqrt_steps<W>());
        const Z t = mpi::mul<W>(s, u);
        const int jr = pivot ? q + 1 : j;
        if (i == (pivot ? q + 1 : q)) {
          r[jr] = s;
          if (row) put_r(jr, s);
        }
        if (pivot) {
          Q = t;
          if (row) put_q(jr, t);
        } else {
          v = mpi::sub<W>(v, t);
          a[j] = v;
          if (j == q + 1) nxt = v;
          if (row && q + 1 == cols) put_q(j, v);
        }
      }
    // back substitution: lane j forms x_j from its right-hand side and the
    // products it has collected (one exact sum), then every lane above
    // collects its product with x_j
    for (int k = 0; k < nrhs; ++k)
      for (int j = cols - 1; j >= 0; --j) {
        Z x;
        x.f = 0;
#pragma unroll
        for (int l = 0; l < W; ++l) x.r[l] = x.i[l] = 0;
        if (i == j && row) {
          Z S[MAXC];
          int cnt = 0;
          S[cnt++] = r[cols + k];
          for (int l = j + 1; l < cols; ++l) S[cnt++] = a[l];
          x = mpi::mul<W>(mpi::first_minus_rest<W, MAXC>(S, cnt), static_cast<Z>(r[j]));
          put_x(k, x);
        }
        if (j == 0) break;
        const int src = min(base + j, 31);
        x.f = __shfl_sync(0xffffffffu, x.f, src);
#pragma unroll
        for (int l = 0; l < W; ++l) {
          x.r[l] = __shfl_sync(0xffffffffu, x.r[l], src);
          x.i[l] = __shfl_sync(0xffffffffu, x.i[l], src);
        }
        if (i < j && row) a[j] = mpi::mul<W>(static_cast<Z>(r[j]), x);
      }
  }
};

}  // namespace ht
