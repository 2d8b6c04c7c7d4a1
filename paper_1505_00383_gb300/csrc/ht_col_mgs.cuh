// Modified Gram-Schmidt least squares in double with one matrix column per
// lane, for groups of few paths (device only).
//
// GB300 issues a double-precision warp instruction every 64 clocks on each SM
// sub-partition whatever number of lanes it has, so with a system per lane a
// round costs a group of one path what it costs 32.  Here a warp serves
// 32 / (n + nrhs - 1) systems: lane (system, column), the column in registers
// and the pivot column in shared memory, so that one instruction projects all
// columns of its systems.  Every column sees the operations of mgs_team in
// their order, so the bits are the same.  While the columns behind the pivot
// die off their lanes idle, which is why it is slower per path once every SM
// has more than four warps of it (n = 16: 2 systems a warp; the crossover is
// near 8 paths an SM).
#pragma once
#include "ht_eval.cuh"

namespace ht {

struct ColLanes {
  static constexpr int MAX = 16;    // largest n
  static constexpr int WARPS = 4;   // warps of a CTA that solve (one per sub-partition)

  static __host__ __device__ int lanes(int n, int nrhs) { return n + nrhs - 1; }
  static __host__ __device__ int systems(int n, int nrhs) { return 32 / lanes(n, nrhs); }
  // double2 words of shared memory of one warp: per system the pivot column
  // [n], R [n][n + nrhs] and the solutions [nrhs][n]
  static __host__ __device__ int words(int n, int nrhs) {
    return systems(n, nrhs) * (n + n * (n + nrhs) + nrhs * n);
  }

  // All 32 lanes call it.  load(i, j): entry (i, j) of [A | b] of this lane's
  // system; put(k, i, z): coordinate i of solution k (called by one lane);
  // live: this lane's system exists.  n <= N: the loops over the rows are
  // unrolled N times, and a row past n still holds the FP64 pipe (predicated
  // off: n = 6 with N = 16 took 106,000 clocks, as many per column as n = 16).
  template <int N, class Load, class Put>
  static __device__ __forceinline__ void solve(int n, int nrhs, bool live, double2* sh, Load load, Put put) {
    const int lane = threadIdx.x & 31, lp = lanes(n, nrhs), sys = min(lane / lp, systems(n, nrhs) - 1), W = n + nrhs;
    const int c = lane - (lane / lp) * lp;
    double2* q = sh + sys * (n + n * W + nrhs * n);
    double2 *R = q + n, *xs = R + n * W;
    live = live && lane < lp * systems(n, nrhs);
    int j = c < n ? c : n + 1;  // this lane's column: lane 0 takes the first right-hand side once column 0 is done
    cx<1> a[N];
    auto load_column = [&]() {
#pragma unroll
      for (int i = 0; i < N; ++i)
        if (i < n) a[i] = live ? load(i, j) : czero<1>();
    };
    load_column();
    double s = 0.0;
    if (c == 0) {
#pragma unroll
      for (int i = 0; i < N; ++i)
        if (i < n) s = fma(a[i].im, a[i].im, fma(a[i].re, a[i].re, s));
    }
    for (int p = 0; p < n; ++p) {
      if (c == p && live) {  // normalise the pivot column (s is its squared norm)
        const double inv = r_div(1.0, r_sqrt(s));
#pragma unroll
        for (int i = 0; i < N; ++i)
          if (i < n) {
            const cx<1> v = cscale_r(a[i], inv);
            q[i] = make_double2(v.re, v.im);
          }
        R[p * W + p] = make_double2(inv, 0.0);
      }
      __syncwarp();
      if (p == 0 && c == 0) {
        j = n;
        load_column();
      }
      if (j > p && live) {
        cx<1> r = czero<1>();
#pragma unroll
        for (int i = 0; i < N; ++i)
          if (i < n) {
            const double2 u = q[i];
            r.re = fma(u.x, a[i].re, r.re);
            r.re = fma(u.y, a[i].im, r.re);
            r.im = fma(u.x, a[i].im, r.im);
            r.im = fma(-u.y, a[i].re, r.im);
          }
        R[p * W + j] = make_double2(r.re, r.im);
#pragma unroll
        for (int i = 0; i < N; ++i)
          if (i < n) {
            const double2 u = q[i];
            a[i].re = fma(-r.re, u.x, a[i].re);
            a[i].re = fma(r.im, u.y, a[i].re);
            a[i].im = fma(-r.re, u.y, a[i].im);
            a[i].im = fma(-r.im, u.x, a[i].im);
          }
        if (j == p + 1 && j < n) {
          s = 0.0;
#pragma unroll
          for (int i = 0; i < N; ++i)
            if (i < n) s = fma(a[i].im, a[i].im, fma(a[i].re, a[i].re, s));
        }
      }
      __syncwarp();
    }
    // back substitution: the first nrhs lanes of a system, one right-hand side each
    if (c < nrhs && live) {
      double2* x = xs + c * n;
      for (int p = n - 1; p >= 0; --p) {
        const double2 y = R[p * W + n + c];
        cx<1> acc{y.x, y.y};
        for (int k = p + 1; k < n; ++k) {
          const double2 r = R[p * W + k], u = x[k];
          acc.re = fma(-r.x, u.x, acc.re);
          acc.re = fma(r.y, u.y, acc.re);
          acc.im = fma(-r.x, u.y, acc.im);
          acc.im = fma(-r.y, u.x, acc.im);
        }
        const cx<1> v = cscale_r(acc, R[p * W + p].x);
        x[p] = make_double2(v.re, v.im);
        put(c, p, v);
      }
    }
    __syncwarp();  // the shared memory may be reused
  }
  template <class Load, class Put>
  static __device__ __forceinline__ void solve_any(int n, int nrhs, bool live, double2* sh, Load load, Put put) {
    if (n <= 4)
      solve<4>(n, nrhs, live, sh, load, put);
    else if (n <= 6)
      solve<6>(n, nrhs, live, sh, load, put);
    else if (n <= 8)
      solve<8>(n, nrhs, live, sh, load, put);
    else if (n <= 10)
      solve<10>(n, nrhs, live, sh, load, put);
    else if (n <= 12)
      solve<12>(n, nrhs, live, sh, load, put);
    else
      solve<MAX>(n, nrhs, live, sh, load, put);
  }
};

}  // namespace ht
