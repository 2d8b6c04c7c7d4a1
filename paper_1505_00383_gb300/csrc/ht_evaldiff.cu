// Fused evaluation and differentiation of a polynomial system at many points
// (Section 3 of Verschelde & Yu 2015: the coeff, mon and sum kernels of
// Table tabcpugpu, here one kernel).
//
// Work decomposition.  A unit is (32 consecutive points, one polynomial).  One
// warp evaluates a unit: each lane owns one point, all lanes walk the same
// monomials in the same order, so every branch and every load of the system
// ("instructions" of Table tabmemory) is warp-uniform and served by one
// broadcast.  Units are dealt round-robin to the warps of a grid sized to the
// SMs, which balances the per-SMSP arithmetic pipe the kernel is bound by.
//
// Per monomial c * prod_{r} x_{v_r}^{a_r} with k variables of positive exponent:
//   cf    = c * prod_{a_r > 1} x_{v_r}^(a_r - 1)        (common factor, Section 1)
//   P_r   = cf * x_{v_0} ... x_{v_r}                    forward products, k mults
//   value = P_{k-1}
//   dv_r  = a_r * P_{r-1} * (x_{v_{r+1}} ... x_{v_{k-1}}) backward sweep
// which is the reverse mode of Table tabmoneval with the common factor folded
// into the first forward product: 3k - 3 complex multiplications for value and
// all k derivatives (the table's 3k - 5 products plus k + 1 multiplications by
// the common factor would take 4k - 4).
//
// Outputs are written in the vertical layout of Table tabtranspose; the
// Jacobian row of the unit's polynomial accumulates in place in the output
// array (it stays in L2 while the unit runs), so no scratch memory is used.
#ifndef HT_LIMBS
#error "compile once per precision with -DHT_LIMBS=1, 2 or 4"
#endif
#include <cooperative_groups.h>

#include <algorithm>

#include "ht_eval.cuh"
#include "ht_internal.h"
#include "ht_int_row.cuh"

namespace ht {

struct EvalArgs {
  PolyView v;
  const int32_t* poly_off;  // advanced to the first polynomial of the range
  int nv, np;               // np: polynomials in the range; val and jac hold them from index 0
  int j0;                   // first polynomial of the range
  double* val;
  double* jac;
  int64_t n_units;
};

template <int L, bool LOOP>
__global__ void __launch_bounds__(256) evaldiff_kernel(EvalArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t n = a.v.npts;
  const int64_t plane = (int64_t)a.nv * 2 * L * n;  // doubles per Jacobian row
  for (int64_t u = warp; u < a.n_units; u += n_warps) {
    const int j = (int)(u % a.np);
    const int64_t p = (u / a.np) * 32 + lane;
    if (p >= n) continue;  // lanes past the ragged tail sit the unit out
    cx<L> v = eval_poly<L, LOOP>(a.v, __ldg(a.poly_off + j), __ldg(a.poly_off + j + 1), a.nv, p, a.jac + (int64_t)j * plane);
    st<L>(a.val, j, n, p, v);
  }
}

#if HT_LIMBS == 1
// The same for few points, in double: a cluster of CTAs takes one polynomial
// for 32 points and deals its monomials to its warps.  A monomial's value and
// derivatives go to slots in its CTA's shared memory (the forward products
// wait in the derivatives' slots), and one warp per output then adds that
// output's terms in monomial order, from the whole cluster's shared memory,
// so every operation and its order are those of evaldiff_kernel, and so are
// the bits.  Polynomials of more terms than there are slots go in chunks.
//
// Why: GB300 issues a double-precision warp instruction every 64 clocks on
// each SM sub-partition, so a polynomial's time on one warp (evaldiff_kernel)
// is its instruction count times 64 clocks, whatever the batch; here the
// sub-partitions of one to eight SMs share it.
__global__ void __launch_bounds__(512) evaldiff_split_kernel(EvalArgs a, const int32_t* __restrict__ term_off,
                                                             const uint32_t* __restrict__ terms, int n_slots, int max_k) {
  extern __shared__ __align__(16) double sm[];  // slots [n_slots][2][32], sums [nv + 1][2][32], points [nv][2][32]
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, T = blockDim.x >> 5;
  __shared__ int cut_m[9], cut_s[9];  // the parts' first monomials and slots
  const auto cluster = cooperative_groups::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  double* sums = sm + (int64_t)n_slots * 64;
  double* xs = sums + (int64_t)(a.nv + 1) * 64;
  int* cursor = reinterpret_cast<int*>(xs + (int64_t)a.nv * 64);  // [nv + 1] next term of each output
  const int64_t n = a.v.npts, plane = (int64_t)a.nv * 2 * n;
  for (int64_t u = blockIdx.x / C; u < a.n_units; u += gridDim.x / C) {
    const int j = (int)(u % a.np);
    const int64_t pt = (u / a.np) * 32 + lane, p = pt < n ? pt : n - 1;  // lanes past the end repeat the last point
    const int m0 = __ldg(a.poly_off + j), m1 = __ldg(a.poly_off + j + 1), o0 = (a.j0 + j) * (a.nv + 1);
    // slot of monomial m (its value, then its derivatives), from the polynomial's first
    auto slot_of = [&](int m) { return __ldg(a.v.mon_off + m) - __ldg(a.v.mon_off + m0) + (m - m0); };
    for (int v = warp; v < a.nv; v += T) st<1>(xs, v, 32, lane, ld<1>(a.v.x, v, n, p));
    __syncthreads();
    for (int c0 = m0; c0 < m1;) {
      // the chunk from monomial c0 in C parts, CTA k's beginning at the first
      // monomial at or past slot s0 + k q; a part overshoots q by less than
      // one monomial, so it fits in n_slots
      const int s0 = slot_of(c0), q = min((slot_of(m1) - s0 + C - 1) / C, n_slots - max_k);
      if (threadIdx.x <= C) {
        int lo = c0, hi = m1;
        while (lo < hi) {
          const int mid = (lo + hi) / 2;
          if (slot_of(mid) - s0 < (int)threadIdx.x * q)
            lo = mid + 1;
          else
            hi = mid;
        }
        cut_m[threadIdx.x] = lo;
        cut_s[threadIdx.x] = slot_of(lo);
      }
      __syncthreads();
      const int cb = cut_m[rank], ce = cut_m[rank + 1], c1 = cut_m[C], sb = cut_s[rank];
      for (int m = cb + warp; m < ce; m += T) {
        const int beg = __ldg(a.v.mon_off + m), k = __ldg(a.v.mon_off + m + 1) - beg;
        const uint16_t* pr = a.v.pairs + beg;
        double* sl = sm + (int64_t)(slot_of(m) - sb) * 64;
        cx<1> cf = ld_coef<1>(a.v.coef + (int64_t)m * 2);
        for (int r = 0; r < k; ++r) {
          const uint16_t w = __ldg(pr + r);
          if ((w >> 8) == 1) continue;
          const cx<1> xr = ld<1>(xs, w & 0xff, 32, lane);
          for (int e = 1; e < (w >> 8); ++e) cf = cmul(cf, xr);
        }
        cx<1> P = cf;
        for (int r = 0; r < k; ++r) {
          st<1>(sl, 1 + r, 32, lane, P);
          P = cmul(P, ld<1>(xs, __ldg(pr + r) & 0xff, 32, lane));
        }
        st<1>(sl, 0, 32, lane, P);
        if (k < 2) continue;
        cx<1> S = ld<1>(xs, __ldg(pr + k - 1) & 0xff, 32, lane);
        for (int r = k - 2; r >= 1; --r) {
          st<1>(sl, 1 + r, 32, lane, cmul(ld<1>(sl, 1 + r, 32, lane), S));
          S = cmul(S, ld<1>(xs, __ldg(pr + r) & 0xff, 32, lane));
        }
        st<1>(sl, 1, 32, lane, cmul(cf, S));
      }
      cluster.sync();
      for (int o = rank + C * warp; o <= a.nv; o += C * T) {
        const int end = __ldg(term_off + o0 + o + 1);
        int t = c0 == m0 ? __ldg(term_off + o0 + o) : cursor[o];
        cx<1> acc = c0 == m0 ? czero<1>() : ld<1>(sums, o, 32, lane);
        // the terms' loads go ahead of the additions, which wait for each other
        for (int k = 0; k < C; ++k) {  // the parts hold ascending slots
          const int b = cut_s[k];
          const double* part = cluster.map_shared_rank(sm, k);
          int te = t, hi = end;  // terms t..te lie in this part
          while (te < hi) {
            const int mid = (te + hi) / 2;
            if ((int)(__ldg(terms + mid) & 0xffffffu) < cut_s[k + 1])
              te = mid + 1;
            else
              hi = mid;
          }
          constexpr int U = 8;
          while (t < te) {
            uint32_t w[U];
            cx<1> v[U];
#pragma unroll
            for (int i = 0; i < U; ++i) w[i] = __ldg(terms + min(t + i, te - 1));
#pragma unroll
            for (int i = 0; i < U; ++i) v[i] = ld<1>(part, (int)(w[i] & 0xffffffu) - b, 32, lane);
#pragma unroll
            for (int i = 0; i < U; ++i) {
              if (t + i >= te) break;
              // (an exponent's conversion costs as much as an addition on the
              // FP64 pipe; an FMA by 1 rounds as the addition does)
              const int ex = (int)(w[i] >> 24);
              if (ex <= 1)
                acc = cadd(acc, v[i]);
              else if (ex == 2)
                acc = caxpy(acc, 2.0, v[i]);
              else if (ex == 3)
                acc = caxpy(acc, 3.0, v[i]);
              else
                acc = caxpy(acc, (double)ex, v[i]);
            }
            t = min(t + U, te);
          }
        }
        if (c1 < m1) {
          st<1>(sums, o, 32, lane, acc);
          if (lane == 0) cursor[o] = t;
        } else if (pt < n) {
          if (o == 0)
            st<1>(a.val, j, n, p, acc);
          else
            st<1>(a.jac + (int64_t)j * plane, o - 1, n, p, acc);
        }
        __syncwarp();
      }
      cluster.sync();  // the slots are read: the next chunk, or the end of the CTA
      c0 = c1;
    }
  }
}

// Shared memory of the split kernel with n_slots slots.
static size_t split_smem(int nv, int n_slots) {
  return (size_t)n_slots * 512 + (size_t)(2 * nv + 1) * 512 + (size_t)(nv + 1) * sizeof(int);
}
#endif

template <int L, bool LOOP>
static int launch_v(const EvalArgs& a, int threads, cudaStream_t st) {
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, evaldiff_kernel<L, LOOP>, threads, 0);
  if (per_sm < 1) per_sm = 1;
  const int wpb = threads / 32;
  int64_t want = (a.n_units + wpb - 1) / wpb;
  int64_t grid = (int64_t)sm_count() * per_sm;
  if (grid > want) grid = want;
  evaldiff_kernel<L, LOOP><<<(unsigned)grid, threads, 0, st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "ht_eval_diff: launch");
  return HT_OK;
}


// ------------------------------------------------------------------------
// Integer-pipe variant for double double and quad double (see ht_mpi.cuh):
// the same reverse-mode sweep on multi-limb integer complex numbers.  Per unit
// (polynomial j, 32 points) each lane
//   1. converts its point's variables once (local memory) and their log2 moduli;
//   2. bounds every term of polynomial j -- log2|c| + sum a log2|x| for the
//      value, minus log2|x_v| plus log2 a_v for a derivative -- and fixes one
//      accumulator frame above the largest bound plus log2 of the term count;
//   3. accumulates value and Jacobian row as fixed-point limbs in local memory;
//   4. converts the accumulators to L doubles and writes the outputs.
template <int L>
__global__ void __launch_bounds__(128, 4) evaldiff_int_kernel(EvalArgs a, IntPoly ip,
                                                           const mpi::fz<IntW<L>::W>* __restrict__ cfz) {
  using Z = mpi::fz<IntW<L>::W>;
  Z X[kIntMaxVars];
  float lg[kIntMaxVars];
  mpi::fzs<IntW<L>::W> P[64];
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t n = a.v.npts;
  const int64_t plane = (int64_t)a.nv * 2 * L * n;
  for (int64_t u = warp; u < a.n_units; u += n_warps) {
    const int j = (int)(u % a.np);
    const int64_t p = (u / a.np) * 32 + lane;
    if (p >= n) continue;
    int_point<L>(a.v.x, a.nv, n, p, X, lg);
    int_row<L>(ip, cfz, a.poly_off[j], a.poly_off[j + 1], X, lg, a.nv, a.val + (int64_t)j * 2 * L * n,
               a.jac + (int64_t)j * plane, n, p, P);
  }
}

// The block's 32 points as limb strings and log2 moduli in shared memory; all
// threads of the CTA take part (lanes past the last point store zeros).
template <int L>
__device__ __forceinline__ void stage_points(const double* __restrict__ x, int nv, int64_t n, int64_t p, int32_t* xs,
                                             float* lgs) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, T = blockDim.x >> 5;
  for (int v = warp; v < nv; v += T) {
    double re[L], im[L];
#pragma unroll
    for (int l = 0; l < L; ++l) {
      re[l] = p < n ? x[((int64_t)(v * 2) * L + l) * n + p] : 0.0;
      im[l] = p < n ? x[((int64_t)(v * 2 + 1) * L + l) * n + p] : 0.0;
    }
    store_point<L>(xs, v, lane, mpi::from_doubles<IntW<L>::W, L>(re, im));
    lgs[v * 32 + lane] = mpi::log2_mod(re[0], im[0]);
  }
}

// Largest CTA of the block organisation, in warps: 32 for double double (64
// registers a thread without spills to speak of), 16 for quad double.  The
// integer multiply-add pipe bounds both, and at n = 32, 65,536 points twice
// the warps take DD from 33.2 to 29.4 ms; QD at 64 registers spills, and
// gained 2 % there while it lost 3 to 8 % on smaller systems.
template <int L>
constexpr int kBlkWarps = L == 4 ? 16 : 32;
// Row slots that pass through shared memory at a time in the split kernel
// (4 KB a warp).
template <int L>
constexpr int kSplitSlots = 8 / RowAcc<L>::Q;

// Block organisation of the same unit: a CTA takes a block of 32 points and
// a group of polynomials (as many as it has warps: one each).  The block's
// converted points live once in shared memory instead of once per lane and
// unit in local memory; the warp still walks one monomial with all lanes in
// step.
// Work items (polynomial group, point block) are ordered group-major, so a
// CTA keeps one group's monomials and coefficients (a QD coefficient is 68
// bytes) in its L1 across point blocks; the points are converted once per
// item.  The sums are the same exact integers, so the results are those of
// the per-unit kernel bit for bit.
//
// What bounds it: the integer multiply-add pipe (QD: 63 % busy, four fifths
// of that the limb products), then the arithmetic around the products.  At
// n = 32, 65,536 points: QD 79.4 -> 58.6 ms and DD 43.9 -> 29.4 ms with the
// steps of ht_mpi_eval.cuh (one operand of every product stays in registers:
// 27 % fewer instructions), the points and the row accumulators in 128-bit
// words, and the column-by-column product.
template <int L>
__global__ void __launch_bounds__(32 * kBlkWarps<L>, 1) evaldiff_intblk_kernel(
    EvalArgs a, IntPoly ip, const mpi::fz<IntW<L>::W>* __restrict__ cfz) {
  extern __shared__ __align__(16) int32_t xs[];  // [nv][32][NW] limb strings, then [nv][32] log2 moduli
  float* lgs = reinterpret_cast<float*>(xs + a.nv * 32 * SmemPoints<L>::NW);
  mpi::fzs<IntW<L>::W> P[64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, T = blockDim.x >> 5;
  const int64_t n = a.v.npts, plane = (int64_t)a.nv * 2 * L * n, n_blocks = (n + 31) / 32;
  const int n_groups = (a.np + T - 1) / T;
  const SmemPoints<L> X{xs, lane};
  const SmemLog lg{lgs, lane};
  for (int64_t item = blockIdx.x; item < n_blocks * n_groups; item += gridDim.x) {
    const int64_t b = item % n_blocks;
    const int j = (int)(item / n_blocks) * T + warp;
    const int64_t p = b * 32 + lane;
    __syncthreads();  // the previous block's points are no longer read
    stage_points<L>(a.v.x, a.nv, n, p, xs, lgs);
    __syncthreads();
    if (p >= n || j >= a.np) continue;  // lanes past the ragged tail and warps past the last polynomial
    int_row<L>(ip, cfz, a.poly_off[j], a.poly_off[j + 1], X, lg, a.nv, a.val + (int64_t)j * 2 * L * n,
               a.jac + (int64_t)j * plane, n, p, P);
  }
}

// The same for few points: the monomials of a polynomial are dealt to S warps
// of the CTA (contiguous ranges of about equal numbers of steps), G = T / S
// polynomials at a time.  Each warp bounds its own monomials' terms; the
// largest bounds over the S warps fix the frames.  Each accumulates its part
// of the row, and the parts are added as integers, so the results are the
// bits of the unsplit sums.  The time is one warp's share of a polynomial:
// the 16 polynomials of 246 monomials at 999 points (512 polynomials x
// blocks for 2,432 resident warps) took 4.4 ms unsplit, 1.14 ms with S = 4.
template <int L>
__global__ void __launch_bounds__(512, 1) evaldiff_intsplit_kernel(EvalArgs a, IntPoly ip,
                                                                 const mpi::fz<IntW<L>::W>* __restrict__ cfz, int S) {
  constexpr int W = IntW<L>::W, WA = IntW<L>::WA, Q = RowAcc<L>::Q, R = kSplitSlots<L>;
  extern __shared__ __align__(16) int32_t xs[];
  float* lgs = reinterpret_cast<float*>(xs + a.nv * 32 * SmemPoints<L>::NW);
  float* red = lgs + a.nv * 32;                 // bounds [T][nv + 1][32], then
  int4* part = reinterpret_cast<int4*>(red);    // row slots [T][R][Q][32]
  mpi::fzs<W> P[64];
  float Ev[kIntMaxVars + 1];
  int Fv[kIntMaxVars + 1];
  int4 acc[(kIntMaxVars + 1) * Q];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, T = blockDim.x >> 5, G = T / S;
  const int s = warp % S, w0 = warp - s;  // this warp's part, its polynomial's first warp
  const int nv = a.nv, n_slots = nv + 1;
  const int64_t n = a.v.npts, plane = (int64_t)nv * 2 * L * n, n_blocks = (n + 31) / 32;
  const int n_groups = (a.np + G - 1) / G;
  const SmemPoints<L> X{xs, lane};
  const SmemLog lg{lgs, lane};
  RowAcc<L> row{acc, Fv, nv};
  for (int64_t item = blockIdx.x; item < n_blocks * n_groups; item += gridDim.x) {
    const int64_t p = (item % n_blocks) * 32 + lane;
    const int j = (int)(item / n_blocks) * G + warp / S;
    const bool work = j < a.np;  // uniform in a warp; every warp takes every barrier
    __syncthreads();
    stage_points<L>(a.v.x, nv, n, p, xs, lgs);
    __syncthreads();
    int m0 = 0, m1 = 0, mb = 0, me = 0;
    if (work) {
      m0 = a.poly_off[j];
      m1 = a.poly_off[j + 1];
      // monomials [mb, me): the first whose steps begin at or past s/S and (s+1)/S of the polynomial's
      const int b0 = ip.step_off[m0];
      const int64_t len = ip.step_off[m1] - b0;
      auto cut = [&](int k) {
        const int target = b0 + (int)(len * k / S);
        int lo = m0, hi = m1;
        while (lo < hi) {
          const int mid = (lo + hi) / 2;
          if (ip.step_off[mid] < target)
            lo = mid + 1;
          else
            hi = mid;
        }
        return lo;
      };
      mb = cut(s);
      me = cut(s + 1);
      Ev[nv] = mpi::bounds_for_poly(ip.mon_off, ip.pairs, ip.clg, mb, me, lg, nv, Ev);
      for (int i = 0; i < n_slots; ++i) red[(warp * n_slots + i) * 32 + lane] = Ev[i];
    }
    __syncthreads();
    if (work) {
      for (int i = 0; i < n_slots; ++i) {
        float E = red[(w0 * n_slots + i) * 32 + lane];
        for (int k = 1; k < S; ++k) E = fmaxf(E, red[((w0 + k) * n_slots + i) * 32 + lane]);
        Fv[i] = mpi::frame_of<WA>(E, m1 - m0);
        row.zero(i);
      }
      mpi::run_steps<L>(ip.steps + ip.step_off[mb], ip.steps + ip.step_off[me], cfz + mb, X, row, P);
    }
    // R slots of every polynomial at a time through shared memory
    for (int i0 = 0; i0 < n_slots; i0 += R) {
      __syncthreads();  // the bounds, or the previous slots, are no longer read
      if (work)
        for (int r = 0; r < R && i0 + r < n_slots; ++r)
#pragma unroll
          for (int k = 0; k < Q; ++k) part[((warp * R + r) * Q + k) * 32 + lane] = acc[(i0 + r) * Q + k];
      __syncthreads();
      for (int r = s; r < R; r += S) {
        const int i = i0 + r;
        if (!work || i >= n_slots || p >= n) continue;
        int64_t c[4 * Q];
#pragma unroll
        for (int k = 0; k < 4 * Q; ++k) c[k] = 0;
        for (int q = 0; q < S; ++q)
#pragma unroll
          for (int k = 0; k < Q; ++k) {
            const int4 v = part[(((w0 + q) * R + r) * Q + k) * 32 + lane];
            c[4 * k] += v.x;
            c[4 * k + 1] += v.y;
            c[4 * k + 2] += v.z;
            c[4 * k + 3] += v.w;
          }
        mpi::carry<WA>(c);
        mpi::carry<WA>(c + WA);
        int32_t ar[WA], ai[WA];
#pragma unroll
        for (int k = 0; k < WA; ++k) {
          ar[k] = (int32_t)c[k];
          ai[k] = (int32_t)c[WA + k];
        }
        store_slot<L>(ar, ai, Fv[i], (i == nv ? a.val + (int64_t)j * 2 * L * n : a.jac + (int64_t)j * plane + (int64_t)i * 2 * L * n) + p, n);
      }
    }
  }
}

template <int L>
static int launch_int(const EvalArgs& a, const ht_system* s, int threads, cudaStream_t st) {
  const auto* cf = reinterpret_cast<const mpi::fz<IntW<L>::W>*>(s->d_coef_fz);
  const IntPoly ip{s->d_mon_off, s->d_pairs, s->d_step_off, s->d_steps, s->d_coef_lg};
  if (threads == 256) {  // block organisation (points in shared memory)
    const int64_t n_blocks = (a.v.npts + 31) / 32, sms = sm_count();
    const size_t xbytes = smem_points_bytes<L>(a.nv);
    EvalShape shape = s->shape;
    shape.np = a.np;  // of this range of polynomials
    const EvalSplit split = eval_split(shape, L, n_blocks, sms);
    const int S = split.S, G = split.G;
    const size_t smem_split = xbytes + (size_t)(S * G) * 32 *
                                           std::max<size_t>((a.nv + 1) * sizeof(float), kSplitSlots<L> * RowAcc<L>::Q * sizeof(int4));
    if (S > 1 && smem_split <= 220 * 1024) {
      raise_smem((const void*)evaldiff_intsplit_kernel<L>, smem_split);
      int per_sm = 0;
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, evaldiff_intsplit_kernel<L>, 32 * S * G, smem_split);
      if (per_sm < 1) per_sm = 1;
      const int64_t want = n_blocks * ((a.np + G - 1) / G);
      const int64_t grid = want < sms * per_sm ? want : sms * per_sm;
      evaldiff_intsplit_kernel<L><<<(unsigned)grid, 32 * S * G, smem_split, st>>>(a, ip, cf, S);
    } else {
      // as few groups of polynomials as the largest CTA allows, of equal size
      const int groups = (a.np + kBlkWarps<L> - 1) / kBlkWarps<L>;
      const int cta = 32 * ((a.np + groups - 1) / groups);
      raise_smem((const void*)evaldiff_intblk_kernel<L>, xbytes);
      int per_sm = 0;
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, evaldiff_intblk_kernel<L>, cta, xbytes);
      if (per_sm < 1) per_sm = 1;
      const int64_t want = n_blocks * groups;  // (point block, polynomial group) items
      const int64_t grid = want < sms * per_sm ? want : sms * per_sm;
      evaldiff_intblk_kernel<L><<<(unsigned)grid, cta, xbytes, st>>>(a, ip, cf);
    }
  } else {
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, evaldiff_int_kernel<L>, 128, 0);
    if (per_sm < 1) per_sm = 1;
    int64_t want = (a.n_units + 3) / 4;
    int64_t grid = (int64_t)sm_count() * per_sm;
    if (grid > want) grid = want;
    evaldiff_int_kernel<L><<<(unsigned)grid, 128, 0, st>>>(a, ip, cf);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "ht_eval_diff: launch");
  return HT_OK;
}

#if HT_LIMBS == 1
// A cluster of C CTAs per unit: the largest of 1, 2, 4, 8 that the SMs and
// the monomials have room for (10 points, the call: 10 polynomials of 10
// monomials 77 us on one warp each, 30 us with C = 1, 25 us with 4; 16 of 246
// monomials 709, 205 and, with 8, 71 us).  Returns false where one warp per
// unit is faster, or if the system needs more shared memory.
static bool launch_split(const EvalArgs& a, const ht_system* s, cudaStream_t st, int* rc) {
  const int64_t sms = sm_count(), max_terms = s->shape.max_terms, max_slots = s->shape.max_slots;
  int C = 8;
  while (C > 1 && (a.n_units * C > sms || C * 2 > max_terms)) C /= 2;
  // 16 warps, fewer when a part has fewer monomials and outputs
  const int warps = (int)std::max<int64_t>(1, std::min<int64_t>(16, std::max<int64_t>(max_terms, a.nv + 1)));
  // slots for a CTA's part of a polynomial, up to 96 KB of them (two CTAs a SM)
  const int n_slots = (int)std::min<int64_t>(192, (max_slots + C - 1) / C + s->max_k);
  const size_t smem = split_smem(a.nv, n_slots);
  if (smem > 220 * 1024) return false;
  if (C == 1) {
    const int64_t q = std::min<int64_t>(max_slots, n_slots - s->max_k);  // a chunk, as the kernel cuts it
    if (!double_split_pays(s->shape, a.n_units, sms, warps, (max_slots + q - 1) / q)) return false;
  }
  raise_smem((const void*)evaldiff_split_kernel, smem);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, evaldiff_split_kernel, 32 * warps, smem);
  if (per_sm < 1) per_sm = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(std::min<int64_t>(a.n_units, std::max<int64_t>(1, sms * per_sm / C)) * C));
  cfg.blockDim = dim3(32 * warps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, evaldiff_split_kernel, a, (const int32_t*)s->d_term_off,
                                     (const uint32_t*)s->d_terms, n_slots, s->max_k);
  if (e == cudaSuccess) e = cudaGetLastError();
  *rc = e == cudaSuccess ? HT_OK : cuda_fail(e, "ht_eval_diff: launch");
  return true;
}
#endif

template <int L>
int launch_evaldiff_l(const ht_system* s, int64_t n_pts, int j0, int j1, const double* x, double* val, double* jac,
                      cudaStream_t st) {
  EvalArgs a;
  a.v.mon_off = s->d_mon_off;
  a.v.pairs = s->d_pairs;
  a.v.coef = s->d_coef;
  a.v.x = x;
  a.v.npts = n_pts;
  a.poly_off = s->d_poly_off + j0;  // polynomials j0 .. j1 - 1, written from output row 0
  a.nv = s->nv;
  a.np = j1 - j0;
  a.j0 = j0;
  a.val = val;
  a.jac = jac;
  a.n_units = ((n_pts + 31) / 32) * a.np;
  const int threads = s->eval_threads > 0 ? s->eval_threads : 128;
  if (s->eval_variant == 2 && s->d_steps && s->nv <= kIntMaxVars && s->max_k <= 64)
    return launch_int<L>(a, s, threads, st);
  const bool loop = s->eval_variant != 0;  // default: compact bodies
#if HT_LIMBS == 1
  if (loop && s->d_terms) {  // few units: polynomials over the warps of a CTA or cluster
    int rc;
    if (launch_split(a, s, st, &rc)) return rc;
  }
#endif
  return loop ? launch_v<L, true>(a, threads, st) : launch_v<L, false>(a, threads, st);
}

template int launch_evaldiff_l<HT_LIMBS>(const ht_system*, int64_t, int, int, const double*, double*, double*,
                                         cudaStream_t);

}  // namespace ht
