// Host build of the limb-string routines of csrc/ht_mpi_ops.cuh that the
// tracker's predictor and least squares use, on raw limbs.
#include <cstdint>

#include "../paper_1505_00383_gb300/csrc/ht_mpi.cuh"
#include "../paper_1505_00383_gb300/csrc/ht_mpi_ops.cuh"

using namespace ht::mpi;

template <int W>
static fz<W> get(const int32_t* p) {
  fz<W> z;
  z.f = p[0];
  for (int k = 0; k < W; ++k) {
    z.r[k] = p[1 + k];
    z.i[k] = p[1 + W + k];
  }
  return z;
}
template <int W>
static void put(const fz<W>& z, int32_t* p) {
  p[0] = z.f;
  for (int k = 0; k < W; ++k) {
    p[1 + k] = z.r[k];
    p[1 + W + k] = z.i[k];
  }
}
template <int W>
static void add_sub_all(int64_t n, const int32_t* a, const int32_t* b, int32_t* sum, int32_t* diff) {
  for (int64_t q = 0; q < n; ++q, a += 2 * W + 1, b += 2 * W + 1, sum += 2 * W + 1, diff += 2 * W + 1) {
    put<W>(add<W>(get<W>(a), get<W>(b)), sum);
    put<W>(sub<W>(get<W>(a), get<W>(b)), diff);
  }
}
template <int WA, int W>
static void to_fz(int64_t n, const int32_t* ar, const int32_t* ai, int F, int32_t* out) {
  for (int64_t q = 0; q < n; ++q) put<W>(fixed_to_fz<WA, W>(ar + q * WA, ai + q * WA, F), out + q * (2 * W + 1));
}
static rz<8> real4(const double* d) {
  const double zero[4] = {0.0, 0.0, 0.0, 0.0};
  return real_of<8>(from_doubles<8, 4>(d, zero));
}
static void put_real(const rz<8>& z, int32_t* p) {
  p[0] = z.f;
  for (int k = 0; k < 8; ++k) p[1 + k] = z.r[k];
}

extern "C" {

int ops_add_sub(int W, int64_t n, const int32_t* a, const int32_t* b, int32_t* sum, int32_t* diff) {
  if (W == 5) add_sub_all<5>(n, a, b, sum, diff);
  else if (W == 8) add_sub_all<8>(n, a, b, sum, diff);
  else return -1;
  return 0;
}
int ops_to_fz(int W, int64_t n, const int32_t* ar, const int32_t* ai, int F, int32_t* out) {
  if (W == 5) to_fz<6, 5>(n, ar, ai, F, out);
  else if (W == 8) to_fz<9, 8>(n, ar, ai, F, out);
  else return -1;
  return 0;
}
// quotients and Hermite weights of quad-double a, b [n][4], u = a / b, d = b
void ops_hermite(int64_t n, const double* a, const double* b, int32_t* quo, int32_t* w) {
  for (int64_t q = 0; q < n; ++q) {
    const rz<8> d = real4(b + 4 * q), u = quotient<8>(real4(a + 4 * q), d, b[4 * q]);
    put_real(u, quo + 9 * q);
    rz<8> w4[4];
    hermite_weights<8>(u, d, w4);
    for (int k = 0; k < 4; ++k) put_real(w4[k], w + (4 * q + k) * 9);
  }
}
}
