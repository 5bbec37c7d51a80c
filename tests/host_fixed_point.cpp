// The integer arithmetic of the kernels (eri_scalar.cuh, rys_fixed.h, eri_fixed.cuh) built for the
// host, for test_integer_arithmetic.py.
#include <cmath>
#include <cstring>

using std::fma;
#define __host__
#define __device__
#define __forceinline__ inline
#include "eri_fixed.cuh"
#include "eri_scalar.cuh"
#include "rys_fixed.h"

extern "C" {

int64_t host_rsqrt(int64_t f) { return sx_rsqrt(f); }

int host_places1(const int64_t* c, int64_t f, int e) { return sx_places1(c, f, e); }

// H = 1/zeta + 1/eta; out: g, ge, d[3], k, ti, x0, x1, rT, rTe, rT2, g2, g2e
void host_quartet(double H, const int64_t* P, const int64_t* Q, int pu, int64_t tcut4, int64_t* out) {
  SxQuartet s;
  uint64_t h;
  memcpy(&h, &H, 8);
  sx_quartet(h, P, Q, pu, tcut4, s);
  const int64_t v[] = {s.g, s.ge, s.d[0], s.d[1], s.d[2], s.k, s.ti, s.x0, s.x1, s.rT, s.rTe, s.rT2, s.g2, s.g2e};
  memcpy(out, v, sizeof(v));
}

// sum_i x_i y_i z_i at the scales of biased exponents K (each >= its values').
double host_sum(int n, const double* x, const double* y, const double* z, const int* K) {
  int64_t acc[2] = {0, 0};
  const double* t[3] = {x, y, z};
  for (int i = 0; i < n; ++i) {
    int32_t l[3][2], v[2];
    for (int ax = 0; ax < 3; ++ax) {
      uint64_t u;
      memcpy(&u, t[ax] + i, 8);
      fx_split((uint32_t)(u >> 32), (uint32_t)u, K[ax], fx_top(ax), l[ax]);
    }
    fx_mul(l[0], l[1], v);
    fx_mac(v, l[2], acc);
  }
  return fx_flush(acc, K[0] + K[1] + K[2] - 3 * 1022, 0.0);
}

// The row of polynomial c[0 .. 7] (highest power first) at the position of T in its interval: value, exponent E,
// interval and position.
int64_t host_horner(const double* c, double T, int* E, int* ti, int64_t* x60) {
  int64_t row[8];
  rys_fx_row(c, row);
  uint64_t u;
  memcpy(&u, &T, 8);
  int32_t x0;
  uint32_t x1;
  rys_fx_locate(u, *ti, x0, x1);
  *x60 = ((int64_t)x0 << 29) + x1;
  return rys_fx_horner(row, x0, x1, E);
}

int host_table(int N, int* deg, int* sub, int* tcut, long long* off, const double** coef) {
  *deg = RYS_DEG;
  *sub = RYS_SUB;
  *tcut = RYS_TCUT[N];
  *off = RYS_COEF_OFFSET[N];
  *coef = RYS_COEF;
  return RYS_NMAX;
}
}
