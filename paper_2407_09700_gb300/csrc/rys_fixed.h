// Rys roots and weights from the generated table (rys_table.h) by Horner's rule in 64-bit
// fixed point.
//
// Why: a root and its weight are two degree-7 sums, 14 FP64 FMAs of 64 cycles each on GB300,
// a third to a half of the FP64 work of the one-lane kernels.  In integers one step is three
// IMAD.WIDE and a few shifts (~17 cycles), and the FP64 pipe is left with one conversion per value.
//
// Format.  A polynomial's row is eight 64-bit words: c_0 .. c_6 in units of 2^(E - 62), then
// c_7 in units of 2^(E - 56) in the high and E in the low half of the last word, with
// sum |c_k| < 2^E, so every partial sum fits 63 bits.  x in [-1, 1) is two's complement in units
// of 2^-60: a signed top word (2^-31) and 29 low bits.  A step drops the product of the low
// halves and the lowest two bits of the sum, so the sums are off by at most 72 units of 2^(E - 62), 32 of
// them from c_7 (44 seen), and the value by that and the rounding of its conversion (worst relative
// error 1.2e-16 against the polynomials, 1.15e-16 with FP64 sums).
#pragma once
#include <stdint.h>

#include "rys_table.h"

#ifndef __CUDACC__
#ifndef __host__
#define __host__
#define __device__
#define __forceinline__ inline
#endif
#endif

// Interval ti of T and x = 2 (RYS_SUB T - ti) - 1 from the bits of 0 <= T < 2^7.
__host__ __device__ __forceinline__ void rys_fx_locate(uint64_t bits, int& ti, int32_t& x0, uint32_t& x1) {
  const int e = (int)(bits >> 52);                               // T >= 0: no sign
  const uint64_t m = ((bits & 0xfffffffffffffULL) | 0x10000000000000ULL) << 11;   // leading bit at 63
  // RYS_SUB T (RYS_SUB = 4) in units of 2^-54: m 2^(e - 1023 - 63 + 2 + 54)
  const int r = 1023 + 63 - 2 - 54 - e;                          // e <= 1029: at least 1
  const uint64_t t = r < 64 ? m >> r : 0ull;
  ti = (int)(t >> 54);
  const uint64_t f = (t << 10) ^ 0x8000000000000000ULL;          // 2 frac - 1 in units of 2^-63
  x0 = (int32_t)(f >> 32);
  x1 = (uint32_t)f >> 3;
}

// The row's polynomial at x in units of 2^(*E - 62).
__host__ __device__ __forceinline__ int64_t rys_fx_horner(const int64_t c[8], int32_t x0, uint32_t x1, int* E) {
  *E = (int32_t)(uint32_t)(uint64_t)c[7];
  int64_t t = (c[7] >> 32) << 6;
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
  for (int k = 6; k >= 0; --k) {
    const int32_t t0 = (int32_t)(t >> 31);
    const int32_t t1 = (int32_t)((uint32_t)(t >> 2) & 0x1fffffffu);
    const int64_t d1 = (int64_t)t0 * (int32_t)x1 + (int64_t)t1 * x0;
    t = (int64_t)t0 * x0 + c[k] + (d1 >> 29);
  }
  return t;
}

// The row of a polynomial with coefficients c[0 .. RYS_DEG], highest power first (host).
inline void rys_fx_row(const double* c, int64_t* row) {
  double sum = 0.0;
  for (int k = 0; k <= RYS_DEG; ++k) sum += c[k] < 0 ? -c[k] : c[k];
  int E = 0;
  (void)__builtin_frexp(sum * (1.0 + 1e-12), &E);
  int e7 = 0;
  (void)__builtin_frexp(c[0], &e7);
  if (c[0] != 0.0 && E < e7 + 26) E = e7 + 26;                   // |c_7| < 2^(E - 25)
  for (int k = 0; k < RYS_DEG; ++k) row[k] = __builtin_llrint(__builtin_ldexp(c[RYS_DEG - k], 62 - E));
  const int64_t c7 = __builtin_llrint(__builtin_ldexp(c[0], 56 - E));
  row[7] = (int64_t)(((uint64_t)c7 << 32) | (uint32_t)E);
}
