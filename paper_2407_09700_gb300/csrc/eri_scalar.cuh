// Per-primitive-quartet scalars in integer arithmetic: P - Q, T = rho |P - Q|^2 with
// rho = zeta eta / (zeta + eta), the Rys roots and weights and the recurrence coefficients, for
// the one-lane kernels (eri_small.cu).
//
// Why.  In FP64 these are ~30 operations of 64 cycles (three subtractions, an inverse square
// root, a dozen products, the large-T limit's inverse square root) and 24 per root; the one-lane kernels
// kept the FP64 pipe 85 % busy and the integer pipes 10-15 %.  Here one FP64 addition is left.
//
// With H = 1/zeta + 1/eta (one FP64 addition) and g = 1/sqrt(H): rho = g^2, zeta/(zeta+eta) =
// g^2/eta, eta/(zeta+eta) = g^2/zeta and 1/sqrt(zeta+eta) = g / sqrt(zeta eta), the last factor kept
// with the pair's prefactor.
//
// Formats: "mantissa" = int64 m and exponent e for m 2^(e - 62), 0 <= m < 2^62, relative error
// 2^-60 per product; "fixed" = units of 2^-60 (or limbs h 2^-30 + l 2^-60), values below 2;
// lengths of the bra (ket) in units of 2^a (2^b), chosen per primitive pair so that every
// C = P - A - u eta/(zeta+eta) (P - Q) fits: |C| <= |P - A| + sqrt(c_N / zeta), c_N the largest
// squared zero of the Hermite polynomial of order 2N (u <= min(1, c_N / T)).  Weights are held in
// units of about 1/sqrt(T).  Errors are a few 2^-60 of these units: seven bits below FP64's for
// values of the units' size, above them for a value whose C's are far below theirs.  SX_TMAX bounds
// that for tight shells; the smaller components of a quartet, or ones that vanish nearly by symmetry,
// are accurate relative to its largest rather than to themselves.
#pragma once
#include <stdint.h>

#include "eri_internal.h"
#include "rys_fixed.h"

// Largest zeta |P - Q|^2 of the FP64 launches with pairs of three or more units of angular momentum, odd in all
// ((dp| and (fs|).  On one centre, where P - A = 0, each of their values has a factor C, about
// 1 / (zeta |P - Q|), sqrt(T) below the unit that the half inverse exponent sets, and carries about
// 2^-57.6 sqrt(zeta |P - Q|^2): 1.7e-15 at this limit, where FP64 keeps 1e-15.  Wider classes run in FP64.  Pairs
// of even angular momentum have values of the unit's size, and the unit of a (ps| pair goes by C.
#define SX_TMAX 131072.0

// Fewest binary places of the positions in FP64 and in FP32 launches (64 and 2^28 bohr to either side of
// the molecule's middle).  P - Q is off by up to a unit, the coordinates in FP64 by 2^-53 of themselves:
// with an atom 1e3, 1e5 and 1e7 bohr away the unit cost J of a compact molecule 4e-15, 8e-13 and 6e-11.
#define SX_PU 52
#define SX_PU32 30

#define SX_M30 0x3fffffff
#define SX_M31 0x7fffffff

#ifdef __CUDACC__
#define SX_HD __host__ __device__ __forceinline__
#else
#define SX_HD inline
#endif

// x y 2^-62 for 0 <= x, y < 2^62 (off by at most 2 units)
SX_HD int64_t sx_mulm(int64_t x, int64_t y) {
  const int32_t xh = (int32_t)(x >> 31), yh = (int32_t)(y >> 31);
  const int32_t xl = (int32_t)((uint32_t)x & SX_M31), yl = (int32_t)((uint32_t)y & SX_M31);
  const uint64_t d1 = (uint64_t)((int64_t)xh * yl + (1 << 30)) + (uint64_t)((int64_t)xl * yh);
  return (int64_t)xh * yh + (int64_t)(d1 >> 31);
}

// m 2^-s rounded to nearest for s > 0, m 2^-s (exact by the caller's bounds) for s <= 0; m < 2^62
SX_HD int64_t sx_shift(int64_t m, int s) {
  if (s > 0) return s < 63 ? ((m >> (s - 1)) + 1) >> 1 : 0;
  return -s < 63 ? (int64_t)((uint64_t)m << -s) : 0;
}

// A fixed value in limbs: h 2^-30 + l 2^-60, 0 <= l < 2^30.
struct SxL {
  int32_t h, l;
};
SX_HD SxL sx_limbs(int64_t t60) { return SxL{(int32_t)(t60 >> 30), (int32_t)((uint32_t)t60 & SX_M30)}; }
SX_HD int64_t sx_int(SxL x) { return ((int64_t)x.h << 30) + x.l; }
// sums of products: d0 in units of 2^-60, d1 of 2^-90 (with a half unit of d0 for the rounding; the
// products of low limbs, below 2^-60, stay out).  At most three products of values up to 1.6.
struct SxSum {
  int64_t d0, d1;
  SX_HD SxSum() : d0(0), d1(1 << 29) {}
};
SX_HD void sx_mac(SxSum& s, SxL x, SxL y) {
  s.d0 += (int64_t)x.h * y.h;
  s.d1 += (int64_t)x.h * y.l;
  s.d1 += (int64_t)x.l * y.h;
}
SX_HD int64_t sx_value(const SxSum& s) { return s.d0 + (s.d1 >> 30); }
SX_HD int64_t sx_mul(SxL x, SxL y) {
  SxSum s;
  sx_mac(s, x, y);
  return sx_value(s);
}

// 1 / sqrt(f 2^-60) in units of 2^-60 (at most 2^60 - 1) for 2^60 <= f < 2^62: an FP32 estimate y0 and
// the second-order step y0 (1 + e/2 + 3 e^2 / 8), e = 1 - f y0^2 (|e| < 2^-20, so e^3 is below
// 2^-60).
SX_HD int64_t sx_rsqrt(int64_t f) {
  const float ff = (float)(int32_t)(f >> 32) * (1.0f / 268435456.0f);
#ifdef __CUDA_ARCH__
  int32_t y0 = __float2int_rn(rsqrtf(ff) * 1073741824.0f);
#else
  int32_t y0 = (int32_t)(1073741824.0 / __builtin_sqrt((double)ff));
#endif
  y0 = y0 < 0x3fffffff ? y0 : 0x3fffffff;
  const int64_t s = ((int64_t)y0 * y0) << 2;                           // units of 2^-62
  const int64_t e = (1LL << 60) - sx_mulm(f, s);                       // units of 2^-60
  const int32_t eh = (int32_t)(e >> 21);                               // units of 2^-39
  const int64_t c = (e >> 1) + ((3 * ((int64_t)eh * eh)) >> 21);
  const int64_t y = ((int64_t)y0 << 30) + (((int64_t)y0 * (int32_t)(c >> 16)) >> 14) +
                    (((int64_t)y0 * (int32_t)(c & 0xffff)) >> 30);
  return y < (1LL << 60) ? y : (1LL << 60) - 1;
}

SX_HD int sx_clz(uint64_t v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}

// Most places p with |c0|, |c1| < 2^(60 - p) and hz < 2^(57 - 2 p) (0 if none).
SX_HD int sx_places(const int64_t c0[3], const int64_t c1[3], int64_t hz) {
  uint64_t m = 0;
  for (int i = 0; i < 3; ++i) m |= (uint64_t)(c0[i] ^ (c0[i] >> 63)) | (uint64_t)(c1[i] ^ (c1[i] >> 63));
  const int p = sx_clz(m) - 4, q = (sx_clz((uint64_t)hz) - 7) >> 1;
  const int r = p < q ? p : q;
  return r > 0 ? r : 0;
}

// Most places p with f 2^(e - 62) < 2^-p; f < 2^62.
SX_HD int sx_room(int64_t f, int e) { return sx_clz((uint64_t)f) - 2 - e; }

// Most places p with |c| < 2^(59 - p) and f 2^(e - 62) < 2^(-1 - p) (0 if none).
SX_HD int sx_places1(const int64_t c[3], int64_t f, int e) {
  uint64_t m = 0;
  for (int i = 0; i < 3; ++i) m |= (uint64_t)(c[i] ^ (c[i] >> 63));
  const int p = sx_clz(m) - 5, q = sx_room(f, e) - 1;
  const int r = p < q ? p : q;
  return r > 0 ? r : 0;
}

// The scalars of one primitive quartet.
struct SxQuartet {
  int64_t g;                 // g = g 2^-60 2^ge
  int ge;
  int64_t g2;                // rho = g2 2^(g2e - 62)
  int g2e;
  int64_t d[3];              // P - Q = d 2^-60 2^k, the largest |d| in [2^59, 2^60)
  int k;
  int ti;                    // Rys lookup: interval and position, or the large-T limit (ti = -1)
  int32_t x0;
  uint32_t x1;
  int64_t rT, rT2;           // 1/sqrt(T) and 1/T as mantissas, exponents rTe and 2 rTe (ti = -1)
  int rTe;
};

// P, Q in units of 2^-pu, |P - Q| < 2^60 of them; tcut4: RYS_SUB times the large-T cutoff in units
// of 2^-54 of RYS_SUB T.
SX_HD void sx_quartet(uint64_t hbits, const int64_t P[3], const int64_t Q[3], int pu, int64_t tcut4, SxQuartet& s) {
  // H = f 2^e2, 1 <= f < 4, e2 even
  const int e = (int)(hbits >> 52) - 1023;
  const int e2 = e & ~1;
  const int64_t f = (int64_t)((hbits & 0xfffffffffffffULL) | 0x10000000000000ULL) << (8 + (e & 1));
  s.g = sx_rsqrt(f);
  s.ge = -(e2 >> 1);
  s.g2 = sx_mulm(s.g << 2, s.g << 2);
  s.g2e = -e2;
  int64_t d0 = P[0] - Q[0], d1 = P[1] - Q[1], d2 = P[2] - Q[2];
  const uint64_t big = (uint64_t)(d0 ^ (d0 >> 63)) | (uint64_t)(d1 ^ (d1 >> 63)) | (uint64_t)(d2 ^ (d2 >> 63));
  int sh = sx_clz(big) - 4;                                            // at least 0
  sh = sh < 59 ? sh : 59;
  s.d[0] = (int64_t)((uint64_t)d0 << sh);
  s.d[1] = (int64_t)((uint64_t)d1 << sh);
  s.d[2] = (int64_t)((uint64_t)d2 << sh);
  s.k = 60 - pu - sh;
  SxSum q;
  for (int i = 0; i < 3; ++i) {
    const SxL v = sx_limbs(s.d[i]);
    q.d0 += (int64_t)v.h * v.h;
    q.d1 += (int64_t)v.h * v.l;
  }
  const int64_t S = q.d0 + (q.d1 >> 29);                               // |P - Q|^2 = S 2^-60 2^2k
  const int64_t T = sx_mulm(S > 0 ? S : 0, s.g2);                      // T = T 2^(st - 60)
  const int st = 2 * s.k - e2;
  // RYS_SUB T (RYS_SUB = 4) in units of 2^-54, when T < 128
  bool far = st > 10 || (st > 4 && (T >> (67 - st)) != 0);
  int64_t t54 = 0;
  if (!far) {
    t54 = sx_shift(T, 4 - st);
    far = t54 >= tcut4;
  }
  s.ti = (int)(t54 >> 54);
  const uint64_t fr = ((uint64_t)t54 << 10) ^ 0x8000000000000000ULL;
  s.x0 = (int32_t)(fr >> 32);
  s.x1 = (uint32_t)fr >> 3;
  s.rT = s.rT2 = 0;
  s.rTe = 0;
  if (far) {
    // T = f 2^-60 2^ft, f in [2^60, 2^62), ft even
    const int lz = sx_clz((uint64_t)T) - 2;                            // leading bit to 61 (or 60)
    const int l = (lz + st) & 1 ? lz - 1 : lz;
    s.ti = -1;
    s.rT = sx_rsqrt(l >= 0 ? T << l : T >> -l) << 2;
    s.rTe = -((st - l) >> 1);
    s.rT2 = sx_mulm(s.rT, s.rT);
  }
}

// Root n and its weight as mantissas.  coef: fixed-point rows of N (rys_fixed.h); asym: the limit's
// u T and w sqrt(T) per root as (mantissa, exponent) pairs.
#ifdef __CUDACC__
__device__ __forceinline__ void sx_root(const int64_t* __restrict__ coef, const longlong2* __restrict__ asym, int N,
                                        const SxQuartet& s, int n, int64_t& um, int& ue, int64_t& wm, int& we) {
  if (s.ti >= 0) {
    const longlong2* c = reinterpret_cast<const longlong2*>(coef) + ((size_t)s.ti * N + n) * (RYS_DEG + 1);
    int64_t row[RYS_DEG + 1];
#pragma unroll
    for (int k = 0; k < (RYS_DEG + 1) / 2; ++k) {
      const longlong2 v = __ldg(c + k);
      row[2 * k] = v.x;
      row[2 * k + 1] = v.y;
    }
    um = rys_fx_horner(row, s.x0, s.x1, &ue);
#pragma unroll
    for (int k = 0; k < (RYS_DEG + 1) / 2; ++k) {
      const longlong2 v = __ldg(c + (RYS_DEG + 1) / 2 + k);
      row[2 * k] = v.x;
      row[2 * k + 1] = v.y;
    }
    wm = rys_fx_horner(row, s.x0, s.x1, &we);
    um = um > 0 ? um : 0;
    wm = wm > 0 ? wm : 0;
  } else {
    const longlong2 au = __ldg(asym + 2 * n), aw = __ldg(asym + 2 * n + 1);
    um = sx_mulm(au.x, s.rT2);
    ue = (int)au.y + 2 * s.rTe;
    wm = sx_mulm(aw.x, s.rT);
    we = (int)aw.y + s.rTe;
  }
}
#endif

// 2^k for -1022 <= k <= 1023
SX_HD double sx_pow2(int k) {
  const uint64_t u = (uint64_t)(k + 1023) << 52;
  double d;
  __builtin_memcpy(&d, &u, 8);
  return d;
}

// Mantissa and exponent of a normal v > 0, v = m 2^(e - 62), 2^61 <= m < 2^62 (exact).
SX_HD void sx_from_double(double v, int64_t* m, int* e) {
  uint64_t u;
  __builtin_memcpy(&u, &v, 8);
  *e = (int)(u >> 52) - 1022;
  *m = (int64_t)((u & 0xfffffffffffffULL) | 0x10000000000000ULL) << 9;
}
