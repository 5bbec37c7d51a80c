// Block fixed-point arithmetic for the Eq. 1 assembly of the FP64 path (arXiv 2407.09700,
// Sec. 2): the sum over roots and primitives of I_x I_y I_z on the integer pipe.
//
// Why.  On GB300 an FP64 warp instruction occupies a sub-partition's FP64 unit for 64 cycles, a
// 32 x 32 + 64-bit IMAD.WIDE for 2 (both measured; the two pipes run side by side).  The FP64
// class kernels keep the FP64 pipe 84-93 % busy, about 70 % of it in Eq. 1: one multiply and
// one FMA per value, root and primitive quartet.  As integers an FMA is three IMAD.WIDE.
//
// Format.  A batch of primitive quartets has one power-of-two scale 2^K per 2D-table entry
// (axis, n, m): the smallest that bounds the entry over the batch's primitives and roots, so
// |I| 2^-K < 1.  An entry is two limbs, l0 2^-top + l1 2^-(top + 28), both with its sign: 56
// fraction bits for I_x, 57 for I_y and I_z.  Before the scales are taken, the factor w Theta of
// I_z is spread over the three axes by powers of two (fx_third), so that a tight primitive's
// large prefactor does not meet a diffuse one's large I_x and I_y in the scales' product, and a
// batch holds primitive pairs of neighbouring exponents (sorted in the plan, the ket's up and down
// in turn): with p and d exponents from 0.1 to 400 the error against quadruple precision is
// 3.5e-16 (3.6e-15 unsorted, 1.0e-13 without the spreading too, FP64 8.6e-16).  A product I_x I_y
// keeps 57 fraction bits; the limb products of its sum with I_z accumulate by weight in 64-bit
// integers, exactly (at most FX_TERMS (primitive, root) terms per batch fit the headroom), and a
// batch's sum returns to FP64 once, at scale 2^(K_x + K_y + K_z).
//
// Accuracy.  Every truncation is absolute at 2^-57 of the three scales' product, which bounds the
// batch's products but need not be close to any: the axes' largest entries may come from different
// primitives and roots, and an entry k binades below its scale keeps 57 - k bits.  FP64 rounds each
// product and each partial sum at 2^-53 of itself, so the form pays while the scales' product stays
// within a few binades of the sum, which FX_SPREAD is for.  Measured against quadruple precision on
// 2 500 quartets of random contracted s/p/d pairs (depths 1..6, spreads up to FX_SPREAD, centres up
// to 4 or 10 bohr apart), error relative to the quartet's largest element: geometric means of the
// classes 1.5 to 3.4 times below FP64's ((dd|dd) 4.0e-15 and 8.8e-15 against 9.9e-15 and 2.0e-14),
// their worst quartets below FP64's worst in most classes ((dd|dd) 1.9e-12 and 2.9e-12 against
// 3.3e-12 and 7.9e-12) and at most a third above ((dd|ds) at 10 bohr 4.6e-13 against 3.4e-13); single
// quartets up to 75 times above.  J and K of small s/p/d molecules came out as close as with FP64 or
// closer (relative 2-norm of J, K: 3.0e-16, 6.5e-16 against 4.3e-16, 6.7e-16 on three atoms with p
// shells, 5.9e-16, 1.1e-15 against 6.6e-16, 4.6e-15 on two atoms of the 3s2p1d recipe).
// The entries of f and g classes spread over more binades (57 bits: 5.8e-15 against 2.5e-16), so
// classes above eight units of angular momentum keep FP64; with a third limb (84 bits, 2.0e-16) they
// gained nothing in time (12-atom s..g build 1138 ms against 1012 ms).
#pragma once
#include <stdint.h>

#define FX_TERMS 32      // most (primitive, root) terms accumulated between two returns to FP64
#define FX_LMAX 8        // most angular momentum la + lb + lc + ld of a class
// Most binades (l0 + l1) / 2 log2(zeta ratio) over a pair's primitives: an entry of degree n scales
// like zeta^(-n/2).  6-31G(d)-like shells have 13 and p, d exponents 0.1 .. 400 18 (no larger
// error than FP64); at 30 (0.1 .. 4000 in p and d) the error is 5e-15 against 0.5e-15, so wider
// shells keep FP64.  A mixed plan's primitives are not sorted; its spreads count 6 binades more: unsorted
// up to 14 binades the same random quartets are 1.8 to 3.5 times closer than with FP64 in the geometric mean
// ((dd|dd) 2.6e-15 against 7.3e-15, worst 4.0e-13 against 2.9e-12).
#define FX_SPREAD 20.0
#define FX_LIMB 28
#define FX_MASK 0x0fffffff
#define FX_POISON (1 << 20)   // K of an entry that held an infinity or a NaN

// Fraction bits of l0: axis 0, 1, 2 = x, y, z.
__host__ __device__ constexpr int fx_top(int ax) { return ax == 0 ? 28 : 29; }

// About e / 3 (any integer serves).
__host__ __device__ __forceinline__ int fx_third(int e) { return (e * 21846) >> 16; }

// Limbs of the double with words (hi, lo) at the scale of biased exponent emax >= its own,
// rounded to nearest.
__host__ __device__ __forceinline__ void fx_split(uint32_t hi, uint32_t lo, int emax, int top, int32_t l[2]) {
  const int e = (int)((hi >> 20) & 0x7ffu);
  const int32_t s = (int32_t)hi >> 31;
  const uint64_t m = e ? ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | lo) : 0ull;   // denormals: 0
  const int r = 63 - (top + FX_LIMB) + emax - e;   // (m << 11) 2^(top + 28 - 64 - (emax - e)), one bit more
  const uint64_t t = ((r < 64 ? (m << 11) >> r : 0ull) + 1ull) >> 1;
  l[0] = ((int32_t)(t >> FX_LIMB) ^ s) - s;
  l[1] = ((int32_t)((uint32_t)t & FX_MASK) ^ s) - s;
}

// v = x y (to nearest; v[1] >= 0).
__host__ __device__ __forceinline__ void fx_mul(const int32_t x[2], const int32_t y[2], int32_t v[2]) {
  const int64_t d1 = (int64_t)x[0] * y[1] + (1 << (FX_LIMB - 1)) + (int64_t)x[1] * y[0];
  const int64_t d0 = (int64_t)x[0] * y[0] + (d1 >> FX_LIMB);
  v[1] = (int32_t)((uint32_t)d0 & FX_MASK);
  v[0] = (int32_t)(d0 >> FX_LIMB);
}

// acc += v z, limb products by weight (the product of the low limbs, below 2^-60, is left out).
__host__ __device__ __forceinline__ void fx_mac(const int32_t v[2], const int32_t z[2], int64_t acc[2]) {
  acc[0] += (int64_t)v[0] * z[0];
  acc[1] += (int64_t)v[0] * z[1];
  acc[1] += (int64_t)v[1] * z[0];
}

// 2^k as a double (0 below the normal range, 2^1023 above it); NaN for a poisoned sum of Ks.
__host__ __device__ __forceinline__ double fx_pow2(int k) {
  int b = k + 1023;
  b = b < 0 ? 0 : (b > 0x7fe ? 0x7fe : b);
  if (k >= FX_POISON / 2) b = 0x7ff;
  const uint64_t u = ((uint64_t)(uint32_t)b << 52) | (k >= FX_POISON / 2 ? 1ull << 51 : 0ull);
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double r;
  __builtin_memcpy(&r, &u, 8);
  return r;
#endif
}

// a + the batch's sum, K = K_x + K_y + K_z of the slot's entries (the top limbs of v and z
// together carry 58 fraction bits).
__host__ __device__ __forceinline__ double fx_flush(const int64_t acc[2], int K, double a) {
  return fma((double)(acc[0] + (acc[1] >> FX_LIMB)), fx_pow2(K - 58), a);
}
