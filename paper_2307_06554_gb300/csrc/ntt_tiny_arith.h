// Arithmetic of the unit for the smallest moduli (ntt_tiny.cuh): Plantard's
// multiplication by a constant in 32-bit words (T. Plantard, "Efficient word
// size modular arithmetic", 2021; the signed form for small moduli of Huang
// et al., "Improved Plantard arithmetic for lattice-based cryptography",
// 2022).  Plain C++, so that the bounds are tested on the host too.
//
// With q' = q^-1 mod 2^32 and W the centred residue of -w 2^32, let
// z = a (W q') mod 2^32 (signed); then z q - a W = k 2^32 with k congruent
// to a w, and |k| <= (q - 1) / 2 because |z| <= 2^31 and |a W| < 2^31.
// k comes from the high half of z alone: with zl = z mod 2^16,
//   (z >> 16) q = (k 2^32 + a W - zl q) / 2^16,
// so floor(((z >> 16) q + c) / 2^16) is k exactly when
//   0 <= a W - zl q + c 2^16 < 2^32.
// zl q lies anywhere in [0, 2^16 q), so c = 2^15 + (Q - 1) / 2 with the
// largest modulus Q centres that range for Q and leaves room below it for
// every smaller one: |a W| <= 2^31 - 2^15 (Q + 1) is enough.  (c = 2^15 alone
// is exact only to 2^31 - 2^16 q for negative products: 16897, 17921 and
// 18433 then give wrong products.)  One constant for all moduli is an
// immediate operand; 2^15 + (q - 1) / 2 per modulus, in a register, made
// k_ntt_tiny_shared 2 % slower (14.9 -> 15.2 us, 4096 products).
#pragma once
#include <cstdint>

#include "host_math.h"

#ifdef __CUDACC__
#define PM_HD __host__ __device__ __forceinline__
#else
#define PM_HD inline
#endif

namespace pm {

constexpr uint32_t kTinyQMax = 18500;  // exclusive
constexpr int kTinyLogM = 3;           // coefficients per remaining ring: 2^3
constexpr int kTinyM = 1 << kTinyLogM;
// largest factor of a product by a constant, in units of (q - 1) / 2
constexpr int kTinyLim = 18;

constexpr int kTinyRound = (1 << 15) + (int)(kTinyQMax - 2) / 2;  // c for Q = kTinyQMax - 1

// largest |a W| with an exact quotient, for either sign; the negative side
// shrinks as q grows, so the largest modulus decides both
constexpr int64_t tiny_product_bound(int64_t q) {
  const int64_t below = kTinyRound * (1ll << 16) - (q * ((1ll << 16) - 1));
  const int64_t above = (1ll << 32) - 1 - kTinyRound * (1ll << 16);
  return below < above ? below : above;
}
constexpr int64_t tiny_largest_product(int64_t q) { return (int64_t)kTinyLim * ((q - 1) / 2) * ((q - 1) / 2); }
static_assert(tiny_largest_product(kTinyQMax - 1) <= tiny_product_bound(kTinyQMax - 1),
              "kTinyLim and kTinyQMax keep every product within the exact range");
// the sums of eight products in the small rings, times W = 1 when reduced
static_assert(kTinyM <= kTinyLim, "a ring's sums stay below the largest product");

struct TinyMod {
  int q, qinv;  // the prime, q^-1 mod 2^32
};

// z = a (W q') mod 2^32 -> a w mod q in [-(q-1)/2, (q-1)/2], before the last shift
PM_HD int tiny_pre(int z, const TinyMod& m) { return (z >> 16) * m.q + kTinyRound; }
// the low product wraps: unsigned, where that is defined
PM_HD int tiny_low(int a, int w) { return (int)((uint32_t)a * (uint32_t)w); }
PM_HD int tiny_mul(int a, int w, const TinyMod& m) { return tiny_pre(tiny_low(a, w), m) >> 16; }

// x, y -> x + w y, x - w y
PM_HD void tiny_ct(int& x, int& y, int w, const TinyMod& m) {
  const int s = x + tiny_mul(y, w, m);
  y = 2 * x - s;
  x = s;
}

// the word W q^-1 mod 2^32 of a constant w (host, at plan creation)
inline uint32_t tiny_word(uint64_t w, uint64_t q) {
  const int64_t W = (int64_t)((q - w % q * ((1ull << 32) % q) % q) % q);
  const int64_t centred = W > (int64_t)(q / 2) ? W - (int64_t)q : W;
  return (uint32_t)((uint64_t)centred * pm::host::inv_pow2_64(q));
}

}  // namespace pm
