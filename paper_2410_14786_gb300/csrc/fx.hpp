// Block fixed-point form of float64 dot products (shared by the kernels and
// their host checks).
//
// GB300 issues 2 float64 FMAs per SM and clock but 32 multiply-adds of two
// 32-bit integers into a 64-bit sum, so the float64 operators are held, and
// their dot products formed, in fixed point. A value v is q 2^(E - kFxBits)
// with an integer |q| <= 2^kFxBits and an exponent E shared by a whole operator
// row or operand vector, and q is split into two signed halves, q = h 2^kFxLow
// + l, |h| <= 2^29, |l| <= 2^28. A product of two such values is h h'
// 2^(2 kFxLow) + (h l' + l h') 2^kFxLow, three integer multiply-adds into two
// 64-bit sums; the dropped l l' is below 2^-60 of full scale. Integer sums are
// exact, so a result depends on no order, and its errors are the rounding of
// the inputs (2^-59 of the row's and the vector's scale; a float64 sum rounds
// to 2^-53 of its partial sums at every step), the dropped terms and the final
// rounding to float64.
//
// Sums run over blocks of kFxBlock products: an operator's scale is such that
// the absolute sum of a row over one block is at most kFxBlockSum in its
// units, which keeps the sum of h h' within 2^62, and the mixed sum grows by
// at most 2^58 per product. A block's sum then joins the row's total as
// an integer of 2^kFxShift times its unit and a fraction of kFxFrac bits
// (fx_block_sum). A total is kept as three 32-bit sums, of the fractions and of
// the integers' lower kFxLimb and upper bits: with an absolute row sum of at
// most kFxRowSum and at most kFxMaxBlocks blocks none overflows.
#pragma once

#include <cstdint>

#if defined(__CUDACC__)
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace bddc {

constexpr int kFxBits = 58;       // magnitude bits of a value
constexpr int kFxLow = 29;        // bits of the low half
constexpr int kFxBlock = 32;      // products of one block (16 per 64-bit sum, two sums)
constexpr int kFxBlockSum = 16;   // largest absolute sum of a row over a block, in units of its scale
constexpr int kFxRowSum = 512;    // the same over the whole row
constexpr int kFxMaxBlocks = 124; // blocks of a row
constexpr int kFxShift = 12;      // low bits of a block's h h' sum that go to the fraction
constexpr int kFxFrac = 24;       // bits of the fraction
constexpr int kFxLimb = 25;       // bits of the low limb of a total
constexpr int kFxZero = -8192;    // exponent of a zero
constexpr int kFxNonFinite = 8192;   // exponent of an infinity or NaN

// Smallest E with |x| < 2^E, from the bits of the float64 x.
FX_HD int fx_exponent(uint64_t bits) {
  const int e = (int)(bits >> 52) & 0x7ff;
  if (e == 0x7ff) return kFxNonFinite;
  if (e > 0) return e - 1022;
  return (bits & 0xfffffffffffffull) ? -1022 : kFxZero;
}

// round(x 2^add) for a finite x with |x| 2^add <= 2^kFxBits (halves away
// from zero).
FX_HD int64_t fx_quantize(uint64_t bits, int add) {
  const int e = (int)(bits >> 52) & 0x7ff;
  const uint64_t m = (bits & 0xfffffffffffffull) | (e ? 0x10000000000000ull : 0ull);
  const int s = (e ? e : 1) - 1075 + add;
  uint64_t q;
  if (s >= 0)
    q = s < 12 ? m << s : 0;   // (s <= kFxBits - 53 for the values allowed)
  else
    q = s >= -54 ? (m + (1ull << (-s - 1))) >> -s : 0;
  return (int64_t)(bits >> 63 ? 0 - q : q);
}

// The same for the words {lo, hi} of a finite x with |x| < 2^E, rounded to
// `bits` bits and in fewer instructions: round(x 2^(bits - E)), 54 <= bits <= 58.
// E is at least -1021, so that 0 and subnormal numbers fit too.
FX_HD int64_t fx_quantize_words(int32_t lo, int32_t hi, int E, int bits = kFxBits) {
  const int e = (hi >> 20) & 0x7ff;
  const uint64_t m = ((uint64_t)(uint32_t)((hi & 0xfffff) | (e ? 0x100000 : 0)) << 32 | (uint32_t)lo) << (bits - 52);
  const int d = E - (e ? e : 1) + 1022;   // m < 2^(bits + 1): x 2^(bits - E) = m / 2^(d + 1)
  const int64_t q = d < 62 ? (int64_t)(((m >> d) + 1) >> 1) : 0;
  const int64_t s = hi >> 31;
  return (q ^ s) - s;
}

FX_HD int32_t fx_hi(int64_t q) { return (int32_t)((q + (1ll << (kFxLow - 1))) >> kFxLow); }
FX_HD int32_t fx_lo(int64_t q) { return (int32_t)(q - ((int64_t)fx_hi(q) << kFxLow)); }

// The sum of a block, kept in two pairs of (h h', mixed) sums, as hi + frac
// 2^-kFxFrac in units of 2^kFxShift times that of h h'; 0 <= frac < 2^kFxFrac.
FX_HD void fx_block_sum(int64_t h0, int64_t m0, int64_t h1, int64_t m1, int64_t& hi, uint32_t& frac) {
  const int64_t m = (m0 >> kFxLow) + (m1 >> kFxLow);
  const int64_t l = (m0 & ((1ll << kFxLow) - 1)) + (m1 & ((1ll << kFxLow) - 1));
  const int64_t h = h0 + h1 + m + (l >> kFxLow);
  hi = h >> kFxShift;
  frac = (uint32_t)(h & ((1 << kFxShift) - 1)) << (kFxFrac - kFxShift) |
         ((uint32_t)l & ((1u << kFxLow) - 1)) >> (kFxLow - kFxFrac + kFxShift);
}

FX_HD uint32_t fx_limb0(int64_t hi) { return (uint32_t)hi & ((1u << kFxLimb) - 1); }
FX_HD int32_t fx_limb1(int64_t hi) { return (int32_t)(hi >> kFxLimb); }
FX_HD int64_t fx_total(uint32_t limb0, int32_t limb1) { return ((int64_t)limb1 << kFxLimb) + limb0; }

// Exponent of the unit of fx_block_sum for operands of exponents Ea and Ex.
FX_HD int fx_unit(int Ea, int Ex) { return Ea + Ex + 2 * (kFxLow - kFxBits) + kFxShift; }

}  // namespace bddc
