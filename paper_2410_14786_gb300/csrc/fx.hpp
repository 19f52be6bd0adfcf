// Block fixed-point form of float64 dot products (shared by the kernels and
// their host checks).
//
// GB300 issues 2 float64 FMAs per SM and clock but 32 multiply-adds of two
// 32-bit integers into a 64-bit sum, so the float64 operators are held, and
// their dot products formed, in fixed point. A value v is q 2^(E - kFxBits)
// with an integer |q| <= 2^kFxBits and an exponent E shared by a block of
// values, and q is split into two signed halves, q = h 2^kFxLow + l, |h| <=
// 2^30, |l| <= 2^28. A product of two such values is h h' 2^(2 kFxLow) + (h l'
// + l h') 2^kFxLow, three integer multiply-adds into two 64-bit sums; the
// dropped l l' is below 2^-62 of full scale. Integer sums are exact, so a result
// depends on no order, and its errors are the rounding of the inputs, the dropped
// terms and the final rounding to float64.
//
// Blocks. An operand's blocks are kFxBlock consecutive values, an operator's
// tiles of kFxBlock x kFxBlock entries, each with its own exponent; a block sum
// is formed of one block of the operand and a row (or column) of one tile. A
// value is exact unless it is below 2^-7 of its block's scale (60 bits hold 53
// there), else its error is 2^-61 of that scale. A tile's scale is such that the
// absolute sum of a row or column is at most kFxBlockSum in its units, an operand
// block's such that no half of it (16 values, of one 64-bit sum) has an absolute
// sum above kFxHalfSum: that keeps a sum of h h' within 2^62, of h l' within 2^61
// and of l h' within 2^62.
//
// Rows. A block sum joins the row's total in the unit of the row's largest
// block (fx_shift_sum), as an integer of 2^kFxShift times the unit of h h' and a
// fraction of kFxFrac bits. A total is kept as three 32-bit sums,
// of the fractions and of the integers' lower kFxLimb and upper bits: with at most
// kFxMaxBlocks blocks none overflows.
//
// Certificate. float64 sums are accurate relative to the sum of |a_ij| |x_j| of
// their own row, however small that is; fixed-point sums are accurate relative
// to the scales u_J of the row's blocks (those of tile and operand block
// multiplied). A row's total is therefore used only where the two are the same:
// where the magnitudes of its half-block sums (16 products; their sum is a lower
// bound of sum |a_ij| |x_j|) add up to 2^-kFxCertBits of the blocks' weighted
// mean scale, sum u_J^2 / sum u_J. Every other row is summed in float64, from
// float64 entries.
#pragma once

#include <cstdint>

#if defined(__CUDACC__)
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace bddc {

constexpr int kFxBits = 60;       // magnitude bits of a value
constexpr int kFxLow = 30;        // bits of the low half
constexpr int kFxBlock = 32;      // products of one block (16 per 64-bit sum, two sums)
constexpr int kFxBlockSum = 4;    // largest absolute sum of a row or column of a tile, in units of its scale
constexpr int kFxHalfSum = 8;     // largest absolute sum of half an operand block, in units of its scale
constexpr int kFxMaxBlocks = 124; // blocks of a row
constexpr int kFxShift = 13;      // low bits of a block's h h' sum that go to the fraction
constexpr int kFxFrac = 24;       // bits of the fraction
constexpr int kFxLimb = 25;       // bits of the low limb of a total
constexpr int kFxZero = -8192;    // exponent of a zero
constexpr int kFxNonFinite = 8192;   // exponent of an infinity or NaN
constexpr int kFxCertBits = 7;    // a row's magnitude is at least 2^-this of its scale
constexpr int kFxCertUnit = 20;   // magnitudes are in units of 2^-this of full scale
constexpr int kFxScaleBits = 12;  // blocks further below a row's largest don't count in its mean scale
constexpr int kFxZeroTile = 127;  // shift of a tile of zeros

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
// `bits` bits and in fewer instructions: round(x 2^(bits - E)), 54 <= bits <= 60.
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

// The sum of a block, kept in two pairs of (h h', mixed) sums, 2^d times smaller
// (d >= 0) and rounded down, as hi + frac 2^-kFxFrac in units of 2^kFxShift times
// that of h h'; 0 <= frac < 2^kFxFrac.
FX_HD void fx_scaled_sum(int64_t h0, int64_t m0, int64_t h1, int64_t m1, int d, int64_t& hi, uint32_t& frac) {
  const int64_t m = (m0 >> kFxLow) + (m1 >> kFxLow);
  const int64_t l = (m0 & ((1ll << kFxLow) - 1)) + (m1 & ((1ll << kFxLow) - 1));
  const int64_t h = h0 + h1 + m + (l >> kFxLow);
  constexpr int drop = kFxLow - kFxFrac + kFxShift;   // low bits of h 2^kFxLow + l beyond the fraction
  const uint64_t low = d <= 64 - kFxFrac - drop
                           ? ((uint64_t)h << kFxLow | ((uint64_t)l & ((1ull << kFxLow) - 1))) >> (drop + d)
                           : (uint64_t)(h >> (d + kFxShift - kFxFrac < 63 ? d + kFxShift - kFxFrac : 63));
  frac = (uint32_t)low & ((1u << kFxFrac) - 1);
  hi = h >> (d + kFxShift < 63 ? d + kFxShift : 63);
}

FX_HD void fx_block_sum(int64_t h0, int64_t m0, int64_t h1, int64_t m1, int64_t& hi, uint32_t& frac) {
  fx_scaled_sum(h0, m0, h1, m1, 0, hi, frac);
}

FX_HD uint32_t fx_limb0(int64_t hi) { return (uint32_t)hi & ((1u << kFxLimb) - 1); }
FX_HD int32_t fx_limb1(int64_t hi) { return (int32_t)(hi >> kFxLimb); }
FX_HD int64_t fx_total(uint32_t limb0, int32_t limb1) { return ((int64_t)limb1 << kFxLimb) + limb0; }

// Exponent of the unit of fx_block_sum for operands of exponents Ea and Ex.
FX_HD int fx_unit(int Ea, int Ex) { return Ea + Ex + 2 * (kFxLow - kFxBits) + kFxShift; }


// Magnitudes of two half-block sums h h' (at most kFxBlockSum together), 2^d
// times smaller, rounded down, in units of 2^-kFxCertUnit of full scale.
FX_HD uint32_t fx_magnitude(int64_t h0, int64_t h1, int d) {
  const int32_t a = (int32_t)(h0 >> 32), b = (int32_t)(h1 >> 32);
  const uint32_t s = (uint32_t)(a ^ (a >> 31)) + (uint32_t)(b ^ (b >> 31));
  constexpr int drop = 2 * (kFxBits - kFxLow) - 32 - kFxCertUnit;
  return s >> (d + drop < 31 ? d + drop : 31);
}

// Exponent of an operand value times 2^e, e the exponent of its row.
FX_HD int fx_scaled_exponent(uint64_t bits, int e) {
  const int x = fx_exponent(bits);
  return x == kFxNonFinite || x == kFxZero ? x : e == kFxZero ? kFxZero : x + e;
}
// Whether half an operand block with this sum of fx_part(h) exceeds kFxHalfSum.
FX_HD uint32_t fx_part(int32_t h) { return (uint32_t)(h < 0 ? -h : h) >> 4; }
FX_HD bool fx_half_exceeds(uint32_t sum) { return sum > (uint32_t)kFxHalfSum << (kFxBits - kFxLow - 4); }
// Scale of the products of an operand block (exponent E) and a tile (shift s).
FX_HD int fx_block_scale(int E, int s) {
  return E == kFxNonFinite ? E : E == kFxZero || s == kFxZeroTile ? kFxZero : E - s;
}

// Certificate of a row: sums s1 of u and s2 of u^2 over its blocks, u in units of
// 2^-kFxScaleBits of the largest one (u = 2^-d of it), against its magnitude in
// that unit. s1 = 0, s2 = 1: no row holds; s1 = s2 = 0: every one does.
FX_HD uint32_t fx_s1(int d) { return d <= kFxScaleBits ? 1u << (kFxScaleBits - d) : 0; }
FX_HD uint32_t fx_s2(int d) { return d <= kFxScaleBits ? 1u << (2 * (kFxScaleBits - d)) : 0; }
FX_HD bool fx_holds(uint32_t magnitude, uint32_t s1, uint32_t s2) {
  return (uint64_t)magnitude * s1 >= (uint64_t)s2 << (kFxCertUnit - kFxScaleBits - kFxCertBits);
}

}  // namespace bddc
