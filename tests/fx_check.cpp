// Host check of the block fixed-point form (fx.hpp): conversion, split and
// block sums against 128-bit integers, and the error of whole dot products
// against the same products in float64, both measured against long double
// products. Prints "ok" or the first failure.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "fx.hpp"

using namespace bddc;

static uint64_t bits(double v) {
  uint64_t b;
  std::memcpy(&b, &v, 8);
  return b;
}
#define REQUIRE(c, ...)                  \
  do {                                   \
    if (!(c)) {                          \
      std::printf("failed: " __VA_ARGS__); \
      std::printf("\n");                 \
      return 1;                          \
    }                                    \
  } while (0)

int main() {
  std::mt19937_64 g(7);
  std::normal_distribution<double> nd;
  // exponents and rounding, over the whole range of float64
  const double special[] = {0.0, -0.0, 1.0, -1.0, 0.5, 2.0, 4.9e-324, -4.9e-324, 2.2250738585072014e-308,
                            1.7976931348623157e308, std::nextafter(1.0, 0.0), std::nextafter(2.0, 3.0)};
  for (int i = 0; i < 20000; ++i) {
    const double x = i < 12 ? special[i] : std::ldexp(nd(g), (int)(g() % 2040) - 1020);
    if (x == 0.0) {
      REQUIRE(fx_exponent(bits(x)) == kFxZero, "exponent of 0");
      continue;
    }
    if (!std::isfinite(x)) continue;
    const int E = fx_exponent(bits(x));
    const long double t = std::fabs((long double)x);
    REQUIRE(t < std::ldexp(1.0L, E) && (t >= std::ldexp(1.0L, E - 1) || E == -1022), "exponent of %g", x);
    for (int drop : {0, 3, 30, 57, 70}) {
      const int64_t q = fx_quantize(bits(x), kFxBits - E - drop);
      const long double want = std::ldexp((long double)x, kFxBits - E - drop);
      REQUIRE(std::fabs((long double)q - want) <= 0.5L, "rounding of %g with %d bits dropped", x, drop);
      REQUIRE(q <= (1ll << kFxBits) && q >= -(1ll << kFxBits), "range of %g", x);
      REQUIRE((int64_t)fx_hi(q) * (1ll << kFxLow) + fx_lo(q) == q, "split of %g", x);
      REQUIRE(std::abs((long)fx_hi(q)) <= 1l << (kFxBits - kFxLow) && std::abs((long)fx_lo(q)) <= 1l << (kFxLow - 1),
              "halves of %g", x);
    }
  }
  // the form from words agrees with the long one
  for (int i = 0; i < 20000; ++i) {
    const double x = i < 12 ? special[i] : std::ldexp(nd(g), (int)(g() % 2040) - 1020);
    if (!std::isfinite(x)) continue;
    const uint64_t b = bits(x);
    const int E0 = x == 0.0 ? -1021 : std::max(fx_exponent(b), -1021);
    for (int E : {E0, E0 + 1, E0 + 7, E0 + 58, E0 + 64, E0 + 2000})
      for (int nb : {54, 55, kFxBits})
        REQUIRE(fx_quantize_words((int32_t)b, (int32_t)(b >> 32), E, nb) == fx_quantize(b, nb - E), "words of %g", x);
  }
  REQUIRE(fx_exponent(bits(INFINITY)) == kFxNonFinite && fx_exponent(bits(-INFINITY)) == kFxNonFinite &&
              fx_exponent(bits(NAN)) == kFxNonFinite, "exponent of a non-finite value");
  // block sums: the extreme halves, and random ones
  for (int trial = 0; trial < 2000; ++trial) {
    int64_t h[2] = {0, 0}, m[2] = {0, 0};
    __int128 all = 0;
    for (int j = 0; j < kFxBlock; ++j) {
      int64_t ah, al, xh, xl;
      if (trial < 4) {
        ah = (trial & 1 ? -1 : 1) * (1ll << 28);   // rows of sum kFxBlockSum: 32 entries of 1/2
        al = (trial & 2 ? -1 : 1) * (1ll << 28);
        xh = 1ll << 29;
        xl = 1ll << 28;
      } else {
        ah = (int64_t)(g() % (1ull << 29)) - (1ll << 28);
        al = (int64_t)(g() % (1ull << 29)) - (1ll << 28);
        xh = (int64_t)(g() % (1ull << 30)) - (1ll << 29);
        xl = (int64_t)(g() % (1ull << 29)) - (1ll << 28);
      }
      const int s = j & 1;
      REQUIRE(!__builtin_add_overflow(h[s], ah * xh, &h[s]) && !__builtin_add_overflow(m[s], ah * xl, &m[s]) &&
                  !__builtin_add_overflow(m[s], al * xh, &m[s]), "overflow in a block");
      all += (((__int128)(ah * xh)) << kFxLow) + ah * xl + al * xh;   // in units of 2^kFxLow
    }
    int64_t hi;
    uint32_t f;
    fx_block_sum(h[0], m[0], h[1], m[1], hi, f);
    REQUIRE(f < 1u << kFxFrac, "fraction");
    const __int128 got = ((__int128)hi << (kFxLow + kFxShift)) + ((__int128)f << (kFxLow + kFxShift - kFxFrac));
    REQUIRE(all - got >= 0 && all - got < (__int128)1 << (kFxLow + kFxShift - kFxFrac), "block sum, trial %d", trial);
  }
  // whole dot products of decaying rows against float64 ones: the largest
  // error over many must not be larger (from two terms on; one product is
  // rounded once in float64, so its bound is that rounding)
  for (int n : {1, 2, 31, 32, 33, 64, 343, 386, 1500}) {
    double worst_fx = 0.0, worst_64 = 0.0;
    for (int trial = 0; trial < 200; ++trial) {
      std::vector<double> a(n), x(n);
      double s = 0.0;
      int Ex = kFxZero, Ea = kFxZero;
      for (int j = 0; j < n; ++j) {
        a[j] = std::exp(-0.02 * j) * nd(g);   // a decaying row; its scale as for a row of a local operator
        Ea = std::max(Ea, fx_exponent(bits(a[j])) + 1);
        x[j] = nd(g);
        Ex = std::max(Ex, fx_exponent(bits(x[j])));
      }
      long double exact = 0.0L, mag = 0.0L;
      uint32_t t0 = 0, tf = 0;
      int32_t t1 = 0;
      double part[8] = {0};
      for (int j0 = 0; j0 < n; j0 += kFxBlock) {
        int64_t h[2] = {0, 0}, m[2] = {0, 0};
        for (int j = j0; j < std::min(n, j0 + kFxBlock); ++j) {
          const int64_t qa = a[j] == 0.0 ? 0 : fx_quantize(bits(a[j]), kFxBits - Ea), qx = fx_quantize(bits(x[j]), kFxBits - Ex);
          h[j & 1] += (int64_t)fx_hi(qa) * fx_hi(qx);
          m[j & 1] += (int64_t)fx_hi(qa) * fx_lo(qx) + (int64_t)fx_lo(qa) * fx_hi(qx);
          exact += (long double)a[j] * x[j];
          mag += std::fabs((long double)a[j] * x[j]);
          part[(j / 2) % 8] = std::fma(a[j], x[j], part[(j / 2) % 8]);   // as the float64 kernel sums
        }
        int64_t hi;
        uint32_t f;
        fx_block_sum(h[0], m[0], h[1], m[1], hi, f);
        t0 += fx_limb0(hi);
        t1 += fx_limb1(hi);
        tf += f;
        REQUIRE(fx_total(fx_limb0(hi), fx_limb1(hi)) == hi, "limbs");
      }
      const double y = std::ldexp(std::fma((double)tf, 1.0 / (1 << kFxFrac), (double)fx_total(t0, t1)), fx_unit(Ea, Ex));
      s = ((part[0] + part[4]) + (part[2] + part[6])) + ((part[1] + part[5]) + (part[3] + part[7]));
      worst_fx = std::max(worst_fx, (double)(std::fabs(y - exact) / mag));
      worst_64 = std::max(worst_64, (double)(std::fabs(s - exact) / mag));
    }
    std::printf("n %d: largest error fixed point %.2e, float64 %.2e (of the absolute sum)\n", n, worst_fx, worst_64);
    REQUIRE(worst_fx <= 1.1e-16 || worst_fx <= worst_64, "error at n = %d", n);
  }
  std::printf("ok\n");
  return 0;
}
