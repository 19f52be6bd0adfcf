// Host check of the packed fixed-point operators (fx_pack.hpp, fx.hpp) row by
// row: products with local operators of even and very uneven conductivities and
// with operands that are dense, localised or spread over many decades. A row is
// used in fixed point only where it is as accurate as float64 relative to
// sum |a_ij| |x_j|; every other one must be marked. Prints "ok" or the first
// failure.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <random>
#include <string>
#include <vector>

#include "dense.hpp"
#include "fx_pack.hpp"

using namespace bddc;

#define REQUIRE(c, ...)                    \
  do {                                     \
    if (!(c)) {                            \
      std::printf("failed: " __VA_ARGS__); \
      std::printf("\n");                   \
      return 1;                            \
    }                                      \
  } while (0)

// Inverse of the Q1 stiffness matrix of a cube of m^3 (dim 2: m^2) interior
// nodes, sigma per element.
static std::vector<double> inverse(int dim, int m, const std::function<double(int, int, int)>& sigma) {
  const int n = dim == 3 ? m * m * m : m * m, ez = dim == 3 ? m + 1 : 1;
  const double k3[4] = {1.0 / 3, 0.0, -1.0 / 12, -1.0 / 12}, k2[4] = {4.0 / 6, -1.0 / 6, -2.0 / 6, 0.0};
  std::vector<double> A((size_t)n * n, 0.0);
  for (int z = 0; z < ez; ++z)
    for (int y = 0; y <= m; ++y)
      for (int x = 0; x <= m; ++x) {
        int node[8];
        for (int a = 0; a < 1 << dim; ++a) {
          const int ix = x + (a & 1) - 1, iy = y + ((a >> 1) & 1) - 1, iz = dim == 3 ? z + (a >> 2) - 1 : 0;
          const bool in = ix >= 0 && ix < m && iy >= 0 && iy < m && iz >= 0 && iz < (dim == 3 ? m : 1);
          node[a] = in ? ix + m * (iy + m * iz) : -1;
        }
        const double sg = sigma(x, y, z);
        for (int a = 0; a < 1 << dim; ++a)
          for (int b = 0; b < 1 << dim; ++b)
            if (node[a] >= 0 && node[b] >= 0)
              A[(size_t)node[a] * n + node[b]] += sg * (dim == 3 ? k3 : k2)[__builtin_popcount(a ^ b)];
      }
  if (dense::spd_inverse(n, A.data(), n) >= 0) A.clear();
  return A;
}

// The fixed-point tiles of one operator {low, high}, as the device forms them.
static std::vector<int32_t> halves(const FxPacked& P, int n) {
  std::vector<int32_t> out(2 * fx_packed_elems(n));
  for (int I = 0; I * kFxTile < n; ++I)
    for (int J = 0; J <= I; ++J)
      for (int r = 0; r < kFxTile; ++r)
        for (int k = 0; k < kFxTile; ++k) {
          const int t = fx_tile_at(I, J), i = I * kFxTile + r, j = J * kFxTile + k;
          uint64_t b;
          std::memcpy(&b, &P.values[(size_t)t * kFxTileElems + r * kFxTile + k], 8);
          int32_t* at = &out[2 * ((size_t)t * kFxTileElems + fx_place(r, k))];
          fx_entry(b, i < n ? P.rexp[i] : 0, j < n ? P.rexp[j] : 0, P.shift[t], at[0], at[1]);
        }
  return out;
}

// One product in fixed point, as the kernel forms it; used[i]: row i holds.
static void product(const FxPacked& P, int n, const std::vector<double>& x, std::vector<double>& y,
                    std::vector<char>& used) {
  const int T = (n + kFxTile - 1) / kFxTile;
  const std::vector<int32_t> tiles = halves(P, n);
  std::vector<int> E(T, kFxZero);
  std::vector<int32_t> xh(T * kFxTile, 0), xl(T * kFxTile, 0);
  auto bits = [](double v) { uint64_t b; std::memcpy(&b, &v, 8); return b; };
  for (int J = 0; J < T; ++J) {
    for (int j = J * kFxTile; j < std::min(n, (J + 1) * kFxTile); ++j) E[J] = std::max(E[J], fx_scaled_exponent(bits(x[j]), P.rexp[j]));
    if (E[J] == kFxZero || E[J] == kFxNonFinite) continue;
    auto round = [&]() {
      uint32_t half[4] = {0, 0, 0, 0};   // lower, upper, even, odd
      for (int j = J * kFxTile; j < std::min(n, (J + 1) * kFxTile); ++j) {
        const int64_t q = P.rexp[j] == kFxZero ? 0 : fx_quantize(bits(x[j]), kFxBits - E[J] + P.rexp[j]);
        xh[j] = fx_hi(q);
        xl[j] = fx_lo(q);
        half[j % kFxTile / 16] += fx_part(xh[j]);
        half[2 + j % 2] += fx_part(xh[j]);
      }
      return fx_half_exceeds(std::max(std::max(half[0], half[1]), std::max(half[2], half[3])));
    };
    if (round()) {
      ++E[J];
      round();
    }
  }
  y.assign(n, 0.0);
  used.assign(n, 0);
  for (int I = 0; I < T; ++I) {
    auto scale = [&](int J) { return fx_block_scale(E[J], P.shift[fx_tile_at(I, J)]); };
    int top = kFxZero;
    uint32_t s1 = 0, s2 = 0;
    for (int J = 0; J < T; ++J) top = std::max(top, scale(J));
    if (top >= kFxNonFinite) {
      s2 = 1;
    } else if (top != kFxZero) {
      for (int J = 0; J < T; ++J) {
        s1 += fx_s1(top - scale(J));
        s2 += fx_s2(top - scale(J));
      }
    }
    for (int r = 0; r < kFxTile && I * kFxTile + r < n; ++r) {
      const int i = I * kFxTile + r;
      uint32_t tf = 0, t0 = 0, size = 0;
      int32_t t1 = 0;
      for (int J = 0; J < T; ++J) {
        const int32_t* tile = &tiles[2 * (int64_t)fx_tile_at(I, J) * kFxTileElems];
        int64_t h[2] = {0, 0}, m[2] = {0, 0};
        for (int k = 0; k < kFxTile; ++k) {
          // row r of tile (I, J), or column r of tile (J, I): halves even / odd, or lower / upper
          const int row = J <= I ? r : k, col = J <= I ? k : r, half = J <= I ? k & 1 : k >> 4;
          const int at = fx_place(row, col);
          const int64_t al = tile[2 * at], ah = tile[2 * at + 1];
          if (__builtin_add_overflow(h[half], ah * xh[J * kFxTile + k], &h[half]) ||
              __builtin_add_overflow(m[half], ah * xl[J * kFxTile + k], &m[half]) ||
              __builtin_add_overflow(m[half], al * xh[J * kFxTile + k], &m[half]))
            std::printf("overflow in a block\n"), std::exit(1);
        }
        int64_t hi;
        uint32_t f;
        const int d = std::max(0, top - E[J] + P.shift[fx_tile_at(I, J)]);
        fx_scaled_sum(h[0], m[0], h[1], m[1], d, hi, f);
        size += fx_magnitude(h[0], h[1], d);
        tf += f;
        t0 += fx_limb0(hi);
        t1 += fx_limb1(hi);
      }
      used[i] = fx_holds(size, s1, s2);
      if (P.rexp[i] != kFxZero && top != kFxZero)
        y[i] = std::ldexp(std::fma((double)tf, 1.0 / (1 << kFxFrac), (double)fx_total(t0, t1)), fx_unit(P.rexp[i], top));
    }
  }
}

int main() {
  std::mt19937_64 g(11);
  std::normal_distribution<double> nd;
  std::uniform_real_distribution<double> ud;
  // a scaled block sum is the exact floor, a magnitude a lower bound
  for (int trial = 0; trial < 20000; ++trial) {
    int64_t v[4];
    for (int q = 0; q < 4; ++q) v[q] = (int64_t)(g() >> (3 + g() % 60)) * (g() & 1 ? 1 : -1);
    const int d = (int)(g() % 100);
    int64_t hi;
    uint32_t f;
    fx_scaled_sum(v[0], v[1], v[2], v[3], d, hi, f);
    const __int128 all = (((__int128)v[0] + v[2]) << kFxLow) + v[1] + v[3], got = ((__int128)hi << kFxFrac) + f;
    REQUIRE(got == all >> (kFxLow - kFxFrac + kFxShift + d) && f < 1u << kFxFrac, "scaled sum, %d", d);
    const long double size = std::ldexp(std::fabs((long double)v[0]) + std::fabs((long double)v[2]),
                                        kFxCertUnit - 2 * (kFxBits - kFxLow) - d);
    REQUIRE(fx_magnitude(v[0], v[2], d) <= size && fx_magnitude(v[0], v[2], d) + 2 > size, "magnitude, %d", d);
  }
  struct Op {
    std::string name;
    int n;
    std::vector<double> A;
  };
  std::vector<Op> ops;
  auto add = [&](const char* name, int dim, int m, const std::function<double(int, int, int)>& s) {
    ops.push_back(Op{name, dim == 3 ? m * m * m : m * m, inverse(dim, m, s)});
  };
  auto one = [](int, int, int) { return 1.0; };
  auto lognormal = [&](int, int, int) { return std::exp(nd(g)); };
  add("one 3", 3, 3, one);
  add("one 6", 3, 6, one);
  add("lognormal 6", 3, 6, lognormal);
  add("lognormal 7", 3, 7, lognormal);
  add("decades 6", 3, 6, [&](int, int, int) { return std::pow(10.0, 8 * ud(g) - 4); });
  add("weak slab 1e6", 3, 7, [](int, int, int z) { return z == 3 ? 1e-6 : 1.0; });
  add("weak slab 1e12", 3, 7, [](int, int, int z) { return z == 3 ? 1e-12 : 1.0; });
  add("one 15 (2D)", 2, 15, one);
  add("lognormal 15 (2D)", 2, 15, lognormal);
  // rows that vanish up to rounding and rows that vanish, a diagonal that does
  // not bound its row, huge and tiny scales
  {
    Op o{"odd rows", 70, std::vector<double>(70 * 70)};
    for (int i = 0; i < 70; ++i)
      for (int j = 0; j <= i; ++j) {
        double v = nd(g) * std::pow(2.0, (i % 7) * 40.0 - 120 + (j % 7) * 40.0 - 120);
        if (i == 5 || j == 5 || i == 69 || j == 69) v = 0.0;
        if (i == 40 || j == 40) v *= 1e-17;
        if (i == j && i == 33) v = 0.0;
        o.A[i * 70 + j] = o.A[j * 70 + i] = v;
      }
    ops.push_back(o);
  }
  const char* kinds[] = {"normal", "positive", "one entry", "a few entries", "entries over 1e-8..1", "first third", "one large, others 1e-9", "flat"};
  for (const Op& o : ops) {
    REQUIRE(!o.A.empty(), "%s: not positive definite", o.name.c_str());
    const int n = o.n;
    FxPacked P;
    fx_pack_lower({o.A}, {n}, {0}, {}, 1, P);
    const std::vector<int32_t> tiles = halves(P, n);
    // the packed entries: float64 exactly, fixed point to 2^-59 of the tile's scale
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) {
        const int I = i / kFxTile, J = j / kFxTile;
        if (J > I) continue;
        const int row = i % kFxTile, col = j % kFxTile, t = fx_tile_at(I, J);
        const double s = 0.5 * (o.A[i * n + j] + o.A[j * n + i]);
        REQUIRE(P.values[(size_t)t * kFxTileElems + row * kFxTile + col] == s, "%s: value", o.name.c_str());
        const int64_t at = (int64_t)t * kFxTileElems + fx_place(row, col);
        const int64_t q = (int64_t)tiles[2 * at + 1] * (1ll << kFxLow) + tiles[2 * at];
        if (s == 0.0) {
          REQUIRE(q == 0, "%s: zero", o.name.c_str());
          continue;
        }
        const long double want = std::ldexp((long double)s, kFxBits - P.rexp[i] - P.rexp[j] + P.shift[t]);
        REQUIRE(std::fabs(q - want) <= 0.5L && std::llabs(q) <= 1ll << kFxBits, "%s: entry %d %d", o.name.c_str(), i, j);
      }
    for (int kind = 0; kind < 8; ++kind) {
      double worst = 0.0, worst64 = 0.0;
      int marked = 0, rows = 0;
      for (int trial = 0; trial < (n < 100 ? 200 : 12); ++trial) {
        std::vector<double> x(n, 0.0), y;
        const int at = (int)(g() % n);
        for (int j = 0; j < n; ++j) {
          if (kind == 0) x[j] = nd(g);
          if (kind == 1) x[j] = 1.0 + 0.25 * std::fmax(-2.0, std::fmin(2.0, nd(g)));
          if (kind == 2) x[j] = j == at ? nd(g) : 0.0;
          if (kind == 3) x[j] = g() % 40 == 0 ? nd(g) : 0.0;
          if (kind == 4) x[j] = nd(g) * std::pow(10.0, -8 * ud(g));
          if (kind == 5) x[j] = j < n / 3 ? nd(g) : 0.0;
          if (kind == 7) x[j] = std::ldexp(g() % 2 ? 1.0 - 0x1p-53 : -1.0, -P.rexp[j] == -kFxZero ? 0 : -P.rexp[j]);
          if (kind == 6) x[j] = j == at ? nd(g) : 1e-9 * nd(g);
        }
        std::vector<char> used;
        product(P, n, x, y, used);
        for (int i = 0; i < n; ++i) {
          long double exact = 0.0L, mag = 0.0L;
          double part[32] = {0};
          for (int j = 0; j < n; ++j) {
            const double a = 0.5 * (o.A[i * n + j] + o.A[j * n + i]);
            exact += (long double)a * x[j];
            mag += std::fabs((long double)a * x[j]);
            part[j % 32] = std::fma(a, x[j], part[j % 32]);
          }
          for (int h = 16; h; h >>= 1)
            for (int q = 0; q < h; ++q) part[q] += part[q + h];
          if (mag == 0.0L) {
            REQUIRE(!used[i] || y[i] == 0.0, "%s, %s: row %d of zeros", o.name.c_str(), kinds[kind], i);
            continue;
          }
          ++rows;
          worst64 = std::max(worst64, (double)(std::fabs(part[0] - exact) / mag));
          if (used[i]) worst = std::max(worst, (double)(std::fabs(y[i] - exact) / mag));
          else ++marked;
        }
      }
      std::printf("%-18s %-24s error of sum |a||x|: fixed point %.2e, float64 %.2e; %5.2f %% of the rows marked\n",
                  o.name.c_str(), kinds[kind], worst, worst64, 100.0 * marked / std::max(rows, 1));
      // no larger than float64's, or than what one product at the limit of the
      // certificate may be off: the rounding of the result, 2^-53, and that of the
      // entry and the dropped product of low halves, (2^-61 + 2^-62) 2^kFxCertBits
      REQUIRE(worst <= std::max(worst64, 0x1p-53 + 0.75 * std::ldexp(1.0, kFxCertBits - 60)), "%s, %s: error %.2e against %.2e", o.name.c_str(), kinds[kind], worst, worst64);
    }
  }
  // several operators in several threads: the same as each alone
  {
    std::vector<std::vector<double>> all;
    std::vector<int> dims;
    std::vector<int32_t> voff;
    std::vector<uint8_t> drop;
    int rows = 3;
    for (int q = 0; q < 40; ++q) {
      const Op& o = ops[q % ops.size()];
      all.push_back(q == 17 ? std::vector<double>() : o.A);
      dims.push_back(q == 17 ? 0 : o.n);
      voff.push_back(rows);
      rows += dims.back();
    }
    drop.assign(rows, 0);
    for (int i = 5; i < rows; i += 50) drop[i] = 1;
    FxPacked many;
    fx_pack_lower(all, dims, voff, drop, 4, many);
    for (size_t q = 0; q < all.size(); ++q) {
      if (dims[q] == 0) continue;
      FxPacked P;
      fx_pack_lower({all[q]}, {dims[q]}, {0}, std::vector<uint8_t>(&drop[voff[q]], &drop[voff[q]] + dims[q]), 1, P);
      const int64_t n = fx_packed_elems(dims[q]);
      REQUIRE(many.off[q] % kFxTileElems == 0 &&
                  std::memcmp(many.values.get() + many.off[q], P.values.get(), 8 * n) == 0 &&
                  std::memcmp(&many.rexp[voff[q]], P.rexp.data(), 4 * dims[q]) == 0 &&
                  std::memcmp(&many.shift[many.off[q] / kFxTileElems], P.shift.data(), n / kFxTileElems) == 0,
              "operator %zu packed with others", q);
      for (int i = 0; i < dims[q]; ++i)
        REQUIRE(!drop[voff[q] + i] || P.rexp[i] == kFxZero, "dropped row %d", i);
    }
  }
  // infinities and NaN: every row marked
  {
    FxPacked P;
    const int n = ops[1].n;
    fx_pack_lower({ops[1].A}, {n}, {0}, {}, 1, P);
    for (double bad : {(double)INFINITY, (double)-INFINITY, std::nan("")}) {
      std::vector<double> x(n, 1.0), y;
      std::vector<char> used;
      x[77] = bad;
      product(P, n, x, y, used);
      for (int i = 0; i < n; ++i) REQUIRE(!used[i], "row %d holds with a non-finite operand", i);
    }
    // zeros: exact
    std::vector<double> x(n, 0.0), y;
    std::vector<char> used;
    product(P, n, x, y, used);
    for (int i = 0; i < n; ++i) REQUIRE(used[i] && y[i] == 0.0, "row %d of a zero operand", i);
  }
  std::printf("ok\n");
  return 0;
}
