// Packing of the float64 local operators for the fixed-point kernel (bddc_fx.cu),
// free of CUDA so that it can be checked on the host: the host forms the float64
// tiles, their shifts and the row exponents, the device the fixed-point tiles from
// them (fx_entry), which spares half of the packing and of the upload.
//
// An operator (symmetric: the packing takes (A + A^T) / 2) is stored as the
// lower triangle of its tiles of 32 x 32: tile (I, J), J <= I, at position
// I (I + 1) / 2 + J, the diagonal ones whole, rows and columns beyond n zero.
// Two forms of the same tiles: fixed point (fx.hpp), {low, high} halves, entry
// (i, j) of a tile with shift s in units of 2^(e_i + e_j - s), e_i the exponent of
// row i (about that of sqrt(a_ii): the operators are positive semidefinite in
// exact arithmetic, so |a_ij| <= sqrt(a_ii a_jj)); and float64, for the rows that
// are not accurate enough in fixed point.
//
// Within a fixed-point tile, vector v (two entries) of row r stands at v ^
// (r & 7), which makes reading a row across lanes and one vector of 8 rows
// across lanes both free of bank conflicts.
#pragma once

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <memory>
#include <system_error>
#include <thread>
#include <vector>

#include "fx.hpp"

namespace bddc {

constexpr int kFxTile = kFxBlock;
constexpr int kFxTileElems = kFxTile * kFxTile;

FX_HD int fx_tiles(int n) {
  const int t = (n + kFxTile - 1) / kFxTile;
  return t * (t + 1) / 2;
}
FX_HD int fx_tile_at(int I, int J) { return I >= J ? I * (I + 1) / 2 + J : J * (J + 1) / 2 + I; }
// Entries of one n x n operator.
inline int64_t fx_packed_elems(int n) { return (int64_t)fx_tiles(n) * kFxTileElems; }

struct FxPacked {
  std::vector<int64_t> off;          // first entry of every operator (a multiple of kFxTileElems)
  int64_t elems = 0;
  std::unique_ptr<double[]> values;  // the float64 tiles
  std::vector<int32_t> rexp;         // exponent of every row, at voff[s] + row (kFxZero: a row of zeros)
  std::vector<int8_t> shift;         // of every tile, padded to a multiple of 4
};

inline int fx_exponent_of(double v) {
  uint64_t b;
  std::memcpy(&b, &v, 8);
  return fx_exponent(b);
}

// S = (A + A^T) / 2 by tiles (the transposed reads stay in cache), row-major;
// rows and columns with drop[i] set are zero.
inline void fx_symmetric_part(const double* A, int n, const uint8_t* drop, double* S) {
  for (int i0 = 0; i0 < n; i0 += kFxTile)
    for (int j0 = 0; j0 <= i0; j0 += kFxTile)
      for (int i = i0; i < std::min(n, i0 + kFxTile); ++i)
        for (int j = j0; j < std::min(n, j0 + kFxTile); ++j) {
          const double v = drop && (drop[i] || drop[j]) ? 0.0 : 0.5 * (A[(size_t)i * n + j] + A[(size_t)j * n + i]);
          S[(size_t)i * n + j] = v;
          S[(size_t)j * n + i] = v;
        }
}

// Row exponents of the symmetric S: |s_ij| < 2^(e_i + e_j). From the diagonal,
// raised where rounding (or a row that vanishes in exact arithmetic) breaks the
// bound of the semidefinite case. size: n doubles of scratch.
inline void fx_row_exponents(const double* S, int n, int32_t* e, double* size) {
  for (int i = 0; i < n; ++i) {
    const double d = S[(size_t)i * n + i];
    e[i] = d != 0.0 ? (fx_exponent_of(d) + 2049) / 2 - 1024 : -400;
    size[i] = std::ldexp(1.0, e[i]);
  }
  for (int i = 0; i < n; ++i) {
    const double* row = S + (size_t)i * n;
    for (int j = 0; j < i; ++j) {
      if (std::fabs(row[j]) < size[i] * size[j]) continue;   // the common case
      const int need = fx_exponent_of(row[j]) - e[i] - e[j];
      if (row[j] == 0.0 || need <= 0) continue;
      const int up = e[i] < e[j] ? i : j;
      e[up] += need;
      size[up] = std::ldexp(1.0, e[up]);
    }
  }
  for (int i = 0; i < n; ++i) {
    bool zero = true;
    for (int j = 0; j < n && zero; ++j) zero = S[(size_t)i * n + j] == 0.0;
    if (zero) e[i] = kFxZero;
  }
}

// Largest shift s (of at most 100) with every |s_ij| 2^(s - e_i - e_j) of the
// tile at (i0, j0) below 1 and every absolute sum of a row or column at most
// kFxBlockSum; kFxZeroTile for a tile of zeros.
inline int fx_tile_shift(const double* S, int n, int i0, int j0, const int32_t* e) {
  const int ni = std::min(kFxTile, n - i0), nj = std::min(kFxTile, n - j0);
  double w[kFxTile], col[kFxTile] = {0};
  for (int j = 0; j < nj; ++j) w[j] = e[j0 + j] == kFxZero ? 0.0 : std::ldexp(1.0, -e[j0 + j]);
  double most = 0.0, sum = 0.0;
  for (int i = 0; i < ni; ++i) {
    const double wi = e[i0 + i] == kFxZero ? 0.0 : std::ldexp(1.0, -e[i0 + i]);
    const double* row = S + (size_t)(i0 + i) * n + j0;
    double r = 0.0;
    for (int j = 0; j < nj; ++j) {
      const double a = std::fabs(row[j]) * w[j] * wi;
      most = std::max(most, a);
      r += a;
      col[j] += a;
    }
    sum = std::max(sum, r);
  }
  for (int j = 0; j < nj; ++j) sum = std::max(sum, col[j]);
  if (most == 0.0) return kFxZeroTile;
  int s = std::min(100, -fx_exponent_of(most));
  while (std::ldexp(sum, s) > kFxBlockSum) --s;
  return s;
}

// Fixed-point entry {low, high} of the value v in row i and column j (exponents
// ei and ej) of a tile with shift s, and its place in the tile (in entries).
FX_HD void fx_entry(uint64_t bits, int ei, int ej, int s, int32_t& lo, int32_t& hi) {
  const int64_t q = bits << 1 ? fx_quantize(bits, kFxBits - ei - ej + s) : 0;
  lo = fx_lo(q);
  hi = fx_hi(q);
}
FX_HD int fx_place(int r, int k) { return r * kFxTile + ((k / 2) ^ (r & 7)) * 2 + k % 2; }

// The float64 tiles of one operator and their shifts.
inline void fx_pack_operator(const double* S, int n, const int32_t* e, double* values, int8_t* shift) {
  for (int I = 0; I * kFxTile < n; ++I)
    for (int J = 0; J <= I; ++J) {
      const int i0 = I * kFxTile, j0 = J * kFxTile, nj = std::min(kFxTile, n - j0);
      *shift++ = (int8_t)fx_tile_shift(S, n, i0, j0, e);
      for (int r = 0; r < kFxTile; ++r, values += kFxTile) {
        const int m = i0 + r < n ? nj : 0;
        if (m) std::memcpy(values, S + (size_t)(i0 + r) * n + j0, sizeof(double) * m);
        std::fill(values + m, values + kFxTile, 0.0);
      }
    }
}

// All operators: ops[s] is dims[s] x dims[s], its rows stand at voff[s] of the
// compact numbering; drop: empty, or a flag per row of that numbering.
inline void fx_pack_lower(const std::vector<std::vector<double>>& ops, const std::vector<int>& dims,
                          const std::vector<int32_t>& voff, const std::vector<uint8_t>& drop, int threads, FxPacked& P) {
  P.off.assign(ops.size(), 0);
  int64_t cur = 0, rows = 0;
  int most = 0;
  for (size_t s = 0; s < ops.size(); ++s) {
    P.off[s] = cur;
    cur += fx_packed_elems(dims[s]);
    rows = std::max<int64_t>(rows, (int64_t)voff[s] + dims[s]);
    most = std::max(most, dims[s]);
  }
  P.elems = std::max<int64_t>(cur, kFxTileElems);
  P.values.reset(new double[P.elems]);   // (every entry is written below, by the threads)
  P.rexp.assign((size_t)std::max<int64_t>(rows, 1), 0);
  P.shift.assign((size_t)(P.elems / kFxTileElems + 3) / 4 * 4, 0);
  // a thread per 65536 entries, not more than asked for; no allocation in the threads
  const int nt = (int)std::max<int64_t>(1, std::min<int64_t>(threads, cur >> 16));
  std::vector<double> scratch((size_t)nt * (most + 1) * most);
  std::atomic<size_t> next{0};
  auto work = [&](int t) {
    double *S = scratch.data() + (size_t)t * (most + 1) * most, *size = S + (size_t)most * most;
    for (size_t s; (s = next.fetch_add(1)) < ops.size();) {
      const int n = dims[s];
      if (n == 0) continue;
      int32_t* e = &P.rexp[voff[s]];
      fx_symmetric_part(ops[s].data(), n, drop.empty() ? nullptr : &drop[voff[s]], S);
      fx_row_exponents(S, n, e, size);
      fx_pack_operator(S, n, e, P.values.get() + P.off[s], &P.shift[P.off[s] / kFxTileElems]);
    }
  };
  std::vector<std::thread> pool;
  pool.reserve(nt);
  for (int t = 1; t < nt; ++t) {
    try {
      pool.emplace_back(work, t);
    } catch (const std::system_error&) {
      break;   // the threads there are share the operators
    }
  }
  work(0);
  for (auto& t : pool) t.join();
}

}  // namespace bddc
