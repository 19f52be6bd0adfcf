// Element term of the adjoint gradient in 3D, lambda^T K_ref u over the 8 corners
// of one element (shared by the kernel and its host check).
//
// K_ref of the Q1 element depends only on the number of coordinate bits in which
// two local nodes differ, and its rows sum to 0, so with weights w = -K_ref[a][b]
//   lambda^T K_ref u = sum over node pairs of w (lambda_a - lambda_b) (u_a - u_b).
// w = h / 12 for the pairs two or three bits apart (face and cube diagonals) and 0
// along the edges, so the pairs lie within the two tetrahedra of even and of odd
// corners, plus the four cube diagonals (a, 7 - a) between them:
//   sum / w = sum_a lambda_a (5 u_a - u_(7 - a)) - S_even T_even - S_odd T_odd
// with T, S the sums of u and lambda over a tetrahedron.
//
// That form runs in block fixed point: the values of one element are rounded to
// kEgBits bits of their largest, which is exact for those within 2^-3 of it, and
// the sums of the products are exact but for ten dropped products of low halves,
// below 2^-58 of full scale each. Cancellation between the terms costs nothing,
// but a value far below the largest loses bits, which matters where the largest u
// and the largest lambda meet no weight (K_ref = 0 along the edges). So the result
// is used only where |S_even| |T_even| + |S_odd| |T_odd| (sums of magnitudes, whose
// products all have a weight) is at least 2^-kEgCertBits of full scale: there its error
// relative to sum |K_ab| |u_a| |lambda_b| is no larger than that of the float64
// products.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#include "fx.hpp"

namespace bddc {

constexpr int kEgBits = 56, kEgLow = 28;
constexpr int kEgCertBits = 3;

FX_HD uint64_t eg_bits(double v) {
#if defined(__CUDA_ARCH__)
  return (uint64_t)__double_as_longlong(v);
#else
  uint64_t b;
  std::memcpy(&b, &v, 8);
  return b;
#endif
}

// Largest exponent (of 0 and subnormal numbers: -1021) of N values; above 1024: not all finite.
template <int N>
FX_HD int eg_exponent(const double (&v)[N]) {
  int e = 1;
  for (int a = 0; a < N; ++a) {
    const int x = (int)(eg_bits(v[a]) >> 52) & 0x7ff;
    e = x > e ? x : e;
  }
  return e - 1022;
}

// a b in units of 2^(2 kEgLow), as (h, m): h + m 2^-kEgLow (low halves' product dropped).
FX_HD void eg_mac(int64_t& h, int64_t& m, int64_t a, int64_t b) {
  const int ah = (int)((a + (1ll << (kEgLow - 1))) >> kEgLow), bh = (int)((b + (1ll << (kEgLow - 1))) >> kEgLow);
  const int al = (int)(a - ((int64_t)ah << kEgLow)), bl = (int)(b - ((int64_t)bh << kEgLow));
  h += (int64_t)ah * bh;
  m += (int64_t)ah * bl;
  m += (int64_t)al * bh;
}

// sum / w times 2^-(Eu + El + 2 (kEgLow - kEgBits)), Eu and El the exponents of u
// and lambda; false where it is not accurate enough.
FX_HD bool eg_fixed(const double (&uv)[8], const double (&lv)[8], int Eu, int El, double& sum) {
  int64_t u[8], l[8];
  uint32_t T[2] = {0, 0}, S[2] = {0, 0};   // sums of magnitudes, without their low 32 bits
#if defined(__CUDACC__)
#pragma unroll
#endif
  for (int a = 0; a < 8; ++a) {
    const uint64_t ub = eg_bits(uv[a]), lb = eg_bits(lv[a]);
    u[a] = fx_quantize_words((int32_t)ub, (int32_t)(ub >> 32), Eu, kEgBits);
    l[a] = fx_quantize_words((int32_t)lb, (int32_t)(lb >> 32), El, kEgBits);
    const int odd = (a ^ (a >> 1) ^ (a >> 2)) & 1;   // corners 1, 2, 4 and 7
    const int32_t uh = (int32_t)(u[a] >> 32), lh = (int32_t)(l[a] >> 32);
    T[odd] += (uint32_t)(uh ^ (uh >> 31));
    S[odd] += (uint32_t)(lh ^ (lh >> 31));
  }
  int64_t h = 0, m = 0;
#if defined(__CUDACC__)
#pragma unroll
#endif
  for (int a = 0; a < 8; ++a) eg_mac(h, m, 5 * u[a] - u[7 - a], l[a]);
  eg_mac(h, m, -(u[0] + u[3] + u[5] + u[6]), l[0] + l[3] + l[5] + l[6]);
  eg_mac(h, m, -(u[7] + u[4] + u[2] + u[1]), l[7] + l[4] + l[2] + l[1]);
  h += m >> kEgLow;
  m &= (1ll << kEgLow) - 1;
  sum = fma((double)m, 1.0 / (double)(1 << kEgLow), (double)h);
  return (uint64_t)T[0] * S[0] + (uint64_t)T[1] * S[1] >= 1ull << (2 * (kEgBits - 32) - kEgCertBits);
}

// s + lambda^T K_ref u by the float64 products, coef[d] the entry of K_ref between
// nodes d bits apart.
template <int N>
FX_HD double eg_products(const double (&u)[N], const double (&l)[N], const double (&coef)[4], double s) {
#if defined(__CUDACC__)
#pragma unroll
#endif
  for (int a = 0; a < N; ++a) {
    double t = 0.0;
#if defined(__CUDACC__)
#pragma unroll
#endif
    for (int b = 0; b < N; ++b) {
      const int d = a ^ b, bits = (d & 1) + ((d >> 1) & 1) + (d >> 2);
      t = fma(coef[bits], u[b], t);
    }
    s = fma(l[a], t, s);
  }
  return s;
}

}  // namespace bddc
