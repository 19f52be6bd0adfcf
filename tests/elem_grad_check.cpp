// Host check of the element term of the 3D adjoint gradient (elem_grad.hpp): on
// elements of many kinds of fields, the largest error relative to sum |K_ab| |u_a|
// |lambda_b| of those that take the fixed-point form must not exceed that of the
// float64 products, and elements where values of very different size meet must
// not take it. Prints "ok" or the first failure.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <random>

#include "elem_grad.hpp"

using namespace bddc;

int main() {
  std::mt19937_64 g(5);
  std::normal_distribution<double> nd;
  std::uniform_real_distribution<double> ud;
  const char* kinds[] = {"even", "normal", "edge peaks", "spread", "spread u", "one node", "boundary", "cancelling", "huge and tiny"};
  for (int kind = 0; kind < 9; ++kind) {
    double worst = 0.0, worst64 = 0.0;
    int taken = 0;
    const int trials = 20000;
    for (int t = 0; t < trials; ++t) {
      const double h = 1.0 / (1 + g() % 200), c2 = -h / 12, su = std::pow(10.0, 4 * nd(g)), sl = std::pow(10.0, 4 * nd(g));
      const int peak = (int)(g() % 8), axis = 1 << (g() % 3);
      double u[8], l[8];
      const double coef[4] = {-4.0 * c2, 0.0, c2, c2};
      for (int a = 0; a < 8; ++a) {
        if (kind == 0) u[a] = su * (1 + 0.1 * nd(g)), l[a] = sl * (1 + 0.1 * nd(g));
        if (kind == 1) u[a] = nd(g), l[a] = nd(g);
        if (kind == 2) u[a] = a == peak ? nd(g) : 1e-8 * nd(g), l[a] = a == (peak ^ axis) ? nd(g) : 1e-8 * nd(g);
        if (kind == 3) u[a] = nd(g) * std::pow(10.0, -6 * ud(g)), l[a] = nd(g) * std::pow(10.0, -6 * ud(g));
        if (kind == 4) u[a] = nd(g) * std::pow(10.0, -6 * ud(g)), l[a] = nd(g);
        if (kind == 5) u[a] = a == peak ? nd(g) : 0.0, l[a] = nd(g);
        if (kind == 6) u[a] = a & axis ? su * (1 + 0.1 * nd(g)) : 0.0, l[a] = a & axis ? sl * (1 + 0.1 * nd(g)) : 0.0;
        if (kind == 7) u[a] = 1 + 1e-9 * nd(g), l[a] = 1 + 1e-9 * nd(g);
        if (kind == 8) u[a] = std::ldexp(nd(g), t % 2 ? 300 : -300), l[a] = std::ldexp(nd(g), t % 3 ? 200 : -200);
      }
      long double exact = 0.0L, size = 0.0L;
      for (int a = 0; a < 8; ++a)
        for (int b = 0; b < 8; ++b) {
          const int bits = __builtin_popcount(a ^ b);
          const long double p = (bits == 0 ? -4.0L : bits == 1 ? 0.0L : 1.0L) * c2 * u[b] * l[a];
          exact += p;
          size += std::fabs(p);
        }
      if (size == 0.0L) continue;
      const int Eu = eg_exponent(u), El = eg_exponent(l);
      double v;
      const bool holds = eg_fixed(u, l, Eu, El, v);
      worst64 = std::fmax(worst64, (double)(std::fabs(eg_products(u, l, coef, 0.0) - exact) / size));
      if (holds) {
        ++taken;
        worst = std::fmax(worst, (double)(std::fabs(-c2 * std::ldexp(v, Eu + El + 2 * (kEgLow - kEgBits)) - exact) / size));
      }
    }
    std::printf("%-14s fixed point %.2e, float64 %.2e; %5.1f %% in fixed point\n", kinds[kind], worst, worst64,
                100.0 * taken / trials);
    if (worst > worst64 || (kind == 2 && taken > 0) || ((kind == 0 || kind == 1 || kind == 6) && taken < 0.97 * trials)) {
      std::printf("failed: %s\n", kinds[kind]);
      return 1;
    }
  }
  std::printf("ok\n");
  return 0;
}
