// Host check of csrc/fixed.cuh: digits and scaled integers against long
// double, over exponents, signs and subnormals.  Exit code 0 if all hold.
#include <cmath>
#include <cstdio>
#include <random>

#include "fixed.cuh"

using namespace mg::fx;

int main() {
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> m(-2.0, 2.0);
  for (int it = 0; it < 2000000; ++it) {
    const int E = 1 + (int)(g() % 2046);
    double v = std::ldexp(m(g), (int)(g() % 90) - 88 + E - 1023);
    if (it % 7 == 0) v = std::ldexp(m(g), -1060);
    if (it % 11 == 0) v = it % 2 ? 0.0 : -0.0;
    if (exp_field(v) > E) continue;
    const int64_t X = to_fixed(v, E), Y = to_fixed<61>(v, E);
    const long double a = std::ldexp((long double)v, 57 - (E - 1022)), b = std::ldexp((long double)v, 61 - (E - 1022));
    if (X != (int64_t)std::trunc(a) || Y != (int64_t)std::trunc(b)) return std::printf("value %a %d\n", v, E), 1;
    if ((X < 0 ? -X : X) >= (1ll << 57) || (Y < 0 ? -Y : Y) >= (1ll << 61)) return 2;
    const int hi = digit_hi(X), lo = digit_lo(X);
    if ((int64_t)hi * (1 << 28) + lo != X || lo < -(1 << 27) || lo >= (1 << 27)) return 3;
    if (fold(hi, X) != hi + (int64_t)std::floor(std::ldexp((long double)X, -28) + 0.5L)) return 4;
  }
  // the row unit keeps |X| < 2^58 and the sum below 2^61
  for (int em = -1000; em < 1000; em += 7)
    for (int es = em; es < em + 14; ++es)
      if (em - row_unit(em, es) > 58 || es - row_unit(em, es) > 61) return 5;
  return 0;
}
