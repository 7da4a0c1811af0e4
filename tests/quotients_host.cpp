// Host program of test_quotients.py: the quotients and roots of
// csrc/softfp.cuh against the processor's, on random significands and on
// significands next to powers of two, exponents over the whole range.  The
// FP32 seeds are off by up to two units either way, as the device's are.
// Prints the number of differing results of each function and srsqrt's largest
// error in units of the last place.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>

static int seed_off = 0;
static float nudged(float f) {
  uint32_t u;
  memcpy(&u, &f, 4);
  u += seed_off;
  memcpy(&f, &u, 4);
  return f;
}
#define SF_SEED(f) nudged(f)
#include "softfp.cuh"
using namespace sacra;

int main() {
  std::mt19937_64 g(1);
  auto value = [&](int spread) {
    uint64_t m = g() & ((1ull << 52) - 1);
    const int kind = (int)(g() % 4);
    if (kind == 1) m = g() % 4;                                        // just above a power of two
    if (kind == 2) m = ((1ull << 52) - 1) - g() % 4;                   // just below
    if (kind == 3) m &= ~((1ull << (g() % 52)) - 1);                   // few significant bits
    const uint64_t e = 1023 - spread + g() % (2 * spread + 1);
    const uint64_t b = ((g() & 1) << 63) | (e << 52) | m;
    double d;
    memcpy(&d, &b, 8);
    return d;
  };
  const double special[] = {0.0, -0.0, 1.0, 3.0, INFINITY, -INFINITY, NAN, 5e-324, -2.3e-308, 2.2250738585072014e-308,
                            1.7976931348623157e308, -1.0, 4.0, 2.0};
  long long bad[3] = {};
  double worst = 0.0;
  auto differ = [](double a, double b) { return !(std::isnan(a) && std::isnan(b)) && memcmp(&a, &b, 8) != 0; };
  auto check = [&](double a, double b) {
    bad[0] += differ(sf::sdiv(a, b), a / b);
    bad[1] += differ(sf::srcp(b), 1.0 / b);
    bad[2] += differ(sf::ssqrt(std::fabs(a)), std::sqrt(std::fabs(a)));
    const double x = std::fabs(a);
    if (std::isnormal(x)) {
      const long double ref = 1.0L / std::sqrt((long double)x);
      const double r = sf::srsqrt(x);
      worst = std::fmax(worst, (double)(std::fabs((long double)r - ref) / (std::nextafter((double)ref, INFINITY) - (double)ref)));
    }
  };
  for (seed_off = -2; seed_off <= 2; ++seed_off) {
    for (int i = 0; i < 1000000; ++i) check(value(i & 1 ? 3 : 1000), value(i & 1 ? 3 : 1000));
    // quotients next to ties: a / b = (2 q + 1) / 2 units with an error of order 1 / b
    for (int i = 0; i < 300000; ++i) {
      const uint64_t q = (1ull << 53) | (g() & ((1ull << 53) - 1)) | 1, d = (1ull << 52) | (g() & ((1ull << 52) - 1));
      const unsigned __int128 p = (unsigned __int128)q * d >> 53;
      check((double)(uint64_t)p, (double)d);
      check((double)((uint64_t)p + 1), (double)d);
    }
    // arguments next to squares of half units
    for (int i = 0; i < 300000; ++i) {
      const uint64_t q = (1ull << 53) | (g() & ((1ull << 53) - 1)) | 1;
      const uint64_t m = (uint64_t)((unsigned __int128)q * q >> 54);
      check((double)m, 1.5);
      check((double)(m + 1), 1.5);
      check(2.0 * (double)m, 1.5);
    }
    for (double a : special)
      for (double b : special) check(a, b);
  }
  printf("%lld %lld %lld %.4f\n", bad[0], bad[1], bad[2], worst);
}
