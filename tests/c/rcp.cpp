// gx_rcp (csrc/ba_rcp.h) against the division: prints the largest error in
// units of the last place of the results (long double reference) over random
// significands at every exponent, and how many special values differ from 1 / d.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>

#include "ba_rcp.h"

int main() {
  uint64_t x = 88172645463325252ull;
  auto next = [&] {  // Marsaglia's xorshift
    x ^= x << 13;
    x ^= x >> 7;
    return x ^= x << 17;
  };
  const uint64_t one = 1ull << 52;
  long double worst = 0;
  for (int ex = 23; ex <= 2023; ++ex)
    for (int k = 0; k < 2000; ++k) {
      uint64_t frac = next() & (one - 1);
      if (k < 8) frac = k < 4 ? k : one - 1 - (k - 4);  // the ends of the binade
      const double d = ba::rcp_make((int)(uint32_t)(((uint64_t)ex << 52 | frac) >> 32), (int)(uint32_t)frac);
      const double z = ba::gx_rcp(d);
      const double ulp = std::nextafter(z, std::numeric_limits<double>::infinity()) - z;
      worst = std::fmax(worst, std::fabs((long double)z - 1.0L / d) / ulp);
    }
  const double inf = std::numeric_limits<double>::infinity(), tiny = std::numeric_limits<double>::denorm_min();
  const double special[] = {0.0, -0.0, inf, -inf, std::nan(""), tiny, -tiny, 1e-310, 2.3e-308, 1.7e308, -1.0, -3.0,
                            -1e300, 1.0, 2.0, 0.5, 1024.0};
  int differ = 0;
  for (double d : special) {
    const double a = ba::gx_rcp(d), b = 1.0 / d;
    differ += std::memcmp(&a, &b, 8) != 0 && !(std::isnan(a) && std::isnan(b));
  }
  std::printf("%.6Lf %d\n", worst, differ);
  return 0;
}
