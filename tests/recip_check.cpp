// recip_fixed (fixexp.h) against the division, bit for bit, with the seed moved
// over all that the device's FP32 division may return: mantissas at both ends of
// a binade, hard ones (reciprocals next to the middle of two doubles), random.
#include "fixexp.h"

#include <cstdio>
#include <random>

int main() {
  std::mt19937_64 g(7);
  long bad = 0, n = 0;
  auto check = [&](uint64_t bits) {
    double d;
    std::memcpy(&d, &bits, 8);
    const double want = 1.0 / d;
    uint64_t w;
    std::memcpy(&w, &want, 8);
    if (bd::recip_fixed(d) != want) ++bad;
    const uint32_t fb = 0x3f800000u | (uint32_t(bits >> 29) & 0x7fffffu);
    float f;
    std::memcpy(&f, &fb, 4);
    // the seed's value is in (1/2, 1], whose unit in the last place is 2^-24 (2^8 at 2^32): two
    // units on either side, cut at 2^32 - 1
    const double r = 4294967296.0 / double(f);
    for (int u : {-512, -256, 0, 256, 512}) {
      const double s = r + u;
      const uint32_t r0 = s >= 4294967295.0 ? 0xffffffffu : uint32_t(s);
      if (bd::recip_from_seed(bits, r0) != w) ++bad;
      ++n;
    }
  };
  for (int i = 0; i < 600000; ++i) {
    uint64_t m = g() & 0xfffffffffffffull;
    if (i % 5 == 1) m &= 0x3fffff;
    if (i % 5 == 2) m |= 0xfffffffc00000ull;
    if (i % 5 == 3) m = (m & 0xfffffe0000000ull) | (i % 2 ? 0x1fffffffull : 0);   // the seed's cut at its largest, and none
    if (i % 5 == 4) {                          // 1/m next to a midpoint: m about 2^106 / (2 q + 1)
      const long double h = 2.0L * double((g() >> 11) | 0x10000000000000ull) + 1;
      m = (uint64_t(0x1p106L / h) + g() % 3 - 1) & 0xfffffffffffffull;
    }
    check((g() & 1) << 63 | (1 + g() % 2043) << 52 | m);
  }
  for (uint64_t be : std::initializer_list<uint64_t>{1, 1023, 2043})
    for (uint64_t m : std::initializer_list<uint64_t>{0, 1, 2, 0xfffffffffffffull, 0xffffffffffffeull}) check(be << 52 | m);
  std::printf("%ld %ld\n", bad, n);
  return 0;
}
