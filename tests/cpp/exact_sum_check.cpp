// Host check of tqs::sq_sum_bits against the FPU: pairs over all exponents and
// their differences, subnormals, zeros, both signs, ties and random patterns.
#include "exact_sq.h"
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
int main() {
  std::mt19937_64 g(2);
  long bad = 0, n = 0;
  auto check = [&](uint32_t a, uint32_t b) {
    float x, y;
    std::memcpy(&x, &a, 4);
    std::memcpy(&y, &b, 4);
    if (!std::isfinite(x) || !std::isfinite(y)) return;
    const double xx = double(x) * x, yy = double(y) * y, want = xx + yy;  // exact squares, one rounding
    uint64_t wb;
    std::memcpy(&wb, &want, 8);
    ++n;
    const uint64_t got = tqs::sq_sum_bits(a, b);
    if (got != wb && bad++ < 5)
      std::printf("mismatch %a %a got %016llx want %016llx\n", x, y, (unsigned long long)got, (unsigned long long)wb);
  };
  auto mant = [&](int k) -> uint32_t {
    switch (k) {
      case 0: return 0;
      case 1: return 1;
      case 2: return 0x7fffff;
      case 3: return 0x400000;
      case 4: return 0x7ff000;
      default: return uint32_t(g() & 0x7fffff);
    }
  };
  for (uint32_t e = 0; e < 255; ++e)
    for (int d = -45; d <= 45; ++d) {
      const int f = int(e) + d;
      if (f < 0 || f > 254) continue;
      for (int i = 0; i < 9; ++i)
        for (int j = 0; j < 9; ++j)
          check((e << 23) | mant(i) | (uint32_t(i & 1) << 31), (uint32_t(f) << 23) | mant(j) | (uint32_t(j & 1) << 31));
    }
  for (long i = 0; i < 3000000; ++i) {
    const uint64_t v = g();
    check(uint32_t(v), uint32_t(v >> 32));
    check((uint32_t(v) & 0x87ffffffu) | 0x38000000u, (uint32_t(v >> 32) & 0x87ffffffu) | 0x38000000u);
  }
  std::printf("checked %ld, mismatches %ld\n", n, bad);
  return bad != 0;
}
