// Host check of the fixed-point collision's input conversion: see test_fix64_jam_host.py.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>

#include "../paper_1711_03540_gb300/csrc/lbks_fix64.cuh"

static uint64_t bits(double x) { uint64_t u; std::memcpy(&u, &x, 8); return u; }

int main() {
  std::mt19937_64 rng(5);
  std::uniform_real_distribution<double> U(1.0, 2.0);
  const uint32_t e = 1023 + 7;
  for (int gap = 0; gap <= 70; ++gap) {
    double mean = 0.0;
    const int draws = 4000;
    for (int t = 0; t < 4 + draws; ++t) {
      const double m = t == 0 ? 1.0 : t == 1 ? 1.0 + 0x1p-52 : t == 2 ? 1.5 : t == 3 ? 1.0 + 0x1p-20 : U(rng);
      for (double sign : {1.0, -1.0}) {
        const double v = sign * std::ldexp(m, 7 - gap);
        int32_t h, l, sg;
        lbks::fix64::to_limbs(bits(v), e, h, l, sg);
        const long double grid = std::ldexp(1.0L, (int)e - 1078), x = v / grid, got = (long double)h * 0x1p28L + l;
        const long double cut = std::trunc(x);
        const bool lost = cut != x, odd = std::fmod(std::fabs(cut), 2.0L) != 0.0L;
        const long double want = cut + (lost && !odd ? (long double)sign : 0.0L);
        if (got != want) {
          std::printf("gap %d value %a: %.1Lf, not %.1Lf\n", gap, v, got, want);
          return 1;
        }
        if (t >= 4 && sign > 0.0) mean += (double)(got - x) / draws;
      }
    }
    // unbiased while the grid still resolves the value (an error is below 1, so the mean of
    // 4000 has a deviation below 0.016)
    if (gap < 50 && !(std::fabs(mean) < 5 * 0.016)) {
      std::printf("gap %d: mean error %g of the grid\n", gap, mean);
      return 1;
    }
  }
  int32_t h, l, sg;
  for (double zero : {0.0, -0.0}) {
    lbks::fix64::to_limbs(bits(zero), e, h, l, sg);
    if (h || l) return 1;
  }
  std::printf("ok\n");
  return 0;
}
