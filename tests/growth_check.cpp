// Host check of the constructors' stability decision (csrc/lbks_growth.h): see test_growth_host.py.
#include <cmath>
#include <cstdio>
#include <random>

#include "../include/lb_ks.h"
#include "../paper_1711_03540_gb300/csrc/lbks_growth.h"

int main() {
  std::mt19937_64 rng(29);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  int unstable = 0;
  for (int i = 0; i < 120; ++i) {
    const int Q = i & 1 ? 7 : 5, variant = Q == 7 ? (i / 2) % 4 : 0;
    const double dx = std::pow(10.0, -1.7 + 1.4 * U(rng)), dt = std::pow(10.0, -7.0 + 4.0 * U(rng));
    const double tau = i % 5 == 0 ? 1.0 : 1.0 + 3.0 * U(rng);
    double g = 0.0;
    if (lb_ks_max_growth(Q, dx, dt, tau, variant, 0.0, 128, &g) != LB_KS_OK) return 1;
    for (double limit : {1.05 * 0.25, g + 1e-3 * std::fabs(g) + 1e-6, g - 1e-3 * std::fabs(g) - 1e-6})
      if ((lbks::growth_above(Q, dx, dt, tau, variant, 128, limit, true) > limit) != (g > limit) ||
          std::fabs(lbks::growth_above(Q, dx, dt, tau, variant, 128, limit, false) - std::fmax(g, limit)) >
              1e-9 * std::fabs(g) + 1e-10 / dt) {
        std::printf("D1Q%d dx %g dt %g tau %g variant %d: growth %g limit %g\n", Q, dx, dt, tau, variant, g, limit);
        return 1;
      }
    unstable += g > 1.05 * 0.25;
  }
  if (unstable < 20 || unstable > 100) return 1;
  std::printf("ok\n");
  return 0;
}
