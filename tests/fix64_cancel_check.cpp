// Host check of the fixed-point collision at sites whose populations cancel: see
// test_fix64_cancel_host.py.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>

#include "../include/lb_ks.h"
#include "../paper_1711_03540_gb300/csrc/lbks_fix64.cuh"

using namespace lbks;
typedef long double ld;

static uint64_t bits(double x) { uint64_t u; std::memcpy(&u, &x, 8); return u; }
static double value(uint64_t u) { double x; std::memcpy(&x, &u, 8); return x; }

template <int Q> static int check(double dx, double dt, double tau, double level, unsigned seed) {
  double A[7], B[7], a[7], b[7];
  if (lb_ks_params(Q, dx, dt, tau, 0, A, B, nullptr) != LB_KS_OK) return 1;
  for (int i = 0; i < Q; ++i) { a[i] = A[i] / tau; b[i] = B[i] / tau; }
  const double r = 1.0 - 1.0 / tau;
  const FixCoef k = fix_coef(Q, r, 0.0, a, b);
  std::mt19937_64 rng(seed);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  for (int t = 0; t < 4000; ++t) {
    // neighbours of densities about `level` on either side of a zero, a sum of 2^-1 .. 2^-56 of it
    double g[7];
    ld sum = 0;
    for (int i = 1; i < Q; ++i) {
      const double rho = level * ((i & 1) ? -U(rng) : U(rng));
      g[i] = A[i] * rho + B[i] * rho * rho;
      sum += g[i];
    }
    g[0] = (double)(std::ldexp((t & 1) ? -U(rng) : U(rng), -1 - t % 56) * level - sum);
    uint64_t in[Q], out[Q];
    double top = 0.0;
    sum += g[0];
    for (int i = 0; i < Q; ++i) {
      in[i] = bits(g[i]);
      const double size = std::max({std::fabs(A[i]), 4.0 * std::fabs(B[i]), 1e-300});
      top = std::max(top, std::fabs(g[i]) / (i ? size : 1.0));
    }
    if (!fix_collide<Q>(in, out, k)) continue;
    // 64 units of the last place of g_0 at the neighbours' density: four bits above the sum of
    // what the conversions, the products and the shifts lose
    const ld tol = top * 64 * 0x1p-53L;
    for (int i = 1; i < Q; ++i) {
      const ld e = (ld)r * g[i] + sum * (ld)a[i] + sum * sum * (ld)b[i];
      if (!(std::fabs((double)((ld)value(out[i]) - e)) <= tol)) {
        std::printf("speed %d: %g, not %g (sum %g, scale %g)\n", i, value(out[i]), (double)e, (double)sum, top);
        return 2;
      }
    }
  }
  return 0;
}

int main() {
  const double settings[][3] = {{0.1, 1e-4, 1.5}, {0.1, 1e-4, 3.0}, {0.0245, 5e-6, 3.0}, {0.2, 5e-5, 1.0}, {0.6, 2e-4, 2.0}};
  for (const auto& c : settings)
    for (double level : {0.02, 1.0, 3.0})
      if (check<5>(c[0], c[1], c[2], level, 21) || check<7>(c[0], c[1], c[2], level, 22)) {
        std::printf("dx %g dt %g tau %g level %g\n", c[0], c[1], c[2], level);
        return 1;
      }
  std::printf("ok\n");
  return 0;
}
