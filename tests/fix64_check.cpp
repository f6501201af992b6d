// Host checks of the fixed-point collision (csrc/lbks_fix64.cuh): see test_fix64_host.py.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "../include/lb_ks.h"
#include "../paper_1711_03540_gb300/csrc/lbks_fix64.cuh"

using namespace lbks;
typedef long double ld;

static uint64_t bits(double x) { uint64_t u; std::memcpy(&u, &x, 8); return u; }
static double value(uint64_t u) { double x; std::memcpy(&x, &u, 8); return x; }
static double half_ulp(double x) { return 0.5 * (std::nextafter(std::fabs(x), 1e300) - std::fabs(x)); }

// The FP64 arithmetic of the collision (lbks_device.cuh, collide_rn).
template <int Q> static void native(const double* g, double r, const double* a, const double* b, double* out) {
  double sg = g[0];
  for (int i = 1; i < Q; ++i) sg += g[i];
  const double rho2 = sg * sg;
  double acc = sg;
  for (int p = 1; 2 * p < Q; ++p) {
    const double t = sg * a[2 * p - 1];
    for (int i = 2 * p - 1; i <= 2 * p; ++i) {
      out[i] = std::fma(r, g[i], std::fma(rho2, b[i], t));
      acc -= out[i];
    }
  }
  out[0] = acc;
}

// Random sites of one setting: 0 ok, else the number of a failed check.
template <int Q> static int check(double dx, double dt, double tau, double level, double spread, unsigned seed) {
  double A[7], B[7], a[7], b[7];
  if (lb_ks_params(Q, dx, dt, tau, 0, A, B, nullptr) != LB_KS_OK) return 1;
  for (int i = 0; i < Q; ++i) { a[i] = A[i] / tau; b[i] = B[i] / tau; }
  const double r = 1.0 - 1.0 / tau;
  const FixCoef k = fix_coef(Q, r, 0.0, a, b);
  if (k.z0 == 0) return 2;
  std::mt19937_64 rng(seed);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  int covered = 0;
  const int sites = 20000;
  for (int s = 0; s < sites; ++s) {
    const double rho = level * U(rng);
    double g[7];
    uint64_t in[Q], out[Q];
    ld sum = 0, e[7];
    for (int i = 0; i < Q; ++i) {
      g[i] = (A[i] * rho + B[i] * rho * rho) * (1.0 + spread * U(rng));
      in[i] = bits(g[i]);
      sum += g[i];
    }
    if (!fix_collide<Q>(in, out, k)) continue;
    ++covered;
    int top = 0;
    for (int i = 0; i < Q; ++i) top = std::max(top, (int)((in[i] >> 52) & 0x7ff));
    const double u = std::ldexp(1.0, top - 1079);  // the grid of the results
    // inputs are cut on a grid of 2 u, each with an error below 2 u: 2 r u in r g_i, and with
    // all Q of them in rho 2 Q |a_i| u; products and shifts add at most 4 u, the conversion half an ulp
    e[0] = sum;
    double tol0 = 2.0 * Q * u;
    ld total = 0;
    for (int i = 1; i < Q; ++i) {
      e[i] = (ld)r * g[i] + sum * (ld)a[i] + sum * sum * (ld)b[i];
      e[0] -= e[i];
      const double tol = (2.0 * r + 2.0 * Q * std::fabs(a[i]) + 4.0) * u;
      tol0 += tol;
      if (!(std::fabs((double)((ld)value(out[i]) - e[i])) <= tol + half_ulp(value(out[i])))) return 3;
    }
    if (!(std::fabs((double)((ld)value(out[0]) - e[0])) <= tol0 + half_ulp(value(out[0])))) return 4;
    double conv = 2.0 * Q * u;  // mass: the cut inputs and the conversions alone
    for (int i = 0; i < Q; ++i) {
      total += value(out[i]);
      conv += half_ulp(value(out[i]));
    }
    if (!(std::fabs((double)(total - sum)) <= conv)) return 5;
  }
  if (covered < sites * 9 / 10) return 6;
  return 0;
}

// A periodic lattice advanced n steps in fixed point, in FP64 arithmetic and in long double
// from the same initial populations: rho's error over FP64's.
template <int Q> static double evolve(double dx, double dt, double tau, int N, int n, double amp, double mean) {
  double A[7], B[7], a[7], b[7];
  lb_ks_params(Q, dx, dt, tau, 0, A, B, nullptr);
  for (int i = 0; i < Q; ++i) { a[i] = A[i] / tau; b[i] = B[i] / tau; }
  const double r = 1.0 - 1.0 / tau;
  const FixCoef k = fix_coef(Q, r, 0.0, a, b);
  std::mt19937_64 rng(7);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  std::vector<double> rho(N, mean), f[2][7];  // in fixed point, in FP64 arithmetic
  std::vector<ld> q[7];
  for (int m = 1; m <= 16; ++m) {
    const double am = amp * U(rng), ph = 6.283185307179586 * U(rng);
    for (int x = 0; x < N; ++x) rho[x] += am * std::cos(6.283185307179586 * m * x / N + ph);
  }
  for (int i = 0; i < Q; ++i) {
    q[i].resize(N);
    for (int x = 0; x < N; ++x) q[i][x] = std::fma(B[i], rho[x] * rho[x], A[i] * rho[x]);
    for (int v = 0; v < 2; ++v) f[v][i].assign(q[i].begin(), q[i].end());
  }
  auto shift = [&](auto& p, int i) {
    const int c = i == 0 ? 0 : ((i & 1) ? (i + 1) / 2 : -(i / 2));
    std::rotate(p.begin(), p.begin() + ((N - c) % N), p.end());
  };
  for (int s = 0; s < n; ++s) {
    for (int x = 0; x < N; ++x) {
      double g[7], o[7];
      for (int v = 0; v < 2; ++v) {
        for (int i = 0; i < Q; ++i) g[i] = f[v][i][x];
        uint64_t in[Q], out[Q];
        for (int i = 0; i < Q; ++i) in[i] = bits(g[i]);
        if (v == 0 && fix_collide<Q>(in, out, k)) {
          for (int i = 0; i < Q; ++i) o[i] = value(out[i]);
        } else {
          native<Q>(g, r, a, b, o);
        }
        for (int i = 0; i < Q; ++i) f[v][i][x] = o[i];
      }
      ld sum = 0;
      for (int i = 0; i < Q; ++i) sum += q[i][x];
      ld e0 = sum;
      for (int i = 1; i < Q; ++i) {
        q[i][x] = (ld)r * q[i][x] + sum * (ld)a[i] + sum * sum * (ld)b[i];
        e0 -= q[i][x];
      }
      q[0][x] = e0;
    }
    for (int i = 1; i < Q; ++i) {
      shift(q[i], i);
      for (int v = 0; v < 2; ++v) shift(f[v][i], i);
    }
  }
  ld err[2] = {0, 0};
  for (int x = 0; x < N; ++x) {
    ld ref = 0;
    for (int i = 0; i < Q; ++i) ref += q[i][x];
    for (int v = 0; v < 2; ++v) {
      ld sum = 0;
      for (int i = 0; i < Q; ++i) sum += f[v][i][x];
      err[v] += (sum - ref) * (sum - ref);
    }
  }
  return (double)std::sqrt(err[0] / err[1]);
}

int main() {
  const double settings[][3] = {{0.1, 1e-4, 1.5}, {0.1, 1e-4, 3.0}, {0.0245, 5e-6, 3.0}, {0.2, 5e-5, 1.0},
                                {0.1, 1e-7, 1.0}, {0.05, 1e-4, 2.6}, {0.2, 1e-3, 1.3}, {0.6, 2e-4, 2.0}};
  for (const auto& c : settings)
    for (double level : {1e-30, 1e-6, 0.02, 1.0, 5.0})
      for (double spread : {0.0, 1e-3, 0.5}) {
        const int f5 = check<5>(c[0], c[1], c[2], level, spread, 11), f7 = check<7>(c[0], c[1], c[2], level, spread, 12);
        if (f5 || f7) {
          std::printf("dx %g dt %g tau %g level %g spread %g: D1Q5 %d D1Q7 %d\n", c[0], c[1], c[2], level, spread, f5, f7);
          return 1;
        }
      }
  // (a lattice's error is one draw of a random walk, so the settings are taken together)
  double log5 = 0.0, log7 = 0.0;
  for (const auto& c : settings)
    for (double mean : {0.0, 2.0}) {
      log5 += std::log(evolve<5>(c[0], c[1], c[2], 256, 1500, 0.01, mean));
      log7 += std::log(evolve<7>(c[0], c[1], c[2], 256, 1500, 0.01, mean));
    }
  if (!(log5 <= 0.0 && log7 <= 0.0)) {
    std::printf("errors against FP64 arithmetic's (geometric mean): D1Q5 %g D1Q7 %g\n", std::exp(log5 / 16), std::exp(log7 / 16));
    return 1;
  }
  // not covered: zeros, subnormals, infinities, NaN, values far out of scale, coefficients out of range
  double A[7], B[7], a[7], b[7];
  lb_ks_params(7, 0.1, 1e-4, 2.0, 0, A, B, nullptr);
  for (int i = 0; i < 7; ++i) { a[i] = A[i] / 2.0; b[i] = B[i] / 2.0; }
  const FixCoef k = fix_coef(7, 0.5, 0.0, a, b);
  for (double bad : {0.0, 1e-310, 1e300, 1e6, (double)INFINITY, -(double)INFINITY, (double)NAN}) {
    uint64_t in[7], out[7];
    for (int i = 0; i < 7; ++i) in[i] = bits(bad == 1e6 || bad > 1e299 || bad != bad ? (i == 3 ? bad : 0.1) : bad);
    if (fix_collide<7>(in, out, k)) { std::printf("covered %g\n", bad); return 1; }
  }
  if (fix_coef(7, 0.5, 0.1, a, b).z0 || fix_coef(7, -0.5, 0.0, a, b).z0) return 1;
  a[1] = a[2] = 40.0;
  if (fix_coef(7, 0.5, 0.0, a, b).z0) return 1;
  a[1] = a[2] = NAN;
  if (fix_coef(7, 0.5, 0.0, a, b).z0) return 1;
  std::printf("ok\n");
  return 0;
}
