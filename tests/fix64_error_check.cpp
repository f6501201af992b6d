// Host check of the fixed-point collision's error over long runs: see test_fix64_error_host.py.
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#include <thread>
#include <vector>

#include "../include/lb_ks.h"
#include "../paper_1711_03540_gb300/csrc/lbks_fix64.cuh"

using namespace lbks;
typedef long double ld;

static uint64_t bits(double x) { uint64_t u; std::memcpy(&u, &x, 8); return u; }
static double value(uint64_t u) { double x; std::memcpy(&x, &u, 8); return x; }

struct Setting { double dx, dt, tau, mean; };

template <int Q> struct Run {
  double A[7], B[7], a[7], b[7], r;
  FixCoef k;
  explicit Run(const Setting& c) {
    lb_ks_params(Q, c.dx, c.dt, c.tau, 0, A, B, nullptr);
    for (int i = 0; i < Q; ++i) { a[i] = A[i] / c.tau; b[i] = B[i] / c.tau; }
    r = 1.0 - 1.0 / c.tau;
    k = fix_coef(Q, r, 0.0, a, b);
  }
  // The FP64 arithmetic of the collision (lbks_device.cuh, collide_rn).
  void native(const double* g, double* out) const {
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
  // As the kernels choose (collide in lbks_device.cuh).
  void library(const double* g, double* out) const {
    uint64_t in[Q], o[Q];
    for (int i = 0; i < Q; ++i) in[i] = bits(g[i]);
    if (k.z0 != 0 && fix_collide<Q>(in, o, k)) {
      for (int i = 0; i < Q; ++i) out[i] = value(o[i]);
    } else {
      native(g, out);
    }
  }
};

struct Result { ld err[2] = {0, 0}, mass[2] = {0, 0}; };

// n steps of a periodic lattice of N sites with the library's collision, in FP64 arithmetic and
// in long double, from the same populations: squared errors of rho, and of its mean.
template <int Q> static void evolve(const Setting& c, int N, int n, unsigned seed, Result* res) {
  const Run<Q> run(c);
  std::mt19937_64 rng(seed);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  std::vector<double> rho(N, c.mean), f[2][7];
  std::vector<ld> q[7];
  for (int m = 1; m <= 16; ++m) {
    const double am = 0.01 * U(rng), ph = 6.283185307179586 * U(rng);
    for (int x = 0; x < N; ++x) rho[x] += am * std::cos(6.283185307179586 * m * x / N + ph);
  }
  for (int i = 0; i < Q; ++i) {
    q[i].resize(N);
    for (int x = 0; x < N; ++x) q[i][x] = std::fma(run.B[i], rho[x] * rho[x], run.A[i] * rho[x]);
    for (auto& v : f) v[i].assign(q[i].begin(), q[i].end());
  }
  // (streaming: plane i's value at site x stands at x - c_i s, s the steps done)
  int off[7] = {};
  for (int s = 0; s < n; ++s) {
    for (int x = 0; x < N; ++x) {
      int id[7];
      for (int i = 0; i < Q; ++i) id[i] = x + off[i] < N ? x + off[i] : x + off[i] - N;
      double g[7], o[7];
      for (int v = 0; v < 2; ++v) {
        for (int i = 0; i < Q; ++i) g[i] = f[v][i][id[i]];
        if (v == 0) run.library(g, o);
        else run.native(g, o);
        for (int i = 0; i < Q; ++i) f[v][i][id[i]] = o[i];
      }
      ld sum = 0;
      for (int i = 0; i < Q; ++i) sum += q[i][id[i]];
      ld e0 = sum;
      for (int i = 1; i < Q; ++i) {
        ld& z = q[i][id[i]];
        z = (ld)run.r * z + sum * (ld)run.a[i] + sum * sum * (ld)run.b[i];
        e0 -= z;
      }
      q[0][id[0]] = e0;
    }
    for (int i = 1; i < Q; ++i) {
      const int ci = (i & 1) ? (i + 1) / 2 : -(i / 2);
      off[i] = ((off[i] - ci) % N + N) % N;
    }
  }
  ld mean[2] = {0, 0};
  for (int x = 0; x < N; ++x) {
    ld ref = 0, sum[2] = {0, 0};
    for (int i = 0; i < Q; ++i) {
      const int y = (x + off[i]) % N;
      ref += q[i][y];
      for (int v = 0; v < 2; ++v) sum[v] += f[v][i][y];
    }
    for (int v = 0; v < 2; ++v) {
      res->err[v] += (sum[v] - ref) * (sum[v] - ref);
      mean[v] += (sum[v] - ref) / N;
    }
  }
  for (int v = 0; v < 2; ++v) res->mass[v] += mean[v] * mean[v];
}

// One collision of states near equilibrium: the squared errors of the planes +-3 (D1Q7), the
// smallest, which take nothing of g_0's rounding.
static void planes(const Setting& c, ld* err) {
  const Run<7> run(c);
  std::mt19937_64 rng(9);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  for (int s = 0; s < 20000; ++s) {
    const double level = c.mean + 0.05 * U(rng);
    double g[7], o[2][7];
    ld sum = 0;
    for (int i = 0; i < 7; ++i) {
      const double rho = level * (1.0 + 0.01 * U(rng));
      g[i] = run.A[i] * rho + run.B[i] * rho * rho;
      sum += g[i];
    }
    run.library(g, o[0]);
    run.native(g, o[1]);
    for (int i = 5; i < 7; ++i)
      for (int v = 0; v < 2; ++v) {
        const ld d = o[v][i] - ((ld)run.r * g[i] + sum * (ld)run.a[i] + sum * sum * (ld)run.b[i]);
        err[v] += d * d;
      }
  }
}

int main() {
  const Setting settings[] = {{0.6, 1e-6, 3.0, 0.0}, {0.3, 1e-7, 1.5, 2.0},  {0.3, 1e-6, 1.5, 2.0},  {0.4, 1e-6, 1.3, 3.0},
                              {0.1, 1e-5, 1.5, 3.0}, {0.1, 1e-4, 2.4, 3.0},  {0.1, 1e-4, 1.5, 0.0},  {0.0245, 5e-6, 3.0, 0.0},
                              {0.2, 5e-5, 1.0, 0.0}, {0.6, 1e-8, 2.0, 1.5}};
  constexpr int kSettings = sizeof(settings) / sizeof(settings[0]), kLattices = 3, kSites = 32, kSteps = 200000;
  Result res[kSettings][2][kLattices];
  std::atomic<int> next{0};
  std::vector<std::thread> pool;
  const unsigned cores = std::thread::hardware_concurrency();
  for (unsigned t = 0; t < (cores ? cores : 1); ++t)
    pool.emplace_back([&] {
      for (int j; (j = next++) < kSettings * 2 * kLattices;) {
        const int l = j % kLattices, q = j / kLattices % 2, s = j / (2 * kLattices);
        if (q) evolve<7>(settings[s], kSites, kSteps, 100 + l, &res[s][q][l]);
        else evolve<5>(settings[s], kSites, kSteps, 100 + l, &res[s][q][l]);
      }
    });
  for (auto& t : pool) t.join();
  int bad = 0;
  for (int s = 0; s < kSettings; ++s) {
    const Setting& c = settings[s];
    for (int q = 0; q < 2; ++q) {
      ld err[2] = {0, 0}, mass = 0;
      for (const Result& r : res[s][q]) {
        for (int v = 0; v < 2; ++v) err[v] += r.err[v];
        mass += r.mass[0];
      }
      const double ratio = (double)std::sqrt(err[0] / err[1]), drift = (double)std::sqrt(mass / kLattices);
      // no further from the exact run than FP64 arithmetic; the mass of a lattice whose mean is not
      // zero kept to its last place
      if (!(ratio <= 1.0) || (c.mean != 0.0 && !(drift <= 0x1p-52 * c.mean))) {
        std::printf("dx %g dt %g tau %g mean %g D1Q%d: error %.2f of FP64 arithmetic's, mass off by %.1e\n", c.dx, c.dt,
                    c.tau, c.mean, q ? 7 : 5, ratio, drift);
        bad = 1;
      }
    }
    ld err[2] = {0, 0};
    planes(c, err);
    if (!(err[0] <= err[1])) {
      std::printf("dx %g dt %g tau %g mean %g: planes +-3 of one collision %.2f of FP64 arithmetic's\n", c.dx, c.dt, c.tau,
                  c.mean, (double)std::sqrt(err[0] / err[1]));
      bad = 1;
    }
  }
  if (!bad) std::printf("ok\n");
  return bad;
}
