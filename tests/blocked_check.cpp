// Host checks of the one-site-per-thread kernel's plan (csrc/lbks_plan.h): see
// test_blocked_host.py.
#include <cstdio>
#include <random>

#include "lbks_plan.h"

using namespace lbks;
using namespace lbks::plan;

// 0 if the plan holds every site once with its halo and no two pieces share a thread.
static int check(const std::vector<int64_t>& Ns, bool res, int C, int NT, int k, bool spread) {
  std::vector<Piece> pieces;
  std::vector<int2> bundles;
  if (!plan_blocked(Ns, res, C, NT, k, &pieces)) return NT - 2 * C * k > 0 ? 1 : 0;
  std::vector<Piece> ordered = pieces;
  blocked_bundles(ordered, NT, spread, &bundles);
  if (ordered.size() != pieces.size()) return 2;
  if (bundles.empty())  // one piece each
    for (size_t b = 0; b < ordered.size(); ++b) bundles.push_back(int2{(int)b, 1});
  std::vector<std::vector<int>> seen(Ns.size());
  const int ghost = res ? C : 0;
  for (size_t r = 0; r < Ns.size(); ++r) seen[r].assign((size_t)(Ns[r] + 2 * ghost), 0);
  size_t at = 0;
  for (const int2 b : bundles) {
    if ((size_t)b.x != at || b.y < 1 || b.y > kBlockedPieces) return 3;
    int end = 0;
    for (int q = 0; q < b.y; ++q) {
      const Piece& p = ordered[at + (size_t)q];
      if (p.t0 != end || p.n < 1 || p.n > p.nthr) return 4;  // (a thread's piece is the last one it reaches)
      end = p.t0 + p.nthr;
      const int64_t n = Ns[(size_t)p.run] + 2 * ghost;
      const bool whole = p.n == n;
      if (!whole && !res && (p.x0 < 0 || p.x0 >= n || p.n > n)) return 5;
      for (int j = p.st_lo; j < p.st_hi; ++j) {
        const int64_t y = p.x0 + ghost + j;  // the node's place in [0, n) (reservoir), or a ring site
        if (res && (y < 0 || y >= n)) return 6;
        ++seen[(size_t)p.run][(size_t)(y % n)];
      }
      if (whole) continue;
      const bool left = res && p.x0 == -ghost, right = res && p.x0 + ghost + p.n == n;
      if ((!left && p.st_lo < C * k) || (!right && p.n - p.st_hi < C * k)) return 7;
    }
    if (end > NT) return 8;
    at += (size_t)b.y;
  }
  for (const auto& s : seen)
    for (int c : s)
      if (c != 1) return 9;
  return 0;
}

int main() {
  std::mt19937 rng(3);
  for (int C : {2, 3})
    for (int NT : {64, 96, 128, 256, 384, 512})
      for (int k : {1, 4, 8, 16, 48})
        for (bool res : {false, true})
          for (bool spread : {false, true}) {
            std::vector<int64_t> Ns;
            for (int64_t n : {2 * C + 1, 13, NT - 2 * C - 1, NT - 2 * C, NT - 1, NT, NT + 1, 2 * NT, 2 * NT - 4 * C * k, 5 * NT + 3})
              if (n >= 2 * C + 1) Ns.push_back(n);
            for (int i = 0; i < 60; ++i) Ns.push_back(2 * C + 1 + (int)(rng() % 900u));
            const int e = check(Ns, res, C, NT, k, spread);
            if (e) { std::printf("C %d NT %d k %d reservoir %d spread %d: %d\n", C, NT, k, res, spread, e); return 1; }
          }
  // the chosen tilings hold what they are chosen for
  for (int Q : {5, 7})
    for (bool f64 : {false, true})
     for (bool col : {false, true})
      for (bool res : {false, true})
        for (int64_t n : {7, 60, 400, 513, 4096, 100001, 1 << 24})
          for (int runs : {1, 40, 3000}) {
            if (n * runs > (1 << 24)) continue;
            const std::vector<int64_t> Ns((size_t)runs, n);
            const BlockedTiling b = choose_blocked(Ns, res, Q, blocked_cost(Q, f64, col), 152, 500);
            std::vector<Piece> pieces;
            if (b.NT < 32 || b.NT > (f64 && !col ? 384 : 512) || b.NT % 32 || b.k < 1 ||
                !plan_blocked(Ns, res, (Q - 1) / 2, b.NT, b.k, &pieces)) {
              std::printf("tiling NT %d k %d for %d x %lld\n", b.NT, b.k, runs, (long long)n);
              return 1;
            }
          }
  // the register-resident choice holds every lattice whole that the fixed tiling does, and
  // leaves scaled FP16 batches with segments alone (their launches round)
  for (int Q : {5, 7})
    for (bool f16 : {false, true})
      for (int i = 0; i < 300; ++i) {
        std::vector<int64_t> Ns(1 + rng() % (i % 3 ? 40u : 1500u));
        const unsigned span = 20u << (rng() % 10u);
        for (auto& n : Ns) n = 7 + (int)(rng() % span);
        const ResidentTiling t = choose_resident(Ns, Q, f16, 152, 500, [](int S, int NT) { return (size_t)S * NT * 40; });
        if (t.S == 0) continue;
        int64_t longest = 0;
        for (int64_t n : Ns) longest = std::max(longest, n);
        std::vector<Piece> rings, segs, rings20, segs20;
        const int C = (Q - 1) / 2, cl = longest > t.S * t.NT && longest <= 2 * t.S * t.NT ? 2 : 1;
        const bool held = plan_pieces(Ns, C, t.S, t.NT, cl * t.NT, t.kseg ? t.kseg : 8, cl == 2 ? 32 : 0, &rings, &segs);
        plan_pieces(Ns, C, 20, 256, longest > 5120 ? 512 : 256, 85, 32, &rings20, &segs20);
        if (!held || (f16 && (!segs20.empty() || !segs.empty()))) {
          std::printf("resident tiling S %d NT %d for %zu lattices up to %lld\n", t.S, t.NT, Ns.size(), (long long)longest);
          return 1;
        }
      }
  std::printf("ok\n");
  return 0;
}
