// Host check of the cluster plan of the one-site-per-thread kernel (csrc/lbks_plan.h): see
// test_blocked_cluster_host.py.
#include <cstdio>
#include <map>
#include <random>

#include "lbks_plan.h"

using namespace lbks;
using namespace lbks::plan;

// Moves one step's values as the kernel's threads do (each its own column, those near a
// portion's ends also the columns its neighbours' threads read) and checks what is read.
static int check(const std::vector<int64_t>& Ns, bool res, int C, int NT, int CL, size_t* clusters) {
  std::vector<Piece> pieces;
  std::vector<int2> bundles;
  if (!plan_clusters(Ns, res, C, NT, CL, &pieces, &bundles)) return 1;
  if (bundles.size() % (size_t)CL) return 2;
  *clusters = bundles.size() / (size_t)CL;
  const int XS = NT + 2 * C * kBlockedPieces, ghost = res ? C : 0;
  const auto site = [&](const Piece& p, int j) { return ((int64_t)p.run << 32) + p.x0 + ghost + j; };
  std::map<int64_t, int> seen;
  for (int c = 1; c <= C; ++c)
    for (int sign : {1, -1}) {
      std::vector<std::vector<int64_t>> ex(bundles.size(), std::vector<int64_t>((size_t)XS, -1));
      for (int pass = 0; pass < 2; ++pass)
        for (size_t b = 0; b < bundles.size(); ++b) {
          if (bundles[b].y > kBlockedPieces) return 3;
          int end = 0;
          for (int q = 0; q < bundles[b].y; ++q) {
            const Piece& p = pieces[(size_t)(bundles[b].x + q)];
            const int64_t N = Ns[(size_t)p.run] + 2 * ghost;
            if (p.t0 != end || p.n > p.nthr || p.st_lo != 0 || p.st_hi != p.n || (p.n < 2 * C && p.n != N)) return 4;
            end = p.t0 + p.nthr;
            if (end > NT) return 5;
            for (int j = 0; j < p.n; ++j) {
              const int col = p.t0 + j + C * (2 * q + 1);
              if (pass == 0) {
                if (c == 1 && sign == 1) ++seen[site(p, j)];
                if (ex[b][(size_t)col] != -1) return 6;  // no two threads write a column
                ex[b][(size_t)col] = site(p, j);
                if (sign > 0 ? j >= p.n - c : j < c) {
                  const bool right = j >= p.n - C;
                  const int to = right ? p.pad_ : p.halo, at = (to & 0xffff) + (right ? j - p.n : j);
                  const size_t block = b / (size_t)CL * (size_t)CL + (size_t)(to >> 16);
                  if ((to >> 16) >= CL || at < 0 || at >= XS || ex[block][(size_t)at] != -1) return 7;
                  ex[block][(size_t)at] = site(p, j);
                }
              } else {
                const int64_t y = p.x0 + ghost + j, from = (y - sign * c + N) % N;
                if (ex[b][(size_t)(col - sign * c)] != ((int64_t)p.run << 32) + from) return 8;
              }
            }
          }
        }
    }
  size_t sites = 0;
  for (int64_t n : Ns) sites += (size_t)(n + 2 * ghost);
  if (seen.size() != sites) return 9;
  for (const auto& s : seen)
    if (s.second != 1) return 10;
  return 0;
}

int main() {
  std::mt19937 rng(5);
  for (int C : {2, 3})
    for (int NT : {64, 96, 128, 192, 256, 384})
      for (int CL : {2, 4, 8})
        for (bool res : {false, true})
          for (int runs : {0, 60}) {
            std::vector<int64_t> Ns;
            for (int64_t n : {2 * C + 1, 13, 4 * C, NT - 7, NT - 1, NT, NT + 1, NT + 2 * C - 1, 2 * NT - 4 * C - 1, CL * NT / 2, CL * NT - 64})
              if (n >= 2 * C + 1 && n + 2 * C <= CL * NT - 2 * portion_min(C, NT)) Ns.push_back(n);
            for (int i = 0; i < runs; ++i) Ns.push_back(2 * C + 1 + (int)(rng() % (unsigned)(CL * NT - 2 * C - 1 - 2 * NT / 16 - 4 * C)));
            size_t clusters = 0;
            const int e = check(Ns, res, C, NT, CL, &clusters);
            if (e) { std::printf("C %d NT %d CL %d reservoir %d runs %d: %d\n", C, NT, CL, res, runs, e); return 1; }
          }
  // the chosen tilings hold what they are chosen for
  for (int Q : {5, 7})
    for (bool res : {false, true})
      for (int i = 0; i < 200; ++i) {
        std::vector<int64_t> Ns(1 + rng() % 200u);
        const unsigned span = 400u << (rng() % 4u);
        for (auto& n : Ns) n = 7 + (int)(rng() % span);
        const ClusterTiling t = choose_clusters(Ns, res, Q, 152, 500);
        std::vector<Piece> pieces;
        std::vector<int2> bundles;
        if (t.CL && !plan_clusters(Ns, res, (Q - 1) / 2, t.NT, t.CL, &pieces, &bundles)) {
          std::printf("cluster tiling %d x %d for %zu lattices of up to %u\n", t.CL, t.NT, Ns.size(), span + 7);
          return 1;
        }
      }
  std::printf("ok\n");
  return 0;
}
