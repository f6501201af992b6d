// Host check of the one-site-per-thread tiling of batches with few long lattices: see
// test_blocked_order_host.py.
#include <algorithm>
#include <array>
#include <cstdio>
#include <random>
#include <vector>

#include "lbks_plan.h"

using namespace lbks;
using namespace lbks::plan;

int main() {
  std::mt19937 rng(7);
  std::vector<std::vector<int64_t>> batches;
  const auto mixed = [&](int a, int64_t na, int b, int64_t nb) {
    std::vector<int64_t> v((size_t)a, na);
    for (int i = 0; i < b; ++i) v.insert(v.begin() + (int64_t)((2 * i + 1) % (int)v.size()), nb);
    batches.push_back(v);
  };
  mixed(128, 100, 128, 2048);
  mixed(255, 64, 1, 5000);
  mixed(4096, 200, 1, 8000);
  mixed(256, 300, 1, 6000);
  for (const auto& c : {std::array<int, 3>{2945, 163, 257}, {464, 46, 259}, {177, 19, 269}, {452, 20, 97}, {129, 7, 700}})
    for (int t = 0; t < 20; ++t) {
      std::vector<int64_t> v((size_t)c[0]);
      for (auto& n : v) n = c[1] + (int64_t)(rng() % (unsigned)(c[2] - c[1] + 1));
      batches.push_back(v);
    }
  for (const auto& batch : batches)
    for (int Q : {5, 7})
      for (bool res : {false, true})
        for (bool f64 : {true, false})
          for (int kwhole : {50, 1000}) {
            BlockedTiling first;
            ClusterTiling first_c;
            for (int order = 0; order < 4; ++order) {  // as given, reversed, shuffled
              std::vector<int64_t> Ns = batch;
              if (order == 1) std::reverse(Ns.begin(), Ns.end());
              if (order > 1) std::shuffle(Ns.begin(), Ns.end(), rng);
              const BlockedTiling b = choose_blocked(Ns, res, Q, blocked_cost(Q, f64, false), 152, kwhole);
              const ClusterTiling c = choose_clusters(Ns, res, Q, 152, kwhole);
              if (order == 0) first = b;
              if (order == 0) first_c = c;
              std::vector<Piece> pieces;
              const int64_t longest = *std::max_element(Ns.begin(), Ns.end()) + (res ? Q - 1 : 0);
              if (!plan_blocked(Ns, res, (Q - 1) / 2, b.NT, b.k, &pieces) || (longest > b.NT && b.k > 48) ||
                  b.NT != first.NT || b.k != first.k || b.spread != first.spread || c.NT != first_c.NT || c.CL != first_c.CL) {
                std::printf("%zu lattices up to %lld, order %d: NT %d k %d (first NT %d k %d)\n", Ns.size(),
                            (long long)longest, order, b.NT, b.k, first.NT, first.k);
                return 1;
              }
            }
          }
  std::printf("ok\n");
  return 0;
}
