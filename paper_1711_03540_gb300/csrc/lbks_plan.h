// Host-side planning of the register-resident kernel: how lattices become pieces
// (whole rings, haloed halves for cluster pairs, haloed segments), and how pieces are
// packed into work groups (bundles) of one block or a two-block cluster.  Plain C++
// (no device code), so that host tests can check it directly.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <functional>
#include <initializer_list>
#include <utility>
#include <vector>

#include "lbks_internal.h"

namespace lbks {
namespace plan {

// Sites per tile of the plain kernel family (one thread per site, one block per tile).
constexpr int kPlainTileMax = 256;
constexpr int kPlainTileMin = 32;

// Sites per plain-family tile: the largest of 256, 128, 64 and 32 that still gives every
// SM two tiles, else 32.  A small workload (one lattice of a few thousand sites) in
// 256-site tiles runs on a few SMs, each doing 256 sites' FP64 arithmetic per step at
// GB300's low FP64 rate, while the rest idle; smaller tiles spread the same per-site
// work over more SMs.  Results do not depend on the tiling (each thread updates one
// site on its own).  Reservoir lattices' tiles also cover their 2 c_max ghost nodes.
inline int plain_tile_sites(const std::vector<int64_t>& Ns, bool reservoir, int cmax, int sms) {
  for (int t = kPlainTileMax; t > kPlainTileMin; t /= 2) {
    int64_t tiles = 0;
    for (int64_t n : Ns) tiles += (n + (reservoir ? 2 * cmax : 0) + t - 1) / t;
    if (tiles >= 2 * (int64_t)sms) return t;
  }
  return kPlainTileMin;
}

// The plain family's tiles: run by run, consecutive stretches of plain_tile_sites sites
// (the last one of a run shorter) covering [0, N) of each run, or [-c_max, N + c_max)
// for reservoir lattices; *tile receives the tile length (the launches' block size).
inline std::vector<Tile> plain_tiles(const std::vector<int64_t>& Ns, bool reservoir, int cmax, int sms, int* tile) {
  const int t = plain_tile_sites(Ns, reservoir, cmax, sms);
  std::vector<Tile> pt;
  for (int32_t r = 0; r < (int32_t)Ns.size(); ++r) {
    const int64_t g0 = reservoir ? -cmax : 0, g1 = reservoir ? Ns[r] + cmax : Ns[r];
    for (int64_t x = g0; x < g1; x += t) pt.push_back(Tile{r, (int32_t)x, (int32_t)std::min<int64_t>(t, g1 - x), 0});
  }
  *tile = t;
  return pt;
}

// One half of a ring of N sites for a cluster pair: own sites [x_own, x_own + len) of
// the ring with `halo` sites on each side, lengthened on the right until it splits
// into runs of S and S-1 sites; false if that takes more than NT threads.
inline bool plan_half(int32_t r, int64_t N, int64_t x_own, int64_t len, int halo, int S, int NT, Piece* p) {
  int64_t n = len + 2 * halo;
  int64_t V = (n + S - 1) / S;
  while (n <= V * (S - 1)) { ++n; V = (n + S - 1) / S; }
  if (V > NT) return false;
  *p = Piece{};
  p->run = r; p->t0 = 0; p->nthr = (int)V; p->n = (int)n;
  p->x0 = ((x_own - halo) % N + N) % N;
  p->st_lo = halo; p->st_hi = (int)(halo + len);
  p->halo = halo;
  return true;
}

// Pieces of every run for (S, NT): rings (whole lattices held by at most ring_cap
// threads: NT, or 2 NT for two-block clusters) and segments (for longer lattices,
// held by one block each, with c_max * kseg halo sites per side); false if some
// run cannot be held.  With two-block clusters and kx > 0, a lattice longer than one
// block holds is split into two halves (consecutive in `rings`, halo c_max kx) when
// each half with its halos fits one block, instead of one ring across both blocks.
inline bool plan_pieces(const std::vector<int64_t>& Ns, int C, int S, int NT, int ring_cap, int kseg, int kx,
                        std::vector<Piece>* rings, std::vector<Piece>* segs) {
  rings->clear();
  segs->clear();
  rings->reserve(Ns.size() + Ns.size() / 2);
  for (int32_t r = 0; r < (int32_t)Ns.size(); ++r) {
    const int64_t N = Ns[r];
    // Ring: hold m copies of the lattice around one ring of m N sites (m > 1 only
    // for lattices shorter than S (S-1), which cannot be cut into runs of S and
    // S-1 sites).  Translation invariance keeps the copies bitwise identical;
    // the first one is stored.
    bool ring = false;
    for (int64_t m = 1;; ++m) {
      const int64_t n = m * N;
      const int64_t V = (n + S - 1) / S;
      if (V > ring_cap) break;
      if (n > V * (S - 1)) {
        if (V > NT && kx > 0) {
          const int halo = C * kx;
          const int64_t NA = (N + 1) / 2, NB = N - NA;
          Piece a{}, b{};
          if (NB >= 2 * halo && plan_half(r, N, 0, NA, halo, S, NT, &a) && plan_half(r, N, NA, NB, halo, S, NT, &b)) {
            rings->push_back(a);
            rings->push_back(b);
            ring = true;
            break;
          }
        }
        Piece p{};
        p.run = r; p.t0 = 0; p.nthr = (int)V; p.n = (int)n; p.x0 = 0; p.st_lo = 0; p.st_hi = (int)N;
        rings->push_back(p);
        ring = true;
        break;
      }
    }
    if (ring) continue;
    const int64_t h2 = 2LL * C * kseg;
    const int64_t room = (int64_t)NT * S - h2 - 2 * S;
    if (room <= 0) return false;
    const int64_t nseg = (N + room - 1) / room;
    const int64_t Ls = (N + nseg - 1) / nseg;
    for (int64_t s0 = 0; s0 < N; s0 += Ls) {
      const int64_t len = std::min<int64_t>(Ls, N - s0);
      int64_t n = len + h2;
      int64_t V = (n + S - 1) / S;
      while (n <= V * (S - 1)) { ++n; V = (n + S - 1) / S; }
      if (V > NT) return false;
      Piece p{};
      p.run = r; p.t0 = 0; p.nthr = (int)V; p.n = (int)n;
      p.x0 = ((s0 - (int64_t)C * kseg) % N + N) % N;
      p.st_lo = C * kseg; p.st_hi = (int)(C * kseg + len);
      segs->push_back(p);
    }
  }
  return true;
}

// Steps per launch of the fixed rule for segments of NT S sites: halos of a tenth on each side.
inline int segment_steps(int S, int NT, int C) { return std::max(1, (int)((int64_t)NT * S / (20 * C))); }

// Steps of every trial of the autotuner, whatever tiling a trial runs: one launch of whole
// lattices (kring steps, at most 500), so that launch edges weigh as in a run, and two at least
// of the longest segments (kseg steps) among the trials.
inline int64_t tuner_steps(int kring, int kseg) { return std::max<int64_t>(2LL * kseg, std::min(kring, 500)); }

// Pieces a block of the one-site-per-thread kernel holds at most (plan_blocked gives each
// at least its share of the block's threads).
constexpr int kBlockedPieces = 16;

// Pieces of every run for one site per thread: lattices of up to NT sites whole, longer
// ones in equal stretches with C k halo sites on each side.  Reservoir lattices cover the
// nodes [-C, N + C), their stretches' halos end there.  False if NT holds no stretch.
inline bool plan_blocked(const std::vector<int64_t>& Ns, bool reservoir, int C, int NT, int64_t k,
                         std::vector<Piece>* pieces) {
  pieces->clear();
  const int64_t ghost = reservoir ? C : 0;
  for (int32_t r = 0; r < (int32_t)Ns.size(); ++r) {
    const int64_t n = Ns[r] + 2 * ghost;
    if (n <= NT) {
      Piece p{};
      p.run = r; p.n = (int)n; p.x0 = -ghost; p.st_hi = (int)n;
      p.nthr = std::max(p.n, NT / kBlockedPieces);
      pieces->push_back(p);
      continue;
    }
    const int64_t h = C * k, room = NT - 2 * h;
    if (room <= 0) return false;
    const int64_t nseg = (n + room - 1) / room, len = (n + nseg - 1) / nseg;
    for (int64_t s0 = 0; s0 < n; s0 += len) {
      const int64_t s1 = std::min(s0 + len, n);
      const int64_t lo = reservoir ? std::max<int64_t>(s0 - h, 0) : s0 - h;
      const int64_t hi = reservoir ? std::min(s1 + h, n) : s1 + h;
      Piece p{};
      p.run = r; p.nthr = p.n = (int)(hi - lo);
      p.x0 = reservoir ? lo - ghost : (lo < 0 ? lo + n : lo);
      p.st_lo = (int)(s0 - lo); p.st_hi = (int)(s1 - lo);
      pieces->push_back(p);
    }
  }
  return true;
}

// Tiling of the one-site-per-thread kernel: NT threads per block, k steps per launch (k
// also bounds the halos; lattices that all fit a block need none and run kwhole steps per
// launch), spread: one piece per block instead of packed blocks.  us: the estimated time
// of a step, in microseconds.
struct BlockedTiling {
  int NT = 0, k = 0;
  bool spread = false;
  double us = 1e300;
};

// A model of a step's time in microseconds, fitted to GB300 timings of single lattices of
// 256 to 2^20 sites and of the 4096-lattice ensembles:
//   t0 + t1 max(w, wmin) + launch / k,
// w the warps an SM has to step, t1 the issue time of one, wmin one per scheduler (t0 + 4 t1
// is then the latency of a step: D1Q7 FP64 0.82 us, FP32 0.10 us; the FP64 collapse, in
// FP64 arithmetic, is bound by the FP64 pipe the schedulers share), launch the time
// between two launches' work (with several FP64 blocks an SM kMoreLaunch times as long: the
// last blocks of one launch end apart).
constexpr double kMoreLaunch = 2.4;
struct BlockedCost {
  double t0, t1, launch;
  int wmin, max_threads;
};
inline BlockedCost blocked_cost(int Q, bool f64, bool collapse) {
  BlockedCost c = collapse ? (f64 ? BlockedCost{0.10, 0.21, 3.2, 1, 512} : BlockedCost{0.10, 0.007, 3.2, 4, 512})
                           : (f64 ? BlockedCost{0.48, 0.086, 1.6, 4, 384} : BlockedCost{0.07, 0.0075, 1.6, 4, 512});
  if (Q == 5) {
    c.t0 *= f64 && !collapse ? 0.78 : 0.7;
    c.t1 *= f64 && !collapse ? 0.78 : 0.7;
  }
  return c;
}

// Lengths (plus `ghosts`) in decreasing order: all of up to 129, else the longest and 128 of the
// others, evenly by rank.
inline std::vector<int64_t> length_sample(const std::vector<int64_t>& Ns, int64_t ghosts) {
  std::vector<int64_t> n(Ns);
  const size_t others = n.size() - 1;
  const int64_t longest = *std::max_element(n.begin(), n.end());
  if (n.size() <= 129 || longest > 65536) {
    std::sort(n.begin(), n.end(), std::greater<int64_t>());
  } else {  // (by counting: sorting 4096 lengths took 0.08 ms of creating a handle)
    std::vector<int> count((size_t)longest + 1, 0);
    for (int64_t v : Ns) ++count[(size_t)v];
    size_t at = 0;
    for (int64_t v = longest; v >= 0; --v)
      for (int c = count[(size_t)v]; c > 0; --c) n[at++] = v;
  }
  if (n.size() > 129) {
    for (size_t q = 0; q < 128; ++q) n[1 + q] = n[1 + (2 * q + 1) * others / 256];
    n.resize(129);
  }
  for (int64_t& v : n) v += ghosts;
  return n;
}

// The cheapest tiling.  More steps per launch mean fewer launches and wider halos, which
// cost warps; smaller blocks spread a small workload over more SMs.  FP64 blocks of more
// than 128 threads step 8 to 20 % slower on a full device (their warps meet at the barrier
// and then want the same pipe).  Of a large batch the longest lattice, which decides whether all
// fit a block, and 128 of the others in order of length (so that the caller's order does not
// matter) are looked at.
inline BlockedTiling choose_blocked(const std::vector<int64_t>& Ns, bool reservoir, int Q, const BlockedCost& cost,
                                    int sms, int kwhole) {
  const int C = (Q - 1) / 2;
  const std::vector<int64_t> n = length_sample(Ns, reservoir ? 2 * C : 0);
  const double each = n.size() > 1 ? (double)(Ns.size() - 1) / (double)(n.size() - 1) : 0.0;  // of n[1], n[2], ...
  BlockedTiling best;
  for (int NT : {64, 96, 128, 192, 256, 384, 512}) {
    if (NT > cost.max_threads) break;
    for (int k : {2, 3, 4, 6, 8, 12, 16, 24, 32, 48}) {
      const int64_t h = (int64_t)C * k, room = NT - 2 * h;
      if (room <= 0) break;
      const bool whole = n[0] <= NT;
      double pieces = 0.0, small = 0.0;  // stretches and whole lattices; the latter's threads
      int64_t widest = 0;
      for (size_t r = 0; r < n.size(); ++r) {
        const double w = r ? each : 1.0;
        if (n[r] <= NT) {
          pieces += w;
          small += w * (double)std::max<int64_t>(n[r], NT / kBlockedPieces) / (0.93 * NT);
          widest = std::max(widest, n[r]);
        } else {
          const int64_t nseg = (n[r] + room - 1) / room;
          pieces += w * (double)nseg;
          small += w * (double)nseg;
          widest = std::max(widest, (n[r] + nseg - 1) / nseg + 2 * h);
        }
      }
      const double blocks = std::max(1.0, small);
      BlockedTiling b;
      b.NT = NT;
      b.k = whole ? kwhole : k;
      b.spread = pieces <= (double)sms;
      double w;  // warps per SM
      if (b.spread) {
        w = (double)((widest + 31) / 32);
      } else {
        const double per = blocks / sms;  // blocks per SM, whole blocks while few
        w = (per < 3.0 ? std::ceil(per) : per + 0.5) * NT / 32.0;
        if (cost.max_threads == 384 && NT > 128) w *= NT > 256 ? 1.2 : 1.08;
      }
      b.us = cost.t0 + cost.t1 * std::max<double>(w, cost.wmin) + cost.launch * (b.spread || cost.max_threads != 384 ? 1.0 : kMoreLaunch) / b.k;
      if (b.us < best.us) best = b;
      if (whole) break;
    }
  }
  return best;
}

// Indices 0..n-1 in decreasing order of k (k >= 0), equal keys in index order: the
// order of a stable sort, by counting (keys are thread counts, at most a few thousand).
inline std::vector<int> stable_desc(const std::vector<int>& k) {
  int kmax = 0;
  for (int v : k) kmax = std::max(kmax, v);
  std::vector<int> start((size_t)kmax + 2, 0);  // start[kmax - v]: first slot of key v
  for (int v : k) ++start[(size_t)(kmax - v) + 1];
  for (size_t q = 1; q < start.size(); ++q) start[q] += start[q - 1];
  std::vector<int> idx(k.size());
  for (size_t i = 0; i < k.size(); ++i) idx[(size_t)start[(size_t)(kmax - k[i])]++] = (int)i;
  return idx;
}

// Work groups of one lane during packing: first fit of pieces (threads nthr) into
// groups of `cap` threads.
struct Bins {
  int cap = 0;
  bool pair = false;  // pair work groups: block 0 is threads [0, cap/2), block 1 the rest
  // Members of each group in the order they joined it: a singly linked list over piece
  // indices (head, tail per group; nxt per piece), so that packing allocates nothing
  // per group.
  std::vector<int> head, tail, count, nxt;
  std::vector<int> used;   // threads [0, used) taken (pair work groups: the end of block 1's)
  std::vector<int> used0;  // pair work groups: threads [0, used0) of block 0 taken
  std::vector<int> key;    // queue order (largest first); empty: by occupied threads
  // Segment tree of the largest free run (block 0's or block 1's) over the groups, so
  // that first fit finds the first group with room in O(log groups).
  std::vector<int> tree;
  size_t tn = 0;

  size_t groups() const { return used.size(); }
  std::vector<int> members(size_t b) const {
    std::vector<int> m;
    for (int i = head[b]; i >= 0; i = nxt[(size_t)i]) m.push_back(i);
    return m;
  }
  void link(size_t b, int i) {
    if ((size_t)i >= nxt.size()) nxt.resize(std::max<size_t>((size_t)i + 1, 2 * nxt.size()), -1);
    nxt[(size_t)i] = -1;
    if (tail[b] < 0) head[b] = i;
    else nxt[(size_t)tail[b]] = i;
    tail[b] = i;
    ++count[b];
  }
  // A new, empty group with u0 threads of block 0 (pair groups) and threads [0, u)
  // (pair groups: block 1's up to u) taken.
  size_t new_group(int u0, int u) {
    head.push_back(-1);
    tail.push_back(-1);
    count.push_back(0);
    used.push_back(u);
    if (pair) used0.push_back(u0);
    return used.size() - 1;
  }
  int room(size_t b) const {
    int f = cap - used[b];
    if (pair) f = std::max(f, cap / 2 - used0[b]);
    return f;
  }
  void fix(size_t b) {
    if (b >= tn) {
      tn = std::max<size_t>(64, 2 * tn);
      while (tn <= b) tn *= 2;
      tree.assign(2 * tn, -1);
      for (size_t q = 0; q < used.size(); ++q) tree[tn + q] = room(q);
      for (size_t p = tn - 1; p >= 1; --p) tree[p] = std::max(tree[2 * p], tree[2 * p + 1]);
      return;
    }
    size_t p = tn + b;
    tree[p] = room(b);
    for (p >>= 1; p >= 1; p >>= 1) tree[p] = std::max(tree[2 * p], tree[2 * p + 1]);
  }
  // A new group holding pieces `mem`, with u0 and u as for new_group.
  void add(std::initializer_list<int> mem, int u0, int u) {
    const size_t b = new_group(u0, u);
    for (int i : mem) link(b, i);
    fix(b);
  }
  // The first group with `need` threads free; groups() if none has.
  size_t first_with(int need) const {
    if (tn == 0 || tree[1] < need) return groups();
    size_t p = 1;
    while (p < tn) p = tree[2 * p] >= need ? 2 * p : 2 * p + 1;
    return p - tn;
  }
  // First fit: the first group with room for the piece.  A piece never spans the
  // block edge of a pair work group here: it goes into block 0's free threads or
  // after block 1's taken ones.
  bool first_fit(std::vector<Piece>& pieces, int i) {
    const int need = pieces[i].nthr;
    const size_t b = first_with(need);
    if (b == groups()) return false;
    if (pair && used0[b] + need <= cap / 2) {
      pieces[i].t0 = used0[b];
      used0[b] += need;
    } else {
      pieces[i].t0 = used[b];
      used[b] += need;
    }
    link(b, i);
    fix(b);
    return true;
  }
  void open(std::vector<Piece>& pieces, int i) {
    pieces[i].t0 = 0;
    add({i}, 0, pieces[i].nthr);
  }
  // bundles in decreasing order of occupied threads (longest first)
  void emit(const std::vector<Piece>& pieces, std::vector<Piece>* ordered, std::vector<int2>* bundles) const {
    const std::vector<int> order = stable_desc(key.empty() ? used : key);
    ordered->clear();
    bundles->clear();
    ordered->reserve(pieces.size());
    bundles->reserve(order.size());
    for (int b : order) {
      bundles->push_back(int2{(int)ordered->size(), count[(size_t)b]});
      for (int i = head[(size_t)b]; i >= 0; i = nxt[(size_t)i]) ordered->push_back(pieces[(size_t)i]);
    }
  }
};

inline std::vector<int> by_threads_desc(const std::vector<Piece>& pieces) {
  std::vector<int> nthr(pieces.size());
  for (size_t i = 0; i < pieces.size(); ++i) nthr[i] = pieces[i].nthr;
  return stable_desc(nthr);
}

// ---- one site per thread over the blocks of a cluster: a lattice's sites lie on consecutive
// threads of the cluster's CL blocks of NT threads, cut into portions at block edges, with no
// halos (a portion's edge values go straight into the blocks that hold its neighbours).

// The fewest threads a portion takes: its two edges are apart, and a block holds at most
// kBlockedPieces portions.
inline int portion_min(int C, int NT) { return std::max(2 * C, NT / kBlockedPieces); }

// Places n sites on a cluster whose threads before pos are taken, in portions (pos, length)
// that each lie in one block; returns the position after them.
template <typename F>
inline int64_t place_portions(int64_t pos, int64_t n, int C, int NT, F portion) {
  const int64_t pmin = portion_min(C, NT);
  int64_t room = NT - pos % NT;
  if (std::max(n, pmin) > room && (room < 2 * pmin || n < 2 * pmin)) {  // no cut leaves two portions
    pos += room;
    room = NT;
  }
  for (;;) {
    int64_t len = std::min(n, room);
    if (n > len && n - len < pmin) len = n - pmin;
    portion(pos, len);
    n -= len;
    if (n == 0) return pos + std::max(len, pmin);
    pos += room;  // (shortened portions leave threads idle)
    room = NT;
  }
}

// Pieces (portions) and bundles (one per block, CL consecutive ones a cluster; possibly empty)
// of lattices packed first fit, longest first.  A piece's halo and pad_ say where its edge
// values go: block of the cluster << 16 | column of that block's exchange area, of the left
// neighbour's right guard and of the right neighbour's first site.  False if some lattice does
// not fit a cluster.
inline bool plan_clusters(const std::vector<int64_t>& Ns, bool reservoir, int C, int NT, int CL,
                          std::vector<Piece>* pieces, std::vector<int2>* bundles) {
  pieces->clear();
  bundles->clear();
  const int64_t ghost = reservoir ? C : 0, cap = (int64_t)CL * NT, pmin = portion_min(C, NT);
  std::vector<int> order(Ns.size());
  for (size_t r = 0; r < Ns.size(); ++r) order[r] = (int)r;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return Ns[(size_t)a] > Ns[(size_t)b]; });
  Bins cl;  // used: a cluster's threads before its free ones
  cl.cap = (int)cap;
  std::vector<int> in_block;                    // portions in the block that the last taken thread lies in
  std::vector<std::pair<int64_t, Piece>> held;  // (block, portion)
  const auto end = [&](int64_t pos, int64_t n) { return place_portions(pos, n, C, NT, [](int64_t, int64_t) {}); };
  for (int r : order) {
    const int64_t n = Ns[(size_t)r] + 2 * ghost;
    if (n > cap) return false;
    size_t b = cl.first_with((int)n);
    if (b < cl.groups() && end(cl.used[b], n) > cap) b = cl.first_with((int)(n + 2 * pmin));
    if (b == cl.groups() || end(cl.used[b], n) > cap) {
      if (end(0, n) > cap) return false;
      b = cl.new_group(0, 0);
      in_block.push_back(0);
    }
    const size_t from = held.size();
    int64_t x = -ghost, block = cl.used[b] > 0 ? (cl.used[b] - 1) / NT : 0;
    cl.used[b] = (int)place_portions(cl.used[b], n, C, NT, [&](int64_t pos, int64_t len) {
      if (pos / NT != block) in_block[b] = 0;
      block = pos / NT;
      Piece p{};
      p.run = r; p.t0 = (int)(pos % NT); p.n = (int)len; p.nthr = (int)std::max(len, pmin); p.x0 = x; p.st_hi = p.n;
      p.pad_ = (int)((block << 16) | (p.t0 + C * (2 * in_block[b] + 1)));  // (its own first column, for now)
      ++in_block[b];
      x += len;
      held.emplace_back((int64_t)b * CL + block, p);
    });
    const size_t m = held.size() - from;
    std::vector<int32_t> own(m);
    for (size_t q = 0; q < m; ++q) own[q] = held[from + q].second.pad_;
    for (size_t q = 0; q < m; ++q) {
      const size_t l = (q + m - 1) % m;
      held[from + q].second.halo = own[l] + held[from + l].second.n;
      held[from + q].second.pad_ = own[(q + 1) % m];
    }
    cl.fix(b);
  }
  std::stable_sort(held.begin(), held.end(), [](const auto& a, const auto& b) { return a.first < b.first; });
  bundles->assign(cl.groups() * (size_t)CL, int2{0, 0});
  for (const auto& [block, p] : held) {
    int2& bd = (*bundles)[(size_t)block];
    if (bd.y++ == 0) bd.x = (int)pieces->size();
    pieces->push_back(p);
  }
  return true;
}

struct ClusterTiling {
  int NT = 0, CL = 0;
  double us = 1e300;
};

// The cheapest cluster tiling for FP64 batches with lattices too long for a block.  No halos and
// no launch ends, but a cluster barrier per step: measured (GB300, D1Q7, 4 x 128 clusters that
// fill the device) 1.13, 1.46, 1.67, 2.16, 3.10 us per step with 1, 2, 3, 4 and 6 blocks an SM,
// t0 + t1 w for w warps.  A cluster's blocks lie in one GPC, of 18 or 20 SMs, so fewer clusters
// than SMs / CL have a block an SM each: of eight blocks 16 (17 step as slowly as 36 do, with two
// blocks on some SMs: 1.44 against 1.45 us), with two blocks an SM 36, with three 52.  Blocks
// beyond 768 threads an SM run all their steps after the others.  Blocks of 256 threads take 1.09
// times that, others but 128 1.1.  Of long lattices the packing may need a cluster more than
// counted here, and at such a line a whole round more, hence 2 % more.  The caller asks for 4 %
// less than the launches' estimate: of 680 random batches of 4 to 1400 lattices 102 take clusters,
// at 0.94 to 1.57 (eight below 1, mean 1.15) of the stretches' rate; front tests of 122 lattices
// D1Q7 2.83 -> 2.24 us per step, D1Q5 2.06 -> 1.71.
inline ClusterTiling choose_clusters(const std::vector<int64_t>& Ns, bool reservoir, int Q, int sms, int kwhole) {
  const double t0 = Q == 7 ? 0.68 : 0.63, t1 = Q == 7 ? 0.0975 : 0.071;
  const int C = (Q - 1) / 2;
  const std::vector<int64_t> n = length_sample(Ns, reservoir ? 2 * C : 0);
  const int64_t longest = n.front();
  ClusterTiling best;
  for (int CL : {2, 4, 8})
    for (int NT : {64, 96, 128, 192, 256, 384}) {
      const int64_t pmin = portion_min(C, NT), cap = (int64_t)CL * NT;
      if (longest <= NT || longest + 2 * pmin > cap || cap > 2048) continue;
      std::vector<int64_t> room;
      for (int64_t v : n) {
        size_t b = 0;
        while (b < room.size() && room[b] < v) ++b;
        if (b == room.size()) room.push_back(cap);
        room[b] -= std::max(v, pmin) + (v > NT ? pmin : pmin / 2);
      }
      const double clusters = 1.02 * (double)room.size() * (double)Ns.size() / (double)n.size();
      const auto hold = [&](int blocks) {  // clusters at once, with that many blocks an SM
        const int small = sms / 16 * 2, large = (sms - 8 * small) / 2;  // (eight GPCs; those of two SMs more)
        return (double)((8 - large) * (blocks * small / CL) + large * (blocks * (small + 2) / CL));
      };
      const int per = 768 / NT;
      const double full = std::floor(clusters / std::max(1.0, hold(per))), rest = clusters - full * hold(per);
      int blocks = 1;
      while (blocks < per && hold(blocks) < rest - 1e-9) ++blocks;
      const double slow = NT == 128 ? 1.0 : NT == 256 ? 1.09 : 1.1;
      const auto step = [&](int b) { return slow * (t0 + t1 * std::max(b * NT / 32.0, 4.0)); };
      const double us = full * step(per) + (rest > 1e-9 ? step(blocks) : 0.0) + 4.0 / kwhole;  // (a launch)
      if (us < best.us) best = ClusterTiling{NT, CL, us};
    }
  return best;
}

// Time of a step of the register-resident kernel (D1Q7, microseconds), S sites per thread
// and q warps on each of an SM's schedulers, measured on single lattices and on uniform
// batches that fill the device; 0: not a tiling that choose_resident considers.  Two blocks
// of 128 threads overlap one's barrier with the other's step (1.11e12 and 1.13e12
// site-updates/s at 18 and 16 sites, 1.10e12 at 16 x 256, 0.94e12 at 20 x 256).  pairs: the
// cluster kernel, whose 16-site loop is scheduled worse, with the halves' exchanges.
inline double resident_step_us(int S, int NT, int q, bool pairs) {
  if (pairs && q == 2) return (NT < 256 ? 1.2 : 1.0) * (S == 20 ? 0.866 : S == 18 ? 0.80 : S == 16 ? 0.756 : 0.9);
  if (NT == 128 && q == 2 && (S == 18 || S == 16)) return S == 18 ? 0.629 : 0.549;
  const auto at = [q](double first, double more) { return first + more * (q - 1); };
  switch (S) {
    case 20: return at(0.48, 0.35);
    case 18: return at(0.385, 0.32);
    case 16: return at(0.345, 0.225);
    case 8: return at(0.285, 0.165);
    case 6: return at(0.26, 0.105);
    case 4: return at(0.235, 0.09);
    default: return 0.0;
  }
}

// Tiling of the register-resident kernel for FP32 and scaled FP16 storage.  spread: one
// lattice per block instead of packed ones; kseg: steps per launch of segments (0: the
// fixed rule's); us: the estimated time of a step.
struct ResidentTiling {
  int S = 0, NT = 0, kseg = 0;
  bool spread = false;
  double us = 1e300;
};

// (D1Q5: 0.7 of these times at 20 sites, 0.84 at fewer.)
// The estimate for one tiling of which `bps` blocks fit an SM: blocks run in rounds of
// sms bps, each as long as a full SM's step, so a batch of 1.7 rounds takes as long as
// one of 2, and smaller blocks that need 2 shorter rounds are faster; a batch of less
// than a round runs as fast as its fullest SM.  Segments (FP32 alone: scaled FP16 rounds at
// launch edges, so its launches stay as they are): each launch adds `edge` microseconds per
// round for loads and stores (measured on a 2^24-site lattice), and halos of c_max kseg
// sites; kseg is the cheapest, or kfix.
inline ResidentTiling rate_resident(const std::vector<int64_t>& Ns, int Q, int S, int NT, int bps, int sms, bool f16,
                                    int kmax, bool may_spread, int kfix = 0) {
  const double edge = S == 18 ? 14.5 : 20.0;
  constexpr double kLaunchUs = 3.0, kRingCost = 1.4, kRingUs = 0.4;
  const int C = (Q - 1) / 2, h = C * kPairStepsMax;
  const double scale = Q == 7 ? 1.0 : (S == 20 ? 0.7 : 0.84);
  ResidentTiling t;
  t.S = S;
  t.NT = NT;
  const size_t stride = (Ns.size() + 127) / 128;  // a sample of a large batch is packed
  std::vector<int> threads;  // of the sample's whole lattices and halves
  double all = 0.0, sampled = 0.0;  // their sum over the batch and the sample
  int64_t whole = 0, halves = 0, rings = 0;
  std::vector<int64_t> cut;
  for (size_t r = 0; r < Ns.size(); ++r) {
    int64_t v = (Ns[r] + S - 1) / S;  // (copies of lattices that do not split into S and S - 1, as in plan_pieces)
    for (int64_t n = Ns[r]; n <= v * (S - 1) && v <= 2 * NT;) {
      n += Ns[r];
      v = (n + S - 1) / S;
    }
    const int64_t half = ((Ns[r] + 1) / 2 + 2 * h + S - 1) / S + 1;
    const bool in = r % stride == 0;
    if (v <= NT || half <= NT) {
      const int held = (int)(v <= NT ? v : half), n = v <= NT ? 1 : 2;
      all += (double)held * n;
      whole += n;
      halves += n == 2 ? 2 : 0;
      if (in) {
        threads.insert(threads.end(), (size_t)n, held);
        sampled += (double)held * n;
      }
    } else if (v <= 2 * NT) {  // one ring across a pair waits on the other block every step
      if (!kfix) return t;     // (the fixed tiling's estimate is still wanted)
      ++rings;
    } else {
      cut.push_back(Ns[r]);
    }
  }
  const bool pairs = halves + rings > 0;
  if (pairs && S <= 8 && !kfix) return t;  // (the cluster kernel's time with these is 1.8 times a block's)
  const double pieces = (double)(whole + rings);
  // first fit, largest first: the blocks they fill
  std::sort(threads.begin(), threads.end(), std::greater<int>());
  const int64_t widest = pairs ? NT : (threads.empty() ? 0 : threads.front());
  std::vector<int> room;
  for (int v : threads) {
    size_t b = 0;
    while (b < room.size() && room[b] < v) ++b;
    if (b == room.size()) room.push_back(NT);
    room[b] -= v;
  }
  double blocks = (double)room.size();
  if (stride > 1 && !room.empty()) {  // as full as the sample's, without its emptiest
    const double most = *std::max_element(room.begin(), room.end());
    const double n = (double)room.size(), fill = n > 1.0 ? (sampled - (NT - most)) / (n - 1.0) : (double)NT;
    blocks = all / fill;
  }
  blocks += 2.0 * kRingCost * (double)rings;
  const double slots = (double)sms * bps;
  const auto warps = [&](double per_sm, int64_t threads) {  // per scheduler: a block's first warp is the first's
    return (int)std::ceil(per_sm - 1e-9) * (int)((threads + 127) / 128);
  };
  double us = rings ? kRingUs : 0.0;
  if (pieces > 0.0) {
    t.spread = may_spread && !pairs && cut.empty() && pieces <= slots;
    if (t.spread) {
      us = scale * resident_step_us(S, NT, warps(std::ceil(pieces / sms), widest), false);
    } else {
      const double rounds = std::ceil(blocks / slots);
      us = scale * rounds * resident_step_us(S, NT, warps(std::min<double>(bps, std::ceil(blocks / sms)), NT), pairs);
    }
  }
  if (!cut.empty()) {
    if (f16) return t;
    const double full = scale * resident_step_us(S, NT, warps(bps, NT), false);
    double best = 1e300;
    for (int k = kfix ? kfix : 16; k <= std::min(kmax, 192); k += 8) {
      const int64_t room = (int64_t)NT * S - 2LL * C * k - 2 * S;
      if (room <= 0) break;
      double n = 0.0;
      for (int64_t N : cut) n += (double)((N + room - 1) / room);
      const double rounds = std::ceil(n / slots);
      const double c = rounds * (full + edge / k) + kLaunchUs / k;
      if (c < best) { best = c; t.kseg = k; }
      if (kfix) break;
    }
    us += best;
  }
  t.us = us;
  return t;
}

// The register-resident tiling of a batch.  The fixed tiling (20 sites x 256 threads,
// lattices packed) stays unless another is estimated at least 8 % faster, about the
// estimate's error on large ensembles; S = 0: it stays.  us is the chosen one's estimate.
// smem(S, NT): shared memory of a block.
template <typename F>
ResidentTiling choose_resident(const std::vector<int64_t>& Ns, int Q, bool f16, int sms, int kmax, F smem) {
  const auto fit = [&](int S, int NT) {  // blocks per SM by registers (255 a thread above 8 sites) and shared memory
    const int threads = S <= 8 ? 512 : 256;
    return std::max(1, std::min(threads / NT, (int)(228 * 1024 / (smem(S, NT) + 1024))));
  };
  const ResidentTiling fixed =
      rate_resident(Ns, Q, 20, 256, 1, sms, f16, kmax, false, std::min(kmax, 5120 / (10 * (Q - 1))));
  ResidentTiling best;
  best.us = fixed.us;
  int64_t sites = 0, longest = 0;
  for (int64_t n : Ns) { sites += n; longest = std::max(longest, n); }
  // more than six rounds: little to gain from their number, only from two blocks an SM
  if (longest > 2304 && longest <= 10240 && sites > 6LL * 5120 * sms) return best;
  if (f16 && fixed.us > 1e290) return best;  // segments: their launches round
  for (const auto& c : {std::pair<int, int>{20, 256}, {18, 256}, {16, 256}, {18, 128}, {16, 128}, {8, 512}, {8, 256},
                        {6, 512}, {6, 256}, {4, 512}, {4, 256}, {4, 128}}) {
    const ResidentTiling t = rate_resident(Ns, Q, c.first, c.second, fit(c.first, c.second), sms, f16, kmax, true);
    if (t.us < 0.92 * fixed.us && t.us < best.us) best = t;
  }
  return best;
}

// The register-resident tau = 1 collapse's tiling (FP32).  Step times by blocks per SM, measured
// (GB300, D1Q7 without the terms that add zero; other runs scale them together): 32 sites x 256
// threads 0.865 with one and 1.59 us with two, 32 x 384 1.25, 16 x 384 0.68, 16 x 256 0.51,
// 8 x 384 0.41.  Lattices shorter than S (S - 1) are held as copies, so
// short ones want few sites per thread; a batch of 1.1 to 1.4 rounds of 8192 sites wants
// 32 x 384 (700 lattices of 256 to 8192 sites: 1.59 -> 1.26 us), one of 0.3 rounds 8 x 384 (101
// lattices of 1504 to 3031 sites: 0.86 -> 0.41 us).  32 x 256 stays unless another
// is estimated 8 % faster.  us is the chosen one's estimate.
inline ResidentTiling choose_collapse(const std::vector<int64_t>& Ns, int sms) {
  struct Cost { int S, NT; double first, more; };  // us with one block an SM, and for each further one
  ResidentTiling best;
  const size_t stride = (Ns.size() + 255) / 256;
  for (const Cost c : {Cost{32, 256, 0.865, 0.725}, Cost{32, 384, 1.25, 1.25}, Cost{16, 384, 0.69, 0.69},
                       Cost{16, 256, 0.51, 0.51}, Cost{8, 384, 0.41, 0.41}}) {
    std::vector<int> threads;
    double all = 0.0, sampled = 0.0;
    bool whole = true;
    for (size_t r = 0; r < Ns.size() && whole; ++r) {
      int64_t v = (Ns[r] + c.S - 1) / c.S;
      for (int64_t n = Ns[r]; n <= v * (c.S - 1) && v <= c.NT;) {
        n += Ns[r];
        v = (n + c.S - 1) / c.S;
      }
      whole = v <= c.NT;
      all += (double)v;
      if (r % stride == 0) {
        threads.push_back((int)v);
        sampled += (double)v;
      }
    }
    if (!whole) continue;
    std::sort(threads.begin(), threads.end(), std::greater<int>());
    std::vector<int> room;
    for (int v : threads) {
      size_t b = 0;
      while (b < room.size() && room[b] < v) ++b;
      if (b == room.size()) room.push_back(c.NT);
      room[b] -= v;
    }
    double blocks = (double)room.size();
    if (stride > 1) {  // as full as the sample's, without its emptiest; 2 % for what it misses
      const double most = *std::max_element(room.begin(), room.end());
      blocks = 1.02 * all / (blocks > 1.0 ? (sampled - (c.NT - most)) / (blocks - 1.0) : (double)c.NT);
    }
    const double us = c.first + c.more * (std::max(1.0, std::ceil(blocks / sms - 1e-9)) - 1.0);
    if (best.S == 0 || us < std::min(best.us, best.S == 32 && best.NT == 256 ? 0.92 * best.us : best.us)) {
      best.S = c.S;
      best.NT = c.NT;
      best.us = us;
    }
  }
  return best;
}

// First-fit decreasing packing of whole lattices: a lattice held as two halves opens a
// cluster pair (one half at the start of each block), one longer than one block (more
// than NT threads) opens a pair as a ring across both blocks; the others fill the
// pairs' spare threads first, then blocks of NT threads.
// (spread: these open a block each).
inline void pack_rings(std::vector<Piece>& pieces, int NT, Bins* blocks, Bins* pairs, bool spread = false) {
  blocks->cap = NT;
  pairs->cap = 2 * NT;
  pairs->pair = true;
  for (size_t i = 0; i + 1 < pieces.size(); ++i) {
    if (pieces[i].halo == 0) continue;
    pieces[i].t0 = 0;
    pieces[i + 1].t0 = NT;
    pairs->add({(int)i, (int)i + 1}, pieces[i].nthr, NT + pieces[i + 1].nthr);
    ++i;
  }
  for (int i : by_threads_desc(pieces)) {
    if (pieces[i].halo > 0) continue;
    if (pieces[i].nthr > NT) {
      pieces[i].t0 = 0;
      pairs->add({i}, NT, pieces[i].nthr);
    } else if (spread || (!pairs->first_fit(pieces, i) && !blocks->first_fit(pieces, i))) {
      blocks->open(pieces, i);
    }
  }
  pairs->key.resize(pairs->used.size());
  for (size_t b = 0; b < pairs->used.size(); ++b) pairs->key[b] = pairs->used0[b] + pairs->used[b] - NT;
}

// One queue for every whole lattice: the single-block bundles go two to a cluster
// pair (the second one's pieces shifted by NT threads, so no piece spans the block
// edge and its blocks never wait on each other), queued after the pair bundles whose
// piece spans the edge; within each kind, largest first.
// (Groups appended here take no further pieces.)
inline void merge_blocks_into_pairs(std::vector<Piece>& pieces, int NT, const Bins& blocks, Bins* pairs) {
  pairs->cap = 2 * NT;
  for (size_t b = 0; b < pairs->key.size(); ++b) pairs->key[b] += 4 * NT;
  const std::vector<int> order = stable_desc(blocks.used);
  for (size_t q = 0; q < order.size(); q += 2) {
    const size_t a = (size_t)order[q];
    const size_t g = pairs->new_group(blocks.used[a], q + 1 < order.size() ? NT + blocks.used[(size_t)order[q + 1]]
                                                                           : blocks.used[a]);
    for (int i = blocks.head[a]; i >= 0; i = blocks.nxt[(size_t)i]) pairs->link(g, i);
    if (q + 1 < order.size()) {
      const size_t c = (size_t)order[q + 1];
      for (int i = blocks.head[c]; i >= 0; i = blocks.nxt[(size_t)i]) {
        pieces[(size_t)i].t0 += NT;
        pairs->link(g, i);
      }
    }
    pairs->key.push_back(blocks.used[a]);  // the fuller of the two blocks
  }
}

inline void pack_blocks(std::vector<Piece>& pieces, int NT, Bins* blocks) {
  blocks->cap = NT;
  for (int i : by_threads_desc(pieces))
    if (!blocks->first_fit(pieces, i)) blocks->open(pieces, i);
}

// Bundles of the one-site-per-thread kernel: each stretch of a longer lattice has a block of
// its own (stretches of a lattice are equally long and fill most of it); whole lattices
// too when spread, else packed first fit after them.  `pieces` is put in bundle order;
// `bundles` is left empty when every piece is a bundle of its own.
inline void blocked_bundles(std::vector<Piece>& pieces, int NT, bool spread, std::vector<int2>* bundles) {
  bundles->clear();
  const auto whole = [](const Piece& p) { return p.st_lo == 0 && p.st_hi == p.n; };
  if (spread || std::none_of(pieces.begin(), pieces.end(), whole)) return;
  std::vector<Piece> small, packed;
  std::vector<int2> more;
  size_t n = 0;
  for (const Piece& p : pieces) {
    if (whole(p)) small.push_back(p);
    else pieces[n++] = p;
  }
  Bins bins;
  pack_blocks(small, NT, &bins);
  bins.emit(small, &packed, &more);
  for (size_t b = 0; b < n; ++b) bundles->push_back(int2{(int)b, 1});
  for (int2 b : more) bundles->push_back(int2{b.x + (int)n, b.y});
  std::copy(packed.begin(), packed.end(), pieces.begin() + (int64_t)n);
}

}  // namespace plan
}  // namespace lbks
