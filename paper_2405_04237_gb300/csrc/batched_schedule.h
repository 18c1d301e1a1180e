// The static schedule of the persistent batched launch (k_batched.cu): which
// group of CTAs factors which matrices, from their sizes alone.
#pragma once
#include <stdint.h>

#include <algorithm>
#include <utility>
#include <vector>

namespace cqr {

// Groups of the launch: level l cuts the N CTAs into cnt[l] groups of equal
// size (to within one), group g = CTAs [g N / cnt, (g + 1) N / cnt).  Every
// CTA walks the levels in order; the groups of a level lie inside those of
// the level before.
constexpr int kBLevels = 12;  // 1, 2, 4, .. and N itself: grids of up to 1024 CTAs
struct BLevels {
  int n;
  int cnt[kBLevels];
  int off[kBLevels];   // node of the level's group 0 (node = entry of gstart, barrier counter)
};

// Rough device time of one matrix on a group of G CTAs (for the static
// schedule), fitted to homogeneous batches (500 to 200000 rows, n = 16 to
// 128, G = 1 to 152) to within 10 %: per row the multiply-adds at an SM's
// FP64 rate and the staging of each pass, per pass the barrier, the in-CTA
// sums and the solve's chain, per CholeskyQR the factorisation.
inline double est_seconds(int64_t m, int n, int b, int G) {
  const double k = n / b, rows = (double)m / G;
  const double row = 4.0 * n * n / 8.28e9 + n * (3.0 + 2.4 * k) * 1e-9;
  const double pass = 13e-6 + 0.35e-6 * b, chol = 0.6e-6 * b * (1.0 + b / 128.0);
  return rows * row + (4.0 * k - 1.0) * pass + 2.0 * k * chol;
}

// The static schedule: matrices (order) of every node, and its estimated time.
struct BSchedule {
  BLevels lev;
  int nodes;
  double seconds;
  std::vector<int> order, gstart;
};

inline void finish(BSchedule& S, const std::vector<std::vector<int>>& lists) {
  S.nodes = (int)lists.size();
  for (const auto& l : lists) {
    S.gstart.push_back((int)S.order.size());
    S.order.insert(S.order.end(), l.begin(), l.end());
  }
  S.gstart.push_back((int)S.order.size());
}

// Equal groups of G CTAs: largest estimated time first, each to the group
// with the least work so far.
inline BSchedule schedule_uniform(int batch, const int64_t* m, const int64_t* n, const int* b, int grid, int G) {
  BSchedule S{};
  const int groups = grid / G;
  S.lev.n = 1;
  S.lev.cnt[0] = groups;
  std::vector<std::pair<double, int>> by;
  for (int i = 0; i < batch; ++i) by.push_back({est_seconds(m[i], (int)n[i], b[i], G), i});
  std::stable_sort(by.begin(), by.end(),
                   [](const std::pair<double, int>& x, const std::pair<double, int>& y) { return x.first > y.first; });
  std::vector<double> load((size_t)groups, 0.0);
  std::vector<std::vector<int>> lists((size_t)groups);
  for (const auto& e : by) {
    int g = 0;
    for (int h = 1; h < groups; ++h)
      if (load[h] < load[g]) g = h;
    load[g] += e.first;
    lists[g].push_back(e.second);
  }
  S.seconds = *std::max_element(load.begin(), load.end());
  finish(S, lists);
  return S;
}

// The tree schedule.  A CTA's finishing time is the sum of the loads of the
// nodes it belongs to (the members of a node arrive together, so nobody
// waits).  For a bound on that time, the matrices are placed by decreasing
// work, each on the smallest groups that keep the bound (fewer CTAs waste
// less on barriers and sums), there on the least loaded one.  The bounds
// tried grow from the largest of the mean work per CTA and the longest
// matrix on the whole grid; on a bound that cannot be kept the next is
// tried, and the last takes the best place for every matrix.
inline BSchedule schedule_tree(int batch, const int64_t* m, const int64_t* n, const int* b, int grid) {
  BSchedule S{};
  BLevels& L = S.lev;
  int nodes = 0;
  for (int c = 1;; c *= 2) {
    const bool last = c >= grid || L.n == kBLevels - 1;
    L.cnt[L.n] = last ? grid : c;
    L.off[L.n] = nodes;
    nodes += L.cnt[L.n++];
    if (last) break;
  }
  auto lo_of = [&](int l, int g) { return (int)((int64_t)g * grid / L.cnt[l]); };
  // estimated times per matrix and level (the level's smallest group)
  std::vector<double> est((size_t)batch * L.n);
  std::vector<int> by((size_t)batch);
  double mean = 0.0, longest = 0.0;
  for (int i = 0; i < batch; ++i) {
    by[i] = i;
    double best = 0.0;
    for (int l = 0; l < L.n; ++l) {
      const double t = est[(size_t)i * L.n + l] = est_seconds(m[i], (int)n[i], b[i], grid / L.cnt[l]);
      if (l == 0 || t < best) best = t;
    }
    mean += est[(size_t)i * L.n + L.n - 1] / grid;
    longest = std::max(longest, best);
  }
  std::stable_sort(by.begin(), by.end(), [&](int x, int y) {
    return est[(size_t)x * L.n + L.n - 1] > est[(size_t)y * L.n + L.n - 1];
  });
  std::vector<double> cta((size_t)grid);     // load of each CTA
  std::vector<double> peak((size_t)nodes);   // largest load of the node's CTAs
  std::vector<int> place((size_t)batch);
  double bound = std::max(mean, longest);
  for (int attempt = 0;; ++attempt, bound *= 1.04) {
    const bool last = attempt == 20;
    std::fill(cta.begin(), cta.end(), 0.0);
    std::fill(peak.begin(), peak.end(), 0.0);
    bool ok = true;
    for (int q = 0; q < batch && ok; ++q) {
      const int i = by[q];
      int pl = -1, pg = -1;
      double at = 0.0;
      for (int l = L.n - 1; l >= 0 && pl < 0; --l) {
        int g = 0;
        for (int h = 1; h < L.cnt[l]; ++h)
          if (peak[L.off[l] + h] < peak[L.off[l] + g]) g = h;
        at = peak[L.off[l] + g] + est[(size_t)i * L.n + l];
        if (at <= bound) {
          pl = l;
          pg = g;
        }
      }
      if (pl < 0 && last) {
        for (int l = 0; l < L.n; ++l) {
          int g = 0;
          for (int h = 1; h < L.cnt[l]; ++h)
            if (peak[L.off[l] + h] < peak[L.off[l] + g]) g = h;
          const double t = peak[L.off[l] + g] + est[(size_t)i * L.n + l];
          if (pl < 0 || t < at) {
            at = t;
            pl = l;
            pg = g;
          }
        }
      }
      if (pl < 0) {
        ok = false;
        break;
      }
      place[i] = L.off[pl] + pg;
      // the node's CTAs wait for the slowest of them, then run the matrix
      const int c0 = lo_of(pl, pg), c1 = lo_of(pl, pg + 1);
      for (int c = c0; c < c1; ++c) cta[c] += est[(size_t)i * L.n + pl];
      for (int l = 0; l < L.n; ++l) {
        const int g0 = ((c0 + 1) * L.cnt[l] - 1) / grid, g1 = (c1 * L.cnt[l] - 1) / grid;
        for (int g = g0; g <= g1; ++g) {
          double v = 0.0;
          for (int c = lo_of(l, g); c < lo_of(l, g + 1); ++c) v = std::max(v, cta[c]);
          peak[L.off[l] + g] = v;
        }
      }
    }
    if (ok) break;
  }
  std::vector<std::vector<int>> lists((size_t)nodes);
  for (int i : by) lists[place[i]].push_back(i);
  S.seconds = *std::max_element(cta.begin(), cta.end());
  finish(S, lists);
  return S;
}

// CTAs of the equal groups the default considers: the largest divisor of the
// grid up to 8.
inline int default_group(int grid) {
  int G = 8;
  while (grid % G) --G;
  return G;
}

// The default: of the tree and equal groups the one with the shorter estimated
// time.  The tree's groups have 152, 76, 38, 19, 9 or 10, ... CTAs, so it
// cannot give 19, 38, 57, ... equal matrices eight CTAs each: 19 of 20000 x 128
// (b = 32) take 25.9 ms on the tree and 23.8 on groups of 8, 38 of 100000 x 64
// 72.9 and 62.7, 512 of 20000 x 128 658 and 646; one takes 1.75 and 23.5, 32
// take 42.3 and 47.6.  Over 126 batches of equal matrices (1 to 512 of 300 x 16
// to 100000 x 64) the estimates pick the faster one, but for batches under 0.3
// ms, where the tree may be taken although groups of 8 gain up to 35 us.
inline BSchedule schedule_default(int batch, const int64_t* m, const int64_t* n, const int* b, int grid) {
  BSchedule T = schedule_tree(batch, m, n, b, grid);
  BSchedule U = schedule_uniform(batch, m, n, b, grid, default_group(grid));
  return U.seconds < T.seconds ? U : T;
}

}  // namespace cqr
