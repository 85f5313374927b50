// tri_batch_plan.h -- how the streamed triangle kernel of batched ensembles
// (tri_batch.cuh) cuts the pairs of many independent systems into segments that its CTAs
// take from a queue. Host only, plain C++ (planning, tests).
//
// Each system is cut into rows and units as in tri_plan.h, with the row length of its
// law. A row whose cost is above 1/kTriBatchPieces of a CTA's mean is cut into equal
// segments; all segments are queued, dearest first. A segment adds its source-side sums
// to slot `row` and its target-side sums to slot nb + (its number in its row).
#pragma once

#include <algorithm>
#include <cstdint>
#include <utility>
#include <vector>

#include "tri_plan.h"

namespace nbody {

// Register groups per thread (rows of 64 h targets), gravity and LJC: 512 systems of 64 to
// 4096 particles take 404 us an evaluation with 6 and 4, 408 with 8 and 4, 412 with 4 and
// 4, 424 with 8 and 6, 437 with 4 and 6.
constexpr int kTriBatchGrav = 6, kTriBatchLjc = 4;

struct TriSeg {
  int first;           // the system's first particle
  int n;               // its particles
  int law;
  float eps2;
  int row;
  int d0, d1, o0, o1;  // own groups and groups beyond the row (tri_run)
  int slot;            // target-side slot
};

struct TriBatchSystem {
  int64_t first;
  int n;
  int law;
  float eps2;
};

inline int tri_batch_h(int law) { return law == 0 ? kTriBatchGrav : kTriBatchLjc; }
// Costs, in hundredths of a gravity unit beyond a row: a unit beyond the row, an own unit
// (one-sided, tri_kernel.cuh), and a row's start and end.
inline int64_t tri_batch_unit(int law) { return law == 0 ? 100 : law == 1 ? 104 : 108; }
inline int64_t tri_batch_own(int law, int64_t count) { return count * tri_batch_unit(law) * 3 / 4; }
constexpr int64_t kTriBatchRow = 50;
// Segments per CTA's mean cost. The older of an SM's two CTAs gets four fifths of it, so
// that equal static shares end 300 to 460 us after the start; and with long segments the
// last of them. The same ensemble, us, for 4 / 6 / 8 / 12 / 16: 406, 404, 404, 407, 412
// (each segment loads and stores its row's targets again). In small ensembles not below
// kTriBatchLeast, as far as every CTA still gets one: us a step for 1, 400, 800, 1600 with
// 32 systems to 4096: 60.1, 46.0, 42.2, 53.6; 128 to 2048: 54.7, 46.5, 43.7, 52.5; 300 to
// 700: 38.6, 30.0, 31.7, 32.8.
constexpr int kTriBatchPieces = 8;
constexpr int64_t kTriBatchLeast = 800;

struct TriBatchPlan {
  std::vector<TriSeg> segs;     // dearest first
  std::vector<int> row_shares;  // segments of each row, system after system
  std::vector<int> row_base;    // a system's first row there
  int64_t slots = 1;            // most slots of a system
};

inline TriBatchPlan tri_batch_plan(const std::vector<TriBatchSystem> &sys, int ctas) {
  TriBatchPlan out;
  auto geom = [](const TriBatchSystem &s) {
    TriGeom g{};
    g.n = s.n;
    g.h = tri_batch_h(s.law);
    g.nb = int((int64_t(s.n) + 64 * g.h - 1) / (64 * g.h));
    g.ng = int((int64_t(s.n) + kTriGroup - 1) / kTriGroup);
    return g;
  };
  // cost of units p .. stop-1 of row b
  auto cost = [](const TriBatchSystem &s, const TriGeom &g, int b, int p, int stop) {
    const int d0 = tri_own(g, b, p), d1 = tri_own(g, b, stop);
    return kTriBatchRow + tri_batch_own(s.law, d1 - d0) +
           int64_t(stop - p - (d1 - d0)) * tri_batch_unit(s.law);
  };
  int64_t total = 0;
  for (const auto &s : sys) {
    const TriGeom g = geom(s);
    for (int b = 0; b < g.nb; ++b) total += cost(s, g, b, 0, tri_row_units(g, b));
  }
  const int64_t most = std::max(std::min(kTriBatchLeast, total / ctas + 1),
                                total / (int64_t(ctas) * kTriBatchPieces));
  std::vector<std::pair<int64_t, TriSeg>> all;
  for (const auto &s : sys) {
    const TriGeom g = geom(s);
    out.row_base.push_back(int(out.row_shares.size()));
    int max_k = 0;
    for (int b = 0; b < g.nb; ++b) {
      const int len = tri_row_units(g, b);
      const int k = int(std::min<int64_t>(len, (cost(s, g, b, 0, len) + most - 1) / most));
      for (int j = 0; j < k; ++j) {
        const int p = int(int64_t(len) * j / k), stop = int(int64_t(len) * (j + 1) / k);
        const int d0 = tri_own(g, b, p), d1 = tri_own(g, b, stop);
        all.emplace_back(cost(s, g, b, p, stop),
                         TriSeg{int(s.first), s.n, s.law, s.eps2, b, d0, d1, p - d0, stop - d1,
                                g.nb + j});
      }
      out.row_shares.push_back(k);
      max_k = std::max(max_k, k);
    }
    out.slots = std::max<int64_t>(out.slots, int64_t(g.nb) + max_k);
  }
  std::stable_sort(all.begin(), all.end(),
                   [](const auto &a, const auto &b) { return a.first > b.first; });
  for (const auto &c : all) out.segs.push_back(c.second);
  return out;
}

}  // namespace nbody
