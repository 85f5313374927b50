// Host check of csrc/tri_batch_plan.h: every unit of every row of every system in exactly
// one segment, target-side slots of a row numbered from nb on without a gap, and no segment
// far above its share. Prints "ok <plans>" or the first fault.
#include <cstdio>
#include <set>
#include <tuple>

#include "tri_batch_plan.h"

using namespace nbody;

static bool check(const std::vector<TriBatchSystem> &sys, int ctas) {
  const TriBatchPlan p = tri_batch_plan(sys, ctas);
  if (p.row_base.size() != sys.size()) return false;
  std::set<std::tuple<int64_t, int, int>> seen, slots;
  int64_t units = 0, rows = 0, longest = 0;
  for (const auto &s : sys) {
    const int h = tri_batch_h(s.law), nb = (s.n + 64 * h - 1) / (64 * h), ng = (s.n + 31) / 32;
    for (int b = 0; b < nb; ++b) units += ng - 2 * h * b;
    rows += nb;
  }
  for (const TriSeg &g : p.segs) {
    const int h = tri_batch_h(g.law), nb = (g.n + 64 * h - 1) / (64 * h), ng = (g.n + 31) / 32;
    const int base = 2 * h * g.row;
    if (g.row >= nb || g.slot < nb || g.slot >= p.slots) return false;
    if (!slots.insert({g.first, g.row, g.slot - nb}).second) return false;
    for (int q = base + g.d0; q < base + g.d1; ++q)
      if (q >= base + 2 * h || q >= ng || !seen.insert({g.first, g.row, q}).second) return false;
    for (int q = base + 2 * h + g.o0; q < base + 2 * h + g.o1; ++q)
      if (q >= ng || !seen.insert({g.first, g.row, q}).second) return false;
    longest = std::max<int64_t>(longest, g.d1 - g.d0 + g.o1 - g.o0);
    if (g.d1 - g.d0 + g.o1 - g.o0 < 1) return false;
  }
  if (int64_t(seen.size()) != units || int64_t(p.row_shares.size()) != rows) return false;
  for (size_t k = 0; k < sys.size(); ++k) {
    const int h = tri_batch_h(sys[k].law), nb = (sys[k].n + 64 * h - 1) / (64 * h);
    for (int b = 0; b < nb; ++b)
      for (int j = 0; j < p.row_shares[p.row_base[k] + b]; ++j)
        if (!slots.erase({sys[k].first, b, j})) return false;
  }
  // no segment far above a piece: own units cost 3/4, so 4/3 of it, and the roundings
  const int64_t total = units * 108 + rows * kTriBatchRow;
  const int64_t piece = std::max(std::min(kTriBatchLeast, total / ctas + 1),
                                 total / (int64_t(ctas) * kTriBatchPieces));
  return slots.empty() && longest <= 4 * piece / (3 * 75) + 3;
}

int main() {
  int plans = 0;
  unsigned r = 1;
  for (int sizes : {1, 40, 300, 700, 2000, 5000})
    for (int nsys : {1, 2, 7, 60})
      for (int want : {1, 3, 152, 304}) {
        std::vector<TriBatchSystem> sys;
        int64_t at = 5;
        for (int k = 0; k < nsys; ++k) {
          r = r * 1664525u + 1013904223u;
          const int n = 1 + int((r >> 8) % unsigned(sizes));
          sys.push_back(TriBatchSystem{at, n, int((r >> 5) % 3), 0.0f});
          at += n + (k & 1);
        }
        if (!check(sys, want)) {
          std::printf("fault: sizes to %d, %d systems, %d shares\n", sizes, nsys, want);
          return 1;
        }
        ++plans;
      }
  std::printf("ok %d\n", plans);
  return 0;
}
