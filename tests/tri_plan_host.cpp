// Host check of csrc/tri_plan.h: every unit of every row in exactly one share, found by
// walking the shares as the kernel does, and the shares that the finalize kernel counts
// for a row those that own units of it. Prints "ok <plans>" or the first fault.
#include <cstdio>
#include <set>

#include "tri_plan.h"

using namespace nbody;

static bool check(int n, int h, int want) {
  const TriGeom t = tri_geom(n, h, want);
  std::set<long long> seen;
  long long units = 0;
  for (int b = 0; b < t.nb; ++b) units += tri_row_units(t, b);
  for (int c = 0; c < t.nshare; ++c) {
    int b, p, b1, p1;
    tri_locate(t, tri_share_start(t, c), b, p);
    tri_locate(t, tri_share_start(t, c + 1), b1, p1);
    for (; b < b1 || (b == b1 && p < p1); ++b, p = 0) {
      if (b >= t.nb) return false;
      const int stop = b == b1 ? p1 : tri_row_units(t, b);
      if (p >= stop) continue;
      int first, count;
      tri_row_shares(t, b, first, count);
      if (c < first || c >= first + count || count > tri_max_row_shares(t)) return false;
      const int d0 = tri_own(t, b, p), d1 = tri_own(t, b, stop);
      const int o0 = p - d0, o1 = stop - d1, base = 2 * h * b;
      for (int g = base + d0; g < base + d1; ++g)
        if (g >= base + 2 * h || g >= t.ng || !seen.insert((long long)b * t.ng + g).second)
          return false;
      for (int g = base + 2 * h + o0; g < base + 2 * h + o1; ++g)
        if (g >= t.ng || !seen.insert((long long)b * t.ng + g).second) return false;
      for (int u = p; u < stop; ++u)
        if (tri_share_of(t, b, u) != c) return false;
    }
  }
  if ((long long)seen.size() != units) return false;
  for (int b = 0; b < t.nb; ++b) {
    std::set<int> own;
    for (int u = 0; u < tri_row_units(t, b); ++u) own.insert(tri_share_of(t, b, u));
    int first, count;
    tri_row_shares(t, b, first, count);
    if (*own.begin() != first || int(own.size()) != count) return false;
  }
  return true;
}

int main() {
  int plans = 0;
  for (int h : {2, 4, 5, 6, 8})
    for (int n : {1, 2, 31, 32, 33, 64, 65, 255, 256, 257, 383, 384, 385, 511, 512, 513, 1000,
                  2500, 3071, 3072, 3073, 4001, 8191, 8192, 8193, 16384, 30011})
      for (int want : {1, 2, 7, 40, 152, 304, 608}) {
        if (!check(n, h, want)) {
          std::printf("fault: n %d h %d shares %d\n", n, h, want);
          return 1;
        }
        ++plans;
      }
  std::printf("ok %d\n", plans);
  return 0;
}
