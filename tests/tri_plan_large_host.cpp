// Host check of csrc/tri_plan.h at large sizes: the shares follow each other without a gap,
// the first and the last unit that a share takes of a row are its own, and the shares that
// the finalize kernels count for a row are those that take units of it. Prints "ok <plans>" or
// the first fault.
#include <cstdio>
#include <vector>

#include "tri_plan.h"

using namespace nbody;

static bool check(int n, int h, int want) {
  const TriGeom t = tri_geom(n, h, want);
  std::vector<long long> units(size_t(t.nb), 0);
  std::vector<int> shares(size_t(t.nb), 0);
  for (int c = 0; c < t.nshare; ++c) {
    int b, p, b1, p1;
    tri_locate(t, tri_share_start(t, c), b, p);
    tri_locate(t, tri_share_start(t, c + 1), b1, p1);
    for (; b < b1 || (b == b1 && p < p1); ++b, p = 0) {
      if (b >= t.nb) return false;
      const int stop = b == b1 ? p1 : tri_row_units(t, b);
      if (p >= stop) continue;
      if (units[size_t(b)] != p) return false;  // goes on where the one before ended
      int first, count;
      tri_row_shares(t, b, first, count);
      if (c < first || c >= first + count || count > tri_max_row_shares(t)) return false;
      if (tri_share_of(t, b, p) != c || tri_share_of(t, b, stop - 1) != c) return false;
      const int d0 = tri_own(t, b, p), d1 = tri_own(t, b, stop);
      if (d0 < 0 || d1 < d0 || d1 - d0 > stop - p || 2 * h * b + d1 > t.ng) return false;
      if (stop - d1 > 0 && 2 * h * (b + 1) + stop - d1 > t.ng) return false;
      units[size_t(b)] = stop;
      ++shares[size_t(b)];
    }
  }
  for (int b = 0; b < t.nb; ++b) {
    int first, count;
    tri_row_shares(t, b, first, count);
    if (units[size_t(b)] != tri_row_units(t, b) || shares[size_t(b)] != count) return false;
  }
  const int most = tri_max_row_shares(t);
  return 4LL * (tri_slots(t) - t.nb - most) >= most;  // a float for each share and particle
}

int main() {
  int plans = 0;
  for (int n : {30012, 65536, 65537, 114687, 131071, 163839, 262144, 1000003, 2147479551})
    for (int h : {4, 6, 8})
      for (int want : {152, 296, 304}) {
        if (!check(n, h, want)) {
          std::printf("fault: n %d h %d shares %d\n", n, h, want);
          return 1;
        }
        ++plans;
      }
  std::printf("ok %d\n", plans);
  return 0;
}
