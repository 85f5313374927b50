// tri_plan.h -- how the streamed triangle kernels (tri_kernel.cuh) cut the N (N - 1) / 2
// unordered pairs of one system into equal shares, one per CTA. Plain integer
// arithmetic, the same on the host (planning, tests) and on the device (the kernel
// itself and the finalize kernels that read its partial sums).
//
// Particles are cut into rows of R = 64 h targets (h f32x2 register groups of 64
// targets per warp) and groups of 32 sources. The unit of work is row b against
// source group g >= 2 h b: the first 2 h groups of a row are its own particles, the
// others lie beyond it. The units are put in a line, row after row, each of cost 1; a
// row costs kTriRowCost more, for loading its targets and adding up its sums. Within a
// row the own units, whose pairs are met twice but from one side (tri_kernel.cuh), are
// spread evenly among the others (tri_own), so that every share of a row gets its part of
// them. The line is cut into nshare shares of equal cost.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define NBODY_HD __host__ __device__ __forceinline__
#else
#define NBODY_HD inline
#endif

namespace nbody {

constexpr int kTriGroup = 32;  // sources per group

// Cost of a row besides its units (fitted to the SMs' times at 8192 and 16384
// particles: 0.8 to 2 us a row, units of 0.7 to 1.5 us).
constexpr int kTriRowCost = 1;

struct TriGeom {
  int n;       // particles
  int h;       // f32x2 register groups per thread: a row is 64 h particles
  int nb;      // rows
  int ng;      // source groups
  int nshare;  // shares
  int extra;   // cost of a row besides its units
  long long total;  // cost of the line
  int low;     // the shares' low parts follow the slots (tri_slots)
};

// Units of row b, and how many of the first p of them are own units (the others are
// the first p - tri_own(t, b, p) groups beyond the row).
NBODY_HD int tri_row_units(const TriGeom &t, int b) { return t.ng - 2 * t.h * b; }
NBODY_HD int tri_own(const TriGeom &t, int b, int p) {
  const int len = tri_row_units(t, b), own = 2 * t.h < len ? 2 * t.h : len;
  return int((long long)p * own / len);
}

// Cost of the rows before row b.
NBODY_HD long long tri_row_start(const TriGeom &t, long long b) {
  return b * (t.ng + t.extra) - (long long)t.h * (b * (b - 1));
}

NBODY_HD TriGeom tri_geom(int n, int h, int max_share) {
  TriGeom t;
  t.n = n;
  t.h = h;
  t.nb = int(((long long)n + 64 * h - 1) / (64 * h));
  t.ng = int(((long long)n + kTriGroup - 1) / kTriGroup);
  t.extra = kTriRowCost;
  t.low = 0;
  t.total = tri_row_start(t, t.nb);
  // Shares between a row's first and last must own units of it (tri_row_shares): with
  // the row cost they do when a share is longer than 2 (kTriRowCost + 1); where shares
  // are shorter (a few rows over the whole GPU) the row cost is left out
  t.nshare = max_share;
  if (t.total < (long long)max_share * (2 * kTriRowCost + 3)) {
    t.extra = 0;
    t.total = tri_row_start(t, t.nb);
    if (t.total < max_share) t.nshare = int(t.total);
  }
  return t;
}

// First cost position of share c.
NBODY_HD long long tri_share_start(const TriGeom &t, int c) { return t.total * c / t.nshare; }

// Row b of cost position q and the first unit of the row at or after it (the row's
// length when none follows); (nb, 0) for the end.
NBODY_HD void tri_locate(const TriGeom &t, long long q, int &b, int &p) {
  if (q >= t.total) {
    b = t.nb;
    p = 0;
    return;
  }
  int lo = 0, hi = t.nb - 1;  // the last row that starts at or before q
  while (lo < hi) {
    const int mid = lo + (hi - lo + 1) / 2;
    if (tri_row_start(t, mid) <= q) lo = mid;
    else hi = mid - 1;
  }
  b = lo;
  const long long len = tri_row_units(t, b);
  p = int((q - tri_row_start(t, b)) * len / (len + t.extra));
}

// Share that owns unit p of row b: the one whose cost range ends first at or beyond
// the position from which p + 1 units are counted (tri_locate).
NBODY_HD int tri_share_of(const TriGeom &t, int b, int p) {
  const long long len = tri_row_units(t, b);
  const long long q = tri_row_start(t, b) + ((p + 1) * (len + t.extra) + len - 1) / len;
  // the smallest c with tri_share_start(c + 1) >= q
  return int((q * t.nshare + t.total - 1) / t.total - 1);
}

// Shares that own units of row b: the first, and how many (all between own some).
NBODY_HD void tri_row_shares(const TriGeom &t, int b, int &first, int &count) {
  first = tri_share_of(t, b, 0);
  count = tri_share_of(t, b, tri_row_units(t, b) - 1) - first + 1;
}

// Most shares that a row can have: rows get shorter, so row 0's length decides.
NBODY_HD int tri_max_row_shares(const TriGeom &t) {
  return int((long long)(t.ng + t.extra) * t.nshare / t.total + 2);
}

// Slots (of a float4 for each particle) of a force evaluation: a source-side one per row,
// target-side ones of the row with the most shares, and a float for each of the latter.
NBODY_HD int tri_slots(const TriGeom &t) {
  const int shares = tri_max_row_shares(t);
  return t.nb + shares + (shares + 3) / 4;
}

}  // namespace nbody
