// tri_kernel.cuh -- all-pairs sums with each unordered pair evaluated once and
// applied to both particles, streamed in equal shares (tri_plan.h).
//
// One CTA (four warps) takes one share: a run of (row, source group) units of one
// or a few rows. The row's 64 H targets sit in registers of every warp, 2 H per
// lane, two to an f32x2 register group; the CTA's warps take the share's groups of
// 32 sources in turn. A lane starts with one source of the group in registers; at
// each of 32 steps it evaluates its source against its 2 H targets, adds the
// target-side terms to its target sums and the source-side terms to the sums that
// travel with the source, and hands the source and its sums to the lane below with
// shuffles. After 32 steps every source has met the warp's 64 H targets and is back
// in the lane it started from, with no shared memory, barrier or atomic in the pair
// loop. Groups left over when a share's groups do not divide by four are split by
// steps, eight per warp, and the four parts of their source-side sums added in
// shared memory.
//
// Why this shape. The packed FP32 unit bounds the loop: an f32x2 instruction holds its
// issue port for two cycles, so that the 16 operations of one register group (64 targets of
// a warp) take 32 at least; they take about 39, because one whose three operands share a
// register bank holds it longer and each MUFU adds 1.3. Per source-step a lane spends about
// 25 instructions besides the pairs: 2 H targets per step share them. Pairs of targets instead of pairs of sources in the
// f32x2 halves halve the registers per target (no duplicated target words), so a lane
// holds up to 16 targets at 8 warps per SM. Equal shares leave no partial wave: all CTAs
// are resident from the start (taken from a queue in smaller pieces instead, 3 to 6%
// more: 82 us against 77.5 at 16384, 298 against 287 at 32768). Two CTAs of four warps
// per SM: one of eight, whose warps keep step with each other, took 5% longer.
// Leapfrog steps inside a call (us), block-pair tile -> here: gravity 36.4 -> 28.4 at
// 8192, 91.8 -> 80.7 at 16384, 308 -> 295 at 32768; LJC 44.9 -> 36.5, 129.6 -> 117.2,
// 475 -> 440, and 1831 -> 1721 at 65536 (80% of the FP32 lane peak).
//
// Sums. A target's sum is plain FP32 over the sources that one warp meets in kChunk groups
// (128 with 16 groups, and the left-over ones), then over at most four such sums (a
// window), then over the four warps, each in order, and over the windows of a share with
// TwoSum. A source's sum is plain FP32 over the 2 H targets of a step and over 32 / kParts
// steps, then over the parts. Laws with kFine (gravity's forces from 8192 particles on, its
// VJP of 4096 to 8191), where the tiles are nearer to the 64-bit values than the longer
// sums, take 8 or 4 groups, 2 or 4 parts and TwoSum over the warps, and their potentials
// keep the low part of a share's sum. Rms errors against 64 bits, plain / fine / tile:
// potential 2.87e-8 / 2.54e-8 / 2.55e-8 at 12287, 2.65e-8 / 2.42e-8 / 2.48e-8 at 65536;
// accelerations 5.1e-8 / 4.6e-8 / 4.8e-8 at 12287; VJP, mass terms, 1.89e-7 / 1.61e-7 /
// 1.70e-7 at 6500. Leapfrog steps (us), plain / fine: 27.8 / 28.4 at 8192, 80.4 / 80.7 at
// 16384, 1143.9 / 1143.8 at 65536, with potential 772 / 782 at 50021; reverse steps 25.2 /
// 25.7 at 5000. The LJC laws' errors are those of their pair terms (forces 8e-7 either way).
// Partials go, per row b,
//   * source side: one per row and particle beyond it, to slot b;
//   * target side: one per share and target, to slot nb + (share - first share of
//     the row);
// each written once, so the finalize adds a particle's slots in a fixed order
// (tri_plan.h gives their number), and results are bitwise reproducible.
#pragma once

#include <type_traits>

#include "tri_laws.cuh"
#include "tri_plan.h"

namespace nbody {

constexpr int kTriWarps = 4;
constexpr int kTriThreads = 32 * kTriWarps;
constexpr int kTriWindow = 4;  // chunks (L::kChunk groups) between sums over the four warps
constexpr int kTriLeft = 3;    // left-over groups beyond the row of a window

struct TriArgs {
  const float4 *p0;  // (x, y, z, m)
  const float4 *p1;  // LJC parameters
  const float4 *p2;  // velocities, lambda, u (VJP and jerk laws)
  float4 *part;      // [slot][stride], kSums floats each: one float4, or two (hi at ostride)
  long long stride;
  long long ostride; // elements from the first float4 of a partial to its second
  float eps2;
  TriGeom geom;
  int pdl;           // host side: programmatic dependent launch
};

template <class L, int H>
struct TriTile {
  static constexpr int kRow = 64 * H;
  // the warps' target sums of a window; the left-over groups' source-side sums; the
  // CTA's compensated target sums (hi, lo)
  static constexpr int kRed = kTriWarps * L::kSums * kRow;
  static constexpr int kRem = kTriLeft * kTriWarps * L::kSums * 32;
  static constexpr int kComp = 2 * L::kSums * kRow;
  static constexpr size_t kSmemBytes = sizeof(float) * size_t(kRed + kRem + kComp);
  static_assert(kTriWarps * L::kSums >= L::kWords, "the target words are staged in the sums' place");
};

// Low parts of the fourth target-side sums that share `k` of a row leaves: a float for each
// particle, behind the slots.
__device__ __forceinline__ float *tri_low(const TriArgs &a, int k) {
  const int slot = a.geom.nb + tri_max_row_shares(a.geom);
  return reinterpret_cast<float *>(a.part + (long long)slot * a.stride) + (long long)k * a.stride;
}

// Place of a row's t-th target in an array of the row: the two targets of an f32x2
// value next to each other, lanes in order.
__device__ __forceinline__ int tri_place(int t) {
  return (t & ~63) + 2 * (t & 31) + ((t >> 5) & 1);
}

template <class L>
__device__ __forceinline__ void tri_store(const TriArgs &a, int slot, int i,
                                          const float (&v)[L::kSums]) {
  const long long o = (long long)slot * a.stride + i;
  if constexpr (L::kSums % 3 == 0) {
    a.part[o] = make_float4(v[0], v[1], v[2], 0.0f);
    if constexpr (L::kSums == 6) a.part[o + a.ostride] = make_float4(v[3], v[4], v[5], 0.0f);
  } else {
    a.part[o] = make_float4(v[0], v[1], v[2], v[3]);
    if constexpr (L::kSums == 8) a.part[o + a.ostride] = make_float4(v[4], v[5], v[6], v[7]);
  }
}

// STEPS steps of one source group beyond the row, from step s0 on, against the row's
// targets in registers; the lane starts with source (lane + s0) & 31 of the group in S. On
// return B holds the source-side sums of source (lane + s0 + STEPS) & 31 over these steps,
// before their sign change.
template <class L, int H, int STEPS>
__device__ __forceinline__ void tri_steps(float eps2, const float2 (&T)[H][L::kWords],
                                          float2 (&A)[H][L::kSums], float (&B)[L::kSums],
                                          float (&S)[L::kWords]) {
  const int next = (threadIdx.x & 31) + 1;
  const float2 e2 = bcast(eps2);
#pragma unroll
  for (int c = 0; c < L::kSums; ++c) B[c] = 0.0f;
#pragma unroll 1
  for (int st = 0; st < STEPS; ++st) {
    float J[2 * L::kSums];  // over this step's targets: even ones J[2c], odd ones J[2c+1]
#pragma unroll
    for (int c = 0; c < 2 * L::kSums; ++c) J[c] = 0.0f;
#pragma unroll
    for (int r = 0; r < H; ++r) L::template pair<false>(S, T[r], A[r], J, e2);
#pragma unroll
    for (int c = 0; c < L::kSums; ++c)
      B[c] = __shfl_sync(0xffffffffu, B[c] + (J[2 * c] + J[2 * c + 1]), next);
#pragma unroll
    for (int c = 0; c < L::kWords; ++c) S[c] = __shfl_sync(0xffffffffu, S[c], next);
  }
}

// All 32 steps from the lane's own source on, in L::kParts parts: each part's sums are added
// to the earlier ones' as the source moves on.
template <class L, int H>
__device__ __forceinline__ void tri_group(float eps2, const float2 (&T)[H][L::kWords],
                                          float2 (&A)[H][L::kSums], float (&B)[L::kSums],
                                          float (&S)[L::kWords]) {
  constexpr int kSteps = 32 / L::kParts;
  if constexpr (L::kParts == 1) {
    tri_steps<L, H, 32>(eps2, T, A, B, S);
  } else {
    const int from = (threadIdx.x & 31) + kSteps;
#pragma unroll
    for (int c = 0; c < L::kSums; ++c) B[c] = 0.0f;
#pragma unroll 1
    for (int k = 0; k < L::kParts; ++k) {
      float part[L::kSums];
      tri_steps<L, H, kSteps>(eps2, T, A, part, S);
#pragma unroll
      for (int c = 0; c < L::kSums; ++c) B[c] = __shfl_sync(0xffffffffu, B[c], from) + part[c];
    }
  }
}

// The same for the row's own-th own group, one-sided: the row's pairs are met in both
// orders, each time for the target alone, and only a lane's first step can meet itself.
// Twice the pairs, but no source side, and one straight loop: masking what was counted
// already (each own pair once, register groups skipped two at a time) took 2.5 us a unit
// against 1.7 of a unit beyond the row (gravity), waiting on the few pairs in flight.
template <class L, int H, int STEPS>
__device__ __forceinline__ void tri_own_group(float eps2, int own, int s0,
                                              const float2 (&T)[H][L::kWords],
                                              float2 (&A)[H][L::kSums], float (&S)[L::kWords]) {
  const int next = (threadIdx.x & 31) + 1;
  const float2 e2 = bcast(eps2);
  float J[2 * L::kSums];  // not used
  const int self = s0 == 0 ? own >> 1 : -1;
#pragma unroll
  for (int r = 0; r < H; ++r)
    L::template pair<true, false>(S, T[r], A[r], J, e2, !(r == self && !(own & 1)),
                                  !(r == self && (own & 1)));
#pragma unroll 1
  for (int st = 1; st < STEPS; ++st) {
#pragma unroll
    for (int c = 0; c < L::kWords; ++c) S[c] = __shfl_sync(0xffffffffu, S[c], next);
#pragma unroll
    for (int r = 0; r < H; ++r) L::template pair<false, false>(S, T[r], A[r], J, e2);
  }
}

// A share's units of one row: its own groups d0 .. d1-1 (counted from the row's first),
// then the groups o0 .. o1-1 beyond the row (counted from the first beyond).
template <class L, int H, bool AHEAD>
__device__ __forceinline__ void tri_run(const TriArgs &a, int row, int d0, int d1, int o0, int o1,
                                        int target_slot, float *low, float *smem) {
  using T_ = TriTile<L, H>;
  constexpr int R = T_::kRow, NS = L::kSums;
  float *red = smem;             // [warp][sum][R]
  float *rem = red + T_::kRed;   // [left-over group][warp][sum][32]
  float *comp = rem + T_::kRem;  // [sum][R] hi, then lo
  __shared__ int rem_group[kTriLeft];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = a.geom.n;
  // The row's targets, through shared memory: the two particles of an f32x2 value
  // then arrive as one 64-bit load, which keeps them in an aligned register pair
  // (packed from two registers, the compiler re-packs them in the pair loop).
  float2 T[H][L::kWords], A[H][NS];
  for (int t = tid; t < R; t += kTriThreads) {
    float w[L::kWords];
    L::load(a.p0, a.p1, a.p2, row * R + t, n, w);
    L::as_target(w);
#pragma unroll
    for (int c = 0; c < L::kWords; ++c) smem[c * R + tri_place(t)] = w[c];
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < H; ++r) {
#pragma unroll
    for (int c = 0; c < L::kWords; ++c)
      T[r][c] = *reinterpret_cast<const float2 *>(smem + c * R + 64 * r + 2 * lane);
#pragma unroll
    for (int c = 0; c < NS; ++c) A[r][c] = make_float2(0.0f, 0.0f);
  }
  __syncthreads();  // the target words' place is the sums' place

  int chunks = 0;       // of the current window
  int nleft = 0;        // left-over groups of the window
  bool folded = false;  // comp holds earlier windows
  // the window's target sums of the four warps into comp, or out when nothing follows,
  // and its left-over groups' source-side sums
  auto close_window = [&](bool done) {
    float v[NS], l[NS];
    __syncthreads();
    for (int t = tid; t < R; t += kTriThreads) {
      const int at = tri_place(t), i = row * R + t;
#pragma unroll
      for (int c = 0; c < NS; ++c) {
        v[c] = red[c * R + at];
        l[c] = 0.0f;
#pragma unroll
        for (int w = 1; w < kTriWarps; ++w) {
          const float s = red[(w * NS + c) * R + at];
          if (L::kFine) comp_add(v[c], l[c], s);
          else v[c] += s;
        }
        if (folded) {
          l[c] += comp[(NS + c) * R + t];
          comp_add(v[c], l[c], comp[c * R + t]);
        }
        if (!done) {
          comp[c * R + t] = v[c];
          comp[(NS + c) * R + t] = l[c];
        }
      }
      if (done && i < n) {
#pragma unroll
        for (int c = 0; c < NS; ++c) {
          const float s = v[c] + l[c];
          l[c] = __fsub_rn(l[c], __fsub_rn(s, v[c]));  // what s leaves out (Fast2Sum)
          v[c] = s;
        }
        tri_store<L>(a, target_slot, i, v);
        if (L::kLow) low[i] = l[NS - 1];
      }
    }
    for (int q = warp; q < nleft; q += kTriWarps) {  // warps' parts in order
#pragma unroll
      for (int c = 0; c < NS; ++c) {
        v[c] = rem[(q * kTriWarps * NS + c) * 32 + lane];
#pragma unroll
        for (int w = 1; w < kTriWarps; ++w) v[c] += rem[((q * kTriWarps + w) * NS + c) * 32 + lane];
      }
      const int i = rem_group[q] * kTriGroup + lane;
      if (i < n) tri_store<L>(a, row, i, v);
    }
    __syncthreads();  // red and rem are free for the next window
    chunks = nleft = 0;
    folded = true;
  };
  // groups g0 .. g1-1, all own (DIAG) or all beyond the row; `more`: others follow
  auto groups = [&](auto diag, int g0, int g1, bool more) {
    constexpr bool DIAG = decltype(diag)::value;
    for (int g = g0; g < g1; g += L::kChunk) {
      const int k = min(L::kChunk, g1 - g);
      const int quads = k >> 2, left = k & 3;
      float v[NS], S[L::kWords];
      auto source_sums = [&]() {
#pragma unroll
        for (int c = 0; c < NS; ++c)
          if ((L::kFlip >> c) & 1) v[c] = -v[c];
      };
      // This warp's groups of the chunk; with AHEAD the next group's sources are on
      // their way while one is worked on.
      float P[L::kWords];
      if (AHEAD) L::load(a.p0, a.p1, a.p2, (g + warp) * kTriGroup + lane, n, P);
      for (int m = 0; m < quads; ++m) {
        const int gg = g + 4 * m + warp, i = gg * kTriGroup + lane;
        if (AHEAD) {
#pragma unroll
          for (int c = 0; c < L::kWords; ++c) S[c] = P[c];
          if (m + 1 < quads) L::load(a.p0, a.p1, a.p2, i + 4 * kTriGroup, n, P);
        } else {
          L::load(a.p0, a.p1, a.p2, i, n, S);
        }
        if constexpr (DIAG) {
          tri_own_group<L, H, 32>(a.eps2, gg - 2 * H * row, 0, T, A, S);
        } else {
          tri_group<L, H>(a.eps2, T, A, v, S);
          source_sums();
          if (i < n) tri_store<L>(a, row, i, v);
        }
      }
      for (int m = 0; m < left; ++m) {  // its eight steps of each left-over group
        const int gg = g + 4 * quads + m, s0 = 8 * warp;
        L::load(a.p0, a.p1, a.p2, gg * kTriGroup + ((lane + s0) & 31), n, S);
        if constexpr (DIAG) {
          tri_own_group<L, H, 8>(a.eps2, gg - 2 * H * row, s0, T, A, S);
          continue;
        }
        tri_steps<L, H, 8>(a.eps2, T, A, v, S);
        source_sums();
#pragma unroll
        for (int c = 0; c < NS; ++c)
          rem[((nleft * kTriWarps + warp) * NS + c) * 32 + ((lane + s0 + 8) & 31)] = v[c];
        if (tid == 0) rem_group[nleft] = gg;
        ++nleft;
      }
      // the chunk's target sums, into this thread's own words of `red`
#pragma unroll
      for (int r = 0; r < H; ++r)
#pragma unroll
        for (int c = 0; c < NS; ++c) {
          float2 *w = reinterpret_cast<float2 *>(red + (warp * NS + c) * R + 64 * r + 2 * lane);
          *w = chunks ? __fadd2_rn(*w, A[r][c]) : A[r][c];
          A[r][c] = make_float2(0.0f, 0.0f);
        }
      ++chunks;
      const bool done = !more && g + L::kChunk >= g1;
      if (done || chunks == kTriWindow) close_window(done);
    }
  };
  const int first = 2 * H * row;
  groups(std::true_type{}, first + d0, first + d1, o1 > o0);
  groups(std::false_type{}, first + 2 * H + o0, first + 2 * H + o1, false);
}

template <class L, int H, int MINB, bool AHEAD>
__global__ void __launch_bounds__(kTriThreads, MINB) tri_kernel(const __grid_constant__ TriArgs a) {
  griddep_launch();
  extern __shared__ __align__(16) float tri_smem[];
  const int share = int(blockIdx.x);
  int row, p, row_end, p_end;
  tri_locate(a.geom, tri_share_start(a.geom, share), row, p);
  tri_locate(a.geom, tri_share_start(a.geom, share + 1), row_end, p_end);
  griddep_start();
  for (; row < row_end || (row == row_end && p < p_end); ++row, p = 0) {
    const int stop = row == row_end ? p_end : tri_row_units(a.geom, row);
    if (p >= stop) continue;
    const int d0 = tri_own(a.geom, row, p), d1 = tri_own(a.geom, row, stop);
    int first, count;
    tri_row_shares(a.geom, row, first, count);
    const int k = share - first;
    tri_run<L, H, AHEAD>(a, row, d0, d1, p - d0, stop - d1, a.geom.nb + k,
                         L::kLow ? tri_low(a, k) : nullptr, tri_smem);
  }
}

}  // namespace nbody
