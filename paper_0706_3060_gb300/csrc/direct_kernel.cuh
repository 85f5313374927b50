// direct_kernel.cuh -- forces on few targets in one launch: the targets' sums over all
// sources, their accelerations, and (steps of nbody_step) their kicks and drifts.
//
// For systems of a few thousand particles and for subsets of active particles. A CTA of
// 256 threads owns 2 H targets; every thread holds all of them in registers, two to an
// f32x2 register group, and its lanes take the sources in turn, straight from global
// memory (each source is read by one thread of the CTA). A cluster of up to eight CTAs
// shares the sources of one set of targets. The per-thread sums are added over the
// lanes (halving the values at each exchange) and, compensated, over the warps and,
// through distributed shared memory, the CTAs of the cluster, always in the same order,
// so results are bitwise reproducible.
//
// Sums. A thread adds 32 sources in plain FP32, then such sums in shared memory, and the
// first two exchanges between lanes are plain. Gravity's forces (kFine) fold every 12
// sources (none up to 20), carry what a fold's sum leaves out into the next fold (Kahan's
// summation) and, where direct_fine says so, compensate every exchange: a close pair's large
// pull is rounded again with each later add. Rms errors against 64 bits, plain / so / tile:
// 1500 targets of 65536 3.80e-8 / 3.66e-8 / 3.65e-8, 4000 of 131072 3.66e-8 / 3.46e-8 /
// 3.49e-8, the same with a close companion for every particle 1.55e-7 / 1.35e-7 / 1.35e-7,
// all of 3600 5.06e-8 / 4.93e-8 / 5.02e-8. Time (us, calls in a loop), plain / so: 55.5 /
// 60.1, 236 / 257, a step of 4001 particles 11.6 / 12.2 (folds of 16 56.8, with errors to 2%
// above the tiles'; of 8 61.1; with the low parts kept beside the sums 64.3). The LJC laws'
// errors are those of their pair terms (1.2e-6 either way), and the VJPs and the jerk run
// here up to 2432 particles, without folds.
//
// What bounds it: launch and latency up to about 1500 particles (one launch where the
// tile path takes an interleave, a force and a finalize launch), then the packed FP32
// unit (12 operations per gravity pair, one-sided; 66% of its cycles at 1500 targets of
// 65536, the folds among them). The pair symmetry is not used: it pays only where its
// partial sums cost less than the pairs it saves (tri_kernel.cuh). Measured, against the
// tile kernels (us): gravity steps at 1024 3.6 / 7.1, 2048 5.4 / 8.9, 4001 12.0 / 21.9; LJC
// 1024 4.4 / 8.2, 2048 7.2 / 11.1; gravity subsets of 65536: 300 targets 16 / 40, 1500
// 53 / 183, 6000 180 / 333; LJC 1500 99 / 230.
#pragma once

#include <cooperative_groups.h>

#include "aux_types.h"
#include "leapfrog.cuh"
#include "tri_laws.cuh"

namespace nbody {

constexpr int kDirectThreads = 256;
constexpr int kDirectWarps = kDirectThreads / 32;
constexpr int kDirectFold = 32;  // sources per register sum
// Laws with finer sums (kFine): sources per register sum, and the most without folds
constexpr int kFineFold = 12, kFineChain = 20;
template <class L>
constexpr int direct_chain() { return L::kFine ? kFineChain : kDirectFold; }

struct DirectArgs {
  const float4 *pos;  // sources (x, y, z, m)
  const float4 *prm;  // LJC parameters or null
  const float4 *vec;  // velocities or lambda (jerk and VJP laws), else null
  const int *idx;     // targets (a subset's indices), or null: all particles
  int n_t;
  int n;
  int slices;         // CTAs of a cluster: source slices
  int *err;
  float eps2;
  float G;
  int law;
  // what the targets' sums become; mode: kFinWriteAcc, kFinKickSync, kFinKickDrift, or 0:
  // nothing (acc and acc_lo get the sums and their low parts, for a finalize launch)
  int mode;
  float dt;
  float4 *acc;       // element per target
  float4 *acc_lo;
  long long ostride; // mode 0, laws of more than four sums: elements to their second row
  float4 *vel;
  float4 *pos_out;   // drifted positions (not `pos`: other CTAs still read it)
  float4 *trace;     // drifted positions as well, or null
  float4 *x_lo;      // two-float state or null
  float4 *v_lo;
  int fine;          // kFine: compensate every exchange between lanes (direct_fine)
  int pdl;           // host side
};

// Two CTAs on an SM where their registers fit (16 targets of gravity without a
// potential: 51 us for 1500 targets of 65536, with one 85).
template <class L, int H, int U>
__global__ void __launch_bounds__(kDirectThreads,
                                  L::kWords * (H + 1) + L::kSums * H <= 60 ? 2 : 0) direct_kernel(
    const __grid_constant__ DirectArgs a) {
  namespace cg = cooperative_groups;
  constexpr int NS = L::kSums, TG = 2 * H, V = TG * NS;
  __shared__ __align__(16) float words[L::kWords][TG];
  __shared__ float red[2][kDirectWarps][V];
  __shared__ float sums[2][V];  // and their low parts
  __shared__ int tidx[TG];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tile = int(blockIdx.x) / a.slices, slice = int(blockIdx.x) - tile * a.slices;
  const int t0 = tile * TG;
  griddep_start();
  if (tid < TG) {
    int g = -1;
    float w[L::kWords];
    if (t0 + tid < a.n_t) {
      g = a.idx ? __ldg(a.idx + t0 + tid) : t0 + tid;
      if (g < 0 || g >= a.n) {  // reported; the row is computed for particle 0
        set_error(a.err, kDevBadItem);
        g = 0;
      }
    }
    L::template load<true>(a.pos, a.prm, a.vec, g >= 0 ? g : a.n, a.n, w);
    L::as_target(w);
#pragma unroll
    for (int c = 0; c < L::kWords; ++c) words[c][tid] = w[c];
    tidx[tid] = g;
  }
  __syncthreads();
  float2 T[H][L::kWords], A[H][NS];
#pragma unroll
  for (int r = 0; r < H; ++r) {
#pragma unroll
    for (int c = 0; c < L::kWords; ++c)
      T[r][c] = *reinterpret_cast<const float2 *>(&words[c][2 * r]);
#pragma unroll
    for (int c = 0; c < NS; ++c) A[r][c] = make_float2(0.0f, 0.0f);
  }
  const int mine = lane < TG ? tidx[lane] : -1;
  const float2 e2 = bcast(a.eps2);
  // slice bounds at multiples of the CTA's stride
  const int blocks = (a.n + kDirectThreads - 1) / kDirectThreads;
  const int b0 = int((long long)blocks * slice / a.slices);
  const int b1 = int((long long)blocks * (slice + 1) / a.slices);
  extern __shared__ __align__(16) float2 folded[];
  constexpr int kFold = L::kFine ? kFineFold : kDirectFold;
  static_assert(kFold % U == 0, "folds between prefetch groups");
  const bool many = b1 - b0 > direct_chain<L>();
  // sources: U of this thread's are on their way while one is worked on
  float P[U][L::kWords];
#pragma unroll
  for (int u = 0; u < U; ++u)
    L::template load<true>(a.pos, a.prm, a.vec, min(b0 + u, b1) * kDirectThreads + tid, a.n, P[u]);
  int fold_at = b0;  // the block after the last fold
  for (int b = b0; b < b1; b += U) {
    // every kFold sources the sums go to this thread's own words in shared memory:
    // a close pair's large pull is not rounded again with each of hundreds of sources
    if (many && b - fold_at == kFold) {
      const bool first = fold_at == b0;
      fold_at = b;
#pragma unroll
      for (int r = 0; r < H; ++r)
#pragma unroll
        for (int c = 0; c < NS; ++c) {
          const int at = (r * NS + c) * kDirectThreads + tid;
          float2 *f = folded + at;
          if (first) {
            *f = A[r][c];
            A[r][c] = make_float2(0.0f, 0.0f);
          } else if (L::kFine) {
            const float2 h = *f, s = __fadd2_rn(h, A[r][c]);
            // what the sum leaves out, A - (s - h), goes into the next fold
            A[r][c] = __ffma2_rn(__ffma2_rn(h, bcast(-1.0f), s), bcast(-1.0f), A[r][c]);
            *f = s;
          } else {
            *f = __fadd2_rn(*f, A[r][c]);
            A[r][c] = make_float2(0.0f, 0.0f);
          }
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (b + u >= b1) break;
      const int first = (b + u) * kDirectThreads + 32 * warp, j = first + lane;
      float J[2 * NS];  // not used one-sided
      if (!__any_sync(0xffffffffu, mine >= first && mine < first + 32)) {
#pragma unroll
        for (int r = 0; r < H; ++r) L::template pair<false, false>(P[u], T[r], A[r], J, e2);
      } else {  // a target among the warp's sources: drop the self pairs by index
#pragma unroll
        for (int r = 0; r < H; ++r)
          L::template pair<true, false>(P[u], T[r], A[r], J, e2, tidx[2 * r] != j,
                                        tidx[2 * r + 1] != j);
      }
      if (b + u + U < b1)
        L::template load<true>(a.pos, a.prm, a.vec, j + U * kDirectThreads, a.n, P[u]);
    }
  }
  if (many) {
#pragma unroll
    for (int r = 0; r < H; ++r)
#pragma unroll
      for (int c = 0; c < NS; ++c) {
        const int at = (r * NS + c) * kDirectThreads + tid;
        A[r][c] = __fadd2_rn(folded[at], A[r][c]);
      }
  }
  // sums over the lanes: at each exchange a lane keeps half of its values (all of
  // them once their number is odd); compensated (unless `fine`, from the third exchange on,
  // where few values are left and their sums are large)
  constexpr int kHalvings = V % 32 == 0 ? 5 : V % 16 == 0 ? 4 : V % 8 == 0 ? 3 : V % 4 == 0 ? 2 : 1;
  constexpr int kLeft = V >> kHalvings, kComp = 2;
  static_assert(kHalvings >= kComp, "compensated exchanges start at a quarter of the values");
  float v[V], l[L::kFine ? V : V >> kComp];
#pragma unroll
  for (int r = 0; r < H; ++r)
#pragma unroll
    for (int c = 0; c < NS; ++c) {
      v[c * TG + 2 * r] = A[r][c].x;
      v[c * TG + 2 * r + 1] = A[r][c].y;
    }
#pragma unroll
  for (int k = 0; k < (L::kFine ? V : V >> kComp); ++k) l[k] = 0.0f;
  const bool fine = L::kFine && a.fine;
  int base = 0, spare = 0;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const int off = 16 >> q;
    const bool halve = q < kHalvings, up = halve && (lane & off) != 0;
    const int keep = halve ? V >> (q + 1) : kLeft;  // values after this exchange
#pragma unroll
    for (int k = 0; k < V / 2; ++k) {
      if (k >= keep) break;
      const int o = halve ? k + keep : k;  // the upper half's
      const float own = up ? v[o] : v[k];
      const float got = __shfl_xor_sync(0xffffffffu, up ? v[k] : v[o], off);
      if (q < kComp && !fine) {
        v[k] = own + got;
      } else {
        float e;
        const float own_l = up ? l[o] : l[k];
        const float got_l =
            q > kComp || (q > 0 && fine)
                ? __shfl_xor_sync(0xffffffffu, up ? l[k] : l[o], off) : 0.0f;
        two_sum(own, got, v[k], e);
        l[k] = (own_l + got_l) + e;
      }
    }
    if (up) base += keep;
    if (!halve) spare |= lane & off;
  }
  if (!spare) {
#pragma unroll
    for (int k = 0; k < kLeft; ++k) {
      red[0][warp][base + k] = v[k];
      red[1][warp][base + k] = l[k];
    }
  }
  __syncthreads();
  if (tid < V) {
    float hi = red[0][0][tid], lo = red[1][0][tid];
#pragma unroll
    for (int w = 1; w < kDirectWarps; ++w) {
      comp_add(hi, lo, red[0][w][tid]);
      lo += red[1][w][tid];
    }
    sums[0][tid] = hi;
    sums[1][tid] = lo;
  }
  if (a.slices > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    if (slice == 0 && tid < V) {
      float hi = sums[0][tid], lo = sums[1][tid];
      for (int k = 1; k < a.slices; ++k) {
        const float *other = cluster.map_shared_rank(&sums[0][0], k);
        comp_add(hi, lo, other[tid]);
        lo += other[V + tid];
      }
      sums[0][tid] = hi;
      sums[1][tid] = lo;
    }
    cluster.sync();  // the other CTAs' shared memory stays until it has been read
    if (slice != 0) return;
  }
  __syncthreads();
  const int t = t0 + tid;
  if (tid >= TG || t >= a.n_t) return;
  const int g = tidx[tid];
  auto row = [&](const float (&v)[V], int c0) {
    constexpr int kRow = NS == 6 ? 3 : NS < 4 ? NS : 4;  // sums in a row
    return make_float4(v[c0 * TG + tid], v[(c0 + 1) * TG + tid], v[(c0 + 2) * TG + tid],
                       kRow > 3 ? v[(c0 + 3) * TG + tid] : 0.0f);
  };
  const float4 hi = row(sums[0], 0), lo = row(sums[1], 0);
  if (!a.mode) {
    a.acc[t] = hi;
    a.acc_lo[t] = lo;
    if constexpr (NS > 4) {
      a.acc[t + a.ostride] = row(sums[0], NS / 2);
      a.acc_lo[t + a.ostride] = row(sums[1], NS / 2);
    }
    return;
  }
  float4 x = a.pos[g], ac;
  const float4 f = make_float4(hi.x + lo.x, hi.y + lo.y, hi.z + lo.z, hi.w + lo.w);
  if (a.law == 0) {  // a = G sum m y^3 d, phi = -G sum m y
    ac = make_float4(a.G * f.x, a.G * f.y, a.G * f.z, -a.G * f.w);
  } else {  // F = -sum f d, a = F / m; phi = sum of pair energies
    const float inv_m = 1.0f / x.w;
    ac = make_float4(-f.x * inv_m, -f.y * inv_m, -f.z * inv_m, f.w);
  }
  if (a.mode & kFinWriteAcc) a.acc[t] = ac;
  if (!(a.mode & (kFinKickSync | kFinKickDrift))) return;
  float4 vel = a.vel[g];
  const float h = 0.5f * a.dt;
  const bool two = a.x_lo != nullptr;
  float4 xl = two ? a.x_lo[g] : make_float4(0.f, 0.f, 0.f, 0.f);
  float4 vl = two ? a.v_lo[g] : make_float4(0.f, 0.f, 0.f, 0.f);
  auto kick = [&]() {
    if (two) {
      comp_axpy(vel, vl, h, ac);
    } else {
      vel.x = fmaf(h, ac.x, vel.x);
      vel.y = fmaf(h, ac.y, vel.y);
      vel.z = fmaf(h, ac.z, vel.z);
    }
  };
  if (a.mode & kFinKickSync) kick();
  if (a.mode & kFinKickDrift) {
    kick();
    if (two) {  // drift with the full two-float velocity
      comp_axpy(x, xl, a.dt, make_float4(vel.x + vl.x, vel.y + vl.y, vel.z + vl.z, 0.f));
    } else {
      x.x = fmaf(a.dt, vel.x, x.x);
      x.y = fmaf(a.dt, vel.y, x.y);
      x.z = fmaf(a.dt, vel.z, x.z);
    }
    a.pos_out[g] = x;
    if (a.trace) a.trace[g] = x;
  }
  a.vel[g] = vel;
  if (two) {
    a.x_lo[g] = xl;
    a.v_lo[g] = vl;
  }
}

}  // namespace nbody
