// direct_tiles.h -- host side of direct_kernel.cuh: the rule that picks targets per CTA
// and source slices, and the launch.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "direct_kernel.cuh"

namespace nbody {

// Launch with 16 (big) or 8 targets per CTA.
using DirectLauncher = cudaError_t (*)(const DirectArgs &, bool big, bool pot, bool precise,
                                       cudaStream_t);
cudaError_t direct_grav(const DirectArgs &a, bool big, bool pot, bool precise, cudaStream_t s);
cudaError_t direct_ljc(const DirectArgs &a, bool big, bool pot, bool precise, cudaStream_t s);
cudaError_t direct_ljclin(const DirectArgs &a, bool big, bool pot, bool precise, cudaStream_t s);

struct DirectPlan {
  bool big;
  int slices;
};

// Targets per CTA (16 or 8) and source slices for n_t targets and n sources: the least
// modelled time. The CTAs run in waves of what the GPU holds in clusters of that size
// (measured on 152 SMs, two CTAs or one on an SM; fewer than two per SM where a
// cluster's size does not divide an SM group's); a wave takes `fixed` to start, add up
// its sums and end, and `block` for every 256 sources of its slice, less (`alone`) where
// a CTA has its SM to itself. Fitted to 1300 timings of 20 to 12000 targets and 2048 to
// 131072 sources within 7% rms; the picks take 1% more than the best in the mean, e.g.
// 1500 targets of 65536 in 16s and 3 slices 51 us (8s and 3 slices 69, 16s and 4 slices
// 57); fitted without gravity's folds of 12 sources, which add a tenth to `block`. False
// where a thread would take more than 1024 sources at the most slices (n above two million).
struct DirectCost {
  double block, fixed, alone, launch;  // us
  bool one;                            // one CTA on an SM
};
// The least time over the slices (added to *out with `big` if less than *best).
inline void direct_slices(const DirectCost &c, bool big, int64_t targets_per_cta, int64_t n_t,
                          int64_t n, int sms, double *best, DirectPlan *out) {
  constexpr int64_t kChain = 32 * kDirectFold;
  static constexpr int kTwo[8] = {304, 304, 291, 296, 290, 276, 266, 288};
  static constexpr int kOne[8] = {152, 152, 138, 144, 140, 138, 105, 120};
  for (int s = 1; s <= 8; ++s) {
    if (n > kChain * kDirectThreads * s) continue;
    if (s > 1 && (s - 1) * kDirectThreads >= n) continue;  // an empty slice
    const int64_t ctas = (n_t + targets_per_cta - 1) / targets_per_cta * s;
    const int64_t held =
        std::max<int64_t>(int64_t(c.one ? kOne[s - 1] : kTwo[s - 1]) * sms / 152, 1);
    const int64_t waves = (ctas + held - 1) / held, last = ctas - (waves - 1) * held;
    const double work = double((n + kDirectThreads * s - 1) / (kDirectThreads * s)) * c.block;
    const double us = c.launch + (s > 1 ? 0.6 : 0.0) + double(waves) * c.fixed +
                      work * (double(waves - 1) + (2 * last <= held ? c.alone : 1.0));
    if (*best < 0.0 || us < *best) {
      *best = us;
      *out = DirectPlan{big, s};
    }
  }
}
inline bool direct_plan(int law, bool pot, int64_t n_t, int64_t n, int sms, DirectPlan *out) {
  static constexpr DirectCost kGrav[2] = {{0.296, 2.84, 0.66, 0.45, false},
                                          {0.503, 3.06, 0.59, 0.61, false}};
  static constexpr DirectCost kLjc[2] = {{0.533, 2.87, 0.76, 0.53, false},
                                         {0.496, 3.24, 1.0, 0.57, true}};
  if (n_t > (int64_t(1) << 28)) return false;
  double best = -1.0;
  for (int big = 0; big < 2; ++big) {
    if (big && law == 0 && pot) continue;  // 16 targets' potentials leave one CTA on an SM
    direct_slices(law == 0 ? kGrav[big] : kLjc[big], big == 1, big ? 16 : 8, n_t, n, sms, &best,
                  out);
  }
  return best >= 0.0;
}

// Whether forces on all n particles run in one direct launch: one wave of two CTAs on
// every SM, of 16 targets for gravity and 8 for the LJC laws (4864 and 2432 particles on
// 152 SMs). Above, where a second wave would run, the streamed triangle kernels are faster
// (us per step: gravity direct 13.1 at 4864, streamed 18.4 at 4865 where two direct waves
// take 21; LJC direct 8.1 at 2432, 19.6 at 3000 where streamed takes 13.8).
inline bool direct_all(int law, int64_t n, int sms) { return n <= (law == 0 ? 32 : 16) * sms; }

// Whether gravity's sums compensate every exchange between lanes (0.6 us of a launch): where
// with two plain ones the rms error of accelerations or potentials passes the tiles'. All n:
// 0.99 and 1.00 of it at 2432, 0.99 and 1.01 at 2700, 1.02 and 1.01 at 3300 and 4095
// (compensated 0.97 to 1.00), half of it from 4096 on; subsets of n sources, accelerations:
// 0.97 at 8192, 1.00 at 12000, 1.01 at 16000 (0.96, 0.98, 1.00).
inline bool direct_fine(bool subset, int64_t n) {
  return subset ? n > 12000 : n > 2432 && n < 4096;
}

// The jerk and VJP laws (tile tables of tri_vjp.cu): 8 targets per CTA, 4 for the LJC
// VJPs; mode 0 only.
cudaError_t direct_vjp(int table, const DirectArgs &a, cudaStream_t s);

}  // namespace nbody
