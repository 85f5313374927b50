// tri_tiles.h -- the compiled streamed triangle kernels (tri_kernel.cuh) and the rule
// that picks one by law and size.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "tri_kernel.cuh"

namespace nbody {

struct TriDesc {
  int h;         // f32x2 register groups per thread: rows of 64 h particles
  int per_sm;    // CTAs per SM (by registers): the grid is one wave
  bool low;      // evaluations with the potential leave its sums' low parts (kLow)
  cudaError_t (*launch)(const TriArgs &, bool pot, bool precise, cudaStream_t);
};

// Kernel for a force law (0 gravity, 1 LJC, 2 LJC linear) at n particles.
const TriDesc *tri_grav(int64_t n);
const TriDesc *tri_ljc(int64_t n);
const TriDesc *tri_ljclin(int64_t n);
// Kernel for a VJP or jerk tile table (tri_vjp.cu; no potential or precise variants).
const TriDesc *tri_vjp(int table, int64_t n);

}  // namespace nbody
