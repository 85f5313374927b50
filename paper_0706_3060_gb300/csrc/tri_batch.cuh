// tri_batch.cuh -- the streamed triangle kernel (tri_kernel.cuh) over many independent
// systems of mixed law and uneven size: one wave of CTAs that take segments of rows from a
// queue (tri_batch_plan.h).
//
// What bounds it: the packed FP32 unit, as for one system, and the pairs within a row,
// which are met twice (a quarter of the work at the mean size of 1000). Per step with
// BatchPlan, against the block-pair tiles (us): 512 systems of 64 to 4096 399 / 449, 128
// to 4096 110 / 127, 128 to 2048 43.7 / 64, 32 to 4096 42 / 65, 300 to 700 32 / 58, 32 to
// 1024 15.9 / 31, 16 to 512 9.8 / 25.
#pragma once

#include "tri_batch_plan.h"
#include "tri_kernel.cuh"
#include "tri_laws.cuh"

namespace nbody {

struct TriBatchArgs {
  const float4 *pos;
  const float4 *prm;
  float4 *part;        // [slot][stride]
  long long stride;    // particles of the ensemble
  const TriSeg *segs;
  int nseg;
  int *counter;        // segments taken beyond the first of each CTA; zero at the launch
  int grid;            // host side
  int pdl;             // host side
};

cudaError_t tri_batch(const TriBatchArgs &a, bool precise, cudaStream_t s);
int tri_batch_per_sm();

template <bool PRECISE>
__global__ void __launch_bounds__(kTriThreads, 2) tri_batch_kernel(
    const __grid_constant__ TriBatchArgs a) {
  griddep_launch();
  extern __shared__ __align__(16) float tri_smem[];
  __shared__ int next;
  griddep_start();
  for (int s = int(blockIdx.x); s < a.nseg;) {
    // the next segment's number is on its way while this one is worked on
    const int mine = threadIdx.x == 0 ? int(gridDim.x) + atomicAdd(a.counter, 1) : 0;
    const TriSeg g = a.segs[s];
    TriArgs t{};
    t.p0 = a.pos + g.first;
    t.p1 = a.prm + g.first;
    t.part = a.part + g.first;
    t.stride = a.stride;
    t.eps2 = g.eps2;
    t.geom.n = g.n;
    if (g.law == 0)
      tri_run<TriGrav<false, PRECISE, false>, kTriBatchGrav, true>(t, g.row, g.d0, g.d1, g.o0, g.o1,
                                                            g.slot, nullptr, tri_smem);
    else if (g.law == 1)
      tri_run<TriLjc<false, false, PRECISE>, kTriBatchLjc, true>(t, g.row, g.d0, g.d1, g.o0, g.o1,
                                                                 g.slot, nullptr, tri_smem);
    else
      tri_run<TriLjc<true, false, PRECISE>, kTriBatchLjc, true>(t, g.row, g.d0, g.d1, g.o0, g.o1,
                                                                g.slot, nullptr, tri_smem);
    if (threadIdx.x == 0) next = mine;
    __syncthreads();
    s = next;
    __syncthreads();
  }
}

}  // namespace nbody
