// direct_impl.h -- launch of one instantiation of direct_kernel.cuh.
#pragma once

#include <atomic>

#include "direct_tiles.h"
#include "tiles.h"

namespace nbody {

template <class L, int H, int U>
inline cudaError_t direct_go(const DirectArgs &a, cudaStream_t s) {
  auto k = direct_kernel<L, H, U>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned((a.n_t + 2 * H - 1) / (2 * H) * a.slices));
  cfg.blockDim = dim3(kDirectThreads);
  cfg.stream = s;
  // a thread's folded sums, where its slice has more than one fold
  const int blocks = (a.n + kDirectThreads - 1) / kDirectThreads;
  if ((blocks + a.slices - 1) / a.slices > direct_chain<L>()) {
    constexpr size_t kBytes = size_t(H) * L::kSums * kDirectThreads * sizeof(float2);
    cfg.dynamicSmemBytes = kBytes;
    static std::atomic<bool> opted[kMaxDevicesTile];
    int dev = 0;
    const bool known = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevicesTile;
    if (!known || !opted[dev].load(std::memory_order_acquire)) {
      const cudaError_t e = cudaFuncSetAttribute(
          k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kBytes));
      if (e != cudaSuccess) return e;
      if (known) opted[dev].store(true, std::memory_order_release);
    }
  }
  cudaLaunchAttribute attr[2];
  unsigned na = 0;
  if (a.slices > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = unsigned(a.slices);
    attr[na].val.clusterDim.y = 1;
    attr[na++].val.clusterDim.z = 1;
  }
  if (a.pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na++].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, k, a);
}

// U: sources on their way per thread (the L2 latency of about 700 cycles against the
// time of one source; 16 targets of gravity with 1 / 2 / 4: 61 / 86 / 49 us for 1500
// targets of 65536). Without BIG_POT potentials take 8 targets (16 would leave one CTA on an SM;
// the same sums: their order depends on the slices alone).
template <template <bool, bool> class LAW, int U, bool BIG_POT>
inline cudaError_t direct_law(const DirectArgs &a, bool big, bool pot, bool precise,
                              cudaStream_t s) {
  if (pot) {
    if constexpr (BIG_POT) {
      if (big)
        return precise ? direct_go<LAW<true, true>, 8, U>(a, s)
                       : direct_go<LAW<true, false>, 8, U>(a, s);
    }
    return precise ? direct_go<LAW<true, true>, 4, U>(a, s)
                   : direct_go<LAW<true, false>, 4, U>(a, s);
  }
  if (big)
    return precise ? direct_go<LAW<false, true>, 8, U>(a, s)
                   : direct_go<LAW<false, false>, 8, U>(a, s);
  return precise ? direct_go<LAW<false, true>, 4, U>(a, s)
                 : direct_go<LAW<false, false>, 4, U>(a, s);
}

}  // namespace nbody
