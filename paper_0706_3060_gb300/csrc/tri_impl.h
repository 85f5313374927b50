// tri_impl.h -- host side of one streamed triangle kernel: per-device opt-in to its
// shared memory and the launch.
#pragma once

#include "tiles.h"
#include "tri_tiles.h"

namespace nbody {

template <class L, int H, int MINB, bool AHEAD>
inline cudaError_t tri_go(const TriArgs &a, cudaStream_t s) {
  auto k = tri_kernel<L, H, MINB, AHEAD>;
  static std::atomic<bool> opted[kMaxDevicesTile];
  int dev = 0;
  const bool known = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevicesTile;
  if (!known || !opted[dev].load(std::memory_order_acquire)) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               int(TriTile<L, H>::kSmemBytes));
    if (e != cudaSuccess) return e;
    if (known) opted[dev].store(true, std::memory_order_release);
  }
  return launch_kernel(k, a.geom.nshare, kTriThreads, TriTile<L, H>::kSmemBytes, s, a.pdl != 0, a);
}

// LAW<POT, PRECISE>: the law's pair functions.
template <template <bool, bool> class LAW, int H, int MINB, bool AHEAD>
struct TriImpl {
  static cudaError_t launch(const TriArgs &a, bool pot, bool precise, cudaStream_t s) {
    if (pot)
      return precise ? tri_go<LAW<true, true>, H, MINB, AHEAD>(a, s)
                     : tri_go<LAW<true, false>, H, MINB, AHEAD>(a, s);
    return precise ? tri_go<LAW<false, true>, H, MINB, AHEAD>(a, s)
                   : tri_go<LAW<false, false>, H, MINB, AHEAD>(a, s);
  }
  static TriDesc desc() { return TriDesc{H, MINB, LAW<true, false>::kLow, &launch}; }
};

}  // namespace nbody
