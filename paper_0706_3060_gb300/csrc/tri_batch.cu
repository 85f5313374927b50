// tri_batch.cu -- launch of the batched streamed triangle kernel.
#include <algorithm>
#include <atomic>

#include "tiles.h"
#include "tri_batch.cuh"

namespace nbody {
namespace {

template <bool PRECISE>
cudaError_t go(const TriBatchArgs &a, cudaStream_t s) {
  auto k = tri_batch_kernel<PRECISE>;
  constexpr size_t kSmem =
      std::max(TriTile<TriGrav<false, PRECISE, false>, kTriBatchGrav>::kSmemBytes,
               TriTile<TriLjc<false, false, PRECISE>, kTriBatchLjc>::kSmemBytes);
  static std::atomic<bool> opted[kMaxDevicesTile];
  int dev = 0;
  const bool known = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevicesTile;
  if (!known || !opted[dev].load(std::memory_order_acquire)) {
    const cudaError_t e =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmem));
    if (e != cudaSuccess) return e;
    if (known) opted[dev].store(true, std::memory_order_release);
  }
  return launch_kernel(k, a.grid, kTriThreads, kSmem, s, a.pdl != 0, a);
}

}  // namespace

cudaError_t tri_batch(const TriBatchArgs &a, bool precise, cudaStream_t s) {
  return precise ? go<true>(a, s) : go<false>(a, s);
}
int tri_batch_per_sm() { return 2; }

}  // namespace nbody
