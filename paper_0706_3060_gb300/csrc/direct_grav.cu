// direct_grav.cu -- one-launch forces on few targets: softened gravity (Eq. 1).
#include "direct_impl.h"

namespace nbody {

namespace {
template <bool POT, bool PRECISE>
using Law = TriGrav<POT, PRECISE, true>;
}

cudaError_t direct_grav(const DirectArgs &a, bool big, bool pot, bool precise, cudaStream_t s) {
  return direct_law<Law, 4, false>(a, big, pot, precise, s);
}

}  // namespace nbody
