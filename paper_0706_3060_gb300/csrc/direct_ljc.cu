// direct_ljc.cu -- one-launch forces on few targets: LJ + Coulomb, constant dielectric (Table 1).
#include "direct_impl.h"

namespace nbody {

namespace {
template <bool POT, bool PRECISE>
using Law = TriLjc<false, POT, PRECISE>;
}

cudaError_t direct_ljc(const DirectArgs &a, bool big, bool pot, bool precise, cudaStream_t s) {
  return direct_law<Law, 2, true>(a, big, pot, precise, s);
}

}  // namespace nbody
