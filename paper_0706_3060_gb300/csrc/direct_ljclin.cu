// direct_ljclin.cu -- one-launch forces on few targets: LJ + Coulomb, linear dielectric (Table 1).
#include "direct_impl.h"

namespace nbody {

namespace {
template <bool POT, bool PRECISE>
using Law = TriLjc<true, POT, PRECISE>;
}

cudaError_t direct_ljclin(const DirectArgs &a, bool big, bool pot, bool precise, cudaStream_t s) {
  return direct_law<Law, 2, true>(a, big, pot, precise, s);
}

}  // namespace nbody
