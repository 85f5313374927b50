// tri_ljc.cu -- streamed triangle kernels for Lennard-Jones plus Coulomb with a constant
// dielectric (Table 1).
#include "tri_impl.h"

namespace nbody {

namespace {
template <bool POT, bool PRECISE>
using Law = TriLjc<false, POT, PRECISE>;
}

const TriDesc *tri_ljc(int64_t n) {
  // As for gravity. Kernel times (us), rows of 256 / 384: 16.2 / 17.6 at 5000, 32.6 / 33.6
  // at 8192, 68.4 / 65.6 at 12288, 116.0 / 112.5 at 16384, 449 / 432 at 32768, 3342 / 3200
  // at 90000.
  static const TriDesc small = TriImpl<Law, 4, 2, true>::desc();
  static const TriDesc large = TriImpl<Law, 6, 2, true>::desc();
  return n < 12288 ? &small : &large;
}

}  // namespace nbody
