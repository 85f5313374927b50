// tri_ljc.cu -- streamed triangle kernels for Lennard-Jones plus Coulomb with a constant
// dielectric (Table 1).
#include "tri_impl.h"

namespace nbody {

namespace {
template <bool POT, bool PRECISE>
using Law = TriLjc<false, POT, PRECISE>;
}

const TriDesc *tri_ljc(int64_t n) {
  // As for gravity. Kernel times (us, constant dielectric), rows of 256 / 384: 36.9 /
  // 38.9 at 8192, 122.8 / 118.8 at 16384, 1043 / 1003 at 50021, 3343 / 3208 at 90000.
  static const TriDesc small = TriImpl<Law, 4, 2, true>::desc();
  static const TriDesc large = TriImpl<Law, 6, 2, true>::desc();
  return n < 12288 ? &small : &large;
}

}  // namespace nbody
