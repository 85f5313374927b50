// tri_ljclin.cu -- streamed triangle kernels for Lennard-Jones plus Coulomb with a linear
// dielectric (Table 1).
#include "tri_impl.h"

namespace nbody {

namespace {
template <bool POT, bool PRECISE>
using Law = TriLjc<true, POT, PRECISE>;
}

const TriDesc *tri_ljclin(int64_t n) {
  // As for gravity. Kernel times (us), rows of 256 / 384: 16.3 / 18.0 at 5000, 33.0 / 34.2
  // at 8192, 69.0 / 67.6 at 12288, 117.1 / 116.0 at 16384, 453 / 446 at 32768, 3367 / 3302
  // at 90000.
  static const TriDesc small = TriImpl<Law, 4, 2, true>::desc();
  static const TriDesc large = TriImpl<Law, 6, 2, true>::desc();
  return n < 12288 ? &small : &large;
}

}  // namespace nbody
