// tri_grav.cu -- streamed triangle kernels for softened gravity (Eq. 1, Table 1
// "Gravity (accel)").
#include "tri_impl.h"

namespace nbody {

const TriDesc *tri_grav(int64_t n) {
  // Rows of 384 targets leave a small system more units for equal shares; rows of 512
  // spend fewer instructions per pair on moving the sources. Kernel times (us), 384 /
  // 512: 28.7 / 30.7 at 8192, 82.0 / 84.0 at 16384, 678 / 670 at 50021, 2162 / 2128 at
  // 90000 (rows of 256, four CTAs per SM: 28.7, 85.0, 713, 2274).
  static const TriDesc small = TriImpl<TriGrav, 6, 2, true>::desc();
  static const TriDesc large = TriImpl<TriGrav, 8, 2, true>::desc();
  return n < 32768 ? &small : &large;
}

}  // namespace nbody
