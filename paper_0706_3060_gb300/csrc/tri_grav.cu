// tri_grav.cu -- streamed triangle kernels for softened gravity (Eq. 1, Table 1
// "Gravity (accel)").
#include "tri_impl.h"

namespace nbody {

namespace {
template <bool POT, bool PRECISE>
using Plain = TriGrav<POT, PRECISE, false>;
template <bool POT, bool PRECISE>
using Fine = TriGrav<POT, PRECISE, true>;
}  // namespace

const TriDesc *tri_grav(int64_t n) {
  // Rows of 384 targets leave a small system more units for equal shares; rows of 512
  // spend fewer instructions per pair on moving the sources. Kernel times (us) with plain
  // sums, 384 / 512: 13.3 / 13.6 at 5000, 24.0 / 24.6 at 8192, 46.1 / 45.5 at 12288, 77.5 / 76.6 at
  // 16384, 294 / 287 at 32768, 2170 / 2116 at 90000 (rows of 256: 15.7, 24.1, 48.5, 82.4,
  // 314, 2328).
  // The finer sums (tri_kernel.cuh, Sums) from 8192 on: below, the tiles' errors were twice
  // those of the plain ones (potential at 5000: 5.8e-8 against 2.7e-8), which take 0.3 us
  // less a step and 2 us less with the potential.
  static const TriDesc few = TriImpl<Plain, 6, 2, true>::desc();
  static const TriDesc small = TriImpl<Fine, 6, 2, true>::desc();
  static const TriDesc large = TriImpl<Fine, 8, 2, true>::desc();
  return n < 8192 ? &few : n < 12288 ? &small : &large;
}

}  // namespace nbody
