// tri_vjp.cu -- streamed triangle and direct kernels of acceleration + jerk (Table 1
// "Gravity (accel & jerk)") and of the gravity and LJC force VJPs.
//
// What bounds them: the packed FP32 unit (33, 35 and 64 operations per pair; 0.72, 0.74
// and 0.81 of its rate at 32768), of which the three-operand multiply-adds take a sixth
// more than the others. Rows of 256 targets: 231, 196 and 255 registers at two CTAs per
// SM; rows of 384 spill (jerk: 642 us at 32768 against 614) or gain nothing (gravity VJP:
// 47.2 us against 44.3 at 8192, 163 against 162 at 16384, 635 against 629 at 32768), rows
// of 128 move the sources twice as often (LJC VJP: 1153 us at 32768 against 1065).
// Per step with the finalize, against the block-pair tiles (us):
//   Hermite 8192 45.8 / 79.2, 16384 161 / 215, 32768 616 / 685
//   gravity reverse step 4096 20.4 / 27.4, 8192 47.3 / 61.7, 16384 166 / 185
//   LJC reverse step 4096 32.5 / 46.3, 8192 77.6 / 105, 32768 1077 / 2186
// The next group's sources are on their way in all but jerk (600 us at 32768 without,
// 609 with).
#include "api_common.h"
#include "direct_impl.h"
#include "tri_impl.h"
#include "tri_vjp_laws.cuh"

namespace nbody {
namespace {

template <class L, int H, bool AHEAD>
cudaError_t tri_one(const TriArgs &a, bool, bool, cudaStream_t s) {
  return tri_go<L, H, 2, AHEAD>(a, s);
}

}  // namespace

// Gravity VJPs that take the finer sums (tri_kernel.cuh, Sums): from 4096 particles to 8191
// the one-sided tile of that size was nearer to the 64-bit values than the plain sums (mass
// terms at 6500: 1.70e-7 against 1.89e-7), below and above the tiles are not (4095: 1.85e-7
// against 1.57e-7, 8192: 2.11e-7 against 1.99e-7).
inline bool vjp_fine(int64_t n) { return n >= 4096 && n < 8192; }

const TriDesc *tri_vjp(int table, int64_t n) {
  static const TriDesc jerk{4, 2, false, &tri_one<TriJerk, 4, false>};
  static const TriDesc fine{4, 2, false, &tri_one<TriGravVjp<true>, 4, true>};
  static const TriDesc grav{4, 2, false, &tri_one<TriGravVjp<false>, 4, true>};
  static const TriDesc ljc{4, 2, false, &tri_one<TriLjcVjp<false>, 4, true>};
  static const TriDesc ljclin{4, 2, false, &tri_one<TriLjcVjp<true>, 4, true>};
  switch (table) {
    case kTableJerk: return &jerk;
    case kTableVjpGrav: return vjp_fine(n) ? &fine : &grav;
    case kTableVjpLJC: return &ljc;
    case kTableVjpLJCLin: return &ljclin;
  }
  return nullptr;
}

cudaError_t direct_vjp(int table, const DirectArgs &a, cudaStream_t s) {
  switch (table) {
    case kTableJerk: return direct_go<TriJerk, 4, 2>(a, s);
    case kTableVjpGrav: return direct_go<TriGravVjp<false>, 4, 2>(a, s);
    case kTableVjpLJC: return direct_go<TriLjcVjp<false>, 2, 2>(a, s);
    case kTableVjpLJCLin: return direct_go<TriLjcVjp<true>, 2, 2>(a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace nbody
