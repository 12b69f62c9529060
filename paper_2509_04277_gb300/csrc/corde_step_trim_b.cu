// Step-kernel instantiations with four elements per thread and thread counts between the plan's
// powers of two (288 to 384): a bin of rods takes the smallest block that holds them.
#include "corde_step_launch.cuh"

namespace corde {

const StepVariant kStepTrimB[] = {step_variant<4, 288>(), step_variant<4, 320>(), step_variant<4, 352>(), step_variant<4, 384>()};
const int kNumStepTrimB = 4;

}  // namespace corde
