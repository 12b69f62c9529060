// Step-kernel instantiations with four elements per thread and thread counts between the plan's
// powers of two (416 to 480): a bin of rods takes the smallest block that holds them.
#include "corde_step_launch.cuh"

namespace corde {

const StepVariant kStepTrimC[] = {step_variant<4, 416>(), step_variant<4, 448>(), step_variant<4, 480>()};
const int kNumStepTrimC = 3;

}  // namespace corde
