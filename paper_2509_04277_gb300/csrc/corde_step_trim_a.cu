// Step-kernel instantiations with four elements per thread and thread counts between the plan's
// powers of two (96 to 224): a bin of rods takes the smallest block that holds them.
#include "corde_step_launch.cuh"

namespace corde {

const StepVariant kStepTrimA[] = {step_variant<4, 96>(), step_variant<4, 160>(), step_variant<4, 192>(), step_variant<4, 224>()};
const int kNumStepTrimA = 4;

}  // namespace corde
