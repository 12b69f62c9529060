// Step-kernel instantiations with 4 elements per thread.
#include "corde_step_launch.cuh"

namespace corde {

const StepVariant kStepVariantsE4[] = {step_variant<4, 32>(), step_variant<4, 64>(), step_variant<4, 128>(),
                                         step_variant<4, 256>(), step_variant<4, 512>()};
const int kNumStepVariantsE4 = 5;

}  // namespace corde
