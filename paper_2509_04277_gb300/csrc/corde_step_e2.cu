// Step-kernel instantiations with 2 elements per thread.
#include "corde_step_launch.cuh"

namespace corde {

const StepVariant kStepVariantsE2[] = {step_variant<2, 32>(), step_variant<2, 64>(), step_variant<2, 128>(),
                                         step_variant<2, 256>(), step_variant<2, 512>()};
const int kNumStepVariantsE2 = 5;

}  // namespace corde
