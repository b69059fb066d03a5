// Binary32 stepper with the binary64 log-weight sum, and the choice between the two.
#include "stepper_f32.cuh"

namespace fpt {

StepperKernel stepper_f32_kahan(int model, bool wall, int k_steps);

StepperKernel stepper_f32(int precision, int model, bool wall, int k_steps) {
    if (precision == FPT_PREC_F32_KAHAN) return stepper_f32_kahan(model, wall, k_steps);
    if (precision == FPT_PREC_F32_F64ACC) return by_model<FPT_PREC_F32_F64ACC>(model, wall, k_steps);
    return StepperKernel{};
}

}  // namespace fpt
