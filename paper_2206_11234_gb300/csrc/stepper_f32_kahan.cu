// Binary32 stepper with the compensated binary32 log-weight sum.
#include "stepper_f32.cuh"

namespace fpt {

StepperKernel stepper_f32_kahan(int model, bool wall, int k_steps) {
    return by_model<FPT_PREC_F32_KAHAN>(model, wall, k_steps);
}

}  // namespace fpt
