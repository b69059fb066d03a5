// Binary64 (reference) instantiations of the persistent stepper.  Built with
// FMA contraction off (-fmad=false) so that every operation is rounded exactly
// as written.
#include "stepper.cuh"
#include "stepper_few.cuh"
#include "stepper_launch.h"

namespace fpt {
namespace {

constexpr int kBlock64 = 16;  // steps of a scheduling block, whatever k_steps folds

template <int MODEL, bool WALL, int FOLD>
cudaError_t launch(const StepperParams& a, int grid, int block, cudaStream_t stream) {
    const size_t smem = stepper_table_bytes(a.n_sets) + (size_t)(block / 32) * warp_smem_bytes<double, FPT_PREC_F64>();
    stepper_kernel<double, FPT_PREC_F64, MODEL, WALL, kBlock64, FOLD><<<grid, block, smem, stream>>>(a);
    return cudaGetLastError();
}

template <int MODEL, bool WALL, int FOLD>
cudaError_t launch_few(const StepperParams& a, int grid, int block, cudaStream_t stream) {
    stepper_few_kernel<double, FPT_PREC_F64, MODEL, WALL, FOLD>
        <<<grid, block, stepper_table_bytes(a.n_sets) + few_smem_bytes<double, FPT_PREC_F64>(), stream>>>(a);
    return cudaGetLastError();
}

template <int MODEL, bool WALL, int FOLD>
StepperKernel make() {
    StepperKernel k{(const void*)stepper_kernel<double, FPT_PREC_F64, MODEL, WALL, kBlock64, FOLD>,
                    warp_smem_bytes<double, FPT_PREC_F64>(), &launch<MODEL, WALL, FOLD>};
    if constexpr (MODEL == FPT_MODEL_QUADRATIC) {
        k.few_func = (const void*)stepper_few_kernel<double, FPT_PREC_F64, MODEL, WALL, FOLD>;
        k.few_per_sm = 4;
        k.few_smem = few_smem_bytes<double, FPT_PREC_F64>();
        k.few_launch = &launch_few<MODEL, WALL, FOLD>;
    }
    return k;
}

template <int MODEL, bool WALL>
StepperKernel by_ks(int ks) {
    switch (ks) {
        case 4: return make<MODEL, WALL, 4>();
        case 8: return make<MODEL, WALL, 8>();
        default: return StepperKernel{};
    }
}

template <int MODEL>
StepperKernel by_wall(bool wall, int ks) {
    return wall ? by_ks<MODEL, true>(ks) : by_ks<MODEL, false>(ks);
}

}  // namespace

StepperKernel stepper_f64(int model, bool wall, int k_steps) {
    if (model == FPT_MODEL_QUADRATIC) return by_wall<FPT_MODEL_QUADRATIC>(wall, k_steps);
    if (model == FPT_MODEL_CONSTANT) return by_wall<FPT_MODEL_CONSTANT>(wall, k_steps);
    if (model == FPT_MODEL_POLYNOMIAL) return by_wall<FPT_MODEL_POLYNOMIAL>(wall, k_steps);
    if (model == kModelPowReal) return by_wall<kModelPowReal>(wall, k_steps);
    return StepperKernel{};
}

}  // namespace fpt
