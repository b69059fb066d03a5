// Binary32-state instantiations of the persistent stepper with the power-law
// bias B = A_p phi^p (§3.4 Eq. (26)): p in 0..4 specialised, any other real p
// through exp2/log2; folds of 32 steps.
#define FPT_NO_F64
#include "stepper.cuh"
#include "stepper_few.cuh"
#include "stepper_launch.h"

namespace fpt {
namespace {

constexpr int kPowKS = 32;

template <int PREC, int MODEL, bool WALL, bool BENCH, int KS = 2 * kPowKS>
cudaError_t launch(const StepperParams& a, int grid, int block, cudaStream_t stream) {
    const size_t smem = stepper_table_bytes(a.n_sets) +
                        (size_t)(block / 32) * (warp_smem_bytes<float, PREC>() + a.bench * kParkWords * 4);
    stepper_kernel<float, PREC, MODEL, WALL, KS, kPowKS, BENCH><<<grid, block, smem, stream>>>(a);
    return cudaGetLastError();
}

template <int PREC, int MODEL, bool WALL>
cudaError_t launch_few(const StepperParams& a, int grid, int block, cudaStream_t stream) {
    stepper_few_kernel<float, PREC, MODEL, WALL, kPowKS><<<grid, block, stepper_table_bytes(a.n_sets) + few_smem_bytes<float, PREC>(), stream>>>(a);
    return cudaGetLastError();
}

template <int PREC, int MODEL, bool WALL>
StepperKernel make() {
    StepperKernel k{(const void*)stepper_kernel<float, PREC, MODEL, WALL, 2 * kPowKS, kPowKS, false>,
                    warp_smem_bytes<float, PREC>(), &launch<PREC, MODEL, WALL, false>};
    k.bench_func = (const void*)stepper_kernel<float, PREC, MODEL, WALL, 2 * kPowKS, kPowKS, true>;
    k.bench_launch = &launch<PREC, MODEL, WALL, true>;
    k.few_func = (const void*)stepper_few_kernel<float, PREC, MODEL, WALL, kPowKS>;
    k.few_smem = few_smem_bytes<float, PREC>();
    k.few_launch = &launch_few<PREC, MODEL, WALL>;
    k.brief_func = (const void*)stepper_kernel<float, PREC, MODEL, WALL, kPowKS, kPowKS, false>;
    k.brief_launch = &launch<PREC, MODEL, WALL, false, kPowKS>;
    k.fold = kPowKS;
    return k;
}

template <int PREC, bool WALL>
StepperKernel by_power(int p_code) {
    switch (p_code) {
        case 0: return make<PREC, kModelPow + 0, WALL>();
        case 1: return make<PREC, kModelPow + 1, WALL>();
        case 2: return make<PREC, kModelPow + 2, WALL>();
        case 3: return make<PREC, kModelPow + 3, WALL>();
        case 4: return make<PREC, kModelPow + 4, WALL>();
        default: return make<PREC, kModelPowReal, WALL>();
    }
}

template <int PREC>
StepperKernel by_wall(bool wall, int p_code) {
    return wall ? by_power<PREC, true>(p_code) : by_power<PREC, false>(p_code);
}

}  // namespace

int pow_code(double p) {
    for (int k = 0; k <= 4; ++k)
        if (p == (double)k) return k;
    return kModelPowReal - kModelPow;
}

StepperKernel stepper_f32_pow(int precision, double p, bool wall, int k_steps) {
    if (k_steps != kPowKS) return StepperKernel{};
    if (precision == FPT_PREC_F32_KAHAN) return by_wall<FPT_PREC_F32_KAHAN>(wall, pow_code(p));
    if (precision == FPT_PREC_F32_F64ACC) return by_wall<FPT_PREC_F32_F64ACC>(wall, pow_code(p));
    return StepperKernel{};
}

}  // namespace fpt
