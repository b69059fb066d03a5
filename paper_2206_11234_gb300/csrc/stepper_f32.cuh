// Binary32-state instantiations of the persistent stepper, for one of the two
// log-weight sums per translation unit.
#pragma once
#define FPT_NO_F64
#include "stepper.cuh"
#include "stepper_few.cuh"
#include "stepper_launch.h"

namespace fpt {
namespace {

constexpr int kBlock32 = 64;  // steps of a scheduling block, whatever k_steps folds

template <int PREC, int MODEL, bool WALL, int FOLD, bool BENCH, int KS = kBlock32>
cudaError_t launch(const StepperParams& a, int grid, int block, cudaStream_t stream) {
    const size_t smem = stepper_table_bytes(a.n_sets) +
                        (size_t)(block / 32) * (warp_smem_bytes<float, PREC>() + a.bench * kParkWords * 4);
    stepper_kernel<float, PREC, MODEL, WALL, KS, FOLD, BENCH><<<grid, block, smem, stream>>>(a);
    return cudaGetLastError();
}

template <int PREC, int MODEL, bool WALL, int FOLD>
cudaError_t launch_few(const StepperParams& a, int grid, int block, cudaStream_t stream) {
    stepper_few_kernel<float, PREC, MODEL, WALL, FOLD><<<grid, block, stepper_table_bytes(a.n_sets) + few_smem_bytes<float, PREC>(), stream>>>(a);
    return cudaGetLastError();
}

template <int PREC, int MODEL, bool WALL, int FOLD>
StepperKernel make() {
    StepperKernel k{(const void*)stepper_kernel<float, PREC, MODEL, WALL, kBlock32, FOLD, false>,
                    warp_smem_bytes<float, PREC>(), &launch<PREC, MODEL, WALL, FOLD, false>};
    if constexpr (MODEL == FPT_MODEL_QUADRATIC || MODEL == kModelPolyLow) {
        k.bench_func = (const void*)stepper_kernel<float, PREC, MODEL, WALL, kBlock32, FOLD, true>;
        k.bench_launch = &launch<PREC, MODEL, WALL, FOLD, true>;
        k.few_func = (const void*)stepper_few_kernel<float, PREC, MODEL, WALL, FOLD>;
        k.few_smem = few_smem_bytes<float, PREC>();
        k.few_launch = &launch_few<PREC, MODEL, WALL, FOLD>;
    }
    if constexpr (FOLD < kBlock32) {
        k.brief_func = (const void*)stepper_kernel<float, PREC, MODEL, WALL, FOLD, FOLD, false>;
        k.brief_launch = &launch<PREC, MODEL, WALL, FOLD, false, FOLD>;
        k.fold = FOLD;
        if (MODEL == FPT_MODEL_POLYNOMIAL) k.brief_warps = 16;
    }
    return k;
}

template <int PREC, int MODEL, bool WALL>
StepperKernel by_ks(int ks) {
    switch (ks) {
        case 16: return make<PREC, MODEL, WALL, 16>();
        case 32: return make<PREC, MODEL, WALL, 32>();
        case 64: return make<PREC, MODEL, WALL, 64>();
        default: return StepperKernel{};
    }
}

template <int PREC, int MODEL>
StepperKernel by_wall(bool wall, int ks) {
    return wall ? by_ks<PREC, MODEL, true>(ks) : by_ks<PREC, MODEL, false>(ks);
}

template <int PREC>
StepperKernel by_model(int model, bool wall, int ks) {
    if (model == FPT_MODEL_QUADRATIC) return by_wall<PREC, FPT_MODEL_QUADRATIC>(wall, ks);
    if (model == FPT_MODEL_CONSTANT) return by_wall<PREC, FPT_MODEL_CONSTANT>(wall, ks);
    if (model == FPT_MODEL_POLYNOMIAL) return by_wall<PREC, FPT_MODEL_POLYNOMIAL>(wall, ks);
    if (model == kModelPolyLow) return by_wall<PREC, kModelPolyLow>(wall, ks);
    return StepperKernel{};
}

}  // namespace

}  // namespace fpt
