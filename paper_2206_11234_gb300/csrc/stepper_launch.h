// Type-erased access to the stepper instantiations (one per precision, model,
// wall and block length), used by the C ABI layer.
#pragma once
#include <cuda_runtime.h>

#include "stepper_types.h"

namespace fpt {

struct StepperKernel {
    const void* func = nullptr;  // for occupancy queries; nullptr = no such instantiation
    int warp_smem_bytes = 0;     // dynamic shared memory per warp (replay queue + parking)
    cudaError_t (*launch)(const StepperParams&, int grid, int block, cudaStream_t stream) = nullptr;
    // the same with runs that take turns (StepperParams::bench > 0), if there is one
    const void* bench_func = nullptr;
    cudaError_t (*bench_launch)(const StepperParams&, int grid, int block, cudaStream_t stream) = nullptr;
    // the stepper for few runs (stepper_few.cuh; blocks of kFewThreads, 32 runs each), if there is one,
    // and up to how many of its blocks per SM it is the faster
    const void* few_func = nullptr;
    cudaError_t (*few_launch)(const StepperParams&, int grid, int block, cudaStream_t stream) = nullptr;
    int few_per_sm = 3;
    int few_smem = 0;  // dynamic shared memory of a block but for the set table
    // the same in scheduling blocks of one fold, for brief runs, if there is one, and from how many
    // warps per SM on it is the faster whatever the runs' length
    const void* brief_func = nullptr;
    int fold = 0;  // steps of its block
    unsigned long long brief_warps = 1ull << 40;
    cudaError_t (*brief_launch)(const StepperParams&, int grid, int block, cudaStream_t stream) = nullptr;
};

inline size_t stepper_smem(const StepperKernel& k, int block, int n_sets, int bench) {
    return stepper_table_bytes(n_sets) + (size_t)(block / 32) * (size_t)(k.warp_smem_bytes + bench * kParkWords * 4);
}

// k_steps (steps of a fold) with an instantiation: binary32 16/32/64, binary64 4/8; the
// power-law bias (model = kModelPowReal in binary64): binary32 32, binary64 4/8.
StepperKernel stepper_f32(int precision, int model, bool wall, int k_steps);
StepperKernel stepper_f64(int model, bool wall, int k_steps);
StepperKernel stepper_f32_pow(int precision, double p, bool wall, int k_steps);

}  // namespace fpt
