// sweep_policies.cuh -- the one-family sweep's entry points per value layout
// (each defined in a translation unit of its own); _count: instances with a
// global count constraint.
#pragma once

#include "dlm_impl.cuh"

namespace dlm {

cudaError_t sweep_prepare_f32(int smem_limit);
cudaError_t sweep_prepare_bf16(int smem_limit);
cudaError_t sweep_prepare_f32_count(int smem_limit);
cudaError_t sweep_prepare_bf16_count(int smem_limit);
cudaError_t launch_sweep_f32(const SweepLaunch& L, bool stats);
cudaError_t launch_sweep_bf16(const SweepLaunch& L, bool stats);
cudaError_t launch_sweep_f32_count(const SweepLaunch& L, bool stats);
cudaError_t launch_sweep_bf16_count(const SweepLaunch& L, bool stats);

}  // namespace dlm
