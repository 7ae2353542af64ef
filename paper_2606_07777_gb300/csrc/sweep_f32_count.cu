// sweep_f32_count.cu -- the one-family sweep for FP32 values and a count constraint.
#include "sweep_kernels.cuh"
#include "sweep_policies.cuh"

namespace dlm {

cudaError_t sweep_prepare_f32_count(int smem_limit) { return prepare_policy<Counted<Narrow<F32Pair>>>(smem_limit); }
cudaError_t launch_sweep_f32_count(const SweepLaunch& L, bool stats) {
  return launch_policy<Counted<Narrow<F32Pair>>>(L, stats);
}

}  // namespace dlm
