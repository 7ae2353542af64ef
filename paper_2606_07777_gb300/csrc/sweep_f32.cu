// sweep_f32.cu -- the one-family sweep for FP32 values.
#include "sweep_kernels.cuh"
#include "sweep_policies.cuh"

namespace dlm {

cudaError_t sweep_prepare_f32(int smem_limit) { return prepare_policy<Narrow<F32Pair>>(smem_limit); }
cudaError_t launch_sweep_f32(const SweepLaunch& L, bool stats) { return launch_policy<Narrow<F32Pair>>(L, stats); }

}  // namespace dlm
