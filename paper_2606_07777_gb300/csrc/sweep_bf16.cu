// sweep_bf16.cu -- the one-family sweep for BF16 values.
#include "sweep_kernels.cuh"
#include "sweep_policies.cuh"

namespace dlm {

cudaError_t sweep_prepare_bf16(int smem_limit) { return prepare_policy<Narrow<BF16Pair>>(smem_limit); }
cudaError_t launch_sweep_bf16(const SweepLaunch& L, bool stats) { return launch_policy<Narrow<BF16Pair>>(L, stats); }

}  // namespace dlm
