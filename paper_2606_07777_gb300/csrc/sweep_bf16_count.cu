// sweep_bf16_count.cu -- the one-family sweep for BF16 values and a count constraint.
#include "sweep_kernels.cuh"
#include "sweep_policies.cuh"

namespace dlm {

cudaError_t sweep_prepare_bf16_count(int smem_limit) { return prepare_policy<Counted<Narrow<BF16Pair>>>(smem_limit); }
cudaError_t launch_sweep_bf16_count(const SweepLaunch& L, bool stats) {
  return launch_policy<Counted<Narrow<BF16Pair>>>(L, stats);
}

}  // namespace dlm
