// sweep.cu -- dispatch of the one-family sweep (sweep_kernels.cuh) over the
// value layouts, and its shared-memory sizes.
#include <algorithm>

#include "dlm_impl.cuh"
#include "sweep_policies.cuh"

namespace dlm {

size_t sweep_smem_bytes(int smemJ, bool stats) { return sweep_stats_smem_bytes(smemJ, stats ? smemJ : 0); }

size_t sweep_stats_smem_bytes(int smemJ, int win) {
  const size_t J = static_cast<size_t>(smemJ);
  const size_t acc = win > 0 ? 3 * static_cast<size_t>(win) : J;
  return acc * 8 + ((J + 1) & ~static_cast<size_t>(1)) * 4 + 32 * 8;
}

int sweep_stats_window(int smemJ) {
  const size_t lim = sweep_smem_limit();
  if (sweep_stats_smem_bytes(smemJ, smemJ) <= lim) return smemJ;
  const size_t fixed = sweep_stats_smem_bytes(smemJ, 0) - static_cast<size_t>(smemJ) * 8;
  if (fixed >= lim) return 0;
  return static_cast<int>(std::min<size_t>((lim - fixed) / 24, static_cast<size_t>(smemJ)));
}

size_t sweep_smem_limit() {
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return 0;
  return optin > 1024 ? static_cast<size_t>(optin - 1024) : 0;  // room for static shared memory
}

cudaError_t sweep_prepare(bool bf16) {
  const int lim = static_cast<int>(sweep_smem_limit());
  cudaError_t e = bf16 ? sweep_prepare_bf16(lim) : sweep_prepare_f32(lim);
  if (e == cudaSuccess) e = bf16 ? sweep_prepare_bf16_count(lim) : sweep_prepare_f32_count(lim);
  return e != cudaSuccess ? e : sweep_short_prepare(bf16);
}

cudaError_t launch_sweep(const SweepLaunch& L, bool stats, bool bf16) {
  // iteration sweeps of a handle with the short-row sweep on take it alone
  if (!stats && L.short_rows) return launch_sweep_short(L, bf16);
  if (L.count) return bf16 ? launch_sweep_bf16_count(L, stats) : launch_sweep_f32_count(L, stats);
  return bf16 ? launch_sweep_bf16(L, stats) : launch_sweep_f32(L, stats);
}

}  // namespace dlm
