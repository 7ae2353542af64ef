// update.cu -- the O(J) kernels that follow a sweep: the accelerated
// projected dual step with gamma continuation, and the dual objective /
// certified-gap statistics.  Every reduction runs in a fixed order, so results
// are bit-identical from run to run.
#include <math.h>

#include "dlm_impl.cuh"

namespace dlm {
namespace {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ double to_real(unsigned long long v, double inv_scale) {
  return static_cast<double>(static_cast<long long>(v)) * inv_scale;
}

// Sum over the block in a fixed order; result valid in thread 0.
__device__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int k = 0; k < static_cast<int>(blockDim.x >> 5); ++k) s += sh[k];
  __syncthreads();
  return s;
}
// Accelerated projected step (Sec. 4.4; App. B.2), for iteration t at y:
//   G_j    = (A x(y))_j - b_j
//   lam+_j = max(0, y_j + step_j G_j),  step_j = gamma / max_k h_k  (1/L)
//                                         or gamma / h_j (row normalization)
//   theta+ = (1 + sqrt(1 + 4 theta^2)) / 2,  y+ = lam+ + (theta - 1)/theta+ (lam+ - lam)
// and, when iteration t+1 starts a stage with a different gamma, a momentum
// restart (theta = 1, y+ = lam+).  With adaptive restart on, the momentum also
// restarts when the step just taken points against the momentum in the
// step metric: sum_j (lam+_j - y_j) (lam+_j - lam_j) / step_j < 0 (the
// gradient-mapping test of O'Donoghue & Candes 2015, for ascent).
// The iterate lam, y is FP64 (G from the exact fixed-point sum minus b in
// FP64; products and sums rounded separately, no fused multiply-add, as the
// FP64 reference arithmetic of the method takes them); the sweeps read FP32
// copies written here.  The update also records the dual objective at the
// sweep point (Sec. 3.2, Eq. dual):
//   g(y) = sum_i (c x + gamma/2 x^2) + y^T G,
// from the sweep's exact fixed-point objective sum and an FP64 dot product,
// into the trajectory slot t mod kTrajCap.
//
// Grid: CTA x of row y takes coordinates x kUpdChunk .. of instance y, one per
// thread.  The step is bound by latency and by the FP64 rate (two lanes per
// clock and SM, so a warp's FP64 instruction holds the pipe for 16 clocks):
// the chunk is two warps, which spreads the coordinates over the SMs, and the
// scalars of the iteration (a square root and three divisions) are taken by
// one thread of each CTA instead of all of them.  (256 threads each computing
// the scalars: 9-15 us a launch for 100 to 10,000 items; 25 iterations of
// 1M x 1,000 with the adaptive restart and its test kernel went from 2,354 to
// 2,041 us with this kernel and the sweeps' constants taken by one thread.)
// Scalars that need every coordinate -- the dot product of g, the restart
// test, the finiteness flag -- are summed per CTA in a fixed order, written as
// partials, and added in a fixed order by the last CTA of the instance to
// finish (an integer ticket; no CTA waits for another), which also writes the
// new iteration state.  With the adaptive restart every CTA takes the step
// with its momentum, and the last one puts y back to lam when the test fails
// (a rare copy of D values), so the test needs no launch of its own.
constexpr int kUpdChunk = 64;  // coordinates per update CTA (one per thread)
constexpr int kUpdParts = 3;   // partials per CTA: y^T G, restart test, finiteness

// The step's scalars for iteration t of an instance.
struct StepScalars {
  DevState st;
  int64_t s1;
  double gamma1, th1, beta, step0;
  bool stage_restart, test;
};
__device__ __forceinline__ void step_scalars(const UpdInst& U, StepScalars& c) {
  static_assert(sizeof(DevState) % 8 == 0, "read in 64-bit words");
#pragma unroll
  for (int k = 0; k < static_cast<int>(sizeof(DevState) / 8); ++k)
    reinterpret_cast<uint64_t*>(&c.st)[k] = __ldcg(reinterpret_cast<const unsigned long long*>(U.state) + k);
  const int64_t t1 = c.st.iter + 1;
  c.s1 = t1 / U.iters_per_stage;
  c.gamma1 = U.gamma_tab[c.s1 < U.nstages ? c.s1 : U.nstages - 1];
  c.stage_restart = c.gamma1 != c.st.gamma;
  c.th1 = 0.5 * (1.0 + sqrt(1.0 + 4.0 * c.st.theta * c.st.theta));
  c.beta = (c.st.theta - 1.0) / c.th1;
  c.step0 = U.curv_max > 0.0 ? c.st.gamma / U.curv_max : 0.0;
  c.test = U.adaptive_restart && !c.stage_restart;
}

__global__ void __launch_bounds__(kUpdChunk) fista_update_kernel(const UpdInst* __restrict__ tab) {
  constexpr int kW = kUpdChunk / 32;
  __shared__ UpdInst U;
  __shared__ StepScalars c;
  __shared__ double sh[kUpdParts][kW];
  __shared__ int s_last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const UpdInst* __restrict__ I = tab + blockIdx.y;
  if (static_cast<int>(blockIdx.x) >= I->nct) {
    chain_wait();
    return;
  }
  chain_go();  // (the sweep after it waits for this kernel's end)
  for (int k = tid; k < static_cast<int>(sizeof(UpdInst) / 8); k += kUpdChunk)
    reinterpret_cast<uint64_t*>(&U)[k] = __ldg(reinterpret_cast<const uint64_t*>(I) + k);
  __syncthreads();
  // Read ahead of chain_wait(): what the sweep between does not write.  The last
  // update wrote the state, y and lam; it had ended, its writes with it, when this
  // sweep's blocks passed their own chain_wait(), and they let this kernel start only after that
  // (chain_go()).  A wait's promise covers reads after one's own, so these go past L1, which may
  // hold a line of an earlier iteration.
  if (tid == 0) step_scalars(U, c);
  // everything that does not depend on the sweep or on the scalars
  const int NC = U.ncap, D = NC + (U.count_on ? 1 : 0);
  const int j = blockIdx.x * kUpdChunk + tid;
  const bool in = j < D;
  double yj = 0.0, lam0 = 0.0, h = 0.0, bj = 0.0;
  if (in) {
    yj = __ldcg(U.y64 + j);
    lam0 = __ldcg(U.lam64 + j);
    if (U.precondition) h = __ldg(U.curv + j);
    bj = j < NC ? __ldg(U.b + j) : U.count_M;
  }
  __syncthreads();
  double step = c.step0;
  if (U.precondition) step = h > 0.0 ? c.st.gamma / h : 0.0;
  double lg = 0.0, dot = 0.0, bad = 0.0;
  chain_wait();  // the sweep's sums
  if (in) {
    const double G =
        j < NC ? to_real(U.acc[j], U.inv_scaleG) - bj : to_real(*U.cnt, U.inv_scaleN) - bj;
    const double v = __dadd_rn(yj, __dmul_rn(step, G));
    const double ln = v > 0.0 ? v : 0.0;
    lg = static_cast<double>(U.y[j]) * G;
    if (c.test && step > 0.0) dot = __ddiv_rn(__dmul_rn(ln - yj, ln - lam0), step);
    const double yn = c.stage_restart ? ln : __dadd_rn(ln, __dmul_rn(c.beta, ln - lam0));
    U.lam64[j] = ln;
    U.y64[j] = yn;
    U.lam[j] = static_cast<float>(ln);
    U.y[j] = static_cast<float>(yn);
    if (j < NC) U.acc[j] = 0ull;
    if (!isfinite(G) || !isfinite(yj) || !isfinite(yn)) bad = 1.0;
  }
  // sums over the block in a fixed order
  bad = __any_sync(kFull, bad != 0.0) ? 1.0 : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lg += __shfl_down_sync(kFull, lg, o);
    if (c.test) dot += __shfl_down_sync(kFull, dot, o);
  }
  if (lane == 0) {
    sh[0][warp] = lg;
    sh[1][warp] = dot;
    sh[2][warp] = bad;
  }
  __syncthreads();
  if (tid == 0) {
    double p[kUpdParts];
#pragma unroll
    for (int q = 0; q < kUpdParts; ++q) {
      p[q] = sh[q][0];
#pragma unroll
      for (int w = 1; w < kW; ++w) p[q] += sh[q][w];
      U.part[kUpdParts * blockIdx.x + q] = p[q];
    }
    __threadfence();
    const unsigned prev = atomicAdd(U.ticket, 1u);
    s_last = prev == static_cast<unsigned>(U.nct) - 1u;
    if (s_last) *U.ticket = 0u;
  }
  __syncthreads();
  if (!s_last) return;
  // the last CTA of the instance: every partial and every coordinate is visible
  __threadfence();
  double L = 0.0, Dt = 0.0, B = 0.0;
  if (warp == 0) {
    for (int k = lane; k < U.nct; k += 32) {
      L += __ldcg(U.part + kUpdParts * k);
      Dt += __ldcg(U.part + kUpdParts * k + 1);
      B += __ldcg(U.part + kUpdParts * k + 2);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      L += __shfl_down_sync(kFull, L, o);
      if (c.test) Dt += __shfl_down_sync(kFull, Dt, o);
    }
    const bool any_bad = __any_sync(kFull, B != 0.0);
    if (lane == 0) {
      const bool again = c.test && Dt < 0.0;
      s_last = again ? 2 : 1;
      const double g = to_real(*U.objq, U.inv_scaleO) + L;
      *U.objq = 0ull;
      if (U.count_on) *U.cnt_rw = 0ull;
      U.traj[c.st.iter % kTrajCap] = g;
      DevState n = c.st;
      n.iter = c.st.iter + 1;
      n.theta = (c.stage_restart || again) ? 1.0 : c.th1;
      n.gamma = c.gamma1;
      n.stage = static_cast<int32_t>(c.s1 < 0x7fffffff ? c.s1 : 0x7fffffff);
      if (any_bad || !isfinite(g)) n.status |= kStatNumeric;
      *U.state = n;
    }
  }
  if (!c.test) return;
  __syncthreads();
  if (s_last == 2) {  // the momentum restart: y <- lam
    for (int k = tid; k < D; k += kUpdChunk) {
      const double l = __ldcg(U.lam64 + k);
      U.y64[k] = l;
      U.y[k] = static_cast<float>(l);
    }
  }
}

// Dual value and certified gap at the dual point of the certificate sweep
// (Sec. 3.2 Eq. dual; scaled-point gap as defined in the header):
//   G_j = (A x)_j - b_j,  g = sum_i (c x + gamma/2 x^2) + lam^T G,
//   s_j = min(1, b_j / (A x)_j),  P = sum_j s_j (c x)_j + gamma/2 s_j^2 (x^2)_j.
// With a count constraint sum x <= M (dual mu = lam[J]): g gains mu (sum x - M)
// and every s_j is multiplied by t = min(1, M / sum x), which keeps the scaled
// point within the count (sum_j s_j (sum_i x_ij) <= sum x).  With m capacity
// families, s_j = min over the families of min(1, b_kj / (A_k x)_j).
// Grid as the update's: 64 items per CTA, fixed-order partials, the last CTA
// of the instance finishes.  (One CTA of 1,024 threads per instance: 28 us at
// 1,000 items, most of it FP64 issue and serial sums.)
__global__ void __launch_bounds__(kUpdChunk) stats_kernel(const StatsInst* __restrict__ tab,
                                                          const __grid_constant__ StatsInst one) {
  constexpr int kW = kUpdChunk / 32;
  __shared__ StatsInst S;
  __shared__ double sh[kUpdParts][kW];
  __shared__ int s_last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int k = tid; k < static_cast<int>(sizeof(StatsInst) / 8); k += kUpdChunk)
    reinterpret_cast<uint64_t*>(&S)[k] =
        tab ? __ldg(reinterpret_cast<const uint64_t*>(tab + blockIdx.y) + k) : reinterpret_cast<const uint64_t*>(&one)[k];
  __syncthreads();
  const int nct = (S.J + kUpdChunk - 1) / kUpdChunk;
  if (static_cast<int>(blockIdx.x) >= nct) return;
  const double gamma = S.gamma ? *S.gamma : S.gamma_val;
  // count constraint: sum x and the common scaling t = min(1, M / sum x)
  const double total = S.count_on ? to_real(*S.cnt, S.inv_sN) : 0.0;
  const double t = (S.count_on && total > S.count_M) ? S.count_M / total : 1.0;
  double lg = 0.0, P = 0.0, viol = 0.0;
  const int m = S.m > 0 ? S.m : 1;
  const int j = blockIdx.x * kUpdChunk + tid;
  if (j < S.J) {
    double s = t;
    for (int f = 0; f < m; ++f) {
      const int q = f * S.J + j;
      const double Ax = to_real(S.acc[q], S.inv_sG);
      const double G = Ax - S.b[q];
      lg += static_cast<double>(S.lam[q]) * G;
      if (Ax > S.b[q]) s = fmin(s, t * (S.b[q] / Ax));
      viol = fmax(viol, G);
      if (S.grad_out) S.grad_out[q] = static_cast<float>(G);
      S.acc[q] = 0ull;
    }
    const double Cx = to_real(S.accC[j], S.inv_sC);
    const double Qx = to_real(S.accQ[j], S.inv_sQ);
    P = s * Cx + 0.5 * gamma * s * s * Qx;
    S.accC[j] = 0ull;
    S.accQ[j] = 0ull;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lg += __shfl_down_sync(kFull, lg, o);
    P += __shfl_down_sync(kFull, P, o);
    viol = fmax(viol, __shfl_down_sync(kFull, viol, o));
  }
  if (lane == 0) {
    sh[0][warp] = lg;
    sh[1][warp] = P;
    sh[2][warp] = viol;
  }
  __syncthreads();
  if (tid == 0) {
    double p0 = sh[0][0], p1 = sh[1][0], p2 = sh[2][0];
#pragma unroll
    for (int w = 1; w < kW; ++w) {
      p0 += sh[0][w];
      p1 += sh[1][w];
      p2 = fmax(p2, sh[2][w]);
    }
    S.part[kUpdParts * blockIdx.x] = p0;
    S.part[kUpdParts * blockIdx.x + 1] = p1;
    S.part[kUpdParts * blockIdx.x + 2] = p2;
    __threadfence();
    s_last = atomicAdd(S.ticket, 1u) == static_cast<unsigned>(nct) - 1u;
    if (s_last) *S.ticket = 0u;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // the last CTA: warp 0 adds the partials, warp 1 the objective's
  double obj = 0.0;
  lg = P = viol = 0.0;
  if (warp == 0) {
    for (int k = lane; k < nct; k += 32) {
      lg += __ldcg(S.part + kUpdParts * k);
      P += __ldcg(S.part + kUpdParts * k + 1);
      viol = fmax(viol, __ldcg(S.part + kUpdParts * k + 2));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lg += __shfl_down_sync(kFull, lg, o);
      P += __shfl_down_sync(kFull, P, o);
      viol = fmax(viol, __shfl_down_sync(kFull, viol, o));
    }
  } else if (!S.obj_in) {
    for (int k = lane; k < S.nseg; k += 32) obj += S.seg_obj[S.seg_list[k]];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) obj += __shfl_down_sync(kFull, obj, o);
    if (lane == 0) sh[0][0] = obj;
  }
  __syncthreads();
  if (tid == 0) {
    obj = S.obj_in ? *S.obj_in : sh[0][0];
    if (S.count_on) {
      const double G = total - S.count_M;
      lg += static_cast<double>(S.lam[m * S.J]) * G;
      viol = fmax(viol, G);
      if (S.grad_out) S.grad_out[m * S.J] = static_cast<float>(G);
      *S.cnt = 0ull;
    }
    const double g = obj + lg;
    const double den = fabs(g) > 1e-30 ? fabs(g) : 1e-30;
    S.out[0] = g;
    S.out[1] = P;
    S.out[2] = S.certified ? (P - g) / den : NAN;
    S.out[3] = -lg / den;
    S.out[4] = viol;
    S.out[5] = obj;
    S.out[6] = S.state ? static_cast<double>(S.state->iter) : 0.0;
    S.out[7] = S.state ? static_cast<double>(S.state->status) : 0.0;
    S.out[8] = S.state ? S.state->gamma : gamma;
  }
}

// The objective partials of instance 0's certificate-sweep segments, summed
// in a fixed order (a shard's share of the certificate objective).
__global__ void __launch_bounds__(kUpdThreads) seg_sum_kernel(const StatsInst* __restrict__ tab, double* out) {
  __shared__ double sh[32];
  const StatsInst S = tab[0];
  double obj = 0.0;
  for (int k = threadIdx.x; k < S.nseg; k += blockDim.x) obj += S.seg_obj[S.seg_list[k]];
  obj = block_sum(obj, sh);
  if (threadIdx.x == 0) *out = obj;
}

}  // namespace

cudaError_t launch_update(const UpdInst* dev_tab, int ninst, int max_cta, cudaStream_t s, bool chain) {
  const dim3 grid(static_cast<unsigned>(max_cta > 0 ? max_cta : 1), static_cast<unsigned>(ninst));
  return launch_chained(chain, &fista_update_kernel, grid, kUpdChunk, 0, s, dev_tab);
}

int update_parts(int64_t D) { return kUpdParts * update_ctas(D); }

int update_ctas(int64_t D) { return static_cast<int>((D + kUpdChunk - 1) / kUpdChunk); }

cudaError_t launch_stats(const StatsInst* dev_tab, const StatsInst* one, int ninst, int maxJ, cudaStream_t s) {
  const dim3 grid(static_cast<unsigned>((maxJ + kUpdChunk - 1) / kUpdChunk), static_cast<unsigned>(ninst));
  stats_kernel<<<grid, kUpdChunk, 0, s>>>(dev_tab, one ? *one : StatsInst{});
  return cudaGetLastError();
}

cudaError_t launch_seg_sum(const StatsInst* dev_tab, double* out, cudaStream_t s) {
  seg_sum_kernel<<<1, kUpdThreads, 0, s>>>(dev_tab, out);
  return cudaGetLastError();
}

}  // namespace dlm
