// noalloc.cu -- one dual evaluation that allocates no device memory.
//
// For callers that cannot allocate device memory (code running under a
// memory budget that forbids cudaMalloc, inside an allocator of its own, or
// in a process whose memory is owned by another framework), this file gives
// a variant of the dual evaluation that reads the caller's CSR arrays
// directly and keeps all of its scratch (fixed-point item sums, per-block
// objective partials, value bounds, an error word) in one file-scope
// __device__ array of fixed size.  Every GPU that loads the library holds that
// array until the process exits.  Calls that overlap on the GPU share it and
// race; run them one after another on one stream.
#include <cmath>
#include <mutex>

#include "dlm_impl.cuh"

namespace {

constexpr int64_t kStaticMaxItems = 65536;  // largest num_items accepted
constexpr int kStaticBlocks = 512;          // fixed grid of the bounds pass; most blocks of the sweep
constexpr int kStaticThreads = 512;         // threads of a sweep block
constexpr int kStaticWarps = kStaticThreads / 32;
constexpr int kLanes = 8;                   // lanes of a row: a warp takes four rows at a time
constexpr int kSlots = 8;                   // edges a lane holds in registers (rows of at most kLanes * kSlots edges)
constexpr unsigned kFull = 0xffffffffu;

struct StaticScratch {
  unsigned long long acc[kStaticMaxItems];  // fixed-point sum a x per item
  double obj[kStaticBlocks];                // objective partial per block
  unsigned int amax[kStaticBlocks];         // max |a| per block of the bounds pass (float bits)
  unsigned int bad;                         // error word
};

static __device__ __align__(256) StaticScratch g_scratch;

// Device address of g_scratch, looked up once per device (host code may not
// use the symbol itself as a device address).  The address belongs to the
// device's primary context: it is not valid after cudaDeviceReset.
constexpr size_t kStaticSmem2 = 100 * 1024;  // shared memory of a sweep block while two fit an SM
std::mutex g_sym_mu;
void* g_sym_addr[64] = {nullptr};
int g_sms[64] = {0};      // multiprocessors, at most kStaticBlocks / 2 used
size_t g_smem[64] = {0};  // the most shared memory a sweep block may use

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ int warp_sumi(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o));
  return v;
}

struct F2 {
  float h, l;
};
__device__ __forceinline__ F2 two_sum(float a, float b) {
  const float s = a + b;
  const float bp = s - a;
  return {s, (a - (s - bp)) + (b - bp)};
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  const F2 s = two_sum(a.h, b.h);
  return {s.h, s.l + (a.l + b.l)};
}
__device__ __forceinline__ F2 u_pair(float c, float a, float y) {
  const float p = a * y;
  const float pe = fmaf(a, y, -p);
  const F2 s = two_sum(-c, -p);
  return {s.h, s.l - pe};
}

__device__ __forceinline__ int shift_for(double bound) {
  if (!(bound > 0)) return 60;
  int s = static_cast<int>(floor(61.0 - log2(bound)));
  return s > 100 ? 100 : (s < 0 ? 0 : s);
}

// Exponent of the item sums: no sum of nnz terms a x overflows, while that leaves
// it at 0 or above (beyond, the sums have to fit by themselves).
__device__ __forceinline__ int sum_shift(int64_t nnz, float amax, double z) {
  return shift_for(static_cast<double>(nnz > 0 ? nnz : 1) * amax * z);
}

// Clears the item sums and the error word, and bounds |a| (for the
// fixed-point scale): one pass at memory bandwidth, four values a load.
__global__ void __launch_bounds__(256) k_static_begin(const float* __restrict__ a, int64_t nnz, int64_t J,
                                                      StaticScratch* S) {
  __shared__ unsigned sm[8];
  const int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  const int64_t nt = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = t; i < J; i += nt) S->acc[i] = 0ull;
  if (t == 0) S->bad = 0u;
  // the part of a that starts on a 16-byte boundary, by four; the ends one by one
  const int64_t lead = static_cast<int64_t>((0u - static_cast<unsigned>(reinterpret_cast<uintptr_t>(a) >> 2)) & 3u);
  const int64_t h = lead < nnz ? lead : nnz;
  const int64_t n4 = (nnz - h) >> 2;
  unsigned m = 0;
  const float4* __restrict__ a4 = reinterpret_cast<const float4*>(a + h);
#pragma unroll 4
  for (int64_t e = t; e < n4; e += nt) {
    const float4 v = __ldg(a4 + e);
    m = max(max(m, __float_as_uint(fabsf(v.x))), __float_as_uint(fabsf(v.y)));
    m = max(max(m, __float_as_uint(fabsf(v.z))), __float_as_uint(fabsf(v.w)));
  }
  for (int64_t e = t; e < h; e += nt) m = max(m, __float_as_uint(fabsf(a[e])));
  for (int64_t e = h + 4 * n4 + t; e < nnz; e += nt) m = max(m, __float_as_uint(fabsf(a[e])));
  m = __reduce_max_sync(kFull, m);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) m = max(m, sm[w]);
    S->amax[blockIdx.x] = m;
  }
}

// max |a| of the bounds pass; every thread of the block calls it.
__device__ __forceinline__ float static_amax(const StaticScratch* S, unsigned* sh) {
  unsigned m = 0;
  for (int k = threadIdx.x; k < kStaticBlocks; k += blockDim.x) m = max(m, S->amax[k]);
  m = __reduce_max_sync(kFull, m);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  m = 0;
  for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) m = max(m, sh[w]);
  __syncthreads();
  return __uint_as_float(m);
}

struct RowConst {
  float gamma, invg, gz, gzl, z, scG;
  bool eq, box;
};

// x of an edge of value pair up at the row's threshold (tau, taul).
__device__ __forceinline__ float static_x(const RowConst& C, bool zero, float tau, float taul, F2 up) {
  if (C.box) return fminf(fmaxf((up.h + up.l) * C.invg, 0.f), C.z);
  return zero ? fmaxf(up.h + up.l, 0.f) * C.invg : fmaxf((up.h - tau) + (up.l - taul), 0.f) * C.invg;
}

// The threshold over the active set's pair sum (sum - gamma z) / cnt.
__device__ __forceinline__ void static_refine(const RowConst& C, F2 sum, int cnt, float& tau, float& taul, bool& zero) {
  const F2 num = f2_add(sum, F2{-C.gz, -C.gzl});
  const float fn = static_cast<float>(cnt > 0 ? cnt : 1);
  const float th = __fdiv_rn(num.h, fn);
  const float tl = __fdiv_rn(fmaf(-th, fn, num.h) + num.l, fn);
  if (!C.eq && th + tl <= 0.f) {
    zero = true;
  } else {
    tau = th;
    taul = tl;
  }
}

// The sweep.  Per row: the simplex threshold by the Michelot iteration from
// max(u) - gamma z, refined in float-pair arithmetic, then x, the item sums
// and the objective.  The iteration stops once the threshold no longer rises (from the
// lower bound it cannot in exact arithmetic; in FP32 two sets whose
// thresholds round past each other would otherwise alternate), so every
// further pass strictly shrinks the active set and d + 1 passes always reach
// the stop.
//
// Eight lanes take a row, a warp four neighbouring rows, and a lane holds its
// up to eight edges in registers: the caller's arrays are read once, coalesced
// (the four rows are contiguous), and every pass of the iteration is register
// work and three shuffles.  Rows of more than 64 edges are taken after, one by
// one by the whole warp, re-reading.  Item sums are kept in shared memory
// (SMEM; J items of 12 bytes with lambda) and flushed once per block, in
// the global scratch for more items than fit.  With a warp per row, its passes
// re-reading the row and every active edge an atomic on the global scratch, the call
// took 592 us on 500,000 rows (12.4M edges, 1,000 items); now 220 us.
template <bool SMEM>
__global__ void __launch_bounds__(kStaticThreads, 2)
    k_static_sweep(const int64_t* __restrict__ rp, const int32_t* __restrict__ col, const float* __restrict__ c,
                   const float* __restrict__ a, int64_t I, int64_t J, int64_t nnz, int kind, double z,
                   const float* __restrict__ lam, double gamma, float* __restrict__ xout, StaticScratch* S) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* acc = SMEM ? reinterpret_cast<unsigned long long*>(smem_raw) : S->acc;
  float* sl = reinterpret_cast<float*>(acc + (SMEM ? J : 0));
  __shared__ RowConst sC;
  __shared__ unsigned s_red[kStaticWarps];
  __shared__ double s_obj[kStaticWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float amax = static_amax(S, s_red);
  if (SMEM) {
    for (int j = threadIdx.x; j < static_cast<int>(J); j += blockDim.x) {
      acc[j] = 0ull;
      sl[j] = lam[j];
    }
  }
  if (threadIdx.x == 0) {  // FP64 work once per block
    sC.scG = ldexpf(1.f, sum_shift(nnz, amax, z));
    sC.gamma = static_cast<float>(gamma);
    sC.invg = static_cast<float>(1.0 / gamma);
    const double gzd = gamma * z;
    sC.gz = static_cast<float>(gzd);
    sC.gzl = static_cast<float>(gzd - static_cast<double>(sC.gz));
    sC.z = static_cast<float>(z);
    sC.eq = kind == DLM_SIMPLEX_EQ;
    sC.box = kind == DLM_BOX;
  }
  __syncthreads();
  const RowConst C = sC;
  const float* __restrict__ ys = SMEM ? sl : lam;
  unsigned bad = 0;
  double wobj = 0.0;
  float ob = 0.f;  // objective of the lane's edges of the rows in hand
  auto put = [&](int j, float cv, float av, float x) {
    // one conversion, exact up to 2^63: with max |a| z above 2^55 the exponent is 0 and terms are as large
    atomicAdd(&acc[j], static_cast<unsigned long long>(__float2ll_rn(av * x * C.scG)));
    ob += fmaf(0.5f * C.gamma * x, x, cv * x);
  };
  // edge e of the caller's arrays: its item (-1: out of range, flagged), values, u
  auto edge = [&](int64_t e, int& j, float& cv, float& av) {
    j = __ldg(col + e);
    cv = __ldg(c + e);
    av = __ldg(a + e);
    if (static_cast<unsigned>(j) >= static_cast<unsigned>(J)) {
      j = -1;
      bad = 1;
      return -INFINITY;
    }
    return -fmaf(av, ys[j], cv);
  };
  auto sum8 = [&](float v) {
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
  };

  const int64_t nq = (I + 3) / 4;  // groups of four rows
  const int64_t step = static_cast<int64_t>(gridDim.x) * kStaticWarps;
  const int sub = lane & (kLanes - 1);
  for (int64_t q = static_cast<int64_t>(blockIdx.x) * kStaticWarps + warp; q < nq; q += step) {
    const int64_t u = 4 * q + (lane >> 3);
    int64_t s = 0, d = 0;
    if (u < I) {
      s = __ldg(rp + u);
      d = __ldg(rp + u + 1) - s;
      if (s < 0 || d < 0 || s > nnz || d > nnz - s) {  // invalid row pointer: no access, flagged
        bad = 1;
        s = d = 0;
      }
    }
    const bool wide = d > kLanes * kSlots;
    const int n = wide ? 0 : static_cast<int>(d);
    const int most = __reduce_max_sync(kFull, n);  // slots in use: (most + 7) / 8, warp-uniform
    int j[kSlots];
    float cv[kSlots], av[kSlots], uv[kSlots];
    float m = -INFINITY;
#pragma unroll
    for (int k = 0; k < kSlots; ++k) {
      j[k] = -1;
      cv[k] = av[k] = 0.f;
      uv[k] = -INFINITY;
      if (kLanes * k < most) {
        const int i = kLanes * k + sub;
        if (i < n) {
          j[k] = __ldg(col + s + i);
          cv[k] = __ldg(c + s + i);
          av[k] = __ldg(a + s + i);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kSlots; ++k) {
      if (kLanes * k < most && kLanes * k + sub < n) {
        if (static_cast<unsigned>(j[k]) >= static_cast<unsigned>(J)) {
          bad = 1;
          j[k] = -1;
        } else {
          uv[k] = -fmaf(av[k], ys[j[k]], cv[k]);
        }
      }
      m = fmaxf(m, uv[k]);
    }
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
    float tau = 0.f, taul = 0.f;
    bool zero = C.box;
    const bool solve = !C.box && n > 0 && (C.eq || m > 0.f);
    if (!C.box) {
      zero = !solve;
      bool run = solve;
      if (solve) tau = m - C.gz;
      int prevn = -1;
      while (__any_sync(kFull, run)) {
        float sm = 0.f;
        int cnt = 0;
#pragma unroll
        for (int k = 0; k < kSlots; ++k) {
          if (kLanes * k < most && uv[k] > tau) {
            sm += uv[k];
            ++cnt;
          }
        }
        sm = sum8(sm);
#pragma unroll
        for (int o = kLanes / 2; o > 0; o >>= 1) cnt += __shfl_xor_sync(kFull, cnt, o);
        if (run) {
          if (cnt == prevn || cnt == 0) {
            run = false;
          } else {
            prevn = cnt;
            const float tn = __fdiv_rn(sm - C.gz, static_cast<float>(cnt));
            if (!(tn > tau))
              run = false;
            else
              tau = tn;
          }
        }
      }
      if (solve) zero = !C.eq && tau <= 0.f;
      const bool refine = solve && !zero;
      if (__any_sync(kFull, refine)) {
        F2 sum{0.f, 0.f};
        int cnt = 0;
#pragma unroll
        for (int k = 0; k < kSlots; ++k) {
          if (kLanes * k < most && refine && uv[k] > tau) {
            sum = f2_add(sum, u_pair(cv[k], av[k], ys[j[k]]));
            ++cnt;
          }
        }
#pragma unroll
        for (int o = kLanes / 2; o > 0; o >>= 1) {
          const F2 other{__shfl_xor_sync(kFull, sum.h, o), __shfl_xor_sync(kFull, sum.l, o)};
          sum = f2_add(sum, other);
          cnt += __shfl_xor_sync(kFull, cnt, o);
        }
        if (refine) static_refine(C, sum, cnt, tau, taul, zero);
      }
    }
    if (zero) tau = taul = 0.f;
#pragma unroll
    for (int k = 0; k < kSlots; ++k) {
      if (kLanes * k < most) {
        float x = 0.f;
        if (uv[k] > tau) {
          x = static_x(C, zero, tau, taul, u_pair(cv[k], av[k], ys[j[k]]));
          if (x > 0.f) put(j[k], cv[k], av[k], x);
        }
        const int i = kLanes * k + sub;
        if (xout && i < n) xout[s + i] = x;
      }
    }
    wobj += static_cast<double>(ob);
    ob = 0.f;
    // rows of more than kLanes * kSlots edges: the whole warp, re-reading
    unsigned todo = __ballot_sync(kFull, wide && sub == 0);
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const int64_t ws = __shfl_sync(kFull, s, src), wd = __shfl_sync(kFull, d, src);
      float wt = 0.f, wtl = 0.f;
      bool wz = C.box;
      if (!C.box) {
        float wm = -INFINITY;
        for (int64_t i = lane; i < wd; i += 32) {
          int jj;
          float cc, aa;
          wm = fmaxf(wm, edge(ws + i, jj, cc, aa));
        }
        wm = warp_max(wm);
        if (C.eq || wm > 0.f) {
          wt = wm - C.gz;
          int prevn = -1;
          for (int64_t it = 0; it <= wd; ++it) {
            float sm = 0.f;
            int cnt = 0;
            for (int64_t i = lane; i < wd; i += 32) {
              int jj;
              float cc, aa;
              const float v = edge(ws + i, jj, cc, aa);
              if (v > wt) {
                sm += v;
                ++cnt;
              }
            }
            sm = warp_sum(sm);
            cnt = warp_sumi(cnt);
            if (cnt == prevn || cnt == 0) break;
            prevn = cnt;
            const float tn = __fdiv_rn(sm - C.gz, static_cast<float>(cnt));
            if (!(tn > wt)) break;
            wt = tn;
          }
          wz = !C.eq && wt <= 0.f;
          if (!wz) {
            F2 sum{0.f, 0.f};
            int cnt = 0;
            for (int64_t i = lane; i < wd; i += 32) {
              int jj;
              float cc, aa;
              if (edge(ws + i, jj, cc, aa) > wt) {
                sum = f2_add(sum, u_pair(cc, aa, ys[jj]));
                ++cnt;
              }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
              const F2 other{__shfl_xor_sync(kFull, sum.h, o), __shfl_xor_sync(kFull, sum.l, o)};
              sum = f2_add(sum, other);
              cnt += __shfl_xor_sync(kFull, cnt, o);
            }
            static_refine(C, sum, cnt, wt, wtl, wz);
          }
        } else {
          wz = true;
        }
      }
      if (wz) wt = wtl = 0.f;
      for (int64_t i = lane; i < wd; i += 32) {
        int jj;
        float cc, aa;
        const float v = edge(ws + i, jj, cc, aa);
        float x = 0.f;
        if (v > wt) {
          x = static_x(C, wz, wt, wtl, u_pair(cc, aa, ys[jj]));
          if (x > 0.f) put(jj, cc, aa, x);
        }
        if (xout) xout[ws + i] = x;
      }
      wobj += static_cast<double>(ob);
      ob = 0.f;
    }
  }
  if (__any_sync(kFull, bad) && lane == 0) atomicOr(&S->bad, 1u);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) wobj += __shfl_xor_sync(kFull, wobj, o);
  if (lane == 0) s_obj[warp] = wobj;
  __syncthreads();
  if (SMEM) {
    for (int j = threadIdx.x; j < static_cast<int>(J); j += blockDim.x) {
      const unsigned long long v = acc[j];
      if (v) atomicAdd(&S->acc[j], v);
    }
  }
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kStaticWarps; ++w) t += s_obj[w];
    S->obj[blockIdx.x] = t;
  }
}

// g = sum_i (c x + gamma/2 x^2) + lam^T (A x - b), grad = A x - b.  A flagged
// invalid item gives NaN.  (k_static_begin clears the scratch for each call.)
__global__ void __launch_bounds__(1024) k_static_finish(const double* __restrict__ b, int64_t J, int64_t nnz, double z,
                                                        int blocks, const float* __restrict__ lam, double* g_out,
                                                        float* __restrict__ grad_out, StaticScratch* S) {
  __shared__ double sh[2][32];
  __shared__ unsigned shm[32];
  __shared__ double s_inv;
  const float amax = static_amax(S, shm);
  if (threadIdx.x == 0) s_inv = ldexp(1.0, -sum_shift(nnz, amax, z));
  __syncthreads();
  const double invG = s_inv;
  const bool bad = S->bad != 0u;
  double lg = 0.0, obj = 0.0;
  for (int k = threadIdx.x; k < blocks; k += blockDim.x) obj += S->obj[k];
  for (int64_t j = threadIdx.x; j < J; j += blockDim.x) {
    const double G = static_cast<double>(static_cast<long long>(S->acc[j])) * invG - b[j];
    lg += static_cast<double>(lam[j]) * G;
    if (grad_out) grad_out[j] = bad ? NAN : static_cast<float>(G);
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lg += __shfl_down_sync(kFull, lg, o);
    obj += __shfl_down_sync(kFull, obj, o);
  }
  if (lane == 0) {
    sh[0][w] = lg;
    sh[1][w] = obj;
  }
  __syncthreads();
  if (w == 0) {
    lg = sh[0][lane];
    obj = sh[1][lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lg += __shfl_down_sync(kFull, lg, o);
      obj += __shfl_down_sync(kFull, obj, o);
    }
    if (lane == 0) *g_out = bad ? NAN : obj + lg;
  }
}

dlm_status sfail(dlm_status s, const char* m) {
  dlm::set_last_error(m);
  return s;
}

}  // namespace

extern "C" {

dlm_status dlm_calculate_static(int64_t num_users, int64_t num_items, int64_t nnz, const int64_t* row_ptr,
                                const int32_t* item_idx, const float* c, const float* a, const double* b,
                                int32_t kind, double z, const float* lambda, double gamma, double* g, float* grad,
                                float* x, void* stream) {
  dlm::set_last_error("");
  if (num_users < 0 || num_items <= 0 || nnz < 0) return sfail(DLM_ERR_INVALID_ARG, "bad sizes");
  if (num_items > kStaticMaxItems)
    return sfail(DLM_ERR_UNSUPPORTED, "num_items exceeds the static scratch limit of 65536 items");
  if (!row_ptr || (nnz > 0 && (!item_idx || !c || !a)) || !b || !lambda || !g)
    return sfail(DLM_ERR_INVALID_ARG, "null pointer");
  if (kind == DLM_BOX_CUT) return sfail(DLM_ERR_UNSUPPORTED, "DLM_BOX_CUT needs a handle (dlm_create)");
  if (kind != DLM_SIMPLEX_LE && kind != DLM_SIMPLEX_EQ && kind != DLM_BOX)
    return sfail(DLM_ERR_INVALID_ARG, "bad simple-set kind");
  if (!(z > 0) || !std::isfinite(z) || !(gamma > 0) || !std::isfinite(gamma))
    return sfail(DLM_ERR_INVALID_ARG, "z and gamma must be finite and > 0");
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
    return sfail(DLM_ERR_CUDA, "no current CUDA device");
  void* sym = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_sym_mu);
    if (!g_sym_addr[dev]) {
      void* p = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
      if (e != cudaSuccess || !p) return sfail(DLM_ERR_CUDA, "cudaGetSymbolAddress of the static scratch failed");
      int sms = 0;
      const size_t lim = dlm::sweep_smem_limit();
      cudaError_t e2 = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      if (e2 == cudaSuccess)
        e2 = cudaFuncSetAttribute(&k_static_sweep<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(lim));
      if (e2 != cudaSuccess) return sfail(DLM_ERR_CUDA, cudaGetErrorString(e2));
      g_sms[dev] = sms < kStaticBlocks / 2 ? sms : kStaticBlocks / 2;
      g_smem[dev] = lim;
      g_sym_addr[dev] = p;
    }
    sym = g_sym_addr[dev];
  }
  StaticScratch* S = static_cast<StaticScratch*>(sym);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  k_static_begin<<<kStaticBlocks, 256, 0, st>>>(a, nnz, num_items, S);
  // item sums in shared memory while they fit (two blocks per SM where both do)
  const size_t sm = 12 * static_cast<size_t>(num_items);
  const bool smem = sm <= g_smem[dev];
  const int most = (!smem || sm <= kStaticSmem2 ? 2 : 1) * g_sms[dev];
  const int64_t want = (num_users + 4 * kStaticWarps - 1) / (4 * kStaticWarps);
  const int blocks = static_cast<int>(want < 1 ? 1 : (want < most ? want : most));
  if (smem)
    k_static_sweep<true><<<blocks, kStaticThreads, sm, st>>>(row_ptr, item_idx, c, a, num_users, num_items, nnz, kind,
                                                             z, lambda, gamma, x, S);
  else
    k_static_sweep<false><<<blocks, kStaticThreads, 0, st>>>(row_ptr, item_idx, c, a, num_users, num_items, nnz, kind,
                                                             z, lambda, gamma, x, S);
  k_static_finish<<<1, 1024, 0, st>>>(b, num_items, nnz, z, blocks, lambda, g, grad, S);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return sfail(DLM_ERR_CUDA, cudaGetErrorString(e));
  return DLM_OK;
}

}  // extern "C"
