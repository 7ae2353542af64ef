// sweep_kernels.cuh -- the fused dual sweep (the per-iteration hot path).  Included by
// one translation unit per value layout (sweep_f32.cu, sweep_bf16.cu and their
// counted forms), which compile in parallel; sweep.cu dispatches.
//
// For every user i and dual point y (Sec. 3.2, Eq. primal-recovery):
//     u_ik = -(c_ik + a_ik * y_j(k))                 (v = u / gamma)
//     x_i  = Proj_C_i(u_i / gamma)
// and per item j (Eq. dual-gradient): (A x)_j = sum_i a_ij x_ij.
// With STATS it also accumulates per item sum c x and sum x^2 and the
// objective sum (c x + gamma/2 x^2) for the dual value and the certified gap,
// and optionally writes x in the caller's edge order.
//
// Layout and mapping: users sit in degree-sorted slices of 32 (layout.cu);
// lane t of a warp owns user t of its slice and walks the user's edges four
// at a time with 128-bit loads (512 contiguous bytes per warp load).  The item dual y lives in
// shared memory (gathered by item index); item sums are accumulated in
// shared memory and flushed once per CTA.
//
// Simplex projection (Sec. 4.3 gets the threshold by sorting the whole row;
// no sort here).  In u-space the threshold tau solves
// sum max(u - tau, 0) = gamma z.  One pass over the row keeps its four
// largest u in a sorted register network, with the positions of the first
// three; the sort-based rule applied to those four either fixes the active
// set (at most three edges active: nearly every row at the paper's gammas,
// and for one edge x = z on it exactly) or shows that at least four are
// active.  With at most three, the threshold is recomputed over the recorded
// edges in float-pair arithmetic, so that x = (u - tau) / gamma keeps full
// FP32 relative accuracy when u and tau nearly cancel, and x is deposited on
// them: no second pass over the row.  With four or more the lane (or the
// whole warp, when few lanes need it) runs the iteration
// tau <- (sum_{u > tau} u - gamma z) / #{u > tau} from tau_4 (Michelot 1986;
// monotone from below, it stops when the active set stops changing), the
// pair-arithmetic refinement and a deposit pass.  The inequality simplex
// takes max(tau, 0) (the early exit of Sec. 4.3).  Box: x = clip(u / gamma,
// 0, z).
//
// Determinism: item sums are 64-bit fixed point (value * 2^s rounded, s chosen
// at set-up so no sum can overflow), exact and order independent, and so is the
// iteration's objective.  A certificate's objective is FP64: one part per slice,
// summed over its rows in lane order, the parts of a CTA's slices in slice order, the
// CTAs' in task order.
#pragma once

#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "dlm_impl.cuh"
#include "sweep_common.cuh"

namespace dlm {
namespace {

// The same value layouts for instances with a global count constraint: the
// count dual mu floors the threshold and every deposit adds x to the count.
// (A separate instantiation, so that instances without one keep the plain
// code: the register and comparison cost measured 4 % on the sweep.)
template <class Base>
struct Counted : Base {
  static constexpr bool kCount = true;
};

// Where a certificate sweep writes a row's x, in the caller's order: the
// output is cleared before the sweep (by the caller) and only the edges with
// x > 0 are written, as they are deposited.  (Every edge written by the row's lane, its
// position decoded from the lead record each time: 315 us for 1M rows, 25M
// edges FP32; that evaluation went from 378 to 166 us with this and the
// reductions of stats_kernel spread over CTAs.)
struct XRow {
  float* x;  // the row's first edge, or nullptr
  uint64_t lead;
  int d;
  __device__ __forceinline__ void put(int k, float v) const {
    if (x != nullptr) x[lead_caller_pos(lead, k, d)] = v;
  }
};

// Threshold of user t of the slice computed by the whole warp: lane l takes
// edges l, l + 32, ... of the user (re-read from L1/L2; the warp has just
// streamed them), the Michelot sums and the pair-arithmetic refinement are
// warp reductions in a fixed order, and every lane deposits the x of its own
// edges.  tau0 is the starting threshold (a lower bound on the equality
// threshold); with `exact` it is already the threshold of the final active
// set and the iteration is skipped.  Returns the threshold (tau, taul) and
// whether the inequality simplex took tau = 0.
template <class P, bool STATS>
__device__ __forceinline__ void coop_user(const Seg& S, const float* __restrict__ ys, unsigned long long* accG,
                                          unsigned long long* accC, unsigned long long* accQ,
                                          const typename P::IX* __restrict__ cp0, const typename P::T* __restrict__ vp0,
                                          int w, int w4, int t, float tau0, bool exact, const XRow& xr, float& tau,
                                          float& taul, bool& zero, float& ob, unsigned long long& cn) {
  const int lane = threadIdx.x & 31;
  const bool box = S.kind == DLM_BOX;
  const bool eq = S.kind == DLM_SIMPLEX_EQ;
  auto uval = [&](int k, int& j, float& c, float& a) {
    const int e = sell_el(k, t, w4);
    j = static_cast<int>(__ldg(cp0 + e));
    P::get(__ldg(vp0 + e), c, a);
    return -fmaf(a, ys[j], c);
  };
  tau = 0.f;
  taul = 0.f;
  zero = box;
  if (!box) {
    tau = tau0;
    if (!exact) {
      int prevn = -1;
      for (int it = 0; it < 256; ++it) {
        float sm = 0.f;
        int n = 0;
        for (int k = lane; k < w; k += 32) {
          int j;
          float c, a;
          const float u = uval(k, j, c, a);
          if (u > tau) {
            sm += u;
            ++n;
          }
        }
        sm = warp_sum(sm);
        n = warp_sumi(n);
        if (n == prevn || n == 0) break;
        prevn = n;
        const float tn = __fdiv_rn(sm - S.gz, static_cast<float>(n));
        if (tn == tau) break;
        tau = tn;
      }
    }
    zero = !eq && tau <= (P::kCount ? S.mu : 0.f);
    if (!zero) {
      F2 sum{0.f, 0.f};
      int n = 0;
      for (int k = lane; k < w; k += 32) {
        int j;
        float c, a;
        if (uval(k, j, c, a) > tau) {
          sum = f2_add(sum, u_pair(c, a, ys[j]));
          ++n;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const F2 other{__shfl_xor_sync(kFull, sum.h, o), __shfl_xor_sync(kFull, sum.l, o)};
        sum = f2_add(sum, other);
        n += __shfl_xor_sync(kFull, n, o);
      }
      const F2 t2 = f2_threshold(sum, S.gz, S.gzl, n > 0 ? n : 1);
      if (!eq && t2.h + t2.l <= (P::kCount ? S.mu : 0.f)) {
        zero = true;
      } else {
        tau = t2.h;
        taul = t2.l;
      }
    }
  }
  if (zero) {
    tau = (P::kCount ? S.mu : 0.f);
    taul = 0.f;
  }
  for (int k = lane; k < w; k += 32) {
    int j;
    float c, a;
    if (uval(k, j, c, a) > tau) {
      const float x = x_general(S, box, tau, taul, c, a, ys[j]);
      if (x > 0.f) {
        deposit<P, STATS>(S, j, c, a, x, accG, accC, accQ, ob, cn);
        if (STATS) xr.put(k, x);
      }
    }
  }
}

// A row whose simplex active set is the r <= 3 recorded edges (on the
// inequality simplex with tau <= 0: those of them with u > 0): load them once,
// compute the threshold over them in pair arithmetic, deposit x on each.
// Returns the objective part.  (Iteration sweeps.)  Loading them once saves a
// re-read (4 % on the 64-instance batch, 6 % on the appendix instance once its
// rows have several active edges; no change on the precision sweep).
template <class P, int K>
__device__ __forceinline__ float rows_upto(const Seg& S, const float* __restrict__ ys, unsigned long long* accG,
                                         const typename P::IX* __restrict__ col0, const typename P::T* __restrict__ ca0,
                                         int w4, int lane, int r, const int (&pos)[K - 1], float tau, bool eq,
                                         unsigned long long& cn) {
  int jr[K - 1];
  float cr[K - 1], ar[K - 1];
#pragma unroll
  for (int i = 0; i < K - 1; ++i) {
    jr[i] = 0;
    cr[i] = ar[i] = 0.f;
    if (i < r) {
      const int el = sell_el(pos[i], lane, w4);
      jr[i] = static_cast<int>(__ldg(col0 + el));
      P::get(__ldg(ca0 + el), cr[i], ar[i]);
    }
  }
  bool zero = !eq && tau <= (P::kCount ? S.mu : 0.f);
  float taul = 0.f;
  if (!zero) {
    F2 sum = u_pair(cr[0], ar[0], ys[jr[0]]);
#pragma unroll
    for (int i = 1; i < K - 1; ++i)
      if (i < r) sum = f2_add(sum, u_pair(cr[i], ar[i], ys[jr[i]]));
    const F2 t2 = f2_threshold_small<K - 1>(sum, S.gz, S.gzl, r);
    if (!eq && t2.h + t2.l <= (P::kCount ? S.mu : 0.f)) {
      zero = true;
    } else {
      tau = t2.h;
      taul = t2.l;
    }
  }
  if (zero) {
    tau = (P::kCount ? S.mu : 0.f);
    taul = 0.f;
  }
  float ob = 0.f;
#pragma unroll
  for (int i = 0; i < K - 1; ++i) {
    if (i < r) {
      const float x = x_general(S, false, tau, taul, cr[i], ar[i], ys[jr[i]]);
      if (x > 0.f) deposit<P, false>(S, jr[i], cr[i], ar[i], x, accG, nullptr, nullptr, ob, cn);
    }
  }
  return ob;
}

// Users of a slice whose active set is larger than the four tracked values
// (mode 3 below) are handled by the whole warp, one after another, unless at
// least coop_max of the 32 need it (then each lane runs its own user, which
// keeps the lanes busy).  coop_max is a tuning parameter (0: always per lane,
// 33: always cooperative).

// The K largest u of a row (v[0] >= ... >= v[K-1]) and the edge positions
// id[0..K-2] of the first K - 1.  K = 4 for most instances; K = 8 resolves
// rows with up to seven active edges without the threshold iteration.
template <int K>
struct TopK {
  float v[K];
  int id[K - 1];
};
template <int K>
__device__ __forceinline__ TopK<K> topk_empty() {
  TopK<K> t;
#pragma unroll
  for (int q = 0; q < K; ++q) t.v[q] = -INFINITY;
#pragma unroll
  for (int q = 0; q < K - 1; ++q) t.id[q] = 0;
  return t;
}
// Sorted insertion of edge k with value u (strict comparisons: among equal
// values the earlier edge ranks first; for K = 4 the network of top4_insert).
template <int K>
__device__ __forceinline__ void topk_insert(float u, int k, TopK<K>& t) {
  float x = u;
  int xi = k;
#pragma unroll
  for (int q = 0; q < K - 1; ++q) {
    const bool c = x > t.v[q];
    const float lo = c ? t.v[q] : x;
    const int loi = c ? t.id[q] : xi;
    t.v[q] = c ? x : t.v[q];
    t.id[q] = c ? xi : t.id[q];
    x = lo;
    xi = loi;
  }
  t.v[K - 1] = fmaxf(t.v[K - 1], x);
}

// After pass A over a row: the threshold, x and the deposits (modes below);
// col0/ca0 are the slice's element streams.  The lane finishes row ut of the
// slice when act is set: its own (ut = lane), or with Q (a quarter slice, rows
// 8 quarter .. 8 quarter + 7) row 8 quarter + lane / 4 in the first lane of each four.
// part: where a certificate sweep puts the objective of these rows (slice_part).
template <class P, bool STATS, int K, bool Q = false>
__device__ __forceinline__ void finish_slice(const InstDesc& D, const Seg& S, const float* __restrict__ ys,
                                             unsigned long long* accG, unsigned long long* accC,
                                             unsigned long long* accQ, int64_t s, int w,
                                             const typename P::IX* __restrict__ col0,
                                             const typename P::T* __restrict__ ca0, const TopK<K>& tk, int coop_max,
                                             int64_t part, unsigned long long& cn, unsigned long long& oq,
                                             int quarter = 0) {
  const int lane = Q ? 8 * quarter + static_cast<int>((threadIdx.x & 31) >> 2) : static_cast<int>(threadIdx.x & 31);
  const bool act = !Q || (threadIdx.x & 3) == 0;
  const int w4 = w >> 2;
  const bool box = S.kind == DLM_BOX;
  const bool eq = S.kind == DLM_SIMPLEX_EQ;
  const float v0 = tk.v[0];
  const int i0 = tk.id[0];
  XRow xr{nullptr, 0, 0};
  if (STATS && D.xout != nullptr && act) {
    const int64_t u = 32 * s + lane;
    if (u < D.nusers) xr = XRow{D.xout + __ldg(D.orig_off + u), __ldg(D.lead + u), __ldg(D.udeg + u)};
  }

  // The equality threshold solves sum_k max(u_k - tau, 0) = gamma z.  With
  // the values sorted, tau_r = (v_0 + ... + v_{r-1} - gamma z) / r and the
  // active count is the first r with v_r <= tau_r; scanning the K largest
  // either finds it (the active set lies among them) or shows that at least
  // K edges are active, and then tau_K is a lower bound for the iteration.
  // mode 0: no edge active; 1: the maximum alone, x = z; 2: threshold of the
  // final active set known (tau); 3: iterate from tau.
  int mode;
  float tau = 0.f, taul = 0.f;
  bool zero = box;
  int r = 0;
  if (box) {
    mode = (v0 > (P::kCount ? S.mu : 0.f)) ? 3 : 0;
  } else if (v0 == -INFINITY || (!eq && v0 <= (P::kCount ? S.mu : 0.f))) {
    mode = 0;
  } else {
    float sm = v0;
    r = 1;
    tau = v0 - S.gz;
#pragma unroll
    for (int q = 1; q < K; ++q) {
      if (r == q && tk.v[q] > tau) {
        sm += tk.v[q];
        r = q + 1;
        tau = div_by(sm - S.gz, static_cast<float>(q + 1), 1.f / static_cast<float>(q + 1));
      }
    }
    mode = (r == 1 && (eq || tau >= (P::kCount ? S.mu : 0.f))) ? 1 : (r < K ? 2 : 3);
  }

  if (!act) mode = 0;
  float ob = 0.f;
  if (!STATS && mode == 2) {
    ob += rows_upto<P, K>(S, ys, accG, col0, ca0, w4, lane, r, tk.id, tau, eq, cn);
  } else if (mode == 2) {
    // The certificate sweeps have no registers to hold the edges: they read them again from L1.
    zero = !eq && tau <= (P::kCount ? S.mu : 0.f);
    if (!zero) {
      F2 sum{0.f, 0.f};
#pragma unroll
      for (int i = 0; i < K - 1; ++i) {
        if (i >= r) break;
        const int el = sell_el(tk.id[i], lane, w4);
        const int j = static_cast<int>(__ldg(col0 + el));
        float c, a;
        P::get(__ldg(ca0 + el), c, a);
        sum = f2_add(sum, u_pair(c, a, ys[j]));
      }
      const F2 t2 = f2_threshold_small<K - 1>(sum, S.gz, S.gzl, r);
      if (!eq && t2.h + t2.l <= (P::kCount ? S.mu : 0.f)) {
        zero = true;
      } else {
        tau = t2.h;
        taul = t2.l;
      }
    }
    if (zero) {
      tau = (P::kCount ? S.mu : 0.f);
      taul = 0.f;
    }
#pragma unroll
    for (int i = 0; i < K - 1; ++i) {
      if (i >= r) break;
      const int el = sell_el(tk.id[i], lane, w4);
      const int j = static_cast<int>(__ldg(col0 + el));
      float c, a;
      P::get(__ldg(ca0 + el), c, a);
      const float x = x_general(S, false, tau, taul, c, a, ys[j]);
      if (x > 0.f) {
        deposit<P, STATS>(S, j, c, a, x, accG, accC, accQ, ob, cn);
        xr.put(tk.id[i], x);
      }
    }
  } else if (mode == 1) {
    // (the maximum alone; folded into the path above, the 16M x 5,000 BF16 sweep took 1.5 % longer)
    const int el = sell_el(i0, lane, w4);
    const int j = static_cast<int>(__ldg(col0 + el));
    float c, a;
    P::get(__ldg(ca0 + el), c, a);
    deposit<P, STATS>(S, j, c, a, S.z, accG, accC, accQ, ob, cn);
    if (STATS) xr.put(i0, S.z);
  }

  // Mode 3 (K or more active edges, or the box): the whole warp per user
  // while few lanes need it, else each lane over its own row.
  const unsigned mask3 = __ballot_sync(kFull, mode == 3);
  const bool coop = mask3 != 0u && __popc(mask3) < coop_max;  // warp-uniform
  if (coop) {
    unsigned m = mask3;
    while (m) {
      const int t = __ffs(m) - 1;
      m &= m - 1;
      const float tt = __shfl_sync(kFull, tau, t);
      const int row = Q ? 8 * quarter + (t >> 2) : t;
      float ta, tl;
      bool zr;
      // every lane adds the objective of its edges of user t: that piece
      // goes to fixed point on its own, so the total does not depend on
      // which users share the warp
      float obu = 0.f;
      XRow xt{nullptr, 0, 0};
      if (STATS)
        xt = XRow{reinterpret_cast<float*>(__shfl_sync(kFull, reinterpret_cast<unsigned long long>(xr.x), t)),
                  __shfl_sync(kFull, xr.lead, t), __shfl_sync(kFull, xr.d, t)};
      coop_user<P, STATS>(S, ys, accG, accC, accQ, col0, ca0, w, w4, row, tt, false, xt, ta, tl, zr, obu, cn);
      if (STATS)
        ob += obu;
      else
        oq += fixp(obu, S.scaleO);
    }
  } else if (mode == 3) {
    // Each lane over its own row, in groups of four edges (128-bit loads, as
    // in pass A) and then the tail, so every pass visits edges 0 .. w-1 in
    // order.
    auto row_pass = [&](auto&& visit) {
      for (int g = 0; g < w4; ++g) {
        const int q = 32 * g + lane;
        int jj[4];
        P::idx4(col0, q, jj);
        float c[4], a[4];
        P::get4(ca0, q, c, a);
#pragma unroll
        for (int e = 0; e < 4; ++e) visit(4 * g + e, jj[e], c[e], a[e]);
      }
      for (int k = 4 * w4; k < w; ++k) {
        const int el = 128 * w4 + 32 * (k - 4 * w4) + lane;
        float c, a;
        P::get(__ldg(ca0 + el), c, a);
        visit(k, static_cast<int>(__ldg(col0 + el)), c, a);
      }
    };
    if (!box) {
      // Michelot iteration from tau_K, a lower bound of the threshold: the
      // active sets {u > tau} shrink until two passes agree.  Each pass also
      // sums its active set in pair arithmetic, so the pass that finds the
      // set unchanged already holds the sum the threshold is refined from.
      F2 psum{0.f, 0.f};
      int n = 0;
      bool settled = false;
      int prevn = -1;
      for (int it = 0; it < 256; ++it) {
        float sm = 0.f;
        int cnt = 0;
        F2 ps{0.f, 0.f};
        row_pass([&](int k, int j, float c, float a) {
          const float y = ys[j];
          const float u = -fmaf(a, y, c);
          if (u > tau) {
            sm += u;
            ++cnt;
            ps = f2_add(ps, u_pair(c, a, y));
          }
        });
        psum = ps;
        n = cnt;
        if (cnt == prevn || cnt == 0) {
          settled = true;
          break;
        }
        prevn = cnt;
        const float tn = __fdiv_rn(sm - S.gz, static_cast<float>(cnt));
        if (tn == tau) {
          settled = true;
          break;
        }
        tau = tn;
      }
      zero = !eq && tau <= (P::kCount ? S.mu : 0.f);
      if (!zero) {
        if (!settled) {  // iteration cap: the sum over the current set
          psum = F2{0.f, 0.f};
          n = 0;
          row_pass([&](int k, int j, float c, float a) {
            if (-fmaf(a, ys[j], c) > tau) {
              psum = f2_add(psum, u_pair(c, a, ys[j]));
              ++n;
            }
          });
        }
        const F2 t2 = f2_threshold(psum, S.gz, S.gzl, n > 0 ? n : 1);
        if (!eq && t2.h + t2.l <= (P::kCount ? S.mu : 0.f)) {
          zero = true;
        } else {
          tau = t2.h;
          taul = t2.l;
        }
      }
    }
    if (zero) {
      tau = (P::kCount ? S.mu : 0.f);
      taul = 0.f;
    }
    // x on the active edges (u > tau; for the box and tau = 0, u > 0)
    row_pass([&](int k, int j, float c, float a) {
      const float y = ys[j];
      if (-fmaf(a, y, c) > tau) {
        const float x = x_general(S, box, tau, taul, c, a, y);
        if (x > 0.f) {
          deposit<P, STATS>(S, j, c, a, x, accG, accC, accQ, ob, cn);
          if (STATS) xr.put(k, x);
        }
      }
    });
  }

  if (STATS) {
    // FP64, to a place of its own: the warps may then take slices by ticket (dealt
    // statically for the sake of one running sum's order, a third of them waited for those
    // with the widest: 1M x 1,000 FP32, one evaluation 157 us, now 136).
    double o = static_cast<double>(ob);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) o += __shfl_xor_sync(kFull, o, d);
    if ((threadIdx.x & 31) == 0) D.slice_obj[part] = o;
  } else {
    // the user's objective part, added exactly (64-bit fixed point)
    oq += fixp(ob, S.scaleO);
  }
}

// Pass A over a slice: lane t = user t; edge k of lane t is element
// sell_el(k, t, w/4) of the slice.  Streams the rows in groups of four edges and
// keeps their K largest u with the positions of the first K - 1.
template <class P, int K>
__device__ __forceinline__ TopK<K> scan_slice(const float* __restrict__ ys, int w,
                                              const typename P::IX* __restrict__ col0,
                                              const typename P::T* __restrict__ ca0) {
  const int lane = threadIdx.x & 31;
  const int w4 = w >> 2;
  TopK<K> tk = topk_empty<K>();
  // groups of four edges in chunks of CH groups: the chunk's loads are issued
  // together, then each group is inserted unless no lane's group maximum tops
  // its K-th largest value (then the insertions change no record: strict
  // comparisons); the rows' lowest-cost edges come first (lead order,
  // layout.cu), so most groups after the first are skipped by the warp
  constexpr int CH = sizeof(typename P::T) == 4 ? 4 : 2;
  auto insert_group = [&](int g, const int (&jj)[4], const float (&c)[4], const float (&a)[4]) {
    float u[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) u[e] = -fmaf(a[e], ys[jj[e]], c[e]);
    const float m4 = fmaxf(fmaxf(u[0], u[1]), fmaxf(u[2], u[3]));
    if (__any_sync(kFull, m4 > tk.v[K - 1])) {
#pragma unroll
      for (int e = 0; e < 4; ++e) topk_insert<K>(u[e], 4 * g + e, tk);
    }
  };
  int g = 0;
  for (; g + CH <= w4; g += CH) {
    int jj[CH][4];
    float c[CH][4], a[CH][4];
#pragma unroll
    for (int h = 0; h < CH; ++h) {
      P::idx4(col0, 32 * (g + h) + lane, jj[h]);
      P::get4(ca0, 32 * (g + h) + lane, c[h], a[h]);
    }
#pragma unroll
    for (int h = 0; h < CH; ++h) insert_group(g + h, jj[h], c[h], a[h]);
  }
  // the rest, at most three groups, in one round trip (16M x 5,000 BF16, ten
  // iterations: 4,460 us with one for each group, 4,219)
  auto rest = [&](auto n) {
    constexpr int N = decltype(n)::value;
    int jj[N][4];
    float c[N][4], a[N][4];
#pragma unroll
    for (int h = 0; h < N; ++h) {
      P::idx4(col0, 32 * (g + h) + lane, jj[h]);
      P::get4(ca0, 32 * (g + h) + lane, c[h], a[h]);
    }
#pragma unroll
    for (int h = 0; h < N; ++h) insert_group(g + h, jj[h], c[h], a[h]);
  };
  if (CH > 2 && g + 3 <= w4)
    rest(std::integral_constant<int, 3>{});
  else if (CH > 2 && g + 2 <= w4)
    rest(std::integral_constant<int, 2>{});
  else if (g < w4)
    rest(std::integral_constant<int, 1>{});
  for (int k = 4 * w4; k < w; ++k) {
    const int e2 = 128 * w4 + 32 * (k - 4 * w4) + lane;
    const int j = static_cast<int>(__ldg(col0 + e2));
    float c, a;
    P::get(__ldg(ca0 + e2), c, a);
    topk_insert<K>(-fmaf(a, ys[j], c), k, tk);
  }
  return tk;
}

// One slice.  `ahead` runs between the pass and the finish (the next slice's
// header is fetched there, so that it is at hand when the slice is done).
// (Rows of four to seven active edges settled by a second pass with the
// eight-wide record instead of the threshold iteration: no gain on any workload,
// 2 % lost on 16M x 5,000 BF16.)
template <class P, bool STATS, int K, class Ahead>
__device__ __forceinline__ void do_slice(const InstDesc& D, const Seg& S, const float* __restrict__ ys,
                                         unsigned long long* accG, unsigned long long* accC,
                                         unsigned long long* accQ, int64_t s, int64_t off, int w, int coop_max,
                                         int64_t part, unsigned long long& cn, unsigned long long& oq, Ahead&& ahead) {
  const typename P::IX* __restrict__ col0 = P::idx(D) + off;
  const typename P::T* __restrict__ ca0 = static_cast<const typename P::T*>(D.ca) + off;
  const TopK<K> tk = scan_slice<P, K>(ys, w, col0, ca0);
  ahead();
  finish_slice<P, STATS, K>(D, S, ys, accG, accC, accQ, s, w, col0, ca0, tk, coop_max, part, cn, oq);
}

// A quarter of a wide slice: rows 8 quarter .. 8 quarter + 7, four lanes a
// row, lane p of the four taking groups p, p + 4, ...; their records are
// merged (of equal values the earlier edge first, so the record is that of the
// whole row in order) and the first of the four finishes the row.  A warp's
// pass over a slice is a chain of loads, one chunk after another (50 us for 500 FP32
// edges); where that is a large part of the sweep the widest slices are cut into
// four tickets of a quarter of the chain each (wide_slices in api.cu).  Not
// inlined, and in kernels of their own (WIDE): the common path keeps its
// registers.  1M x 1,000 FP32, rows of up to 500 edges, 25 iterations and a
// certificate: 1,976 -> 1,500 us; 2,000 to 50,000 users: 25 -> 18 us an iteration.
template <class P, int K>
__device__ __forceinline__ TopK<K> scan_quarter(const float* __restrict__ ys, int w,
                                                const typename P::IX* __restrict__ col0,
                                                const typename P::T* __restrict__ ca0, int quarter) {
  const int part = threadIdx.x & 3;
  const int row = 8 * quarter + static_cast<int>((threadIdx.x & 31) >> 2);
  const int w4 = w >> 2;
  TopK<K> tk = topk_empty<K>();
  constexpr int CH = 2;  // groups of a chunk, as in the whole slice's pass
  for (int g0 = part; g0 - part < w4; g0 += 4 * CH) {
    int jj[CH][4];
    float c[CH][4], a[CH][4];
#pragma unroll
    for (int h = 0; h < CH; ++h) {
      const int g = g0 + 4 * h;
      if (g < w4) {
        P::idx4(col0, 32 * g + row, jj[h]);
        P::get4(ca0, 32 * g + row, c[h], a[h]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) jj[h][e] = 0, c[h][e] = INFINITY, a[h][e] = 0.f;
      }
    }
#pragma unroll
    for (int h = 0; h < CH; ++h) {
      float u[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) u[e] = -fmaf(a[h][e], ys[jj[h][e]], c[h][e]);
      const float m4 = fmaxf(fmaxf(u[0], u[1]), fmaxf(u[2], u[3]));
      if (__any_sync(kFull, m4 > tk.v[K - 1])) {
#pragma unroll
        for (int e = 0; e < 4; ++e) topk_insert<K>(u[e], 4 * (g0 + 4 * h) + e, tk);
      }
    }
  }
  if (4 * w4 + part < w) {  // the tail's edge `part`
    const int el = 128 * w4 + 32 * part + row;
    float c, a;
    P::get(__ldg(ca0 + el), c, a);
    topk_insert<K>(-fmaf(a, ys[__ldg(col0 + el)], c), 4 * w4 + part, tk);
  }
  __syncwarp();
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    float ov[K];
    int oi[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
      ov[q] = __shfl_xor_sync(kFull, tk.v[q], o);
      oi[q] = q < K - 1 ? __shfl_xor_sync(kFull, tk.id[q < K - 1 ? q : 0], o) : 0x7fffffff;
    }
#pragma unroll
    for (int n = 0; n < K; ++n) {
      float x = ov[n];
      int xi = oi[n];
#pragma unroll
      for (int q = 0; q < K - 1; ++q) {
        const bool b = x > tk.v[q] || (x == tk.v[q] && xi < tk.id[q]);
        const float lo = b ? tk.v[q] : x;
        const int loi = b ? tk.id[q] : xi;
        tk.v[q] = b ? x : tk.v[q];
        tk.id[q] = b ? xi : tk.id[q];
        x = lo;
        xi = loi;
      }
      tk.v[K - 1] = fmaxf(tk.v[K - 1], x);
    }
  }
  return tk;
}
struct QuarterSums {
  unsigned long long cn, oq;
};
template <class P, bool STATS, int K>
__device__ __noinline__ QuarterSums do_quarter(const InstDesc& D, const Seg& S, const float* __restrict__ ys,
                                               unsigned long long* accG, unsigned long long* accC,
                                               unsigned long long* accQ, int64_t s, int quarter, int coop_max) {
  const int64_t off = __ldg(D.slice_off + s);
  const int w = __ldg(D.slice_w + s);
  const typename P::IX* __restrict__ col0 = P::idx(D) + off;
  const typename P::T* __restrict__ ca0 = static_cast<const typename P::T*>(D.ca) + off;
  QuarterSums r{0ull, 0ull};
  const TopK<K> tk = scan_quarter<P, K>(ys, w, col0, ca0, quarter);
  finish_slice<P, STATS, K, true>(D, S, ys, accG, accC, accQ, s, w, col0, ca0, tk, coop_max, 4 * s + quarter, r.cn, r.oq,
                                  quarter);
  return r;
}

// The constants as the sweep's registers: those that the kernel parameter holds are read from it.
template <bool ONE, bool STATS>
__device__ __forceinline__ Seg seg_of(const InstDesc& D, const Seg& sS) {
  Seg S = sS;
  if (ONE) {
    S.z = D.z;
    S.scaleG = D.scaleG;
    S.scaleC = D.scaleC;
    S.scaleQ = D.scaleQ;
    S.scaleN = D.scaleN;
    S.scaleO = D.scaleO;
    S.kind = D.kind;
  }
  return S;
}
// Slices of the task below nwide.
__device__ __forceinline__ int64_t task_wide(const Task& T, int64_t nwide) {
  const int64_t end = nwide < T.end ? nwide : T.end;
  return T.first < end ? (end - T.first + T.stride - 1) / T.stride : 0;
}

// Where slice s leaves its part of a certificate's objective: after the four parts
// of each slice taken in quarters (4 s + quarter).
template <bool WIDE>
__device__ __forceinline__ int64_t slice_part(const InstDesc& D, int64_t s) {
  return WIDE ? s + 3 * D.nwide : s;
}

// The warp's share of a task's slices, by tickets.  AHEAD: the ticket and the
// header (offset, width) of the next slice are fetched before the finish of
// the one in hand (16M x 5,000 BF16: 492 -> 470 us an iteration); not where the CTA meets a barrier at the
// end of every unit, which a slice claimed ahead by a warp still busy delays (16-member batch: 145 -> 163 us).
template <class P, bool STATS, int K, bool ONE, bool WIDE, bool AHEAD>
__device__ __forceinline__ void slices_of(const InstDesc& D, const Seg& sS, const float* __restrict__ ys,
                                          unsigned long long* accG, unsigned long long* accC,
                                          unsigned long long* accQ, const Task& T, unsigned* next, int coop_max,
                                          unsigned long long& cn, unsigned long long& oq) {
  const int n = static_cast<int>((T.end - T.first + T.stride - 1) / T.stride);
  const int nq = WIDE ? static_cast<int>(task_wide(T, D.nwide)) : 0;  // its first slices, taken in quarters
  int i = next_ticket(next);
  if constexpr (WIDE) {
    for (; i < 4 * nq; i = next_ticket(next)) {
      const QuarterSums r = do_quarter<P, STATS, K>(D, sS, ys, accG, accC, accQ,
                                                    T.first + static_cast<int64_t>(i >> 2) * T.stride, i & 3,
                                                          coop_max);
      cn += r.cn;
      oq += r.oq;
    }
    i -= 3 * nq;
  }
  const Seg S = seg_of<ONE, STATS>(D, sS);
  if constexpr (!AHEAD) {
    for (; i < n; i = next_ticket(next) - (WIDE ? 3 * nq : 0)) {
      const int64_t s = T.first + static_cast<int64_t>(i) * T.stride;
      do_slice<P, STATS, K>(D, S, ys, accG, accC, accQ, s, __ldg(D.slice_off + s), __ldg(D.slice_w + s), coop_max,
                            slice_part<WIDE>(D, s), cn, oq, [] {});
    }
    return;
  }
  int64_t off = 0;
  int w = 0;
  auto header = [&](int q, int64_t& o, int& v) {
    if (q < n) {
      const int64_t s = T.first + static_cast<int64_t>(q) * T.stride;
      o = __ldg(D.slice_off + s);
      v = __ldg(D.slice_w + s);
    }
  };
  header(i, off, w);
  while (i < n) {
    int ni = 0, nw = 0;
    int64_t noff = 0;
    const int64_t s = T.first + static_cast<int64_t>(i) * T.stride;
    do_slice<P, STATS, K>(D, S, ys, accG, accC, accQ, s, off, w, coop_max, slice_part<WIDE>(D, s), cn, oq, [&] {
                                  ni = next_ticket(next) - (WIDE ? 3 * nq : 0);
                                  header(ni, noff, nw);
                                });
    i = ni;
    off = noff;
    w = nw;
  }
}

// Certificate sweeps (STATS) keep the item sums of the window of items
// jlo .. jlo + jw - 1 only, so that instances whose three item arrays do not
// fit in shared memory take one launch per window; every launch recomputes
// the same x and writes the same objective partials, and the count sum is
// flushed by the launch with jlo = 0.
//
// ONE: every task is of one instance, whose descriptor comes as a kernel
// parameter: its fields are constant-bank operands and take no registers (the
// kernel sits at the 64 a thread that 1,024 threads allow; with the constants
// in registers the 16M x 5,000 BF16 sweep took 5 % longer).  Otherwise the descriptors are read
// from the table, one per instance.
template <class P, bool STATS, int K, bool ONE, bool WIDE>
__global__ void __launch_bounds__(kSweepThreads, 1)
    sweep_kernel(const __grid_constant__ InstDesc one, const InstDesc* __restrict__ insts,
                 const Task* __restrict__ tasks, const int32_t* __restrict__ cta_task, int smemJ, int coop_max,
                 int jlo, int jw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int accN = STATS ? jw : smemJ;
  unsigned long long* accG = reinterpret_cast<unsigned long long*>(smem_raw);
  unsigned long long* accC = accG + accN;
  unsigned long long* accQ = accC + accN;
  float* ys = reinterpret_cast<float*>(accG + (STATS ? 3 : 1) * static_cast<size_t>(accN));
  double* wsum = reinterpret_cast<double*>(ys + ((smemJ + 1) & ~1));

  __shared__ InstDesc s_inst;
  const InstDesc& sD = ONE ? one : s_inst;
  __shared__ Seg sS;
  __shared__ unsigned s_next;
  __shared__ unsigned long long s_red[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = blockDim.x >> 5;
  const int t_last = cta_task[blockIdx.x + 1];
  int t = cta_task[blockIdx.x];
  if (ONE)  // one segment: its sums are cleared ahead of the wait
    for (int j = threadIdx.x; j < (STATS ? 3 : 1) * accN; j += blockDim.x) accG[j] = 0ull;
  chain_wait();
  chain_go();
  while (t < t_last) {
    const int inst = tasks[t].inst;
    int te = t + 1;
    while (te < t_last && tasks[te].inst == inst) ++te;
    if (!ONE) {
      if (threadIdx.x == 0) s_inst = insts[inst];
      __syncthreads();
    }
    const int J = sD.J;
    // items with sums in this launch (STATS: the window, clipped to J)
    const int nacc = STATS ? max(0, min(J - jlo, jw)) : J;
    for (int j = threadIdx.x; j < J; j += blockDim.x) ys[j] = sD.y[j];
    if (!ONE) {
      for (int j = threadIdx.x; j < nacc; j += blockDim.x) {
        accG[j] = 0ull;
        if (STATS) {
          accC[j] = 0ull;
          accQ[j] = 0ull;
        }
      }
    }
    unsigned long long cn = 0ull, oq = 0ull;
    if (threadIdx.x == 0) {
      fill_seg(sD, STATS ? jlo : 0, nacc, sS);
      s_next = 0;
    }
    __syncthreads();
    for (int k = t; k < te; ++k) {
      const Task T = tasks[k];
      // dynamic order within the CTA (the sums are exact, so the order of
      // slices does not change any result)
      slices_of<P, STATS, K, ONE, WIDE, true>(sD, sS, ys, accG, accC, accQ, T, &s_next, coop_max, cn, oq);
      __syncthreads();
      if (threadIdx.x == 0) s_next = 0;
      __syncthreads();
    }
    if (STATS) {
      // the slices' parts (written before the barrier above), in a fixed order
      double o = 0.0;
      for (int k = t; k < te; ++k) {
        const Task T = tasks[k];
        const int n = static_cast<int>((T.end - T.first + T.stride - 1) / T.stride);
        const int nq = WIDE ? static_cast<int>(task_wide(T, sD.nwide)) : 0;
        for (int i = threadIdx.x; i < n + 3 * nq; i += blockDim.x) {
          const bool q = i < 4 * nq;
          const int64_t s = T.first + static_cast<int64_t>(q ? i >> 2 : i - 3 * nq) * T.stride;
          o += sD.slice_obj[q ? 4 * s + (i & 3) : slice_part<WIDE>(sD, s)];
        }
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) o += __shfl_xor_sync(kFull, o, d);
      if (lane == 0) wsum[warp] = o;
    } else {
      cta_add_u64(oq, s_red, sD.objq);
    }
    if (P::kCount && sD.count_on && (!STATS || jlo == 0)) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) cn += __shfl_xor_sync(kFull, cn, o);
      if (lane == 0 && cn) atomicAdd(sD.cnt, cn);
    }
    __syncthreads();
    {
      const int j0 = STATS ? jlo : 0;
      for (int j = threadIdx.x; j < nacc; j += blockDim.x) {
        const unsigned long long v = accG[j];
        if (v) atomicAdd(sD.acc + j0 + j, v);
        if (STATS) {
          const unsigned long long vc = accC[j], vq = accQ[j];
          if (vc) atomicAdd(sD.accC + j0 + j, vc);
          if (vq) atomicAdd(sD.accQ + j0 + j, vq);
        }
      }
    }
    if (STATS && threadIdx.x == 0) {
      double sum = 0.0;
      for (int w = 0; w < nw; ++w) sum += wsum[w];
      sD.seg_obj[t] = sum;
    }
    __syncthreads();
    t = te;
  }
}

// Sweep with dynamic work distribution (iteration sweeps only): CTAs take
// work units -- a range of slices of one instance -- from a global counter in
// table order.  A CTA keeps an instance's y and item sums in shared memory
// across consecutive units of that instance and flushes the sums when it
// moves to another instance.  The last CTA to finish resets the counters for
// the next launch.  The units are ordered by instance and shrink toward the
// end of the table, so the CTAs finish together.
template <class P, int K, bool WIDE>
__global__ void __launch_bounds__(kSweepThreads, 1)
    sweep_dyn_kernel(const InstDesc* __restrict__ insts, const Task* __restrict__ units, int nunits,
                     unsigned* __restrict__ ctr, int smemJ, int coop_max) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* accG = reinterpret_cast<unsigned long long*>(smem_raw);
  float* ys = reinterpret_cast<float*>(accG + smemJ);

  __shared__ InstDesc sD;
  __shared__ Seg sS;
  __shared__ unsigned s_unit;
  __shared__ unsigned s_next;
  __shared__ unsigned long long s_red[32];
  const int lane = threadIdx.x & 31;
  int cur = -1;
  unsigned long long cn = 0ull, oq = 0ull;
  chain_wait();
  chain_go();
  for (;;) {
    if (threadIdx.x == 0) {
      s_unit = atomicAdd(ctr, 1u);
      s_next = 0;
    }
    __syncthreads();
    const unsigned u = s_unit;
    const bool out_of_work = u >= static_cast<unsigned>(nunits);
    const int inst = out_of_work ? -1 : units[u].inst;
    if (out_of_work || inst != cur) {
      if (cur >= 0) {
        if (P::kCount && sD.count_on) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) cn += __shfl_xor_sync(kFull, cn, o);
          if (lane == 0 && cn) atomicAdd(sD.cnt, cn);
        }
        cn = 0ull;
        for (int j = threadIdx.x; j < sD.J; j += blockDim.x) {
          const unsigned long long v = accG[j];
          if (v) atomicAdd(sD.acc + j, v);
        }
        cta_add_u64(oq, s_red, sD.objq);
        oq = 0ull;
      }
      __syncthreads();
      if (out_of_work) break;
      if (threadIdx.x == 0) sD = insts[inst];
      __syncthreads();
      for (int j = threadIdx.x; j < sD.J; j += blockDim.x) {
        ys[j] = sD.y[j];
        accG[j] = 0ull;
      }
      if (threadIdx.x == 0) fill_seg(sD, 0, sD.J, sS);
      cur = inst;
      __syncthreads();
    }
    const Task T = units[u];
    slices_of<P, false, K, false, WIDE, false>(sD, sS, ys, accG, nullptr, nullptr, T, &s_next, coop_max, cn, oq);
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned prev = atomicAdd(ctr + 1, 1u);
    if (prev == gridDim.x - 1) {
      ctr[0] = 0u;
      ctr[1] = 0u;
    }
  }
}

template <class P, int K, bool WIDE>
cudaError_t prepare_kernels(int lim) {
  const auto smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(&sweep_dyn_kernel<P, K, WIDE>, smem, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(&sweep_kernel<P, false, K, true, WIDE>, smem, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(&sweep_kernel<P, false, K, false, WIDE>, smem, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(&sweep_kernel<P, true, K, true, WIDE>, smem, lim);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(&sweep_kernel<P, true, K, false, WIDE>, smem, lim);
  return e;
}

// Quarters are taken of FP32 instances and with the four-wide record only.
template <class P, int K>
constexpr bool kQuarters = K == 4 && sizeof(typename P::T) == 8;

template <class P, int K>
cudaError_t prepare_width(int lim) {
  const cudaError_t e = prepare_kernels<P, K, false>(lim);
  if constexpr (kQuarters<P, K>) return e != cudaSuccess ? e : prepare_kernels<P, K, true>(lim);
  return e;
}

template <class P>
cudaError_t prepare_policy(int lim) {
  const cudaError_t e = prepare_width<P, 4>(lim);
  return e != cudaSuccess ? e : prepare_width<P, 8>(lim);
}

template <class P, int K, bool WIDE>
cudaError_t launch_kernels(const SweepLaunch& L, bool stats) {
  const int th = L.threads > 0 ? L.threads : kSweepThreads;
  const int cm = L.coop_max;
  const InstDesc one = L.inst0 != nullptr ? *L.inst0 : InstDesc{};
  if (stats) {
    const int w = L.win > 0 ? std::min(L.win, L.smemJ) : L.smemJ;
    if (w < 1) return cudaErrorInvalidValue;
    const size_t sm = sweep_stats_smem_bytes(L.smemJ, w);
    for (int jlo = 0; jlo < L.smemJ || jlo == 0; jlo += w) {
      if (L.inst0 != nullptr)
        sweep_kernel<P, true, K, true, WIDE>
            <<<L.grid, th, sm, L.stream>>>(one, L.inst, L.tasks, L.cta_task, L.smemJ, cm, jlo, w);
      else
        sweep_kernel<P, true, K, false, WIDE>
            <<<L.grid, th, sm, L.stream>>>(one, L.inst, L.tasks, L.cta_task, L.smemJ, cm, jlo, w);
      const cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  const size_t sm = sweep_smem_bytes(L.smemJ, false);
  if (L.units != nullptr)
    return launch_chained(L.chain, &sweep_dyn_kernel<P, K, WIDE>, L.grid, th, sm, L.stream, L.inst, L.units, L.nunits,
                          L.ctr, L.smemJ, cm);
  if (L.inst0 != nullptr)
    return launch_chained(L.chain, &sweep_kernel<P, false, K, true, WIDE>, L.grid, th, sm, L.stream, one, L.inst, L.tasks,
                          L.cta_task, L.smemJ, cm, 0, L.smemJ);
  return launch_chained(L.chain, &sweep_kernel<P, false, K, false, WIDE>, L.grid, th, sm, L.stream, one, L.inst, L.tasks,
                        L.cta_task, L.smemJ, cm, 0, L.smemJ);
}

template <class P, int K>
cudaError_t launch_width(const SweepLaunch& L, bool stats) {
  if constexpr (kQuarters<P, K>)
    if (L.wide) return launch_kernels<P, K, true>(L, stats);
  return launch_kernels<P, K, false>(L, stats);
}

template <class P>
cudaError_t launch_policy(const SweepLaunch& L, bool stats) {
  return L.topk == 8 ? launch_width<P, 8>(L, stats) : launch_width<P, 4>(L, stats);
}

}  // namespace
}  // namespace dlm
