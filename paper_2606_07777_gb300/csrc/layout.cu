// layout.cu -- one-time set-up of an instance: input validation, the
// degree-sorted sliced layout the sweep reads, and per-item constants
// (sum_i a_ij^2 for the step size and row normalization, App. B.2; item
// degrees and value bounds for the fixed-point scales).
//
// The caller's CSR is user-major (one row per user; the paper's CSC with one
// column per source, Sec. 4.1).  Users are stably sorted by degree, largest
// first (the paper buckets by degree to limit padding, Sec. 4.2; sorting by
// the exact degree takes that to its limit), and cut into slices of 32
// consecutive users.  A slice of width w (its largest degree) holds 32 w
// elements per stream (item index; interleaved (c, a)).  Its first 4 (w / 4)
// edges of every user are stored in groups of four: edge k < 4 (w / 4) of
// user t at slice_off + 4 (32 (k / 4) + t) + k % 4, so that lane t reads four
// consecutive edges of its user with one 128-bit value load (one float2 pair
// per edge in FP32: two 128-bit loads) and a warp load covers 512 contiguous
// bytes.  The remaining w % 4 edges follow edge-major: edge k at
// slice_off + 128 (w / 4) + 32 (k - 4 (w / 4)) + t.  Edges past a user's
// degree are padding with c = +inf, a = 0 (they give u = -inf and are never
// active).  Users with no edges are dropped from the slices.  The item index
// stream is written as uint16 (every handle has fewer than 65,536 items), so
// four indices are one 64-bit load.
//
// Device memory comes from a stream-ordered pool per device that keeps what
// handles free (dev_alloc / dev_free): a daily re-creation of an instance of
// the same size then maps no new memory.
#include <cub/cub.cuh>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "dlm_impl.cuh"

namespace dlm {
namespace {

constexpr int kT = 256;

enum : int { kBadRowPtr = 1, kBadItem = 2, kBadValue = 4, kBadB = 8, kNegA = 16, kDupItem = 32 };
constexpr unsigned kFullMask = 0xffffffffu;
const char* const kDupMsg = "an item appears twice in one row (the eligible items of a user must be distinct)";
constexpr int kDupThreads = 256;

__device__ __forceinline__ float load_val(const void* p, int64_t e, bool bf16) {
  if (bf16) {
    const unsigned short b = reinterpret_cast<const unsigned short*>(p)[e];
    return __uint_as_float(static_cast<unsigned>(b) << 16);
  }
  return reinterpret_cast<const float*>(p)[e];
}

// Row pointer checks; degree of every user; users with no edges.  A row of more
// edges than items repeats one: found here, before a slice is laid out at its length.
__global__ void k_rows(const int64_t* rp, int64_t I, int64_t nnz, int64_t J, int32_t* deg,
                       unsigned long long* zero_cnt, int* bad) {
  int flag = 0;
  unsigned long long z = 0;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < I;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t r0 = rp[i], r1 = rp[i + 1];
    const int64_t d = r1 - r0;
    if (d < 0 || r0 < 0 || r1 > nnz || d > 0x7fffffff) flag |= kBadRowPtr;
    if (d > J) flag |= kDupItem;
    deg[i] = d < 0 ? 0 : static_cast<int32_t>(d);
    z += (d == 0);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (rp[0] != 0 || rp[I] != nnz) flag |= kBadRowPtr;
  }
  if (flag) atomicOr(bad, flag);
  if (z) atomicAdd(zero_cnt, z);
}

// Four consecutive values from edge 4 q on (aligned: see aligned4), as floats.
__device__ __forceinline__ void load_val4(const void* p, int64_t q, bool bf16, float (&v)[4]) {
  if (bf16) {
    const uint2 w = __ldg(static_cast<const uint2*>(p) + q);
    v[0] = __uint_as_float(w.x << 16), v[1] = __uint_as_float(w.x & 0xffff0000u);
    v[2] = __uint_as_float(w.y << 16), v[3] = __uint_as_float(w.y & 0xffff0000u);
  } else {
    const float4 w = __ldg(static_cast<const float4*>(p) + q);
    v[0] = w.x, v[1] = w.y, v[2] = w.z, v[3] = w.w;
  }
}
// Whether the caller's arrays start on the boundaries that loads of four
// edges need (any array of its own does; a view into one may not).
inline bool aligned4(const int32_t* col, const void* c, const void* a, bool bf16) {
  const uintptr_t m = bf16 ? 7 : 15;
  return (reinterpret_cast<uintptr_t>(col) & 15) == 0 &&
         ((reinterpret_cast<uintptr_t>(c) | reinterpret_cast<uintptr_t>(a)) & m) == 0;
}

// Edge checks, item degrees, max |a|, max |c|.  With J <= 16384 each block
// counts its share of the edges in shared memory and flushes once per item.
// Bound by the loads in flight: with `quad` (aligned arrays) a thread takes
// four edges a step, two steps at a time (50M BF16 edges, 1,000 items: 233 us with
// one edge a step).
__global__ void __launch_bounds__(1024) k_edges(const int32_t* __restrict__ col, const void* __restrict__ c,
                                                const void* __restrict__ a, bool bf16, int64_t nnz, int64_t J, bool quad,
                                                unsigned long long* item_deg, unsigned* max_a, unsigned* max_c,
                                                int* bad) {
  extern __shared__ unsigned scnt[];
  __shared__ unsigned s_ma, s_mc;
  const bool sm = J <= 16384;
  if (threadIdx.x == 0) s_ma = s_mc = 0;
  if (sm)
    for (int64_t j = threadIdx.x; j < J; j += blockDim.x) scnt[j] = 0u;
  __syncthreads();
  int flag = 0;
  unsigned ma = 0, mc = 0;
  auto take = [&](int32_t j, float cv, float av) {
    if (j < 0 || j >= J)
      flag |= kBadItem;
    else if (sm)
      atomicAdd(&scnt[j], 1u);
    else
      atomicAdd(&item_deg[j], 1ull);
    if (!isfinite(cv) || !isfinite(av)) flag |= kBadValue;
    if (av < 0.f) flag |= kNegA;
    ma = max(ma, __float_as_uint(fabsf(av)));
    mc = max(mc, __float_as_uint(fabsf(cv)));
  };
  const int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  const int64_t nt = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t n4 = quad ? nnz >> 2 : 0;
#pragma unroll 2
  for (int64_t q = t; q < n4; q += nt) {
    const int4 j = __ldg(reinterpret_cast<const int4*>(col) + q);
    float cv[4], av[4];
    load_val4(c, q, bf16, cv);
    load_val4(a, q, bf16, av);
    take(j.x, cv[0], av[0]);
    take(j.y, cv[1], av[1]);
    take(j.z, cv[2], av[2]);
    take(j.w, cv[3], av[3]);
  }
  for (int64_t e = 4 * n4 + t; e < nnz; e += nt) take(col[e], load_val(c, e, bf16), load_val(a, e, bf16));
  ma = __reduce_max_sync(kFullMask, ma);
  mc = __reduce_max_sync(kFullMask, mc);
  if (flag) atomicOr(bad, flag);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&s_ma, ma);
    atomicMax(&s_mc, mc);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicMax(max_a, s_ma);
    atomicMax(max_c, s_mc);
  }
  if (sm)
    for (int64_t j = threadIdx.x; j < J; j += blockDim.x)
      if (scnt[j]) atomicAdd(&item_deg[j], static_cast<unsigned long long>(scnt[j]));
}

// Items distinct within each row (the eligible set of Sec. 3.3 is a set of
// (user, item) pairs).  A warp takes 32 consecutive rows, whose edges are
// contiguous: it touches them once (prefetch to L1), then checks one row at a
// time -- a row of at most 32 edges by __match_any_sync over the lanes'
// items, a longer one by marking its items in a per-warp bitmap of J bits in
// shared memory, cleared again after the row.  Runs after the row pointers
// are checked; items outside [0, J) are skipped here (k_edges flags them).
__global__ void k_dups(const int64_t* rp, const int32_t* col, int64_t I, int64_t J, int* bad) {
  extern __shared__ unsigned bm[];
  const int lane = threadIdx.x & 31;
  const int words = static_cast<int>((J + 31) >> 5);
  unsigned* my = bm + static_cast<size_t>(threadIdx.x >> 5) * words;
  for (int k = lane; k < words; k += 32) my[k] = 0u;
  __syncwarp();
  const int64_t gw = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
  const int64_t nw = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  int flag = 0;
  for (int64_t i0 = 32 * gw; i0 < I; i0 += 32 * nw) {
    const int nrow = static_cast<int>(I - i0 < 32 ? I - i0 : 32);
    const int64_t rk = lane < nrow ? rp[i0 + lane] : 0;
    const int64_t rend = rp[i0 + nrow];
    const int64_t e0 = __shfl_sync(kFullMask, rk, 0);
    for (int64_t e = e0 + 32 * static_cast<int64_t>(lane); e < rend; e += 32 * 32)
      asm volatile("prefetch.global.L1 [%0];" ::"l"(col + e));
    for (int r = 0; r < nrow; ++r) {
      const int64_t s = __shfl_sync(kFullMask, rk, r);
      const int64_t t = __shfl_sync(kFullMask, rk, r + 1 < nrow ? r + 1 : 0);
      const int64_t e = r + 1 < nrow ? t : rend;
      const int64_t d = e - s;
      if (d <= 1) continue;  // warp-uniform
      if (d > J) {           // more edges than items: some item repeats
        flag = 1;
        continue;
      }
      if (d <= 32) {
        const int j = lane < d ? col[s + lane] : -1 - lane;  // idle lanes: distinct negative keys
        if (__popc(__match_any_sync(kFullMask, j)) > 1) flag = 1;
      } else {
        for (int64_t q = s + lane; q < e; q += 32) {
          const int j = col[q];
          if (static_cast<unsigned>(j) >= static_cast<unsigned>(J)) continue;
          const unsigned bit = 1u << (j & 31);
          if (atomicOr(&my[j >> 5], bit) & bit) flag = 1;
        }
        __syncwarp();
        for (int64_t q = s + lane; q < e; q += 32) {
          const int j = col[q];
          if (static_cast<unsigned>(j) < static_cast<unsigned>(J)) my[j >> 5] = 0u;
        }
        __syncwarp();
      }
    }
  }
  if (__any_sync(kFullMask, flag) && lane == 0) atomicOr(bad, kDupItem);
}

__global__ void k_b(const double* b, int64_t J, int* bad) {
  int flag = 0;
  for (int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; j < J;
       j += static_cast<int64_t>(gridDim.x) * blockDim.x)
    if (!isfinite(b[j]) || b[j] < 0.0) flag |= kBadB;
  if (flag) atomicOr(bad, flag);
}

__global__ void k_iota(int32_t* v, int64_t n) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    v[i] = static_cast<int32_t>(i);
}

// Slice widths (edges per lane) and slice sizes in elements (32 w).
__global__ void k_slices(const int32_t* sdeg, int64_t nslices, bool bf16, int32_t* width, int64_t* size) {
  for (int64_t s = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; s < nslices;
       s += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    // the slice's largest degree (sorted descending).  Three edges past the
    // groups of four -- in BF16, whose edges are smaller, two -- are made a
    // group with padding: the sweeps read the tail an edge at a time, a round trip
    // each (16M x 5,000 BF16: 470 -> 454 us an iteration with three, 451 with two; 8M x 2,000 FP32: 308
    // -> 305 us with three, 306 with two).  Rows of a few edges gain and lose by it: with widths under 12
    // left as they are, ten iterations of 4M x 1,000 at mean 10 take 823 -> 868 us in BF16, 891 -> 917 in
    // FP32; at mean 4 615 -> 564, 612 -> 638; at mean 2 468 -> 458, 445 -> 442; the short-row sweep 1 % less to 5 % more.
    const int32_t d = sdeg[32 * s];
    const int32_t w = (d & 3) >= (bf16 ? 2 : 3) ? (d | 3) + 1 : d;
    width[s] = w;
    size[s] = 32 * static_cast<int64_t>(w);
  }
}

// CA = float2 {c, a} (FP32) or uint32 (bf16 c low, bf16 a high).
template <typename CA>
__device__ __forceinline__ CA pack_ca(const void* c, const void* a, int64_t e);
template <>
__device__ __forceinline__ float2 pack_ca<float2>(const void* c, const void* a, int64_t e) {
  return make_float2(static_cast<const float*>(c)[e], static_cast<const float*>(a)[e]);
}
template <>
__device__ __forceinline__ uint32_t pack_ca<uint32_t>(const void* c, const void* a, int64_t e) {
  return static_cast<uint32_t>(static_cast<const unsigned short*>(c)[e]) |
         (static_cast<uint32_t>(static_cast<const unsigned short*>(a)[e]) << 16);
}
template <typename CA>
__device__ __forceinline__ CA pad_ca();
template <>
__device__ __forceinline__ float2 pad_ca<float2>() {
  return make_float2(INFINITY, 0.f);
}
template <>
__device__ __forceinline__ uint32_t pad_ca<uint32_t>() {
  return 0x00007F80u;  // c = bf16 +inf, a = 0
}

// Lanes' keys that order like the floats they encode (-0 as +0).
__device__ __forceinline__ unsigned cost_key(float c) {
  const unsigned u = __float_as_uint(c + 0.f);
  return (u & 0x80000000u) ? ~u : u | 0x80000000u;
}

// Four edges of a lane written at 16-byte pieces (q: quadruple).
__device__ __forceinline__ void put4(uint32_t* o, int64_t q, const uint32_t (&v)[4]) {
  reinterpret_cast<uint4*>(o)[q] = make_uint4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void put4(float2* o, int64_t q, const float2 (&v)[4]) {
  reinterpret_cast<float4*>(o)[2 * q] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  reinterpret_cast<float4*>(o)[2 * q + 1] = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
}

// A lane's four lowest edges by cost, of equal costs the earlier one: the
// cost's key above the position, so that an insertion is minima and maxima --
// 32 bits a key for BF16 costs and positions of up to 16 bits, 64 for FP32.
template <typename CA>
using LeadKey = typename std::conditional<sizeof(CA) == 4, unsigned, unsigned long long>::type;
__device__ __forceinline__ unsigned lead_key(uint32_t v, int k) {
  return (cost_key(__uint_as_float(v << 16)) & 0xffff0000u) | static_cast<unsigned>(k);
}
__device__ __forceinline__ unsigned long long lead_key(float2 v, int k) {
  return static_cast<unsigned long long>(cost_key(v.x)) << 32 | static_cast<unsigned>(k);
}
template <typename K>
__device__ __forceinline__ void lowest4(K x, K (&lk)[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const K lo = min(x, lk[q]);
    x = max(x, lk[q]);
    lk[q] = lo;
  }
}
// Adds the record of the lane o away.
template <typename K>
__device__ __forceinline__ void lowest4_merge(int o, K (&lk)[4]) {
  K x[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) x[q] = __shfl_xor_sync(kFullMask, lk[q], o);
#pragma unroll
  for (int q = 0; q < 4; ++q) lowest4(x[q], lk);
}
// The record as lead edges (0xFFFF past the row's d edges).
template <typename K>
__device__ __forceinline__ uint64_t lead_of(const K (&lk)[4], int d) {
  uint64_t ld = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    ld |= static_cast<uint64_t>(q < d ? static_cast<unsigned>(lk[q]) & 0xFFFFu : 0xFFFFu) << (16 * q);
  return ld;
}

// The slices' edge streams, rows in lead order (dlm_impl.cuh: the four
// lowest-cost edges first, of equal costs the earlier one).
//
// A warp takes a slice.  Rows of up to kRawWidth edges (gather_raw) are read
// once, with consecutive lanes (the caller's rows are contiguous, where a lane per row
// read every sector eight times over), as many rows at a time as fill 32 reads of
// the warp, eight of which are in flight together; they stay in shared memory
// in the caller's order while the lead edges are picked (warp minima of the costs'
// keys), the items checked (no item twice: a bitmap of the items in shared
// memory), and the slice's elements written, four positions of a row per
// lane.  Longer rows (gather_strips) are read for the lead edges, for the check and then
// once more, 32 slice positions of every row at a time, put into the slice's
// order in shared memory -- groups of four edges 4 elements further apart than
// in the slice, so that a row's groups fall into different banks -- and
// written out in whole 128-bit pieces.  There are few such slices and each is long, so
// the whole block takes one: its warps share the rows, then the strips (a new handle of
// 3,000 rows of 2,000 FP32 edges: 3,844 us with a warp a slice, 889 with a block; 30,000 rows: 5,322, 3,000).
// Slices are dealt by a counter, widest first.
// 50M BF16 edges (2M rows of 25 on average, the longest 500): 939 us with every
// row read twice and the longest rows' chains of loads at the end, now 439 us.
// Every item is in [0, J) here (checked before).
constexpr int kGatherWarps = 8;
constexpr int kStripGroups = 8;                           // groups of four edges of a strip
constexpr int kStripElems = kStripGroups * 132 + 3 * 32;  // staged elements: the groups, then the slice's tail
constexpr int kRawWidth = 1024;                           // longest rows of gather_raw
constexpr int kRawElems = 32 * 33;                        // its staged elements, at most: R rows of 32 nc + 1
static_assert(kRawElems <= kStripElems, "one buffer");

// What a warp works on: its slice, lane t's row of it, its shared memory.
template <typename CA>
struct GatherWarp {
  const int32_t* __restrict__ col;
  const void* __restrict__ c;
  const void* __restrict__ a;
  uint16_t* __restrict__ col_o;  // the slice's elements
  CA* __restrict__ ca_o;
  CA* sca;
  uint16_t* scol;
  unsigned* seen;
  int64_t r;  // first edge and degree of the lane's row
  int d, w, J;
};

// A row's lead edges in ascending order of position (0x7fff after the last),
// 16 bits each: with it a slice position past them is found by four comparisons.
__device__ __forceinline__ uint64_t lead_sorted(uint64_t lead, int d) {
  unsigned p[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) p[i] = i < d ? static_cast<unsigned>(lead >> (16 * i)) & 0xffffu : 0x7fffu;
  auto order = [&](int i, int j) {
    const unsigned lo = min(p[i], p[j]), hi = max(p[i], p[j]);
    p[i] = lo;
    p[j] = hi;
  };
  order(0, 1), order(2, 3), order(0, 2), order(1, 3), order(1, 2);
  return p[0] | static_cast<uint64_t>(p[1]) << 16 | static_cast<uint64_t>(p[2]) << 32 | static_cast<uint64_t>(p[3]) << 48;
}

// Slices of rows of up to kRawWidth edges.  Returns the lane's row's lead edges.
template <typename CA>
__device__ __forceinline__ uint64_t gather_raw(const GatherWarp<CA>& W, bool& twice) {
  const int lane = threadIdx.x & 31;
  const int w4 = W.w >> 2;
  const int nc = (W.w + 31) >> 5;  // reads of a row
  const int lg = nc > 1 ? 32 - __clz(nc - 1) : 0;
  const int R = 32 >> lg;  // rows at a time: R nc <= 32
  const int rs = 32 * nc + 1;
  using K = LeadKey<CA>;
  uint64_t lead = 0;
  for (int t0 = 0; t0 < 32; t0 += R) {
    // the rows as they are
    int row = 0, ch = 0;
    for (int x = 0; x < R * nc; x += 8) {
      int j[8], at[8];
      CA v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int64_t rt = __shfl_sync(kFullMask, W.r, (t0 + row) & 31);
        const int dt = __shfl_sync(kFullMask, W.d, (t0 + row) & 31);
        const int k = 32 * ch + lane;
        at[i] = -1;
        if (row < R && k < dt) {
          at[i] = row * rs + k;
          j[i] = __ldg(W.col + rt + k);
          v[i] = pack_ca<CA>(W.c, W.a, rt + k);
        }
        if (++ch == nc) ch = 0, ++row;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (at[i] >= 0) {
          W.scol[at[i]] = static_cast<uint16_t>(j[i]);
          W.sca[at[i]] = v[i];
        }
    }
    __syncwarp();
    // no item repeats: the row's items set their bits, and clear them again
    if (nc == 1) {
#pragma unroll 4
      for (int t = 0; t < 32; ++t) {
        const bool on = lane < __shfl_sync(kFullMask, W.d, t);
        const int j = on ? W.scol[t * rs + lane] : 0;
        const unsigned bit = on ? 1u << (j & 31) : 0u;
        if (on && (atomicOr(&W.seen[j >> 5], bit) & bit)) twice = true;
        __syncwarp();
        if (on) W.seen[j >> 5] = 0u;
        __syncwarp();
      }
    } else {
      for (int t = 0; t < R; ++t) {
        const int dt = __shfl_sync(kFullMask, W.d, t0 + t);
        for (int k = lane; k < dt; k += 32) {
          const int j = W.scol[t * rs + k];
          const unsigned bit = 1u << (j & 31);
          if (atomicOr(&W.seen[j >> 5], bit) & bit) twice = true;
        }
        __syncwarp();
        for (int k = lane; k < dt; k += 32) W.seen[W.scol[t * rs + k] >> 5] = 0u;
        __syncwarp();
      }
    }
    // 1 << lg lanes a row, R apart: its lead edges (every one of them holds the record at the end)
    const int t = lane & (R - 1), part = lane >> (5 - lg);
    const int dt = __shfl_sync(kFullMask, W.d, t0 + t);
    K lk[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) lk[q] = ~K{0};
#pragma unroll 2
    for (int k = part; k < dt; k += 1 << lg) lowest4<K>(lead_key(W.sca[t * rs + k], k), lk);
    __syncwarp();
    for (int o = R; o < 32; o <<= 1) lowest4_merge<K>(o, lk);
    const uint64_t lt = lead_of<K>(lk, dt);
    {
      const uint64_t mine = __shfl_sync(kFullMask, lt, lane & (R - 1));
      if (lane >= t0 && lane < t0 + R) lead = mine;
    }
    // the rows' slice elements: a lane writes a group of four positions of a row
    const uint64_t ls = lead_sorted(lt, dt);
    const unsigned p0 = ls & 0xffffu, p1 = (ls >> 16) & 0xffffu, p2 = (ls >> 32) & 0xffffu, p3 = ls >> 48;
    auto edge = [&](int k, CA& v, unsigned& j) {
      v = pad_ca<CA>();
      j = 0u;
      if (k < dt) {
        unsigned e;
        if (k < 4) {
          e = static_cast<unsigned>(lt >> (16 * k)) & 0xffffu;
        } else {
          e = static_cast<unsigned>(k - 4);
          e += e >= p0;
          e += e >= p1;
          e += e >= p2;
          e += e >= p3;
        }
        v = W.sca[t * rs + e];
        j = W.scol[t * rs + e];
      }
    };
    for (int g = part; g < w4; g += 1 << lg) {
      CA v[4];
      unsigned j[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) edge(4 * g + e, v[e], j[e]);
      const int64_t q = 32 * static_cast<int64_t>(g) + t0 + t;
      reinterpret_cast<uint2*>(W.col_o)[q] = make_uint2(j[0] | j[1] << 16, j[2] | j[3] << 16);
      put4(W.ca_o, q, v);
    }
    for (int k = 4 * w4 + part; k < W.w; k += 1 << lg) {  // the tail
      CA v;
      unsigned j;
      edge(k, v, j);
      const int64_t q = 128 * static_cast<int64_t>(w4) + 32 * (k - 4 * w4) + t0 + t;
      W.col_o[q] = static_cast<uint16_t>(j);
      W.ca_o[q] = v;
    }
    __syncwarp();
  }
  return lead;
}

// A slice of longer rows, by the whole block (every warp has the same slice in W).
template <typename CA>
__device__ __noinline__ uint64_t gather_strips(const GatherWarp<CA>& W, uint64_t* s_lead, bool& twice) {
  using K = LeadKey<CA>;
  constexpr bool kBf = sizeof(CA) == 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int w4 = W.w >> 2;
  for (int t = warp; t < 32; t += kGatherWarps) {
    const int64_t rt = __shfl_sync(kFullMask, W.r, t);
    const int dt = __shfl_sync(kFullMask, W.d, t);
    K lk[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) lk[q] = ~K{0};
    const int de = dt < 0xFFFF ? dt : 0xFFFF;  // (positions fit 16 bits)
#pragma unroll 4
    for (int k = lane; k < de; k += 32) lowest4<K>(lead_key(pack_ca<CA>(W.c, W.a, rt + k), k), lk);
    __syncwarp();
    for (int o = 1; o < 32; o <<= 1) lowest4_merge<K>(o, lk);
    const uint64_t ld = lead_of<K>(lk, dt);
    if (lane == 0) s_lead[t] = ld;
#pragma unroll 4
    for (int k = lane; k < dt; k += 32) {
      const int j = __ldg(W.col + rt + k);
      const unsigned bit = 1u << (j & 31);
      if (atomicOr(&W.seen[j >> 5], bit) & bit) twice = true;
    }
    __syncwarp();
#pragma unroll 4
    for (int k = lane; k < dt; k += 32) W.seen[__ldg(W.col + rt + k) >> 5] = 0u;
    __syncwarp();
  }
  __syncthreads();
  const uint64_t lead = s_lead[lane];
  // positions 32 st .. of every row, then the strip's elements in order
  for (int st = warp; 32 * st < W.w; st += kGatherWarps) {
    const int k = 32 * st + lane;
    const int at = k < 4 * w4 ? (lane >> 2) * 132 + (lane & 3) : kStripGroups * 132 + 32 * (k - 4 * w4);
    const int by = k < 4 * w4 ? 4 : 1;
#pragma unroll 4
    for (int t = 0; t < 32; ++t) {
      const int64_t rt = __shfl_sync(kFullMask, W.r, t);
      const int dt = __shfl_sync(kFullMask, W.d, t);
      const uint64_t lt = __shfl_sync(kFullMask, lead, t);
      CA v = pad_ca<CA>();
      uint16_t j = 0;
      if (k < dt) {
        const int64_t src = rt + lead_caller_pos(lt, k, dt);
        v = pack_ca<CA>(W.c, W.a, src);
        j = static_cast<uint16_t>(__ldg(W.col + src));
      }
      if (k < W.w) {
        W.sca[at + by * t] = v;
        W.scol[at + by * t] = j;
      }
    }
    __syncwarp();
    const int ng = min(kStripGroups, w4 - kStripGroups * st);
    const int64_t o = 128 * static_cast<int64_t>(kStripGroups * st);
    for (int g = 0; g < ng; ++g) {
      reinterpret_cast<uint4*>(W.ca_o + o + 128 * g)[lane] = reinterpret_cast<const uint4*>(W.sca + 132 * g)[lane];
      if (!kBf)
        reinterpret_cast<uint4*>(W.ca_o + o + 128 * g)[32 + lane] =
            reinterpret_cast<const uint4*>(W.sca + 132 * g)[32 + lane];
      reinterpret_cast<uint2*>(W.col_o + o + 128 * g)[lane] = reinterpret_cast<const uint2*>(W.scol + 132 * g)[lane];
    }
    if (W.w - 32 * st <= 32) {  // the last strip holds the tail
      for (int q = 0; q < W.w - 4 * w4; ++q) {
        const int64_t e = 128 * static_cast<int64_t>(w4) + 32 * q + lane;
        W.ca_o[e] = W.sca[kStripGroups * 132 + 32 * q + lane];
        W.col_o[e] = W.scol[kStripGroups * 132 + 32 * q + lane];
      }
    }
    __syncwarp();
  }
  return lead;
}

template <typename CA>
__global__ void __launch_bounds__(32 * kGatherWarps, sizeof(CA) == 4 ? 4 : 2)
    k_gather(const int64_t* __restrict__ rp, const int32_t* __restrict__ col, const void* __restrict__ c,
             const void* __restrict__ a, const int32_t* __restrict__ perm, const int32_t* __restrict__ sdeg, int64_t In,
             int64_t nslices, const int64_t* __restrict__ slice_off, const int32_t* __restrict__ width,
             uint16_t* __restrict__ col_o, CA* __restrict__ ca_o, int64_t* __restrict__ orig_off,
             int32_t* __restrict__ udeg, uint64_t* __restrict__ lead_o, int J, unsigned* __restrict__ ticket,
             int* __restrict__ dup) {
  extern __shared__ __align__(16) unsigned char gsm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  CA* sca = reinterpret_cast<CA*>(gsm + static_cast<size_t>(warp) * kStripElems * (sizeof(CA) + 2));
  uint16_t* scol = reinterpret_cast<uint16_t*>(sca + kStripElems);
  const int words = (J + 31) >> 5;
  unsigned* seen = reinterpret_cast<unsigned*>(gsm + static_cast<size_t>(kGatherWarps) * kStripElems * (sizeof(CA) + 2)) +
                   warp * words;
  for (int k = lane; k < words; k += 32) seen[k] = 0u;
  __syncwarp();
  __shared__ uint64_t s_lead[32];
  __shared__ unsigned s_ticket;
  bool twice = false;
  // slice s of every warp of the caller: its rows, and where its elements go
  auto slice = [&](int64_t s, bool write) {
    const int64_t u = 32 * s + lane;
    int64_t r = 0;
    int d = 0;
    if (u < In) {
      r = rp[perm[u]];
      d = sdeg[u];
      if (write) {
        orig_off[u] = r;
        udeg[u] = d;
      }
    }
    const int64_t base = slice_off[s];
    return GatherWarp<CA>{col, c, a, col_o + base, ca_o + base, sca, scol, seen, r, d, width[s], J};
  };
  // slices of long rows first, a block each; the first ticket that has none is warp 0's
  int64_t mine = -1;
  for (;;) {
    if (threadIdx.x == 0) s_ticket = atomicAdd(ticket, 1u);
    __syncthreads();
    const int64_t s = s_ticket;
    if (s >= nslices || width[s] <= kRawWidth) {
      if (warp == 0) mine = s;
      break;
    }
    bool again = false;  // (copies: W and `twice` stay in registers)
    const GatherWarp<CA> V = slice(s, warp == 0);
    const uint64_t lead = gather_strips(V, s_lead, again);
    twice = twice || again;
    if (warp == 0 && 32 * s + lane < In) lead_o[32 * s + lane] = lead;
    __syncthreads();  // s_lead and s_ticket have been read
  }
  for (;;) {
    int64_t s = mine;
    if (s < 0) {
      unsigned tk = 0;
      if (lane == 0) tk = atomicAdd(ticket, 1u);
      s = __shfl_sync(kFullMask, tk, 0);
    }
    mine = -1;
    if (s >= nslices) break;
    const GatherWarp<CA> W = slice(s, true);
    const uint64_t lead = gather_raw(W, twice);
    if (32 * s + lane < In) lead_o[32 * s + lane] = lead;
  }
  if (__any_sync(kFullMask, twice) && lane == 0) *dup = 1;
}

// sum_i a_ij^2 (sums[0 .. J)) and sum_i a_ij (sums[J .. 2 J)) per item in
// 64-bit fixed point (exact, order independent); SQ, S1: which of the two.
// Blocks add in shared memory where it holds the sums (SMEM) and flush once per
// item.  Bound by the shared-memory atomics of the popular items: one pass
// over the edges for both sums instead of two, four edges a step
// (`quad`: aligned arrays).  50M BF16 edges, 1,000 items: 168 us (2 x 338 in two passes).
template <bool SQ, bool S1, bool SMEM>
__global__ void __launch_bounds__(1024)
    k_item_sums(const int32_t* __restrict__ col, const void* __restrict__ a, bool bf16, int64_t nnz, int64_t J,
                float scale_sq, float scale_s1, bool quad, unsigned long long* __restrict__ sums) {
  extern __shared__ unsigned long long sacc[];
  unsigned long long* sq = SMEM ? sacc : sums;
  unsigned long long* s1 = (SMEM && !SQ) ? sacc : sq + J;
  const int64_t held = (SQ && S1) ? 2 * J : J;
  if (SMEM) {
    for (int64_t j = threadIdx.x; j < held; j += blockDim.x) sacc[j] = 0ull;
    __syncthreads();
  }
  auto add = [](unsigned long long* p, unsigned long long v) {
    if (SMEM)
      shared_add64(p, v);
    else
      atomicAdd(p, v);
  };
  auto take = [&](int32_t j, float av) {
    if (SQ) add(&sq[j], static_cast<unsigned long long>(__float2ll_rn(av * av * scale_sq)));
    if (S1) add(&s1[j], static_cast<unsigned long long>(__float2ll_rn(av * scale_s1)));
  };
  const int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  const int64_t nt = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t n4 = quad ? nnz >> 2 : 0;
#pragma unroll 2
  for (int64_t q = t; q < n4; q += nt) {
    const int4 j = __ldg(reinterpret_cast<const int4*>(col) + q);
    float av[4];
    load_val4(a, q, bf16, av);
    take(j.x, av[0]);
    take(j.y, av[1]);
    take(j.z, av[2]);
    take(j.w, av[3]);
  }
  for (int64_t e = 4 * n4 + t; e < nnz; e += nt) take(col[e], load_val(a, e, bf16));
  if (SMEM) {
    __syncthreads();
    unsigned long long* out = sums + (SQ ? 0 : J);
    for (int64_t j = threadIdx.x; j < held; j += blockDim.x)
      if (sacc[j]) atomicAdd(&out[j], sacc[j]);
  }
}

// Both sums into sums[2 J] (cleared here): one pass where shared memory holds
// both, two passes where it holds one, else global atomics.
cudaError_t launch_item_sums(const int32_t* col, const void* a, bool bf16, int64_t nnz, int64_t J, int ssq, int ss1,
                             unsigned long long* sums, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(sums, 0, sizeof(unsigned long long) * 2 * (J > 0 ? J : 1), s);
  if (e != cudaSuccess || nnz <= 0) return e;
  const size_t lim = sweep_smem_limit();
  const size_t one = sizeof(unsigned long long) * static_cast<size_t>(J);
  const float fq = std::ldexp(1.0f, ssq), f1 = std::ldexp(1.0f, ss1);
  const bool quad = aligned4(col, a, a, bf16);
  int dev = 0, sms = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int g = static_cast<int>(std::min<int64_t>(sms, nnz / 8192 + 1));  // one block of 1,024 threads per SM
  auto go = [&](auto kernel, size_t smem) {
    // (the limit is the process's: the same for every instance, or another thread's launch might find it lowered)
    cudaError_t f = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(lim));
    if (f != cudaSuccess) return f;
    kernel<<<g, 1024, smem, s>>>(col, a, bf16, nnz, J, fq, f1, quad, sums);
    return cudaGetLastError();
  };
  if (2 * one <= lim) return go(&k_item_sums<true, true, true>, 2 * one);
  if (one <= lim) {
    e = go(&k_item_sums<true, false, true>, one);
    return e != cudaSuccess ? e : go(&k_item_sums<false, true, true>, one);
  }
  return go(&k_item_sums<true, true, false>, 0);
}

int grid_for(int64_t n) {
  int64_t g = (n + kT - 1) / kT;
  if (g > 152 * 16) g = 152 * 16;
  if (g < 1) g = 1;
  return static_cast<int>(g);
}

std::mutex g_pool_mu;
cudaMemPool_t g_pool[64] = {};

}  // namespace

cudaError_t dev_alloc(void** p, size_t bytes, cudaStream_t s) {
  *p = nullptr;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  cudaMemPool_t pool;
  {
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (!g_pool[dev]) {
      cudaMemPoolProps props = {};
      props.allocType = cudaMemAllocationTypePinned;
      props.handleTypes = cudaMemHandleTypeNone;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      e = cudaMemPoolCreate(&g_pool[dev], &props);
      if (e != cudaSuccess) {
        g_pool[dev] = nullptr;
        return e;
      }
      uint64_t keep = UINT64_MAX;  // freed memory stays with the pool until dlm_release_cached_memory
      e = cudaMemPoolSetAttribute(g_pool[dev], cudaMemPoolAttrReleaseThreshold, &keep);
      if (e != cudaSuccess) return e;
    }
    pool = g_pool[dev];
  }
  return cudaMallocFromPoolAsync(p, bytes > 0 ? bytes : 16, pool, s);
}

void dev_free(void* p, cudaStream_t s) {
  if (p) cudaFreeAsync(p, s);
}

cudaError_t release_cached_memory() {
  std::lock_guard<std::mutex> lk(g_pool_mu);
  cudaError_t first = cudaSuccess;
  for (cudaMemPool_t& q : g_pool) {
    if (!q) continue;
    const cudaError_t e = cudaMemPoolTrimTo(q, 0);
    if (e != cudaSuccess && first == cudaSuccess) first = e;
  }
  return first;
}

// Fixed-point exponent for sums bounded by `bound`: the largest s with
// bound * 2^s <= 2^61 (two bits of headroom), clamped to [0, 100].
int fixed_point_shift(double bound) {
  if (!(bound > 0)) return 60;
  int s = static_cast<int>(std::floor(61.0 - std::log2(bound)));
  if (s > 100) s = 100;
  return s;
}

#define DLM_CK(x)                                                            \
  do {                                                                       \
    cudaError_t e_ = (x);                                                    \
    if (e_ != cudaSuccess) {                                                 \
      *msg = std::string("CUDA error in layout: ") + cudaGetErrorString(e_); \
      goto fail;                                                             \
    }                                                                        \
  } while (0)

void item_sum_shifts(int64_t max_item_deg, double max_abs_a, int* ssq, int* ss1) {
  *ssq = fixed_point_shift(static_cast<double>(max_item_deg) * max_abs_a * max_abs_a);
  *ss1 = fixed_point_shift(static_cast<double>(max_item_deg) * max_abs_a);
}

dlm_status item_sums(int64_t J, int64_t nnz, const int32_t* col, const void* a, bool bf16, int ssq, int ss1,
                     cudaStream_t s, int64_t* sq, int64_t* s1, std::string* msg) {
  unsigned long long* acc = nullptr;
  dlm_status st = DLM_OK;
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&acc), sizeof(unsigned long long) * 2 * (J > 0 ? J : 1), s));
  DLM_CK(launch_item_sums(col, a, bf16, nnz, J, ssq, ss1, acc, s));
  DLM_CK(cudaMemcpyAsync(sq, acc, sizeof(int64_t) * J, cudaMemcpyDeviceToHost, s));
  DLM_CK(cudaMemcpyAsync(s1, acc + J, sizeof(int64_t) * J, cudaMemcpyDeviceToHost, s));
  DLM_CK(cudaStreamSynchronize(s));
  goto done;
fail:
  st = DLM_ERR_CUDA;
done:
  dev_free(acc, s);
  cudaStreamSynchronize(s);
  return st;
}

dlm_status build_layout(int64_t I, int64_t J, int64_t nnz, const int64_t* rp, const int32_t* col, const void* c,
                        const void* a, const double* b, bool bf16, cudaStream_t s, LayoutOut* out,
                        std::string* msg, RowStats* measure, const ShardGlobal* shard) {
  const auto t_start = std::chrono::steady_clock::now();
  auto lap = [&](int k) {
    out->phase_s[k] = std::chrono::duration<double>(std::chrono::steady_clock::now() - t_start).count() -
                      (k > 0 ? out->phase_s[0] : 0.0) - (k > 1 ? out->phase_s[1] : 0.0);
  };
  const size_t vs = bf16 ? 2 : 4;
  // the kernels' limits are the process's: the same for every instance, or another thread's launch might find
  // one lowered
  const int smem_limit = static_cast<int>(sweep_smem_limit());
  cudaFuncSetAttribute(k_edges, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * 16384);
  dlm_status st = DLM_OK;
  int32_t *deg = nullptr, *sdeg = nullptr, *idx = nullptr, *perm = nullptr;
  int64_t* ssize = nullptr;
  unsigned long long *zero_cnt = nullptr, *item_deg = nullptr, *sq = nullptr;
  unsigned* mx = nullptr;
  int* bad = nullptr;
  void* tmp = nullptr;
  size_t tmp_bytes = 0;
  int h_bad = 0, h_dup = 0;
  unsigned h_mx[2] = {0, 0};
  unsigned long long h_zero = 0;
  std::vector<unsigned long long> h_deg;
  int ssq = 0, ss1 = 0;
  int64_t In = 0, ns = 0;

  DLM_CK(dev_alloc(reinterpret_cast<void**>(&deg), sizeof(int32_t) * (I > 0 ? I : 1), s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&zero_cnt), sizeof(unsigned long long), s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&item_deg), sizeof(unsigned long long) * (J > 0 ? J : 1), s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&mx), sizeof(unsigned) * 2, s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&bad), 2 * sizeof(int), s));
  DLM_CK(cudaMemsetAsync(zero_cnt, 0, sizeof(unsigned long long), s));
  DLM_CK(cudaMemsetAsync(item_deg, 0, sizeof(unsigned long long) * (J > 0 ? J : 1), s));
  DLM_CK(cudaMemsetAsync(mx, 0, sizeof(unsigned) * 2, s));
  DLM_CK(cudaMemsetAsync(bad, 0, sizeof(int), s));
  if (I > 0) k_rows<<<grid_for(I), kT, 0, s>>>(rp, I, nnz, J, deg, zero_cnt, bad);
  DLM_CK(cudaGetLastError());
  if (J > 0) k_b<<<grid_for(J), kT, 0, s>>>(b, J, bad);
  DLM_CK(cudaGetLastError());
  DLM_CK(cudaMemcpyAsync(&h_bad, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
  DLM_CK(cudaMemcpyAsync(&h_zero, zero_cnt, sizeof(h_zero), cudaMemcpyDeviceToHost, s));
  DLM_CK(cudaStreamSynchronize(s));
  if (h_bad & kBadRowPtr) {
    *msg = "row_ptr must start at 0, be non-decreasing and end at nnz";
    st = DLM_ERR_INVALID_ARG;
    goto done;
  }
  if (h_bad & kBadB) {
    *msg = "b must be finite and >= 0";
    st = DLM_ERR_INVALID_ARG;
    goto done;
  }
  if (nnz > 0) {
    int dev = 0, sms = 0;
    DLM_CK(cudaGetDevice(&dev));
    DLM_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int g = static_cast<int>(std::min<int64_t>(sms, nnz / 8192 + 1));  // one block of 1,024 threads per SM
    const size_t smem = J <= 16384 ? sizeof(unsigned) * J : 0;
    k_edges<<<g, 1024, smem, s>>>(col, c, a, bf16, nnz, J, aligned4(col, c, a, bf16), item_deg, mx, mx + 1, bad);
    DLM_CK(cudaGetLastError());
    if (measure) {  // no layout is built: the items' repeats are checked apart
      const size_t dsm = sizeof(unsigned) * static_cast<size_t>((J + 31) / 32) * (kDupThreads / 32);
      DLM_CK(cudaFuncSetAttribute(k_dups, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit));
      const int64_t want = (I + kDupThreads - 1) / kDupThreads;
      const int gd = static_cast<int>(want < 8LL * sms ? (want > 0 ? want : 1) : 8LL * sms);
      k_dups<<<gd, kDupThreads, dsm, s>>>(rp, col, I, J, bad);
    }
  }
  DLM_CK(cudaGetLastError());
  DLM_CK(cudaMemcpyAsync(&h_bad, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
  DLM_CK(cudaMemcpyAsync(h_mx, mx, sizeof(unsigned) * 2, cudaMemcpyDeviceToHost, s));
  h_deg.resize(J > 0 ? J : 1);
  DLM_CK(cudaMemcpyAsync(h_deg.data(), item_deg, sizeof(unsigned long long) * h_deg.size(), cudaMemcpyDeviceToHost,
                         s));
  DLM_CK(cudaStreamSynchronize(s));
  lap(0);
  if (h_bad & kBadItem) {
    *msg = "item_idx out of range [0, num_items)";
    st = DLM_ERR_INVALID_ARG;
    goto done;
  }
  if (h_bad & kBadValue) {
    *msg = "c and a must be finite";
    st = DLM_ERR_INVALID_ARG;
    goto done;
  }
  if (h_bad & kDupItem) {
    *msg = kDupMsg;
    st = DLM_ERR_INVALID_ARG;
    goto done;
  }
  out->a_nonneg = !(h_bad & kNegA);
  {
    float fa, fc;
    memcpy(&fa, &h_mx[0], 4);
    memcpy(&fc, &h_mx[1], 4);
    out->max_abs_a = fa;
    out->max_abs_c = fc;
  }
  out->max_item_deg = 0;
  for (int64_t j = 0; j < J; ++j)
    if (static_cast<int64_t>(h_deg[j]) > out->max_item_deg) out->max_item_deg = static_cast<int64_t>(h_deg[j]);
  if (measure) {
    measure->nnz = nnz;
    measure->active_users = I - static_cast<int64_t>(h_zero);
    measure->max_item_deg = out->max_item_deg;
    measure->max_abs_a = out->max_abs_a;
    measure->max_abs_c = out->max_abs_c;
    measure->a_nonneg = out->a_nonneg;
    measure->item_deg.assign(h_deg.begin(), h_deg.begin() + J);
    goto done;
  }
  if (shard) {  // bounds of the whole instance: the fixed-point exponents must agree on every shard
    out->max_item_deg = shard->max_item_deg;
    out->max_abs_a = shard->max_abs_a;
    out->max_abs_c = shard->max_abs_c;
    out->a_nonneg = shard->a_nonneg;
  }

  // ---- stable sort of users by degree, largest first ----
  In = I - static_cast<int64_t>(h_zero);
  ns = (In + 31) / 32;
  out->num_active_users = In;
  out->nslices = ns;
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&sdeg), sizeof(int32_t) * (I + 32), s));
  DLM_CK(cudaMemsetAsync(sdeg, 0, sizeof(int32_t) * (I + 32), s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&idx), sizeof(int32_t) * (I > 0 ? I : 1), s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&perm), sizeof(int32_t) * (I > 0 ? I : 1), s));
  if (I > 0) {
    k_iota<<<grid_for(I), kT, 0, s>>>(idx, I);
    DLM_CK(cudaGetLastError());
    DLM_CK(cub::DeviceRadixSort::SortPairsDescending(nullptr, tmp_bytes, deg, sdeg, idx, perm, I, 0, 32, s));
    DLM_CK(dev_alloc(reinterpret_cast<void**>(&tmp), tmp_bytes > 0 ? tmp_bytes : 16, s));
    DLM_CK(cub::DeviceRadixSort::SortPairsDescending(tmp, tmp_bytes, deg, sdeg, idx, perm, I, 0, 32, s));
    dev_free(tmp, s);
    tmp = nullptr;
  }

  // ---- slices ----
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&out->slice_w), sizeof(int32_t) * (ns + 1), s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&out->slice_off), sizeof(int64_t) * (ns + 1), s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&ssize), sizeof(int64_t) * (ns + 1), s));
  DLM_CK(cudaMemsetAsync(out->slice_off, 0, sizeof(int64_t), s));
  if (ns > 0) {
    k_slices<<<grid_for(ns), kT, 0, s>>>(sdeg, ns, bf16, out->slice_w, ssize);
    DLM_CK(cudaGetLastError());
    tmp_bytes = 0;
    DLM_CK(cub::DeviceScan::InclusiveSum(nullptr, tmp_bytes, ssize, out->slice_off + 1, ns, s));
    DLM_CK(dev_alloc(reinterpret_cast<void**>(&tmp), tmp_bytes > 0 ? tmp_bytes : 16, s));
    DLM_CK(cub::DeviceScan::InclusiveSum(tmp, tmp_bytes, ssize, out->slice_off + 1, ns, s));
    dev_free(tmp, s);
    tmp = nullptr;
  }
  DLM_CK(cudaMemcpyAsync(&out->padded_nnz, out->slice_off + ns, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  DLM_CK(cudaStreamSynchronize(s));
  lap(1);

  // ---- edge streams in slice order (16-bit item indices: every handle has
  // fewer than 65,536 items) ----
  if (J > 65536) {
    *msg = "num_items above 65,536";
    st = DLM_ERR_UNSUPPORTED;
    goto done;
  }
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&out->col16), sizeof(uint16_t) * (out->padded_nnz + 64), s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&out->ca), 2 * vs * (out->padded_nnz + 32), s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&out->orig_off), sizeof(int64_t) * (In + 32), s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&out->udeg), sizeof(int32_t) * (In + 32), s));
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&out->lead), sizeof(uint64_t) * (In + 32), s));
  DLM_CK(cudaMemsetAsync(out->col16 + out->padded_nnz, 0, sizeof(uint16_t) * 64, s));
  if (ns > 0) {
    // `bad` has been read: its words serve as the slice counter and the flag of a repeated item
    DLM_CK(cudaMemsetAsync(bad, 0, 2 * sizeof(int), s));
    unsigned* ticket = reinterpret_cast<unsigned*>(bad);
    int dev = 0, sms = 0;
    DLM_CK(cudaGetDevice(&dev));
    DLM_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int gsm = kGatherWarps * (kStripElems * static_cast<int>(2 + 2 * vs) + 4 * static_cast<int>((J + 31) / 32));
    // blocks that fit at once, or one a slice (a block takes a slice of long rows, a warp another)
    const int g = static_cast<int>(std::min<int64_t>(ns, static_cast<int64_t>(sms) * (bf16 ? 4 : 2)));
    if (bf16) {
      DLM_CK(cudaFuncSetAttribute(&k_gather<uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit));
      k_gather<uint32_t><<<g, 32 * kGatherWarps, gsm, s>>>(rp, col, c, a, perm, sdeg, In, ns, out->slice_off,
                                                           out->slice_w, out->col16, static_cast<uint32_t*>(out->ca),
                                                           out->orig_off, out->udeg, out->lead, static_cast<int>(J),
                                                           ticket, bad + 1);
    } else {
      DLM_CK(cudaFuncSetAttribute(&k_gather<float2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit));
      k_gather<float2><<<g, 32 * kGatherWarps, gsm, s>>>(rp, col, c, a, perm, sdeg, In, ns, out->slice_off,
                                                         out->slice_w, out->col16, static_cast<float2*>(out->ca),
                                                         out->orig_off, out->udeg, out->lead, static_cast<int>(J),
                                                           ticket, bad + 1);
    }
    DLM_CK(cudaGetLastError());
  }

  // ---- n_j = sum_i a_ij^2 and s_j = sum_i a_ij (exact fixed point; the
  // whole instance's sums for a shard) ----
  if (shard) {
    DLM_CK(cudaMemcpyAsync(&h_dup, bad + 1, sizeof(int), cudaMemcpyDeviceToHost, s));
    DLM_CK(cudaStreamSynchronize(s));
    int sq_shift = 0, s1_shift = 0;
    item_sum_shifts(out->max_item_deg, out->max_abs_a, &sq_shift, &s1_shift);
    out->h_n2.assign(J > 0 ? J : 1, 0.0);
    out->h_s1.assign(J > 0 ? J : 1, 0.0);
    out->n2max = 0;
    for (int64_t j = 0; j < J; ++j) {
      out->h_n2[j] = static_cast<double>(shard->item_sq[j]) * std::ldexp(1.0, -sq_shift);
      out->h_s1[j] = static_cast<double>(shard->item_sum[j]) * std::ldexp(1.0, -s1_shift);
      out->n2max = out->h_n2[j] > out->n2max ? out->h_n2[j] : out->n2max;
    }
    DLM_CK(cudaStreamSynchronize(s));
    lap(2);
    goto checked;
  }
  item_sum_shifts(out->max_item_deg, out->max_abs_a, &ssq, &ss1);
  DLM_CK(dev_alloc(reinterpret_cast<void**>(&sq), sizeof(unsigned long long) * 2 * (J > 0 ? J : 1), s));
  DLM_CK(launch_item_sums(col, a, bf16, nnz, J, ssq, ss1, sq, s));
  {
    std::vector<unsigned long long> q(2 * static_cast<size_t>(J > 0 ? J : 1));
    DLM_CK(cudaMemcpyAsync(&h_dup, bad + 1, sizeof(int), cudaMemcpyDeviceToHost, s));
    DLM_CK(cudaMemcpyAsync(q.data(), sq, sizeof(unsigned long long) * q.size(), cudaMemcpyDeviceToHost, s));
    DLM_CK(cudaStreamSynchronize(s));
    out->h_n2.assign(J > 0 ? J : 1, 0.0);
    out->h_s1.assign(J > 0 ? J : 1, 0.0);
    out->n2max = 0;
    for (int64_t j = 0; j < J; ++j) {
      out->h_n2[j] = static_cast<double>(static_cast<long long>(q[j])) * std::ldexp(1.0, -ssq);
      out->h_s1[j] = static_cast<double>(static_cast<long long>(q[J + j])) * std::ldexp(1.0, -ss1);
      out->n2max = out->h_n2[j] > out->n2max ? out->h_n2[j] : out->n2max;
    }
  }
  lap(2);
checked:
  if (ns > 0 && h_dup) {
    *msg = kDupMsg;
    st = DLM_ERR_INVALID_ARG;
  }
  goto done;

fail:
  st = DLM_ERR_CUDA;
done:
  dev_free(deg, s);
  dev_free(sdeg, s);
  dev_free(idx, s);
  dev_free(perm, s);
  dev_free(ssize, s);
  dev_free(zero_cnt, s);
  dev_free(item_deg, s);
  dev_free(sq, s);
  dev_free(mx, s);
  dev_free(bad, s);
  dev_free(tmp, s);
  if (st != DLM_OK) {
    dev_free(out->slice_w, s);
    dev_free(out->slice_off, s);
    dev_free(out->col16, s);
    dev_free(out->ca, s);
    dev_free(out->orig_off, s);
    dev_free(out->udeg, s);
    dev_free(out->lead, s);
    out->slice_w = nullptr;
    out->slice_off = nullptr;
    out->col16 = nullptr;
    out->ca = nullptr;
    out->orig_off = nullptr;
    out->udeg = nullptr;
    out->lead = nullptr;
  }
  return st;
}

}  // namespace dlm
