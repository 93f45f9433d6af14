// Per-node top-k of the logits (Sec. 3.1 "Progressive Expansion" and "Width Control":
// each node's draft token d_v and at most k children; Sec. 3.2: the greedy verification
// token V_n is entry 0).  Pure HBM streaming.
//
// One kernel: a row's parts to the CTAs of a cluster, merged through distributed shared memory (no
// global scratch), or, for the step's large batches, to single CTAs that merge through scratch.
//
// Order: a 64-bit key (order-preserving bits of the fp32 value) << 32 | ~index, so a
// larger key is a larger value or, on equal values, a lower index.  -0.0 is folded into
// +0.0 before the key is formed.  NaN come after every number, in the order of their indices.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "launch.cuh"
#include "ptd_device.cuh"
#include "topk.cuh"
#include "verify_tree.cuh"

namespace cg = cooperative_groups;

namespace ptd {
namespace topk {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxCluster = 8;

__device__ __forceinline__ uint32_t ordered_bits(float f) {
  uint32_t u = __float_as_uint(f);
  if (u == 0x80000000u) u = 0u;   // -0.0 == +0.0
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float from_ordered(uint32_t o) {
  const uint32_t u = (o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o;
  return __uint_as_float(u);
}

__device__ __forceinline__ uint64_t make_key(uint32_t ord, uint32_t idx) {
  return ((uint64_t)ord << 32) | (uint64_t)(~idx);
}

// Largest key of the warp: the largest high word (one warp reduction), then the largest low
// word among the lanes that hold it (a second one).
__device__ __forceinline__ uint64_t warp_max_u64(uint64_t v) {
  const uint32_t hi = (uint32_t)(v >> 32);
  const uint32_t mhi = __reduce_max_sync(0xffffffffu, hi);
  const uint32_t mlo = __reduce_max_sync(0xffffffffu, hi == mhi ? (uint32_t)v : 0u);
  return ((uint64_t)mhi << 32) | mlo;
}

template <typename T>
struct Vec;
template <>
struct Vec<__nv_bfloat16> {
  static constexpr int kN = 8;
  __device__ __forceinline__ static void unpack(const uint4& v, float (&f)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      f[2 * j] = __uint_as_float(w[j] << 16);
      f[2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
    }
  }
  __device__ __forceinline__ static float scalar(const __nv_bfloat16* p) {
    return __uint_as_float((uint32_t)(*reinterpret_cast<const uint16_t*>(p)) << 16);
  }
};
template <>
struct Vec<float> {
  static constexpr int kN = 4;
  __device__ __forceinline__ static void unpack(const uint4& v, float (&f)[8]) {
    f[0] = __uint_as_float(v.x);
    f[1] = __uint_as_float(v.y);
    f[2] = __uint_as_float(v.z);
    f[3] = __uint_as_float(v.w);
  }
  __device__ __forceinline__ static float scalar(const float* p) { return *p; }
};

// ------------------------------------------------------------------ the step's verification
// Trees that no row can complete (an empty or out-of-range node range, or offsets that do not
// run from 0 to n_total): their outputs and the status are written at once (one warp).
__device__ __forceinline__ void flag_bad_trees_warp(const VerifyArgs& va) {
  const int lane = threadIdx.x & 31;
  for (int b = lane; b < va.batch; b += 32) {
    const int n0 = va.node_offsets[b], n1 = va.node_offsets[b + 1];
    const bool bad = n1 - n0 < 1 || n1 - n0 > va.max_nodes || n0 < 0 || n1 > va.n_total ||
                     (b == 0 && n0 != 0) || (b == va.batch - 1 && n1 != va.n_total);
    if (bad) {
      for (int j = 0; j < va.max_nodes; ++j) va.accepted[(size_t)b * va.max_nodes + j] = -1;
      va.accept_len[b] = 0;
      va.bonus[b] = -1;
      atomicMax(va.dev_status, (int)PTD_ERR_INVALID_TREE);
    }
  }
}

// Greedy verification of tree b on the calling warp, on column 0 of the top-k rows already
// written (and made visible to this warp), and the tree's outputs.
__device__ __forceinline__ void verify_and_write_warp(const VerifyArgs& va, int b, const vt::TreeInputs& tin,
                                                      const int32_t* out_idx, int k, vt::VerifyScratch& sc,
                                                      vt::TreeVerdict& vd) {
  const int lane = threadIdx.x & 31;
  vt::verify_tree_warp(tin, out_idx, k, sc, &vd);
  __syncwarp();
  int len = vd.len;
  if (len > va.max_nodes) len = va.max_nodes;
  int32_t* acc_row = va.accepted + (size_t)b * va.max_nodes;
  for (int j = lane; j < va.max_nodes; j += 32) acc_row[j] = j < len ? vd.path[j] : -1;
  if (lane == 0) {
    va.accept_len[b] = len;
    va.bonus[b] = vd.bonus;
    if (vd.invalid) atomicMax(va.dev_status, (int)PTD_ERR_INVALID_TREE);
  }
}

// ------------------------------------------------------------------ selection
// A row (bf16 or fp32 logits) is cut into contiguous parts, one CTA each:
//   1. every lane's maximum over its vectors, and of each eight lanes' (32 groups over the CTA);
//   2. T = the k-th largest of the 32 group maxima: k elements of the part are >= T, so
//      nothing below T is among the part's top-k (about 32 ln(32 / (32 - k)) elements are
//      >= T: 4 for k = 4, 22 for k = 16);
//   3. the few lanes whose maximum reaches T read their vectors again (L2) and put the elements
//      >= T into a candidate buffer as 64-bit keys, in any order; a candidate's place among
//      the part's top-k is the number of larger candidates.
// A part whose candidates do not fit the buffer (long runs of equal values, or fewer than k
// groups above -inf), or that has NaN and fewer than k numbers (NaN is never >= T), selects by k
// rounds of "largest key below the last", so that every entry is written.  The parts' keys are
// placed among each other the same way:
//   kCluster, kClusterVerify  in the shared memory of the first CTA of the row's cluster, which
//       the others write to before they leave;
//   kWhole  (a row in one part) not at all: they are the row's entries (15 fp32 rows of 1000, k = 2: 3.0 us
//       with the merge, 2.4 without; 1500 rows 10.7 / 7.0);
//   kSlotsVerify  (the step's "streamed" form) by the CTA that counts in the row's last part,
//       from slots in global scratch: parts of all rows run one by one wherever an SM has
//       room, with no cluster to place, and a CTA leaves as soon as its part is done.
// With verification (the step's tail), whoever writes the last row of a tree then verifies that
// tree (greedy, on one warp), so no separate verification launch follows.
//
// The kernel holds little (40 registers a thread, ~8 KB of shared memory a CTA) so that in the
// step its CTAs fit beside the attention's and run while that does (`beside`, see below): a
// batched paged step 82.4 -> 55 us, one 8-head layer with 63 rows of 128256 logits 68.5 -> 30,
// the tiny fp32 step 13.4 -> 10.8, the 32-layer step ~240 -> ~236.
//
// What bounds it alone: for a few rows the chain of two reads, selection and merge; for many the
// reads in flight (four or eight 16-byte loads a thread, six or four CTAs per SM).  Measured (GB300; at first with
// per-thread sorted lists and k rounds of warp maxima at four levels, each thread's list taking
// every element for fp32), 128256 logits a row: fp32, 63 rows, k = 4 21.1 -> 7.8 us, k = 16
// 62.6 -> 10.2, 512 rows, k = 16 352 -> 61.4; bf16, 63 rows, k = 4 8.5 -> 7.3, 512 rows 39.6 -> 34.3
// (k = 16 102 -> 44.3).  Parts staged in shared memory by bulk copies took 32.1 us for the 512 bf16
// rows and 72.5 for the fp32 ones, but left no room beside the attention; a persistent grid
// with double-buffered parts took 66 (the chain of a row is longer than its copy).
constexpr int kTargetVec = 2048;   // 32 KB: the part that the cluster size aims at
constexpr int kMaxK = 16;
constexpr int kCand = 256;         // candidate buffer (keys)
constexpr int kCluster = 0, kClusterVerify = 1, kSlotsVerify = 2, kWhole = 3;

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
// Lane-wise maximum of two bf16 pairs in one instruction (exact: a maximum only compares)
__device__ __forceinline__ uint32_t bf16x2_max(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
constexpr uint32_t kBf16x2NegInf = 0xFF80FF80u;

// The largest logit of a 16-byte vector.
template <typename T>
__device__ __forceinline__ float vec_max(const uint4& x) {
  if constexpr (sizeof(T) == 2) {
    const uint32_t h = bf16x2_max(bf16x2_max(x.x, x.y), bf16x2_max(x.z, x.w));
    return fmaxf(bf16_lo(h), bf16_hi(h));
  } else {
    return fmax3(__uint_as_float(x.x), __uint_as_float(x.y), fmaxf(__uint_as_float(x.z), __uint_as_float(x.w)));
  }
}

// The k-th largest of the warp's 32 order-preserving values (0 = a lane without one), or 0 when
// fewer than k lanes hold one: one warp maximum and one ballot per distinct value, equal values
// counted together.  Any x with k elements >= x bounds the warp's top-k from below.
__device__ __forceinline__ uint32_t kth_largest_ord(uint32_t v, int k) {
  int count = 0;
  for (int s = 0; s < k; ++s) {
    const uint32_t m = __reduce_max_sync(0xffffffffu, v);
    if (m == 0u) return 0u;
    count += __popc(__ballot_sync(0xffffffffu, v == m));
    if (count >= k) return m;
    if (v == m) v = 0u;
  }
  return 0u;
}

// The k-th largest (k <= 32) of 32 shared values, by every warp on its own: a lane's value with
// k - 1 values before it (larger, or equal at a lower lane).
__device__ __forceinline__ uint32_t kth_of_32(const uint32_t* v_s, int k) {
  const int lane = threadIdx.x & 31;
  const uint32_t mine = v_s[lane];
  int before = 0;
#pragma unroll
  for (int i = 0; i < 32; i += 4) {
    const uint4 o = *reinterpret_cast<const uint4*>(v_s + i);
    before += (o.x > mine || (o.x == mine && i < lane)) + (o.y > mine || (o.y == mine && i + 1 < lane)) +
              (o.z > mine || (o.z == mine && i + 2 < lane)) + (o.w > mine || (o.w == mine && i + 3 < lane));
  }
  const uint32_t at = __ballot_sync(0xffffffffu, before == k - 1);
  return __shfl_sync(0xffffffffu, mine, __ffs(at) - 1);
}

// `beside`: the logits (and the trees) were complete before the stream's previous grid let this one
// be placed, so the CTAs start on them at once, beside that grid; the outputs and counters
// belong to no grid still running.  One CTA waits for the previous grid before it leaves, so
// that this grid's completion implies that one's.
// The counters that this kernel adds to (rows done per tree, parts done per row) were cleared by CTA 0 of that
// grid, and being placed makes nothing visible by itself.  What orders the two: CTA 0 stores the zeros, then
// fences device-wide, then (after a barrier) gives its permission, and this grid has no CTA before every CTA
// there has given it or left; the stores are then performed in L2, where the counts, atomics all of them, are
// made.  A plain load of a counter would have to wait for that grid.
//
// Vectors in flight per thread and CTAs per SM (registers).  Kernels that run beside the tensor-core
// attention keep to four and 40 registers, and bf16 rows do best so (eight: 512 rows of 128256
// 34.3 -> 43.8 us); a part of fp32 logits is twice as many vectors (four -> eight: 63 rows 11.2 -> 7.8
// us, 512 rows with k = 16 59.2 -> 61.4).
template <typename T, int kMode>
struct Depth {
  static constexpr bool kDeep = (kMode == kCluster || kMode == kWhole) && sizeof(T) == 4;
  static constexpr int kLoads = kDeep ? 8 : 4, kCtas = kDeep ? 4 : 6;
};

template <typename T, int kMode>
__global__ void __launch_bounds__(kThreads, Depth<T, kMode>::kCtas)
    topk_rows_kernel(const T* __restrict__ logits, int64_t rows, int vocab, int64_t row_stride, int k, int per, int beside,
                     int32_t* __restrict__ out_idx, float* __restrict__ out_val, int32_t* dev_status,
                     unsigned int* row_counters, unsigned long long* slots, const __grid_constant__ VerifyArgs va) {
  constexpr int VN = Vec<T>::kN, kLoads = Depth<T, kMode>::kLoads;
  constexpr bool kClustered = kMode == kCluster || kMode == kClusterVerify;
  __shared__ __align__(16) uint64_t cand_s[kCand];
  __shared__ __align__(16) uint64_t all_keys[kMaxCluster * kMaxK];   // the row's parts' keys, at its last merger
  __shared__ __align__(16) uint32_t group_max_s[32];
  __shared__ __align__(8) uint64_t keys_bar_s;
  __shared__ uint64_t round_s[kWarps];
  __shared__ int n_cand_s, abort_s, last_s;

  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)blockIdx.x, parts = (int)gridDim.x;   // the grid's x is one row's parts
  const int64_t r = (int64_t)blockIdx.z * gridDim.y + blockIdx.y;
  const bool waiter = beside != 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;
  if (r >= rows) return;   // the whole cluster
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t keys_bar = smem_u32(&keys_bar_s);
  if (tid == 0) {
    if (kClustered) {
      mbar_init(keys_bar, (uint32_t)(parts * k));   // one arrival per key (rank 0's is used)
      fence_mbar_init();
    }
    abort_s = 0;
    n_cand_s = 0;
  }
  if (kMode != kWhole && rank == 0 && tid < kMaxCluster * kMaxK) all_keys[tid] = 0ull;
  __syncthreads();
  if (tid == 0) grid_launch_dependents();   // the next grid may be placed now; it waits for this one
  // the cluster's CTAs are there and rank 0's keys and barrier are set up (waited for before the
  // first key is sent)
  if (kClustered) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  if (!beside) grid_dependency_wait();   // the logits, the trees and the outputs belong to the stream's previous work
  // this CTA's part: the vector body starts at the row's first 16-byte boundary (head and tail
  // elements outside it go to the first and last CTA one by one)
  const T* row = logits + r * row_stride;
  int a0 = (int)(((16 - (reinterpret_cast<uintptr_t>(row) & 15)) & 15) / sizeof(T));
  if (a0 > vocab) a0 = vocab;
  const int nvec = (vocab - a0) / VN;
  const int a1 = a0 + nvec * VN;
  const int v_begin = min(nvec, rank * per), nv = min(nvec, v_begin + per) - v_begin;
  const uint4* vrow = reinterpret_cast<const uint4*>(row + a0) + v_begin;
  const bool own_head = rank == 0 && tid == 0, own_tail = rank == parts - 1 && tid == kThreads - 1;
  if constexpr (kMode == kClusterVerify || kMode == kSlotsVerify) {
    // Trees that no row completes (an empty or out-of-range node range, or offsets that do not
    // run from 0 to n_total): their outputs and the status are written here, by warp 1 of the
    // first CTA; a tree whose rows all arrive is verified below.
    if (r == 0 && rank == 0 && warp == 1) flag_bad_trees_warp(va);
  }

  // 1. lane maxima, then of eight lanes
  float tmax = -INFINITY;
  {
    constexpr uint32_t kNone = VN == 8 ? kBf16x2NegInf : 0xFF800000u;   // -inf
    uint32_t h0 = kBf16x2NegInf, h1 = kBf16x2NegInf;
    float m0 = -INFINITY, m1 = -INFINITY;
#pragma unroll 1
    for (int v0 = tid; v0 < nv; v0 += kLoads * kThreads) {
      uint4 x[kLoads];
#pragma unroll
      for (int u = 0; u < kLoads; ++u) {
        const int v = v0 + u * kThreads;
        x[u] = v < nv ? __ldg(vrow + v) : make_uint4(kNone, kNone, kNone, kNone);
      }
#pragma unroll
      for (int u = 0; u < kLoads; ++u) {
        if constexpr (VN == 8) {
          h0 = bf16x2_max(h0, bf16x2_max(x[u].x, x[u].y));
          h1 = bf16x2_max(h1, bf16x2_max(x[u].z, x[u].w));
        } else {
          m0 = fmax3(m0, __uint_as_float(x[u].x), __uint_as_float(x[u].y));
          m1 = fmax3(m1, __uint_as_float(x[u].z), __uint_as_float(x[u].w));
        }
      }
    }
    if constexpr (VN == 8) {
      h0 = bf16x2_max(h0, h1);
      tmax = fmaxf(bf16_lo(h0), bf16_hi(h0));
    } else {
      tmax = fmaxf(m0, m1);
    }
  }
  float smax = tmax;   // with the head and tail elements
  if (own_head)
    for (int i = 0; i < a0; ++i) smax = fmaxf(smax, Vec<T>::scalar(row + i));
  if (own_tail)
    for (int i = a1; i < vocab; ++i) smax = fmaxf(smax, Vec<T>::scalar(row + i));
  {
    const bool has_elems = tid < nv || (own_head && a0 > 0) || (own_tail && a1 < vocab);
    uint32_t o = has_elems ? ordered_bits(smax) : 0u;
#pragma unroll
    for (int d = 1; d < 8; d <<= 1) o = max(o, __shfl_xor_sync(0xffffffffu, o, d));
    if ((lane & 7) == 0) group_max_s[warp * 4 + (lane >> 3)] = o;
  }
  __syncthreads();

  // 2. T (0: fewer than k groups hold elements, so every element is a candidate)
  const uint32_t kth = k <= 8 ? kth_largest_ord(group_max_s[lane], k) : kth_of_32(group_max_s, k);
  const float thr = kth != 0u ? from_ordered(kth) : -INFINITY;

  // 3. the candidates
  auto push = [&](float f, uint32_t idx) {
    const int at = atomicAdd(&n_cand_s, 1);
    if (at < kCand) cand_s[at] = make_key(ordered_bits(f), idx);
  };
  if (own_head)
    for (int i = 0; i < a0; ++i) {
      const float f = Vec<T>::scalar(row + i);
      if (f >= thr) push(f, (uint32_t)i);
    }
  if (own_tail)
    for (int i = a1; i < vocab; ++i) {
      const float f = Vec<T>::scalar(row + i);
      if (f >= thr) push(f, (uint32_t)i);
    }
  if (tmax >= thr) {   // about k lanes of the 256
#pragma unroll 1
    for (int v0 = tid; v0 < nv; v0 += kLoads * kThreads) {
      uint4 x[kLoads];
#pragma unroll
      for (int u = 0; u < kLoads; ++u) x[u] = __ldg(vrow + min(v0 + u * kThreads, nv - 1));
      if (*(volatile int*)&n_cand_s > kCand) break;   // the buffer is already lost
#pragma unroll
      for (int u = 0; u < kLoads; ++u) {
        const int v = v0 + u * kThreads;
        if (v < nv && vec_max<T>(x[u]) >= thr) {
          float f[8];
          Vec<T>::unpack(x[u], f);
          const uint32_t i0 = (uint32_t)(a0 + (v_begin + v) * VN);
#pragma unroll
          for (int e = 0; e < VN; ++e)
            if (f[e] >= thr) push(f[e], i0 + e);
        }
      }
    }
  }
  __syncthreads();
  if (kClustered) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  // where a key of this part goes: rank 0's shared memory, with an arrival that releases it, or the
  // part's slot
  uint64_t* dst_keys = nullptr;
  uint32_t dst_bar = 0;
  if constexpr (kClustered) {
    dst_keys = cluster.map_shared_rank(all_keys, 0) + rank * kMaxK;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(dst_bar) : "r"(keys_bar));
  } else if constexpr (kMode == kSlotsVerify) {
    dst_keys = reinterpret_cast<uint64_t*>(slots) + (r * parts + rank) * k;
  }
  auto write_entry = [&](int at, uint64_t key) {   // entry `at` of the row
    out_idx[r * k + at] = (int32_t)(~(uint32_t)(key & 0xFFFFFFFFull));
    out_val[r * k + at] = from_ordered((uint32_t)(key >> 32));
  };
  auto arrive = [&](int count) {
    if constexpr (kClustered)
      asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(dst_bar), "r"(count)
                   : "memory");
  };
  const int n = n_cand_s;
  const int n_elems = nv * VN + (rank == 0 ? a0 : 0) + (rank == parts - 1 ? vocab - a1 : 0);
  if (n <= kCand && n >= min(k, n_elems)) {
    for (int i = tid; i < n; i += kThreads) {
      const uint64_t key = cand_s[i];
      int before = 0;
      for (int j = 0; j < n; ++j) before += cand_s[j] > key ? 1 : 0;
      if (before < k) {
        if constexpr (kMode == kWhole) {
          write_entry(before, key);
        } else {
          dst_keys[before] = key;
          arrive(1);
        }
      }
    }
    if (kMode != kWhole && n < k) {   // fewer elements than k in this part
      if (kMode == kSlotsVerify) {
        if (tid >= n && tid < k) dst_keys[tid] = 0ull;
      } else if (tid == 0) {
        arrive(k - n);
      }
    }
  } else {
    // k rounds over the part (rare; every thread takes part); 0 is below every number's order
    uint64_t last = ~0ull;
    for (int q = 0; q < k; ++q) {
      uint64_t best = 0ull;
      auto take = [&](float f, uint32_t idx) {
        const uint64_t key = make_key(f == f ? ordered_bits(f) : 0u, idx);
        if (key < last && key > best) best = key;
      };
      if (own_head)
        for (int i = 0; i < a0; ++i) take(Vec<T>::scalar(row + i), (uint32_t)i);
      if (own_tail)
        for (int i = a1; i < vocab; ++i) take(Vec<T>::scalar(row + i), (uint32_t)i);
      for (int v = tid; v < nv; v += kThreads) {
        float f[8];
        Vec<T>::unpack(__ldg(vrow + v), f);
#pragma unroll
        for (int e = 0; e < VN; ++e) take(f[e], (uint32_t)(a0 + (v_begin + v) * VN + e));
      }
      best = warp_max_u64(best);
      if (lane == 0) round_s[warp] = best;
      __syncthreads();
      best = round_s[0];
#pragma unroll
      for (int w = 1; w < kWarps; ++w) best = best > round_s[w] ? best : round_s[w];
      if (tid == 0) {
        if constexpr (kMode == kWhole) {
          write_entry(q, best);
        } else {
          dst_keys[q] = best;
          arrive(1);
        }
      }
      last = best;
      __syncthreads();   // round_s is read
    }
  }

  // ---- the row's top-k from its parts' keys
  constexpr int kMergers = kMaxCluster * kMaxK;   // the first four warps
  bool merger = kMode != kWhole && rank == 0;
  if constexpr (kMode == kSlotsVerify) {
    __syncthreads();   // the part's keys are written before it is counted
    if (tid == 0) last_s = (int)atom_add_acq_rel_gpu(row_counters + r, 1u) + 1 == parts ? 1 : 0;
    __syncthreads();
    merger = last_s != 0;
  }
  if (merger && tid < kMergers) {
    const int q = tid / kMaxK, at = tid % kMaxK;
    uint64_t key;
    if constexpr (kMode == kSlotsVerify) {
      key = q < parts && at < k ? __ldcg(slots + (r * parts + q) * k + at) : 0ull;
      all_keys[tid] = key;
      asm volatile("bar.sync 1, %0;" ::"n"(kMergers) : "memory");
    } else {
      mbar_wait_cluster(keys_bar, 0u, &abort_s, dev_status);
      key = all_keys[tid];
    }
    if (key != 0ull) {
      int before = 0;
      for (int c = 0; c < parts; ++c)
        for (int j = 0; j < k; ++j) before += all_keys[c * kMaxK + j] > key ? 1 : 0;
      if (before < k) write_entry(before, key);
    }
    if constexpr (kMode == kClusterVerify || kMode == kSlotsVerify) {
      // the last row of a tree to be written: its tree is verified
      asm volatile("bar.sync 1, %0;" ::"n"(kMergers) : "memory");   // the row's entries precede its count
      if (warp == 0) {
        int lo = 0, hi = va.batch;   // the tree of the row
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (va.node_offsets[mid] <= r) lo = mid; else hi = mid;
        }
        int vb = -1;
        if (lane == 0) {
          // release: this row's top-k before its count; acquire: the other rows' top-k (each
          // written before its own count) before this warp reads them
          if ((int)atom_add_acq_rel_gpu(va.counters + lo, 1u) + 1 == va.node_offsets[lo + 1] - va.node_offsets[lo]) vb = lo;
        }
        vb = __shfl_sync(0xffffffffu, vb, 0);
        if (vb >= 0) {
          __shared__ vt::VerifyScratch vsc;
          __shared__ vt::TreeVerdict verdict;
          __syncwarp();   // lane 0's acquire precedes every lane's reads of the tree's rows
          vt::TreeInputs tin;
          vt::load_tree_warp(va.node_offsets, va.parents, va.tokens, va.n_total, va.max_nodes, vb, tin);
          verify_and_write_warp(va, vb, tin, out_idx, k, vsc, verdict);
        }
      }
    }
  }
  if (waiter) grid_dependency_wait();
}

// Parts of a row: 32 KB each, at most eight.
template <typename T>
int row_parts(int vocab) {
  const int64_t c = ((int64_t)vocab / Vec<T>::kN + kTargetVec) / kTargetVec;
  return c > kMaxCluster ? kMaxCluster : (int)c;
}

template <typename T, int kMode>
cudaError_t launch_rows(const T* logits, int64_t rows, int vocab, int64_t row_stride, int k, int parts, int beside,
                        int32_t* out_idx, float* out_val, int32_t* dev_status, unsigned int* row_counters,
                        unsigned long long* slots, const VerifyArgs& va, cudaStream_t stream) {
  const int per = (vocab / Vec<T>::kN + parts - 1) / parts;   // vectors per CTA (rows off 16 bytes have one fewer)
  const unsigned gy = (unsigned)(rows < 32768 ? rows : 32768), gz = (unsigned)((rows + gy - 1) / gy);
  return launch_chained(topk_rows_kernel<T, kMode>, dim3((unsigned)parts, gy, gz), dim3(kThreads), 0, stream,
                        kMode == kSlotsVerify || kMode == kWhole ? 0u : (unsigned)parts, logits, rows, vocab, row_stride, k, per, beside,
                        out_idx, out_val, dev_status, row_counters, slots, va);
}

// Parts of each of many rows: where 32 KB parts are more CTAs than run at once, the next power of two
// below that fits, while a part stays under 128 KB.  GB300, us, 32 KB parts -> these: 300 bf16 rows of 50257,
// k = 1 9.0 -> 7.4, 700 rows 17.2 -> 11.3; fp32, 300 rows of 50257 15.0 -> 8.3, 512 rows of 32000 13.7 -> 7.7;
// over 600 sizes 8 % less on average, none more than 2 % slower.
template <typename T>
int row_parts_of_many(int vocab, int64_t rows, int sms) {
  const int most = row_parts<T>(vocab);
  const int64_t slots = (int64_t)Depth<T, kCluster>::kCtas * sms, bytes = (int64_t)vocab * (int64_t)sizeof(T);
  if (rows * most <= slots) return most;
  int parts = kMaxCluster;
  while (parts > 1 && (parts >= most || rows * parts > slots) && bytes / (parts / 2) <= 128000) parts /= 2;
  return parts < most ? parts : most;
}

template <typename T>
cudaError_t launch_plain(const T* logits, int64_t rows, int vocab, int64_t row_stride, int k, int beside,
                         int32_t* out_idx, float* out_val, int32_t* dev_status, int sms, cudaStream_t stream) {
  constexpr int64_t kMost = 32768ll * 32768;   // rows of one grid
  const int parts = beside ? row_parts<T>(vocab) : row_parts_of_many<T>(vocab, rows, sms);
  for (int64_t r = 0; r < rows; r += kMost) {
    auto* const launch = parts == 1 ? launch_rows<T, kWhole> : launch_rows<T, kCluster>;
    const cudaError_t e = launch(logits + r * row_stride, rows - r < kMost ? rows - r : kMost, vocab, row_stride, k, parts,
                                 beside, out_idx + r * k, out_val + r * k, dev_status, nullptr, nullptr, VerifyArgs{},
                                 stream);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace topk

bool topk_stream_ok(const void* logits, int vocab) {
  return vocab >= 8 && vocab % 8 == 0 && (reinterpret_cast<uintptr_t>(logits) & 15u) == 0;
}

size_t topk_stream_slot_bytes(int64_t rows) {
  return (size_t)rows * topk::kMaxK * sizeof(unsigned long long);
}

cudaError_t launch_topk_stream(const void* logits, int64_t rows, int vocab, int k, bool beside, int32_t* out_idx,
                               float* out_val, int32_t* dev_status, const VerifyArgs& va, unsigned int* row_counters,
                               unsigned long long* slots, cudaStream_t stream) {
  if (!topk_stream_ok(logits, vocab) || rows < 1 || k < 1 || k > topk::kMaxK) return cudaErrorInvalidValue;
  int parts = topk::row_parts<__nv_bfloat16>(vocab);
  if (parts * k > topk::kMaxK) parts = topk::kMaxK / k;   // a row's slots hold kMaxK keys
  return topk::launch_rows<__nv_bfloat16, topk::kSlotsVerify>(static_cast<const __nv_bfloat16*>(logits), rows, vocab, vocab,
                                                              k, parts, beside ? 1 : 0, out_idx, out_val, dev_status,
                                                              row_counters, slots, va, stream);
}

int topk_slices(int vocab) { return (int)(((int64_t)vocab / 8 + 4096) / 4096); }

cudaError_t launch_topk(const void* logits, bool bf16, int64_t rows, int vocab, int64_t row_stride, int k, bool beside,
                        int32_t* out_idx, float* out_val, int32_t* dev_status, const VerifyArgs* va, int sms,
                        cudaStream_t stream) {
  if (va != nullptr) {
    if (!bf16) return cudaErrorInvalidValue;
    // Beside the attention an SM takes one or two CTAs: no more parts than one wave of six per SM
    // holds, as a cluster also waits for all its places (322 rows of 128256 with the step 61.3 ->
    // 57.1 us, 640 rows 76.1 -> 69.0).  Alone, or without clusters, full parts are no slower.
    const int64_t wave = (6 * (int64_t)sms + rows - 1) / rows;
    int parts = topk::row_parts<__nv_bfloat16>(vocab);
    if (parts > wave) parts = (int)wave;
    return topk::launch_rows<__nv_bfloat16, topk::kClusterVerify>(
        static_cast<const __nv_bfloat16*>(logits), rows, vocab, row_stride, k, parts, beside ? 1 : 0,
        out_idx, out_val, dev_status, nullptr, nullptr, *va, stream);
  }
  if (bf16)
    return topk::launch_plain(static_cast<const __nv_bfloat16*>(logits), rows, vocab, row_stride, k, beside ? 1 : 0,
                              out_idx, out_val, dev_status, sms, stream);
  return topk::launch_plain(static_cast<const float*>(logits), rows, vocab, row_stride, k, beside ? 1 : 0, out_idx,
                            out_val, dev_status, sms, stream);
}

}  // namespace ptd
