// Tree-masked attention in fp32 on the CUDA cores, and the choice between it and the kernel that
// splits fp32 operands for the tensor cores (D = 128, many rows and keys).
//
// Same operation as the tensor-core kernel (Sec. 3.1 ancestor-only visibility over the
// committed prefix plus the tree, Sec. 3.2), and the same dense view of it: the T nodes times
// the G query heads of a KV head form M = T * G rows that share every K/V row.  A unit is one
// (layer, tree, KV head, block of BM rows); a cluster of `csize` CTAs computes it, CTA r taking
// the r-th share of the keys, and the CTAs' partial softmax states (m, l, O) are combined
// through distributed shared memory, so the split needs no scratch and no second launch.
//
// In a CTA (128 threads as 8 row groups x 16 lanes) keys come in tiles of 64 whose K and V one
// thread brings in by TMA (K of the next tile during this tile's P V, V during its Q K^T; row
// copies issued by a warp's lanes held the other warps up at the next barrier).  Thread (row
// group, lane g) scores its RM = BM / 8 rows against keys g + 16 j (packed fp32 pairs over two
// columns, fma.rn.f32x2, so Q and K are used as they lie; K in 32-column boxes with the 128-byte
// swizzle, so that eight consecutive keys' 16-byte reads hit distinct banks), the row maxima
// reduce over the 16 lanes, P goes transposed to shared memory, and the thread accumulates RM
// rows x D / 16 columns of O (pairs over two rows).
//
// What bounds it: shared-memory reads and the fp32 FMA pipe (an 8 x 4 tile of S reads 12 floats
// per 32 FMAs, an 8 x 8 tile of O 16 per 64; the pipe gives ~110 FMA per cycle and SM) for many
// rows, the latency of a tile's chain and the K/V stream for few.  Measured (GB300, one layer,
// against one CTA per (node, head) over all keys, which read every K/V row T * G times): 32 query
// / 8 KV heads, D 128, 2048 + 63 keys, 63 nodes 628 -> 69.5 us (31 TFLOP/s; the tensor-core kernel 29.4); the same with one
// node 86 -> 26 us; 8 heads, D 64, 256 + 15 keys, 15 nodes 14.5 -> 6.6 us.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <type_traits>

#include "attention.cuh"
#include "ptd_device.cuh"
#include "row_division.cuh"

namespace cg = cooperative_groups;

namespace ptd {
namespace simt {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;
constexpr int kLanes = 16;                   // lanes that share a row group
constexpr int kGroups = kThreads / kLanes;   // row groups
constexpr int kBN = 64;                      // keys per tile
constexpr int kKeys = kBN / kLanes;          // keys per lane and tile
constexpr int kMaxCluster = 8;
constexpr int kMaxNodes = 128;

constexpr int kBoxRows = 16;                 // rows of a box of a paged cache (a tile starts on a multiple of 16)

// Shared memory (floats) of a block of kGroups * RM rows (D = 128, 64 rows: two CTAs per SM).
template <int D, int RM>
struct Layout {
  static constexpr int BM = kGroups * RM;
  static constexpr int kK = 0;                // K [D / 32][kBN][32], 128-byte swizzle
  static constexpr int kV = kK + kBN * D;     // V [kBN][D]
  static constexpr int kP = kV + kBN * D;     // P^T [kBN][BM], 16-byte chunk c of row n at c ^ p_swizzle(n)
  static constexpr int kQ = kP + kBN * BM;    // Q [BM][D]
  static constexpr int kBar = kQ + BM * D;    // Q, K and V barriers, abort flag
  static constexpr int kEnd = kBar + 8;
  static constexpr int kPar = kP;             // set-up: the tree's parents (before P is written)
  static constexpr int kO = kV;               // end: the partial rows [BM][D] (over V: BM <= kBN)
  static constexpr int kMl = kP;              // end: [BM][2] running maximum and row sum (over P)
  static constexpr size_t kBytes = (size_t)kEnd * sizeof(float);
  static_assert(BM <= kBN && kBN * BM >= kMaxNodes && 2 * (kBytes + 1024) <= 233472, "shared memory");
  // eight consecutive keys' stores of the same rows hit distinct banks
  static __device__ __forceinline__ int p_swizzle(int n) { return BM >= 32 ? n & 7 : (n >> 1) & 3; }
};

// Maximum / sum over the 16 lanes that share a row group.
__device__ __forceinline__ float group_max(float v) {
#pragma unroll
  for (int o = kLanes / 2; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int o = kLanes / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// N consecutive floats (1, or 2 or a multiple of 4 with the alignment of a 16-byte load).
template <int N>
__device__ __forceinline__ void load_n(const float* p, float (&x)[N]) {
  if constexpr (N == 1) {
    x[0] = *p;
  } else if constexpr (N == 2) {
    const float2 a = *reinterpret_cast<const float2*>(p);
    x[0] = a.x, x[1] = a.y;
  } else {
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      const float4 a = *reinterpret_cast<const float4*>(p + i);
      x[i] = a.x, x[i + 1] = a.y, x[i + 2] = a.z, x[i + 3] = a.w;
    }
  }
}
template <int N>
__device__ __forceinline__ void store_n(float* p, const float (&x)[N]) {
  if constexpr (N == 1) {
    *p = x[0];
  } else if constexpr (N == 2) {
    *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
  } else {
#pragma unroll
    for (int i = 0; i < N; i += 4) *reinterpret_cast<float4*>(p + i) = make_float4(x[i], x[i + 1], x[i + 2], x[i + 3]);
  }
}
// A lane's DC = D / 16 columns: two runs of four (D = 128), or one run.
template <int D>
__device__ __forceinline__ void load_cols(const float* row, int g, float (&x)[D / kLanes]) {
  if constexpr (D == 128) {
    const float4 a = *reinterpret_cast<const float4*>(row + 4 * g);
    const float4 c = *reinterpret_cast<const float4*>(row + 64 + 4 * g);
    x[0] = a.x, x[1] = a.y, x[2] = a.z, x[3] = a.w, x[4] = c.x, x[5] = c.y, x[6] = c.z, x[7] = c.w;
  } else {
    load_n<D / kLanes>(row + D / kLanes * g, x);
  }
}

// One tile of K or V, rows [k0, min(k0 + kBN, k_hi)), by one thread; bar receives the bytes.  A
// contiguous cache's tile is whole rows of the tensor whatever the share's end (rows past it are
// some other slot's, or zeros past the tensor); a paged one's comes in boxes of 16 rows, those at
// or past k_hi left out.
template <int D, bool kIsK>
__device__ __forceinline__ void load_tile(const AttnParams& p, const CUtensorMap* map, float* dst_f, uint32_t bar, int b,
                                          int layer, int hkv, int k0, int k_hi) {
  constexpr int kCols = kIsK ? 32 : D;   // columns of a box
  const uint32_t dst = smem_u32(dst_f);
  if (p.page_size == 0) {
    const int row0 = (layer * p.batch + b) * p.seq_capacity + k0;
    mbar_arrive_expect_tx(bar, kBN * D * 4);
#pragma unroll
    for (int c = 0; c < D / kCols; ++c) tma_load_3d(dst + (uint32_t)(c * kBN * kCols) * 4u, map, bar, c * kCols, hkv, row0);
  } else {
    const int shift = __ffs(p.page_size) - 1;   // pages are powers of two
    const int* table = p.block_table + (size_t)b * p.max_pages;
    const int n = min(kBN, (k_hi - k0 + kBoxRows - 1) & ~(kBoxRows - 1));
    mbar_arrive_expect_tx(bar, (uint32_t)(n * D * 4));
#pragma unroll 1
    for (int r = 0; r < n; r += kBoxRows) {
      const int row0 = ((layer * p.num_pages + table[(k0 + r) >> shift]) << shift) + ((k0 + r) & (p.page_size - 1));
#pragma unroll
      for (int c = 0; c < D / kCols; ++c)
        tma_load_3d(dst + (uint32_t)((c * kBN + r) * kCols) * 4u, map, bar, c * kCols, hkv, row0);
    }
  }
}

// Rare path, one warp: a row over the visible keys of [k_lo, k_hi) alone, in order (the tiles multiply the
// P = 0 of hidden nodes into their V, which must not be infinite or NaN).  O (unnormalised) to dst;
// returns the running maximum (log2 units) and the row sum.
template <int D>
__device__ __noinline__ float2 visible_row(const AttnParams& p, const float* q, int layer, int b, int hkv, int k_lo, int k_hi,
                                           int C, const int* parents, int node, float* dst) {
  constexpr int WC = D / 32;
  const int lane = threadIdx.x & 31;
  uint32_t am[4] = {0, 0, 0, 0};
  for (int a = node; a >= 0; a = parents[a])
#pragma unroll
    for (int w = 0; w < 4; ++w) am[w] |= (a >> 5) == w ? 1u << (a & 31) : 0u;
  float qv[WC], o[WC], m = -INFINITY, l = 0.f;
  load_n<WC>(q + WC * lane, qv);
#pragma unroll
  for (int c = 0; c < WC; ++c) o[c] = 0.f;
#pragma unroll 1
  for (int key = k_lo; key < k_hi; ++key) {
    const int a = key - C;
    if (a >= 0 && !((a < 32 ? am[0] : a < 64 ? am[1] : a < 96 ? am[2] : am[3]) >> (a & 31) & 1u)) continue;
    long long row;
    bool there = true;
    if (p.page_size > 0) {
      const int page = p.block_table[(size_t)b * p.max_pages + key / p.page_size];
      there = (unsigned)page < (unsigned)p.num_pages;
      row = ((long long)layer * p.num_pages + page) * p.page_size + key % p.page_size;
    } else {
      row = ((long long)layer * p.batch + b) * p.seq_capacity + key;
    }
    const long long at = (row * p.hkv + hkv) * D + WC * lane;
    float kv[WC], vv[WC], x = 0.f;
#pragma unroll
    for (int c = 0; c < WC; ++c) kv[c] = vv[c] = 0.f;
    if (there) {
      load_n<WC>(static_cast<const float*>(p.k) + at, kv);
      load_n<WC>(static_cast<const float*>(p.v) + at, vv);
    }
#pragma unroll
    for (int c = 0; c < WC; ++c) x = fmaf(qv[c], kv[c], x);
    x = warp_sum(x);
    const float m_new = fmaxf(m, x * p.scale_log2);
    const float m_use = m_new == -INFINITY ? 0.f : m_new;
    const float alpha = exp2f(m - m_use), w = exp2f(fmaf(x, p.scale_log2, -m_use));
    m = m_new;
    l = fmaf(l, alpha, w);
#pragma unroll
    for (int c = 0; c < WC; ++c) o[c] = fmaf(o[c], alpha, w * vv[c]);
  }
  store_n<WC>(dst + WC * lane, o);
  return make_float2(m, l);
}

template <int D, int RM>
__global__ void __launch_bounds__(kThreads, 2)
    tree_attn_simt_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                          const __grid_constant__ AttnParams p, int csize, int m_blocks, GroupDivisor by_group) {
  using L = Layout<D, RM>;
  constexpr int BM = L::BM;
  constexpr int DC = D / kLanes;            // output columns per thread
  extern __shared__ __align__(1024) float sm[];
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane & (kLanes - 1);        // key / column lane
  const int rg = tid / kLanes;              // row group
  const int rank = blockIdx.x % csize;
  int u = blockIdx.x / csize;
  const int mb = u % m_blocks;
  u /= m_blocks;
  const int hkv = u % p.hkv;
  u /= p.hkv;
  const int b = u % p.batch;
  const int lq = u / p.batch;
  const int layer = p.layer_begin + lq;
  const int G = p.group;
  auto node_of = [&](int m) { return divide_by_group(m, by_group); };   // row m's node
  const uint32_t bar_q = smem_u32(sm + L::kBar), bar_k = bar_q + 8, bar_v = bar_q + 16;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + L::kBar + 6);

  if (tid == 0) {
    mbar_init(bar_q, 1);
    mbar_init(bar_k, 1);
    mbar_init(bar_v, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tensormap(&map_k);
    prefetch_tensormap(&map_v);
  }
  grid_dependency_wait();   // the trees, Q, the cache and the output belong to the stream's previous work
  // the next grid may be placed now (not before the wait: the step's top-k starts on its logits
  // beside this kernel)
  if (tid == 0) grid_launch_dependents();
  // ---- the tree (every CTA of the cluster decides alike, so all of them leave here or none)
  const int node0 = p.node_offsets[b];
  const int T = p.node_offsets[b + 1] - node0;
  const int C = p.ctx_lens[b];
  const int N = C + T;
  bool bad_shape = T < 1 || T > p.max_nodes || T > kMaxNodes || node0 < 0 || node0 + T > p.n_total || C < 0;
  if (!bad_shape) bad_shape = p.page_size > 0 ? N > p.max_pages * p.page_size : N > p.seq_capacity;
  // nodes that no tree owns
  if (tid == 0 && ((b == 0 && node0 != 0) || (b == p.batch - 1 && node0 + T != p.n_total)))
    atomicMax(p.dev_status, (int)PTD_ERR_INVALID_TREE);
  if (bad_shape) {
    if (tid == 0) atomicMax(p.dev_status, (int)PTD_ERR_INVALID_TREE);
    return;
  }
  const int M = T * G;
  const int row0 = mb * BM;
  if (row0 >= M) return;
  const int rows = min(BM, M - row0);
  const size_t out_row0 = ((size_t)lq * p.n_total + node0) * p.hq + (size_t)hkv * G;   // + node * hq + head
  auto q_row = [&](int r) {   // row r of the block in q and out
    const int m = row0 + r, node = node_of(m);
    return out_row0 + (size_t)node * p.hq + (m - node * G);
  };

  // this CTA's keys: the rank-th of csize shares, in steps of 16
  const int per = ((N + csize - 1) / csize + 15) & ~15;
  const int k_lo = min(N, rank * per), k_hi = min(N, k_lo + per);
  const int n_tiles = (k_hi - k_lo + kBN - 1) / kBN;
  // the tree is checked before any copy starts, so that leaving needs no drain
  int* const par_s = reinterpret_cast<int*>(sm + L::kPar);
  bool bad = false;
  if (tid < T) {
    const int pp = p.parents[node0 + tid];
    par_s[tid] = pp;
    bad = tid == 0 ? (pp != -1) : (pp < 0 || pp >= tid);
  }
  if (__syncthreads_or(bad)) {
    if (tid == 0) atomicMax(p.dev_status, (int)PTD_ERR_INVALID_TREE);
    if (rank == 0)
      for (int e = tid; e < rows * (D / 4); e += kThreads) {
        const int r = e / (D / 4);
        reinterpret_cast<float4*>(static_cast<float*>(p.out) + q_row(r) * D)[e % (D / 4)] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    return;
  }
  if (n_tiles > 0) {
    if (tid == 0) load_tile<D, true>(p, &map_k, sm + L::kK, bar_k, b, layer, hkv, k_lo, k_hi);
    if (tid == 32) load_tile<D, false>(p, &map_v, sm + L::kV, bar_v, b, layer, hkv, k_lo, k_hi);
    if (warp == 2) {   // Q rows of the block (padding rows keep what is there: their results are not written)
      if (lane == 0) mbar_arrive_expect_tx(bar_q, (uint32_t)(rows * D * 4));
      __syncwarp();
      for (int r = lane; r < rows; r += 32)
        bulk_load(smem_u32(sm + L::kQ + r * D), static_cast<const float*>(p.q) + q_row(r) * D, D * 4, bar_q);
    }
  }
  // ancestor masks (walk up the strictly decreasing parents), for tiles past the context: lane i
  // of a half warp holds its row group's row i
  uint32_t am[4] = {0, 0, 0, 0};
  if (k_hi > C && g < RM && rg * RM + g < rows)
    for (int a = node_of(row0 + rg * RM + g); a >= 0; a = par_s[a]) {
      const uint32_t bit = 1u << (a & 31);
#pragma unroll
      for (int w = 0; w < 4; ++w) am[w] |= (a >> 5) == w ? bit : 0u;
    }

  float m_run[RM], l_run[RM];           // running maximum (log2 units), this thread's share of the row sum
  unsigned long long o[DC][RM / 2];     // O, pairs of rows
#pragma unroll
  for (int i = 0; i < RM; ++i) m_run[i] = -INFINITY, l_run[i] = 0.f;
#pragma unroll
  for (int c = 0; c < DC; ++c)
#pragma unroll
    for (int i = 0; i < RM / 2; ++i) o[c][i] = 0ull;
  const float sl2 = p.scale_log2;
  // A wait that gave up (the status says so) leaves the walk going without further waits, so
  // that every thread meets every barrier.
  bool ok = true;

  if (n_tiles > 0) ok = mbar_wait(bar_q, 0, abort_flag, p.dev_status);
  for (int t = 0; t < n_tiles; ++t) {
    const int k0 = k_lo + t * kBN;
    const int nk = min(kBN, k_hi - k0);
    __syncthreads();   // the previous tile's V is read, the parents are read
    if (t > 0 && tid == 32 && ok) load_tile<D, false>(p, &map_v, sm + L::kV, bar_v, b, layer, hkv, k0, k_hi);
    if (ok) ok = mbar_wait(bar_k, (uint32_t)(t & 1), abort_flag, p.dev_status);
    // ---- S = Q K^T, pairs over columns
    float pr[kKeys][RM];
    {
      unsigned long long s[kKeys][RM];
#pragma unroll
      for (int j = 0; j < kKeys; ++j)
#pragma unroll
        for (int i = 0; i < RM; ++i) s[j][i] = 0ull;
      const float* kp = sm + L::kK + g * 32;
      const int x = (smem_u32(kp) >> 7) & 7;   // the swizzle of keys g + 16 j: chunk c lies at c ^ x
      const float* qp = sm + L::kQ + rg * RM * D;
      auto dot = [&](auto keys) {
        constexpr int NK = decltype(keys)::value;
#pragma unroll 4
        for (int d = 0; d < D; d += 4) {
          ulonglong2 kf[NK];
#pragma unroll
          for (int j = 0; j < NK; ++j) kf[j] = *reinterpret_cast<const ulonglong2*>(kp + (d >> 5) * (kBN * 32) + j * kLanes * 32 + (((d >> 2) & 7) ^ x) * 4);
#pragma unroll
          for (int i = 0; i < RM; ++i) {
            const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(qp + i * D + d);
#pragma unroll
            for (int j = 0; j < NK; ++j) s[j][i] = f2_fma(q.y, kf[j].y, f2_fma(q.x, kf[j].x, s[j][i]));
          }
        }
      };
      if (nk > kBN / 2)
        dot(std::integral_constant<int, kKeys>{});
      else   // a share's last tile may hold few keys
        dot(std::integral_constant<int, kKeys / 2>{});
#pragma unroll
      for (int j = 0; j < kKeys; ++j)
#pragma unroll
        for (int i = 0; i < RM; ++i) {
          float a, c;
          f2_unpack(s[j][i], a, c);
          pr[j][i] = a + c;
        }
    }
    // ---- mask, row maxima, P
    if (k0 + nk > C || nk < kBN) {
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        uint32_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = __shfl_sync(0xffffffffu, am[q], (lane & kLanes) + i);
#pragma unroll
        for (int j = 0; j < kKeys; ++j) {
          const int key = g + kLanes * j, a = k0 + key - C;
          const uint32_t word = a < 32 ? w[0] : a < 64 ? w[1] : a < 96 ? w[2] : w[3];
          if (key >= nk || (a >= 0 && !((word >> (a & 31)) & 1u))) pr[j][i] = -INFINITY;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < RM; i += 2) {
      float alpha[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float mx = pr[0][i + h];
#pragma unroll
        for (int j = 1; j < kKeys; ++j) mx = fmaxf(mx, pr[j][i + h]);
        mx = group_max(mx) * sl2;
        const float m_new = fmaxf(m_run[i + h], mx);
        const float m_use = m_new == -INFINITY ? 0.f : m_new;   // -inf only while nothing is visible
        alpha[h] = exp2f(m_run[i + h] - m_use);                 // 0 from the first visible key's tile
        m_run[i + h] = m_new;
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < kKeys; ++j) {
          pr[j][i + h] = exp2f(fmaf(pr[j][i + h], sl2, -m_use));
          sum += pr[j][i + h];
        }
        l_run[i + h] = fmaf(l_run[i + h], alpha[h], sum);
      }
      const unsigned long long a2 = f2_pack(alpha[0], alpha[1]);
#pragma unroll
      for (int c = 0; c < DC; ++c) o[c][i / 2] = f2_mul(o[c][i / 2], a2);
    }
    // P^T (a row group is one half warp: it reads only what it wrote here)
    constexpr int RC = RM < 4 ? RM : 4;   // rows per store
#pragma unroll
    for (int j = 0; j < kKeys; ++j) {
      const int key = g + kLanes * j;
#pragma unroll
      for (int i = 0; i < RM; i += RC) {
        const int r = rg * RM + i;
        float x[RC];
#pragma unroll
        for (int e = 0; e < RC; ++e) x[e] = pr[j][i + e];
        store_n<RC>(sm + L::kP + key * BM + ((r >> 2) ^ L::p_swizzle(key)) * 4 + (r & 3), x);
      }
    }
    __syncthreads();   // K is read
    if (t + 1 < n_tiles && tid == 0 && ok)
      load_tile<D, true>(p, &map_k, sm + L::kK, bar_k, b, layer, hkv, k0 + kBN, k_hi);
    if (ok) ok = mbar_wait(bar_v, (uint32_t)(t & 1), abort_flag, p.dev_status);
    if (nk < kBN) {   // the share's last tile: P is 0 past its keys, and 0 must not meet a NaN of V
      for (int r = nk; r < ((nk + 3) & ~3); ++r)
        for (int d = tid; d < D; d += kThreads) sm[L::kV + r * D + d] = 0.f;
      __syncthreads();
    }
    // ---- O += P V, pairs over rows
    const float* vp = sm + L::kV;
#pragma unroll 1
    for (int k4 = 0; k4 < nk; k4 += 4) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k = k4 + e;
        float pk[RM], v[DC];
#pragma unroll
        for (int i = 0; i < RM; i += RC) {
          const int r = rg * RM + i;
          float x[RC];
          load_n<RC>(sm + L::kP + k * BM + ((r >> 2) ^ L::p_swizzle(k)) * 4 + (r & 3), x);
#pragma unroll
          for (int q = 0; q < RC; ++q) pk[i + q] = x[q];
        }
        load_cols<D>(vp + k * D, g, v);
#pragma unroll
        for (int c = 0; c < DC; ++c) {
          const unsigned long long vv = f2_pack(v[c], v[c]);
#pragma unroll
          for (int i = 0; i < RM / 2; ++i) o[c][i] = f2_fma(f2_pack(pk[2 * i], pk[2 * i + 1]), vv, o[c][i]);
        }
      }
    }
  }

  if (!ok) {   // copies in flight land (bounded) before shared memory is reused or given up
    for (int ph = 0; ph < 2; ++ph) {
      mbar_drain(bar_q, (uint32_t)ph, 50000000ull);
      mbar_drain(bar_k, (uint32_t)ph, 50000000ull);
      mbar_drain(bar_v, (uint32_t)ph, 50000000ull);
    }
  }
  // ---- this CTA's partial rows into shared memory (over V and P)
  bool wild = false;   // a row of this thread is not finite
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    bool x = !(fabsf(l_run[i]) < INFINITY);
#pragma unroll
    for (int c = 0; c < DC; ++c) {
      float lo, hi;
      f2_unpack(o[c][i / 2], lo, hi);
      x = x || !(fabsf(i & 1 ? hi : lo) < INFINITY);
    }
    wild = wild || (x && rg * RM + i < rows);
  }
  wild = cta_any_unless_aborted(wild, abort_flag);
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    const float l = group_sum(l_run[i]);
    if (g == 0) *reinterpret_cast<float2*>(sm + L::kMl + (rg * RM + i) * 2) = make_float2(m_run[i], l);
  }
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    float x[DC];
#pragma unroll
    for (int c = 0; c < DC; ++c) {
      float lo, hi;
      f2_unpack(o[c][i / 2], lo, hi);
      x[c] = i & 1 ? hi : lo;
    }
    float* dst = sm + L::kO + (rg * RM + i) * D;
    if constexpr (D == 128) {
      *reinterpret_cast<float4*>(dst + 4 * g) = make_float4(x[0], x[1], x[2], x[3]);
      *reinterpret_cast<float4*>(dst + 64 + 4 * g) = make_float4(x[4], x[5], x[6], x[7]);
    } else {
      store_n<DC>(dst + DC * g, x);
    }
  }
  constexpr int WC = D / 32;   // columns per lane of a whole warp
  if (wild) {
    __syncthreads();
#pragma unroll 1
    for (int r = warp; r < rows; r += kWarps) {
      float* const row = sm + L::kO + r * D;
      float2* const ml = reinterpret_cast<float2*>(sm + L::kMl + 2 * r);
      bool x = !(fabsf(ml->y) < INFINITY);
#pragma unroll
      for (int c = 0; c < WC; ++c) x = x || !(fabsf(row[WC * lane + c]) < INFINITY);
      if (!__any_sync(0xffffffffu, x)) continue;
      const float2 y = visible_row<D>(p, static_cast<const float*>(p.q) + q_row(r) * D, layer, b, hkv, k_lo, k_hi, C,
                                      p.parents + node0, node_of(row0 + r), row);
      __syncwarp();
      if (lane == 0) *ml = y;
    }
  }
  cluster.sync();
  // ---- combine: CTA r writes the r-th share of the rows, one row per warp at a time
  const int r_lo = rank * rows / csize, r_hi = (rank + 1) * rows / csize;
#pragma unroll 1
  for (int r = r_lo + warp; r < r_hi; r += kWarps) {
    float part[kMaxCluster][WC];
#pragma unroll
    for (int c = 0; c < kMaxCluster; ++c)
      if (c < csize) load_n<WC>(cluster.map_shared_rank(sm + L::kO, c) + r * D + WC * lane, part[c]);
    float m = -INFINITY, l = 0.f;
    if (lane < csize) {
      const float2 ml = *reinterpret_cast<const float2*>(cluster.map_shared_rank(sm + L::kMl, lane) + 2 * r);
      m = ml.x, l = ml.y;
    }
    const float mm = warp_max(m);
    const float w = l > 0.f ? exp2f(m - mm) : 0.f;
    const float lw = warp_sum(l * w);
    const float inv = lw > 0.f ? 1.f / lw : 0.f;
    float acc[WC];
#pragma unroll
    for (int e = 0; e < WC; ++e) acc[e] = 0.f;
#pragma unroll
    for (int c = 0; c < kMaxCluster; ++c) {
      const float wc = __shfl_sync(0xffffffffu, w, c);
      if (c < csize) {
#pragma unroll
        for (int e = 0; e < WC; ++e) acc[e] = fmaf(wc, part[c][e], acc[e]);
      }
    }
#pragma unroll
    for (int e = 0; e < WC; ++e) acc[e] *= inv;
    store_n<WC>(static_cast<float*>(p.out) + q_row(r) * D + WC * lane, acc);
  }
  cluster.sync();   // keep this CTA's shared memory alive until the others have read it
}

template <int D, int RM>
cudaError_t launch(const CUtensorMap& map_k, const CUtensorMap& map_v, const AttnParams& p, int csize, int m_blocks, cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((long long)csize * m_blocks * p.hkv * p.batch * p.layers), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = Layout<D, RM>::kBytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // placed while the previous kernel drains
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const cudaError_t e = cudaFuncSetAttribute(tree_attn_simt_kernel<D, RM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)Layout<D, RM>::kBytes);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, tree_attn_simt_kernel<D, RM>, map_k, map_v, p, csize, m_blocks,
                            group_divisor(p.group));
}

// Rows per block: the smallest that holds M, up to 64 (two such CTAs fit an SM's shared memory;
// 128-row blocks, one per SM, left a unit's cluster of 8 CTAs short of SMs in some GPCs).
int block_rows(int M) {
  int bm = 16;
  while (bm < 64 && bm < M) bm *= 2;
  return bm;
}

template <int D>
cudaError_t launch_d(const CUtensorMap& map_k, const CUtensorMap& map_v, const AttnParams& p, int csize, cudaStream_t stream) {
  const int M = p.max_nodes * p.group, bm = block_rows(M), m_blocks = (M + bm - 1) / bm;
  if ((long long)m_blocks * p.hkv * p.batch * p.layers * csize > 0x7fffffffll) return cudaErrorInvalidValue;
  switch (bm) {
    case 16:
      return launch<D, 16 / kGroups>(map_k, map_v, p, csize, m_blocks, stream);
    case 32:
      return launch<D, 32 / kGroups>(map_k, map_v, p, csize, m_blocks, stream);
    default:
      return launch<D, 64 / kGroups>(map_k, map_v, p, csize, m_blocks, stream);
  }
}

}  // namespace simt

F32Plan choose_tree_attn_f32(const AttnParams& p, int max_ctx, int sms) {
  using simt::kMaxCluster;
  const int M = p.max_nodes * p.group, bm = simt::block_rows(M);
  const long long units = (long long)((M + bm - 1) / bm) * p.hkv * p.batch * p.layers;
  // CTAs per unit (a cluster): the split whose waves over the SMs take the fewest keys, a CTA's
  // fixed part (set-up, combination) counted as 48 keys
  const int keys = max_ctx + p.max_nodes;
  const long long slots = 2ll * sms;
  int csize = 1;
  double best = 1e300;
  for (int c = 1; c <= kMaxCluster; ++c) {
    const double waves = (double)((units * c + slots - 1) / slots);
    const double cost = waves * (((keys + c - 1) / c + 15) / 16 * 16 + 48);
    if (cost < best) best = cost, csize = c;
  }
  if (p.head_dim != 128) return {false, csize};
  // The tensor-core kernel where it is estimated to be faster (us, fitted to measurements of 70
  // shapes on 152 SMs: one runs 7 % slower than it would on the other kernel, the rest within 4 %):
  // on the cores a fixed part and a time per key of a CTA's share that depends on the rows of a block and
  // on whether two CTAs share an SM; on the tensor cores a fixed part, the rows' combination and a time per tile of 64
  // keys.  Tensor cores / CUDA cores, 32 query and 8 KV heads: 63 nodes 64 keys 14.1 / 16.5, 300 keys
  // 13.9 / 22.3, 1000 keys 19.9 / 43.7, 4000 keys 46.3 / 117.7; 8 heads without groups: 32 nodes 1000 keys
  // 17.5 / 17.2, 4000 keys 34.0 / 41.0, 8 nodes 4000 keys 33.6 / 33.2.
  const double share = ((keys + csize - 1) / csize + 15) / 16 * 16;
  const double waves = (double)((units * csize + slots - 1) / slots);
  auto fit = [&](int c) { return clusters_at_once(c, sms); };
  const bool shared_sm = units > fit(csize);
  const double fixed = bm == 16 ? 5.5 : bm == 32 ? 7.3 : 11.;
  const double per_key = bm == 16 ? (shared_sm ? 0.085 : 0.054) : bm == 32 ? (shared_sm ? 0.117 : 0.069)
                                                                          : (shared_sm ? 0.205 : 0.112);
  const double t_here = waves * (fixed + per_key * share);
  const int split_blocks = (M + 127) / 128;
  const long long split_units = (long long)split_blocks * p.hkv * p.batch * p.layers;
  int split_csize = 0;
  double t_split = t_here;
  for (int c = 1; c <= kMaxCluster; ++c) {
    const int tiles = (((keys + c - 1) / c + 15) / 16 * 16 + 63) / 64;
    const double t = (double)((split_units + fit(c) - 1) / fit(c)) * (8.5 + 2.5 * (M < 128 ? M : 128) / 128 + 3.25 * tiles);
    if (t < t_split) t_split = t, split_csize = c;
  }
  return split_csize > 0 ? F32Plan{true, split_csize} : F32Plan{false, csize};
}

cudaError_t launch_tree_attn_simt(const CUtensorMap& map_k, const CUtensorMap& map_v, const AttnParams& p, int csize, cudaStream_t stream) {
  if (p.hq > 65535 || p.n_total > 65535 || p.layers > 65535) return cudaErrorInvalidValue;
  switch (p.head_dim) {
    case 32:
      return simt::launch_d<32>(map_k, map_v, p, csize, stream);
    case 64:
      return simt::launch_d<64>(map_k, map_v, p, csize, stream);
    case 128:
      return simt::launch_d<128>(map_k, map_v, p, csize, stream);
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace ptd
