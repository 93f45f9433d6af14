// Tree-masked attention in fp32 on the tensor cores (tcgen05), D = 128: every fp32 operand is split
// into three bf16 parts, x = h + m + l (each the nearest bf16 to what is left; exact from 2^-110 up, below
// that off by at most 2^-134, half of bf16's smallest subnormal), and a product x y is taken as the six
// partial products
//   h l' + l h' + m m' + h m' + m h' + h h'
// (exact in fp32, summed in fp32; what is left out is below 2^-26 of x y).  The small ones are
// summed first and apart from h h'.
//
// Same operation and same work split as the fp32 kernel on the CUDA cores: the T nodes times the G
// query heads of a KV head are M = T * G rows, a unit is one (layer, tree, KV head, block of 128
// rows), and a cluster of `csize` CTAs computes it, CTA r taking the r-th share of the keys; the
// CTAs' partial states (m, l, O) are combined through distributed shared memory.
//
// A CTA (384 threads):
//   warps 0-7   rows: thread (row = TMEM lane, half).  They bring K and V of a tile of 64 keys from
//               global memory and write the three bf16 parts to shared memory, take the softmax
//               (thread: its row, 32 of the 64 keys; the row maximum is exchanged by the two
//               halves), put the three parts of P into TMEM, and keep O (64 columns of the row) in
//               registers: the P V of a tile comes in a TMEM tile of its own and is added in fp32
//               with rounding to nearest.
//   warp 8      issues the GEMMs: S of the next tile while the softmax of this one runs.
//   warps 9-11  idle (they give their registers to the others).
// TMEM: two S sets of 192 columns (h h' over columns 0-63 and 64-127 of Q and K, the other five
// products), P over the first 96 columns of its set, the P V tile.
//
// What bounds it: per tile the GEMMs, 48 instructions of S and 24 of P V in series (~7,400 cycles; the
// conversions and the softmax run beside them), and about 9 us of set-up (Q and the first tiles
// are read, converted and the code is fetched) and combination.  The tile is 64 keys because the three
// parts of 128 rows of Q (96 KB) and of K and V (48 KB each) fill shared memory.  Measured (GB300,
// one layer, against the CUDA-core kernel): 32 query / 8 KV heads, 2048 + 63 keys, 63 nodes 69.2 ->
// 29.4 us (74 TFLOP/s); 4000 keys 115.5 -> 46.4; 128 nodes, 4000 keys 229 -> 64.7.  (Set-up written out
// per piece, with divisions by the group, and the combination one row after the other: 30.8; without the
// checks for tiny results and huge operands 29.1.)
//
// Precision: relative error against 64 bits over 14 shapes drawn for it, at scores of deviation 1/4,
// 1 and 4: 1.0e-7 .. 1.3e-7, 1.5e-7 .. 1.9e-7, 2.5e-7 .. 4.2e-7; the CUDA-core kernel's, whose chains of
// fp32 sums are longer, 1.2e-7 .. 3.2e-7, 2.3e-7 .. 3.9e-7, 4.5e-7 .. 8.0e-7.  The tensor core
// truncates its fp32 sums, so few h h' are chained: four instructions per accumulator of S, four per
// tile of O.
//
// A row is taken again, over its CTA's share of the keys, by plain fp32 loops where the parts do not
// carry it: one that comes out infinite or NaN (an input that is, or whose nearest bf16 is, or an
// overflow); one with a column below 2^-88 (the 2^-134 then count: V of 2^-120 was off by 4e-5); and all
// rows of a CTA that meets an operand of 2^90 or more (which the 2^-134 of its partner, or of a
// probability, may stand against: Q of 2^120 on K of 2^-120 was off by 4e-5).  Such inputs run at a
// fraction of the speed.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "attention.cuh"
#include "attention_tc.cuh"
#include "launch.cuh"
#include "ptd_device.cuh"
#include "row_division.cuh"

namespace cg = cooperative_groups;

namespace ptd {
namespace split {

constexpr int kThreads = 384;
constexpr int kRowWarps = 8;                   // then the warp that issues the GEMMs
constexpr int kBM = 128;                       // rows per block
constexpr int kBN = 64;                        // keys per tile
constexpr int kD = 128;
constexpr int kMaxCluster = 8;
constexpr int kMaxNodes = 128;
constexpr uint32_t kQPart = kBM * kD * 2;      // bytes of one bf16 part of Q
constexpr uint32_t kKvPart = kBN * kD * 2;     //   of a K or V tile
constexpr uint32_t kQHalf = kQPart / 2;        // 64 columns (one 128-byte swizzle column) of all rows
constexpr uint32_t kKvHalf = kKvPart / 2;
constexpr uint32_t kOffK = 3 * kQPart;
constexpr uint32_t kOffV = kOffK + 3 * kKvPart;
constexpr uint32_t kOffX = kOffV + 3 * kKvPart;    // [tile parity][2][kBM] row maxima of the halves
constexpr uint32_t kOffMl = kOffX + 4 * kBM * 4;   // [kBM][2] partial (m, l), read by the cluster
constexpr uint32_t kOffPar = kOffMl + kBM * 8;     // the tree's parents
constexpr uint32_t kOffBar = kOffPar + kMaxNodes * 4;   // k and p ready, o full, drain, s full[2]
constexpr uint32_t kOffTmem = kOffBar + 6 * 8;
constexpr uint32_t kOffAbort = kOffTmem + 4;
constexpr uint32_t kOffHuge = kOffAbort + 4;
constexpr uint32_t kSmemBytes = kOffHuge + 4 + 1024;   // slack to align the base to 1024 B
static_assert(kSmemBytes <= 232448, "shared memory budget");
// O of the block, fp32 [kBM][kD], over Q at the end: 16-byte chunk c of row r at c ^ (r & 7)
static_assert(kBM * kD * 4 <= 3 * kQPart, "O lies over Q");

constexpr float kHuge = 0x1p90f, kTiny = 0x1p-88f;   // operands from which, columns of O up to which plain loops run

constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kSetCols = 192;             // S set: h h' (columns 0-63) | h h' (64-127) | the rest
constexpr uint32_t kColO = 2 * kSetCols;       // P V of a tile
constexpr uint32_t kIdescS = idesc_bf16_f32(128, 64, 0, 0);
constexpr uint32_t kIdescPV = idesc_bf16_f32(128, 128, 0, 1);

// Two fp32 values as three packed bf16 pairs.
__device__ __forceinline__ void split2(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = pack_bf16x2(a, b);
  a = __fsub_rn(a, __uint_as_float(h << 16));
  b = __fsub_rn(b, __uint_as_float(h & 0xFFFF0000u));
  m = pack_bf16x2(a, b);
  a = __fsub_rn(a, __uint_as_float(m << 16));
  b = __fsub_rn(b, __uint_as_float(m & 0xFFFF0000u));
  l = pack_bf16x2(a, b);
}
// Columns [4 lane, 4 lane + 4) of row r, split, into three parts of `part` bytes (128-byte swizzle,
// 64 columns of all rows before the other 64).
__device__ __forceinline__ void store_split(uint32_t dst, uint32_t part, int r, int lane, float4 x) {
  uint32_t h0, h1, m0, m1, l0, l1;
  split2(x.x, x.y, h0, m0, l0);
  split2(x.z, x.w, h1, m1, l1);
  const uint32_t at = dst + (uint32_t)(lane >> 4) * (part / 2) + (uint32_t)r * 128u +
                      ((((uint32_t)(lane & 15) >> 1) ^ (uint32_t)(r & 7)) << 4) + (uint32_t)(lane & 1) * 8u;
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at), "r"(h0), "r"(h1) : "memory");
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at + part), "r"(m0), "r"(m1) : "memory");
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at + 2 * part), "r"(l0), "r"(l1) : "memory");
}

// Four floats, or zeros where `there` is false, as one predicated load: nothing waits for it before its use.
__device__ __forceinline__ float4 load_or_zero(const float* src, bool there) {
  float4 x;
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\t"
      "mov.b32 %3, 0;\n\t@p ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
      : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w)
      : "l"(src), "r"((int)there));
  return x;
}

// Key `key` of tree b's sequence as an offset in K and V; negative when its page number lies
// outside the cache.
__device__ __forceinline__ long long kv_row(const AttnParams& p, int layer, int b, int hkv, int key, const int* table,
                                            int shift) {
  long long r;
  if (p.page_size > 0) {
    const int page = table[key >> shift];
    if ((unsigned)page >= (unsigned)p.num_pages) return -kD;
    r = ((long long)layer * p.num_pages + page) * p.page_size + (key & (p.page_size - 1));
  } else {
    r = ((long long)layer * p.batch + b) * p.seq_capacity + key;
  }
  return (r * p.hkv + hkv) * kD;
}

// Rare path: a row's share of the keys in plain fp32, O (unnormalised, 64 columns) to dst (16-byte
// chunk c at c ^ sw); returns the maximum (log2 units) and the row sum.
__device__ __noinline__ float2 plain_row(const AttnParams& p, const float* q, int layer, int b, int hkv, int k_lo, int k_hi,
                                         int C, uint4 am, int half, float* dst, int sw) {
  const float* const kg = static_cast<const float*>(p.k);
  const float* const vg = static_cast<const float*>(p.v) + 64 * half;
  const int* const table = p.block_table + (size_t)b * p.max_pages;
  const int shift = p.page_size > 0 ? __ffs(p.page_size) - 1 : 0;
  float m = -INFINITY, l = 0.f;
#pragma unroll 1
  for (int c = 0; c < 16; ++c) *reinterpret_cast<float4*>(dst + (((half * 16 + c) ^ sw) << 2)) = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int key = k_lo; key < k_hi; ++key) {
    const int a = key - C;
    if (a >= 0 && !((a < 32 ? am.x : a < 64 ? am.y : a < 96 ? am.z : am.w) >> (a & 31) & 1u)) continue;
    const long long at = kv_row(p, layer, b, hkv, key, table, shift);
    float s0 = 0.f, s1 = 0.f;
#pragma unroll 8
    for (int d = 0; d < kD; d += 4) {
      const float4 y = *reinterpret_cast<const float4*>(q + d), z = load_or_zero(kg + at + d, at >= 0);
      s0 = fmaf(y.x, z.x, s0);
      s1 = fmaf(y.y, z.y, s1);
      s0 = fmaf(y.z, z.z, s0);
      s1 = fmaf(y.w, z.w, s1);
    }
    const float x = s0 + s1;
    const float m_new = fmaxf(m, x * p.scale_log2);
    const float m_use = m_new == -INFINITY ? 0.f : m_new;
    const float alpha = exp2f(m - m_use), w = exp2f(fmaf(x, p.scale_log2, -m_use));
    m = m_new;
    l = fmaf(l, alpha, w);
#pragma unroll 8
    for (int c = 0; c < 16; ++c) {
      float4* const o = reinterpret_cast<float4*>(dst + (((half * 16 + c) ^ sw) << 2));
      const float4 v = load_or_zero(vg + at + 4 * c, at >= 0);
      float4 y = *o;
      y.x = fmaf(y.x, alpha, w * v.x);
      y.y = fmaf(y.y, alpha, w * v.y);
      y.z = fmaf(y.z, alpha, w * v.z);
      y.w = fmaf(y.w, alpha, w * v.w);
      *o = y;
    }
  }
  return make_float2(m, l);
}

__global__ void __launch_bounds__(kThreads, 1)
    tree_attn_split_kernel(const __grid_constant__ AttnParams p, int csize, int m_blocks, GroupDivisor by_group) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint32_t base = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (base & 1023u)) & 1023u;   // the same in every CTA of the launch
  uint8_t* const smem = smem_raw + pad;
  base += pad;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // known to be uniform, for the GEMM issue
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
  const uint32_t k_ready = base + kOffBar, p_ready = k_ready + 8, o_full = k_ready + 16, drain = k_ready + 24;
  // one per S set: a set is written again only after the row warps have passed its last S
  auto s_full = [&](int t) { return k_ready + 32 + 8u * (uint32_t)(t & 1); };
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(smem + kOffAbort);
  volatile int* const huge_s = reinterpret_cast<volatile int*>(smem + kOffHuge);   // an operand reached kHuge
  float* const x_s = reinterpret_cast<float*>(smem + kOffX);
  float* const ml_s = reinterpret_cast<float*>(smem + kOffMl);
  int* const par_s = reinterpret_cast<int*>(smem + kOffPar);

  if (tid == 0) {
    mbar_init(k_ready, kRowWarps);   // one arrival per warp
    mbar_init(p_ready, kRowWarps);
    mbar_init(s_full(0), 1);
    mbar_init(s_full(1), 1);
    mbar_init(o_full, 1);
    mbar_init(drain, 1);
    *abort_flag = 0;
    *huge_s = 0;
    fence_mbar_init();
  }
  grid_dependency_wait();   // the trees, Q, the cache and the output belong to the stream's previous work
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
  const int row0 = mb * kBM;
  if (row0 >= M) return;
  const int rows = min(kBM, M - row0);
  const size_t out_row0 = ((size_t)lq * p.n_total + node0) * p.hq + (size_t)hkv * G;   // + node * hq + head
  auto node_of = [&](int m) { return divide_by_group(m, by_group); };   // row m's node
  auto q_row = [&](int r) {   // row r of the block in q and out
    const int m = row0 + r, node = node_of(m);
    return out_row0 + (size_t)node * p.hq + (m - node * G);
  };
  // this CTA's keys: the rank-th of csize shares, in steps of 16
  const int per = ((N + csize - 1) / csize + 15) & ~15;
  const int k_lo = min(N, rank * per), k_hi = min(N, k_lo + per);
  const int n_tiles = __shfl_sync(0xffffffffu, (k_hi - k_lo + kBN - 1) / kBN, 0);
  const float* const kg = static_cast<const float*>(p.k);
  const float* const vg = static_cast<const float*>(p.v);
  const int shift = p.page_size > 0 ? __ffs(p.page_size) - 1 : 0;   // pages are powers of two
  const int* const table = p.block_table + (size_t)b * p.max_pages;
  // this lane's four columns of rows warp, warp + 8, .. of tile t (rows past the share: zeros)
  constexpr int kRowsPerWarp = kBN / kRowWarps;
  auto load = [&](float4(&x)[kRowsPerWarp], const float* src, int t) {
    const int key0 = k_lo + t * kBN + warp;
    if (p.page_size > 0) {
      long long at[kRowsPerWarp];
#pragma unroll
      for (int i = 0; i < kRowsPerWarp; ++i)
        at[i] = key0 + kRowWarps * i < k_hi ? kv_row(p, layer, b, hkv, key0 + kRowWarps * i, table, shift) : -1;
#pragma unroll
      for (int i = 0; i < kRowsPerWarp; ++i) x[i] = load_or_zero(src + at[i] + 4 * lane, at[i] >= 0);
    } else {
      const float* at = src + kv_row(p, layer, b, hkv, key0, table, shift) + 4 * lane;
      const size_t step = (size_t)kRowWarps * p.hkv * kD;
#pragma unroll
      for (int i = 0; i < kRowsPerWarp; ++i, at += step) x[i] = load_or_zero(at, key0 + kRowWarps * i < k_hi);
    }
  };
  // and of the block's Q, rows warp + 64 h, warp + 64 h + 8, ..
  auto load_q = [&](float4(&x)[kRowsPerWarp], int h) {
#pragma unroll
    for (int i = 0; i < kRowsPerWarp; ++i) {
      const int r = warp + kRowWarps * i + kBN * h;
      x[i] = load_or_zero(static_cast<const float*>(p.q) + (r < rows ? q_row(r) : 0) * kD + 4 * lane, r < rows);
    }
  };
  bool bad = false;
  if (tid < T) {
    const int pp = p.parents[node0 + tid];
    par_s[tid] = pp;
    bad = tid == 0 ? (pp != -1) : (pp < 0 || pp >= tid);
  }
  if (__syncthreads_or(bad)) {
    if (tid == 0) atomicMax(p.dev_status, (int)PTD_ERR_INVALID_TREE);
    if (rank == 0)
      for (int e = tid; e < rows * (kD / 4); e += kThreads)
        reinterpret_cast<float4*>(static_cast<float*>(p.out) + q_row(e / (kD / 4)) * kD)[e % (kD / 4)] =
            make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  if (warp == kRowWarps) {
    tmem_alloc(base + kOffTmem, kTmemCols);
    tmem_relinquish();
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + kOffTmem);

  const int row = (warp & 3) * 32 + lane, half = (warp >> 2) & 1;   // row warps
  bool ok = true;

  // A wait that gave up (the status says so) leaves the walks going without further waits, so
  // that every thread meets every barrier.
  if (warp >= kRowWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    if (warp == kRowWarps) {
      // ================================================================ GEMM issue
      // The warp walks together and one lane issues by predication (see tc::issue_s): a GEMM
      // instruction takes 80-100 cycles instead of 95-110 (54 in a kernel that does nothing else).
      const uint32_t leader = lane == 0 ? 1u : 0u;
      // descriptors of the first part's first 16 columns (Q, K) or keys (V); the address field counts
      // 16-byte units, so the others are sums
      const uint32_t dq = (uint32_t)smem_desc_sw128(base, 16, 1024), dk = (uint32_t)smem_desc_sw128(base + kOffK, 16, 1024),
                     dv = (uint32_t)smem_desc_sw128(base + kOffV, kKvHalf, 1024);
      // the products, the smallest first: parts of the two operands, four bits each (a loop over
      // them: unrolled, the descriptors would be kept over the tiles and spill)
      constexpr uint32_t kPartA = 0x010120u, kPartB = 0x001102u;
      auto gemm_s = [&](int t) {
        if (!__shfl_sync(0xffffffffu, (int)mbar_wait_warp(k_ready, (uint32_t)(t & 1), abort_flag, p.dev_status), 0)) return false;
        tc_fence_after();
        const uint32_t set = __shfl_sync(0xffffffffu, tmem, 0) + (uint32_t)(t & 1) * kSetCols;
        const uint32_t dqt = __shfl_sync(0xffffffffu, dq, 0), dkt = __shfl_sync(0xffffffffu, dk, 0);
#pragma unroll 2
        for (int i = 0; i < 6; ++i) {
          const uint32_t a = dqt + ((kPartA >> (4 * i)) & 3u) * (kQPart / 16);
          const uint32_t c = dkt + ((kPartB >> (4 * i)) & 3u) * (kKvPart / 16);
          const bool hh = i == 5;
          const uint32_t d0 = hh ? set : set + 128u, d1 = hh ? set + 64u : set + 128u;
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            mma_ss_if(leader, kk < 4 ? d0 : d1, a + (uint32_t)((kk >> 2) * (int)(kQHalf / 16) + (kk & 3) * 2),
                      c + (uint32_t)((kk >> 2) * (int)(kKvHalf / 16) + (kk & 3) * 2), tc::kDescHi, kIdescS,
                      kk == 0 ? (i > 0 && !hh ? 1u : 0u) : kk == 4 ? (hh ? 0u : 1u) : 1u);
        }
        if (leader) mma_commit(s_full(t));
        return true;
      };
      auto gemm_pv = [&](int t) {
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0), pt = tm + (uint32_t)(t & 1) * kSetCols;
        const uint32_t dvt = __shfl_sync(0xffffffffu, dv, 0);
#pragma unroll 2
        for (int i = 0; i < 6; ++i) {
          const uint32_t a = pt + ((kPartA >> (4 * i)) & 3u) * 32u;
          const uint32_t c = dvt + ((kPartB >> (4 * i)) & 3u) * (kKvPart / 16);
#pragma unroll
          for (int kk = 0; kk < kBN / 16; ++kk)
            mma_ts_if(leader, tm + kColO, a + (uint32_t)kk * 8u, c + (uint32_t)(kk * 128), tc::kDescHi, kIdescPV,
                      i > 0 || kk > 0 ? 1u : 0u);
        }
        if (leader) mma_commit(o_full);
      };
      if (n_tiles > 0) ok = gemm_s(0);
      for (int t = 0; t < n_tiles && ok; ++t) {
        // S of tile t + 1 goes over P of tile t - 1: its P V has ended
        if (t > 0 && !(ok = mbar_wait_warp(o_full, (uint32_t)((t - 1) & 1), abort_flag, p.dev_status))) break;
        if (t + 1 < n_tiles && !(ok = gemm_s(t + 1))) break;
        if (!(ok = mbar_wait_warp(p_ready, (uint32_t)(t & 1), abort_flag, p.dev_status))) break;
        tc_fence_after();
        gemm_pv(t);
      }
      // what was issued ends (bounded) before shared memory and TMEM are reused or given up
      if (leader) {
        mma_commit(drain);
        mbar_drain(drain, 0, 100000000ull);
      }
    }
    __syncwarp();
    __syncthreads();   // every GEMM has ended, the row warps have read TMEM
    if (warp == kRowWarps) {
      tc_fence_after();
      tmem_dealloc(tmem, kTmemCols);
    }
    cluster.sync();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
    // ================================================================ rows
    float m_run = -INFINITY, l_run = 0.f;   // running maximum (log2 units), this thread's share of the row sum
    float o[64];                            // columns [64 half, 64 half + 64) of the row
    uint32_t am[4] = {0, 0, 0, 0};
    auto note = [&](const float4(&y)[kRowsPerWarp]) {
      float m[4] = {0.f, 0.f, 0.f, 0.f};   // (four chains: one of sixteen maxima takes 29.55 us instead of 29.41, 63 nodes over 2048 keys)
#pragma unroll
      for (int i = 0; i < kRowsPerWarp; i += 2) {
        m[0] = fmax3(fabsf(y[i].x), fabsf(y[i].y), m[0]);
        m[1] = fmax3(fabsf(y[i].z), fabsf(y[i].w), m[1]);
        m[2] = fmax3(fabsf(y[i + 1].x), fabsf(y[i + 1].y), m[2]);
        m[3] = fmax3(fabsf(y[i + 1].z), fabsf(y[i + 1].w), m[3]);
      }
      if (fmaxf(fmax3(m[0], m[1], m[2]), m[3]) >= kHuge) *huge_s = 1;
    };
    auto store = [&](uint32_t off, const float4(&y)[kRowsPerWarp]) {
#pragma unroll
      for (int i = 0; i < kRowsPerWarp; ++i) store_split(base + off, kKvPart, warp + kRowWarps * i, lane, y[i]);
      fence_proxy_async_smem();
    };
    // Q in two halves, then the first tile's K, each stored while the next (V last) is on its way: one
    // loop with one copy of each piece of code, as it is fetched cold
    float4 kx[kRowsPerWarp], vx[kRowsPerWarp];
    if (n_tiles > 0) {
#pragma unroll 1
      for (int j = 0; j < 4; ++j) {
        if (j < 2)
          load_q(vx, j);
        else
          load(vx, j == 2 ? kg : vg, 0);
        if (j > 0) {
          const uint32_t part = j < 3 ? kQPart : kKvPart, off = j < 3 ? 0u : kOffK;
#pragma unroll
          for (int i = 0; i < kRowsPerWarp; ++i)
            store_split(base + off, part, warp + kRowWarps * i + (j == 2 ? kBN : 0), lane, kx[i]);
          note(kx);
        }
        if (j < 3) {
#pragma unroll
          for (int i = 0; i < kRowsPerWarp; ++i) kx[i] = vx[i];
        }
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(k_ready);
      if (n_tiles > 1) load(kx, kg, 1);
    }
    // the row's ancestor mask (walk up the strictly decreasing parents), for keys past the context
    if (k_hi > C && row < rows)
      for (int a = node_of(row0 + row); a >= 0; a = par_s[a]) {
        const uint32_t bit = 1u << (a & 31);
#pragma unroll
        for (int w = 0; w < 4; ++w) am[w] |= (a >> 5) == w ? bit : 0u;
      }
#pragma unroll
    for (int c = 0; c < 64; ++c) o[c] = 0.f;
    const uint32_t lane_t = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const float sl2 = p.scale_log2;
    float alpha_o = 0.f;   // what O is to be multiplied by before the tile in TMEM is added
    // O = alpha O + the P V tile in TMEM
    auto add_tile = [&](int t) {
      if (ok) ok = mbar_wait_warp(o_full, (uint32_t)(t & 1), abort_flag, p.dev_status);
      tc_fence_after();
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint32_t r[16];
        tmem_ld16(lane_t + kColO + (uint32_t)half * 64u + (uint32_t)q * 16u, r);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) o[16 * q + e] = fmaf(o[16 * q + e], alpha_o, __uint_as_float(r[e]));
      }
    };
#pragma unroll 1
    for (int t = 0; t < n_tiles; ++t) {
      const int k0 = k_lo + t * kBN + half * 32;   // this thread's keys
      if (ok) ok = mbar_wait_warp(s_full(t), (uint32_t)((t >> 1) & 1), abort_flag, p.dev_status);
      tc_fence_after();
      if (t + 1 < n_tiles) {   // K of tile t is read: the next one's place
        store(kOffK, kx);
        __syncwarp();
        if (lane == 0) mbar_arrive(k_ready);
        note(kx);
        if (t + 2 < n_tiles) load(kx, kg, t + 2);
      }
      // ---- S, mask, row maximum, P
      float s[32];
      const uint32_t set = lane_t + (uint32_t)(t & 1) * kSetCols;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint32_t a[16], c[16];
        tmem_ld16(set + (uint32_t)(half * 32 + q * 16), a);
        tmem_ld16(set + 64u + (uint32_t)(half * 32 + q * 16), c);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) s[16 * q + e] = __uint_as_float(a[e]) + __uint_as_float(c[e]);
        tmem_ld16(set + 128u + (uint32_t)(half * 32 + q * 16), c);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) s[16 * q + e] += __uint_as_float(c[e]);
      }
      if (k0 + 32 > C || k0 + 32 > k_hi) {
        uint32_t vis = tc::vis_word(k0 - C, am[0], am[1], am[2], am[3]);
        if (k0 + 32 > k_hi) vis &= k_hi > k0 ? (1u << (k_hi - k0)) - 1u : 0u;
#pragma unroll
        for (int e = 0; e < 32; ++e) s[e] = ((vis >> e) & 1u) ? s[e] : -INFINITY;
      }
      float mx = s[0];
#pragma unroll
      for (int e = 1; e < 32; ++e) mx = fmaxf(mx, s[e]);
      float* const xt = x_s + (t & 1) * 2 * kBM;
      xt[half * kBM + row] = mx;
      tc_fence_before();
      // both halves of these rows have read S, over which P goes
      asm volatile("bar.sync %0, 64;" ::"r"(1 + (warp & 3)) : "memory");
      tc_fence_after();
      mx = fmaxf(mx, xt[(half ^ 1) * kBM + row]) * sl2;
      const float m_new = fmaxf(m_run, mx);
      const float m_use = m_new == -INFINITY ? 0.f : m_new;   // -inf only while nothing is visible
      const float alpha = exp2f(m_run - m_use);               // 0 from the first visible key's tile
      m_run = m_new;
      float sum = 0.f;
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        s[e] = ptx_exp2(fmaf(s[e], sl2, -m_use));
        sum += s[e];
      }
      l_run = fmaf(l_run, alpha, sum);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        uint32_t h[8], m[8], l[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) split2(s[16 * q + 2 * e], s[16 * q + 2 * e + 1], h[e], m[e], l[e]);
        tmem_st8(set + (uint32_t)(half * 16 + q * 8), h);
        tmem_st8(set + 32u + (uint32_t)(half * 16 + q * 8), m);
        tmem_st8(set + 64u + (uint32_t)(half * 16 + q * 8), l);
      }
      if (t > 0) add_tile(t - 1);
      alpha_o = alpha;
      store(kOffV, vx);   // V of tile t - 1 is read
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_ready);
      note(vx);
      if (t + 1 < n_tiles) load(vx, vg, t + 1);
    }
    if (n_tiles > 0) add_tile(n_tiles - 1);
    // ---- a row that the parts do not carry (see above): the share again, in plain fp32
    bool redo = !(fabsf(l_run) < INFINITY);
    uint32_t least = 0xFFFFFFFFu, most = 0u;   // magnitudes as integers, less one: 0 is the largest of all
#pragma unroll
    for (int c = 0; c < 64; ++c) {
      const uint32_t a = 2u * __float_as_uint(o[c]);
      least = min(least, a - 1u);
      most = max(most, a);
    }
    redo = redo || most >= 2u * 0x7F800000u || least < 2u * __float_as_uint(kTiny) - 1u;
    {   // for both halves of the row
      float* const xt = x_s + (n_tiles & 1) * 2 * kBM;
      xt[half * kBM + row] = redo ? 1.f : 0.f;
      asm volatile("bar.sync 5, 256;" ::: "memory");   // the row warps
      redo = redo || xt[(half ^ 1) * kBM + row] != 0.f || *huge_s != 0;
    }
    // ---- this CTA's partial rows into shared memory (over Q: the last P V followed every S)
    float* const dst = reinterpret_cast<float*>(smem) + row * kD;
    if (ok && redo && row < rows) {
      const float2 ml = plain_row(p, static_cast<const float*>(p.q) + q_row(row) * kD, layer, b, hkv, k_lo, k_hi, C,
                                  make_uint4(am[0], am[1], am[2], am[3]), half, dst, row & 7);
      m_run = ml.x;
      l_run = half == 0 ? ml.y : 0.f;
    } else {
#pragma unroll
      for (int c = 0; c < 16; ++c)
        *reinterpret_cast<float4*>(dst + (((half * 16 + c) ^ (row & 7)) << 2)) =
            make_float4(o[4 * c], o[4 * c + 1], o[4 * c + 2], o[4 * c + 3]);
    }
    float* const xt = x_s + ((n_tiles + 1) & 1) * 2 * kBM;
    xt[half * kBM + row] = l_run;
    asm volatile("bar.sync %0, 64;" ::"r"(1 + (warp & 3)) : "memory");
    if (half == 0) *reinterpret_cast<float2*>(ml_s + 2 * row) = make_float2(m_run, l_run + xt[kBM + row]);
    tc_fence_before();
    __syncthreads();
    cluster.sync();
    // ---- combine: CTA r writes the r-th share of the rows, one row per warp at a time
    const int r_lo = rank * rows / csize, r_hi = (rank + 1) * rows / csize;
    float4 part[kMaxCluster], next[kMaxCluster];
    float2 ml = make_float2(-INFINITY, 0.f), ml_next = ml;
#pragma unroll 1
    for (int r = r_lo + warp - kRowWarps; r < r_hi; r += kRowWarps) {   // (a row's reads are issued one row ahead)
      const int rn = r + kRowWarps;
      if (rn < r_hi) {
        if (lane < csize) ml_next = *reinterpret_cast<const float2*>(cluster.map_shared_rank(ml_s, lane) + 2 * rn);
#pragma unroll
        for (int c = 0; c < kMaxCluster; ++c)
          if (c < csize)
            next[c] = *reinterpret_cast<const float4*>(cluster.map_shared_rank(reinterpret_cast<float*>(smem), c) +
                                                       rn * kD + ((lane ^ (rn & 7)) << 2));
      }
      if (r >= r_lo) {
        float mm = ml.x;
#pragma unroll
        for (int d = 4; d > 0; d >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, d));
        const float w = ml.y > 0.f ? exp2f(ml.x - mm) : 0.f;
        float lw = ml.y * w;
#pragma unroll
        for (int d = 4; d > 0; d >>= 1) lw += __shfl_xor_sync(0xffffffffu, lw, d);
        lw = __shfl_sync(0xffffffffu, lw, 0);
        const float inv = lw > 0.f ? 1.f / lw : 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int c = 0; c < kMaxCluster; ++c) {
          const float wc = __shfl_sync(0xffffffffu, w, c);
          if (c < csize) {
            acc.x = fmaf(wc, part[c].x, acc.x);
            acc.y = fmaf(wc, part[c].y, acc.y);
            acc.z = fmaf(wc, part[c].z, acc.z);
            acc.w = fmaf(wc, part[c].w, acc.w);
          }
        }
        reinterpret_cast<float4*>(static_cast<float*>(p.out) + q_row(r) * kD)[lane] =
            make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
      }
#pragma unroll
      for (int c = 0; c < kMaxCluster; ++c) part[c] = next[c];
      ml = ml_next;
    }
  }
  cluster.sync();   // keep this CTA's shared memory alive until the others have read it
}

}  // namespace split

cudaError_t launch_tree_attn_split(const AttnParams& p, int csize, cudaStream_t stream) {
  if (p.hq > 65535 || p.n_total > 65535 || p.layers > 65535) return cudaErrorInvalidValue;
  const int m_blocks = (p.max_nodes * p.group + split::kBM - 1) / split::kBM;
  const long long grid = (long long)csize * m_blocks * p.hkv * p.batch * p.layers;
  if (grid > 0x7fffffffll) return cudaErrorInvalidValue;
  const cudaError_t e = cudaFuncSetAttribute(split::tree_attn_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)split::kSmemBytes);
  if (e != cudaSuccess) return e;
  return launch_chained(split::tree_attn_split_kernel, dim3((unsigned)grid), dim3(split::kThreads), split::kSmemBytes, stream,
                        (unsigned)csize, p, csize, m_blocks,
                        group_divisor(p.group));
}

}  // namespace ptd
