// Tree-masked attention on the tensor cores for few short units (bf16): a cluster of CTAs per
// (layer, tree, KV head, pair of 128-row M tiles), each CTA an equal share of the unit's key
// tiles, the partial results combined through distributed shared memory.
//
// Same operation, tiles, GEMMs and softmax as attention_tc.cu.  That kernel's balanced cut needs
// a schedule walk before the first copy, fp32 partials in global memory and a second kernel to
// merge them: for a layer of a few us of work these took most of the time (32 MHA heads, 2048 + 31
// keys: of 25 us, 5.5 us were key tiles; 26.9 -> 12.6 us here).  Here a CTA's work follows from its block index, the
// first copies start as soon as the tree's sizes are read, and the merge is two cluster
// barriers and one pass over shared memory (no scratch): the partials go to shared memory as they are,
// and a warp per row weighs and adds them (with the weights applied before, three barriers and 1-2
// us more).
//
// Units of one M tile run their key tiles as two streams: softmax warps 2-5 take the even tiles
// and warps 6-9 the odd ones, each with S, O, maximum and sum of its own (the TMEM that a second M
// tile would use), so that a tile's chain (S GEMM, softmax, P V) overlaps the next tile's; the
// streams are two more partials of the merge.  A key tile takes ~0.8 us this way against ~1.5 us as
// one stream: 32 MHA heads, 32768 keys 105.7 -> 82.6 us (79.4 with the GEMMs issued as now: 6.6 TB/s).
//
// Warp roles (352 threads): warp 0 K producer (and Q), warp 10 V producer (their copies of a paged
// tile are 16 each: one thread issuing both took longer than a tile's GEMMs), warp 1 TMEM and
// MMA issuer, warps 2-9 softmax; all warps combine and write the output.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <type_traits>

#include "attention.cuh"
#include "attention_tc.cuh"
#include "launch.cuh"
#include "ptd_device.cuh"

namespace cg = cooperative_groups;

namespace ptd {
namespace tcc {

using namespace tc;

constexpr int kThreads = 352;
constexpr int kWarps = kThreads / 32;
constexpr int kVWarp = 10;
constexpr int kStages = 2;
constexpr int kMaxNodes = 128;
constexpr uint32_t kOffQ = 0;
constexpr uint32_t kOffRing = 2 * kTileBytes;   // K/V stages; at the end the partial O of both M tiles / streams
constexpr uint32_t kOffMl = kOffRing + kStages * kStageBytes;   // [2][128] (running maximum, row sum)
constexpr uint32_t kOffPar = kOffMl + 2 * 128 * 8;
constexpr uint32_t kOffBar = kOffPar + kMaxNodes * 4;
// full_k[2], full_v[2], empty_k[2], empty_v[2], v_load[2], s_full[2], p_full[2], o_full[2], q_ready[2], drain
constexpr uint32_t kNumBars = 19;
constexpr uint32_t kOffTmemPtr = kOffBar + kNumBars * 8;
constexpr uint32_t kOffAbort = kOffTmemPtr + 4;
constexpr uint32_t kSmemBytes = kOffAbort + 16 + 1024;   // slack to align the base to 1024 B
static_assert(kSmemBytes <= 232448 && kStages * kStageBytes >= 2 * 128 * 128 * 4, "shared memory");

// (A bound of 512 threads keeps the kernel at 128 registers: two CTAs of the step's top-k then fit
// beside each of its CTAs.)
template <bool kPaged, bool kQTma>
__global__ void __launch_bounds__(512, 1)
    tree_attn_cluster_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v,
                             const __grid_constant__ CUtensorMap map_q, const __grid_constant__ AttnParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint32_t base = smem_u32(smem_raw);
  const uint32_t pad = (1024u - (base & 1023u)) & 1023u;   // the same in every CTA
  uint8_t* smem = smem_raw + pad;
  base += pad;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // known to be uniform, for the GEMM issue
  auto bar = [&](int i) { return base + kOffBar + 8u * (uint32_t)i; };
  auto fullk_bar = [&](int s) { return bar(s); };
  auto fullv_bar = [&](int s) { return bar(2 + s); };
  auto emptyk_bar = [&](int s) { return bar(4 + s); };
  auto emptyv_bar = [&](int s) { return bar(6 + s); };
  auto vload_bar = [&](int s) { return bar(8 + s); };   // V of a tile that reaches past the sequence (its tail is zeroed)
  auto sfull_bar = [&](int t) { return bar(10 + t); };
  auto pfull_bar = [&](int t) { return bar(12 + t); };
  auto ofull_bar = [&](int t) { return bar(14 + t); };
  auto qready_bar = [&](int t) { return bar(16 + t); };
  const uint32_t drain_bar = bar(18);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffAbort);
  int* const par_s = reinterpret_cast<int*>(smem + kOffPar);
  float2* const ml_s = reinterpret_cast<float2*>(smem + kOffMl);

  // ---- set-up that reads no global memory: it may overlap the stream's previous grid
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(fullk_bar(i), 1);
      mbar_init(fullv_bar(i), 1);
      mbar_init(emptyk_bar(i), 1);
      mbar_init(emptyv_bar(i), 1);
      mbar_init(vload_bar(i), 1);
      mbar_init(sfull_bar(i), 1);
      mbar_init(pfull_bar(i), 4);                // one arrival per softmax warp
      mbar_init(ofull_bar(i), 1);
      mbar_init(qready_bar(i), kQTma ? 1 : 4);   // the TMA issuer, or one arrival per softmax warp
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tensormap(&map_k);
    prefetch_tensormap(&map_v);
    if (kQTma) prefetch_tensormap(&map_q);
  }
  if (warp == 1) {
    tmem_alloc(base + kOffTmemPtr, kTmemCols);
    tmem_relinquish();
    tc_fence_before();
  }
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + kOffTmemPtr);
  grid_dependency_wait();   // every input (trees, Q, the cache) and output belongs to the stream's previous work
  if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) {   // counters of the step's tail (see AttnParams)
    for (int i = tid; i < p.zero_count; i += kThreads) p.zero_ptr[i] = 0u;
    __threadfence();
  }

  // ---- this CTA's share (every CTA of the cluster decides alike on its unit)
  const int rank = (int)blockIdx.x, csize = (int)gridDim.x;
  const int b = (int)(blockIdx.z % (unsigned)p.batch), lq = (int)(blockIdx.z / (unsigned)p.batch);
  const int hkv = p.pairs == 1 ? (int)blockIdx.y : (int)blockIdx.y / p.pairs;
  const int mp = (int)blockIdx.y - hkv * p.pairs;
  const int G = p.group;
  const int node0 = p.node_offsets[b];
  const int T = p.node_offsets[b + 1] - node0;
  const int C = p.ctx_lens[b];
  const int N = C + T;
  const bool bad = T < 1 || T > p.max_nodes || node0 < 0 || node0 + T > p.n_total || C < 0 ||
                   (p.page_size > 0 ? N > p.max_pages * p.page_size : N > p.seq_capacity);
  const int m_tiles = bad ? 0 : (T * G + 127) / 128;
  const int nt = min(2, m_tiles - 2 * mp);   // M tiles of this unit (below 1: none)
  if (bad && rank == 0 && blockIdx.y == 0 && tid == 0) atomicMax(p.dev_status, (int)PTD_ERR_INVALID_TREE);
  if (nt < 1) {
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
    return;
  }
  const bool dual = nt == 1;
  const int n_kt = (N + 127) >> 7;
  const int kt0 = rank * n_kt / csize;
  const int n = (rank + 1) * n_kt / csize - kt0;   // this CTA's key tiles (may be none)
  const int layer = p.layer_begin + lq;
  const size_t out_row0 = ((size_t)lq * p.n_total + node0) * p.hq + (size_t)hkv * G;   // + node * hq + head

  // one tile of K or V (one thread)
  const uint64_t kv_policy = l2_policy_evict_first();
  auto load_tile = [&](int j, bool is_v) {
    const int st = j & 1, t0 = (kt0 + j) * 128;
    const CUtensorMap* map = is_v ? &map_v : &map_k;
    const uint32_t fb = is_v ? (t0 + 128 > N ? vload_bar(st) : fullv_bar(st)) : fullk_bar(st);
    const uint32_t d = base + kOffRing + (uint32_t)st * kStageBytes + (is_v ? kTileBytes : 0u);
    if (!kPaged) {
      const int row = (layer * p.batch + b) * p.seq_capacity + t0;
      mbar_arrive_expect_tx(fb, kTileBytes);
      tma_load_3d_hint(d, map, fb, 0, hkv, row, kv_policy);
      tma_load_3d_hint(d + kHalfBytes, map, fb, 64, hkv, row, kv_policy);
    } else {
      const int ps = p.page_size, first = t0 / ps;
      const int nvalid = min(128 / ps, (N + ps - 1) / ps - first);
      const int* bt = p.block_table + (size_t)b * p.max_pages + first;
      int phys[8];   // loaded together, so that the copies do not each wait for their own
#pragma unroll
      for (int pg = 0; pg < 8; ++pg) phys[pg] = pg < nvalid ? bt[pg] : 0;
      mbar_arrive_expect_tx(fb, (uint32_t)(nvalid * 2 * ps * 128));
#pragma unroll
      for (int pg = 0; pg < 8; ++pg) {
        if (pg < nvalid) {
          const int row = (layer * p.num_pages + phys[pg]) * ps;
          const uint32_t off = (uint32_t)(pg * ps * 128);
          tma_load_3d_hint(d + off, map, fb, 0, hkv, row, kv_policy);
          tma_load_3d_hint(d + kHalfBytes + off, map, fb, 64, hkv, row, kv_policy);
        }
      }
    }
  };
  // the first tiles (both stages are free) and Q are asked for before the tree is read
  if (n > 0 && lane == 0) {
    if (warp == 0) {
      load_tile(0, false);
      if (kQTma) {
        for (int t = 0; t < nt; ++t) {   // 128 / G nodes x G heads, two 64-column halves
          const int qrow = lq * p.n_total + node0 + ((2 * mp + t) * 128) / G;
          const uint32_t dst = base + kOffQ + (uint32_t)t * kTileBytes;
          mbar_arrive_expect_tx(qready_bar(t), kTileBytes);
          tma_load_3d(dst, &map_q, qready_bar(t), 0, hkv * G, qrow);
          tma_load_3d(dst + kHalfBytes, &map_q, qready_bar(t), 64, hkv * G, qrow);
        }
      }
      if (n > 1) load_tile(1, false);
    } else if (warp == kVWarp) {
      load_tile(0, true);
      if (n > 1) load_tile(1, true);
    }
  }
  bool bad_par = false;
  if (tid < T) {
    const int pp = p.parents[node0 + tid];
    par_s[tid] = pp;
    bad_par = tid == 0 ? (pp != -1) : (pp < 0 || pp >= tid);
  }
  const bool invalid = __syncthreads_or(bad_par) != 0;
  // the grids after this one may be placed from here on (as in attention_tc.cu)
  if (tid == 0) grid_launch_dependents();
  if (invalid && rank == 0 && tid == 0) atomicMax(p.dev_status, (int)PTD_ERR_INVALID_TREE);

  float m_run = -INFINITY, l_run = 0.f;
  const int t = (warp - 2) >> 2;              // softmax warps: M tile, or stream
  const int row = (warp & 3) * 32 + lane;     // = TMEM lane this warp may access
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  const uint32_t tO = tmem + lane_base + 256u + (uint32_t)(t & 1) * 128u;
  int mine = 0;                               // key tiles this softmax warp took
  if (warp == 0 || warp == kVWarp) {
    // ================================================================ producers (K; V)
    const bool is_v = warp == kVWarp;
    bool ok = true;
    int issued = n < 2 ? n : 2;
    for (int j = 0; j < n && ok; ++j) {
      const int st = j & 1;
      if (j >= 2) {
        if (lane == 0) {
          ok = mbar_wait(is_v ? emptyv_bar(st) : emptyk_bar(st), (uint32_t)(((j >> 1) & 1) ^ 1), abort_flag, p.dev_status);
          if (ok) load_tile(j, is_v);
        }
        ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        if (!ok) break;
        issued = j + 1;
      }
      const int t0 = (kt0 + j) * 128;
      if (is_v && t0 + 128 > N) {
        // V rows past the sequence: zero them so that P = 0 never meets a non-finite value (the
        // unit's last tile only, so v_load of a stage completes once)
        ok = mbar_wait_warp(vload_bar(st), 0u, abort_flag, p.dev_status);
        if (ok) {
          const uint32_t vbase = base + kOffRing + (uint32_t)st * kStageBytes + kTileBytes;
          const int r0 = N - t0;
          for (int c = lane; c < (128 - r0) * 16; c += 32) {
            const int r = r0 + (c >> 4), hc = c & 15;
            st_shared_v4(vbase + (uint32_t)(hc >> 3) * kHalfBytes + (uint32_t)r * 128u + (uint32_t)(hc & 7) * 16u, 0, 0,
                         0, 0);
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(fullv_bar(st));
        }
      }
    }
    if (!ok && lane == 0) {
      // drain the copies already issued (bounded) before the CTA can exit
      for (int back = 1; back <= kStages && issued - back >= 0; ++back) {
        const int j2 = issued - back;
        mbar_drain(is_v ? fullv_bar(j2 & 1) : fullk_bar(j2 & 1), (uint32_t)((j2 >> 1) & 1), 100000000ull);
        if (is_v) mbar_drain(vload_bar(j2 & 1), 0u, 100000000ull);
        if (!is_v && kQTma) mbar_drain(qready_bar(back - 1), 0u, 100000000ull);
      }
    }
  } else if (warp == 1) {
    // ================================================================ MMA issuer
    if (n > 0) {
      const uint32_t dq = (uint32_t)smem_desc_sw128(base + kOffQ, 16, 1024), dk = (uint32_t)smem_desc_sw128(base + kOffRing, 16, 1024),
                     dv = (uint32_t)smem_desc_sw128(base + kOffRing + kTileBytes, kHalfBytes, 1024);
      const uint32_t leader = lane == 0 ? 1u : 0u;
      auto commit = [&](uint32_t b) {
        if (leader) mma_commit(b);
      };
      auto wait = [&](uint32_t bar_, uint32_t parity) { return mbar_wait_warp(bar_, parity, abort_flag, p.dev_status); };
      auto s_gemm = [&](int tt, int j) {   // S_tt of tile j
        issue_s(leader, tmem + (uint32_t)tt * 128u, dq + (dual ? 0u : (uint32_t)tt * (kTileBytes >> 4)),
                dk + (uint32_t)(j & 1) * (kStageBytes >> 4));
        commit(sfull_bar(tt));
      };
      auto pv_gemm = [&](int tt, int j, bool acc) {
        issue_pv(leader, tmem + (uint32_t)tt * 128u, dv + (uint32_t)(j & 1) * (kStageBytes >> 4), acc);
      };
      bool ok = true;
      for (int tt = 0; tt < nt && ok; ++tt) ok = wait(qready_bar(tt), 0u);
      if (dual) {
        // tile j in stream j % 2: S(j + 2) follows P V(j) (they share the stream's TMEM)
        for (int j = 0; j < (n < 2 ? n : 2) && ok; ++j) {
          if (!(ok = wait(fullk_bar(j), 0u))) break;
          tc_fence_after();
          s_gemm(j, j);
          commit(emptyk_bar(j));
        }
        for (int j = 0; j < n && ok; ++j) {
          const int tt = j & 1;
          const uint32_t ph = (uint32_t)((j >> 1) & 1);
          if (!(ok = wait(fullv_bar(tt), ph))) break;
          if (!(ok = wait(pfull_bar(tt), ph))) break;
          tc_fence_after();
          pv_gemm(tt, j, j >= 2);
          commit(emptyv_bar(tt));
          if (j + 2 >= n) {
            commit(ofull_bar(tt));
          } else {
            if (!(ok = wait(fullk_bar(tt), ph ^ 1u))) break;
            tc_fence_after();
            s_gemm(tt, j + 2);
            commit(emptyk_bar(tt));
          }
        }
      } else {
        ok = ok && wait(fullk_bar(0), 0u);
        if (ok) {
          tc_fence_after();
          s_gemm(0, 0);
          s_gemm(1, 0);
          commit(emptyk_bar(0));
        }
        for (int j = 0; j < n && ok; ++j) {
          const int st = j & 1, st1 = st ^ 1;
          const bool more = j + 1 < n;
          if (!(ok = wait(fullv_bar(st), (uint32_t)((j >> 1) & 1)))) break;
          if (!(ok = wait(pfull_bar(0), (uint32_t)(j & 1)))) break;
          tc_fence_after();
          pv_gemm(0, j, j > 0);
          if (more) {
            if (!(ok = wait(fullk_bar(st1), (uint32_t)(((j + 1) >> 1) & 1)))) break;
            tc_fence_after();
            s_gemm(0, j + 1);
          } else {
            commit(ofull_bar(0));
          }
          if (!(ok = wait(pfull_bar(1), (uint32_t)(j & 1)))) break;
          tc_fence_after();
          pv_gemm(1, j, j > 0);
          commit(emptyv_bar(st));
          if (more) {
            s_gemm(1, j + 1);
            commit(emptyk_bar(st1));
          } else {
            commit(ofull_bar(1));
          }
        }
      }
      if (!ok && leader) {   // error path: let the tensor core finish what was issued before TMEM is freed
        mma_commit(drain_bar);
        mbar_drain(drain_bar, 0, 100000000ull);
      }
    }
  } else {
    // ================================================================ softmax
    const int grow = (2 * mp + (dual ? 0 : t)) * 128 + row;
    const int node = grow / G;
    const bool row_valid = node < T;
    if (!kQTma && n > 0 && (!dual || t == 0)) {
      // this thread's Q row into shared memory (128-byte swizzle)
      const uint4* src = reinterpret_cast<const uint4*>(p.q) +
                         (row_valid ? (out_row0 + (size_t)node * p.hq + (grow - node * G)) * 16 : 0);
      const uint32_t dst = base + kOffQ + (uint32_t)t * kTileBytes + (uint32_t)row * 128u;
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const uint4 v = row_valid ? __ldg(src + c) : make_uint4(0, 0, 0, 0);
        st_shared_v4(dst + (uint32_t)(c >> 3) * kHalfBytes + (uint32_t)(((c & 7) ^ (row & 7)) << 4), v.x, v.y, v.z, v.w);
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(qready_bar(t));
    }
    uint32_t am0 = 0, am1 = 0, am2 = 0, am3 = 0;   // ancestor mask of this row's node
    if (row_valid && !invalid && (kt0 + n) * 128 > C) {
      for (int q = node; q >= 0; q = par_s[q]) {
        const uint32_t bit = 1u << (q & 31);
        const int w = q >> 5;
        am0 |= w == 0 ? bit : 0u;
        am1 |= w == 1 ? bit : 0u;
        am2 |= w == 2 ? bit : 0u;
        am3 |= w == 3 ? bit : 0u;
      }
    }
    const uint32_t tS = tmem + lane_base + (uint32_t)t * 128u;
    const int todo = dual ? (n + 1 - t) >> 1 : n;
    bool ok = true;
    for (; mine < todo; ++mine) {
      if (!(ok = mbar_wait_warp(sfull_bar(t), (uint32_t)(mine & 1), abort_flag, p.dev_status))) break;
      tc_fence_after();
      const int t0 = (kt0 + (dual ? 2 * mine + t : mine)) * 128;
      softmax_tile(tS, tO, mine > 0, t0 + 128 > C, t0 - C, am0, am1, am2, am3, p.scale_log2, m_run, l_run);
      __syncwarp();
      if (lane == 0) mbar_arrive(pfull_bar(t));
    }
    if (todo > 0 && ok) ok = mbar_wait_warp(ofull_bar(t), 0u, abort_flag, p.dev_status);
    tc_fence_after();
    // ---- this thread's partial row, as it is, into shared memory: the ring is free once both halves of
    // the softmax warps have seen their last P V
    asm volatile("bar.sync 1, 256;" ::: "memory");
    ml_s[t * 128 + row] = make_float2(m_run, ok ? l_run : 0.f);   // (a failed wait: the status says so)
    if (todo > 0) {   // (else O was not written; its weight is 0)
      float4* dst = reinterpret_cast<float4*>(smem + kOffRing) + (size_t)(t * 128 + row) * 32;
#pragma unroll 1
      for (int c = 0; c < 4; ++c) {
        uint32_t r[32];
        tmem_ld32(tO + (uint32_t)c * 32u, r);
        tmem_ld_wait();
#pragma unroll
        for (int g = 0; g < 8; ++g)   // chunk c of row r at c ^ (r & 31), and r & 31 = lane
          dst[(c * 8 + g) ^ lane] = make_float4(__uint_as_float(r[4 * g]), __uint_as_float(r[4 * g + 1]),
                                                __uint_as_float(r[4 * g + 2]), __uint_as_float(r[4 * g + 3]));
      }
    }
    tc_fence_before();
  }

  // ---- combine: a warp per row of this CTA's share, over the row's partials (CTA, and stream where
  // there are two) in a fixed order: O = sum_c 2^(m_c - M) O_c / sum_c 2^(m_c - M) l_c
  cluster.sync();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
  {
    const float4* const o_s = reinterpret_cast<const float4*>(smem + kOffRing);
    const int rows = min(nt * 128, T * G - 256 * mp);
    const int r_lo = rank * rows / csize, r_hi = (rank + 1) * rows / csize;
    const int np = dual ? 2 * csize : csize;   // partial i: CTA i / 2, stream i % 2, or CTA i
    auto cta_of = [&](int i) { return dual ? i >> 1 : i; };
    auto row_of = [&](int r, int i) { return r + (dual ? (i & 1) * 128 : 0); };
    // rows of at most NP partials each, eight partials in flight per lane (16 with NP = 16)
    auto reduce = [&](auto np_max) {
      constexpr int NP = decltype(np_max)::value, R = NP < 8 ? 8 / NP : 1;
#pragma unroll 1
      for (int r0 = r_lo + warp * R; r0 < r_hi; r0 += kWarps * R) {
        float2 ml = make_float2(-INFINITY, 0.f);   // lane: row r0 + lane / NP, partial lane % NP
        const int li = lane % NP, lr = r0 + lane / NP;
        if (lane < R * NP && li < np && lr < r_hi) ml = *(cluster.map_shared_rank(ml_s, cta_of(li)) + row_of(lr, li));
        float4 part[R][NP];
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll
          for (int i = 0; i < NP; ++i)
            if (i < np && r0 + q < r_hi)
              part[q][i] = *(cluster.map_shared_rank(o_s, cta_of(i)) + (size_t)row_of(r0 + q, i) * 32 + lane);
        float M = partial_counts(ml.y) ? ml.x : -INFINITY;
#pragma unroll
        for (int o = NP / 2; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        const float w = partial_counts(ml.y) ? ptx_exp2(ml.x - M) : 0.f;
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const int r = r0 + q;
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
          float L = 0.f;
#pragma unroll
          for (int i = 0; i < NP; ++i) {
            const float wi = __shfl_sync(0xffffffffu, w, q * NP + i), l = __shfl_sync(0xffffffffu, ml.y, q * NP + i);
            if (partial_counts(l)) {
              L = fmaf(wi, l, L);
              acc.x = fmaf(wi, part[q][i].x, acc.x);
              acc.y = fmaf(wi, part[q][i].y, acc.y);
              acc.z = fmaf(wi, part[q][i].z, acc.z);
              acc.w = fmaf(wi, part[q][i].w, acc.w);
            }
          }
          const float inv = L > 0.f ? 1.f / L : 0.f;
          if (r < r_hi) {
            const int grow = 256 * mp + r, node = grow / G;
            uint2* dst = reinterpret_cast<uint2*>(p.out) + (out_row0 + (size_t)node * p.hq + (grow - node * G)) * 32;
            const uint2 v = make_uint2(pack_bf16x2(acc.x * inv, acc.y * inv), pack_bf16x2(acc.z * inv, acc.w * inv));
            dst[lane ^ (r & 31)] = invalid ? make_uint2(0u, 0u) : v;
          }
        }
      }
    };
    if (np <= 2)
      reduce(std::integral_constant<int, 2>{});
    else if (np <= 4)
      reduce(std::integral_constant<int, 4>{});
    else if (np <= 8)
      reduce(std::integral_constant<int, 8>{});
    else
      reduce(std::integral_constant<int, 16>{});
  }
  cluster.sync();   // keep this CTA's shared memory alive until the others have read it
}

}  // namespace tcc

cudaError_t launch_tree_attn_cluster(const CUtensorMap& map_k, const CUtensorMap& map_v, const CUtensorMap& map_q,
                                     const AttnParams& p, int csize, cudaStream_t stream) {
  const dim3 grid((unsigned)csize, (unsigned)(p.hkv * p.pairs), (unsigned)(p.batch * p.layers));
  auto* kernel = p.page_size > 0
                     ? (p.q_tma ? tcc::tree_attn_cluster_kernel<true, true> : tcc::tree_attn_cluster_kernel<true, false>)
                     : (p.q_tma ? tcc::tree_attn_cluster_kernel<false, true> : tcc::tree_attn_cluster_kernel<false, false>);
  const cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tcc::kSmemBytes);
  if (e != cudaSuccess) return e;
  return launch_chained(kernel, grid, dim3(tcc::kThreads), tcc::kSmemBytes, stream, (unsigned)csize, map_k, map_v, map_q, p);
}

}  // namespace ptd
