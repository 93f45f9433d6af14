// Pieces shared by the tensor-core attention kernels (attention_tc.cu, attention_cluster.cu):
// tile geometry, the GEMM issue, and the softmax of one key tile.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "attention.cuh"
#include "ptd_device.cuh"

namespace ptd {
namespace tc {

constexpr uint32_t kTileBytes = 32768;   // 128 rows x 128 bf16
constexpr uint32_t kHalfBytes = 16384;   // 128 rows x 64 bf16 (one 128-byte swizzle column)
constexpr uint32_t kStageBytes = 2 * kTileBytes;   // a K tile, then a V tile
constexpr uint32_t kTmemCols = 512;                // S_0 | S_1 | O_0 | O_1, 128 fp32 columns each
constexpr float kRescaleLog2 = 8.0f;               // lazy rescale threshold (log2 units)

constexpr uint32_t kIdescS = idesc_bf16_f32(128, 128, 0, 0);    // Q (K-major) x K (K-major)
constexpr uint32_t kIdescPV = idesc_bf16_f32(128, 128, 0, 1);   // P (K-major) x V (MN-major)

// Bits [a0, a0+32) of "is slot C + a visible": a < 0 is committed context (visible),
// 0 <= a < 128 reads the node's ancestor mask, a >= 128 is past the tree.
__device__ __forceinline__ uint32_t vis_word(int a0, uint32_t m0, uint32_t m1, uint32_t m2, uint32_t m3) {
  if (a0 <= -32) return 0xFFFFFFFFu;
  if (a0 < 0) {
    const int sh = -a0;   // 1..31
    return (m0 << sh) | ((1u << sh) - 1u);
  }
  if (a0 >= 128) return 0u;
  const int w = a0 >> 5, sh = a0 & 31;
  const uint32_t lo = w == 0 ? m0 : w == 1 ? m1 : w == 2 ? m2 : m3;
  const uint32_t hi = w == 0 ? m1 : w == 1 ? m2 : w == 2 ? m3 : 0u;
  return __funnelshift_r(lo, hi, sh);
}

// Rare path of the softmax, kept out of the hot loop: O_t (n_o 16-column groups) and the
// bf16 P chunks [0, c) of S_t scaled by alpha.  Warp-collective.
static __device__ __noinline__ void rescale_tmem(uint32_t tO, uint32_t tS, int n_o, int c, float alpha) {
  for (int q = 0; q < n_o; ++q) {
    uint32_t o16[16];
    tmem_ld16(tO + (uint32_t)q * 16u, o16);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 16; ++e) o16[e] = __float_as_uint(__uint_as_float(o16[e]) * alpha);
    tmem_st16(tO + (uint32_t)q * 16u, o16);
  }
  if (c > 0) tmem_st_wait();
  for (int q = 0; q < c; ++q) {
    uint32_t p16[16];
    tmem_ld16(tS + (uint32_t)q * 16u, p16);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 16; ++e)
      p16[e] = pack_bf16x2(__uint_as_float(p16[e] << 16) * alpha, __uint_as_float(p16[e] & 0xFFFF0000u) * alpha);
    tmem_st16(tS + (uint32_t)q * 16u, p16);
  }
}

// GEMM issue.  The whole warp calls, in a branch on a broadcast warp number (so that the compiler
// knows it uniform), and the lane with `leader` != 0 issues, by predication: descriptors and TMEM
// addresses then lie in uniform registers, where the instruction takes them.  Against one thread
// issuing in a branch of its own (back to back): 32768 keys under 128 nodes of 64 heads 117.4 -> 112.4 us, 32
// layers of 8192 keys under 63 nodes with the step's tail 234.7 -> 225.8, a 32-head MHA layer 13.4 -> 12.6, 611
// keys 8.5 -> 8.25.  Descriptors come as their low words; the high word is the same for all.
constexpr uint32_t kDescHi = (1u << 14) | (1024u >> 4) | (2u << 29);   // stride 1024, version 1, 128-byte swizzle
// S_t (TMEM, 128 columns at s_tmem) = Q K^T: descriptor words of the Q tile and the K tile.
__device__ __forceinline__ void issue_s(uint32_t leader, uint32_t s_tmem, uint32_t q_desc, uint32_t k_desc) {
#pragma unroll
  for (int kk = 0; kk < 8; ++kk) {
    const uint32_t o = (uint32_t)(kk >> 2) * (kHalfBytes >> 4) + (uint32_t)(kk & 3) * 2u;
    mma_ss_if(leader, s_tmem, q_desc + o, k_desc + o, kDescHi, kIdescS, kk > 0 ? 1u : 0u);
  }
}
// O_t (TMEM, 256 columns past S_t) (+)= P V: P_t (bf16, 16 keys = 8 packed columns per step) over S_t,
// descriptor word of the V tile.
__device__ __forceinline__ void issue_pv(uint32_t leader, uint32_t s_tmem, uint32_t v_desc, bool acc) {
#pragma unroll
  for (int kk = 0; kk < 8; ++kk)
    mma_ts_if(leader, s_tmem + 256u, s_tmem + (uint32_t)kk * 8u, v_desc + (uint32_t)kk * 128u, kDescHi, kIdescPV,
              (acc || kk > 0) ? 1u : 0u);
}

// A partial (m, l, O) of a row counts unless the row saw no key in it: then l is exactly 0, m = -inf and O
// was not written.  (Not l > 0: a NaN among the scores makes l NaN, and has to reach the output.)
__device__ __forceinline__ bool partial_counts(float l) { return !(l == 0.f); }

// Softmax of one key tile of this thread's row: S (TMEM at tS) becomes the bf16 P over its first
// 64 columns, against the reference maximum m_run (log2 units), which only moves up, and only
// when a 32-column chunk exceeds it by more than 2^8; then the row sum, O (TMEM at tO, if `has_o`)
// and the P chunks already written are rescaled.  c0 = the tile's first key less the context
// length; the ancestor mask am applies when `need_mask` (warp-uniform).  Warp-collective.
__device__ __forceinline__ void softmax_tile(uint32_t tS, uint32_t tO, bool has_o, bool need_mask, int c0, uint32_t am0,
                                             uint32_t am1, uint32_t am2, uint32_t am3, float sl2, float& m_run,
                                             float& l_run) {
  const unsigned long long sl2x2 = f2_pack(sl2, sl2);
  uint32_t r[32];
  unsigned long long sum = f2_pack(0.f, 0.f);
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    tmem_ld32(tS + (uint32_t)c * 32u, r);
    tmem_ld_wait();
    if (need_mask) {
      const uint32_t vw = vis_word(c0 + c * 32, am0, am1, am2, am3);
#pragma unroll
      for (int e = 0; e < 32; ++e) r[e] = ((vw >> e) & 1u) ? r[e] : __float_as_uint(-INFINITY);
    }
    float cm;
    {
      float a0 = -INFINITY, a1 = -INFINITY;
#pragma unroll
      for (int e = 0; e < 32; e += 4) {
        a0 = fmax3(a0, __uint_as_float(r[e]), __uint_as_float(r[e + 1]));
        a1 = fmax3(a1, __uint_as_float(r[e + 2]), __uint_as_float(r[e + 3]));
      }
      cm = fmaxf(a0, a1) * sl2;
    }
    // The TMEM accesses of a rescale are warp-collective, so the whole warp takes the
    // branch when any of its rows needs it; the other rows rescale by exactly 1.  (Rows
    // differ when a piece starts on a key tile past the committed context: each row
    // first meets a visible ancestor in whichever chunk holds one.)
    const bool raise = cm > m_run + kRescaleLog2;
    if (__any_sync(0xffffffffu, raise)) {
      // raise the reference: rescale everything taken against the old one
      float alpha = 1.f;
      if (raise) {
        alpha = m_run == -INFINITY ? 0.f : ptx_exp2(m_run - cm);
        m_run = cm;
      }
      float s0, s1;
      f2_unpack(sum, s0, s1);
      sum = f2_pack(s0 * alpha, s1 * alpha);
      l_run *= alpha;
      rescale_tmem(tO, tS, has_o ? 8 : 0, c, alpha);
    }
    const float m_use = m_run == -INFINITY ? 0.f : m_run;   // -inf only while nothing is visible
    const unsigned long long negm = f2_pack(-m_use, -m_use);
    uint32_t pk[16];
#pragma unroll
    for (int e = 0; e < 32; e += 2) {
      const unsigned long long x =
          f2_fma(f2_pack(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), sl2x2, negm);
      float x0, x1;
      f2_unpack(x, x0, x1);
      const float p0 = ptx_exp2(x0), p1 = ptx_exp2(x1);
      sum = f2_add(sum, f2_pack(p0, p1));
      pk[e >> 1] = pack_bf16x2(p0, p1);
    }
    tmem_st16(tS + (uint32_t)c * 16u, pk);   // P chunk c: columns [16c, 16c+16) of S_t
  }
  {
    float s0, s1;
    f2_unpack(sum, s0, s1);
    l_run += s0 + s1;
  }
  tmem_st_wait();
  tc_fence_before();
}

}  // namespace tc
}  // namespace ptd
