// Internal launch parameters of the tree-attention kernels (not part of the C ABI).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace ptd {

struct AttnParams {
  const void* q;               // [layers][n_total][hq][D]
  void* out;                   // [layers][n_total][hq][D]
  float* part_o;               // piece partials: [slot][M tile][D / 4][128 rows][4] fp32 (O unnormalised)
  float* part_ml;              // [slot][256 rows][2] (running max in log2 units, row sum)
  unsigned long long* counters;   // persistent schedule: pieces finished per (unit, 32-row block):
                                  // (epoch << 32) | count, a value of another epoch counting as 0
  uint32_t epoch;                 // this launch's epoch (never 0)
  unsigned int* zero_ptr;         // zero_count words that CTA 0 clears after its dependency wait and before
  int zero_count;                 // it lets later grids be placed: the step's tail counters
  const int32_t* node_offsets;
  const int32_t* parents;
  const int32_t* ctx_lens;
  const int32_t* block_table;
  const void* k;               // cache base pointers (SIMT path)
  const void* v;
  int32_t* dev_status;
  int batch, hq, hkv, group, head_dim;
  int layer_begin, layers;     // layers of this call
  int n_total, max_nodes;
  int pairs;                   // 256-row M-tile pairs per (tree, KV head)
  int persistent;              // 1: balanced persistent schedule, one CTA per SM
  int defer_merge;             // persistent: every piece leaves a partial; tree_attn_merge_kernel merges
  int ctas;                    // persistent: the attention grid's CTAs (the cut the merge kernel follows)
  int q_tma;                   // 1: Q tiles arrive by TMA (map_q), else by per-thread loads
  int page_size, seq_capacity, num_pages, max_pages;
  float scale_log2;            // scale * log2(e)
};

size_t tc_smem_bytes();
// Launched with programmatic stream serialization: the kernel's set-up (barriers, tensor
// memory, descriptor prefetch) may overlap the stream's previous grid; it waits for that grid
// before its first global access.
cudaError_t launch_tree_attn_tc(const CUtensorMap& map_k, const CUtensorMap& map_v, const CUtensorMap& map_q,
                                const AttnParams& p, dim3 grid, cudaStream_t stream);
// How many clusters of c CTAs (1 to 8), each filling an SM, run at once: cudaOccupancyMaxActiveClusters'
// answers on the 152 SMs of a GB300, whose clusters lie within a GPC; by proportion for another number
// of SMs (an estimate only, for the choice between kernels).
inline int clusters_at_once(int c, int sms) {
  constexpr int fit152[9] = {0, 152, 76, 46, 36, 28, 23, 15, 15};
  const int f = fit152[c] * sms / 152;
  return f > 0 ? f : 1;
}

// Few short units: a cluster of `csize` CTAs per unit (csize <= 8), no scratch; p.pairs set as for
// one CTA per unit.  Programmatic dependent launch.
cudaError_t launch_tree_attn_cluster(const CUtensorMap& map_k, const CUtensorMap& map_v, const CUtensorMap& map_q,
                                     const AttnParams& p, int csize, cudaStream_t stream);
// fp32 attention on the CUDA cores, a cluster of `csize` CTAs (csize <= 8) per block of rows.  map_k:
// boxes of 32 columns (128-byte swizzle), map_v: of D columns, both of one KV head and
// simt_box_rows(page_size) rows.
cudaError_t launch_tree_attn_simt(const CUtensorMap& map_k, const CUtensorMap& map_v, const AttnParams& p, int csize,
                                  cudaStream_t stream);
// fp32 attention on the tensor cores, D = 128: a cluster of `csize` CTAs (csize <= 8) per block of 128
// rows.  Programmatic dependent launch.
cudaError_t launch_tree_attn_split(const AttnParams& p, int csize, cudaStream_t stream);
// Which of the two, and the cluster size, from the shapes (batch, hkv, group, head_dim, layers, max_nodes).
struct F32Plan {
  bool tensor;
  int csize;
};
F32Plan choose_tree_attn_f32(const AttnParams& p, int max_ctx, int sms);
inline int simt_box_rows(int page_size) { return page_size > 0 ? 16 : 64; }
// The merge of the units the persistent cut split, after the attention kernel (programmatic
// dependent launch): one CTA per unit, the pieces' partials combined in CTA order.
cudaError_t launch_tree_attn_merge(const AttnParams& p, int units, int sms, cudaStream_t stream);

}  // namespace ptd
