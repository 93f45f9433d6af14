// Internal launcher of the per-node top-k kernel (not part of the C ABI).
#pragma once
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

namespace ptd {
// Greedy verification of each tree by the top-k cluster that completes the tree's rows (the
// step's tail): rows are the trees' nodes, back to back.
struct VerifyArgs {
  const int32_t* node_offsets;   // [batch + 1]
  const int32_t* parents;        // [n_total]
  const int32_t* tokens;         // [n_total]
  unsigned int* counters;        // [batch] rows done per tree, zero before the launch
  int batch, n_total, max_nodes;
  int32_t* accepted;             // [batch][max_nodes]
  int32_t* accept_len;           // [batch]
  int32_t* bonus;                // [batch]
  int32_t* dev_status;
};

// `beside` (below): the kernel's CTAs start on the logits at once, beside the stream's previous grid,
// instead of waiting for it.  For a previous grid that lets its successors be placed only after
// its own dependency wait, and inputs that were complete before that grid began; the outputs are
// written while it runs.  The kernel completes after that grid has.

// The step's streamed top-k with verification (bf16 rows back to back, vocab a multiple of 8,
// logits 16-byte aligned): parts of the rows without clusters, merged through scratch.
// row_counters [rows] (and va.counters) must be zero before the launch; slots holds
// topk_stream_slot_bytes(rows) bytes of scratch (no clearing needed).
bool topk_stream_ok(const void* logits, int vocab);
size_t topk_stream_slot_bytes(int64_t rows);
cudaError_t launch_topk_stream(const void* logits, int64_t rows, int vocab, int k, bool beside, int32_t* out_idx,
                               float* out_val, int32_t* dev_status, const VerifyArgs& va, unsigned int* row_counters,
                               unsigned long long* slots, cudaStream_t stream);

// 64 KB slices of a row of bf16 logits.
int topk_slices(int vocab);

// Launched with programmatic stream serialization; without `beside` the kernel waits for the
// stream's previous grid before its first global access, and it lets the next grid be placed
// early.  With `va` (bf16 only) it also verifies every tree, as ptd_verify_greedy on its column 0
// would; the node_offsets / parents / tokens it reads must have been complete before the
// stream's previous grid began.
cudaError_t launch_topk(const void* logits, bool bf16, int64_t rows, int vocab, int64_t row_stride, int k, bool beside,
                        int32_t* out_idx, float* out_val, int32_t* dev_status, const VerifyArgs* va, int sms,
                        cudaStream_t stream);
}  // namespace ptd
