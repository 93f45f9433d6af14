// Tree positions, the rotary encoding and the tree's K/V append (Sec. 3.1 "Tree
// Construction": a node's position is set by |pi(v)|).
//
// Node i of tree b sits at position p = C_b + |pi(i)| - 1.  One CTA per (node, group of
// layers): it asks for its rows of q, k and v, stages its tree's parent array in shared memory
// (one load per thread), counts |pi(i)| by walking up (<= 128 shared-memory reads), builds the
// node's D/2 (cos, sin) pairs once, then, with 16-byte vectors where rows allow, turns every pair
// (x_j, x_{j+D/2}) of the node's query heads (in place) and key heads by p * base^(-2j/D)
// (RoFormer's rotation, rotate-half layout; the angle p * f is carried as an fp32 pair
// from a float-float f computed in double on the host, so that its rounding error is
// corrected to first order after sincosf) and writes the rotated keys and the values into
// cache slot C_b + i of each layer (contiguous or paged); a slot outside the cache (or a
// page number outside the pool) writes nothing and sets the status.
//
// What bounds it: the reads and writes (49.5 MB for 32 layers of 63 nodes, 32 query / 8 KV heads)
// and, for few layers, the chain tree, parents, slot, angles.  Measured (GB300; at first with
// that chain before the first read of a row, one thread walking, four layers one after the other):
// 32 layers 14.2 -> 10.4 us (4.8 TB/s), one layer 6.2 -> 3.7, eight fp32 layers 10.4 -> 5.6.  Three
// items a thread at four CTAs per SM: two items 14.1, four 11.7, six 13.3 us.  An item's layer and head by
// multiplications: by division, six a thread and round, batches of some hundred nodes were slower than
// they had been with one item at a time (8 layers of ~345 nodes, 64 / 8 heads 15.9 us, then 21.7, now 17.3).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "launch.cuh"
#include "ptd_device.cuh"
#include "row_division.cuh"
#include "tree_rope.cuh"

namespace ptd {
namespace tr {

constexpr int kThreads = 256;

template <typename T>
__device__ __forceinline__ float ld(const T* p);
template <>
__device__ __forceinline__ float ld<float>(const float* p) { return *p; }
template <>
__device__ __forceinline__ float ld<__nv_bfloat16>(const __nv_bfloat16* p) { return __bfloat162float(*p); }
template <typename T>
__device__ __forceinline__ void st(T* p, float x);
template <>
__device__ __forceinline__ void st<float>(float* p, float x) { *p = x; }
template <>
__device__ __forceinline__ void st<__nv_bfloat16>(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }

// One 16-byte vector of T: 16 / sizeof(T) elements, widened to fp32.
template <typename T>
struct Vec {
  static constexpr int N = 16 / sizeof(T);
  float x[N];
};
template <typename T>
__device__ __forceinline__ Vec<T> unpack16(const uint4& u) {
  Vec<T> r;
  if constexpr (sizeof(T) == 2) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      r.x[2 * i] = __uint_as_float(w[i] << 16);
      r.x[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
    }
  } else {
    r.x[0] = __uint_as_float(u.x), r.x[1] = __uint_as_float(u.y), r.x[2] = __uint_as_float(u.z),
    r.x[3] = __uint_as_float(u.w);
  }
  return r;
}
template <typename T>
__device__ __forceinline__ uint4 pack16(const Vec<T>& r) {
  if constexpr (sizeof(T) == 2) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(r.x[2 * i], r.x[2 * i + 1]);
      w[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
  } else {
    return make_uint4(__float_as_uint(r.x[0]), __float_as_uint(r.x[1]), __float_as_uint(r.x[2]), __float_as_uint(r.x[3]));
  }
}

// What every thread of a CTA works out for its node: the tree, the position and the cache row.
struct Place {
  int pos;      // C + |pi(i)| - 1
  size_t row;   // cache row of its slot, within a layer
  bool fits;
};

// Node n's place (block-wide: one barrier).  Every thread finds the tree, walks the ancestors and
// reads the block table itself: the reads are broadcasts, and no further barrier is needed.
// False (status set) when the tree is not one.
__device__ __forceinline__ bool find_place(const int32_t* node_offsets, const int32_t* parents, const int32_t* ctx_lens,
                                           int batch, int n, int page_size, int seq_capacity, int num_pages,
                                           const int32_t* block_table, int max_pages, bool first, int* par_s,
                                           int32_t* positions_out, int32_t* dev_status, Place& out) {
  const int t = threadIdx.x, lane = t & 31;
  int b = batch - 1;   // the first tree that ends after node n
  for (int b0 = 0; b0 < batch - 1; b0 += 32) {
    const int q = b0 + lane;
    const uint32_t hit = __ballot_sync(0xffffffffu, q < batch - 1 && node_offsets[q + 1] > n);
    if (hit != 0u) {
      b = b0 + __ffs(hit) - 1;
      break;
    }
  }
  const int node0 = node_offsets[b];
  const int T = node_offsets[b + 1] - node0;
  const int C = ctx_lens[b];
  const int i = n - node0;
  bool bad = T < 1 || T > kThreads || i < 0 || i >= T;
  if (!bad && t < T) {
    const int p = parents[node0 + t];
    par_s[t] = p;
    bad = t == 0 ? p != -1 : (p < 0 || p >= t);
  }
  if (__syncthreads_or(bad)) {
    if (t == 0) atomicMax(dev_status, (int)PTD_ERR_INVALID_TREE);
    return false;
  }
  const int slot = C + i;
  const int cap = page_size > 0 ? max_pages * page_size : seq_capacity;
  out.fits = C >= 0 && slot < cap;
  out.row = (size_t)b * seq_capacity + slot;
  if (out.fits && page_size > 0) {
    const int pg = block_table[(size_t)b * max_pages + slot / page_size];
    out.fits = pg >= 0 && pg < num_pages;
    out.row = (size_t)page_size * pg + slot % page_size;
  }
  int depth = 0;
  for (int a = i; a != -1; a = par_s[a]) ++depth;
  out.pos = C + depth - 1;
  if (t == 0 && first) {
    if (positions_out) positions_out[n] = out.pos;
    if (!out.fits) atomicMax(dev_status, (int)PTD_ERR_INVALID_TREE);
  }
  return true;
}

// cos and sin of pos * f_j for j < half, into shared memory (the caller's barrier follows).
__device__ __forceinline__ void make_table(const RopeFreqs& freqs, int pos_i, int half, float* cos_s, float* sin_s) {
  for (int j = threadIdx.x; j < half; j += kThreads) {
    // angle = pos * (hi + lo) = a_hi + a_err (a_err exact up to pos * lo's rounding); sin
    // and cos of a_hi, corrected to first order in a_err (|a_err| < 1e-3)
    const float pos = (float)pos_i, fh = freqs.hi[j];
    const float a_hi = __fmul_rn(pos, fh);
    const float a_err = fmaf(pos, fh, -a_hi) + pos * freqs.lo[j];
    float s0, c0;
    sincosf(a_hi, &s0, &c0);
    sin_s[j] = fmaf(a_err, c0, s0);
    cos_s[j] = fmaf(-a_err, s0, c0);
  }
}

// Rows of 16-byte vectors.  A row of q, k or v is cut into items of two vectors, columns j and
// j + D/2; a CTA takes all items of one node in `layers_per_cta` layers, kItems per thread at a
// time, and asks for the first kItems before it looks the node up, so that the reads (which
// depend on no position) overlap the chain tree, parents, slot, angles.
// kItems = 3 at four CTAs per SM; two at five where that saves a wave (see launch_tree_rope).
template <typename T, int kItems>
__global__ void __launch_bounds__(kThreads, kItems == 3 ? 4 : 5)
    tree_rope_kernel(const int32_t* node_offsets, const int32_t* parents, const int32_t* ctx_lens, int batch,
                     int n_total, int num_layers, int layers_per_cta, int D, int hq, int hkv, T* q, const T* k, const T* v,
                     T* k_cache, T* v_cache, int layer_begin, int page_size, int seq_capacity, int num_pages,
                     const int32_t* block_table, int max_pages, const __grid_constant__ RopeFreqs freqs,
                     int32_t* positions_out, int32_t* dev_status, GroupDivisor by_layer, GroupDivisor by_chunks) {
  __shared__ int par_s[kThreads];
  __shared__ float cos_s[kMaxRopeHalf], sin_s[kMaxRopeHalf];
  const int n = blockIdx.x, t = threadIdx.x;
  const int l0 = blockIdx.y * layers_per_cta;   // first layer of this CTA, relative to layer_begin
  const int layers = min(num_layers - l0, layers_per_cta);
  if (t == 0) grid_launch_dependents();   // the next grid may be placed now; it waits for this one
  grid_dependency_wait();   // the trees, q, k, v and the cache belong to the stream's previous work
  constexpr int V = Vec<T>::N;
  const int half = D / 2, chunks = half / V;
  const int heads = hq + 2 * hkv, per_layer = heads * chunks, items = layers * per_layer;
  // item e: its layer (relative), head (q heads, then k heads, then v heads) and first column
  auto place_of = [&](int e, int& lq, int& h, int& j) {
    lq = layers > 1 ? divide_by_group(e, by_layer) : 0;
    const int r = e - lq * per_layer;
    h = divide_by_group(r, by_chunks);
    j = (r - h * chunks) * V;
  };
  auto src_of = [&](int e) -> const T* {
    int lq, h, j;
    place_of(e, lq, h, j);
    const size_t node = (size_t)(l0 + lq) * n_total + n;
    if (h < hq) return q + (node * hq + h) * D + j;
    if (h < hq + hkv) return k + (node * hkv + (h - hq)) * D + j;
    return v + (node * hkv + (h - hq - hkv)) * D + j;
  };
  uint4 lo[kItems], hi[kItems];
  auto load_items = [&](int e0) {
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
      const int e = e0 + u * kThreads;
      if (e < items) {
        const T* src = src_of(e);
        lo[u] = *reinterpret_cast<const uint4*>(src);   // plain loads: q is also written
        hi[u] = *reinterpret_cast<const uint4*>(src + half);
      }
    }
  };
  load_items(t);
  Place at;
  if (!find_place(node_offsets, parents, ctx_lens, batch, n, page_size, seq_capacity, num_pages, block_table, max_pages,
                  l0 == 0, par_s, positions_out, dev_status, at))
    return;
  if (!at.fits) return;   // the node's slot is outside the cache: nothing is written
  make_table(freqs, at.pos, half, cos_s, sin_s);
  __syncthreads();
  const size_t layer_rows = page_size > 0 ? (size_t)num_pages * page_size : (size_t)batch * seq_capacity;
  for (int e0 = t;; load_items(e0)) {
#pragma unroll
    for (int u = 0; u < kItems; ++u) {
      const int e = e0 + u * kThreads;
      if (e >= items) continue;
      int lq, h, j;
      place_of(e, lq, h, j);
      uint4 a = lo[u], b = hi[u];
      if (h < hq + hkv) {
        const Vec<T> x = unpack16<T>(a), y = unpack16<T>(b);
        Vec<T> rx, ry;
#pragma unroll
        for (int i = 0; i < V; ++i) {
          const float c = cos_s[j + i], s = sin_s[j + i];
          rx.x[i] = x.x[i] * c - y.x[i] * s;
          ry.x[i] = x.x[i] * s + y.x[i] * c;
        }
        a = pack16(rx);
        b = pack16(ry);
      }
      T* dst;
      if (h < hq) {
        dst = q + (((size_t)(l0 + lq) * n_total + n) * hq + h) * D + j;
      } else {
        const size_t crow = (size_t)(layer_begin + l0 + lq) * layer_rows + at.row;
        dst = h < hq + hkv ? k_cache + (crow * hkv + (h - hq)) * D + j : v_cache + (crow * hkv + (h - hq - hkv)) * D + j;
      }
      *reinterpret_cast<uint4*>(dst) = a;
      *reinterpret_cast<uint4*>(dst + half) = b;
    }
    e0 += kItems * kThreads;
    if (e0 - t >= items) break;
  }
}

// Rows that are not 16-byte vectors: one element at a time, one CTA per (node, layer).
template <typename T>
__global__ void __launch_bounds__(kThreads)
    tree_rope_scalar_kernel(const int32_t* node_offsets, const int32_t* parents, const int32_t* ctx_lens, int batch,
                            int n_total, int D, int hq, int hkv, T* q, const T* k, const T* v, T* k_cache, T* v_cache,
                            int layer_begin, int page_size, int seq_capacity, int num_pages, const int32_t* block_table,
                            int max_pages, const __grid_constant__ RopeFreqs freqs, int32_t* positions_out,
                            int32_t* dev_status) {
  __shared__ int par_s[kThreads];
  __shared__ float cos_s[kMaxRopeHalf], sin_s[kMaxRopeHalf];
  const int n = blockIdx.x, t = threadIdx.x, lq = blockIdx.y;
  if (t == 0) grid_launch_dependents();   // the next grid may be placed now; it waits for this one
  grid_dependency_wait();   // the trees, q, k, v and the cache belong to the stream's previous work
  Place at;
  if (!find_place(node_offsets, parents, ctx_lens, batch, n, page_size, seq_capacity, num_pages, block_table, max_pages,
                  lq == 0, par_s, positions_out, dev_status, at))
    return;
  if (!at.fits) return;   // the node's slot is outside the cache: nothing is written
  const int half = D / 2;
  make_table(freqs, at.pos, half, cos_s, sin_s);
  __syncthreads();
  const size_t layer_rows = page_size > 0 ? (size_t)num_pages * page_size : (size_t)batch * seq_capacity;
  T* qn = q + ((size_t)lq * n_total + n) * hq * D;
  const T* kn = k + ((size_t)lq * n_total + n) * hkv * D;
  const T* vn = v + ((size_t)lq * n_total + n) * hkv * D;
  const size_t crow = ((size_t)(layer_begin + lq) * layer_rows + at.row) * hkv * D;
  for (int e = t; e < (hq + hkv) * half; e += kThreads) {
    const bool isq = e < hq * half;
    const int e2 = isq ? e : e - hq * half;
    const int h = e2 / half, j = e2 - h * half;
    const T* src = (isq ? (const T*)qn : kn) + (size_t)h * D;
    T* dst = isq ? qn + (size_t)h * D : k_cache + crow + (size_t)h * D;
    const float a = ld(src + j), bb = ld(src + j + half);
    const float c = cos_s[j], s = sin_s[j];
    st(dst + j, a * c - bb * s);
    st(dst + j + half, a * s + bb * c);
  }
  for (int e = t; e < hkv * D; e += kThreads) v_cache[crow + e] = vn[e];
}

}  // namespace tr

cudaError_t launch_tree_rope(const int32_t* node_offsets, const int32_t* parents, const int32_t* ctx_lens,
                             int batch, int n_total, bool bf16, int head_dim, int hq, int hkv, void* q, const void* k,
                             const void* v, void* k_cache, void* v_cache, int layer_begin, int num_layers,
                             int page_size, int seq_capacity, int num_pages, const int32_t* block_table, int max_pages,
                             const RopeFreqs& freqs, int32_t* positions_out, int32_t* dev_status, int sms,
                             cudaStream_t stream) {
  const auto al16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
  const bool aligned = al16(q) && al16(k) && al16(v) && al16(k_cache) && al16(v_cache);
  const int vec = bf16 ? 8 : 4;
  // (2^26 items a layer: the bound of the kernel's quotients)
  if (aligned && (head_dim / 2) % vec == 0 && ((int64_t)hq + 2 * (int64_t)hkv) * (head_dim / 2 / vec) < (1 << 26)) {
    // As many layers a CTA as fill three items of its threads; twice that over more than two waves of CTAs
    // (few heads' remainders, and half the look-ups: 32 layers of 128 nodes, 64 / 8 heads, bf16 31.1 -> 26.9
    // us, 8 layers of ~345 nodes 19.3 -> 17.3).  A grid just above one wave of four CTAs per SM runs with
    // five (~650 nodes, one layer, 32 / 8 heads 6.1 -> 4.7 us, 64 / 8 heads 7.2 -> 6.5); with five everywhere
    // the others lose 5 % (geometric mean over 249 sizes).
    const int chunks = head_dim / 2 / vec, per_layer = (hq + 2 * hkv) * chunks;
    auto layers_of = [&](int items) {
      const int l = items * tr::kThreads / per_layer;
      return l < 1 ? 1 : (l > num_layers ? num_layers : l);
    };
    auto ctas_of = [&](int l) { return (int64_t)n_total * ((num_layers + l - 1) / l); };
    int layers = layers_of(3);
    const int64_t ctas = ctas_of(layers), slots = 4 * (int64_t)sms;
    const bool five = ctas > slots && ctas_of(layers_of(2)) <= 5 * (int64_t)sms;
    if (five) layers = layers_of(2);
    if (ctas > 2 * slots) layers = layers_of(6);
    const dim3 grid(n_total, (num_layers + layers - 1) / layers);
#define PTD_ROPE_LAUNCH(T, ITEMS)                                                                                   \
  return launch_chained(tr::tree_rope_kernel<T, ITEMS>, grid, dim3(tr::kThreads), 0, stream, 0, node_offsets, parents,     \
                        ctx_lens, batch, n_total, num_layers, layers, head_dim, hq, hkv, static_cast<T*>(q),        \
                        static_cast<const T*>(k), static_cast<const T*>(v), static_cast<T*>(k_cache),               \
                        static_cast<T*>(v_cache), layer_begin, page_size, seq_capacity, num_pages, block_table,     \
                        max_pages, freqs, positions_out, dev_status, group_divisor(per_layer), group_divisor(chunks))
    if (bf16) {
      if (five) PTD_ROPE_LAUNCH(__nv_bfloat16, 2);
      PTD_ROPE_LAUNCH(__nv_bfloat16, 3);
    }
    if (five) PTD_ROPE_LAUNCH(float, 2);
    PTD_ROPE_LAUNCH(float, 3);
#undef PTD_ROPE_LAUNCH
  }
  const dim3 grid(n_total, num_layers);
#define PTD_ROPE_LAUNCH(T)                                                                                          \
  return launch_chained(tr::tree_rope_scalar_kernel<T>, grid, dim3(tr::kThreads), 0, stream, 0, node_offsets,       \
                        parents, ctx_lens, batch, n_total, head_dim, hq, hkv, static_cast<T*>(q),                   \
                        static_cast<const T*>(k), static_cast<const T*>(v), static_cast<T*>(k_cache),               \
                        static_cast<T*>(v_cache), layer_begin, page_size, seq_capacity, num_pages, block_table,     \
                        max_pages, freqs, positions_out, dev_status)
  if (bf16) PTD_ROPE_LAUNCH(__nv_bfloat16);
  PTD_ROPE_LAUNCH(float);
#undef PTD_ROPE_LAUNCH
}

}  // namespace ptd
