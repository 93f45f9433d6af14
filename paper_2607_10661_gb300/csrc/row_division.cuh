// Row number / query heads per KV head by a multiplication (internal; also compiled as plain C++).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define PTD_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define PTD_HOST_DEVICE inline
#endif

namespace ptd {

// m / group as floor(m mul / 2^(32 + shift)), mul = ceil(2^(32 + shift) / group) = (2^(32 + shift) + e) / group
// with 0 <= e < group: exact while m e < 2^(32 + shift).  Rows are below 128 * group, so shift 0 does below
// 5793 = sqrt(2^32 / 128) heads (from 5843 on it takes row 128 * group - 1 of most sizes for one of the next
// node); 12 does up to 2^16 heads, and mul still fits.  mul 0: group 1, the row itself.
struct GroupDivisor {
  uint32_t mul;
  uint32_t shift;
};

inline GroupDivisor group_divisor(int group) {
  if (group <= 1) return {0u, 0u};
  const uint32_t shift = group < 5793 ? 0u : 12u;
  return {(uint32_t)(((1ull << (32 + shift)) + (unsigned)group - 1) / (unsigned)group), shift};
}

PTD_HOST_DEVICE int divide_by_group(int m, GroupDivisor d) {
  if (d.mul == 0u) return m;
#ifdef __CUDA_ARCH__
  return (int)(__umulhi((uint32_t)m, d.mul) >> d.shift);
#else
  return (int)((((uint64_t)(uint32_t)m * d.mul) >> 32) >> d.shift);
#endif
}

}  // namespace ptd
