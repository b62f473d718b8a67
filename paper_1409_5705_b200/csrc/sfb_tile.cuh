// Device helpers that the tensor-core translation units share.
#pragma once

#include <algorithm>

#include "sfb_internal.h"
#include "sfb_ptx.cuh"

namespace sfb {

// Exchange of the partial tiles of a split contraction through the shared memory of the cluster's CTAs, in chunks of 32
// columns x 128 rows of fp32 (16 KB, the operand stages' memory, which nothing uses any more); a warp writes and reads its 32
// rows with the 16-byte pieces of a row swizzled.  Each of them finishes every parts-th chunk.  The sums are in rank order, so they do not depend on timing.
constexpr int kXchgCols = 32;
constexpr int kXchgBytes = 128 * kXchgCols * 4;
// the 16-byte piece j of a row of 32 fp32 values
__device__ __forceinline__ uint32_t slot_addr(uint32_t base, int row, int j) {
  return base + row * (kXchgCols * 4) + ((j ^ (row & 7)) << 4);
}
__device__ __forceinline__ uint32_t xchg_addr(uint8_t* smem, int c, int row, int j) {
  return slot_addr(ptx::smem_u32(smem) + c * kXchgBytes, row, j);
}
__device__ __forceinline__ void slot_put(uint32_t base, int row, const uint32_t (&acc)[32]) {
#pragma unroll
  for (int j = 0; j < 8; ++j)
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(slot_addr(base, row, j)), "r"(acc[4 * j]), "r"(acc[4 * j + 1]),
                 "r"(acc[4 * j + 2]), "r"(acc[4 * j + 3]) : "memory");
}
__device__ __forceinline__ void xchg_put(uint8_t* smem, int c, int row, const uint32_t (&acc)[32]) {
  slot_put(ptx::smem_u32(smem) + c * kXchgBytes, row, acc);
}
__device__ __forceinline__ void xchg_sum(uint8_t* smem, int c, int row, int parts, uint32_t (&acc)[32]) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t at = xchg_addr(smem, c, row, j);
    float4 s = ptx::ld_cluster_f4(at, 0);
    for (int g = 1; g < parts; ++g) {
      const float4 v = ptx::ld_cluster_f4(at, g);
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    acc[4 * j] = __float_as_uint(s.x); acc[4 * j + 1] = __float_as_uint(s.y);
    acc[4 * j + 2] = __float_as_uint(s.z); acc[4 * j + 3] = __float_as_uint(s.w);
  }
}

__device__ __forceinline__ float soft_threshold(float w, float t) {
  const float a = fabsf(w) - t;
  return a > 0.f ? copysignf(a, w) : 0.f;
}

// Blocks of a grid-stride kernel over `items`, at most 16 per SM.
inline unsigned grid1d(int64_t items, int per_block) {
  const int64_t g = (items + per_block - 1) / per_block;
  return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(g, static_cast<int64_t>(sm_count()) * 16)));
}

}  // namespace sfb
