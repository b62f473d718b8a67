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

// What a pair of CTAs computes of a product's tiles, in its order: whole tiles (the `whole` first of them, a multiple of the pairs;
// all when nothing is cut), then, of the others, whose k-blocks are shared out evenly, the part of a tile that another pair
// completes and the tiles that it completes (the one it completes for others last).  k-blocks [k0, k1) of each.
struct Segment { int tile, k0, k1; };
struct Segments {
  int pair, pairs, kseg, whole, own, t0, n;      // own: whole tiles of this pair ahead of its part of the others
  int64_t units, beg, end;                       // k-blocks of the tiles that are shared out; of this pair
  bool cut, leaves;
  __device__ Segments(int kseg_, bool cut_, int whole_, int ntiles, int pair_, int pairs_)
      : pair(pair_), pairs(pairs_), kseg(kseg_), whole(whole_), units(static_cast<int64_t>(ntiles - whole_) * kseg_), cut(cut_) {
    own = whole / pairs;
    beg = units * pair / pairs;
    end = units * (pair + 1) / pairs;
    t0 = static_cast<int>(beg / kseg);
    leaves = cut && end > beg && end % kseg != 0;
    n = cut ? own + (end > beg ? static_cast<int>((end - 1) / kseg) - t0 + 1 : 0) : pair < ntiles ? (ntiles - 1 - pair) / pairs + 1 : 0;
  }
  __device__ Segment get(int i) const {
    if (!cut || i < own) return Segment{pair + i * pairs, 0, kseg};
    i -= own;
    if (leaves) {
      const int last = t0 + n - own - 1;
      const int64_t first = static_cast<int64_t>(last) * kseg;
      if (i == 0) return Segment{whole + last, static_cast<int>((beg > first ? beg : first) - first), static_cast<int>(end - first)};
      --i;
    }
    const int mine = n - own - (leaves ? 1 : 0), t = i < mine - 1 ? t0 + 1 + i : t0;
    const int64_t first = static_cast<int64_t>(t) * kseg;
    return Segment{whole + t, beg > first ? static_cast<int>(beg - first) : 0, kseg};
  }
  // of the pairs that have a part of the tile which this one completes
  __device__ int first_part(const Segment& sg) const {
    if (sg.k0 == 0) return pair;
    const int64_t first = static_cast<int64_t>(sg.tile - whole) * kseg;
    int j = pair - 1;
    while (j > 0 && units * j / pairs > first) --j;
    return j;
  }
};

__device__ __forceinline__ float soft_threshold(float w, float t) {
  const float a = fabsf(w) - t;
  return a > 0.f ? copysignf(a, w) : 0.f;
}

// Blocks of a grid-stride kernel over `items`, at most 16 per SM.
inline unsigned grid1d(int64_t items, int per_block) {
  const int64_t g = (items + per_block - 1) / per_block;
  return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(g, static_cast<int64_t>(sm_count()) * 16)));
}

// Opts a kernel of CTA pairs (thread blocks of a fixed cluster of two) into `smem` bytes; at most *max_pairs of them at a time.
template <typename Kernel>
cudaError_t prepare_pair_kernel(Kernel kernel, int threads, int smem, int* max_pairs) {
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(2, 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 2; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  e = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg);
  if (e != cudaSuccess) return e;
  *max_pairs = std::min(*max_pairs, n);
  return cudaSuccess;
}

}  // namespace sfb
