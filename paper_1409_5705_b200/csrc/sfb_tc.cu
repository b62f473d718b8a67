// Tensor-core (bf16 operand) path of the SFB step on sm_100a: sufficient-factor computation for multiclass
// logistic regression (Sections 1 and 2: u = softmax(W x) - onehot(y), v = x) and the operand packing of the
// update product.  The update product itself is in sfb_update.cu, the products of (hi | lo) pairs in sfb_split.cu.
//
// Forward product (of 65 to 128 samples, of others where logits_kernel does not prefer those of sfb_forward.cu, and of tf32 words): one
// persistent, warp-specialised kernel computes  Z (K x rows) = X (K x cols) * W^T  with bf16
// operands staged by TMA into 128-byte-swizzled shared memory, tcgen05.mma accumulating in TMEM (two 128 x 256
// fp32 accumulators, so the epilogue of one tile overlaps the main loop of the next).  The epilogue stores Z as
// fp32 and, per (sample, 256-row block), the softmax partials (max, sum of exp).
// Roles: warp 0 TMA producer, warp 1 MMA issuer (and TMEM owner), warps 2-5 epilogue (one TMEM lane quarter each).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <new>

#include "sfb_ptx.cuh"
#include "sfb_tc.h"
#include "sfb_tile.cuh"

namespace sfb {
namespace {

using namespace ptx;

constexpr int BM = 128, BN = 256, BK = 64, UMMA_K = 16;
constexpr int kBytesA = BM * BK * 2, kBytesB = BN * BK * 2;
constexpr int kChunk = 32;                 // accumulator columns handled per epilogue step
constexpr int kSlotBytes = 32 * kChunk * 4;  // one warp's 32 rows x 32 fp32 columns
constexpr int kTmemCols = 512;
constexpr int S = 4;                      // operand pipeline stages of a full-width tile (narrower ones: see forward_stages)
constexpr int S_MAX = 8;
constexpr int R = 2;                      // epilogue ring slots per warp
constexpr int kEpiWarps = 4;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kBars = 2 * S_MAX + 4;
constexpr int kSmem = S * (kBytesA + kBytesB) + kEpiWarps * R * kSlotBytes + kBars * 8 + 16 + 1024;

struct TcParams {
  int32_t M, N, Kc;            // extents of the product: samples, output columns, contraction
  int32_t m_off;               // first sample handled by this launch (per-worker slices)
  int32_t tilesM, tilesN;
  int32_t a_rows;              // rows of A per box (fewer than 128 for a slice of few samples; the rest of a
                               // tile's samples are then never stored)
  int32_t stages;              // forward_kernel: stages of the operand ring
  int32_t pw;                  // columns per softmax partial, a divisor of bn
  int32_t bn;                  // columns per tile, at most BN, a multiple of 32 (chosen so that the tiles fill the SMs)
  // The contraction runs over nseg segments of kseg k-blocks; segment s reads A from column a_off<s> and B from
  // column b_off<s> of their tensors: one segment is the plain product, three segments over [big | small] tf32 operand
  // halves form big*small + small*big + big*big.  (Scalars: an indexed array would send the whole parameter block to local
  // memory.)
  int32_t nseg, kseg;
  int32_t a_off0, a_off1, a_off2, b_off0, b_off1, b_off2;
  float2* part;                // [N / pw][part_ld] (max, sum exp) per sample and pw rows of W
  int64_t part_ld;
  int32_t kparts;              // the contraction of a tile is cut over a cluster of this many CTAs (1: persistent CTAs)
  uint32_t* status;
};

// Tiles are numbered with the sample block fastest: consecutive tiles (which run on different SMs at the same
// time) share one block of W, which therefore stays hot in L2 while all K samples are swept past it.
__device__ __forceinline__ void tile_coords(const TcParams& p, int tile, int& m0, int& n0) {
  const int tm = tile % p.tilesM, tn = tile / p.tilesM;
  m0 = p.m_off + tm * BM;
  n0 = tn * p.bn;
}

// TF32: the operands are 32-bit words read as tf32 (a k-block of 128 bytes is then 32 elements and one MMA contracts
// 8 of them); everything else -- stages, descriptors, epilogues -- is the same.
template <bool TF32>
__global__ void __launch_bounds__(kThreads, 1)
forward_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmC, const TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int ST = p.stages;
  const int stage_bytes = kBytesA + p.bn * BK * 2;       // A, then B: all multiples of 1024
  uint8_t* sRing = smem + S * (kBytesA + kBytesB);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sRing + 4 * R * kSlotBytes);
  uint64_t* full = bars;
  uint64_t* empty = bars + S_MAX;
  uint64_t* tfull = bars + 2 * S_MAX;
  uint64_t* tempty = bars + 2 * S_MAX + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kBars);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int ntiles = p.tilesM * p.tilesN;
  // With a split contraction a CTA has one tile and the k-blocks [kbeg, kend) of its nseg * kseg; else all of them and the
  // tiles blockIdx.x, blockIdx.x + gridDim.x, ...
  const int split = p.kparts, part = split > 1 ? static_cast<int>(blockIdx.x) % split : 0;
  const int tile0 = static_cast<int>(blockIdx.x) / split, tile_step = split > 1 ? ntiles : static_cast<int>(gridDim.x);
  const int kall = p.nseg * p.kseg;
  const int kbeg = part * kall / split, kend = (part + 1) * kall / split;
  pdl_launch_dependents();

  if (threadIdx.x == 0) {
    for (int i = 0; i < ST; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], 4); }
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&tmA); prefetch_tmap(&tmB); prefetch_tmap(&tmC);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, kTmemCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    // A (the K samples) is the small operand every tile re-reads: pinned in L2.
    const uint64_t pol_keep = policy_evict_last();
    uint32_t s = 0, ph = 0;
    bool ok = true;
    for (int tile = tile0; tile < ntiles && ok; tile += tile_step) {
      int m0, n0;
      tile_coords(p, tile, m0, n0);
      for (int seg = 0; seg < p.nseg && ok; ++seg) {
        const int xa0 = seg == 0 ? p.a_off0 : seg == 1 ? p.a_off1 : p.a_off2;
        const int xb0 = seg == 0 ? p.b_off0 : seg == 1 ? p.b_off1 : p.b_off2;
        const int kl1 = min(p.kseg, kend - seg * p.kseg);
        for (int kl = max(0, kbeg - seg * p.kseg); kl < kl1; ++kl) {
          if (!mbar_wait_warp(&empty[s], ph ^ 1, abort_flag)) { ok = false; break; }
          if (elect_one()) {
            uint8_t* st = smem + s * stage_bytes;
            mbar_expect_tx(&full[s], (p.a_rows + p.bn) * BK * 2);
            tma_load_2d_hint(st, &tmA, xa0 + kl * (TF32 ? BK / 2 : BK), m0, &full[s], pol_keep);
            tma_load_2d(st + kBytesA, &tmB, xb0 + kl * (TF32 ? BK / 2 : BK), n0, &full[s]);
          }
          if (++s == static_cast<uint32_t>(ST)) { s = 0; ph ^= 1; }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const uint32_t idesc = TF32 ? umma_idesc_tf32(BM, p.bn) : umma_idesc_bf16(BM, p.bn);
    uint32_t s = 0, ph = 0, tl = 0;
    bool ok = true;
    for (int tile = tile0; tile < ntiles && ok; tile += tile_step, ++tl) {
      const uint32_t a = tl & 1, aph = (tl >> 1) & 1;
      if (!mbar_wait_warp(&tempty[a], aph ^ 1, abort_flag)) { ok = false; break; }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + a * BN;
      for (int kb = 0; kb < kend - kbeg; ++kb) {
        if (!mbar_wait_warp(&full[s], ph, abort_flag)) { ok = false; break; }
        tc_fence_after();
        if (elect_one()) {
          const uint64_t da = umma_desc_k128(smem_u32(smem + s * stage_bytes));
          const uint64_t db = umma_desc_k128(smem_u32(smem + s * stage_bytes + kBytesA));
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k) {          // four MMAs of 32 bytes of contraction each, either kind
            const uint64_t adv = static_cast<uint64_t>(k * UMMA_K * 2 / 16);
            if (TF32) umma_tf32(d_tmem, da + adv, db + adv, idesc, (kb | k) != 0 ? 1u : 0u);
            else umma_bf16(d_tmem, da + adv, db + adv, idesc, (kb | k) != 0 ? 1u : 0u);
          }
          umma_commit(&empty[s]);          // the stage is free once these MMAs have read it
        }
        if (++s == static_cast<uint32_t>(ST)) { s = 0; ph ^= 1; }
      }
      if (ok && elect_one()) umma_commit(&tfull[a]);    // the accumulator is complete once every MMA of the tile is
    }
  } else {
    // ---------------- epilogue: warps 2..5, TMEM lane quarter q ----------------
    const int q = warp & 3;
    uint8_t* ring = sRing + q * R * kSlotBytes;
    const int my_tiles = tile0 < ntiles ? (ntiles - 1 - tile0) / tile_step + 1 : 0;
    bool ok = true;
    // The fp32 result goes out through the ring by TMA; the epilogue keeps a running (max, sum exp) per sample.
    uint32_t gs = 0;                       // stores issued so far: consecutive stores alternate ring slots
    float mx = -INFINITY, sum = 0.f;
    auto finish = [&](uint32_t (&acc)[32], int m0, int n0, int c) {
      uint8_t* sl = ring + (gs % R) * kSlotBytes;
      const int col0 = n0 + c * kChunk, row = m0 + q * 32 + lane;
      if (col0 < p.N) {
        float cm = -INFINITY;
#pragma unroll
        for (int j = 0; j < 32; ++j)
          if (col0 + j < p.N) cm = fmaxf(cm, __uint_as_float(acc[j]));
        const float nm = fmaxf(mx, cm);
        float cs = 0.f;
#pragma unroll
        for (int j = 0; j < 32; ++j)
          if (col0 + j < p.N) cs += __expf(__uint_as_float(acc[j]) - nm);
        sum = sum * __expf(mx - nm) + cs;
        mx = nm;
        if (lane == 0) tma_wait_group_read<R - 1>();   // the store that last used this slot has read it
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 8; ++j)
          *reinterpret_cast<uint4*>(sl + lane * 128 + ((j ^ (lane & 7)) << 4)) =
              make_uint4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          tma_store_2d(&tmC, sl, col0, m0 + q * 32);
          tma_commit_group();
        }
        ++gs;
      }
      if (((c + 1) * kChunk) % p.pw == 0) {      // the end of a group of pw columns
        const int grp = (n0 + (c + 1) * kChunk) / p.pw - 1;
        if (grp * p.pw < p.N && row < p.M) p.part[static_cast<int64_t>(grp) * p.part_ld + row] = make_float2(mx, sum);
        mx = -INFINITY;
        sum = 0.f;
      }
    };
    for (int tl = 0; tl < my_tiles && ok; ++tl) {
      int m0, n0;
      tile_coords(p, tile0 + tl * tile_step, m0, n0);
      const uint32_t a = tl & 1, aph = (tl >> 1) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(&tfull[a], aph, abort_flag))) { ok = false; break; }
      tc_fence_after();
      for (int c = 0; c < p.bn / kChunk; ++c) {
        uint32_t acc[32];
        tmem_ld_32x32(tmem_base + (static_cast<uint32_t>(q * 32) << 16) + a * BN + c * kChunk, acc);
        tmem_ld_wait();
        if (split > 1) xchg_put(smem, c, q * 32 + lane, acc);
        else finish(acc, m0, n0, c);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty[a]);
    }
    if (split > 1) {
      __syncwarp();
      cluster_arrive();
      cluster_wait();
      int m0, n0;
      tile_coords(p, tile0, m0, n0);
      for (int c = part; c < p.bn / kChunk && ok; c += split) {        // (pw is 32: a group is a chunk)
        uint32_t acc[32];
        xchg_sum(smem, c, q * 32 + lane, split, acc);
        finish(acc, m0, n0, c);
      }
    }
    if (lane == 0) tma_wait_group<0>();
  }
  if (split > 1) {
    __syncwarp();
    if (warp < 2) { cluster_arrive(); cluster_wait(); }                // (the epilogue warps have been there)
    cluster_arrive();                                                  // no CTA leaves while a peer still reads its part
    cluster_wait();
  }

  // ---------------- teardown ----------------
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // A wait ran out: report it, give copies in flight a bounded time to land, then release TMEM.
    if (threadIdx.x == 0) atomicOr(p.status, SFB_STATUS_TIMEOUT);
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, kTmemCols); }
}

// ---------------------------------------------------------------------------------------------------------
// Bandwidth-bound companions of the tensor-core products
// ---------------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&v);
}

// fp32 [rows x cols] -> bf16 [rows x ld] (row-major), 8 elements per thread; cols is a multiple of 4.
__global__ void __launch_bounds__(256) convert_rows_kernel(const float* __restrict__ src, int64_t rows, int64_t cols,
                                                           __nv_bfloat16* __restrict__ dst, int64_t ld) {
  pdl_launch_dependents();
  pdl_wait(src, dst);
  const int64_t quads = cols / 4;
  const int64_t total = rows * quads;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total; i += stride) {
    const int64_t r = i / quads, qd = i % quads;
    const float4 v = *reinterpret_cast<const float4*>(src + r * cols + qd * 4);
    *reinterpret_cast<uint2*>(dst + r * ld + qd * 4) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
  }
}

// Pack of the inputs of n samples starting at pair index off (Section 2.1: v = a_i):
//   Xb[off + i][:]  = bf16(x_i), the operand of the forward product and of the update (which contracts over the samples and
//                     takes it as an MN-major operand),   Xf (may be null) = the fp32 sample for the label rows,   labels.
// The label-row slots of the classes that these samples had in the step before are cleared.
// One read of X, 6 bytes written per value, 2 without Xf; bound by HBM (1,024 x 20,000: 33 us with a transposed copy beside
// it, 28 without, 20 without Xf).
__global__ void __launch_bounds__(256) pack_mlr_kernel(const float* __restrict__ X, int64_t n, int64_t cols,
                                                       __nv_bfloat16* __restrict__ Xb, int64_t ldx, int64_t off,
                                                       float* __restrict__ Xf, const int32_t* labels, int32_t* labels_out,
                                                       int32_t* __restrict__ slot, int64_t rows, const Stamp stamp) {
  pdl_launch_dependents();
  pdl_wait(X, Xb, Xf, slot);
  stamp_begin(stamp);
  const uint32_t quads = static_cast<uint32_t>(cols / 4);
  const int64_t total = n * quads, stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t t0 = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  for (int64_t q = t0; q < total; q += stride) {
    const int64_t i = q / quads, c = (q - i * quads) * 4;
    const float4 v = *reinterpret_cast<const float4*>(X + i * cols + c);
    *reinterpret_cast<uint2*>(Xb + (off + i) * ldx + c) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
    if (Xf) *reinterpret_cast<float4*>(Xf + (off + i) * cols + c) = v;
  }
  for (int64_t i = t0; i < n; i += stride) {
    const int32_t old = labels_out[off + i];
    if (old >= 0 && old < rows) slot[old] = kNoSlot;
    labels_out[off + i] = labels[i];
  }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// One warp per sample: merge the per-block (max, sum exp) partials into log sum exp; loss = lse - z_y;
// coef = 1 - p_y, the size of the label entry of u, kept in fp32.
__global__ void __launch_bounds__(256) mlr_lse_kernel(const float2* __restrict__ part, int64_t part_ld, int nblocks,
                                                      const float* __restrict__ Z, int64_t ldz, int64_t rows,
                                                      const int32_t* __restrict__ labels, int64_t off, int64_t n,
                                                      float* __restrict__ lse, float* __restrict__ loss,
                                                      float* __restrict__ coef, int32_t* __restrict__ slot,
                                                      uint32_t* status) {
  pdl_launch_dependents();
  pdl_wait(part, Z, labels, lse, loss, coef, slot);
  const int64_t i = static_cast<int64_t>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  if (i >= n) return;
  const int lane = threadIdx.x & 31;
  const int64_t s = off + i;
  float m = -INFINITY;
  for (int b = lane; b < nblocks; b += 32) m = fmaxf(m, part[static_cast<int64_t>(b) * part_ld + s].x);
  m = warp_max(m);
  float sum = 0.f;
  for (int b = lane; b < nblocks; b += 32) {
    const float2 v = part[static_cast<int64_t>(b) * part_ld + s];
    sum += v.y * __expf(v.x - m);
  }
  sum = warp_sum(sum);
  if (lane == 0) {
    const float l = m + logf(sum);
    lse[s] = l;
    const int32_t y = labels[i];
    const bool okl = y >= 0 && y < rows;
    if (!okl) atomicOr(status, SFB_STATUS_LABEL_RANGE);
    const float zy = okl ? Z[s * ldz + y] : 0.f;
    loss[s] = okl ? l - zy : 0.f;
    coef[s] = okl ? -expm1f(zy - l) : 0.f;        // 1 - p_y = -u_y, formed in fp32 without cancellation
    if (okl && slot) atomicMin(&slot[y], static_cast<int32_t>(s));      // the first sample of its class (see label_delta)
  }
}

// The label entries of the K factors, u_iy = p_iy - 1, which the bf16 operand leaves out (it holds 0 there).  Per class that
// the mini-batch has, in fp32 and in ascending sample order (no atomics: one order):
//     dL[f] = sum_{i : y_i = y} (1 - p_iy) x_i,   W[y] <- W[y] + step * dL[f],   f = slot[y] the class's first sample,
// and the bf16 copy of the row with it; dL is kept for a repeated update.  Work units (first sample, 1024 columns) are dealt
// to nblk blocks; the last block also forms the mean loss.  A popular class (130 of 1,024 samples under Zipf labels) is what
// the kernel waits for, so a unit has eight samples in flight.  It shares a launch with the probabilities where it can.
// (Adding dL in the epilogue of the update, which has the row on chip, cost that kernel 100 us at 10,000 x 20,000: its W
// stream is bound by latency, and any work between a tile's arrival and its departure adds to it.)
// Eight loads in one statement: issued together, whatever the compiler thinks of the registers.
__device__ __forceinline__ void load8(float4 (&x)[8], const float* const (&p)[8]) {
  asm volatile(
      "ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%32];\n\tld.global.nc.v4.f32 {%4, %5, %6, %7}, [%33];\n\t"
      "ld.global.nc.v4.f32 {%8, %9, %10, %11}, [%34];\n\tld.global.nc.v4.f32 {%12, %13, %14, %15}, [%35];\n\t"
      "ld.global.nc.v4.f32 {%16, %17, %18, %19}, [%36];\n\tld.global.nc.v4.f32 {%20, %21, %22, %23}, [%37];\n\t"
      "ld.global.nc.v4.f32 {%24, %25, %26, %27}, [%38];\n\tld.global.nc.v4.f32 {%28, %29, %30, %31}, [%39];"
      : "=&f"(x[0].x), "=&f"(x[0].y), "=&f"(x[0].z), "=&f"(x[0].w), "=&f"(x[1].x), "=&f"(x[1].y), "=&f"(x[1].z), "=&f"(x[1].w),
        "=&f"(x[2].x), "=&f"(x[2].y), "=&f"(x[2].z), "=&f"(x[2].w), "=&f"(x[3].x), "=&f"(x[3].y), "=&f"(x[3].z), "=&f"(x[3].w),
        "=&f"(x[4].x), "=&f"(x[4].y), "=&f"(x[4].z), "=&f"(x[4].w), "=&f"(x[5].x), "=&f"(x[5].y), "=&f"(x[5].z), "=&f"(x[5].w),
        "=&f"(x[6].x), "=&f"(x[6].y), "=&f"(x[6].z), "=&f"(x[6].w), "=&f"(x[7].x), "=&f"(x[7].y), "=&f"(x[7].z), "=&f"(x[7].w)
      : "l"(p[0]), "l"(p[1]), "l"(p[2]), "l"(p[3]), "l"(p[4]), "l"(p[5]), "l"(p[6]), "l"(p[7]));
}
constexpr int kLabelList = 1024, kLabelCols = 1024, kLabelBatch = 8;
struct LabelArgs {
  const float* X;              // the K samples, fp32
  const int32_t* labels;
  const int32_t* slot;
  const float* coef;
  float* dL;                   // [K x cols]
  float* W;                    // [rows x cols]
  __nv_bfloat16* Wb;           // its operand copy, row pitch ldw
  int64_t ldw;
  float step;
  int32_t again;               // dL is there: add it to W once more
  const float* loss;
  float* loss_mean;
  int64_t rows, cols;
  int32_t K;
};
__device__ __forceinline__ void label_delta(const LabelArgs& a, int blk, int nblk) {
  __shared__ int nunits;
  __shared__ int32_t unit[256];
  __shared__ int32_t list[kLabelList];
  __shared__ float lcoef[kLabelList];
  __shared__ int warp_tot[8];
  __shared__ float lsum[8];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  if (blk == nblk - 1) {
    float v = 0.f;
    for (int i = t; i < a.K; i += 256) v += a.loss[i];
    v = warp_sum(v);
    if (lane == 0) lsum[wid] = v;
    __syncthreads();
    if (t == 0) {
      float m = 0.f;
      for (int w = 0; w < 8; ++w) m += lsum[w];
      *a.loss_mean = m / static_cast<float>(a.K);
    }
  }
  const int64_t chunks = (a.cols + kLabelCols - 1) / kLabelCols, total = a.K * chunks;
  for (int64_t base = 0; base * nblk < total; base += 256) {
    if (t == 0) nunits = 0;
    __syncthreads();
    const int64_t u = (base + t) * nblk + blk;
    if (u < total) {
      const int32_t i = static_cast<int32_t>(u / chunks), y = a.labels[i];
      if (y >= 0 && y < a.rows && a.slot[y] == i) unit[atomicAdd(&nunits, 1)] = t;
    }
    __syncthreads();
    const int todo = nunits;
    for (int k = 0; k < todo; ++k) {
      const int64_t v = (base + unit[k]) * nblk + blk;
      const int32_t i = static_cast<int32_t>(v / chunks), y = a.labels[i];
      const int64_t c = (v % chunks) * kLabelCols + 4 * t;
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
      float* d = a.dL + static_cast<int64_t>(i) * a.cols + c;
      float* wp = a.W + static_cast<int64_t>(y) * a.cols + c;
      float4 w = s;
      if (c < a.cols) {
        w = *reinterpret_cast<const float4*>(wp);
        if (a.again) s = *reinterpret_cast<const float4*>(d);
      }
      for (int j0 = a.again ? a.K : i; j0 < a.K; j0 += kLabelList) {
        // ordered compaction of the class's samples in [j0, j0 + kLabelList): a warp looks at 128 labels
        unsigned hit[4];
        int mine = 0;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const int j = j0 + wid * 128 + o * 32 + lane;
          hit[o] = __ballot_sync(0xffffffffu, j < a.K && a.labels[j] == y);
          mine += __popc(hit[o]);
        }
        if (lane == 0) warp_tot[wid] = mine;
        __syncthreads();
        int pre = 0, n = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
          if (w < wid) pre += warp_tot[w];
          n += warp_tot[w];
        }
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          if ((hit[o] >> lane) & 1u) {
            const int at = pre + __popc(hit[o] & ((1u << lane) - 1)), j = j0 + wid * 128 + o * 32 + lane;
            list[at] = j;
            lcoef[at] = a.coef[j];
          }
          pre += __popc(hit[o]);
        }
        __syncthreads();
        if (c < a.cols)
          for (int q0 = 0; q0 < n; q0 += kLabelBatch) {
            float4 x[kLabelBatch];
            const float* xp[kLabelBatch];
#pragma unroll
            for (int e = 0; e < kLabelBatch; ++e) xp[e] = a.X + static_cast<int64_t>(list[min(q0 + e, n - 1)]) * a.cols + c;
            load8(x, xp);
#pragma unroll
            for (int e = 0; e < kLabelBatch; ++e) {
              const float cf = q0 + e < n ? lcoef[q0 + e] : 0.f;
              s.x = fmaf(cf, x[e].x, s.x); s.y = fmaf(cf, x[e].y, s.y);
              s.z = fmaf(cf, x[e].z, s.z); s.w = fmaf(cf, x[e].w, s.w);
            }
          }
        __syncthreads();
      }
      if (c < a.cols) {
        if (!a.again) *reinterpret_cast<float4*>(d) = s;
        w.x = fmaf(a.step, s.x, w.x); w.y = fmaf(a.step, s.y, w.y); w.z = fmaf(a.step, s.z, w.z); w.w = fmaf(a.step, s.w, w.w);
        *reinterpret_cast<float4*>(wp) = w;
        *reinterpret_cast<uint2*>(a.Wb + static_cast<int64_t>(y) * a.ldw + c) = make_uint2(pack_bf16(w.x, w.y), pack_bf16(w.z, w.w));
      }
    }
    __syncthreads();
  }
}
__global__ void __launch_bounds__(256) label_delta_kernel(const LabelArgs a) {
  pdl_launch_dependents();
  pdl_wait();
  label_delta(a, blockIdx.x, gridDim.x);
}
// slot[y] = the smallest index of a sample of class y, for factors that came in several calls.
__global__ void __launch_bounds__(256) label_slots_kernel(const int32_t* __restrict__ labels, int32_t K, int64_t rows,
                                                          int32_t* __restrict__ slot, const Stamp stamp) {
  pdl_launch_dependents();
  pdl_wait(labels, slot);
  stamp_begin(stamp);
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= K) return;
  const int32_t y = labels[i];
  if (y >= 0 && y < rows) atomicMin(&slot[y], i);
}

// Row-sharded form, first half: one warp per sample merges the forward's per-block (max, sum exp) partials over the
// shard's rows into the shard's partial (m_i, s_i, zy_i, has_i); zy_i = z_{i,y_i} and has_i = 1 when the shard owns
// class y_i (labels are global ids; the shard holds rows [row_off, row_off + rows)).
__global__ void __launch_bounds__(256) mlr_shard_partials_tc_kernel(const float2* __restrict__ part, int64_t part_ld, int nblocks,
                                                                    const float* __restrict__ Z, int64_t ldz, int64_t rows,
                                                                    const int32_t* __restrict__ labels, int64_t row_off,
                                                                    int64_t n, float4* __restrict__ out) {
  pdl_launch_dependents();
  pdl_wait(part, Z, labels, out);
  const int64_t i = static_cast<int64_t>(blockIdx.x) * 8 + (threadIdx.x >> 5);
  if (i >= n) return;
  const int lane = threadIdx.x & 31;
  float m = -INFINITY;
  for (int b = lane; b < nblocks; b += 32) m = fmaxf(m, part[static_cast<int64_t>(b) * part_ld + i].x);
  m = warp_max(m);
  float sum = 0.f;
  for (int b = lane; b < nblocks; b += 32) {
    const float2 v = part[static_cast<int64_t>(b) * part_ld + i];
    sum += v.y * __expf(v.x - m);
  }
  sum = warp_sum(sum);
  if (lane == 0) {
    const int64_t yl = static_cast<int64_t>(labels[i]) - row_off;
    const bool mine = yl >= 0 && yl < rows;
    out[i] = make_float4(m, sum, mine ? Z[i * ldz + yl] : 0.f, mine ? 1.f : 0.f);
  }
}

// Second half, one thread per sample: merge the partials of all shards ([shards][n], shard order) into the global
// log-partition; loss = lse - z_y; coef = 1 - p_y for the samples whose class this shard owns (0 otherwise); the class
// ids are rewritten as row indices of this shard (-1: another shard's row).  A class no shard owns sets the status bit.
__global__ void __launch_bounds__(256) mlr_shard_finish_tc_kernel(const float4* __restrict__ parts, int shards, int64_t n,
                                                                  int64_t rows, int64_t row_off,
                                                                  int32_t* __restrict__ labels,
                                                                  float* __restrict__ lse, float* __restrict__ loss,
                                                                  float* __restrict__ coef, uint32_t* status) {
  pdl_launch_dependents();
  pdl_wait(parts, labels, lse, loss, coef);
  const int64_t i = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x;
  if (i >= n) return;
  float M = -INFINITY;
  for (int g = 0; g < shards; ++g) M = fmaxf(M, parts[static_cast<int64_t>(g) * n + i].x);
  float S = 0.f, zy = 0.f, has = 0.f;
  for (int g = 0; g < shards; ++g) {
    const float4 v = parts[static_cast<int64_t>(g) * n + i];
    S += v.y * expf(v.x - M);
    zy += v.z;
    has += v.w;
  }
  const float l = M + logf(S);
  const bool ok = has > 0.5f;
  if (!ok) atomicOr(status, SFB_STATUS_LABEL_RANGE);
  const int64_t yl = static_cast<int64_t>(labels[i]) - row_off;
  const bool mine = ok && yl >= 0 && yl < rows;
  lse[i] = l;
  loss[i] = ok ? l - zy : 0.f;
  coef[i] = mine ? -expm1f(zy - l) : 0.f;
  labels[i] = mine ? static_cast<int32_t>(yl) : -1;
}

// P[off + i][r] = bf16( exp(z_ir - lse_i) ) for r != y_i and 0 for r = y_i, from the logits Z (row pitch a multiple of 32).
// The factor is u_i = p_i - onehot(y_i); its label entry u_iy = p_iy - 1 is left out of the bf16 operand and applied to W in
// fp32 (label_delta), because bf16 cannot hold it when p_iy is close to 1 (spacing 2^-8 next to 1) and a rounded p_iy
// with an exact -1 would not cancel.  Eight values per thread; 6 bytes per value, bound by HBM.
// PLAIN: the values of Z themselves instead of exp(z - lse) (factors received from elsewhere), with the same zero at the label
// entry.
// With K label entries to sum (lab.K > 0) the first lab_blocks blocks do that instead, see label_delta.
template <bool PLAIN>
__global__ void __launch_bounds__(256) mlr_emit_p_kernel(const float* __restrict__ Z, int64_t ldz, int64_t rows,
                                                         const float* __restrict__ lse, int64_t off, int64_t n,
                                                         const int32_t* __restrict__ labels, __nv_bfloat16* __restrict__ P,
                                                         int64_t ldp, int lab_blocks, const LabelArgs lab) {
  pdl_launch_dependents();
  pdl_wait(Z, lse, labels, P);
  if (static_cast<int>(blockIdx.x) < lab_blocks) return label_delta(lab, blockIdx.x, lab_blocks);
  const uint32_t octs = static_cast<uint32_t>((rows + 7) / 8);
  const int64_t total = n * octs, stride = static_cast<int64_t>(gridDim.x - lab_blocks) * blockDim.x;
  for (int64_t q = (blockIdx.x - lab_blocks) * static_cast<int64_t>(blockDim.x) + threadIdx.x; q < total; q += stride) {
    const int64_t i = q / octs, r = (q - i * octs) * 8, s = off + i;
    const float l = PLAIN ? 0.f : lse[s];
    const int64_t yrel = static_cast<int64_t>(labels[i]) - r;           // label row relative to this group of eight
    const float4 a = *reinterpret_cast<const float4*>(Z + s * ldz + r), b = *reinterpret_cast<const float4*>(Z + s * ldz + r + 4);
    float z[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int k = 0; k < 8; ++k) z[k] = k == yrel ? 0.f : (PLAIN ? z[k] : __expf(z[k] - l));
    *reinterpret_cast<uint4*>(P + s * ldp + r) =
        make_uint4(pack_bf16(z[0], z[1]), pack_bf16(z[2], z[3]), pack_bf16(z[4], z[5]), pack_bf16(z[6], z[7]));
  }
}

// Merged softmax of a small mini-batch (up to 128 samples, eight partials): one launch instead of mlr_lse_kernel and mlr_emit_p_kernel,
// 1.2 of the 20 us of a step at 64 x 256 with 128 samples.  Every block merges the partials of all samples itself, a sample per
// thread with all loads under way, in the order of mlr_lse_kernel's lanes; the label blocks find a class's samples in shared
// memory, as its slots are only just being set here, and follow its chain, LONG while the eight samples before are on their way.  (Followed
// between the loads, a popular class made the launch slower than the two: 4 x 256 with 100 Zipf labels 22.5 us a step in two launches,
// 24.9 so, 20.6 now; 4 x 2,000 with 128 uniform ones 34.0 so, 30.8 now.  The next eight as bytes:
// with pointers and coefficients in registers 4 x 256 21.1.  With more partials, a sample's over several lanes and so the samples in
// several passes: 405 x 940 with 102 samples and 13 partials 28 -> 38 us; with more samples the search for a class: 191 x 140 with 225 25.6 ->
// 28.4.  With more than 64 samples of more than 6,000 features 1.02 to 1.06 times as long.)
// LONG: the chain is followed ahead, which takes 80 registers instead of 40; where classes have more than four samples on average. (64 x 256 with
// 128 uniform labels 18.4 us without it, 20.1 with it; 4 x 256 and 4 x 2,000 as above.)
constexpr int kMergeSamples = 128, kMergePartials = 8;
static_assert(kMergeSamples < 255 && kLabelBatch == 8, "");
template <bool LONG>
__global__ void __launch_bounds__(256) mlr_merged_kernel(const float2* __restrict__ part, int64_t part_ld, int nblocks,
                                                         const float* __restrict__ Z, int64_t ldz, int64_t rows, int32_t n,
                                                         const int32_t* __restrict__ labels, float* __restrict__ lse,
                                                         float* __restrict__ loss, float* __restrict__ coef, int32_t* __restrict__ slot,
                                                         __nv_bfloat16* __restrict__ P, int64_t ldp, uint32_t* status, int lab_blocks,
                                                         const LabelArgs lab) {
  pdl_launch_dependents();
  pdl_wait(part, Z, labels, lse, loss, coef, slot, P);
  __shared__ float sh_lse[kMergeSamples], sh_coef[kMergeSamples], sh_loss[kMergeSamples];
  __shared__ int32_t sh_y[kMergeSamples], sh_next[kMergeSamples];
  __shared__ bool sh_first[kMergeSamples];
  const int t = threadIdx.x, lane = t & 31;
  if (t < n) {
    float2 v[kMergePartials];
#pragma unroll
    for (int b = 0; b < kMergePartials; ++b)
      v[b] = b < nblocks ? part[static_cast<int64_t>(b) * part_ld + t] : make_float2(-INFINITY, 0.f);
    const int32_t y = labels[t];
    const bool ok = y >= 0 && y < rows;
    const float zy = ok ? Z[t * ldz + y] : 0.f;
    float m = v[0].x;
#pragma unroll
    for (int b = 1; b < kMergePartials; ++b) m = fmaxf(m, v[b].x);
    float e[kMergePartials];
#pragma unroll
    for (int b = 0; b < kMergePartials; ++b) e[b] = b < nblocks ? v[b].y * __expf(v[b].x - m) : 0.f;
#pragma unroll
    for (int o = kMergePartials / 2; o > 0; o >>= 1)
#pragma unroll
      for (int b = 0; b < o; ++b) e[b] += e[b + o];
    const float l = m + logf(e[0]);
    sh_lse[t] = l;
    sh_y[t] = ok ? y : -1;
    sh_loss[t] = ok ? l - zy : 0.f;
    sh_coef[t] = ok ? -expm1f(zy - l) : 0.f;
  }
  __syncthreads();
  const int blk = static_cast<int>(blockIdx.x);
  if ((blk < lab_blocks || blk == gridDim.x - 1) && t < n) {       // the first sample of this one's class, and the next one
    const int32_t y = sh_y[t];
    int first = n, next = n;
#pragma unroll 8
    for (int j = n - 1; j >= 0; --j)
      if (sh_y[j] == y) {
        first = j;
        if (j > t) next = j;
      }
    sh_first[t] = y >= 0 && first == t;
    sh_next[t] = next;
  }
  __syncthreads();
  if (blk == gridDim.x - 1)                          // for the calls that come after
    for (int i = t; i < n; i += 256) {
      lse[i] = sh_lse[i]; loss[i] = sh_loss[i]; coef[i] = sh_coef[i];
      if (sh_y[i] < 0) atomicOr(status, SFB_STATUS_LABEL_RANGE);
      if (sh_first[i]) slot[sh_y[i]] = i;
    }
  if (blk < lab_blocks) {
    if (blk == lab_blocks - 1) {                     // the mean loss, in label_delta's order
      __shared__ float lsum[8];
      float v = t < n ? sh_loss[t] : 0.f;
      v = warp_sum(v);
      if (lane == 0) lsum[t >> 5] = v;
      __syncthreads();
      if (t == 0) {
        float mean = 0.f;
        for (int w = 0; w < 8; ++w) mean += lsum[w];
        *lab.loss_mean = mean / static_cast<float>(n);
      }
    }
    const int chunks = static_cast<int>((lab.cols + kLabelCols - 1) / kLabelCols);
    for (int u = blk; u < n * chunks; u += lab_blocks) {
      const int i = u / chunks;
      if (!sh_first[i]) continue;
      const int32_t y = sh_y[i];
      const int64_t c = static_cast<int64_t>(u % chunks) * kLabelCols + 4 * t;
      if (c >= lab.cols) continue;
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
      float* wp = lab.W + static_cast<int64_t>(y) * lab.cols + c;
      float4 w = *reinterpret_cast<const float4*>(wp);
      const float* X = lab.X + c;
      auto add = [&](float cf, const float4& x) {
        s.x = fmaf(cf, x.x, s.x); s.y = fmaf(cf, x.y, s.y); s.z = fmaf(cf, x.z, s.z); s.w = fmaf(cf, x.w, s.w);
      };
      int j = i;
      if (sh_next[j] >= n) {                         // a class of one sample
        add(sh_coef[j], *reinterpret_cast<const float4*>(X + static_cast<int64_t>(j) * lab.cols));
      } else if (!LONG) {
        while (j < n) {
          if (sh_next[j] >= n) {                     // the last one by itself
            add(sh_coef[j], *reinterpret_cast<const float4*>(X + static_cast<int64_t>(j) * lab.cols));
            break;
          }
          float4 x[kLabelBatch];
          const float* xp[kLabelBatch];
          float cf[kLabelBatch];
#pragma unroll
          for (int e = 0; e < kLabelBatch; ++e) {
            xp[e] = X + static_cast<int64_t>(j < n ? j : i) * lab.cols;
            cf[e] = j < n ? sh_coef[j] : 0.f;
            if (j < n) j = sh_next[j];
          }
          load8(x, xp);
#pragma unroll
          for (int e = 0; e < kLabelBatch; ++e) add(cf[e], x[e]);
        }
      } else {
        uint32_t at[kLabelBatch / 4], ahead[kLabelBatch / 4];
        auto follow = [&](uint32_t (&q)[kLabelBatch / 4]) {        // the next eight of the chain, a byte each: 255 behind its end
          q[0] = q[1] = 0;
#pragma unroll
          for (int e = 0; e < kLabelBatch; ++e) {
            q[e / 4] |= static_cast<uint32_t>(j < n ? j : 255) << (8 * (e % 4));
            if (j < n) j = sh_next[j];
          }
        };
        auto sample = [&](int e) { return static_cast<int>((at[e / 4] >> (8 * (e % 4))) & 255u); };
        follow(at);
        for (bool more = true; more;) {              // the chain is followed while the samples are on their way
          float4 x[kLabelBatch];
#pragma unroll
          for (int e = 0; e < kLabelBatch; ++e)
            x[e] = __ldg(reinterpret_cast<const float4*>(X + (sample(e) < n ? sample(e) : i) * lab.cols));
          more = j < n;
          if (more) follow(ahead);
#pragma unroll
          for (int e = 0; e < kLabelBatch; ++e) add(sample(e) < n ? sh_coef[sample(e)] : 0.f, x[e]);
          at[0] = ahead[0]; at[1] = ahead[1];
        }
      }
      *reinterpret_cast<float4*>(lab.dL + static_cast<int64_t>(i) * lab.cols + c) = s;
      w.x = fmaf(lab.step, s.x, w.x); w.y = fmaf(lab.step, s.y, w.y); w.z = fmaf(lab.step, s.z, w.z); w.w = fmaf(lab.step, s.w, w.w);
      *reinterpret_cast<float4*>(wp) = w;
      *reinterpret_cast<uint2*>(lab.Wb + static_cast<int64_t>(y) * lab.ldw + c) = make_uint2(pack_bf16(w.x, w.y), pack_bf16(w.z, w.w));
    }
    return;
  }
  const int octs = static_cast<int>((rows + 7) / 8), emit = static_cast<int>(gridDim.x) - lab_blocks;
  for (int q = (blk - lab_blocks) * 256 + t; q < n * octs; q += emit * 256) {
    const int i = q / octs, r = (q - i * octs) * 8, yrel = sh_y[i] - r;
    const float l = sh_lse[i];
    const float4 a = *reinterpret_cast<const float4*>(Z + i * ldz + r), b = *reinterpret_cast<const float4*>(Z + i * ldz + r + 4);
    float z[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int k = 0; k < 8; ++k) z[k] = k == yrel ? 0.f : __expf(z[k] - l);
    *reinterpret_cast<uint4*>(P + i * ldp + r) =
        make_uint4(pack_bf16(z[0], z[1]), pack_bf16(z[2], z[3]), pack_bf16(z[4], z[5]), pack_bf16(z[6], z[7]));
  }
}

// Both for a worker's samples whose label rows are summed later: every block merges the partials of its sample itself, which
// saves a launch (3 us of a call of 37 samples against 4,999 x 3,004).  One sample per grid row, its classes over the grid's
// columns.
__global__ void __launch_bounds__(256) mlr_lse_emit_kernel(const float2* __restrict__ part, int64_t part_ld, int nblocks,
                                                           const float* __restrict__ Z, int64_t ldz, int64_t rows,
                                                           const int32_t* __restrict__ labels, int64_t off, float* __restrict__ lse,
                                                           float* __restrict__ loss, float* __restrict__ coef,
                                                           __nv_bfloat16* __restrict__ P, int64_t ldp, uint32_t* status) {
  pdl_launch_dependents();
  pdl_wait(part, Z, labels, lse, loss, coef, P);
  __shared__ float sh[16];
  const int t = threadIdx.x;
  const int64_t i = blockIdx.y, s = off + i;
  float m = -INFINITY;
  for (int b = t; b < nblocks; b += 256) m = fmaxf(m, part[static_cast<int64_t>(b) * part_ld + s].x);
  m = warp_max(m);
  if ((t & 31) == 0) sh[t >> 5] = m;
  __syncthreads();
  m = sh[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) m = fmaxf(m, sh[w]);
  float sum = 0.f;
  for (int b = t; b < nblocks; b += 256) {
    const float2 v = part[static_cast<int64_t>(b) * part_ld + s];
    sum += v.y * __expf(v.x - m);
  }
  sum = warp_sum(sum);
  if ((t & 31) == 0) sh[8 + (t >> 5)] = sum;
  __syncthreads();
  sum = sh[8];
#pragma unroll
  for (int w = 1; w < 8; ++w) sum += sh[8 + w];
  const float l = m + logf(sum);
  const int64_t y = labels[i];
  if (blockIdx.x == 0 && t == 0) {
    const bool okl = y >= 0 && y < rows;
    if (!okl) atomicOr(status, SFB_STATUS_LABEL_RANGE);
    const float zy = okl ? Z[s * ldz + y] : 0.f;
    lse[s] = l;
    loss[s] = okl ? l - zy : 0.f;
    coef[s] = okl ? -expm1f(zy - l) : 0.f;
  }
  const int octs = static_cast<int>((rows + 7) / 8);
  for (int q = blockIdx.x * 256 + t; q < octs; q += gridDim.x * 256) {
    const int64_t r = static_cast<int64_t>(q) * 8, yrel = y - r;
    const float4 a = *reinterpret_cast<const float4*>(Z + s * ldz + r), b = *reinterpret_cast<const float4*>(Z + s * ldz + r + 4);
    float z[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
    for (int k = 0; k < 8; ++k) z[k] = k == yrel ? 0.f : __expf(z[k] - l);
    *reinterpret_cast<uint4*>(P + s * ldp + r) =
        make_uint4(pack_bf16(z[0], z[1]), pack_bf16(z[2], z[3]), pack_bf16(z[4], z[5]), pack_bf16(z[6], z[7]));
  }
}

// ---------------------------------------------------------------------------------------------------------
// fp32 mode on the tensor cores: every fp32 value x is carried as two tf32 words, big = tf32(x) and
// small = tf32(x - big) (x = big + small to about 2^-22 |x|), and a product runs as big*big + big*small + small*big.
// ---------------------------------------------------------------------------------------------------------
__device__ __forceinline__ float to_tf32(float x) {
  uint32_t u;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(x));
  return __uint_as_float(u);
}

// fp32 [n x dim] (row pitch ld) -> [n x 2*dimp] fp32 words: dst[r][c] = big, dst[r][dimp + c] = small.  Columns
// dim..dimp-1 keep the zeros of set-up.  dim and ld are multiples of 4.
__global__ void __launch_bounds__(256) split32_rows_kernel(const float* __restrict__ F, int64_t n, int64_t dim, int64_t ld,
                                                           float* __restrict__ dst, int64_t dimp) {
  pdl_launch_dependents();
  pdl_wait(F, dst);
  const int64_t quads = dim / 4, total = n * quads;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total; i += stride) {
    const int64_t r = i / quads, qd = i % quads;
    const float4 v = *reinterpret_cast<const float4*>(F + r * ld + qd * 4);
    const float4 b = make_float4(to_tf32(v.x), to_tf32(v.y), to_tf32(v.z), to_tf32(v.w));
    float* d = dst + r * 2 * dimp + qd * 4;
    *reinterpret_cast<float4*>(d) = b;
    *reinterpret_cast<float4*>(d + dimp) = make_float4(to_tf32(v.x - b.x), to_tf32(v.y - b.y), to_tf32(v.z - b.z),
                                                       to_tf32(v.w - b.w));
  }
}

// Gathered fp32 factors F [n x dim] (pair-major, row pitch ld) -> FT [dim x 2*Kp] (pairs contiguous):
// FT[c][i] = big, FT[c][Kp + i] = small; pairs n..Kp-1 are written as zeros.  64 x 64 tiles through shared memory.
__global__ void __launch_bounds__(256) split32_t_kernel(const float* __restrict__ F, int64_t n, int64_t dim, int64_t ld,
                                                        float* __restrict__ FT, int64_t Kp) {
  pdl_launch_dependents();
  pdl_wait(F, FT);
  __shared__ float tile[64][65];
  const int64_t i0 = static_cast<int64_t>(blockIdx.y) * 64, c0 = static_cast<int64_t>(blockIdx.x) * 64;
  const int t = threadIdx.x;
#pragma unroll
  for (int v = 0; v < 16; ++v) {
    const int idx = t + v * 256;            // 64 pairs x 64 columns
    const int i = idx / 64, c = idx % 64;
    tile[i][c] = (i0 + i < n && c0 + c < dim) ? F[(i0 + i) * ld + c0 + c] : 0.f;
  }
  __syncthreads();
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const int idx = t + v * 256;            // 64 columns x 16 groups of 4 pairs
    const int c = idx / 16, ig = (idx % 16) * 4;
    if (c0 + c >= dim || i0 + ig >= Kp) continue;
    const float f0 = tile[ig][c], f1 = tile[ig + 1][c], f2 = tile[ig + 2][c], f3 = tile[ig + 3][c];
    const float4 b = make_float4(to_tf32(f0), to_tf32(f1), to_tf32(f2), to_tf32(f3));
    float* dst = FT + (c0 + c) * 2 * Kp + i0 + ig;          // Kp is a multiple of 32: 16-byte aligned
    *reinterpret_cast<float4*>(dst) = b;
    *reinterpret_cast<float4*>(dst + Kp) = make_float4(to_tf32(f0 - b.x), to_tf32(f1 - b.y), to_tf32(f2 - b.z), to_tf32(f3 - b.w));
  }
}

// u_ij = exp(z_ij - lse_i) - [j = y_i], from the logits Z [n x ldz] to the pair-major fp32 factors U [n x rows]
// (Section 2.1: u = d f / d (W a)).
__global__ void __launch_bounds__(256) mlr_finish_u_kernel(const float* __restrict__ Z, int64_t ldz, int64_t rows,
                                                           const float* __restrict__ lse,
                                                           const int32_t* __restrict__ labels,
                                                           float* __restrict__ U) {
  pdl_launch_dependents();
  pdl_wait(Z, lse, labels, U);
  const int64_t i = blockIdx.y;
  const float l = lse[i];
  const int64_t y = labels[i];
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; j < rows; j += stride) {
    const float z = Z[i * ldz + j];
    U[i * rows + j] = expf(z - l) - (j == y ? 1.f : 0.f);
  }
}

// ---------------------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------------------
template <bool TF32>
cudaError_t launch_forward(sfb_ctx* ctx, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& c, TcParams p) {
  TcState* st = static_cast<TcState*>(ctx->tc);
  const int64_t tiles = static_cast<int64_t>(p.tilesM) * p.tilesN;
  if (tiles <= 0) return cudaSuccess;
  const unsigned grid = static_cast<unsigned>(p.kparts > 1 ? tiles * p.kparts : std::min<int64_t>(tiles, st->sms));
  return launch_kernel_if(tiles * p.kparts <= st->sms, forward_kernel<TF32>, dim3(grid), dim3(kThreads), kSmem, ctx->stream,
                          p.kparts, a, b, c, p);
}

// The shared-memory opt-in is a per-device attribute of each kernel: set for every instantiation when a context is
// created (with its device current), not once per process.
cudaError_t prepare_forward_kernels() {
  cudaError_t e = cudaFuncSetAttribute(forward_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(forward_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  return e;
}

}  // namespace

#define CKC(call)                                       \
  do {                                                  \
    cudaError_t e__ = (call);                           \
    if (e__ != cudaSuccess) {                           \
      ctx->last_cuda = static_cast<int>(e__);           \
      return SFB_ERR_CUDA;                              \
    }                                                   \
  } while (0)

// Stages of the operand ring for tiles of bn columns (192 KB).
static int forward_stages(int bn) { return std::min(S_MAX, S * (kBytesA + kBytesB) / (kBytesA + bn * BK * 2)); }

// Cycles of the forward product of n samples with a rows x cols matrix in tiles of bn columns and `split` parts.  A k-block of
// a tile takes the longest of its MMAs (2 cycles per column), its bytes at about 60 a cycle and the latency of its loads over
// the stages in flight; the exchange of the parts about 3000.
static double forward_cost(int64_t n, int64_t rows, int64_t cols, int bn, int split) {
  const double kb = static_cast<double>((cols + BK - 1) / BK), ar = static_cast<double>(std::min<int64_t>(BM, round_up(n, 8)));
  const int64_t ctas = ((n + BM - 1) / BM) * ((rows + bn - 1) / bn) * split;
  const double rounds = static_cast<double>((ctas + kModelSms - 1) / kModelSms);
  const double per_kb = std::max(std::max(2.0 * bn, (ar + bn) * BK * 2 / 60.0), 1200.0 / forward_stages(bn));
  return rounds * (kb / split * per_kb + 2500.0 + (split > 1 ? 3000.0 : 0.0));
}
// Tile width: a power of two from `least` to 256 (128 with a split contraction, whose parts are exchanged through the operand
// stages).  Wide tiles read the samples less often, narrow ones occupy more SMs when W has few rows (a worker's 37 samples
// against 4,999 x 3,004: 23 us with 256-wide tiles on 20 SMs).
static int pick_forward_width(int64_t n, int64_t rows, int64_t cols, int least, int split) {
  int best = split > 1 ? 128 : 256;
  double cost = forward_cost(n, rows, cols, best, split);
  for (int bn = best / 2; bn >= least; bn /= 2) {
    const double c = forward_cost(n, rows, cols, bn, split);
    if (c < 0.97 * cost) { cost = c; best = bn; }
  }
  return best;
}
// Parts that the contraction of the forward product is cut into when the tiles of all K samples do not fill the SMs (72 rows of
// 14,240 columns: 223 k-blocks in a row on one SM, 68 us).  One choice per context, for the calls that forward_kernel takes: its sums
// then have one order.  (By their number of samples others go to the kernels of sfb_forward.cu, whose sums have another one.)
static int pick_forward_split(int64_t K, int64_t rows, int64_t cols) {
  int best = 1;
  double cost = forward_cost(K, rows, cols, pick_forward_width(K, rows, cols, 32, 1), 1);
  for (int s = 2; s <= 8 && (cols + BK - 1) / BK >= 2 * s; s *= 2) {
    const double c = forward_cost(K, rows, cols, pick_forward_width(K, rows, cols, 32, s), s);
    if (c < 0.9 * cost) { cost = c; best = s; }
  }
  return best;
}

// Whether the logits of n samples take the kernel of CTA pairs.  Not beyond five rounds of its tiles, where an uneven last one matters
// little (325,000 x 10,000 with 1,024 samples: 5,280 us of the factors' time here, 5,470 there) and the softmax has twice the partials to
// merge: from 30,000 classes on, steps with 129 to 200 samples of up to 1,000 features take 1.5 to 1.7 times as long on pairs, with 300 to 500
// 1.45, with more than 1,000 1.02 to 1.05, although their factors by calls take 0.91 to 1.03.
// What forward_cost has for a split contraction chooses among splits; against another kernel it needs 22,000 cycles more, and its rounds are
// those of the clusters that are resident at a time (15 of eight CTAs, 120 of the 148 SMs: the factors of 281 x 7,060 with 146 samples,
// 144 CTAs, 33.6 us, 22.9 on pairs; 870 x 1,012 with 218, 112 CTAs, 16.5 and 14.0).
static bool forward_on_pairs(const sfb_config& c, const Layout& L, int64_t n, int* parts) {
  if (n <= BM || ((n + 255) / 256) * ((c.rows + 255) / 256) >= 5 * (kModelSms / 2)) return false;
  const int bn = pick_forward_width(n, c.rows, c.cols, L.pw, L.split);
  double cost = forward_cost(n, c.rows, c.cols, bn, L.split);
  if (L.split > 1) {
    const int64_t clusters = ((n + BM - 1) / BM) * ((c.rows + bn - 1) / bn), resident = L.split == 2 ? 74 : L.split == 4 ? 33 : 15;
    const int64_t by_ctas = (clusters * L.split + kModelSms - 1) / kModelSms, rounds = (clusters + resident - 1) / resident;
    cost = (cost / static_cast<double>(by_ctas) - 3000.0 + 22000.0) * static_cast<double>(rounds);
  }
  return forward_pair_pays(n, c.rows, c.cols, cost, (c.rows + L.pw - 1) / L.pw, parts);
}

// The kernel that forms the logits of n samples, in bf16 mode; step: in a call that goes on to the update.
enum LogitsKernel { kLogitsTiles = 1, kLogitsPairs = 2, kLogitsFew = 3 };
static LogitsKernel logits_kernel(const sfb_config& c, const Layout& L, int64_t n, bool step, int* parts) {
  *parts = L.split;
  if (forward_few_fits(n, c.rows, c.cols, step)) return kLogitsFew;
  return forward_on_pairs(c, L, n, parts) ? kLogitsPairs : kLogitsTiles;
}

// Whether the softmax of a step's n samples, `partials` of each, is merged by mlr_merged_kernel.
static bool softmax_merged(int64_t n, int64_t cols, int64_t partials) {
  return n <= (cols > 6000 ? kMergeSamples / 2 : kMergeSamples) && partials <= kMergePartials;
}

int tc_logits_plan(const sfb_config& c, const Layout& L, int64_t n, bool step, int* parts, bool* merged) {
  const LogitsKernel k = logits_kernel(c, L, n, step, parts);
  const int64_t pw = k == kLogitsFew ? 32 : L.pw;
  *merged = k != kLogitsPairs && softmax_merged(n, c.cols, (c.rows + pw - 1) / pw);
  if (k == kLogitsFew) *parts = 1;
  return k;
}

// fp32 mode on the tensor cores (MLR): fp32 pair-major factors as in the FFMA path, plus the (big | small) tf32
// operands of the two products and the logits.
void tc32_extend_layout(const sfb_config& c, Layout& L, size_t& off) {
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + kAlign - 1) / kAlign * kAlign; return o; };
  const size_t K = static_cast<size_t>(c.workers) * c.batch;
  L.Kp = round_up(static_cast<int64_t>(K), 32);
  L.colsp = round_up(c.cols, 32);
  const size_t ldz = static_cast<size_t>(round_up(c.rows, 32));
  const size_t nblk = static_cast<size_t>((c.rows + BN - 1) / BN);
  L.V = take(K * static_cast<size_t>(c.cols) * 4);
  L.U = take(K * static_cast<size_t>(c.rows) * 4);
  L.Ws = take(static_cast<size_t>(c.rows) * 2 * L.colsp * 4);        // W, rows x (big | small)
  L.As = take(K * 2 * static_cast<size_t>(L.colsp) * 4);             // the samples, K x (big | small)
  L.VT = take(static_cast<size_t>(c.cols) * 2 * L.Kp * 4);
  L.UT = take(static_cast<size_t>(c.rows) * 2 * L.Kp * 4);
  L.ZT = take(K * ldz * 4);
  L.part = take(nblk * K * 8);
  L.lse = take(K * 4);
  L.coef = take(K * 4);
  L.labels = take(K * 4);
}

void tc_extend_layout(const sfb_config& c, Layout& L, size_t& off) {
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + kAlign - 1) / kAlign * kAlign; return o; };
  const size_t K = static_cast<size_t>(c.workers) * c.batch;
  L.Kp = round_up(static_cast<int64_t>(K), 64);
  L.colsb = round_up(c.cols, 64);
  if (c.model != SFB_MLR) return split_extend_layout(c, L, off);
  const size_t ldz = static_cast<size_t>(round_up(c.rows, 32));
  L.split = pick_forward_split(static_cast<int64_t>(K), c.rows, c.cols);
  L.pw = L.split > 1 ? 32 : pick_forward_width(c.batch, c.rows, c.cols, 32, 1);
  size_t nblk = static_cast<size_t>((c.rows + L.pw - 1) / L.pw);
  if (forward_few_fits(c.batch, c.rows, c.cols, true)) nblk = std::max(nblk, static_cast<size_t>(forward_few_groups(c.rows)));
  // For the kernel of CTA pairs, where a worker's call, one of all samples or a part of sfb_step_host's takes it: parts of tiles, 256 KB
  // a pair that leaves some (19 MB in all; whatever the context, 325,000 x 10,000 had them for nothing).
  for (int64_t parts = 0; parts <= HostSide::kParts; parts = parts ? 2 * parts : 1) {
    const int64_t n = parts ? static_cast<int64_t>(K) / parts : c.batch;
    int cut = 1;
    if (n < 1 || logits_kernel(c, L, n, parts != 0, &cut) != kLogitsPairs) continue;
    L.on_pairs = true;
    L.cut_pairs = std::max(L.cut_pairs, static_cast<int32_t>(forward_pair_cut(n, c.rows, c.cols)));
  }
  if (L.on_pairs) nblk = std::max(nblk, static_cast<size_t>(forward_pair_groups(c.rows)));
  if (L.cut_pairs > 0) {
    L.partial = take(forward_pair_partial_bytes(L.cut_pairs));
    L.ready = take(forward_pair_ready_bytes());
  }
  L.Wb = take(static_cast<size_t>(c.rows) * L.colsb * 2);
  L.Xb = take(K * L.colsb * 2);
  L.ZT = take(K * ldz * 4);                      // logits Z, sample-major [K x ldz]
  L.ldp = round_up(c.rows, 64);
  L.P = take(K * static_cast<size_t>(L.ldp) * 2);
  L.part = take(nblk * K * 8);
  L.V = take(K * 4);                             // log-sum-exp per sample
  L.Xf = take(K * static_cast<size_t>(c.cols) * 4);   // fp32 copy of the K samples (exact label-row term)
  L.labels = take(K * 4);                        // class ids of the K samples
  L.coef = take(K * 4);                          // 1 - p_y per sample (fp32 label entry of u)
  L.slot = take(static_cast<size_t>(c.rows) * 4);     // per class of W: its first sample in the mini-batch (kNoSlot: none)
  L.dL = take(K * static_cast<size_t>(c.cols) * 4);   // per such sample: the fp32 sum that the class's row of W takes
  L.U = 0;
}

int tc_init(sfb_ctx* ctx) {
  TcState* st = new (std::nothrow) TcState();
  if (!st) return SFB_ERR_ARG;
  ctx->tc = st;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  CKC(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres));
  if (qres != cudaDriverEntryPointSuccess || !fn) return SFB_ERR_CUDA;
  st->encode = reinterpret_cast<EncodeTiledFn>(fn);
  int dev = 0;
  CKC(cudaGetDevice(&dev));
  CKC(cudaDeviceGetAttribute(&st->sms, cudaDevAttrMultiProcessorCount, dev));
  CKC(prepare_forward_kernels());
  CKC(forward_few_prepare(st->few));
  {
    const int rc = tc_update_init(ctx, st);
    if (rc) return rc;
  }
  const sfb_config& c = ctx->cfg;
  if (ctx->tf32) {
    // pad columns of the split operands are never written by the kernels: clear the buffers once
    const Layout& L = ctx->lay;
    CKC(cudaMemsetAsync(ctx->at<char>(L.Ws), 0, static_cast<size_t>(c.rows) * 2 * L.colsp * 4, ctx->stream));
    CKC(cudaMemsetAsync(ctx->at<char>(L.As), 0, static_cast<size_t>(ctx->K) * 2 * L.colsp * 4, ctx->stream));
    return tc_refresh_operands(ctx);
  }
  if (c.model != SFB_MLR || ctx->h16) return split_init(ctx);
  if (ctx->lay.ready) CKC(cudaMemsetAsync(ctx->at<char>(ctx->lay.ready), 0, forward_pair_ready_bytes(), ctx->stream));
  CKC(cudaMemsetAsync(ctx->at<char>(ctx->lay.labels), 0xff, static_cast<size_t>(ctx->K) * 4, ctx->stream));
  CKC(cudaMemsetAsync(ctx->at<char>(ctx->lay.slot), 0x7f, static_cast<size_t>(c.rows) * 4, ctx->stream));
  // bf16 copy of W for the forward product; afterwards the update's epilogue keeps it current
  return tc_refresh_operands(ctx);
}

int tc_refresh_operands(sfb_ctx* ctx) {
  const sfb_config& c = ctx->cfg;
  if (c.model != SFB_MLR) return SFB_OK;          // the split copies of W are rebuilt by the first factors call of a step
  TcState* st = static_cast<TcState*>(ctx->tc);
  if (ctx->tf32) {
    CKC(launch_kernel(split32_rows_kernel, dim3(static_cast<unsigned>(st->sms * 16)), dim3(256), 0, ctx->stream, 1,
                      ctx->W, c.rows, c.cols, c.cols, ctx->at<float>(ctx->lay.Ws), ctx->lay.colsp));
      return SFB_OK;
  }
  CKC(launch_kernel(convert_rows_kernel, dim3(st->sms * 8), dim3(256), 0, ctx->stream, 1, ctx->W, c.rows, c.cols,
                    ctx->at<__nv_bfloat16>(ctx->lay.Wb), ctx->lay.colsb));
  return SFB_OK;
}

void tc_destroy(sfb_ctx* ctx) {
  delete static_cast<TcState*>(ctx->tc);
  ctx->tc = nullptr;
}

// v = x, the (big | small) samples, and the logits of n samples at pair offset off against this context's rows as
// the three-term tf32 product, with the per-(sample, 256-row block) softmax partials.
static int mlr32_forward(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, int* tiles_n) {
  const sfb_config& c = ctx->cfg;
  TcState* st = static_cast<TcState*>(ctx->tc);
  const Layout& L = ctx->lay;
  const int64_t rows = c.rows, cols = c.cols, K = ctx->K;
  const int64_t ldz = round_up(rows, 32);
  cudaStream_t s = ctx->stream;
  float* Ws = ctx->at<float>(L.Ws);
  float* As = ctx->at<float>(L.As);
  float* Z = ctx->at<float>(L.ZT);
  float* V = ctx->at<float>(L.V) + off * cols;
  // Ws, the (big | small) copy of W, is built at set-up and rewritten by the update's epilogue together with W
  CKC(pack_copy(s, V, X, nullptr, n * cols, take_stamp(ctx)));                             // v = x
  CKC(launch_kernel(split32_rows_kernel, dim3(grid1d(n * cols / 4, 256)), dim3(256), 0, s, 1, X, n, cols, cols,
                    As + off * 2 * L.colsp, L.colsp));
  CUtensorMap ma, mb, mc;
  if (!make_map(st, &ma, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, As, 2 * L.colsp, off + n, 2 * L.colsp * 4, BK / 2, BM) ||
      !make_map(st, &mb, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, Ws, 2 * L.colsp, rows, 2 * L.colsp * 4, BK / 2, BN) ||
      !make_map(st, &mc, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, Z, rows, off + n, ldz * 4, kChunk, 32))
    return SFB_ERR_CUDA;
  TcParams p{};
  p.M = static_cast<int32_t>(off + n); p.N = static_cast<int32_t>(rows); p.Kc = static_cast<int32_t>(L.colsp);
  p.m_off = static_cast<int32_t>(off);
  p.tilesM = static_cast<int32_t>((n + BM - 1) / BM);
  p.bn = BN; p.kparts = 1; p.pw = BN; p.a_rows = BM; p.stages = S;
  p.tilesN = static_cast<int32_t>((rows + BN - 1) / BN);
  p.part = ctx->at<float2>(L.part); p.part_ld = K; p.status = ctx->at<uint32_t>(L.status);
  p.nseg = 3; p.kseg = static_cast<int32_t>(L.colsp / (BK / 2));          // cross terms first, big*big last
  p.a_off0 = 0; p.a_off1 = static_cast<int32_t>(L.colsp); p.a_off2 = 0;
  p.b_off0 = static_cast<int32_t>(L.colsp); p.b_off1 = 0; p.b_off2 = 0;
  CKC((launch_forward<true>(ctx, ma, mb, mc, p)));                                // z_i = W x_i
  ctx->stats.flops += 3.0 * 2.0 * n * rows * cols;
  *tiles_n = p.tilesN;
  return SFB_OK;
}

// Row-sharded form in the tensor-core fp32 mode: partials of all K samples against this shard's rows ...
int tc32_forward_partials(sfb_ctx* ctx, const float* X, const int32_t* labels, float* part_out) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  int tiles_n = 0;
  const int rc = mlr32_forward(ctx, 0, ctx->K, X, &tiles_n);
  if (rc) return rc;
  CKC(cudaMemcpyAsync(ctx->at<int32_t>(L.labels), labels, static_cast<size_t>(ctx->K) * 4, cudaMemcpyDeviceToDevice, ctx->stream));
  CKC(launch_kernel(mlr_shard_partials_tc_kernel, dim3(static_cast<unsigned>((ctx->K + 7) / 8)), dim3(256), 0,
                    ctx->stream, 1, ctx->at<float2>(L.part), ctx->K, tiles_n, ctx->at<float>(L.ZT), round_up(c.rows, 32),
                    c.rows, ctx->at<int32_t>(L.labels), ctx->row_offset, ctx->K, reinterpret_cast<float4*>(part_out)));
  return SFB_OK;
}

// ... and the fp32 factors from the partials of all shards.
int tc32_finish_factors(sfb_ctx* ctx, const float* parts, int shards) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t K = ctx->K, rows = c.rows;
  CKC(launch_kernel(mlr_shard_finish_tc_kernel, dim3(static_cast<unsigned>((K + 255) / 256)), dim3(256), 0, ctx->stream,
                    1, reinterpret_cast<const float4*>(parts), shards, K, rows, ctx->row_offset,
                    ctx->at<int32_t>(L.labels), ctx->at<float>(L.lse), ctx->at<float>(L.loss), ctx->at<float>(L.coef),
                    ctx->at<uint32_t>(L.status)));
  dim3 ugrid(static_cast<unsigned>(std::min<int64_t>((rows + 255) / 256, 64)), static_cast<unsigned>(K));
  CKC(launch_kernel(mlr_finish_u_kernel, ugrid, dim3(256), 0, ctx->stream, 1, ctx->at<float>(L.ZT), round_up(rows,
                    32), rows, ctx->at<float>(L.lse), ctx->at<int32_t>(L.labels), ctx->at<float>(L.U)));
  return SFB_OK;
}

// fp32 mode on the tensor cores: factors of n MLR samples at pair offset off.  The logits are the three-term tf32
// product of the (big | small) samples and the (big | small) rows of W; softmax, loss and the factors in fp32.
// sdca_ids != nullptr: the dual changes of the SDCA step instead of softmax - onehot.
int tc32_factors(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const int32_t* labels, const int32_t* sdca_ids,
                 float inv_lam_n) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t rows = c.rows, K = ctx->K;
  const int64_t ldz = round_up(rows, 32);
  cudaStream_t s = ctx->stream;
  float* Z = ctx->at<float>(L.ZT);
  float* U = ctx->at<float>(L.U) + off * rows;
  int tiles_n = 0;
  {
    const int rc = mlr32_forward(ctx, off, n, X, &tiles_n);
    if (rc) return rc;
  }
  dim3 ugrid(static_cast<unsigned>(std::min<int64_t>((rows + 255) / 256, 64)), static_cast<unsigned>(n));
  if (sdca_ids) {
    SdcaArgs a = sdca_args(ctx, off, n, X, labels, sdca_ids, inv_lam_n);
    a.Z = Z + off * ldz; a.ldz = ldz; a.out = U; a.ldo = rows;
    CKC(sdca_dual_rows(s, a));
  } else {
    float* lse = ctx->at<float>(L.lse);
    CKC(launch_kernel(mlr_lse_kernel, dim3(static_cast<unsigned>((n + 7) / 8)), dim3(256), 0, s, 1,
                      ctx->at<float2>(L.part), K, tiles_n, Z, ldz, rows, labels, off, n, lse, ctx->at<float>(L.loss),
                      ctx->at<float>(L.coef), nullptr, ctx->at<uint32_t>(L.status)));
    CKC(launch_kernel(mlr_finish_u_kernel, ugrid, dim3(256), 0, s, 1, Z + off * ldz, ldz, rows, lse + off, labels,
                      U));
  }
  return SFB_OK;
}

// The gathered fp32 pairs (computed here or received) become the (big | small) operands of the update product.
int tc32_gather(sfb_ctx* ctx) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const unsigned gy = static_cast<unsigned>((L.Kp + 63) / 64);
  CKC(launch_kernel(split32_t_kernel, dim3(static_cast<unsigned>((c.rows + 63) / 64), gy), dim3(256), 0, ctx->stream, 1,
                    ctx->at<float>(L.U), ctx->K, c.rows, c.rows, ctx->at<float>(L.UT), L.Kp));
  CKC(launch_kernel(split32_t_kernel, dim3(static_cast<unsigned>((c.cols + 63) / 64), gy), dim3(256), 0, ctx->stream, 1,
                    ctx->at<float>(L.V), ctx->K, c.cols, c.cols, ctx->at<float>(L.VT), L.Kp));
  return SFB_OK;
}

// Pack of n samples at pair offset off and their logits against the rows of this context's W:
// Z[off .. off+n) = X W^T with the softmax partials.  fused: see tc_factors.
static int mlr_forward(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const int32_t* labels, bool fused, int* parts) {
  const sfb_config& c = ctx->cfg;
  TcState* st = static_cast<TcState*>(ctx->tc);
  const Layout& L = ctx->lay;
  const int64_t rows = c.rows, cols = c.cols, K = ctx->K;
  const int64_t ldz = round_up(rows, 32);
  __nv_bfloat16* Xb = ctx->at<__nv_bfloat16>(L.Xb);
  ctx->labels = sfb_ctx::kLabelsNone;
  ctx->stats.flops += 2.0 * n * rows * cols;
  // (samples that come by a copy on another stream: that one has to be complete before the kernel starts at all)
  const bool early = !ctx->host || ctx->host->parts <= 1;
  if (!ctx->packed)
    CKC(launch_kernel_if(early, pack_mlr_kernel, dim3(grid1d(n * cols / 4, 256)), dim3(256), 0, ctx->stream, 1, X, n, cols, Xb,
                    L.colsb, off,
                    fused ? nullptr : ctx->at<float>(L.Xf), labels, ctx->at<int32_t>(L.labels), ctx->at<int32_t>(L.slot),
                    rows,
                    take_stamp(ctx)));
  int cut = 1;
  const LogitsKernel kernel = logits_kernel(c, L, n, fused, &cut);
  if (kernel == kLogitsFew) {
    CKC(forward_few(ctx, off, n));
    *parts = static_cast<int>(forward_few_groups(rows));
    return SFB_OK;
  }
  if (kernel == kLogitsPairs && L.on_pairs) {
    int pw = 0;
    CKC(forward_pair(ctx, off, n, &pw));
    *parts = static_cast<int>((rows + pw - 1) / pw);
    return SFB_OK;
  }
  // samples on the lanes (A), rows of W on the accumulator columns (B)
  const int bn = pick_forward_width(n, rows, cols, L.pw, L.split);
  const int ar = static_cast<int>(std::min<int64_t>(BM, round_up(n, 8)));
  CUtensorMap ma, mb, mc;
  if (!make_map(st, &ma, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, Xb, cols, K, L.colsb * 2, BK, ar) ||
      !make_map(st, &mb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, ctx->at<__nv_bfloat16>(L.Wb), cols, rows, L.colsb * 2, BK, bn) ||
      !make_map(st, &mc, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, ctx->at<float>(L.ZT), rows, off + n, ldz * 4, kChunk, 32))
    return SFB_ERR_CUDA;
  TcParams p{};
  p.M = static_cast<int32_t>(off + n); p.N = static_cast<int32_t>(rows); p.Kc = static_cast<int32_t>(cols);
  p.m_off = static_cast<int32_t>(off);
  p.tilesM = static_cast<int32_t>((n + BM - 1) / BM);
  p.bn = bn; p.kparts = L.split; p.pw = L.pw; p.a_rows = ar; p.stages = forward_stages(bn);
  p.tilesN = static_cast<int32_t>((rows + bn - 1) / bn);
  p.part = ctx->at<float2>(L.part); p.part_ld = K; p.status = ctx->at<uint32_t>(L.status);
  p.nseg = 1; p.kseg = (p.Kc + BK - 1) / BK;
  CKC(launch_forward<false>(ctx, ma, mb, mc, p));
  *parts = static_cast<int>((rows + L.pw - 1) / L.pw);
  return SFB_OK;
}

static LabelArgs label_args(sfb_ctx* ctx, const float* X) {
  const Layout& L = ctx->lay;
  LabelArgs a{};
  a.X = X;
  a.labels = ctx->at<int32_t>(L.labels); a.slot = ctx->at<int32_t>(L.slot); a.coef = ctx->at<float>(L.coef);
  a.dL = ctx->at<float>(L.dL);
  a.loss = ctx->at<float>(L.loss); a.loss_mean = &ctx->at<Scalars>(L.scalars)->loss_mean;
  a.rows = ctx->cfg.rows; a.cols = ctx->cfg.cols; a.K = static_cast<int32_t>(ctx->K);
  a.W = ctx->W; a.Wb = ctx->at<__nv_bfloat16>(L.Wb); a.ldw = L.colsb; a.step = ctx->step;
  return a;
}
static int label_blocks(const sfb_ctx* ctx) {
  return static_cast<int>(std::min<int64_t>(ctx->K * ((ctx->cfg.cols + kLabelCols - 1) / kLabelCols), 6 * sm_count()));
}

// Probabilities (or, PLAIN, the values of Z) of n samples as the operand of the update; fused: and the label rows applied.
template <bool PLAIN>
static int emit_p(sfb_ctx* ctx, int64_t off, int64_t n, const int32_t* labels, const float* fused_X) {
  const Layout& L = ctx->lay;
  const int64_t rows = ctx->cfg.rows;
  const int lab = fused_X ? label_blocks(ctx) : 0;
  CKC(launch_kernel(mlr_emit_p_kernel<PLAIN>, dim3(grid1d(n * ((rows + 7) / 8), 256) + lab), dim3(256), 0, ctx->stream, 1,
                    ctx->at<float>(L.ZT), round_up(rows, 32), rows, ctx->at<float>(L.V), off, n, labels,
                    ctx->at<__nv_bfloat16>(L.P), L.ldp, lab, label_args(ctx, fused_X)));
  if (fused_X) ctx->labels = sfb_ctx::kLabelsApplied;
  return SFB_OK;
}

int tc_labels(sfb_ctx* ctx) {
  if (ctx->labels == sfb_ctx::kLabelsApplied) {           // by the factors call of this step
    ctx->labels = sfb_ctx::kLabelsKept;
    return SFB_OK;
  }
  const Layout& L = ctx->lay;
  LabelArgs a = label_args(ctx, ctx->at<float>(L.Xf));
  a.again = ctx->labels == sfb_ctx::kLabelsKept;          // a repeated update
  if (!a.again)
    CKC(launch_kernel(label_slots_kernel, dim3(static_cast<unsigned>((ctx->K + 255) / 256)), dim3(256), 0, ctx->stream, 1,
                      ctx->at<int32_t>(L.labels), static_cast<int32_t>(ctx->K), ctx->cfg.rows, ctx->at<int32_t>(L.slot),
                      take_stamp(ctx)));
  CKC(launch_kernel(label_delta_kernel, dim3(static_cast<unsigned>(label_blocks(ctx))), dim3(256), 0, ctx->stream, 1, a));
  ctx->labels = sfb_ctx::kLabelsKept;
  return SFB_OK;
}

int tc_forward_partials(sfb_ctx* ctx, const float* X, const int32_t* labels, float* part_out) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  int tiles_n = 0;
  const int rc = mlr_forward(ctx, 0, ctx->K, X, labels, false, &tiles_n);
  if (rc) return rc;
  CKC(launch_kernel(mlr_shard_partials_tc_kernel, dim3(static_cast<unsigned>((ctx->K + 7) / 8)), dim3(256), 0,
                    ctx->stream, 1, ctx->at<float2>(L.part), ctx->K, tiles_n, ctx->at<float>(L.ZT), round_up(c.rows, 32),
                    c.rows, ctx->at<int32_t>(L.labels), ctx->row_offset, ctx->K, reinterpret_cast<float4*>(part_out)));
  return SFB_OK;
}

int tc_finish_factors(sfb_ctx* ctx, const float* parts, int shards) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t K = ctx->K;
  CKC(launch_kernel(mlr_shard_finish_tc_kernel, dim3(static_cast<unsigned>((K + 255) / 256)), dim3(256), 0, ctx->stream,
                    1, reinterpret_cast<const float4*>(parts), shards, K, c.rows, ctx->row_offset,
                    ctx->at<int32_t>(L.labels), ctx->at<float>(L.V), ctx->at<float>(L.loss), ctx->at<float>(L.coef),
                    ctx->at<uint32_t>(L.status)));
  return emit_p<false>(ctx, 0, K, ctx->at<int32_t>(L.labels), nullptr);
}

// What a worker sends (Section 3) in bf16 mode: u_ij = exp(z_ij - lse_i) - [j = y_i] in fp32 from the logits and the
// log-partition it holds; one block row per sample.
__global__ void __launch_bounds__(256) mlr_export_u_kernel(const float* __restrict__ Z, int64_t ldz, int64_t rows,
                                                           const float* __restrict__ lse,
                                                           const int32_t* __restrict__ labels,
                                                           int64_t off, float* __restrict__ U_out) {
  pdl_launch_dependents();
  pdl_wait(Z, lse, labels, U_out);
  const int64_t i = blockIdx.y;
  const float l = lse[off + i];
  const int32_t y = labels[off + i];
  const float* z = Z + (off + i) * ldz;
  float* u = U_out + i * rows;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; j < rows; j += stride)
    u[j] = expf(z[j] - l) - (j == y ? 1.f : 0.f);
}

// A received u = p - onehot(y): its smallest entry is the (only negative) one at y.  Per sample: the class, the fp32
// label coefficient 1 - p_y = -u_y and the loss -log p_y, as the local softmax pass leaves them.  One block per sample;
// ties (none for a valid u) go to the smaller index.
__global__ void __launch_bounds__(256) mlr_import_labels_kernel(const float* __restrict__ U_in, int64_t rows, int64_t off,
                                                                int32_t* __restrict__ labels, float* __restrict__ coef,
                                                                float* __restrict__ loss, int32_t* __restrict__ slot) {
  pdl_launch_dependents();
  pdl_wait(U_in, labels, coef, loss, slot);
  __shared__ float sv[256];
  __shared__ int32_t si[256];
  const int64_t i = blockIdx.x;
  const float* u = U_in + i * rows;
  float best = INFINITY;
  int32_t arg = 0;
  for (int64_t j = threadIdx.x; j < rows; j += 256) {
    const float v = u[j];
    if (v < best) { best = v; arg = static_cast<int32_t>(j); }
  }
  sv[threadIdx.x] = best; si[threadIdx.x] = arg;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      const float v = sv[threadIdx.x + o];
      const int32_t a = si[threadIdx.x + o];
      if (v < sv[threadIdx.x] || (v == sv[threadIdx.x] && a < si[threadIdx.x])) { sv[threadIdx.x] = v; si[threadIdx.x] = a; }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const float c = fminf(fmaxf(-sv[0], 0.f), 1.f);
    const int32_t old = labels[off + i];
    if (old >= 0 && old < rows) slot[old] = kNoSlot;
    labels[off + i] = si[0];
    coef[off + i] = c;
    loss[off + i] = -logf(fmaxf(1.f - c, 1e-37f));
  }
}

int tc_export_factors(sfb_ctx* ctx, int64_t off, int64_t n, float* U_out, float* V_out) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t ldz = round_up(c.rows, 32);
  dim3 grid(static_cast<unsigned>(std::min<int64_t>((c.rows + 255) / 256, 64)), static_cast<unsigned>(n));
  CKC(launch_kernel(mlr_export_u_kernel, grid, dim3(256), 0, ctx->stream, 1, ctx->at<float>(L.ZT), ldz, c.rows,
                    ctx->at<float>(L.V), ctx->at<int32_t>(L.labels), off, U_out));
  CKC(cudaMemcpyAsync(V_out, ctx->at<float>(L.Xf) + off * c.cols, static_cast<size_t>(n) * c.cols * 4, cudaMemcpyDeviceToDevice,
                      ctx->stream));
  return SFB_OK;
}

// Received fp32 factors take a worker's place in the bf16 layout: v as the bf16 operand and the fp32 sample copy, u as the bf16
// operand (0 at the class entry), the class entry into the fp32 label coefficients.
int tc_import_factors(sfb_ctx* ctx, int64_t off, int64_t n, const float* U_in, const float* V_in) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t rows = c.rows, cols = c.cols;
  const int64_t ldz = round_up(rows, 32);
  cudaStream_t s = ctx->stream;
  int32_t* labels = ctx->at<int32_t>(L.labels);
  ctx->labels = sfb_ctx::kLabelsNone;
  CKC(launch_kernel(mlr_import_labels_kernel, dim3(static_cast<unsigned>(n)), dim3(256), 0, s, 1, U_in, rows, off, labels,
                    ctx->at<float>(L.coef), ctx->at<float>(L.loss), ctx->at<int32_t>(L.slot)));
  float* Z = ctx->at<float>(L.ZT);
  CKC(cudaMemcpy2DAsync(Z + off * ldz, static_cast<size_t>(ldz) * 4, U_in, static_cast<size_t>(rows) * 4,
                        static_cast<size_t>(rows) * 4, static_cast<size_t>(n), cudaMemcpyDeviceToDevice, s));
  CKC(launch_kernel(pack_mlr_kernel, dim3(grid1d(n * cols / 4, 256)), dim3(256), 0, s, 1, V_in, n, cols,
                    ctx->at<__nv_bfloat16>(L.Xb), L.colsb, off, ctx->at<float>(L.Xf), labels + off, labels,
                    ctx->at<int32_t>(L.slot), rows, Stamp{}));
  return emit_p<true>(ctx, off, n, labels + off, nullptr);
}

// SDCA factors in bf16 mode: logits by the forward product, then the dual changes, solved in fp32, as the bf16 operand U (0 at
// the label entry, which goes to W in fp32 through coef, as for MLR).
int tc_sdca_factors(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const int32_t* labels, const int32_t* ids,
                    float inv_lam_n, bool fused) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t rows = c.rows;
  const int64_t ldz = round_up(rows, 32);
  float* Z = ctx->at<float>(L.ZT);
  int tiles_n = 0;
  const int rc = mlr_forward(ctx, off, n, X, labels, fused, &tiles_n);
  if (rc) return rc;
  SdcaArgs a = sdca_args(ctx, off, n, X, labels, ids, inv_lam_n);
  a.Z = Z + off * ldz; a.ldz = ldz;
  a.P = ctx->at<__nv_bfloat16>(L.P) + off * L.ldp; a.ldp = L.ldp;
  a.coef = ctx->at<float>(L.coef) + off;
  a.slot = fused ? ctx->at<int32_t>(L.slot) : nullptr;
  CKC(sdca_dual_rows(ctx->stream, a));
  if (fused) {
    CKC(launch_kernel(label_delta_kernel, dim3(static_cast<unsigned>(label_blocks(ctx))), dim3(256), 0, ctx->stream, 1,
                      label_args(ctx, X)));
    ctx->labels = sfb_ctx::kLabelsApplied;
  }
  return SFB_OK;
}

// Parts of at least 128 samples: copied at about 45 GB/s; a part's product takes its tensor work or one pass over the bf16 W.  With
// the copies and the products in line, first copy + the slower of the two per part + last product is what passes.
int tc_host_parts(const sfb_ctx* ctx) {
  const sfb_config& c = ctx->cfg;
  if (c.model != SFB_MLR || c.precision != SFB_PREC_BF16 || ctx->lay.split > 1) return 1;
  auto total = [&](int parts) {
    const int64_t n = ctx->K / parts;
    const double copy = 4.0 * static_cast<double>(n) * static_cast<double>(c.cols) / 45e9 + 4e-6;
    int cut = 1;
    const double cycles = logits_kernel(c, ctx->lay, n, true, &cut) == kLogitsPairs
                              ? forward_pair_cost(n, c.rows, c.cols)
                              : forward_cost(n, c.rows, c.cols, pick_forward_width(n, c.rows, c.cols, ctx->lay.pw, 1), 1);
    const double product = std::max(cycles / 1.7e9, 2.0 * static_cast<double>(c.rows) * static_cast<double>(c.cols) / 5e12) + 5e-6;
    // (a product that takes much longer than its copy has little to gain, and a pass over W per part to lose)
    return parts > 1 && product > 2. * copy ? 1e9 : copy + (parts - 1) * std::max(copy, product) + product;
  };
  int best = 1;
  for (int parts = 2; parts <= HostSide::kParts && ctx->K % (parts * BM) == 0; parts *= 2)
    if (total(parts) < 0.95 * total(best)) best = parts;
  return best;
}

int tc_factors(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const float* Y, const int32_t* labels, bool fused,
               float* dml_norm_out) {
  if (ctx->cfg.model == SFB_SC) return split_factors_sc(ctx, off, n, X);
  if (ctx->cfg.model == SFB_DML) {
    const Layout& L = ctx->lay;
    const int rc = split_logits(ctx, off, n, X, Y);                                     // z_i = W v_i
    if (rc) return rc;
    CKC(dml_scale_rows(ctx->stream, ctx->at<float>(L.U) + off * L.ldu, n, ctx->cfg.rows, L.ldu, labels, ctx->cfg.dml_margin,
                       ctx->at<uint16_t>(L.Rs) + off * 2 * L.rowsp, L.rowsp, nullptr, nullptr, dml_norm_out));
    return SFB_OK;
  }
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t rows = c.rows, K = ctx->K;
  const int64_t ldz = round_up(rows, 32);
  float* Z = ctx->at<float>(L.ZT);
  float* lse = ctx->at<float>(L.V);
  int tiles_n = 0;
  const int parts = ctx->host && ctx->host->parts > 1 ? ctx->host->parts : 1;
  for (int i = 0; i < parts; ++i) {                     // (parts: of samples that are still on their way, see sfb_step_host)
    const int64_t m = n / parts;
    if (parts > 1) CKC(cudaStreamWaitEvent(ctx->stream, ctx->host->part[i], 0));
    const int rc = mlr_forward(ctx, off + i * m, m, X + i * m * c.cols, labels + i * m, fused, &tiles_n);
    if (rc) return rc;
  }
  if (!fused && n <= 65535) {
    const int64_t most = (rows + 2047) / 2048, want = (4 * sm_count() + n - 1) / n;      // blocks of at least one pass over 2,048 classes
    CKC(launch_kernel(mlr_lse_emit_kernel, dim3(static_cast<unsigned>(std::min(most, want)), static_cast<unsigned>(n)), dim3(256), 0,
                      ctx->stream, 1, ctx->at<float2>(L.part), K, tiles_n, Z, ldz, rows, labels, off, lse, ctx->at<float>(L.loss),
                      ctx->at<float>(L.coef), ctx->at<__nv_bfloat16>(L.P), L.ldp, ctx->at<uint32_t>(L.status)));
    return SFB_OK;
  }
  if (fused && n == K && softmax_merged(n, c.cols, tiles_n)) {
    const int lab = label_blocks(ctx);
    CKC(launch_kernel(n > 4 * rows ? mlr_merged_kernel<true> : mlr_merged_kernel<false>, dim3(grid1d(n * ((rows + 7) / 8), 256) + lab), dim3(256), 0, ctx->stream, 1,
                      ctx->at<float2>(L.part), K, tiles_n, Z, ldz, rows, static_cast<int32_t>(n), labels, lse, ctx->at<float>(L.loss),
                      ctx->at<float>(L.coef), ctx->at<int32_t>(L.slot), ctx->at<__nv_bfloat16>(L.P), L.ldp, ctx->at<uint32_t>(L.status),
                      lab, label_args(ctx, X)));
    ctx->labels = sfb_ctx::kLabelsApplied;
    return SFB_OK;
  }
  CKC(launch_kernel(mlr_lse_kernel, dim3(static_cast<unsigned>((n + 7) / 8)), dim3(256), 0, ctx->stream, 1,
                    ctx->at<float2>(L.part), K, tiles_n, Z, ldz, rows, labels, off, n, lse, ctx->at<float>(L.loss),
                    ctx->at<float>(L.coef), fused ? ctx->at<int32_t>(L.slot) : nullptr, ctx->at<uint32_t>(L.status)));
  return emit_p<false>(ctx, off, n, labels, fused ? X : nullptr);
}

int tc_get_factors(sfb_ctx* ctx, const void** U, const void** V, int32_t* dtype, int32_t* layout, int64_t* ldu,
                   int64_t* ldv) {
  if (ctx->cfg.model != SFB_MLR) {   // the workers' fp32 factors, pair-major
    if (U) *U = ctx->at<float>(ctx->lay.U);
    if (V) *V = ctx->at<float>(ctx->lay.V);
    if (dtype) *dtype = 0;
    if (layout) *layout = 0;
    if (ldu) *ldu = ctx->lay.ldu;
    if (ldv) *ldv = ctx->cfg.cols;
    return SFB_OK;
  }
  if (U) *U = ctx->at<__nv_bfloat16>(ctx->lay.P);
  if (V) *V = ctx->at<__nv_bfloat16>(ctx->lay.Xb);
  if (dtype) *dtype = 1;
  if (layout) *layout = 0;
  if (ldu) *ldu = ctx->lay.ldp;
  if (ldv) *ldv = ctx->lay.colsb;
  return SFB_OK;
}

}  // namespace sfb
