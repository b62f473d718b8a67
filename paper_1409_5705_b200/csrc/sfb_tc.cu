// Tensor-core (bf16 operand) path of the SFB step on sm_100a: sufficient-factor computation for multiclass
// logistic regression (Sections 1 and 2: u = softmax(W x) - onehot(y), v = x) and the operand packing of the
// update product.  The update product itself is in sfb_update.cu.
//
// Forward product: one persistent, warp-specialised kernel computes  Z (K x rows) = X (K x cols) * W^T  with bf16
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

#ifndef SFB_SPLIT_PREFETCH
#define SFB_SPLIT_PREFETCH 4
#endif

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

// Epilogues of the product  D (samples x N) = A * B^T:
//   F_SOFTMAX  store D as fp32 logits and the softmax partials per (sample, pw columns)            (MLR; forward_kernel)
// and, in forward_split_kernel:
//   F_STORE    store D as fp32                                                                     (DML: z = W v)
//   F_SUB      store D - aux as fp32 and as a (hi | lo) bf16 pair                                  (SC: r = W a - x)
//   F_ISTA     C <- soft(C - D / L, lambda / L) in place, also as a (hi | lo) bf16 pair            (SC: ISTA step)
//   F_ISTAG    C <- soft(C - (D - C2) / L, lambda / L) in place, also as a pair                     (SC: on W^T W)
//   F_ISTA0    C2 = D and C = soft(D / L, lambda / L), also as a pair                               (SC: first iterate)
//   F_GRAM     C (unless null) = D and D as a pair, of a symmetric D: only the tiles that reach the diagonal or lie above
//              it are formed, the others are written as their mirror images                          (SC: W^T W)
enum FwdEpi { F_SOFTMAX = 0, F_STORE = 1, F_SUB = 2, F_ISTA = 3, F_ISTAG = 4, F_ISTA0 = 5, F_GRAM = 6 };
template <int EPI>
constexpr bool kIsta = EPI == F_ISTA || EPI == F_ISTAG || EPI == F_ISTA0;

struct TcParams {
  int32_t M, N, Kc;            // extents of the product: samples, output columns, contraction
  int32_t m_off;               // first sample handled by this launch (per-worker slices)
  int32_t tilesM, tilesN;
  int32_t a_rows;              // forward_kernel: rows of A per box (fewer than 128 for a slice of few samples; the rest of a
                               // tile's samples are then never stored)
  int32_t stages;              // forward_kernel: stages of the operand ring
  int32_t pw;                  // F_SOFTMAX: columns per softmax partial, a divisor of bn
  int32_t bn;                  // columns per tile, at most BN (chosen so that the tiles fill the SMs): a multiple of 32
                               // in forward_kernel, of 16 in forward_split_kernel
  // The contraction runs over nseg segments of kseg k-blocks; segment s reads A from column a_off<s> and B from
  // column b_off<s> of their tensors: one segment is the plain product, three segments over [hi | lo] operand
  // halves form the split-bf16 product hi*hi + hi*lo + lo*hi.  (Scalars: an indexed array would send the whole
  // parameter block to local memory.)
  int32_t nseg, kseg;
  int32_t a_off0, a_off1, a_off2, b_off0, b_off1, b_off2;
  float2* part;                // F_SOFTMAX: [N / pw][part_ld] (max, sum exp) per sample and pw rows of W
  int64_t part_ld;
  const float* aux;            // F_SUB: the matrix subtracted, [M x ldaux]; F_ISTA, F_ISTAG: the matrix updated
  int64_t ldaux;
  float* C2;                   // F_ISTA0 (may be null), F_ISTAG: W^T x, [M x ldc]
  int32_t prefetch;            // k-blocks by which the producer asks L2 for the B operand ahead of its loads (0: off)
  int32_t kparts;              // the contraction of a tile is cut over a cluster of this many CTAs (1: persistent CTAs)
  int32_t four;                // F_GRAM: with the fourth term A_lo B_lo
  const Scalars* sc;           // F_ISTA*: 1 / L
  float lam;                   // F_ISTA*: lambda
  __nv_bfloat16* split;        // all but F_STORE: [M x ld_split] receives hi at column n and lo at column split_half + n
  int64_t ld_split;
  int32_t split_half;          // padded N (a multiple of 64); columns N..split_half-1 are written as zeros
  uint32_t* status;
};

// Tiles are numbered with the sample block fastest: consecutive tiles (which run on different SMs at the same
// time) share one block of W, which therefore stays hot in L2 while all K samples are swept past it.
__device__ __forceinline__ void tile_coords(const TcParams& p, int tile, int& m0, int& n0) {
  const int tm = tile % p.tilesM, tn = tile / p.tilesM;
  m0 = p.m_off + tm * BM;
  n0 = tn * p.bn;
}

// F_GRAM: the tiles of column block tn that are formed are row blocks 0 .. sym_row_blocks - 1 (those that begin above the
// column block's end); numbered column block by column block.
__host__ __device__ __forceinline__ int sym_row_blocks(int tilesM, int bn, int tn) {
  const int n = ((tn + 1) * bn - 1) / BM + 1;
  return n < tilesM ? n : tilesM;
}
__host__ __device__ __forceinline__ int sym_tiles(int tilesM, int tilesN, int bn) {
  int n = 0;
  for (int tn = 0; tn < tilesN; ++tn) n += sym_row_blocks(tilesM, bn, tn);
  return n;
}
template <int EPI>
__device__ __forceinline__ void split_tile_coords(const TcParams& p, int tile, int& m0, int& n0) {
  if (EPI != F_GRAM) return tile_coords(p, tile, m0, n0);
  int tn = 0;
  for (int n; tile >= (n = sym_row_blocks(p.tilesM, p.bn, tn)); ++tn) tile -= n;
  m0 = tile * BM;
  n0 = tn * p.bn;
}

// Exchange of the partial tiles of a split contraction through the shared memory of the cluster's CTAs, in chunks of 32
// columns x 128 rows of fp32 (16 KB, the operand stages' memory, which nothing uses any more); a warp writes and reads its 32
// rows with the 16-byte pieces of a row swizzled.  Rank r then finishes the chunks c = r, r + split, ...; the sums are in rank
// order, so they do not depend on timing.
constexpr int kXchgBytes = BM * kChunk * 4;
__device__ __forceinline__ uint32_t xchg_addr(uint8_t* smem, int c, int row, int j) {
  return smem_u32(smem) + c * kXchgBytes + row * (kChunk * 4) + ((j ^ (row & 7)) << 4);
}
__device__ __forceinline__ void xchg_put(uint8_t* smem, int c, int row, const uint32_t (&acc)[32]) {
#pragma unroll
  for (int j = 0; j < 8; ++j)
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(xchg_addr(smem, c, row, j)), "r"(acc[4 * j]), "r"(acc[4 * j + 1]),
                 "r"(acc[4 * j + 2]), "r"(acc[4 * j + 3]) : "memory");
}
__device__ __forceinline__ void xchg_sum(uint8_t* smem, int c, int row, int split, uint32_t (&acc)[32]) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t at = xchg_addr(smem, c, row, j);
    float4 s = ld_cluster_f4(at, 0);
    for (int g = 1; g < split; ++g) {
      const float4 v = ld_cluster_f4(at, g);
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

// TF32: the operands are 32-bit words read as tf32 (a k-block of 128 bytes is then 32 elements and one MMA contracts
// 8 of them); everything else -- stages, descriptors, epilogues -- is the same.
template <int EPI, bool TF32 = false>
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

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
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
    if (lane == 0) {
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
            if (!mbar_wait(&empty[s], ph ^ 1, abort_flag)) { ok = false; break; }
            // B streams from HBM when it is larger than L2: with the box asked for a few k-blocks early, the load
            // that fills the stage finds it in L2 and the four stages cover the latency
            if (p.prefetch > 0 && kl + p.prefetch < p.kseg)
              tma_prefetch_2d(&tmB, xb0 + (kl + p.prefetch) * (TF32 ? BK / 2 : BK), n0);
            uint8_t* st = smem + s * stage_bytes;
            mbar_expect_tx(&full[s], (p.a_rows + p.bn) * BK * 2);
            tma_load_2d_hint(st, &tmA, xa0 + kl * (TF32 ? BK / 2 : BK), m0, &full[s], pol_keep);
            tma_load_2d(st + kBytesA, &tmB, xb0 + kl * (TF32 ? BK / 2 : BK), n0, &full[s]);
            if (++s == static_cast<uint32_t>(ST)) { s = 0; ph ^= 1; }
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      const uint32_t idesc = TF32 ? umma_idesc_tf32(BM, p.bn) : umma_idesc_bf16(BM, p.bn);
      uint32_t s = 0, ph = 0, tl = 0;
      bool ok = true;
      for (int tile = tile0; tile < ntiles && ok; tile += tile_step, ++tl) {
        const uint32_t a = tl & 1, aph = (tl >> 1) & 1;
        if (!mbar_wait(&tempty[a], aph ^ 1, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + a * BN;
        for (int kb = 0; kb < kend - kbeg; ++kb) {
          if (!mbar_wait(&full[s], ph, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint64_t da = umma_desc_k128(smem_u32(smem + s * stage_bytes));
          const uint64_t db = umma_desc_k128(smem_u32(smem + s * stage_bytes + kBytesA));
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k) {          // four MMAs of 32 bytes of contraction each, either kind
            const uint64_t adv = static_cast<uint64_t>(k * UMMA_K * 2 / 16);
            if (TF32) umma_tf32(d_tmem, da + adv, db + adv, idesc, (kb | k) != 0 ? 1u : 0u);
            else umma_bf16(d_tmem, da + adv, db + adv, idesc, (kb | k) != 0 ? 1u : 0u);
          }
          umma_commit(&empty[s]);          // the stage is free once these MMAs have read it
          if (++s == static_cast<uint32_t>(ST)) { s = 0; ph ^= 1; }
        }
        if (ok) umma_commit(&tfull[a]);    // the accumulator is complete once every MMA of the tile is
      }
    }
  } else {
    // ---------------- epilogue: warps 2..5, TMEM lane quarter q ----------------
    const int q = warp & 3;
    uint8_t* ring = sRing + q * R * kSlotBytes;
    const int my_tiles = tile0 < ntiles ? (ntiles - 1 - tile0) / tile_step + 1 : 0;
    bool ok = true;
    // The fp32 result goes out through the ring by TMA; F_SOFTMAX keeps a running (max, sum exp) per sample.
    uint32_t gs = 0;                       // stores issued so far: consecutive stores alternate ring slots
    float mx = -INFINITY, sum = 0.f;
    auto finish = [&](uint32_t (&acc)[32], int m0, int n0, int c) {
      uint8_t* sl = ring + (gs % R) * kSlotBytes;
      const int col0 = n0 + c * kChunk, row = m0 + q * 32 + lane;
      if (col0 < p.N) {
        if constexpr (EPI == F_SOFTMAX) {
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
        }
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
      if (EPI == F_SOFTMAX && ((c + 1) * kChunk) % p.pw == 0) {      // the end of a group of pw columns
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
// Split-bf16 products of distance metric learning and sparse coding:  D (samples x N) = A * B^T  with both operands
// stored as [hi | lo] bf16 halves,  A_hi B_hi + A_lo B_hi + A_hi B_lo  (fp32-class accuracy; A_lo B_lo, 2^-16 of the
// product, is dropped).  One pipeline stage holds the k-block of all four halves, and the three products of that
// k-block are issued from it: 72 KB of operands per three k-blocks of tensor work instead of 108 KB when the three
// products run as separate passes over the contraction (these products are bound by their operand loads: a 128 x 160
// tile takes 36 KB per 320 cycles of MMA).  Three stages of 72 KB fill the shared memory, so the epilogue writes its
// results straight from registers (the outputs are small: samples x N).  The cross terms have an accumulator of their own: the
// tensor core rounds an fp32 accumulator at every instruction relative to what it holds, so two thirds of the roundings happen
// at a 2^-8 of the size.
// Roles as in forward_kernel: warp 0 TMA producer, warp 1 MMA issuer and TMEM owner, warps 2-5 epilogue.
// ---------------------------------------------------------------------------------------------------------
constexpr int FS_BN = 160;                          // widest tile of this kernel (columns of the accumulator)
constexpr int FS_STAGES = 3;
constexpr int kFsBytesB = FS_BN * BK * 2;           // 20 KB
constexpr int kFsStage = 2 * kBytesA + 2 * kFsBytesB;
constexpr int kFsBars = 2 * FS_STAGES + 4;
constexpr int kFsEpi = 8;                           // epilogue warps: two per TMEM lane quarter, taking turns at the chunks
constexpr int kFsThreads = 64 + 32 * kFsEpi;
constexpr int kFsSmem = FS_STAGES * kFsStage + kFsBars * 8 + 16 + 1024;

template <int EPI>
__global__ void __launch_bounds__(kFsThreads, 1)
forward_split_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, float* __restrict__ C,
                     int64_t ldc, const TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + FS_STAGES * kFsStage);
  uint64_t* full = bars;
  uint64_t* empty = bars + FS_STAGES;
  uint64_t* tfull = bars + 2 * FS_STAGES;
  uint64_t* tempty = bars + 2 * FS_STAGES + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kFsBars);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ntiles = EPI == F_GRAM ? sym_tiles(p.tilesM, p.tilesN, p.bn) : p.tilesM * p.tilesN;
  // the tiles and k-blocks (each serves three products) of this CTA, as in forward_kernel
  const int split = p.kparts, part = split > 1 ? static_cast<int>(blockIdx.x) % split : 0;
  const int tile0 = static_cast<int>(blockIdx.x) / split, tile_step = split > 1 ? ntiles : static_cast<int>(gridDim.x);
  const int kbeg = part * p.kseg / split, kend = (part + 1) * p.kseg / split;
  // Two accumulators per tile: A_hi B_hi, and the cross terms at column `cross` of it.  Tiles of at most 128 columns have room
  // for two such pairs (the epilogue of one tile then overlaps the products of the next), wider ones for one.
  const int nacc = p.bn <= 128 ? 2 : 1, cross = p.bn <= 128 ? 128 : 256;
  const int a_hi = p.a_off0, a_lo = p.a_off2, b_hi = p.b_off0, b_lo = p.b_off1;

  pdl_launch_dependents();
  if (threadIdx.x == 0) {
    for (int i = 0; i < FS_STAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], kFsEpi); }
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&tmA); prefetch_tmap(&tmB);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, kTmemCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();

  if (warp == 0) {
    // ---------------- TMA producer: the four operand halves of a k-block per stage ----------------
    if (lane == 0) {
      const uint64_t pol_keep = policy_evict_last();
      const uint32_t stage_bytes = 2 * kBytesA + 2 * static_cast<uint32_t>(p.bn) * BK * 2;
      uint32_t it = 0;
      bool ok = true;
      for (int tile = tile0; tile < ntiles && ok; tile += tile_step) {
        int m0, n0;
        split_tile_coords<EPI>(p, tile, m0, n0);
        for (int kl = kbeg; kl < kend; ++kl, ++it) {
          const uint32_t s = it % FS_STAGES, ph = (it / FS_STAGES) & 1;
          if (!mbar_wait(&empty[s], ph ^ 1, abort_flag)) { ok = false; break; }
          if (p.prefetch > 0 && kl + p.prefetch < kend) {          // B streams from HBM when it is larger than L2
            tma_prefetch_2d(&tmB, b_hi + (kl + p.prefetch) * BK, n0);
            tma_prefetch_2d(&tmB, b_lo + (kl + p.prefetch) * BK, n0);
          }
          uint8_t* st = smem + s * kFsStage;
          mbar_expect_tx(&full[s], stage_bytes);
          tma_load_2d_hint(st, &tmA, a_hi + kl * BK, m0, &full[s], pol_keep);
          tma_load_2d_hint(st + kBytesA, &tmA, a_lo + kl * BK, m0, &full[s], pol_keep);
          tma_load_2d(st + 2 * kBytesA, &tmB, b_hi + kl * BK, n0, &full[s]);
          tma_load_2d(st + 2 * kBytesA + kFsBytesB, &tmB, b_lo + kl * BK, n0, &full[s]);
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: three products per stage ----------------
    if (lane == 0) {
      const uint32_t idesc = umma_idesc_bf16(BM, p.bn);
      uint32_t it = 0, tl = 0;
      bool ok = true;
      for (int tile = tile0; tile < ntiles && ok; tile += tile_step, ++tl) {
        const uint32_t a = tl % nacc, aph = (tl / nacc) & 1;
        if (!mbar_wait(&tempty[a], aph ^ 1, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + a * BN, d_cross = d_tmem + cross;
        for (int kb = 0; kb < kend - kbeg; ++kb, ++it) {
          const uint32_t s = it % FS_STAGES, ph = (it / FS_STAGES) & 1;
          if (!mbar_wait(&full[s], ph, abort_flag)) { ok = false; break; }
          tc_fence_after();
          uint8_t* st = smem + s * kFsStage;
          const uint64_t dah = umma_desc_k128(smem_u32(st));
          const uint64_t dal = umma_desc_k128(smem_u32(st + kBytesA));
          const uint64_t dbh = umma_desc_k128(smem_u32(st + 2 * kBytesA));
          const uint64_t dbl = umma_desc_k128(smem_u32(st + 2 * kBytesA + kFsBytesB));
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k) {
            const uint64_t adv = static_cast<uint64_t>(k * UMMA_K * 2 / 16);
            const uint32_t more = (kb | k) != 0 ? 1u : 0u;
            umma_bf16(d_cross, dal + adv, dbh + adv, idesc, more);                       // A_lo B_hi
            umma_bf16(d_cross, dah + adv, dbl + adv, idesc, 1u);                         // A_hi B_lo
            if (EPI == F_GRAM && p.four) umma_bf16(d_cross, dal + adv, dbl + adv, idesc, 1u);    // A_lo B_lo
            umma_bf16(d_tmem, dah + adv, dbh + adv, idesc, more);                        // A_hi B_hi
          }
          umma_commit(&empty[s]);
        }
        if (ok) umma_commit(&tfull[a]);
      }
    }
  } else {
    // ---------------- epilogue: warp (q, h) = TMEM lane quarter q, every second chunk; results leave straight from registers
    const int q = warp & 3, h = (warp - 2) >> 2;
    const int my_tiles = tile0 < ntiles ? (ntiles - 1 - tile0) / tile_step + 1 : 0;
    bool ok = true;
    float invL = 0.f, thr = 0.f;
    if (kIsta<EPI>) { invL = p.sc->invL; thr = p.lam * invL; }
    auto finish = [&](uint32_t (&acc)[32], int m0, int n0, int c) {
      const int row = m0 + q * 32 + lane;
      // the tile's columns end at nlim; its width is a multiple of 16, so the last 32-column chunk may be half used
      const int nlim = min(p.N, n0 + p.bn);
      const int col0 = n0 + c * kChunk;
      if (col0 >= nlim || row >= p.M) return;
      if constexpr (EPI == F_ISTAG || EPI == F_ISTA0) {
        // W^T x of the sample (N, hence every pitch, is a multiple of 4 for the products over atoms)
        float* bp = p.C2 ? p.C2 + static_cast<int64_t>(row) * ldc + col0 : nullptr;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (!bp || col0 + 4 * j + 4 > nlim) continue;
          if constexpr (EPI == F_ISTAG) {
            const float4 b4 = *reinterpret_cast<const float4*>(bp + 4 * j);
            acc[4 * j] = __float_as_uint(__uint_as_float(acc[4 * j]) - b4.x);
            acc[4 * j + 1] = __float_as_uint(__uint_as_float(acc[4 * j + 1]) - b4.y);
            acc[4 * j + 2] = __float_as_uint(__uint_as_float(acc[4 * j + 2]) - b4.z);
            acc[4 * j + 3] = __float_as_uint(__uint_as_float(acc[4 * j + 3]) - b4.w);
          } else {
            *reinterpret_cast<uint4*>(bp + 4 * j) = make_uint4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
          }
        }
      }
      if constexpr (EPI != F_STORE) {
        if constexpr (EPI == F_SUB || EPI == F_ISTA || EPI == F_ISTAG) {
          // the sample's values of aux (x, or the current code a) are contiguous: up to 128 bytes per lane
          float xv[32];
          const float* ap = p.aux + static_cast<int64_t>(row) * p.ldaux + col0;
          const bool ap16 = (reinterpret_cast<uintptr_t>(ap) & 15u) == 0;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (ap16 && col0 + 4 * j + 4 <= nlim) {
              const float4 v4 = *reinterpret_cast<const float4*>(ap + 4 * j);
              xv[4 * j] = v4.x; xv[4 * j + 1] = v4.y; xv[4 * j + 2] = v4.z; xv[4 * j + 3] = v4.w;
            } else {
#pragma unroll
              for (int e = 0; e < 4; ++e) xv[4 * j + e] = col0 + 4 * j + e < nlim ? ap[4 * j + e] : 0.f;
            }
          }
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const float d = __uint_as_float(acc[j]);
            acc[j] = __float_as_uint(EPI == F_SUB ? d - xv[j] : soft_threshold(fmaf(-d, invL, xv[j]), thr));
          }
        }
        if constexpr (EPI == F_ISTA0) {
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[j] = __float_as_uint(soft_threshold(__uint_as_float(acc[j]) * invL, thr));
        }
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = col0 + j < p.N ? acc[j] : 0u;
        // (hi | lo) bf16 pair of the result: the operand of the next product (zero in the padding past N; the
        // columns past this tile's width belong to the next tile)
        __nv_bfloat16* hp = p.split + static_cast<int64_t>(row) * p.ld_split + col0;
        const int split_lim = min(p.split_half, n0 + p.bn);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (col0 + 8 * j < split_lim) {
            uint32_t hi[4], lo[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float f0 = __uint_as_float(acc[8 * j + 2 * e]), f1 = __uint_as_float(acc[8 * j + 2 * e + 1]);
              const __nv_bfloat16 h0 = __float2bfloat16_rn(f0), h1 = __float2bfloat16_rn(f1);
              hi[e] = static_cast<uint32_t>(__bfloat16_as_ushort(h0)) |
                      (static_cast<uint32_t>(__bfloat16_as_ushort(h1)) << 16);
              const __nv_bfloat162 l2 = __floats2bfloat162_rn(f0 - __bfloat162float(h0), f1 - __bfloat162float(h1));
              lo[e] = *reinterpret_cast<const uint32_t*>(&l2);
            }
            *reinterpret_cast<uint4*>(hp + 8 * j) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4*>(hp + p.split_half + 8 * j) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
          }
        }
      }
      if constexpr (EPI == F_GRAM) {
        // the mirror images of the entries whose own tile is not formed: lanes are neighbouring columns there
        const int own_end = (row / p.bn + 1) * p.bn;              // end of the column block that row lies in
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const int n = col0 + j;
          if (n >= nlim || own_end > n / BM * BM) continue;
          const float f = __uint_as_float(acc[j]);
          const __nv_bfloat16 hi = __float2bfloat16_rn(f);
          __nv_bfloat16* hp = p.split + static_cast<int64_t>(n) * p.ld_split + row;
          hp[0] = hi;
          hp[p.split_half] = __float2bfloat16_rn(f - __bfloat162float(hi));
          if (C) C[static_cast<int64_t>(n) * ldc + row] = f;
        }
        if (!C) return;
      }
      // the fp32 result: this lane's consecutive columns of its row
      float* cp = C + static_cast<int64_t>(row) * ldc + col0;
      const bool cp16 = (reinterpret_cast<uintptr_t>(cp) & 15u) == 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (cp16 && col0 + 4 * j + 4 <= nlim) {
          *reinterpret_cast<uint4*>(cp + 4 * j) = make_uint4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (col0 + 4 * j + e < nlim) cp[4 * j + e] = __uint_as_float(acc[4 * j + e]);
        }
      }
    };
    const int chunks = (p.bn + kChunk - 1) / kChunk;
    for (int tl = 0; tl < my_tiles && ok; ++tl) {
      int m0, n0;
      split_tile_coords<EPI>(p, tile0 + tl * tile_step, m0, n0);
      const uint32_t a = tl % nacc, aph = (tl / nacc) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(&tfull[a], aph, abort_flag))) { ok = false; break; }
      tc_fence_after();
      for (int c = h; c < chunks; c += 2) {
        uint32_t acc[32];
        {
          uint32_t small[32];
          const uint32_t at = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + a * BN + c * kChunk;
          tmem_ld_32x32(at, acc);
          tmem_ld_32x32(at + cross, small);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[j] = __float_as_uint(__uint_as_float(acc[j]) + __uint_as_float(small[j]));
        }
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
      split_tile_coords<EPI>(p, tile0, m0, n0);
      for (int c = part + split * h; c < chunks && ok; c += 2 * split) {
        uint32_t acc[32];
        xchg_sum(smem, c, q * 32 + lane, split, acc);
        finish(acc, m0, n0, c);
      }
    }
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
  pdl_wait();
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
constexpr int32_t kNoSlot = 0x7f7f7f7f;              // above every sample index (K <= 2^20)
__global__ void __launch_bounds__(256) pack_mlr_kernel(const float* __restrict__ X, int64_t n, int64_t cols,
                                                       __nv_bfloat16* __restrict__ Xb, int64_t ldx, int64_t off,
                                                       float* __restrict__ Xf, const int32_t* labels, int32_t* labels_out,
                                                       int32_t* __restrict__ slot, int64_t rows, const Stamp stamp) {
  pdl_launch_dependents();
  pdl_wait();
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

// W [n x dim] -> its transpose as a (hi | lo) bf16 operand FT [dim x 2*Kp] (the coder's W^T): FT[c][i] = hi(F[i][c]),
// FT[c][Kp + i] = lo(F[i][c]) with hi = bf16(f), lo = bf16(f - hi); rows n..Kp-1 are written as zeros.  64 x 64 tiles through
// shared memory.
__global__ void __launch_bounds__(256) pack_split_t_kernel(const float* __restrict__ F, int64_t n, int64_t dim,
                                                           int64_t ld, __nv_bfloat16* __restrict__ FT, int64_t Kp) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ float tile[64][65];
  const int64_t i0 = static_cast<int64_t>(blockIdx.y) * 64, c0 = static_cast<int64_t>(blockIdx.x) * 64;
  const int t = threadIdx.x;
  const bool vec = (ld % 4) == 0;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const int idx = t + v * 256;            // 64 samples x 16 quads
    const int i = idx / 16, cq = (idx % 16) * 4;
    float f[4] = {0.f, 0.f, 0.f, 0.f};
    if (i0 + i < n) {
      const float* src = F + (i0 + i) * ld + c0 + cq;
      if (vec && c0 + cq + 3 < dim) {
        const float4 q4 = *reinterpret_cast<const float4*>(src);
        f[0] = q4.x; f[1] = q4.y; f[2] = q4.z; f[3] = q4.w;
      } else {
        for (int k = 0; k < 4; ++k)
          if (c0 + cq + k < dim) f[k] = src[k];
      }
    }
    tile[i][cq + 0] = f[0]; tile[i][cq + 1] = f[1]; tile[i][cq + 2] = f[2]; tile[i][cq + 3] = f[3];
  }
  __syncthreads();
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    const int idx = t + v * 256;            // 64 features x 8 groups of 8 samples
    const int c = idx / 8, ig = (idx % 8) * 8;
    if (c0 + c >= dim) continue;
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float f0 = tile[ig + 2 * k][c], f1 = tile[ig + 2 * k + 1][c];
      const __nv_bfloat16 h0 = __float2bfloat16_rn(f0), h1 = __float2bfloat16_rn(f1);
      hi[k] = static_cast<uint32_t>(__bfloat16_as_ushort(h0)) | (static_cast<uint32_t>(__bfloat16_as_ushort(h1)) << 16);
      lo[k] = pack_bf16(f0 - __bfloat162float(h0), f1 - __bfloat162float(h1));
    }
    __nv_bfloat16* dst = FT + (c0 + c) * 2 * Kp + i0 + ig;     // Kp is a multiple of 64: 16-byte aligned
    *reinterpret_cast<uint4*>(dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(dst + Kp) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

// fp32 [n x dim] (row pitch ld) -> the (hi | lo) bf16 operand [n x 2*dimp], no transpose: dst[r][c] = hi,
// dst[r][dimp + c] = lo with hi = bf16(f), lo = bf16(f - hi).  Columns dim..dimp-1 are left as they are (zero since
// set-up).
__global__ void __launch_bounds__(256) pack_split_rows_kernel(const float* __restrict__ F, int64_t n, int64_t dim,
                                                              int64_t ld, __nv_bfloat16* __restrict__ dst, int64_t dimp,
                                                              const Stamp stamp) {
  pdl_launch_dependents();
  pdl_wait();
  stamp_begin(stamp);
  const int64_t quads = (dim + 3) / 4, total = n * quads;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const bool vec = ld % 4 == 0 && dim % 4 == 0;          // else (samples with an odd number of features) value by value
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < total; i += stride) {
    const int64_t r = i / quads, qd = i % quads;
    const float* src = F + r * ld + qd * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (vec) {
      v = *reinterpret_cast<const float4*>(src);
    } else {
      v.x = src[0];
      if (qd * 4 + 1 < dim) v.y = src[1];
      if (qd * 4 + 2 < dim) v.z = src[2];
      if (qd * 4 + 3 < dim) v.w = src[3];
    }
    const __nv_bfloat16 h0 = __float2bfloat16_rn(v.x), h1 = __float2bfloat16_rn(v.y), h2 = __float2bfloat16_rn(v.z),
                        h3 = __float2bfloat16_rn(v.w);
    __nv_bfloat16* d = dst + r * 2 * dimp + qd * 4;
    *reinterpret_cast<uint2*>(d) =
        make_uint2(static_cast<uint32_t>(__bfloat16_as_ushort(h0)) | (static_cast<uint32_t>(__bfloat16_as_ushort(h1)) << 16),
                   static_cast<uint32_t>(__bfloat16_as_ushort(h2)) | (static_cast<uint32_t>(__bfloat16_as_ushort(h3)) << 16));
    *reinterpret_cast<uint2*>(d + dimp) = make_uint2(pack_bf16(v.x - __bfloat162float(h0), v.y - __bfloat162float(h1)),
                                                     pack_bf16(v.z - __bfloat162float(h2), v.w - __bfloat162float(h3)));
  }
}

// DML: v = x - y of n pairs (Section 2) in fp32 and as the (hi | lo) operand, one pass (16 bytes per value; as two kernels 24).
__global__ void __launch_bounds__(256) pack_pairs_kernel(const float* __restrict__ X, const float* __restrict__ Y, int64_t n,
                                                         int64_t dim, float* __restrict__ V,
                                                         __nv_bfloat16* __restrict__ dst,
                                                         int64_t dimp, const Stamp stamp) {
  pdl_launch_dependents();
  pdl_wait();
  stamp_begin(stamp);
  const uint32_t quads = static_cast<uint32_t>(dim / 4);
  const int64_t total = n * quads, stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t q = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; q < total; q += stride) {
    const int64_t i = q / quads, c = (q - i * quads) * 4;
    const float4 x = reinterpret_cast<const float4*>(X)[q], y = reinterpret_cast<const float4*>(Y)[q];
    const float4 v = make_float4(x.x - y.x, x.y - y.y, x.z - y.z, x.w - y.w);
    reinterpret_cast<float4*>(V)[q] = v;
    const uint32_t h01 = pack_bf16(v.x, v.y), h23 = pack_bf16(v.z, v.w);
    const float2 f01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h01));
    const float2 f23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&h23));
    __nv_bfloat16* d = dst + i * 2 * dimp + c;
    *reinterpret_cast<uint2*>(d) = make_uint2(h01, h23);
    *reinterpret_cast<uint2*>(d + dimp) = make_uint2(pack_bf16(v.x - f01.x, v.y - f01.y), pack_bf16(v.z - f23.x, v.w - f23.y));
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
  pdl_wait();
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
  pdl_wait();
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
  pdl_wait();
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
  pdl_wait();
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
  pdl_wait();
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
  pdl_wait();
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
  pdl_wait();
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
  pdl_wait();
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
template <int EPI, bool TF32 = false>
cudaError_t launch_forward(sfb_ctx* ctx, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& c, TcParams p) {
  TcState* st = static_cast<TcState*>(ctx->tc);
  const int64_t tiles = static_cast<int64_t>(p.tilesM) * p.tilesN;
  if (tiles <= 0) return cudaSuccess;
  const unsigned grid = static_cast<unsigned>(p.kparts > 1 ? tiles * p.kparts : std::min<int64_t>(tiles, st->sms));
  return launch_kernel_if(tiles * p.kparts <= st->sms, forward_kernel<EPI, TF32>, dim3(grid), dim3(kThreads), kSmem, ctx->stream,
                          p.kparts, a, b, c, p);
}

template <int EPI>
cudaError_t launch_forward_split(sfb_ctx* ctx, const CUtensorMap& a, const CUtensorMap& b, float* C, int64_t ldc, TcParams p) {
  TcState* st = static_cast<TcState*>(ctx->tc);
  const int64_t tiles = EPI == F_GRAM ? sym_tiles(p.tilesM, p.tilesN, p.bn) : static_cast<int64_t>(p.tilesM) * p.tilesN;
  if (tiles <= 0) return cudaSuccess;
  const unsigned grid = static_cast<unsigned>(p.kparts > 1 ? tiles * p.kparts : std::min<int64_t>(tiles, st->sms));
  return launch_kernel_if(tiles * p.kparts <= st->sms, forward_split_kernel<EPI>, dim3(grid), dim3(kFsThreads), kFsSmem, ctx->stream,
                          p.kparts, a, b, C, ldc, p);
}

// The shared-memory opt-in is a per-device attribute of each kernel: set for every instantiation when a context is
// created (with its device current), not once per process.
cudaError_t prepare_forward_kernels() {
  cudaError_t e = cudaFuncSetAttribute(forward_kernel<F_SOFTMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(forward_split_kernel<F_STORE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFsSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(forward_split_kernel<F_SUB>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFsSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(forward_split_kernel<F_ISTA>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFsSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(forward_split_kernel<F_ISTAG>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFsSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(forward_split_kernel<F_ISTA0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFsSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(forward_split_kernel<F_GRAM>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFsSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(forward_kernel<F_SOFTMAX, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
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
  const double rounds = static_cast<double>((ctas + sm_count() - 1) / sm_count());
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
// 14,240 columns: 223 k-blocks in a row on one SM, 68 us).  One choice per context: it fixes the order of the sums.
static int pick_forward_split(int64_t K, int64_t rows, int64_t cols) {
  int best = 1;
  double cost = forward_cost(K, rows, cols, pick_forward_width(K, rows, cols, 32, 1), 1);
  for (int s = 2; s <= 8 && (cols + BK - 1) / BK >= 2 * s; s *= 2) {
    const double c = forward_cost(K, rows, cols, pick_forward_width(K, rows, cols, 32, s), s);
    if (c < 0.9 * cost) { cost = c; best = s; }
  }
  return best;
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
  if (c.model != SFB_MLR) {
    // fp32 factors as the workers write them, and the split-bf16 operands of the forward and update products
    L.colsp = round_up(c.cols, 64);
    L.rowsp = round_up(c.rows, 64);
    L.ldu = round_up(c.rows, 4);                                        // TMA stores need a 16-byte row pitch
    L.V = take(K * static_cast<size_t>(c.cols) * 4);
    L.U = take(K * static_cast<size_t>(L.ldu) * 4);
    L.Rs = take(K * 2 * static_cast<size_t>(L.rowsp) * 2);              // u (SC: first x, then the residuals)
    L.Ws = take(static_cast<size_t>(c.rows) * 2 * L.colsp * 2);         // W, rows x (hi | lo)
    L.As = take(K * 2 * static_cast<size_t>(L.colsp) * 2);              // v (DML) or the codes a (SC)
    if (c.model == SFB_SC) {
      L.WTs = take(static_cast<size_t>(c.cols) * 2 * L.rowsp * 2);      // W^T, atoms x (hi | lo)
      if (sc_use_gram(c)) {
        L.Gs = take(static_cast<size_t>(c.cols) * 2 * L.colsp * 2);     // W^T W, atoms x (hi | lo)
        L.G = take(c.sc_lipschitz > 0.f ? 0 : static_cast<size_t>(c.cols) * c.cols * 4);   // in fp32 for the power iteration
        L.Bx = take(K * static_cast<size_t>(c.cols) * 4);               // W^T x
        L.As2 = take(K * 2 * static_cast<size_t>(L.colsp) * 2);         // the codes of every other iteration
      }
    }
    return;
  }
  const size_t ldz = static_cast<size_t>(round_up(c.rows, 32));
  L.split = pick_forward_split(static_cast<int64_t>(K), c.rows, c.cols);
  L.pw = L.split > 1 ? 32 : pick_forward_width(c.batch, c.rows, c.cols, 32, 1);
  const size_t nblk = static_cast<size_t>((c.rows + L.pw - 1) / L.pw);
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
  if (c.model != SFB_MLR) {
    // pad columns of the split operands are never written by the kernels: clear the buffers once
    const Layout& L = ctx->lay;
    const size_t K = static_cast<size_t>(ctx->K);
    CKC(cudaMemsetAsync(ctx->at<char>(L.Ws), 0, static_cast<size_t>(c.rows) * 2 * L.colsp * 2, ctx->stream));
    CKC(cudaMemsetAsync(ctx->at<char>(L.As), 0, K * 2 * L.colsp * 2, ctx->stream));
    CKC(cudaMemsetAsync(ctx->at<char>(L.Rs), 0, K * 2 * L.rowsp * 2, ctx->stream));
    if (c.model == SFB_SC) {
      CKC(cudaMemsetAsync(ctx->at<char>(L.WTs), 0, static_cast<size_t>(c.cols) * 2 * L.rowsp * 2, ctx->stream));
      if (L.Gs) {
        CKC(cudaMemsetAsync(ctx->at<char>(L.Gs), 0, static_cast<size_t>(c.cols) * 2 * L.colsp * 2, ctx->stream));
        CKC(cudaMemsetAsync(ctx->at<char>(L.As2), 0, K * 2 * L.colsp * 2, ctx->stream));
      }
    }
    return SFB_OK;
  }
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

namespace {

inline unsigned grid1d(int64_t items, int per_block) {
  int64_t g = (items + per_block - 1) / per_block;
  return static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(g, static_cast<int64_t>(sm_count()) * 16)));
}

// Tile width (a multiple of `step` columns, at most `widest`) for a product with tilesM row blocks and N columns on
// `sms` SMs.  The
// persistent kernel runs ceil(tiles / sms) rounds of tiles; measured, a tile costs about max(width, 128) + 16
// column-equivalents (below 128 columns a k-block is bound by the latency of its operand loads, not by the MMA).
// Narrower tiles fill the SMs of small products, where 256-wide ones leave many idle or need a nearly empty
// second round; ties go to the wider tile.
inline int pick_tile_width(int sms, int64_t tilesM, int64_t N, int widest, int step = 32, bool sym = false) {
  int best = widest;
  int64_t best_cost = INT64_MAX;
  if (N <= 112) return static_cast<int>(round_up(N, step));
  for (int bn = widest; bn >= 128; bn -= step) {
    const int64_t tn = (N + bn - 1) / bn;
    const int64_t tiles = sym ? sym_tiles(static_cast<int>(tilesM), static_cast<int>(tn), bn) : tilesM * tn;
    const int64_t cost = ((tiles + sms - 1) / sms) * (bn + 16);
    if (cost < best_cost) { best_cost = cost; best = bn; }
  }
  return best;
}

// Features up to which the coder on W^T W forms W^T x by fp32 FMAs and W^T W with its fourth term.  Every iterate carries
// their error, and for short contractions the rounding of the operands to pairs is most of it (for long ones it is the
// tensor core's own rounding, which the second accumulator brought down).  Error of the codes with / without, and with two
// products per iteration: 700 x 400: 3.7e-6 / 9.1e-6, 5.0e-6; 1,501 x 1,400: 5.1e-6 / 9.9e-6, 7.3e-6.
constexpr int64_t kPreciseRows = 2048;

constexpr int kSplitPrefetch = SFB_SPLIT_PREFETCH;    // k-blocks of look-ahead of the L2 prefetch in the split products

// Cost of a split product in rounds of tiles x columns x k-blocks, its contraction in `split` parts.
double split_cost(int64_t M, int64_t N, int64_t Kc, bool sym, int split) {
  const int sms = sm_count();
  const int64_t tm = (M + BM - 1) / BM;
  const int bn = pick_tile_width(sms / split, tm, N, FS_BN, 16, sym);
  const int64_t tn = (N + bn - 1) / bn;
  const int64_t tiles = sym ? sym_tiles(static_cast<int>(tm), static_cast<int>(tn), bn) : tm * tn;
  const double kb = static_cast<double>((Kc + BK - 1) / BK) / split;
  return static_cast<double>((tiles * split + sms - 1) / sms) * (std::max(bn, 128) + 16) * (kb + 8.0 + (split > 1 ? 6.0 : 0.0));
}
// Parts of the contraction for all M samples of the product (a slice of them takes the same: it fixes the order of the sums):
// where the tiles leave SMs idle and the k-blocks of one follow each other on one SM.
int split_parts(int64_t M, int64_t N, int64_t Kc) {
  int best = 1;
  double cost = split_cost(M, N, Kc, false, 1);
  for (int s = 2; s <= 8 && Kc / BK >= 2 * s; s *= 2) {
    const double c = split_cost(M, N, Kc, false, s);
    if (c < 0.9 * cost) { cost = c; best = s; }
  }
  return best;
}

// One split-bf16 product  D[off..off+n) = A * B^T  with A = [*, 2*Cp] and B = [N x 2*Cp] (hi | lo) operands:
// hi*hi + hi*lo + lo*hi over a contraction of Cp.
template <int EPI>
int split_product(sfb_ctx* ctx, int64_t off, int64_t n, __nv_bfloat16* A, __nv_bfloat16* B, int64_t N, int64_t Cp,
                  float* C, int64_t ldc, TcParams p) {
  TcState* st = static_cast<TcState*>(ctx->tc);
  p.kparts = EPI == F_GRAM ? 1 : split_parts(ctx->K, N, Cp);
  const int bn = pick_tile_width(st->sms / p.kparts, (n + BM - 1) / BM, N, FS_BN, 16, EPI == F_GRAM);
  CUtensorMap ma, mb;
  if (!make_map(st, &ma, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, A, 2 * Cp, off + n, 2 * Cp * 2, BK, BM) ||
      !make_map(st, &mb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, B, 2 * Cp, N, 2 * Cp * 2, BK, bn))
    return SFB_ERR_CUDA;
  p.M = static_cast<int32_t>(off + n); p.N = static_cast<int32_t>(N); p.Kc = static_cast<int32_t>(Cp);
  p.m_off = static_cast<int32_t>(off);
  p.tilesM = static_cast<int32_t>((n + BM - 1) / BM);
  p.bn = bn;
  p.tilesN = static_cast<int32_t>((N + bn - 1) / bn);
  p.nseg = 3; p.kseg = static_cast<int32_t>(Cp / BK);
  p.prefetch = kSplitPrefetch;
  p.a_off0 = 0; p.a_off1 = 0; p.a_off2 = static_cast<int32_t>(Cp);
  p.b_off0 = 0; p.b_off1 = static_cast<int32_t>(Cp); p.b_off2 = 0;
  p.status = ctx->at<uint32_t>(ctx->lay.status);
  CKC(launch_forward_split<EPI>(ctx, ma, mb, C, ldc, p));
  ctx->stats.flops += (EPI == F_GRAM ? 3.0 : 6.0) * n * N * Cp;
  return SFB_OK;
}

// Sufficient factors of distance metric learning and sparse coding in bf16 mode: the same steps as the fp32
// path (Section 2: z = W v with v = x - y; Figure 3: ISTA codes, u = W a - x), every product on the tensor cores
// with (hi | lo) bf16 operands.
int factors_split(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const float* Y, const int32_t* labels,
                  float* dml_norm_out = nullptr) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t rows = c.rows, cols = c.cols;
  cudaStream_t s = ctx->stream;
  float* V = ctx->at<float>(L.V);
  float* U = ctx->at<float>(L.U);
  __nv_bfloat16* Ws = ctx->at<__nv_bfloat16>(L.Ws);
  __nv_bfloat16* As = ctx->at<__nv_bfloat16>(L.As);
  TcParams p{};
  if (c.model == SFB_DML) {
    CKC(launch_kernel(pack_pairs_kernel, dim3(grid1d(n * cols / 4, 256)), dim3(256), 0, s, 1, X, Y, n, cols,
                      V + off * cols, As + off * 2 * L.colsp, L.colsp, Stamp{}));
      int rc = split_product<F_STORE>(ctx, off, n, As, Ws, rows, L.colsp, U, L.ldu, p);    // z_i = W v_i
    if (rc) return rc;
    CKC(dml_scale_rows(s, U + off * L.ldu, n, rows, L.ldu, labels, c.dml_margin,
                       ctx->at<__nv_bfloat16>(L.Rs) + off * 2 * L.rowsp, L.rowsp, dml_norm_out));
    return SFB_OK;
  }
  // Sparse coding: ISTA from a = 0, then u = W a - x, v = a.  The first iterate is soft(W^T x / L).
  const int T = c.sc_ista_iters;
  const bool gram = L.Gs != 0;
  __nv_bfloat16* WTs = ctx->at<__nv_bfloat16>(L.WTs);
  __nv_bfloat16* Rs = ctx->at<__nv_bfloat16>(L.Rs);
  // the iterates as operands: with the Gram matrix a product reads one and writes the next, so two buffers in turn
  __nv_bfloat16* as[2] = {As, gram ? ctx->at<__nv_bfloat16>(L.As2) : As};
  auto ista = [&](int t) {
    TcParams q{};
    q.aux = V; q.ldaux = cols;
    q.sc = ctx->at<Scalars>(L.scalars); q.lam = c.sc_lambda;
    q.split = as[t & 1]; q.ld_split = 2 * L.colsp; q.split_half = static_cast<int32_t>(L.colsp);
    return q;
  };
  auto residual = [&](__nv_bfloat16* a) {                                               // r = W a - x
    TcParams q{};
    q.aux = X - off * rows; q.ldaux = rows;          // X holds this worker's samples: index it by the global row
    q.split = Rs; q.ld_split = 2 * L.rowsp; q.split_half = static_cast<int32_t>(L.rowsp);
    return split_product<F_SUB>(ctx, off, n, a, Ws, rows, L.colsp, U, L.ldu, q);
  };
  int rc = SFB_OK;
  if (T == 0) {
    CKC(cudaMemsetAsync(V + off * cols, 0, static_cast<size_t>(n) * cols * 4, s));
    CKC(cudaMemsetAsync(As + off * 2 * L.colsp, 0, static_cast<size_t>(n) * 2 * L.colsp * 2, s));
  } else {
    if (gram && rows <= kPreciseRows) {                                                 // W^T x, a_1
      EpiArgs e{};
      e.C = V + off * cols; e.ldc = cols; e.C2 = ctx->at<float>(L.Bx) + off * cols; e.ldc2 = cols;
      e.sc = ctx->at<Scalars>(L.scalars); e.lam = c.sc_lambda;
      CKC(sgemm(s, true, false, EPI_ISTA0, n, cols, rows, X, rows, ctx->W, cols, e, ctx->K));
      ctx->stats.flops += 2.0 * n * rows * cols;
      CKC(launch_kernel(pack_split_rows_kernel, dim3(grid1d(n * cols / 4, 256)), dim3(256), 0, s, 1, V + off * cols, n,
                        cols, cols, as[1] + off * 2 * L.colsp, L.colsp, Stamp{}));
    } else {
      CKC(launch_kernel(pack_split_rows_kernel, dim3(grid1d(n * ((rows + 3) / 4), 256)), dim3(256), 0, s, 1, X, n, rows,
                        rows, Rs + off * 2 * L.rowsp, L.rowsp, Stamp{}));
      p = ista(1);
      p.C2 = gram ? ctx->at<float>(L.Bx) : nullptr;
      if ((rc = split_product<F_ISTA0>(ctx, off, n, Rs, WTs, cols, L.rowsp, V, cols, p)) != SFB_OK) return rc;
    }
  }
  for (int t = 2; t <= T; ++t) {
    p = ista(t);
    if (gram) {
      p.C2 = ctx->at<float>(L.Bx);
      rc = split_product<F_ISTAG>(ctx, off, n, as[(t - 1) & 1], ctx->at<__nv_bfloat16>(L.Gs), cols, L.colsp, V, cols, p);
    } else {
      if ((rc = residual(As)) != SFB_OK) return rc;
      rc = split_product<F_ISTA>(ctx, off, n, Rs, WTs, cols, L.rowsp, V, cols, p);      // a <- soft(a - W^T r / L)
    }
    if (rc) return rc;
  }
  return residual(T == 0 ? As : as[T & 1]);                                             // u = W a - x
}

}  // namespace

// The operands that the factors of every worker of a step share: the split copies of the W that all of them see
// (bulk-synchronous consistency), and for sparse coding its transpose and W^T W.
int tc_begin_step(sfb_ctx* ctx) {
  const sfb_config& c = ctx->cfg;
  if (c.model == SFB_MLR) return SFB_OK;
  const Layout& L = ctx->lay;
  const int64_t rows = c.rows, cols = c.cols;
  cudaStream_t s = ctx->stream;
  CKC(launch_kernel(pack_split_rows_kernel, dim3(grid1d(rows * cols / 4, 256)), dim3(256), 0, s, 1, ctx->W, rows, cols,
                    cols, ctx->at<__nv_bfloat16>(L.Ws), L.colsp, take_stamp(ctx)));
  if (c.model == SFB_SC) {
    __nv_bfloat16* WTs = ctx->at<__nv_bfloat16>(L.WTs);
    CKC(launch_kernel(pack_split_t_kernel, dim3(static_cast<unsigned>((cols + 63) / 64),
                      static_cast<unsigned>(L.rowsp / 64)), dim3(256), 0, s, 1, ctx->W, rows, cols, cols, WTs, L.rowsp));
    if (L.Gs) {
      TcParams p{};
      p.four = rows <= kPreciseRows;
      p.split = ctx->at<__nv_bfloat16>(L.Gs); p.ld_split = 2 * L.colsp; p.split_half = static_cast<int32_t>(L.colsp);
      float* G = c.sc_lipschitz > 0.f ? nullptr : ctx->at<float>(L.G);
      const int rc = split_product<F_GRAM>(ctx, 0, cols, WTs, WTs, cols, L.rowsp, G, cols, p);
      if (rc) return rc;
    }
  }
  return SFB_OK;
}

double split_product_cost(int64_t M, int64_t N, int64_t Kc, bool sym) {
  return split_cost(M, N, Kc, sym, sym ? 1 : split_parts(M, N, Kc));
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
  CKC((launch_forward<F_SOFTMAX, true>(ctx, ma, mb, mc, p)));                                // z_i = W x_i
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
  const int64_t rows = c.rows, cols = c.cols, K = ctx->K;
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
  CKC(launch_kernel(pack_mlr_kernel, dim3(grid1d(n * cols / 4, 256)), dim3(256), 0, ctx->stream, 1, X, n, cols, Xb,
                    L.colsb, off,
                    fused ? nullptr : ctx->at<float>(L.Xf), labels, ctx->at<int32_t>(L.labels), ctx->at<int32_t>(L.slot),
                    rows,
                    take_stamp(ctx)));
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
  CKC(launch_forward<F_SOFTMAX>(ctx, ma, mb, mc, p));
  ctx->stats.flops += 2.0 * n * rows * cols;
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
  pdl_wait();
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
  pdl_wait();
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

// Received fp32 factors take a worker's place in the bf16 layout: v into V^T (bf16) and the fp32 sample copy, u into U^T
// (bf16, 0 at the class entry), the class entry into the fp32 label coefficients.
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

int tc_factors(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const float* Y, const int32_t* labels, bool fused,
               float* dml_norm_out) {
  if (ctx->cfg.model != SFB_MLR) return factors_split(ctx, off, n, X, Y, labels, dml_norm_out);
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t rows = c.rows, K = ctx->K;
  const int64_t ldz = round_up(rows, 32);
  float* Z = ctx->at<float>(L.ZT);
  float* lse = ctx->at<float>(L.V);
  int tiles_n = 0;
  const int rc = mlr_forward(ctx, off, n, X, labels, fused, &tiles_n);
  if (rc) return rc;
  CKC(launch_kernel(mlr_lse_kernel, dim3(static_cast<unsigned>((n + 7) / 8)), dim3(256), 0, ctx->stream, 1,
                    ctx->at<float2>(L.part), K, tiles_n, Z, ldz, rows, labels, off, n, lse, ctx->at<float>(L.loss),
                    ctx->at<float>(L.coef), fused ? ctx->at<int32_t>(L.slot) : nullptr, ctx->at<uint32_t>(L.status)));
  return emit_p<false>(ctx, off, n, labels, fused ? X : nullptr);
}

// The (hi | lo) codes or pair differences: the operand V of the update.
__nv_bfloat16* tc_split_v(const sfb_ctx* ctx) {
  const Layout& L = ctx->lay;
  const bool odd = ctx->cfg.model == SFB_SC && L.Gs != 0 && (ctx->cfg.sc_ista_iters & 1);     // which buffer the last iterate is in
  return ctx->at<__nv_bfloat16>(odd ? L.As2 : L.As);
}

// Factors computed elsewhere (DML, SC): fp32 pairs in U and V -> the operands of the update.
int tc_pack_received(sfb_ctx* ctx, int64_t off, int64_t n) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  cudaStream_t s = ctx->stream;
  CKC(launch_kernel(pack_split_rows_kernel, dim3(grid1d(n * ((c.rows + 3) / 4), 256)), dim3(256), 0, s, 1,
                    ctx->at<float>(L.U) + off * L.ldu, n, c.rows, L.ldu, ctx->at<__nv_bfloat16>(L.Rs) + off * 2 * L.rowsp,
                    L.rowsp, Stamp{}));
  CKC(launch_kernel(pack_split_rows_kernel, dim3(grid1d(n * c.cols / 4, 256)), dim3(256), 0, s, 1,
                    ctx->at<float>(L.V) + off * c.cols, n, c.cols, c.cols, tc_split_v(ctx) + off * 2 * L.colsp, L.colsp,
                    Stamp{}));
  return SFB_OK;
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
