// Reconstruct-and-apply step of SFB on sm_100a (Section 3, Figure 1: every worker rebuilds the K rank-1 updates
// from the gathered sufficient factors and applies them):   W <- W + alpha * U^T V,   alpha = -eta,
// as ONE pass over W: the tensor-core product of a tile is combined with the fp32 tile of W while both are on
// the SM, so the reconstructed update matrix never exists in memory and W makes one HBM round trip.
//
// Kernel shape.  Clusters of two CTAs on the two SMs of a TPC drive one tcgen05.mma.cta_group::2: the pair owns a
// 256 x 256 tile of W, CTA r of the pair holds rows [128 r, 128 r + 128) of it in its TMEM (fp32, two accumulator
// stages of 256 columns), loads its own 128 x 64 slice of U^T and its own 128 x 64 half of the V^T slice per
// k-block (32 KB per stage instead of the 48 KB a single-CTA 128 x 256 tile needs), and streams its own
// 128 x 256 fp32 half of the W tile.
// The bf16 operands are the gathered factors as the forward side leaves them, U [pairs x rows] and V [pairs x columns]: the
// contraction runs over pairs, so both are MN-major operands and no transposed copy of either exists (the transposes were
// a sixth of a step of metric learning at 1,000 x 20,000).  The tf32 words are K-major (U^T, V^T).
// Warps of a CTA: 0 = TMA producer, 1 = MMA issuer (leader CTA only) and TMEM owner, 2..9 = epilogue.
// Epilogue warp (q, h): TMEM lane quarter q (32 rows of W), column half h (128 columns), in four chunks of
// 32 x 32.  Each warp owns a ring of 4 KB slots: the W chunk lands there by TMA (two chunks in flight per warp, 64 KB per SM, or
// four), is combined in place with the accumulator chunk and goes back by TMA from the same slot; a lane has a row of the
// chunk and stores its 32 roundings of the bf16 copy as two sectors.  (The copy by rows, read back from the slot with 8 lanes a row,
// was a third of a warp's chain per chunk: 10,000 x 20,000, 64 pairs 480 us of the pass, 420 without, 374 where few rows change.)
// Shared memory is the scarce resource: see UpShape.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "sfb_ptx.cuh"
#include "sfb_tc.h"
#include "sfb_tile.cuh"

namespace sfb {
namespace {

using namespace ptx;

constexpr int UM = 128;                 // rows of W per CTA (256 per pair)
constexpr int UN = 256;                 // columns of W per tile, at most (128 for small matrices, see tile_width)
constexpr int UK = 64, UMMA_K = 16;
constexpr int kBytesA = UM * UK * 2;          // 16 KB: this CTA's rows of U^T
constexpr int kBytesB = (UN / 2) * UK * 2;    // 16 KB: this CTA's half of the V^T rows
constexpr int kStageBytes = kBytesA + kBytesB;
constexpr int kChunk = 32;
constexpr int kSlotBytes = 32 * kChunk * 4;   // 4 KB
constexpr int kPend = 1;                      // TMA stores of a warp that may still be reading their slots
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kTmemCols = 512;
// Two splits of the shared memory.  Four operand stages and a ring of three slots per epilogue warp; FEW, where every tile has a pair of CTAs of
// its own and the contraction fits two stages (up to kFewPairs pairs): two stages and five slots, so that all four chunks of a warp are under
// way at once.  us of a step, 4 + 3 / 2 + 5: 64 x 256 with 128 samples 20.5 / 18.2 to 19.5, 500 x 1,000 28.3 / 28.15, 1,000 x 1,000 30.2 / 30.1,
// 512 x 2,048 with 64 24.7 / 24.6; beyond: 1,000 x 1,000 with 256 30.5 / 31.2, 2,000 x 500 with 256 27.4 / 28.1.  us of an update:
// 5,000 x 3,000 with 128, 256 pairs 31.2, 34.8 / 32.7, 36.3; 10,000 x 20,000 with 64 366 / 367, 1,024 472 / 713;
// 78,798 x 1,716 with 256 272 / 284.  (3 + 4: 552; 5 + 2: 495.)
constexpr int kFewPairs = 128;
template <bool FEW>
struct UpShape {
  static constexpr int kStages = FEW ? 2 : 4, kRing = FEW ? 5 : 3;
  static constexpr int kBars = 2 * kStages + 4 + kEpiWarps * kRing;
  static constexpr int kSmem = kStages * kStageBytes + kEpiWarps * kRing * kSlotBytes + kBars * 8 + 16 + 1024;
};

struct UpdParams {
  int32_t rows, cols;          // shape of W
  int32_t tilesM, tilesN;      // pair tiles: 256 rows x bn columns
  int32_t bn;                  // 256 or 128
  int32_t nseg, kseg;          // contraction: nseg segments of kseg k-blocks (3 segments: tf32 pairs)
  // Segment s reads U^T from column a_off<s> and V^T from column b_off<s>.  Scalars, not arrays: indexing an
  // array of a kernel parameter with a run-time index moves the whole parameter block to local memory.
  int32_t a_off0, a_off1, a_off2, b_off0, b_off1, b_off2;
  float alpha;
  int32_t prox_kind;           // entry-wise prox applied to the updated value (0 none, 1 soft-threshold, 2 scale)
  float prox_a;
  __nv_bfloat16* shadow;       // bf16 copy of the updated W (or null), row pitch shadow_ld elements
  float* shadow32;             // (big | small) tf32 copy of the updated W: big at column c, small at shadow_half + c
  int64_t shadow_ld;
  int64_t shadow_half;
  Stamp begin;
  unsigned long long* end;
  uint32_t* status;
  unsigned long long* copy_counters;   // [0] row pieces of the bf16 copy visited, [1] of them rewritten (or null)
};

__device__ __forceinline__ float to_tf32(float x) {
  uint32_t u;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(u) : "f"(x));
  return __uint_as_float(u);
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&v);
}

// Tile order: row blocks are taken in groups of kGroup; within a group the tiles are numbered row block fastest,
// then column block.  The pairs that run at the same time therefore work on kGroup blocks of U^T (512 KB each) and
// on about 74 / kGroup blocks of V^T: every operand line has a handful of readers at a time instead of one block of
// U^T having forty (measured: groups of 8 are 4-5 % faster than column-block-fastest order, groups of 37 or more
// slower again).  All of V^T (marked evict_last) and the group's blocks of U^T stay in L2.
constexpr int kGroup = 8;
__device__ __forceinline__ void tile_origin(const UpdParams& p, int tile, int& m0, int& n0) {
  const int per_group = kGroup * p.tilesN;
  const int grp = tile / per_group, within = tile - grp * per_group;
  const int gsz = min(kGroup, p.tilesM - grp * kGroup);       // the last group may be smaller
  const int tm = grp * kGroup + within % gsz, tn = within / gsz;
  m0 = tm * (2 * UM);
  n0 = tn * p.bn;
}

// TF32: the operands are 32-bit words read as tf32 (32 elements per 128-byte k-block), see the forward kernel.
// SHADOW: the operand copy of the new W that the epilogue writes beside it for the next forward product:
// 1 bf16, 2 the (big | small) pair of tf32 words of the fp32-on-tensor-cores mode.
template <int SHADOW, bool TF32 = false, bool FEW = false>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
update_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const __grid_constant__ CUtensorMap tmC, const UpdParams p) {
  constexpr int kStages = UpShape<FEW>::kStages, kRing = UpShape<FEW>::kRing, kBars = UpShape<FEW>::kBars;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + kStages * kBytesA;
  uint8_t* sRing = smem + kStages * kStageBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sRing + kEpiWarps * kRing * kSlotBytes);
  uint64_t* full = bars;                       // leader's copy is the one in use: both CTAs' loads signal it
  uint64_t* empty = bars + kStages;            // one per CTA: the MMA's commit arrives on both
  uint64_t* tfull = bars + 2 * kStages;        // one per CTA (commit arrives on both)
  uint64_t* tempty = bars + 2 * kStages + 2;   // leader's copy: 8 epilogue warps of each CTA arrive on it
  uint64_t* rfull = bars + 2 * kStages + 4;    // per epilogue warp and ring slot
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kBars);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int ntiles = p.tilesM * p.tilesN;
  const int my_tiles = pair < ntiles ? (ntiles - 1 - pair) / npairs + 1 : 0;
  const int numK = p.nseg * p.kseg;
  constexpr bool MN = !TF32;                   // the operands are MN-major
  const int half = p.bn / 2;                   // columns per CTA of the V^T slice, and per epilogue warp
  pdl_launch_dependents();

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], 2 * kEpiWarps); }
    for (int i = 0; i < kEpiWarps * kRing; ++i) mbar_init(&rfull[i], 1);
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&tmA); prefetch_tmap(&tmB); prefetch_tmap(&tmC);
  }
  if (warp == 1) { tmem_alloc_pair(tmem_slot, kTmemCols); tmem_relinquish_pair(); }
  tc_fence_before();
  __syncthreads();
  cluster_arrive();          // both CTAs' barriers exist and both have their TMEM before anyone signals the peer
  cluster_wait();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();
  stamp_begin(p.begin);

  if (warp == 0) {
    // ---------------- TMA producer (each CTA loads its own rows of U^T and its own half of the V^T rows) ---------
    const uint64_t pol_keep = policy_evict_last(), pol_norm = policy_evict_normal();
    uint32_t it = 0;
    bool ok = true;
    for (int tl = 0; tl < my_tiles && ok; ++tl) {
      int m0, n0;
      tile_origin(p, pair + tl * npairs, m0, n0);
      const int ma = m0 + static_cast<int>(rank) * UM, nb = n0 + static_cast<int>(rank) * half;
      for (int seg = 0; seg < p.nseg && ok; ++seg) {
        const int xa = seg == 0 ? p.a_off0 : seg == 1 ? p.a_off1 : p.a_off2;
        const int xb = seg == 0 ? p.b_off0 : seg == 1 ? p.b_off1 : p.b_off2;
        for (int kl = 0; kl < p.kseg; ++kl, ++it) {
          const uint32_t s = it % kStages, ph = (it / kStages) & 1;
          if (!mbar_wait_warp(&empty[s], ph ^ 1, abort_flag)) { ok = false; break; }
          if (elect_one()) {
            if (rank == 0) mbar_expect_tx(&full[s], 2 * (kBytesA + half * UK * 2));
            const uint32_t full_leader = mapa_u32(smem_u32(&full[s]), 0);
            if (MN) {                          // boxes of 64 rows (columns) of W x 64 pairs
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                tma_load_2d_pair(sA + s * kBytesA + h * (kBytesA / 2), &tmA, xa + ma + 64 * h, kl * UK, full_leader, pol_norm);
                if (64 * h < half)
                  tma_load_2d_pair(sB + s * kBytesB + h * (kBytesB / 2), &tmB, xb + nb + 64 * h, kl * UK, full_leader, pol_keep);
              }
            } else {
              tma_load_2d_pair(sA + s * kBytesA, &tmA, xa + kl * (UK / 2), ma, full_leader, pol_norm);
              tma_load_2d_pair(sB + s * kBytesB, &tmB, xb + kl * (UK / 2), nb, full_leader, pol_keep);
            }
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: one thread of the leader CTA drives both SMs ----------------
    if (rank == 0) {
      const uint32_t idesc = TF32 ? umma_idesc_tf32(2 * UM, p.bn) : umma_idesc_bf16(2 * UM, p.bn) | kIdescMnMajor;
      uint32_t it = 0;
      bool ok = true;
      for (int tl = 0; tl < my_tiles && ok; ++tl) {
        const uint32_t a = tl & 1, aph = (tl >> 1) & 1;
        if (!mbar_wait_warp(&tempty[a], aph ^ 1, abort_flag)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + a * UN;
        for (int kb = 0; kb < numK; ++kb, ++it) {
          const uint32_t s = it % kStages, ph = (it / kStages) & 1;
          if (!mbar_wait_warp(&full[s], ph, abort_flag)) { ok = false; break; }
          tc_fence_after();
          if (elect_one()) {
            const uint64_t da = MN ? umma_desc_mn128(smem_u32(sA + s * kBytesA)) : umma_desc_k128(smem_u32(sA + s * kBytesA));
            const uint64_t db = MN ? umma_desc_mn128(smem_u32(sB + s * kBytesB)) : umma_desc_k128(smem_u32(sB + s * kBytesB));
#pragma unroll
            for (int k = 0; k < UK / UMMA_K; ++k) {          // four MMAs of 16 pairs (bf16) or 8 (tf32) each
              const uint64_t adv = static_cast<uint64_t>(MN ? k * 2048 / 16 : k * 32 / 16);
              if (TF32) umma_tf32_pair(d_tmem, da + adv, db + adv, idesc, (kb | k) != 0 ? 1u : 0u);
              else umma_bf16_pair(d_tmem, da + adv, db + adv, idesc, (kb | k) != 0 ? 1u : 0u);
            }
            umma_commit_pair(&empty[s], 3);          // both CTAs' stage s is free once these MMAs have read it
          }
        }
        if (ok && elect_one()) umma_commit_pair(&tfull[a], 3);    // both CTAs' halves of the accumulator are complete
      }
    }
  } else {
    // ---------------- epilogue: warp (q, h) = TMEM lane quarter q, column half h ----------------
    const int e = warp - 2, q = warp & 3, h = e >> 2;
    uint8_t* ring = sRing + e * kRing * kSlotBytes;
    uint64_t* rf = rfull + e * kRing;
    const int cshift = p.bn == 256 ? 2 : 1, cpw = 1 << cshift;       // chunks per warp and tile: 4 or 2
    const uint32_t nchunks = static_cast<uint32_t>(my_tiles * cpw);
    // Default L2 priority for the tiles of W: with evict_first on this traffic the written lines are pushed to
    // HBM at once, in small pieces between the reads, and the measured rate drops by a quarter.
    const uint64_t pol_w = policy_evict_normal();
    const uint32_t tempty_leader0 = mapa_u32(smem_u32(&tempty[0]), 0), tempty_leader1 = mapa_u32(smem_u32(&tempty[1]), 0);
    const int row_in_tile = static_cast<int>(rank) * UM + q * 32;
    bool ok = true;
    uint32_t copy_written = 0;           // row pieces of the bf16 copy this lane rewrote
    uint32_t lg = 0;                     // next chunk to request, by the whole warp
    int lm0 = 0, ln0 = 0;                // ... and its tile
    auto issue_load = [&]() {
      if (lg >= nchunks) return;
      if ((lg & (cpw - 1)) == 0) tile_origin(p, pair + static_cast<int>(lg >> cshift) * npairs, lm0, ln0);
      const uint32_t slot = lg % kRing;
      if (elect_one()) {
        mbar_expect_tx(&rf[slot], kSlotBytes);
        tma_load_2d_hint(ring + slot * kSlotBytes, &tmC, ln0 + h * half + static_cast<int>(lg & (cpw - 1)) * kChunk,
                         lm0 + row_in_tile, &rf[slot], pol_w);
      }
      ++lg;
    };
    for (int i = 0; i < kRing - kPend; ++i) issue_load();
    uint32_t g = 0;
    for (int tl = 0; tl < my_tiles && ok; ++tl) {
      int m0, n0;
      tile_origin(p, pair + tl * npairs, m0, n0);
      const uint32_t a = tl & 1, aph = (tl >> 1) & 1;
      const int y0 = m0 + row_in_tile;
      if (!__all_sync(0xffffffffu, mbar_wait(&tfull[a], aph, abort_flag))) { ok = false; break; }
      tc_fence_after();
      const uint32_t t_addr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + a * UN + h * half;
      uint32_t acc0[32], acc1[32];
      tmem_ld_32x32(t_addr, acc0);
      auto process = [&](uint32_t (&acc)[32], uint32_t (&nxt)[32], int c) -> bool {
        tmem_ld_wait();                                      // chunk c's accumulators are in registers
        if (c + 1 < cpw) {
          tmem_ld_32x32(t_addr + (c + 1) * kChunk, nxt);     // chunk c+1 streams in during this chunk's work
        } else {
          tc_fence_before();                                 // last TMEM read of the tile by this warp: hand the
          __syncwarp();                                      // accumulator stage back to the leader's MMA warp
          if (lane == 0) mbar_arrive_cluster(a ? tempty_leader1 : tempty_leader0);
        }
        const uint32_t rs = g % kRing;
        const uint32_t sl = smem_u32(ring + rs * kSlotBytes);
        const int x0 = n0 + h * half + c * kChunk;
        if (!__all_sync(0xffffffffu, mbar_wait(&rf[rs], (g / kRing) & 1, abort_flag))) return false;
        // All of the row's reads, then the arithmetic, then the writes: with two epilogue warps to a scheduler a chunk's time is its
        // chain of latencies.
        float4 w[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) w[j] = ld_shared_f4(slot_addr(sl, lane, j));
        uint32_t now[16];          // SHADOW == 1: the bf16 rounding of this row's 32 new values
        uint32_t differs = 0;      //   does any of them change?
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          uint32_t o01 = 0, o23 = 0;
          if (SHADOW == 1) { o01 = pack2(w[j].x, w[j].y); o23 = pack2(w[j].z, w[j].w); }
          w[j].x = fmaf(p.alpha, __uint_as_float(acc[4 * j + 0]), w[j].x);
          w[j].y = fmaf(p.alpha, __uint_as_float(acc[4 * j + 1]), w[j].y);
          w[j].z = fmaf(p.alpha, __uint_as_float(acc[4 * j + 2]), w[j].z);
          w[j].w = fmaf(p.alpha, __uint_as_float(acc[4 * j + 3]), w[j].w);
          if (p.prox_kind != 0) {
            w[j].x = prox_entry(w[j].x, p.prox_kind, p.prox_a); w[j].y = prox_entry(w[j].y, p.prox_kind, p.prox_a);
            w[j].z = prox_entry(w[j].z, p.prox_kind, p.prox_a); w[j].w = prox_entry(w[j].w, p.prox_kind, p.prox_a);
          }
          if (SHADOW == 1) {
            now[2 * j] = pack2(w[j].x, w[j].y);
            now[2 * j + 1] = pack2(w[j].z, w[j].w);
            differs |= (o01 ^ now[2 * j]) | (o23 ^ now[2 * j + 1]);
          }
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) st_shared_f4(slot_addr(sl, lane, j), w[j]);
        fence_proxy_async_smem();
        __syncwarp();                                        // every lane has rewritten its row of the slot
        if (elect_one()) {                                   // (the same lane every time: bulk groups are a thread's)
          if (x0 < p.cols && y0 < p.rows) tma_store_2d_at(&tmC, sl, x0, y0, pol_w);
          tma_commit_group();
          if (g >= kPend) tma_wait_group_read<kPend>();      // the store of chunk g-kPend has read its slot:
        }
        __syncwarp();
        issue_load();                                        // refill it with chunk g + kRing - kPend
        if (SHADOW == 2) {
          // (big | small) tf32 copy of the chunk, read back from the slot with 8 lanes per row: 128-byte row pieces
          const int sub = lane >> 3, jj = lane & 7;
#pragma unroll
          for (int r0 = 0; r0 < 32; r0 += 4) {
            const int r = r0 + sub;
            const float4 w = ld_shared_f4(slot_addr(sl, r, jj));
            const int col = x0 + 4 * jj;
            if (y0 + r < p.rows && col < p.cols) {
              const float4 b = make_float4(to_tf32(w.x), to_tf32(w.y), to_tf32(w.z), to_tf32(w.w));
              float* d = p.shadow32 + static_cast<int64_t>(y0 + r) * p.shadow_ld + col;
              *reinterpret_cast<float4*>(d) = b;
              *reinterpret_cast<float4*>(d + p.shadow_half) =
                  make_float4(to_tf32(w.x - b.x), to_tf32(w.y - b.y), to_tf32(w.z - b.z), to_tf32(w.w - b.w));
            }
          }
        }
        if (SHADOW == 1) {
          // The bf16 copy holds bf16(W) when the pass starts (set-up, refresh and this kernel keep it so): a row piece whose 32
          // roundings all stay the same already holds bf16 of the new values and is not rewritten.  With updates of a few
          // fp32 spacings per entry that is most of the matrix; the copy stays exact either way.  (x0 and the copy's pitch are
          // multiples of 32: a piece is inside or outside as a whole.)
          const bool rewrite = differs != 0 && y0 + lane < p.rows && x0 < p.shadow_ld;
          if (rewrite) {
            __nv_bfloat16* d = p.shadow + static_cast<int64_t>(y0 + lane) * p.shadow_ld + x0;
            st_global_v8(d, now, 0);
            st_global_v8(d + 16, now, 8);
          }
          copy_written += rewrite;
        }
        ++g;
        return true;
      };
#pragma unroll 1
      for (int c = 0; c < cpw && ok; c += 2) {
        ok = process(acc0, acc1, c);
        if (ok) ok = process(acc1, acc0, c + 1);
      }
    }
    if (elect_one()) tma_wait_group<0>();
    if (SHADOW == 1 && p.copy_counters) {
      const uint32_t written = __reduce_add_sync(0xffffffffu, copy_written);
      if (lane == 0) {
        atomicAdd(&p.copy_counters[0], 32ull * nchunks);
        atomicAdd(&p.copy_counters[1], static_cast<unsigned long long>(written));
      }
    }
  }

  // ---------------- teardown ----------------
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // A wait ran out: report it and give copies in flight a bounded time to land.
    if (threadIdx.x == 0) atomicOr(p.status, SFB_STATUS_TIMEOUT);
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
    __syncthreads();
  }
  cluster_arrive();          // neither CTA frees its TMEM or exits while the other may still signal or write it
  cluster_wait();
  stamp_end(p.end);
  if (warp == 1) { tc_fence_after(); tmem_dealloc_pair(tmem_base, kTmemCols); }
}

// ---------------------------------------------------------------------------------------------------------
// The update of operands that are (hi | lo) pairs of 16-bit values (metric learning, sparse coding):
//   W <- prox(W + alpha * (U_hi^T V_hi + U_lo^T V_hi + U_hi^T V_lo)).
// As in split_product_kernel, one stage holds a k-block of all four halves and the cross terms have an accumulator of their own;
// U_hi^T V_hi is added to sums in the epilogue warps' registers every 1,024 pairs, while the cross terms of the last k-block
// run.  The sums also free both accumulators (all 512 columns of TMEM) before the pass over W, which therefore runs beside the
// next tile's products although there is no second pair of accumulators.
// Shared memory, in two forms.  Many pairs: three stages of 64 of them (64 KB in a CTA), for the tensor cores' sake, and one 4 KB
// slot of W per epilogue warp.  Few pairs, where the pass over W is what takes the time: three stages of 32 and four slots.
// With one slot that pass waits for every load (2.7 TB/s); with stages of 32 there are twice the copies (K = 1024: 914 -> 980 us).
// ---------------------------------------------------------------------------------------------------------
constexpr int SU_STAGES = 3, kSuFewPairs = 384;
template <bool FEW>
struct SuShape {
  static constexpr int kPairs = FEW ? 32 : 64, kDrain = 1024 / kPairs, kSlots = FEW ? 4 : 1, kPending = FEW ? 1 : 0;
  static constexpr int kBox = 64 * kPairs * 2, kBytes = 2 * kBox, kStage = 4 * kBytes;     // 64 columns; an operand half; all four
  static constexpr int kBars = 2 * SU_STAGES + 4 + kEpiWarps * kSlots;
  static constexpr int kSmem = SU_STAGES * kStage + kEpiWarps * kSlots * kSlotBytes + kBars * 8 + 16 + 1024;
};

struct SplitUpdParams {
  UpdParams t;                 // rows, cols, tiles, bn, kseg, alpha, prox, stamps, status
  int32_t u_lo, v_lo;          // column of the lo half of U and of V
  bool fp16;                   // the form of the pairs
  float lo_scale;              // what an accumulated cross term counts for
  const float* inv;            // inverse scale of the whole sum (or null: 1)
};

template <bool FEW>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
update_split_kernel(const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmV,
                    const __grid_constant__ CUtensorMap tmC, const __grid_constant__ SplitUpdParams sp) {
  using Shape = SuShape<FEW>;
  constexpr int SU_UK = Shape::kPairs, SU_DRAIN = Shape::kDrain, SU_SLOTS = Shape::kSlots, SU_PENDING = Shape::kPending;
  constexpr int kSuBox = Shape::kBox, kSuBytes = Shape::kBytes, kSuStage = Shape::kStage, kSuBars = Shape::kBars;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sRing = smem + SU_STAGES * kSuStage;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sRing + kEpiWarps * SU_SLOTS * kSlotBytes);
  uint64_t* full = bars;                             // as in update_pair_kernel: full, mempty, cempty are the leader's
  uint64_t* empty = bars + SU_STAGES;
  uint64_t* mfull = bars + 2 * SU_STAGES;
  uint64_t* mempty = mfull + 1;
  uint64_t* cfull = mfull + 2;
  uint64_t* cempty = mfull + 3;
  uint64_t* rfull = mfull + 4;                       // per epilogue warp and slot
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kSuBars);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const UpdParams& p = sp.t;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int ntiles = p.tilesM * p.tilesN;
  const int my_tiles = pair < ntiles ? (ntiles - 1 - pair) / npairs + 1 : 0;
  const int nk = p.kseg, half = p.bn / 2;
  pdl_launch_dependents();

  if (threadIdx.x == 0) {
    for (int i = 0; i < SU_STAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(mfull, 1); mbar_init(mempty, 2 * kEpiWarps);
    mbar_init(cfull, 1); mbar_init(cempty, 2 * kEpiWarps);
    for (int i = 0; i < kEpiWarps * SU_SLOTS; ++i) mbar_init(&rfull[i], 1);
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&tmU); prefetch_tmap(&tmV); prefetch_tmap(&tmC);
  }
  if (warp == 1) { tmem_alloc_pair(tmem_slot, kTmemCols); tmem_relinquish_pair(); }
  tc_fence_before();
  __syncthreads();
  cluster_arrive();
  cluster_wait();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();
  stamp_begin(p.begin);

  if (warp == 0) {
    // ---------------- TMA producer: U_hi, U_lo, V_hi, V_lo of a k-block, boxes of 64 columns ----------------
    const uint64_t pol_keep = policy_evict_last(), pol_norm = policy_evict_normal();
    uint32_t it = 0;
    bool ok = true;
    for (int tl = 0; tl < my_tiles && ok; ++tl) {
      int m0, n0;
      tile_origin(p, pair + tl * npairs, m0, n0);
      const int mu = m0 + static_cast<int>(rank) * UM, nv = n0 + static_cast<int>(rank) * half;
      for (int kb = 0; kb < nk; ++kb, ++it) {
        const uint32_t s = it % SU_STAGES, ph = (it / SU_STAGES) & 1;
        if (!mbar_wait_warp(&empty[s], ph ^ 1, abort_flag)) { ok = false; break; }
        if (elect_one()) {
          if (rank == 0) mbar_expect_tx(&full[s], 2 * (2 * kSuBytes + 2 * half * SU_UK * 2));
          const uint32_t bar = mapa_u32(smem_u32(&full[s]), 0);
          uint8_t* st = smem + s * kSuStage;
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            tma_load_2d_pair(st + b * kSuBox, &tmU, mu + 64 * b, kb * SU_UK, bar, pol_norm);
            tma_load_2d_pair(st + kSuBytes + b * kSuBox, &tmU, sp.u_lo + mu + 64 * b, kb * SU_UK, bar, pol_norm);
            if (64 * b < half) {
              tma_load_2d_pair(st + 2 * kSuBytes + b * kSuBox, &tmV, nv + 64 * b, kb * SU_UK, bar, pol_keep);
              tma_load_2d_pair(st + 3 * kSuBytes + b * kSuBox, &tmV, sp.v_lo + nv + 64 * b, kb * SU_UK, bar, pol_keep);
            }
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: one thread of the leader CTA ----------------
    if (rank == 0) {
      const uint32_t idesc = (sp.fp16 ? umma_idesc_fp16(2 * UM, p.bn) : umma_idesc_bf16(2 * UM, p.bn)) | kIdescMnMajor;
      const uint32_t d_main = tmem_base, d_cross = tmem_base + UN;
      uint32_t it = 0, g = 0;
      bool ok = true;
      for (int tl = 0; tl < my_tiles && ok; ++tl) {
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const uint32_t s = it % SU_STAGES, ph = (it / SU_STAGES) & 1;
          const int kc = kb % SU_DRAIN;
          if (!mbar_wait_warp(&full[s], ph, abort_flag)) { ok = false; break; }
          if (kc == 0 && !mbar_wait_warp(mempty, (g & 1) ^ 1, abort_flag)) { ok = false; break; }
          tc_fence_after();
          uint8_t* st = smem + s * kSuStage;
          const uint64_t duh = umma_desc_mn128(smem_u32(st), kSuBox), dul = umma_desc_mn128(smem_u32(st + kSuBytes), kSuBox);
          const uint64_t dvh = umma_desc_mn128(smem_u32(st + 2 * kSuBytes), kSuBox), dvl = umma_desc_mn128(smem_u32(st + 3 * kSuBytes), kSuBox);
          const bool drained = kc == SU_DRAIN - 1 || kb + 1 == nk;
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < SU_UK / UMMA_K; ++k) {
              const uint64_t adv = static_cast<uint64_t>(k * 2048 / 16);
              umma_bf16_pair(d_main, duh + adv, dvh + adv, idesc, (kc | k) != 0 ? 1u : 0u);
            }
            if (drained) umma_commit_pair(mfull, 3);
          }
          if (drained) ++g;
          if (kb == 0) {
            if (!mbar_wait_warp(cempty, (tl & 1) ^ 1, abort_flag)) { ok = false; break; }
            tc_fence_after();
          }
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < SU_UK / UMMA_K; ++k) {
              const uint64_t adv = static_cast<uint64_t>(k * 2048 / 16);
              umma_bf16_pair(d_cross, dul + adv, dvh + adv, idesc, (kb | k) != 0 ? 1u : 0u);
              umma_bf16_pair(d_cross, duh + adv, dvl + adv, idesc, 1u);
            }
            umma_commit_pair(&empty[s], 3);
          }
        }
        if (ok && elect_one()) umma_commit_pair(cfull, 3);
      }
    }
  } else {
    // ---------------- epilogue: warp (q, h) = TMEM lane quarter q, column half h ----------------
    const int e = warp - 2, q = warp & 3, h = e >> 2;
    uint8_t* slots = sRing + e * SU_SLOTS * kSlotBytes;
    uint64_t* arrived = rfull + e * SU_SLOTS;
    const int cpw = half / kChunk;                   // chunks per warp and tile: 4 or 2
    const uint64_t pol_w = policy_evict_normal();
    const uint32_t mempty_leader = mapa_u32(smem_u32(mempty), 0), cempty_leader = mapa_u32(smem_u32(cempty), 0);
    const int row_in_tile = static_cast<int>(rank) * UM + q * 32;
    const uint32_t t_addr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + h * half;
    bool ok = true;
    const uint32_t last = static_cast<uint32_t>(my_tiles * cpw);
    auto issue_load = [&](uint32_t n) {              // (lane 0) the n-th chunk of this warp
      if (n >= last) return;
      const int tl = static_cast<int>(n) / cpw, c = static_cast<int>(n) % cpw;
      int m0, n0;
      tile_origin(p, pair + tl * npairs, m0, n0);
      const uint32_t at = n % SU_SLOTS;
      mbar_expect_tx(&arrived[at], kSlotBytes);
      tma_load_2d_hint(slots + at * kSlotBytes, &tmC, n0 + h * half + c * kChunk, m0 + row_in_tile, &arrived[at], pol_w);
    };
    if (lane == 0)
      for (uint32_t n = 0; n < SU_SLOTS; ++n) issue_load(n);
    const float alpha = p.alpha * (sp.inv ? *sp.inv : 1.f);
    uint32_t g = 0, r = 0;                           // drains and chunks behind
    for (int tl = 0; tl < my_tiles && ok; ++tl) {
      int m0, n0;
      tile_origin(p, pair + tl * npairs, m0, n0);
      float sum[4][32];
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int j = 0; j < 32; ++j) sum[c][j] = 0.f;
      auto drain = [&](uint32_t at, float scale, uint32_t done) {     // sum += scale * the accumulator at column `at`
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (c >= cpw) break;
          uint32_t acc[32];
          tmem_ld_32x32(t_addr + at + c * kChunk, acc);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) sum[c][j] = fmaf(__uint_as_float(acc[j]), scale, sum[c][j]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(done);
      };
      for (int kb = 0; kb < nk && ok; kb += SU_DRAIN, ++g) {
        ok = __all_sync(0xffffffffu, mbar_wait(mfull, g & 1, abort_flag));
        if (ok) drain(0, 1.f, mempty_leader);
      }
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(cfull, tl & 1, abort_flag));
      if (!ok) break;
      drain(UN, sp.lo_scale, cempty_leader);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (c >= cpw || !ok) break;
        const int x0 = n0 + h * half + c * kChunk, y0 = m0 + row_in_tile;
        ok = __all_sync(0xffffffffu, mbar_wait(&arrived[r % SU_SLOTS], (r / SU_SLOTS) & 1, abort_flag));
        if (!ok) break;
        uint8_t* sl = slots + (r % SU_SLOTS) * kSlotBytes;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          float4* wp = reinterpret_cast<float4*>(sl + lane * 128 + ((j ^ (lane & 7)) << 4));
          float4 w = *wp;
          w.x = fmaf(alpha, sum[c][4 * j + 0], w.x);
          w.y = fmaf(alpha, sum[c][4 * j + 1], w.y);
          w.z = fmaf(alpha, sum[c][4 * j + 2], w.z);
          w.w = fmaf(alpha, sum[c][4 * j + 3], w.w);
          if (p.prox_kind != 0) {
            w.x = prox_entry(w.x, p.prox_kind, p.prox_a); w.y = prox_entry(w.y, p.prox_kind, p.prox_a);
            w.z = prox_entry(w.z, p.prox_kind, p.prox_a); w.w = prox_entry(w.w, p.prox_kind, p.prox_a);
          }
          *wp = w;
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (x0 < p.cols && y0 < p.rows) tma_store_2d_hint(&tmC, sl, x0, y0, pol_w);
          tma_commit_group();
          tma_wait_group_read<SU_PENDING>();          // an earlier chunk's slot (or this one's) has been read: refill it
          if (r >= SU_PENDING) issue_load(r - SU_PENDING + SU_SLOTS);
        }
        __syncwarp();
        ++r;
      }
    }
    if (lane == 0) tma_wait_group<0>();
  }

  // ---------------- teardown, as in update_pair_kernel ----------------
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(p.status, SFB_STATUS_TIMEOUT);
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
    __syncthreads();
  }
  cluster_arrive();
  cluster_wait();
  stamp_end(p.end);
  if (warp == 1) { tc_fence_after(); tmem_dealloc_pair(tmem_base, kTmemCols); }
}

// Tile width: 128 where 256-wide tiles leave the pairs short of work.  Cycles of a tile: its k-blocks at the MMA or operand
// rate (measured about 620 a k-block of 64 pairs for 256 columns, 450 for 128; 1600 and 900 with four operand halves) and its
// epilogue.  (Counted with the cycles of the pass over W instead, more shapes take 128, whose half rows it moves more slowly: 4,999 x
// 3,004 with 259 pairs 36.7 -> 41.9 us, 30,000 x 500 with 300 42 -> 50.)
int tile_width(int64_t rows, int64_t cols, int64_t kblocks, int pairs, bool split) {
  auto cost = [&](int bn) {
    const int64_t tiles = ((rows + 2 * UM - 1) / (2 * UM)) * ((cols + bn - 1) / bn);
    const double kb = split ? (bn == 256 ? 1600. : 900.) : (bn == 256 ? 620. : 450.);
    return static_cast<double>((tiles + pairs - 1) / pairs) * (kblocks * kb + (bn == 256 ? 2500. : 1800.));
  };
  return cost(128) < 0.97 * cost(256) ? 128 : 256;
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

int tc_update_init(sfb_ctx* ctx, TcState* st) {
  int n = 1 << 30;
  CKC(prepare_pair_kernel(update_pair_kernel<1>, kThreads, UpShape<false>::kSmem, &n));
  CKC((prepare_pair_kernel(update_pair_kernel<1, false, true>, kThreads, UpShape<true>::kSmem, &n)));
  CKC(prepare_pair_kernel(update_split_kernel<false>, kThreads, SuShape<false>::kSmem, &n));
  CKC(prepare_pair_kernel(update_split_kernel<true>, kThreads, SuShape<true>::kSmem, &n));
  CKC((prepare_pair_kernel(update_pair_kernel<2, true>, kThreads, UpShape<false>::kSmem, &n)));
  CKC(forward_pair_prepare(&n));
  st->max_pairs = n;
  if (n < 1) return SFB_ERR_ARCH;                 // the device cannot host a CTA pair of these kernels
  return SFB_OK;
}

// fp32 mode on the tensor cores (MLR): U^T and V^T are (big | small) pairs of tf32 words, [rows x 2 Kp] and
// [cols x 2 Kp] with Kp the pair count rounded up to 32;  U^T V = Ub Vb + Ub Vs + Us Vb  (Us Vs, 2^-22 of the product,
// is dropped).  The label entries are part of U here: no separate label-row pass, no bf16 copy of W.
int tc32_update(sfb_ctx* ctx) {
  if (ctx->sparse_v) return sparse_update(ctx);         // writes the (big | small) copy as well
  const sfb_config& c = ctx->cfg;
  TcState* st = static_cast<TcState*>(ctx->tc);
  const Layout& L = ctx->lay;
  const int64_t Kp = L.Kp;                                  // a multiple of 32
  CUtensorMap ma, mb, mc;
  if (!make_map(st, &ma, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, ctx->at<float>(L.UT), 2 * Kp, c.rows, 2 * Kp * 4, UK / 2, UM) ||
      !make_map(st, &mb, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, ctx->at<float>(L.VT), 2 * Kp, c.cols, 2 * Kp * 4, UK / 2, UN / 2) ||
      !make_map(st, &mc, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, ctx->W, c.cols, c.rows, c.cols * 4, kChunk, 32))
    return SFB_ERR_CUDA;
  UpdParams p{};
  p.rows = static_cast<int32_t>(c.rows); p.cols = static_cast<int32_t>(c.cols);
  p.tilesM = static_cast<int32_t>((c.rows + 2 * UM - 1) / (2 * UM));
  p.bn = UN;
  p.tilesN = static_cast<int32_t>((c.cols + UN - 1) / UN);
  p.kseg = static_cast<int32_t>(Kp / (UK / 2));
  p.begin = take_stamp(ctx); p.end = &ctx->at<Scalars>(L.scalars)->ns[3];
  p.alpha = -ctx->step;
  p.prox_kind = ctx->prox_kind; p.prox_a = ctx->prox_a;
  p.status = ctx->at<uint32_t>(L.status);
  // The two cross terms first, big*big last: the tensor core rounds its fp32 accumulator at every instruction, by an
  // amount relative to what the accumulator holds, so the many roundings of the small terms should happen while it is
  // still small (measured: 3 times less error than with big*big first).
  p.nseg = 3;
  p.a_off0 = 0; p.a_off1 = static_cast<int32_t>(Kp); p.a_off2 = 0;
  p.b_off0 = static_cast<int32_t>(Kp); p.b_off1 = 0; p.b_off2 = 0;
  // the epilogue also writes the (big | small) copy of the new W, the operand of the next forward product
  p.shadow = nullptr; p.shadow32 = ctx->at<float>(L.Ws); p.shadow_ld = 2 * L.colsp; p.shadow_half = L.colsp;
  const int64_t tiles = static_cast<int64_t>(p.tilesM) * p.tilesN;
  const unsigned grid = 2u * static_cast<unsigned>(std::min<int64_t>(tiles, st->max_pairs));
  CKC(launch_kernel_if(tiles <= st->max_pairs, (update_pair_kernel<2, true>), dim3(grid), dim3(kThreads), UpShape<false>::kSmem, ctx->stream, 1, ma, mb, mc, p));
  return SFB_OK;
}

int tc_update(sfb_ctx* ctx) {
  if (ctx->cfg.model == SFB_MLR && !ctx->h16) {
    const int rc = tc_labels(ctx);                     // the fp32 label entries, unless the factors call has applied them
    if (rc) return rc;
  }
  if (ctx->sparse_v) return sparse_update(ctx);
  const sfb_config& c = ctx->cfg;
  TcState* st = static_cast<TcState*>(ctx->tc);
  const Layout& L = ctx->lay;
  const bool split = c.model != SFB_MLR || ctx->h16;
  // U and V pair-major; the split products have (hi | lo) halves side by side
  const int64_t ldu = split ? 2 * L.rowsp : L.ldp, ldv = split ? 2 * L.colsp : L.colsb;
  const int64_t wu = split ? 2 * L.rowsp : c.rows, wv = split ? 2 * L.colsp : c.cols;
  __nv_bfloat16* U = ctx->at<__nv_bfloat16>(split ? L.Rs : L.P);
  void* V = split ? const_cast<uint16_t*>(split_v(ctx)) : ctx->at<uint16_t>(L.Xb);
  const bool few = split && ctx->K <= kSuFewPairs;
  const int uk = few ? SuShape<true>::kPairs : UK;
  CUtensorMap ma, mb, mc;
  if (!make_map(st, &ma, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, U, wu, ctx->K, ldu * 2, 64, uk) ||
      !make_map(st, &mb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, V, wv, ctx->K, ldv * 2, 64, uk) ||
      !make_map(st, &mc, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, ctx->W, c.cols, c.rows, c.cols * 4, kChunk, 32))
    return SFB_ERR_CUDA;
  UpdParams p{};
  p.rows = static_cast<int32_t>(c.rows); p.cols = static_cast<int32_t>(c.cols);
  p.tilesM = static_cast<int32_t>((c.rows + 2 * UM - 1) / (2 * UM));
  p.kseg = static_cast<int32_t>((ctx->K + uk - 1) / uk);
  p.bn = tile_width(c.rows, c.cols, (ctx->K + UK - 1) / UK, st->max_pairs, split);
  p.tilesN = static_cast<int32_t>((c.cols + p.bn - 1) / p.bn);
  p.begin = take_stamp(ctx); p.end = &ctx->at<Scalars>(L.scalars)->ns[3];
  p.alpha = -ctx->step;
  p.prox_kind = ctx->prox_kind; p.prox_a = ctx->prox_a;
  p.status = ctx->at<uint32_t>(L.status);
  const int64_t tiles = static_cast<int64_t>(p.tilesM) * p.tilesN;
  const unsigned grid = 2u * static_cast<unsigned>(std::min<int64_t>(tiles, st->max_pairs));
  if (split) {
    SplitUpdParams sp{p, static_cast<int32_t>(L.rowsp), static_cast<int32_t>(L.colsp), ctx->h16, ctx->h16 ? 1.f / 2048.f : 1.f,
                      ctx->h16 ? &ctx->at<Scalars>(L.scalars)->iU : nullptr};
    CKC(few ? launch_kernel_if(tiles <= st->max_pairs, update_split_kernel<true>, dim3(grid), dim3(kThreads), SuShape<true>::kSmem,
                               ctx->stream, 1, ma, mb, mc, sp)
            : launch_kernel_if(tiles <= st->max_pairs, update_split_kernel<false>, dim3(grid), dim3(kThreads), SuShape<false>::kSmem,
                               ctx->stream, 1, ma, mb, mc, sp));
    return SFB_OK;
  }
  p.nseg = 1;
  p.shadow = ctx->at<__nv_bfloat16>(L.Wb); p.shadow_ld = L.colsb;
  p.copy_counters = &ctx->at<Scalars>(L.scalars)->copy_pieces;
  CKC(ctx->K <= kFewPairs && tiles <= st->max_pairs
          ? launch_kernel((update_pair_kernel<1, false, true>), dim3(grid), dim3(kThreads),
                             UpShape<true>::kSmem, ctx->stream, 1, ma, mb, mc, p)
          : launch_kernel_if(tiles <= st->max_pairs, update_pair_kernel<1>, dim3(grid), dim3(kThreads), UpShape<false>::kSmem,
                             ctx->stream, 1, ma, mb, mc, p));
  return SFB_OK;
}

}  // namespace sfb
