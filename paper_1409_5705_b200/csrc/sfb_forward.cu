// Logits of multiclass logistic regression in bf16 mode for more than 128 samples, on pairs of CTAs where these are the faster ones:  Z (samples x rows of W) = X W^T
// with the softmax partials of each sample.  (Fewer samples, and the tf32 words: forward_kernel in sfb_tc.cu.)
//
// A pair (cta_group::2) owns a tile of 256 samples x bn classes, a CTA 128 of the samples in its TMEM; it loads its own samples and its
// half of the classes, 32 KB a k-block where a CTA with a 128 x 256 tile of its own loads 48 KB.  Two accumulators: the end of a
// tile runs beside the next one's products.
// What bounds the product is the MMA, as long as no pair waits: 160 tiles of 10,000 x 20,000 with 1,024 samples are 2.2 rounds of the
// 74 pairs, and a third round for twelve tiles took 85 of 390 us.  So the tiles of all rounds but the last whole one are taken
// whole, in step (the tiles that run at the same time share a block of W), and the k-blocks of the rest are shared out evenly, at
// most two tiles a pair and few parts a tile (Segments in sfb_tile.cuh).
// Warps: 0 TMA producer, 1 MMA issuer (leader CTA) and TMEM owner, 2..9 epilogue (TMEM lane quarter q, half h of the columns).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "sfb_tc.h"
#include "sfb_tile.cuh"

namespace sfb {
namespace {

using namespace ptx;

constexpr int PM = 256, BM = 128, BK = 64, UMMA_K = 16;
constexpr int kMaxN = 256, kChunk = 32, kEpi = 8;
constexpr int kStages = 5, kRing = 2;               // operand stages; slots per epilogue warp for the chunks of Z on their way out
constexpr int kInputs = 4;                          // parts of tiles on their way in, per epilogue warp
constexpr int kBytesA = BM * BK * 2, kBytesB = (kMaxN / 2) * BK * 2, kStage = kBytesA + kBytesB;
constexpr int kSlot = 32 * kChunk * 4;
constexpr int kThreads = 64 + 32 * kEpi;
constexpr int kBars = 2 * kStages + 4 + kEpi * kInputs;
constexpr int kSmem = kStages * kStage + kEpi * kRing * kSlot + kBars * 8 + 16 + 1024;
constexpr int kTmemCols = 512;
static_assert(kEpi * kInputs * kSlot <= kStages * kStage, "the parts land in the operand ring");

struct PairParams {
  int32_t M, N, m_off;         // samples end at M and begin at m_off; classes
  int32_t tilesM, tilesN, bn;  // tiles of 256 samples x bn classes, bn a multiple of 64
  int32_t kseg;                // k-blocks
  int32_t cut, whole;          // see Segments
  float2* part;                // [ceil(N / (bn / 2))][part_ld] (max, sum exp) per sample and half a tile's classes
  int64_t part_ld;
  float* partial;              // [pairs][2][kEpi][4] slots: what a pair leaves of a tile that another one completes ...
  uint32_t* ready;             // [pairs][2][kEpi]: ... and that it is there
  uint32_t* status;
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
forward_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmC, const __grid_constant__ PairParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sRing = smem + kStages * kStage;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sRing + kEpi * kRing * kSlot);
  uint64_t* full = bars;                             // full, tempty: the leader's are in use
  uint64_t* empty = bars + kStages;
  uint64_t* tfull = bars + 2 * kStages;
  uint64_t* tempty = tfull + 2;
  uint64_t* ifull = tfull + 4;                       // per epilogue warp and input buffer
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kBars);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int pair = blockIdx.x >> 1, half = p.bn / 2;
  const Segments segs(p.kseg, p.cut != 0, p.whole, p.tilesM * p.tilesN, pair, gridDim.x >> 1);
  // Sample block fastest: the tiles that run at the same time share blocks of W.
  auto tile_coords = [&](int tile, int& m0, int& n0) {
    const int tn = tile / p.tilesM;
    m0 = p.m_off + (tile - tn * p.tilesM) * PM;
    n0 = tn * p.bn;
  };
  pdl_launch_dependents();

  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&tfull[i], 1); mbar_init(&tempty[i], 2 * kEpi); }
    for (int i = 0; i < kEpi * kInputs; ++i) mbar_init(&ifull[i], 1);
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

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const uint64_t pol_keep = policy_evict_last(), pol_norm = policy_evict_normal();    // every tile reads the samples again
    uint32_t s = 0, ph = 0;
    bool ok = true;
    for (int i = 0; i < segs.n && ok; ++i) {
      const Segment sg = segs.get(i);
      int m0, n0;
      tile_coords(sg.tile, m0, n0);
      const int ma = m0 + static_cast<int>(rank) * BM, nb = n0 + static_cast<int>(rank) * half;
      for (int k = sg.k0; k < sg.k1; ++k) {
        if (!mbar_wait_warp(&empty[s], ph ^ 1, abort_flag)) { ok = false; break; }
        if (elect_one()) {
          if (rank == 0) mbar_expect_tx(&full[s], 2 * (kBytesA + half * BK * 2));
          const uint32_t bar = mapa_u32(smem_u32(&full[s]), 0);
          uint8_t* st = smem + s * kStage;
          tma_load_2d_pair(st, &tmA, k * BK, ma, bar, pol_keep);
          tma_load_2d_pair(st + kBytesA, &tmB, k * BK, nb, bar, pol_norm);
        }
        if (++s == static_cast<uint32_t>(kStages)) { s = 0; ph ^= 1; }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (rank == 0) {
      const uint32_t idesc = umma_idesc_bf16(PM, p.bn);
      uint32_t s = 0, ph = 0;
      bool ok = true;
      for (int i = 0; i < segs.n && ok; ++i) {
        const Segment sg = segs.get(i);
        const uint32_t a = i & 1, aph = (i >> 1) & 1, d_tmem = tmem_base + a * kMaxN;
        if (!mbar_wait_warp(&tempty[a], aph ^ 1, abort_flag)) { ok = false; break; }
        tc_fence_after();
        for (int kb = 0; kb < sg.k1 - sg.k0; ++kb) {
          if (!mbar_wait_warp(&full[s], ph, abort_flag)) { ok = false; break; }
          tc_fence_after();
          if (elect_one()) {
            const uint64_t da = umma_desc_k128(smem_u32(smem + s * kStage)), db = umma_desc_k128(smem_u32(smem + s * kStage + kBytesA));
#pragma unroll
            for (int k = 0; k < BK / UMMA_K; ++k) {
              const uint64_t adv = static_cast<uint64_t>(k * UMMA_K * 2 / 16);
              umma_bf16_pair(d_tmem, da + adv, db + adv, idesc, (kb | k) != 0 ? 1u : 0u);
            }
            umma_commit_pair(&empty[s], 3);
          }
          if (++s == static_cast<uint32_t>(kStages)) { s = 0; ph ^= 1; }
        }
        if (ok && elect_one()) umma_commit_pair(&tfull[a], 3);
      }
    }
  } else {
    // ---------------- epilogue ----------------
    const int e = warp - 2, q = warp & 3, h = e >> 2, cpw = half / kChunk;
    const uint32_t ring = smem_u32(sRing + e * kRing * kSlot);
    const int row0 = static_cast<int>(rank) * BM + q * 32;           // first of this warp's 32 samples within the tile
    const int at = static_cast<int>(rank) * kEpi + e;
    const uint32_t tempty_leader0 = mapa_u32(smem_u32(&tempty[0]), 0), tempty_leader1 = mapa_u32(smem_u32(&tempty[1]), 0);
    uint32_t stores = 0;
    bool ok = true;
    // a chunk from registers (a sample per lane) to a slot, when the copy that last used the slot has read it
    auto to_slot = [&](const uint32_t (&acc)[32]) {
      const uint32_t sl = ring + (stores % kRing) * kSlot;
      if (elect_one()) tma_wait_group_read<kRing - 1>();
      __syncwarp();
      slot_put(sl, lane, acc);
      fence_proxy_async_smem();
      __syncwarp();
      ++stores;
      return sl;
    };
    for (int i = 0; i < segs.n && ok; ++i) {
      const Segment sg = segs.get(i);
      int m0, n0;
      tile_coords(sg.tile, m0, n0);
      const uint32_t a = i & 1, aph = (i >> 1) & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(&tfull[a], aph, abort_flag))) { ok = false; break; }
      tc_fence_after();
      const uint32_t t_addr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + a * kMaxN + h * half;
      const bool leave = sg.k1 < p.kseg;
      const int from = leave ? pair : segs.first_part(sg), parts = pair - from, asks = parts * cpw;
      // Parts of the tile from the pairs before this one (the last tile of a pair): their sums come by bulk copies, kInputs of them
      // under way per warp, into the operand ring, which nothing uses any more.
      const uint32_t room = smem_u32(smem) + e * kInputs * kSlot;
      uint64_t* bar = ifull + e * kInputs;
      int asked = 0;
      auto ask = [&]() {                             // the next one: chunk by chunk, each from all of them in their order
        if (asked >= asks) return;
        const int c = asked / parts, w = asked - c * parts, b = asked % kInputs;
        if (elect_one()) {
          mbar_expect_tx(&bar[b], kSlot);
          bulk_load(room + b * kSlot, p.partial + ((static_cast<int64_t>(from + w) * 2 * kEpi + at) * 4 + c) * (kSlot / 4), kSlot, &bar[b]);
        }
        ++asked;
      };
      if (parts > 0) {
        for (int j = from; j < pair && ok; ++j) ok = __all_sync(0xffffffffu, lane != 0 || flag_wait(p.ready + j * 2 * kEpi + at, abort_flag));
        if (!ok) break;
        if (elect_one())
          for (int j = from; j < pair; ++j) p.ready[j * 2 * kEpi + at] = 0;             // for the next launch
        fence_proxy_async_all();
        __syncwarp();
        for (int b = 0; b < kInputs; ++b) ask();
      }
      float mx = -INFINITY, sum = 0.f;
      int taken = 0;
      const int row = m0 + row0 + lane;
#pragma unroll 1
      for (int c = 0; c < cpw && ok; ++c) {
        uint32_t acc[32];
        tmem_ld_32x32(t_addr + c * kChunk, acc);
        tmem_ld_wait();
        if (c + 1 == cpw) {                          // the last read of the accumulator: hand it back
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(a ? tempty_leader1 : tempty_leader0);
        }
        if (leave) {
          const uint32_t sl = to_slot(acc);
          if (elect_one()) {
            bulk_store(p.partial + ((static_cast<int64_t>(pair) * 2 * kEpi + at) * 4 + c) * (kSlot / 4), sl, kSlot);
            tma_commit_group();
          }
          continue;
        }
        for (int w = 0; w < parts && ok; ++w, ++taken) {
          const int b = taken % kInputs;
          ok = __all_sync(0xffffffffu, mbar_wait(&bar[b], (taken / kInputs) & 1, abort_flag));
          if (!ok) break;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float4 t = ld_shared_f4(slot_addr(room + b * kSlot, lane, j));
            acc[4 * j] = __float_as_uint(__uint_as_float(acc[4 * j]) + t.x);
            acc[4 * j + 1] = __float_as_uint(__uint_as_float(acc[4 * j + 1]) + t.y);
            acc[4 * j + 2] = __float_as_uint(__uint_as_float(acc[4 * j + 2]) + t.z);
            acc[4 * j + 3] = __float_as_uint(__uint_as_float(acc[4 * j + 3]) + t.w);
          }
          __syncwarp();
          ask();
        }
        if (!ok) break;
        const int col0 = n0 + h * half + c * kChunk;
        if (col0 >= p.N) continue;
        // running (max, sum exp) of the sample over this warp's classes of the tile
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
        const uint32_t sl = to_slot(acc);
        if (elect_one()) {
          tma_store_2d_at(&tmC, sl, col0, m0 + row0);
          tma_commit_group();
        }
      }
      if (leave && ok) {
        if (elect_one()) {
          tma_wait_group<0>();
          fence_proxy_async_all();
          __threadfence();
          st_release(p.ready + pair * 2 * kEpi + at, 1u);
        }
        __syncwarp();
      } else if (ok && n0 + h * half < p.N && row < p.M) {
        p.part[static_cast<int64_t>(n0 / half + h) * p.part_ld + row] = make_float2(mx, sum);
      }
    }
    if (elect_one()) tma_wait_group<0>();
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
  if (warp == 1) { tc_fence_after(); tmem_dealloc_pair(tmem_base, kTmemCols); }
}

// Cycles of a plan: its k-blocks on a pair at the MMAs' rate or 60 bytes a cycle and SM, at least the 8,000 that the end of a tile of 256
// classes takes; 7,000 from the start to the first MMA and from the last one to the results; 9,000 and 2,000 a part to leave and to
// take over parts of tiles, of which there are no more than pay for that.  (Fitted to 47 shapes, 64 to 100,000 classes, 170 to 20,000 features, 129 to 1,024 samples; whether
// the pairs are taken at all: forward_pair_pays.  us of the product, forward_kernel / here: 10,000 x 20,000 with 1,024 samples 376 / 283, 11,133 x
// 3,364 with 1,024 79 / 67.)
constexpr int64_t kNarrowRows = 4096;               // up to which narrower tiles are looked at (they have more partials)
struct PairPlan { int bn, cut, whole, pairs; double cost; };
PairPlan plan_pairs(int64_t n, int64_t rows, int64_t cols, int64_t max_pairs) {
  PairPlan best{};
  const int64_t kseg = (cols + BK - 1) / BK, tm = (n + PM - 1) / PM;
  for (int bn = kMaxN; bn >= (rows <= kNarrowRows ? 64 : kMaxN); bn -= 64) {
    const int64_t tiles = tm * ((rows + bn - 1) / bn), rounds = (tiles + max_pairs - 1) / max_pairs, full = tiles / max_pairs;
    const double per_kb = std::max(2.1 * bn, (BM + bn / 2) * BK * 2 / 60.0);
    const double tile = std::max(static_cast<double>(kseg) * per_kb, 8000.0 * bn / kMaxN);
    PairPlan p{bn, 0, 0, static_cast<int>(std::min(tiles, max_pairs)), static_cast<double>(rounds) * tile + 7000.0};
    const int64_t whole = std::max<int64_t>(0, full - 1) * max_pairs, rest = tiles - whole;
    const int64_t most = full > 0 ? max_pairs : std::max<int64_t>(1, std::min(max_pairs, rest * kseg / 4));
    for (int64_t parts = 2; (full > 0 && parts == 2) || (parts - 1) * rest < most; ++parts) {      // of a tile
      const int64_t pairs = full > 0 ? max_pairs : std::min(most, parts * rest), shared = (rest * kseg + pairs - 1) / pairs;
      const double cost = static_cast<double>(whole / max_pairs) * tile + static_cast<double>(shared) * per_kb + 16000.0 + 2000.0 * static_cast<double>(parts);
      if (cost < p.cost && rest % pairs != 0) p = PairPlan{bn, 1, static_cast<int>(whole), static_cast<int>(pairs), cost};
    }
    if (bn == kMaxN || p.cost < 0.97 * best.cost) best = p;
  }
  return best;
}
PairPlan plan_pairs(const sfb_ctx* ctx, int64_t n) {
  const int64_t most = std::min(static_cast<TcState*>(ctx->tc)->max_pairs, std::min(sm_count(), kModelSms) / 2);
  return plan_pairs(n, ctx->cfg.rows, ctx->cfg.cols, most);
}

}  // namespace

double forward_pair_cost(int64_t n, int64_t rows, int64_t cols) { return plan_pairs(n, rows, cols, kModelSms / 2).cost; }
// Against a product of `other` cycles (by forward_cost) with `other_groups` softmax partials a sample.  The two models were fitted apart: held
// against each other, on 1,278 shapes of 129 to 2,048 samples, 2 to 300,000 classes and 32 to 24,000 features, the pairs are the better
// ones where a third more, 13,000 cycles where tiles are cut, and 2,400 per 32 partials that the softmax has to merge (a pair's tile
// of 256 classes leaves two) still come to less.  With that the choice costs a step, fused or by calls, more than 3 % in 29 of 2,556 cases,
// by the models as they are in 271 (4,047 more shapes, against the better of the two: steps 0.7 % longer, 2.1 % by the models as they are,
// 2.9 % on forward_kernel alone): 36,667 x 912 with 364 samples 145 us on forward_kernel, 174 on pairs, 78,798 x 1,716 with 156
// 396 and 458, 121 x 3,772 with 180 35.8 and 39.6.
bool forward_pair_pays(int64_t n, int64_t rows, int64_t cols, double other, int64_t other_groups, int* parts) {
  const PairPlan p = plan_pairs(n, rows, cols, kModelSms / 2);
  const int64_t half = p.bn / 2, tiles = (n + PM - 1) / PM * ((rows + p.bn - 1) / p.bn);
  const double groups = static_cast<double>((rows + half - 1) / half - other_groups);
  if (1.35 * p.cost + (p.cut ? 13000.0 : 0.0) + 2400.0 * groups / 32.0 >= other) return false;
  *parts = p.cut ? std::max(2, static_cast<int>((p.pairs + tiles - p.whole - 1) / (tiles - p.whole))) : 1;
  return true;
}
int64_t forward_pair_groups(int64_t rows) { return rows <= kNarrowRows ? (rows + 31) / 32 : (rows + kMaxN / 2 - 1) / (kMaxN / 2); }
size_t forward_pair_partial_bytes(int64_t pairs) { return static_cast<size_t>(pairs) * 2 * kEpi * 4 * kSlot; }
int64_t forward_pair_cut(int64_t n, int64_t rows, int64_t cols) {
  const PairPlan p = plan_pairs(n, rows, cols, kModelSms / 2);
  return p.cut ? p.pairs : 0;
}
size_t forward_pair_ready_bytes() { return static_cast<size_t>(kModelSms / 2) * 2 * kEpi * 4; }

cudaError_t forward_pair_prepare(int* max_pairs) { return prepare_pair_kernel(forward_pair_kernel, kThreads, kSmem, max_pairs); }

cudaError_t forward_pair(sfb_ctx* ctx, int64_t off, int64_t n, int* pw) {
  TcState* st = static_cast<TcState*>(ctx->tc);
  const Layout& L = ctx->lay;
  const int64_t rows = ctx->cfg.rows, cols = ctx->cfg.cols;
  PairPlan plan = plan_pairs(ctx, n);
  if (plan.cut && plan.pairs > L.cut_pairs) {      // (a device with fewer pairs than the workspace was laid out for: whole tiles)
    const int64_t tiles = (n + PM - 1) / PM * ((rows + plan.bn - 1) / plan.bn);
    plan.cut = plan.whole = 0;
    plan.pairs = static_cast<int>(std::min<int64_t>(tiles, plan.pairs));
  }
  CUtensorMap ma, mb, mc;
  if (!make_map(st, &ma, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, ctx->at<uint16_t>(L.Xb), cols, ctx->K, L.colsb * 2, BK, BM) ||
      !make_map(st, &mb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, ctx->at<uint16_t>(L.Wb), cols, rows, L.colsb * 2, BK, plan.bn / 2) ||
      !make_map(st, &mc, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, ctx->at<float>(L.ZT), rows, off + n, round_up(rows, 32) * 4, kChunk, 32))
    return cudaErrorInvalidValue;
  PairParams p{};
  p.M = static_cast<int32_t>(off + n); p.N = static_cast<int32_t>(rows); p.m_off = static_cast<int32_t>(off);
  p.tilesM = static_cast<int32_t>((n + PM - 1) / PM); p.tilesN = static_cast<int32_t>((rows + plan.bn - 1) / plan.bn);
  p.bn = plan.bn; p.kseg = static_cast<int32_t>((cols + BK - 1) / BK);
  p.cut = plan.cut; p.whole = plan.whole;
  p.part = ctx->at<float2>(L.part); p.part_ld = ctx->K;
  p.partial = ctx->at<float>(L.partial); p.ready = ctx->at<uint32_t>(L.ready); p.status = ctx->at<uint32_t>(L.status);
  *pw = plan.bn / 2;
  return launch_kernel_if(p.tilesM * p.tilesN <= plan.pairs, forward_pair_kernel, dim3(2u * static_cast<unsigned>(plan.pairs)),
                          dim3(kThreads), kSmem, ctx->stream, 1, ma, mb, mc, p);
}

}  // namespace sfb

// ---------------------------------------------------------------------------------------------------------
// Logits of up to 64 samples, a worker's mini-batch: the classes are the rows of the accumulator (128 of them a CTA), the samples its
// columns.
// Such a product is bound by the way of W to the SMs and by latency.  With the samples as rows, 128 of which the MMA computes
// whatever their number, an SM had 64 classes and issued four MMAs of 64 columns a k-block of 8 KB of W: 79 CTAs at 400 cycles a
// k-block for 4,999 x 3,004.  Here an MMA has as many columns as there are samples, a k-block is 16 KB of W, and the contraction
// is cut over clusters of up to four CTAs as long as all of them are resident.  us of a worker's call, forward_kernel / here:
// 4,999 x 3,004 with 8, 37, 64 samples 20.5, 20.6, 21.7 / 12.7, 14.5, 17.9; 500 x 3,004 18.2, 28.6, 28.9 / 11.2, 12.6, 13.0.  (With
// the rounding of the samples in this kernel instead of one of its own before it, eight k-blocks of loads under way: 11.4, 16.3,
// 20.9; every CTA then reads all samples in fp32.)
// Warps: 0 TMA producer, 1 MMA issuer and TMEM owner, 2..9 epilogue: parts through shared memory, Z by rows, softmax partials of 32
// classes.
// ---------------------------------------------------------------------------------------------------------
namespace sfb {
namespace {

constexpr int kFewN = 64, kFewStages = 8, kFewParts = 4;
constexpr int kFewA = BM * BK * 2, kFewB = kFewN * BK * 2, kFewStage = kFewA + kFewB;
constexpr int kFewXchg = 4 * kFewN * 32 * 4;        // [lane quarter][sample][32 classes] fp32
constexpr int kFewBars = 2 * kFewStages + 1;
constexpr int kFewSmem = kFewStages * kFewStage + kFewXchg + kFewBars * 8 + 16 + 1024;
constexpr int kFewTmem = 64;

struct FewParams {
  int32_t n, off;              // samples of this call, first pair
  int32_t rows, tiles;         // classes; tiles of 128 of them
  int32_t kseg, parts;         // k-blocks; CTAs of a cluster, which share them
  float* Z;
  int64_t ldz;
  float2* part;
  int64_t part_ld;
  uint32_t* status;
};

__global__ void __launch_bounds__(kThreads, 1)
forward_few_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const __grid_constant__ FewParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* xchg = smem + kFewStages * kFewStage;
  uint64_t* bars = reinterpret_cast<uint64_t*>(xchg + kFewXchg);
  uint64_t* full = bars;
  uint64_t* empty = bars + kFewStages;
  uint64_t* done = bars + 2 * kFewStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kFewBars);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int tile = static_cast<int>(blockIdx.x) / p.parts, mine = static_cast<int>(blockIdx.x) % p.parts;     // (its rank in the cluster)
  const int kbeg = mine * p.kseg / p.parts, nk = (mine + 1) * p.kseg / p.parts - kbeg;
  pdl_launch_dependents();
  if (threadIdx.x == 0) {
    for (int i = 0; i < kFewStages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(done, 1);
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&tmW); prefetch_tmap(&tmX);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, kFewTmem); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();

  if (warp == 0) {
    const uint64_t pol_keep = policy_evict_last();      // every tile reads the samples
    bool ok = true;
    for (int k = 0; k < nk && ok; ++k) {
      const uint32_t s = k % kFewStages, ph = (k / kFewStages) & 1;
      ok = mbar_wait_warp(&empty[s], ph ^ 1, abort_flag);
      if (ok && elect_one()) {
        mbar_expect_tx(&full[s], kFewA + ((p.n + 7) & ~7) * BK * 2);
        tma_load_2d(smem + s * kFewStage, &tmW, (kbeg + k) * BK, tile * BM, &full[s]);
        tma_load_2d_hint(smem + s * kFewStage + kFewA, &tmX, (kbeg + k) * BK, p.off, &full[s], pol_keep);
      }
    }
  } else if (warp == 1) {
    const uint32_t idesc = umma_idesc_bf16(BM, (static_cast<uint32_t>(p.n) + 15u) & ~15u);
    bool ok = true;
    for (int k = 0; k < nk && ok; ++k) {
      const uint32_t s = k % kFewStages, ph = (k / kFewStages) & 1;
      ok = mbar_wait_warp(&full[s], ph, abort_flag);
      tc_fence_after();
      if (ok && elect_one()) {
        const uint64_t da = umma_desc_k128(smem_u32(smem + s * kFewStage)), db = umma_desc_k128(smem_u32(smem + s * kFewStage + kFewA));
#pragma unroll
        for (int j = 0; j < BK / UMMA_K; ++j) {
          const uint64_t adv = static_cast<uint64_t>(j * UMMA_K * 2 / 16);
          umma_bf16(tmem_base, da + adv, db + adv, idesc, (k | j) != 0 ? 1u : 0u);
        }
        umma_commit(&empty[s]);
      }
    }
    if (ok && elect_one()) umma_commit(done);
  } else {
    const int e = warp - 2, q = warp & 3, h = e >> 2;
    const int r4 = lane >> 3, c8 = lane & 7;         // eight lanes take 32 classes of a sample
    // ---------------- the accumulator: lane = class, column = sample ----------------
    if (mbar_wait_warp(done, 0, abort_flag) && h * 32 < p.n) {
      tc_fence_after();
      uint32_t acc[32];
      tmem_ld_32x32(tmem_base + (static_cast<uint32_t>(q * 32) << 16) + h * 32, acc);
      tmem_ld_wait();
      float* out = reinterpret_cast<float*>(xchg) + (q * kFewN + h * 32) * 32 + lane;
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (h * 32 + j < p.n) out[j * 32] = __uint_as_float(acc[j]);
    }
    __syncwarp();
    if (p.parts > 1) { cluster_arrive(); cluster_wait(); }
    else asm volatile("bar.sync 1, 256;" ::: "memory");
    // units of 4 samples x 32 classes, 8 lanes a sample; a unit's sums are in rank order
    const int units = 4 * ((p.n + 3) / 4);
    for (int u = mine * kEpi + e; u < units; u += p.parts * kEpi) {
      const int uq = u & 3, j = (u >> 2) * 4 + r4, grp = tile * 4 + uq;
      const int64_t r0 = static_cast<int64_t>(grp) * 32 + 4 * c8;
      const uint32_t at = smem_u32(xchg) + ((uq * kFewN + j) * 32 + 4 * c8) * 4;      // (j < 64: n is at most that)
      float4 v = ld_cluster_f4(at, 0);
      for (int r = 1; r < p.parts; ++r) {
        const float4 t = ld_cluster_f4(at, r);
        v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
      }
      const int left = p.rows - static_cast<int>(r0);                                   // classes from here on
      float mx = left > 0 ? v.x : -INFINITY;
      if (left > 1) mx = fmaxf(mx, v.y);
      if (left > 2) mx = fmaxf(mx, v.z);
      if (left > 3) mx = fmaxf(mx, v.w);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      float sum = (left > 0 ? __expf(v.x - mx) : 0.f) + (left > 1 ? __expf(v.y - mx) : 0.f) + (left > 2 ? __expf(v.z - mx) : 0.f) +
                  (left > 3 ? __expf(v.w - mx) : 0.f);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (j < p.n && grp * 32 < p.rows) {
        *reinterpret_cast<float4*>(p.Z + (p.off + j) * p.ldz + r0) = v;               // (its pitch is a multiple of 32)
        if (c8 == 0) p.part[static_cast<int64_t>(grp) * p.part_ld + p.off + j] = make_float2(mx, sum);
      }
    }
  }
  if (p.parts > 1) {
    __syncwarp();
    if (warp < 2) { cluster_arrive(); cluster_wait(); }                // (the others have been there)
    cluster_arrive();                                                  // no CTA leaves while a peer still reads its part
    cluster_wait();
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(p.status, SFB_STATUS_TIMEOUT);
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
    __syncthreads();
  }
  if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, kFewTmem); }
}

// CTAs of a cluster: as many as keep all of them resident and leave each four k-blocks.
int few_parts(int64_t tiles, int64_t kseg, const int (&most)[kFewParts + 1]) {
  int best = 1;
  for (int s = 2; s <= kFewParts; ++s)
    if (tiles <= most[s] && kseg >= 4 * s) best = s;
  return best;
}

}  // namespace

// Where two CTAs share a tile (up to 74 tiles); fewer than one tile per SM leaves SMs idle, which pays for few samples or where W comes from
// HBM.  us of a worker's call, forward_kernel / here, 3,004 features: 9,400 classes with 37 and 64 samples 23.2, 24.9 / 21.5, 24.2; 10,000
// with 8 and 64 23.5, 26.0 / 19.4, 29.8; 15,000 with 16 and 37 25.0, 27.3 / 22.0, 30.8; 10,000 x 20,000 with 8 and 64 119, 128 / 80, 88.
// (118 tiles are the 15,000 classes up to which it was measured.  From 15,105 to 30,000 up to 8 samples would take 0.74 to 0.90 times as long
// here too, 9 to 16 0.83 to 0.97, 17 to 32 0.94 to 1.06, more 1.08 to 1.39.)
// Above 40 samples the end of a tile (Z and partials, by rows, through shared memory) takes longer than forward_kernel's, which fewer than 12
// k-blocks do not repay in a call of its own: factors with 49 to 64 samples, up to 500 features 1.06 to 1.20 times as long as with
// forward_kernel, 1,000 to 1,500 0.84 times; 33 to 40 samples 1.02 and 0.85.  (In a step, beside the kernels around it, the same sizes
// take 0.90 to 1.04 times as long.)  And forward_kernel cuts the longest contractions into eight parts where there are few
// tiles: up to 512 classes, 20,000 to 24,000 features 1.04 times as long here, 14,000 to 18,000 0.95.
bool forward_few_fits(int64_t n, int64_t rows, int64_t cols, bool step) {
  const int64_t tiles = (rows + BM - 1) / BM, kseg = (cols + BK - 1) / BK;
  if (n > kFewN || (!step && n > 40 && kseg < 12) || (tiles <= 4 && cols > 18000)) return false;
  return tiles <= kModelSms / 2 || (tiles <= 118 && (n <= 24 || rows * cols >= 100000000));
}
int64_t forward_few_groups(int64_t rows) { return (rows + 31) / 32; }

cudaError_t forward_few_prepare(int (&most)[5]) {
  static_assert(kFewParts + 1 == 5, "");
  cudaError_t e = cudaFuncSetAttribute(forward_few_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFewSmem);
  for (int s = 1; s <= kFewParts && e == cudaSuccess; ++s) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(s, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kFewSmem;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = s; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(&most[s], forward_few_kernel, &cfg);
  }
  return e;
}

cudaError_t forward_few(sfb_ctx* ctx, int64_t off, int64_t n) {
  TcState* st = static_cast<TcState*>(ctx->tc);
  const Layout& L = ctx->lay;
  const int64_t rows = ctx->cfg.rows, cols = ctx->cfg.cols;
  CUtensorMap mw, mx;
  if (!make_map(st, &mw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, ctx->at<uint16_t>(L.Wb), cols, rows, L.colsb * 2, BK, BM) ||
      !make_map(st, &mx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, ctx->at<uint16_t>(L.Xb), cols, ctx->K, L.colsb * 2, BK,
                static_cast<int>(round_up(n, 8))))
    return cudaErrorInvalidValue;
  FewParams p{};
  p.n = static_cast<int32_t>(n); p.off = static_cast<int32_t>(off);
  p.rows = static_cast<int32_t>(rows); p.tiles = static_cast<int32_t>((rows + BM - 1) / BM);
  p.kseg = static_cast<int32_t>((cols + BK - 1) / BK);
  p.parts = few_parts(p.tiles, p.kseg, st->few);
  p.Z = ctx->at<float>(L.ZT); p.ldz = round_up(rows, 32);
  p.part = ctx->at<float2>(L.part); p.part_ld = ctx->K;
  p.status = ctx->at<uint32_t>(L.status);
  return launch_kernel(forward_few_kernel, dim3(static_cast<unsigned>(p.tiles * p.parts)), dim3(kThreads), kFewSmem, ctx->stream, p.parts,
                       mw, mx, p);
}

}  // namespace sfb
