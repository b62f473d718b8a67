// Products on the tensor cores whose operands carry each value as a (hi | lo) pair of 16-bit words, three products per term:
//     A B^T = A_hi B_hi^T + A_lo B_hi^T + A_hi B_lo^T.
// Two forms of the pair, chosen by the precision mode:
//   bf16 mode, metric learning and sparse coding (their u comes from a cancelling residual):  hi = bf16(x), lo = bf16(x - hi);
//     16 bits of x, no scale.
//   fp32 mode:  hi = fp16(s x), lo = fp16(2^11 (s x - hi)) with a power of two s per row of the operand that puts the row's
//     largest entry at 2^13.  23 of fp32's 24 bits (the last one is lost for a quarter of the values), for entries down to
//     2^-27 of the row's largest; below that the error stays at 2^-49 of the largest.  Twice the rate of tf32 words in half the
//     bytes, with the same number of bits.
// and the per-step work around them: operand packing, the factors of metric learning and sparse coding (Section 2: z = W v
// with v = x - y; Figure 3: ISTA codes, u = W a - x), the logits of logistic regression in fp32 mode.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "sfb_tc.h"
#include "sfb_tile.cuh"

namespace sfb {
namespace {

using namespace ptx;

constexpr float kLoScale = 2048.f;                  // of the lo word in the fp16 form

// Epilogues of the product  D (samples x N) = A * B^T:
//   F_STORE    C = D                                                                  (z = W v)
//   F_SUB      C = D - aux, also as a pair                                            (sparse coding: r = W a - x)
//   F_ISTA     C <- soft(C - D / L, lambda / L) in place, also as a pair              (ISTA step)
//   F_ISTAG    C <- soft(C - (D - C2) / L, lambda / L) in place, also as a pair       (the same on W^T W; C2 = W^T x)
//   F_ISTA0    C2 (unless null) = D and C = soft(D / L, lambda / L), also as a pair   (first iterate)
//   F_GRAM     C (unless null) = D and, in the bf16 form, D as a pair, of a symmetric D: only the tiles that reach the diagonal or
//              lie above it are formed, the others are written as their mirror images (W^T W)
enum FwdEpi { F_STORE = 0, F_SUB = 1, F_ISTA = 2, F_ISTAG = 3, F_ISTA0 = 4, F_GRAM = 5 };
// The result also goes out as an operand.  (fp32 mode has W^T W for the power iteration only.)
template <int EPI, bool F16>
constexpr bool kPairOut = EPI != F_STORE && !(EPI == F_GRAM && F16);
template <int EPI>
constexpr bool kIsta = EPI == F_ISTA || EPI == F_ISTAG || EPI == F_ISTA0;

struct SplitParams {
  int32_t M, N, m_off;         // samples end at M and begin at m_off (a worker's slice); output columns
  int32_t tilesM, tilesN, bn;  // tiles of 256 samples x bn columns, bn a multiple of 32
  int32_t a_rows;              // rows of A per box (fewer than 128 for a slice of few samples)
  int32_t stages, kseg;        // operand ring; k-blocks
  int32_t a_lo, b_lo;          // first column of the lo halves
  int32_t cut;                 // the k-blocks are shared out; else the tiles are taken whole, pair by pair
  float* partial;              // [pairs][2][kEpi][4][8][32] float4: sums of the tile that a pair leaves to another one ...
  uint32_t* ready;             // [pairs][2][kEpi]: ... and that they are there
  int32_t four;                // F_GRAM: with the fourth term A_lo B_lo
  float* C;
  int64_t ldc;
  const float* aux;            // F_SUB: the matrix subtracted; F_ISTA, F_ISTAG: the matrix updated; [M x ldaux]
  int64_t ldaux;
  float* C2;                   // [M x ldc]
  int32_t copies;              // F_SUB, F_ISTA, F_ISTAG: aux and C2 as tensor maps (16-byte pitch and address); the first row of
  int32_t aux_row0;            // aux's map
  const Scalars* sc;           // F_ISTA*: 1 / L
  float lam;                   // F_ISTA*: lambda
  uint16_t* split;             // where kPairOut: [M x ld_split] receives hi at column n and lo at column split_half + n
  int64_t ld_split;
  int32_t split_half;          // padded N (a multiple of 64); columns N..split_half-1 are written as zeros
  // fp16 form: inverse scales of A per row, of B per column of D, a factor for all (null: 1)
  const float* ia;
  const float* ib;
  const float* iab;
  // ... and of the pair that goes out, per row: from the largest value so far, most_in, whose inverse scale goes to io and which
  // with the values of this product becomes most_out.  (Iterations that diverge, on an L below ||W||^2 / 2, keep their precision as
  // long as no value grows by more than 2^12 in one of them.)
  const float* most_in;
  float* most_out;
  float* io;
  uint32_t* status;
};

// ---------------------------------------------------------------------------------------------------------
// Pairs
// ---------------------------------------------------------------------------------------------------------
// The power of two that brings a largest entry m into [2^top, 2^(top+1)); the largest one, 2^120, for 0 (its inverse is looked
// at for the smallest scale of several rows), 1 for what is not finite.
__device__ __forceinline__ float pow2_scale(float m, int top) {
  const int ex = ((__float_as_int(m) >> 23) & 255) - 127;
  if (ex == 128) return 1.f;
  return __int_as_float((min(max(top - ex, -120), 120) + 127) << 23);
}
constexpr int kTop = 3;                             // of the largest value so far of a sample's codes and residuals
// two neighbouring values (already scaled in the fp16 form) as packed words
template <bool F16>
__device__ __forceinline__ void split2(float f0, float f1, uint32_t& hi, uint32_t& lo) {
  if (F16) {
    const __half2 h = __floats2half2_rn(f0, f1);
    const float2 b = __half22float2(h);
    const __half2 l = __floats2half2_rn((f0 - b.x) * kLoScale, (f1 - b.y) * kLoScale);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
  } else {
    const __nv_bfloat162 h = __floats2bfloat162_rn(f0, f1);
    const float2 b = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(f0 - b.x, f1 - b.y);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    lo = *reinterpret_cast<const uint32_t*>(&l);
  }
}
template <bool F16>
__device__ __forceinline__ void put_pair4(uint16_t* d, int64_t half, float4 v) {
  uint32_t h0, l0, h1, l1;
  split2<F16>(v.x, v.y, h0, l0);
  split2<F16>(v.z, v.w, h1, l1);
  *reinterpret_cast<uint2*>(d) = make_uint2(h0, h1);
  *reinterpret_cast<uint2*>(d + half) = make_uint2(l0, l1);
}
__device__ __forceinline__ float4 scale4(float4 v, float s) { return make_float4(v.x * s, v.y * s, v.z * s, v.w * s); }

// ---------------------------------------------------------------------------------------------------------
// The product kernel.  Pairs of CTAs (cta_group::2): 256 samples x bn columns per tile, CTA r of the pair holds 128 of the
// samples in its TMEM, loads its own samples and its own half of the columns.  What bounds such a product is the way of the
// operands into the tensor core: with a CTA of its own per 128 x 160 tile an SM's shared memory moved 9 KB per 80 cycles of
// MMA and took 75 bytes per cycle from L2 (0.70 of the tensor rate); a pair at 256 columns moves 8 KB per 128 cycles and
// takes 43.  One stage holds the k-block of all four operand halves, from which the three products are issued.
// The tensor core rounds an fp32 accumulator towards zero at every instruction, so the error grows with the instructions that
// add to one.  Hence the cross terms have an accumulator of their own (2^-8 or 2^-11 of the size), and A_hi B_hi is drained
// every eight k-blocks, while the A_lo B_hi of the last of them run: the epilogue warps add it to sums in their registers.
// A product of fewer tiles than pairs is cut along the contraction: its k-blocks are shared out evenly, a pair
// has a run of them that begins within one tile and ends within another (or the same).  The part at the end of a run, which
// does not reach the end of its tile, is computed first and left in memory; the part at the beginning, which completes a tile,
// last: the parts that it waits for come from the pairs before this one.  The sums are in the order of the pairs, so they do
// not depend on timing.
// Warps: 0 TMA producer, 1 MMA issuer (leader CTA) and TMEM owner, 4..11 epilogue; the first four give their registers to
// the epilogue (384 threads x 168 = 128 x 40 + 256 x 232).
// Rates: see plan_width.
// ---------------------------------------------------------------------------------------------------------
constexpr int PM = 256, BM = 128, BK = 64, UMMA_K = 16;
constexpr int kMaxN = 256;
constexpr int kBytesA = BM * BK * 2;
constexpr int kChunk = 32, kEpi = 8;
constexpr int kStagesMax = 6;
constexpr int kRegion = 192 << 10;                  // of the operand ring
constexpr int kSlot = 32 * kChunk * 4;              // per epilogue warp: 32 rows x 32 columns of fp32
// k-blocks of A_hi B_hi per drain.  Sparse coding in fp32 mode drains every one: the gradient of its iterations cancels, and the
// rounding towards zero of the 32 instructions of eight k-blocks made the codes up to 2.5 times less exact than those of the FMA
// kernels (676 x 1,148, K = 649, 20 iterations; one drain a k-block: 0.95).
template <int EPI, bool F16>
constexpr int kDrain = F16 && EPI != F_STORE ? 1 : 8;
constexpr int kThreads = 128 + 32 * kEpi;
constexpr int kInputs = 3;                          // buffers per epilogue warp for what the end of the last tile reads
static_assert((4 + kInputs - 1) * kEpi * kSlot <= kRegion, "see there");
constexpr int kBars = 2 * kStagesMax + 4 + kEpi * kInputs;
constexpr int kSmem = kRegion + kEpi * kSlot + kBars * 8 + 16 + 1024;
constexpr int kTmemCols = 512;

inline int ring_stages(int bn) { return std::min(kStagesMax, kRegion / (2 * kBytesA + bn * BK * 2)); }

// F_GRAM: the tiles of column block tn that are formed are row blocks 0 .. sym_row_blocks - 1 (those that begin above the
// column block's end); numbered column block by column block.
__host__ __device__ __forceinline__ int sym_row_blocks(int tilesM, int bn, int tn) {
  const int n = ((tn + 1) * bn - 1) / PM + 1;
  return n < tilesM ? n : tilesM;
}
__host__ __device__ __forceinline__ int sym_tiles(int tilesM, int tilesN, int bn) {
  int n = 0;
  for (int tn = 0; tn < tilesN; ++tn) n += sym_row_blocks(tilesM, bn, tn);
  return n;
}
// Sample block fastest: the tiles that run at the same time share blocks of W.
template <int EPI>
__device__ __forceinline__ void tile_coords(const SplitParams& p, int tile, int& m0, int& n0) {
  int tn = 0;
  if (EPI == F_GRAM) {
    for (int n; tile >= (n = sym_row_blocks(p.tilesM, p.bn, tn)); ++tn) tile -= n;
  } else {
    tn = tile / p.tilesM;
    tile -= tn * p.tilesM;
  }
  m0 = p.m_off + tile * PM;
  n0 = tn * p.bn;
}

template <int EPI, bool F16>
__global__ void __launch_bounds__(kThreads, 1)
split_product_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                     const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmY,
                     const __grid_constant__ SplitParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kRegion + kEpi * kSlot);
  uint64_t* full = bars;                             // full, mempty, cempty: the leader's are in use
  uint64_t* empty = bars + kStagesMax;
  uint64_t* mfull = bars + 2 * kStagesMax;
  uint64_t* mempty = mfull + 1;
  uint64_t* cfull = mfull + 2;
  uint64_t* cempty = mfull + 3;
  uint64_t* ifull = mfull + 4;                       // per epilogue warp and buffer
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kBars);
  volatile uint32_t* abort_flag = tmem_slot + 1;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int ST = p.stages, half = p.bn / 2;
  const int bytesB = half * BK * 2, stage_bytes = 2 * kBytesA + 2 * bytesB;
  const int ntiles = EPI == F_GRAM ? sym_tiles(p.tilesM, p.tilesN, p.bn) : p.tilesM * p.tilesN;
  const int pair = blockIdx.x >> 1;
  const Segments segs(p.kseg, p.cut != 0, 0, ntiles, pair, gridDim.x >> 1);

  pdl_launch_dependents();
  if (threadIdx.x == 0) {
    for (int i = 0; i < ST; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(mfull, 1); mbar_init(mempty, 2 * kEpi);
    mbar_init(cfull, 1); mbar_init(cempty, 2 * kEpi);
    for (int i = 0; i < kEpi * kInputs; ++i) mbar_init(&ifull[i], 1);
    *abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&tmA); prefetch_tmap(&tmB);
  }
  if (warp == 1) { tmem_alloc_pair(tmem_slot, kTmemCols); tmem_relinquish_pair(); }
  tc_fence_before();
  __syncthreads();
  cluster_arrive();
  cluster_wait();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == 0) {
      // ---------------- TMA producer ----------------
      const uint64_t pol_keep = policy_evict_last(), pol_norm = policy_evict_normal();
      uint32_t s = 0, ph = 0;
      bool ok = true;
      for (int i = 0; i < segs.n && ok; ++i) {
        const Segment sg = segs.get(i);
        int m0, n0;
        tile_coords<EPI>(p, sg.tile, m0, n0);
        const int ma = m0 + static_cast<int>(rank) * BM, nb = n0 + static_cast<int>(rank) * half;
        for (int k = sg.k0; k < sg.k1; ++k) {
          const int x = k * BK;
          if (!mbar_wait_warp(&empty[s], ph ^ 1, abort_flag)) { ok = false; break; }
          if (elect_one()) {
            if (k + 4 < sg.k1) {                        // B streams from HBM when it is larger than L2: asked for early
              tma_prefetch_2d(&tmB, x + 4 * BK, nb);
              tma_prefetch_2d(&tmB, p.b_lo + x + 4 * BK, nb);
            }
            if (rank == 0) mbar_expect_tx(&full[s], 2 * (2 * p.a_rows * BK * 2 + 2 * bytesB));
            const uint32_t bar = mapa_u32(smem_u32(&full[s]), 0);
            uint8_t* st = smem + s * stage_bytes;
            tma_load_2d_pair(st, &tmA, x, ma, bar, pol_keep);
            tma_load_2d_pair(st + kBytesA, &tmA, p.a_lo + x, ma, bar, pol_keep);
            tma_load_2d_pair(st + 2 * kBytesA, &tmB, x, nb, bar, pol_norm);
            tma_load_2d_pair(st + 2 * kBytesA + bytesB, &tmB, p.b_lo + x, nb, bar, pol_norm);
          }
          if (++s == static_cast<uint32_t>(ST)) { s = 0; ph ^= 1; }
        }
      }
    } else if (warp == 1 && rank == 0) {
      // ---------------- MMA issuer ----------------
      const uint32_t idesc = F16 ? umma_idesc_fp16(PM, p.bn) : umma_idesc_bf16(PM, p.bn);
      const uint32_t d_main = tmem_base, d_cross = tmem_base + kMaxN;
      uint32_t s = 0, ph = 0, g = 0;
      bool ok = true;
      for (int i = 0; i < segs.n && ok; ++i) {
        const Segment sg = segs.get(i);
        const int nk = sg.k1 - sg.k0;
        for (int kb = 0; kb < nk; ++kb) {
          const int kc = kb % kDrain<EPI, F16>;
          if (!mbar_wait_warp(&full[s], ph, abort_flag) || (kc == 0 && !mbar_wait_warp(mempty, (g & 1) ^ 1, abort_flag)) ||
              (kb == 0 && !mbar_wait_warp(cempty, (i & 1) ^ 1, abort_flag))) { ok = false; break; }
          tc_fence_after();
          const bool drained = kc == kDrain<EPI, F16> - 1 || kb + 1 == nk;
          if (elect_one()) {
            uint8_t* st = smem + s * stage_bytes;
            const uint64_t dah = umma_desc_k128(smem_u32(st)), dal = umma_desc_k128(smem_u32(st + kBytesA));
            const uint64_t dbh = umma_desc_k128(smem_u32(st + 2 * kBytesA)), dbl = umma_desc_k128(smem_u32(st + 2 * kBytesA + bytesB));
#pragma unroll
            for (int k = 0; k < BK / UMMA_K; ++k) {
              const uint64_t adv = static_cast<uint64_t>(k * UMMA_K * 2 / 16);
              umma_bf16_pair(d_main, dah + adv, dbh + adv, idesc, (kc | k) != 0 ? 1u : 0u);      // A_hi B_hi
              umma_bf16_pair(d_cross, dah + adv, dbl + adv, idesc, (kb | k) != 0 ? 1u : 0u);     // A_hi B_lo
            }
            if (drained) umma_commit_pair(mfull, 3);
#pragma unroll
            for (int k = 0; k < BK / UMMA_K; ++k) {
              const uint64_t adv = static_cast<uint64_t>(k * UMMA_K * 2 / 16);
              umma_bf16_pair(d_cross, dal + adv, dbh + adv, idesc, 1u);                          // A_lo B_hi
              if (EPI == F_GRAM && !F16 && p.four) umma_bf16_pair(d_cross, dal + adv, dbl + adv, idesc, 1u);
            }
            umma_commit_pair(&empty[s], 3);
          }
          if (drained) ++g;
          if (++s == static_cast<uint32_t>(ST)) { s = 0; ph ^= 1; }
        }
        if (ok && elect_one()) umma_commit_pair(cfull, 3);
      }
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: warp (q, h) = TMEM lane quarter q, every second chunk of 32 columns ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
    const int q = warp & 3, h = (warp - 4) >> 2;
    bool ok = true;
    float invL = 0.f, thr = 0.f;
    if (kIsta<EPI>) { invL = p.sc->invL; thr = p.lam * invL; }
    const int row0 = static_cast<int>(rank) * BM + q * 32;           // first of this warp's 32 rows within the tile
    const uint32_t slot = smem_u32(smem + kRegion + (warp - 4) * kSlot);
    // The result leaves by rows: 8 lanes take the 32 columns of a row, 4 rows at a time.  (With a row per lane, as it comes out
    // of TMEM, every access touched 32 lines and the loads of an ISTA step waited for one another: 20 us at the end of each
    // product of 512 x 5,000.)
    const int rg = lane >> 3, cj = lane & 7;
    constexpr bool kAux = EPI == F_SUB || EPI == F_ISTA || EPI == F_ISTAG;
    // Four columns of a row: the factors, what the epilogue does, the result and its pair.
    struct Place { int col; bool in4; float4 fb; };
    auto place = [&](int n0, int c) {
      Place o;
      o.col = n0 + c * kChunk + 4 * cj;
      o.in4 = o.col + 4 <= p.N;
      o.fb = make_float4(1.f, 1.f, 1.f, 1.f);
      if constexpr (F16) {
        if (p.ib) o.fb = *reinterpret_cast<const float4*>(p.ib + o.col);                // (padded to whole chunks)
        if (p.iab) o.fb = scale4(o.fb, *p.iab);
      }
      return o;
    };
    auto put = [&](const Place& o, int row, float4 v, const float4& x, const float4& b) {
      if constexpr (F16) {
        if (p.ia) v = scale4(v, p.ia[row]);
        v = make_float4(v.x * o.fb.x, v.y * o.fb.y, v.z * o.fb.z, v.w * o.fb.w);
      }
      // (N, hence every pitch, is a multiple of 4 for the products over atoms)
      if constexpr (EPI == F_ISTAG) v = make_float4(v.x - b.x, v.y - b.y, v.z - b.z, v.w - b.w);
      if constexpr (EPI == F_ISTA0) {
        if (p.C2 && o.in4) *reinterpret_cast<float4*>(p.C2 + static_cast<int64_t>(row) * p.ldc + o.col) = v;
        v = make_float4(soft_threshold(v.x * invL, thr), soft_threshold(v.y * invL, thr), soft_threshold(v.z * invL, thr),
                        soft_threshold(v.w * invL, thr));
      }
      if constexpr (EPI == F_SUB) v = make_float4(v.x - x.x, v.y - x.y, v.z - x.z, v.w - x.w);
      if constexpr (EPI == F_ISTA || EPI == F_ISTAG)
        v = make_float4(soft_threshold(fmaf(-v.x, invL, x.x), thr), soft_threshold(fmaf(-v.y, invL, x.y), thr),
                        soft_threshold(fmaf(-v.z, invL, x.z), thr), soft_threshold(fmaf(-v.w, invL, x.w), thr));
      if (p.C) {
        float* to = p.C + static_cast<int64_t>(row) * p.ldc + o.col;
        if (o.in4) {                                                // (its pitch is a multiple of 4)
          *reinterpret_cast<float4*>(to) = v;
        } else {
          if (o.col < p.N) to[0] = v.x;
          if (o.col + 1 < p.N) to[1] = v.y;
          if (o.col + 2 < p.N) to[2] = v.z;
        }
      }
      if constexpr (kPairOut<EPI, F16>) {            // the operand of the next product, zero in the padding past N
        if (o.col < p.split_half) {
          if (!o.in4) v = make_float4(o.col < p.N ? v.x : 0.f, o.col + 1 < p.N ? v.y : 0.f, o.col + 2 < p.N ? v.z : 0.f, 0.f);
          uint16_t* to = p.split + static_cast<int64_t>(row) * p.ld_split + o.col;
          if constexpr (F16) {
            const float most = p.most_in[row], so = pow2_scale(most, kTop);
            const float here = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
            if (here > most) atomicMax(reinterpret_cast<int*>(p.most_out + row), __float_as_int(here));
            if (o.col == 0) {
              atomicMax(reinterpret_cast<int*>(p.most_out + row), __float_as_int(most));
              p.io[row] = 1.f / so;
            }
            v = scale4(v, so);
          }
          put_pair4<F16>(to, p.split_half, v);
        }
      }
    };
    // A chunk from shared memory, with loads of what else it reads.
    auto finish = [&](int m0, int n0, int c, uint32_t from) {
      if (n0 + c * kChunk >= p.N) return;
      const Place o = place(n0, c);
      const int row = m0 + row0 + rg, nv = (p.M - row + 3) >> 2;    // nv: of the lane's rows row + 4 e inside the matrix
      float4 x[8], b[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        x[e] = b[e] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e >= nv) continue;
        if constexpr (kAux) {
          const float* ap = p.aux + static_cast<int64_t>(row + 4 * e) * p.ldaux + o.col;
          if (o.in4 && (reinterpret_cast<uintptr_t>(ap) & 15u) == 0) {
            x[e] = *reinterpret_cast<const float4*>(ap);
          } else {
            if (o.col < p.N) x[e].x = ap[0];
            if (o.col + 1 < p.N) x[e].y = ap[1];
            if (o.col + 2 < p.N) x[e].z = ap[2];
            if (o.col + 3 < p.N) x[e].w = ap[3];
          }
        }
        if (EPI == F_ISTAG && o.in4)
          b[e] = *reinterpret_cast<const float4*>(p.C2 + static_cast<int64_t>(row + 4 * e) * p.ldc + o.col);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (e < nv) put(o, row + 4 * e, ld_shared_f4(slot_addr(from, rg + 4 * e, cj)), x[e], b[e]);
    };
    // F_GRAM: the mirror images of the entries whose own tile is not formed; a row per lane makes neighbouring columns there.
    auto mirror = [&](const uint32_t (&acc)[32], int m0, int n0, int c) {
      const int row = m0 + row0 + lane, col0 = n0 + c * kChunk;
      if (row >= p.M) return;
      const int own_end = (row / p.bn + 1) * p.bn;                  // end of the column block that row lies in
      const float f = F16 ? *p.iab : 1.f;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const int n = col0 + j;
        if (n >= p.N || own_end > n / PM * PM) continue;
        const float v = __uint_as_float(acc[j]) * f;
        if constexpr (kPairOut<EPI, F16>) {
          uint32_t hi, lo;
          split2<F16>(v, 0.f, hi, lo);
          uint16_t* mp = p.split + static_cast<int64_t>(n) * p.ld_split + row;
          mp[0] = static_cast<uint16_t>(hi);
          mp[p.split_half] = static_cast<uint16_t>(lo);
        }
        if (p.C) p.C[static_cast<int64_t>(n) * p.ldc + row] = v;
      }
    };

    const int chunks = p.bn / kChunk;
    const uint32_t t_addr = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
    const uint32_t mempty_leader = mapa_u32(smem_u32(mempty), 0), cempty_leader = mapa_u32(smem_u32(cempty), 0);
    uint32_t g = 0;
    for (int sgi = 0; sgi < segs.n && ok; ++sgi) {
      const Segment sg = segs.get(sgi);
      const int nk = sg.k1 - sg.k0;
      int m0, n0;
      tile_coords<EPI>(p, sg.tile, m0, n0);
      float sum[4][32];                              // chunks h, h + 2, h + 4, h + 6
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 32; ++j) sum[i][j] = 0.f;
      // sum += scale * (the accumulator at column `at`), which is then given back
      auto drain = [&](uint32_t at, float scale, uint32_t done) {
        tc_fence_after();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (h + 2 * i >= chunks) break;
          uint32_t acc[32];
          tmem_ld_32x32(t_addr + at + (h + 2 * i) * kChunk, acc);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) sum[i][j] = fmaf(__uint_as_float(acc[j]), scale, sum[i][j]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(done);
      };
      for (int kb = 0; kb < nk && ok; kb += kDrain<EPI, F16>, ++g) {
        ok = __all_sync(0xffffffffu, mbar_wait(mfull, g & 1, abort_flag));
        if (ok) drain(0, 1.f, mempty_leader);
      }
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(cfull, sgi & 1, abort_flag));
      if (!ok) break;
      drain(kMaxN, F16 ? 1.f / kLoScale : 1.f, cempty_leader);
      const int at = static_cast<int>(rank) * kEpi + warp - 4;
      auto chunk_to_slot = [&](int i) {
        uint32_t acc[32];
#pragma unroll
        for (int j = 0; j < 32; ++j)
          acc[j] = __float_as_uint(i == 0 ? sum[0][j] : i == 1 ? sum[1][j] : i == 2 ? sum[2][j] : sum[3][j]);
        slot_put(slot, lane, acc);
      };
      if (sg.k1 < p.kseg) {                          // the rest of the tile is another pair's: leave it the sums
        float* out = p.partial + (static_cast<int64_t>(pair) * 2 * kEpi + at) * 4 * (kSlot / 4);
#pragma unroll 1
        for (int i = 0; h + 2 * i < chunks; ++i) {
          chunk_to_slot(i);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) { bulk_store(out + i * (kSlot / 4), slot, kSlot); tma_commit_group(); tma_wait_group_read<0>(); }
          __syncwarp();
        }
        if (lane == 0) {
          tma_wait_group<0>();
          fence_proxy_async_all();
          __threadfence();
          st_release(p.ready + pair * 2 * kEpi + at, 1u);
        }
        continue;
      }
      if (EPI != F_GRAM && sgi + 1 == segs.n) {
        // The last tile, the one that may take parts from other pairs.  Nothing uses the operand ring any more: its memory takes
        // the sums and, with the slot, what the end of the tile reads -- per chunk the parts, aux, C2 -- by bulk copies, kInputs
        // of them under way per warp.
        // (Loads go through what is left of L1, 28 KB, which held them to 14 bytes per cycle: 30,000 cycles at the end of an
        // ISTA step of 512 x 5,000, 27,000 to add up five parts.)
        const int from = segs.first_part(sg), parts = pair - from;
        const bool copies = kAux && p.copies;
        constexpr int kAfter = EPI == F_ISTAG ? 2 : 1;
        const int per = parts + (copies ? kAfter : 0);
        int mine = 0;
        while (mine < 4 && h + 2 * mine < chunks && n0 + (h + 2 * mine) * kChunk < p.N) ++mine;
        const uint32_t room = smem_u32(smem) + (warp - 4) * (4 + kInputs - 1) * kSlot;
        auto buffer = [&](int k) { return k % kInputs == 0 ? slot : room + (3 + k % kInputs) * kSlot; };
        uint64_t* bar = ifull + (warp - 4) * kInputs;
        for (int j = from; j < pair && ok; ++j) ok = __all_sync(0xffffffffu, lane != 0 || flag_wait(p.ready + j * 2 * kEpi + at, abort_flag));
        if (!ok) break;
        int asked = 0, taken = 0;                    // copies
        auto ask = [&]() {                           // (lane 0) the next one
          if (asked >= mine * per) return;
          const int i = asked / per, w = asked - i * per, buf = asked % kInputs;
          const uint32_t to = buffer(asked);
          const int x0 = n0 + (h + 2 * i) * kChunk;
          mbar_expect_tx(&bar[buf], kSlot);
          if (w < parts) bulk_load(to, p.partial + ((static_cast<int64_t>(from + w) * 2 * kEpi + at) * 4 + i) * (kSlot / 4), kSlot, &bar[buf]);
          else if (w == parts) tma_load_2d_at(to, &tmX, x0, m0 + row0 - p.aux_row0, &bar[buf]);
          else tma_load_2d_at(to, &tmY, x0, m0 + row0, &bar[buf]);
          ++asked;
        };
        auto take = [&](int ahead) {                 // waits for the copy `ahead` places on; where it is
          const int k = taken + ahead;
          ok = ok && __all_sync(0xffffffffu, mbar_wait(&bar[k % kInputs], (k / kInputs) & 1, abort_flag));
          return buffer(k);
        };
        auto give = [&](int n) {                     // their buffers are free
          __syncwarp();
          taken += n;
          if (lane == 0) for (int k = 0; k < n; ++k) ask();
        };
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (i >= mine) break;
          uint32_t acc[32];
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[j] = __float_as_uint(sum[i][j]);
          slot_put(room + i * kSlot, lane, acc);
        }
        __syncwarp();
        if (lane == 0) {
          for (int j = from; j < pair; ++j) p.ready[j * 2 * kEpi + at] = 0;             // for the next launch
          fence_proxy_async_all();
          for (int k = 0; k < kInputs; ++k) ask();
        }
#pragma unroll 1
        for (int i = 0; i < mine && ok; ++i) {
          const uint32_t own = room + i * kSlot;
          const Place o = place(n0, h + 2 * i);
          const int row = m0 + row0 + rg, nv = (p.M - row + 3) >> 2;
          float4 v[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) v[e] = ld_shared_f4(slot_addr(own, rg + 4 * e, cj));
          for (int w = 0; w < parts && ok; ++w) {
            const uint32_t a = take(0);
            if (!ok) break;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const float4 t = ld_shared_f4(slot_addr(a, rg + 4 * e, cj));
              v[e] = make_float4(v[e].x + t.x, v[e].y + t.y, v[e].z + t.z, v[e].w + t.w);
            }
            give(1);
          }
          if (!ok) break;
          const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
          if (!kAux) {
#pragma unroll
            for (int e = 0; e < 8; ++e)
              if (e < nv) put(o, row + 4 * e, v[e], none, none);
          } else if (copies) {
            const uint32_t xa = take(0), ba = kAfter > 1 ? take(1) : 0;
            if (!ok) break;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const float4 x = ld_shared_f4(slot_addr(xa, rg + 4 * e, cj));
              const float4 b = kAfter > 1 ? ld_shared_f4(slot_addr(ba, rg + 4 * e, cj)) : none;
              if (e < nv) put(o, row + 4 * e, v[e], x, b);
            }
            give(kAfter);
          } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) st_shared_f4(slot_addr(own, rg + 4 * e, cj), v[e]);
            __syncwarp();
            finish(m0, n0, h + 2 * i, own);
          }
        }
        break;
      }
#pragma unroll 1
      for (int i = 0; h + 2 * i < chunks; ++i) {
        const int c = h + 2 * i;
        if (EPI == F_GRAM) {
          uint32_t acc[32];
#pragma unroll
          for (int j = 0; j < 32; ++j)
            acc[j] = __float_as_uint(i == 0 ? sum[0][j] : i == 1 ? sum[1][j] : i == 2 ? sum[2][j] : sum[3][j]);
          mirror(acc, m0, n0, c);
        }
        chunk_to_slot(i);
        __syncwarp();
        finish(m0, n0, c, slot);
        __syncwarp();
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
  cluster_arrive();          // no CTA frees its TMEM or exits while another may still signal it or read its shared memory
  cluster_wait();
  if (warp == 1) { tc_fence_after(); tmem_dealloc_pair(tmem_base, kTmemCols); }
}

// ---------------------------------------------------------------------------------------------------------
// Operand packing
// ---------------------------------------------------------------------------------------------------------
// W [n x dim] -> its transpose as an operand FT [dim x 2*Kp] (the coder's W^T); rows n..Kp-1 are written as zeros.  64 x 64
// tiles through shared memory.  inv: the inverse of the scale (fp16 form).
// FR (bf16 form): the rows as an operand [n x 2*dimp] too (fp16 pairs have a scale per row there and one for all here); columns
// dim..dimp-1 are left as they are.  One read of W for both: 124 us for 10,000 x 5,000, 190 in two kernels.
template <bool F16>
__global__ void __launch_bounds__(256) pack_t_kernel(const float* __restrict__ F, int64_t n, int64_t dim, int64_t ld,
                                                     uint16_t* __restrict__ FT, int64_t Kp, const float* __restrict__ inv,
                                                     uint16_t* __restrict__ FR, int64_t dimp, const Stamp stamp) {
  pdl_launch_dependents();
  pdl_wait(F, FT, inv, FR);
  stamp_begin(stamp);
  __shared__ float tile[64][65];
  const int64_t cblocks = (dim + 63) / 64, i0 = blockIdx.x / cblocks * 64, c0 = blockIdx.x % cblocks * 64;
  const int t = threadIdx.x;
  const float s = F16 ? 1.f / *inv : 1.f;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const int idx = t + v * 256;            // 64 rows x 16 quads (dim and ld are multiples of 4)
    const int i = idx / 16, cq = (idx % 16) * 4;
    float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i0 + i < n && c0 + cq < dim) {
      f = *reinterpret_cast<const float4*>(F + (i0 + i) * ld + c0 + cq);
      if (!F16) put_pair4<false>(FR + (i0 + i) * 2 * dimp + c0 + cq, dimp, f);
    }
    tile[i][cq + 0] = f.x * s; tile[i][cq + 1] = f.y * s; tile[i][cq + 2] = f.z * s; tile[i][cq + 3] = f.w * s;
  }
  __syncthreads();
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    const int idx = t + v * 256;            // 64 columns x 8 groups of 8 rows
    const int c = idx / 8, ig = (idx % 8) * 8;
    if (c0 + c >= dim) continue;
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) split2<F16>(tile[ig + 2 * k][c], tile[ig + 2 * k + 1][c], hi[k], lo[k]);
    uint16_t* dst = FT + (c0 + c) * 2 * Kp + i0 + ig;     // Kp is a multiple of 64: 16-byte aligned
    *reinterpret_cast<uint4*>(dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(dst + Kp) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

// bf16 form: rows of F (or of F - Y, which then also go to V in fp32) -> the operand [n x 2*dimp].  TPR threads per row, four
// quads of columns each at a time.  Columns dim..dimp-1 are left as they are (zero since set-up).  For the rows that
// pack_long_kernel does not take (1,000 x 20,000 there: 49 -> 42 us).
template <int TPR, bool SUB>
__global__ void __launch_bounds__(256) pack_rows_kernel(const float* __restrict__ F, const float* __restrict__ Y, int64_t n, int dim,
                                                        int64_t ld, float* __restrict__ V, uint16_t* __restrict__ dst, int64_t dimp,
                                                        const Stamp stamp) {
  pdl_launch_dependents();
  pdl_wait(F, Y, V, dst);
  stamp_begin(stamp);
  const int64_t r = static_cast<int64_t>(blockIdx.x) * (256 / TPR) + threadIdx.x / TPR;
  const int t = threadIdx.x % TPR, quads = dim / 4;
  if (r >= n) return;
  uint16_t* d = dst + r * 2 * dimp;
  if (ld % 4 == 0 && dim % 4 == 0) {
    const float4* src = reinterpret_cast<const float4*>(F + r * ld);
    const float4* sub = reinterpret_cast<const float4*>(Y + r * ld);
    float4* v4 = reinterpret_cast<float4*>(V + r * dim);
    for (int q0 = t; q0 < quads; q0 += 4 * TPR) {
      float4 v[4], y[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (q0 + k * TPR < quads) v[k] = src[q0 + k * TPR];
        if (SUB && q0 + k * TPR < quads) y[k] = sub[q0 + k * TPR];
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int q = q0 + k * TPR;
        if (q >= quads) continue;
        if (SUB) {
          v[k] = make_float4(v[k].x - y[k].x, v[k].y - y[k].y, v[k].z - y[k].z, v[k].w - y[k].w);
          v4[q] = v[k];
        }
        put_pair4<false>(d + 4 * q, dimp, v[k]);
      }
    }
  } else {                                             // samples with an odd number of features: value by value
    const float* src = F + r * ld;
    for (int c = t; c < dim; c += TPR) {
      uint32_t hi, lo;
      split2<false>(src[c], 0.f, hi, lo);
      d[c] = static_cast<uint16_t>(hi);
      d[dimp + c] = static_cast<uint16_t>(lo);
    }
  }
}

// fp16 form: rows of F (or of F - Y) with a scale per row, its inverse to inv.  A row takes TPR threads, which hold up to 64
// values each in registers between the search for the largest entry and the conversion (the rest is read again, from L2):
// one pass over memory.
struct Pack16 {
  const float* F;
  const float* Y;              // subtracted, same pitch (may be null)
  int64_t n, dim, ld;
  float* V;                    // the fp32 values, pitch dim (may be null)
  uint16_t* dst;
  int64_t dimp;
  float* inv;
  float* inv2;                 // the same again (may be null)
  // sparse coding: what the sample's residuals and codes begin with as their largest values, ||x|| and ||x|| / sqrt(L), in both of
  // the buffers that the iterations take in turn (of `samples` each), and the inverse scale of codes that no iteration makes
  float* res;
  float* code;
  float* inv_code;
  int64_t samples;
  const Scalars* sc;
  Stamp stamp;
};
__device__ __forceinline__ void row_scales(const Pack16& p, int64_t r, float s, float ss) {
  p.inv[r] = 1.f / s;
  if (p.inv2) p.inv2[r] = 1.f / s;
  if (p.res) {
    const float norm = sqrtf(ss), code = norm * sqrtf(p.sc->invL);
    p.res[r] = p.res[p.samples + r] = norm;
    p.code[r] = p.code[p.samples + r] = code;
    p.inv_code[r] = 1.f / pow2_scale(code, kTop);
  }
}
template <int TPR>
__global__ void __launch_bounds__(256) pack16_kernel(const __grid_constant__ Pack16 p) {
  pdl_launch_dependents();
  pdl_wait();
  stamp_begin(p.stamp);
  constexpr int kHeld = 16;
  __shared__ float sh[16];
  const int t = threadIdx.x % TPR;
  const int64_t r = static_cast<int64_t>(blockIdx.x) * (256 / TPR) + threadIdx.x / TPR;
  if (r >= p.n) return;                                // (whole warps; whole blocks when TPR is 256)
  const float* src = p.F + r * p.ld;
  const float* sub = p.Y ? p.Y + r * p.ld : nullptr;
  const bool vec = p.ld % 4 == 0 && p.dim % 4 == 0;
  const int quads = static_cast<int>(p.dim / 4), dim = static_cast<int>(p.dim);
  auto get = [&](int q) {
    float4 v = reinterpret_cast<const float4*>(src)[q];
    if (sub) {
      const float4 y = reinterpret_cast<const float4*>(sub)[q];
      v.x -= y.x; v.y -= y.y; v.z -= y.z; v.w -= y.w;
    }
    return v;
  };
  float m = 0.f, ss = 0.f;
  auto look = [&](const float4& v) {
    m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
    if (p.res) ss = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, ss))));
  };
  float4 held[kHeld];
  if (vec) {
#pragma unroll
    for (int k = 0; k < kHeld; ++k)
      if (t + k * TPR < quads) held[k] = get(t + k * TPR);
#pragma unroll
    for (int k = 0; k < kHeld; ++k)
      if (t + k * TPR < quads) look(held[k]);
    for (int q = t + kHeld * TPR; q < quads; q += TPR) look(get(q));
  } else {
    for (int c = t; c < dim; c += TPR) look(make_float4(src[c], 0.f, 0.f, 0.f));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
  }
  if (TPR > 32) {
    if ((t & 31) == 0) { sh[t >> 5] = m; sh[8 + (t >> 5)] = ss; }
    __syncthreads();
    m = sh[0]; ss = sh[8];
#pragma unroll
    for (int w = 1; w < 8; ++w) { m = fmaxf(m, sh[w]); ss += sh[8 + w]; }
  }
  const float s = pow2_scale(m, 13);
  if (t == 0) row_scales(p, r, s, ss);
  uint16_t* d = p.dst + r * 2 * p.dimp;
  if (vec) {
    float4* v4 = p.V ? reinterpret_cast<float4*>(p.V + r * p.dim) : nullptr;
#pragma unroll
    for (int k = 0; k < kHeld; ++k) {
      const int q = t + k * TPR;
      if (q >= quads) continue;
      if (v4) v4[q] = held[k];
      put_pair4<true>(d + 4 * q, p.dimp, scale4(held[k], s));
    }
    for (int q = t + kHeld * TPR; q < quads; q += TPR) {
      const float4 v = get(q);
      if (v4) v4[q] = v;
      put_pair4<true>(d + 4 * q, p.dimp, scale4(v, s));
    }
  } else {
    for (int c = t; c < dim; c += TPR) {
      uint32_t hi, lo;
      split2<true>(src[c] * s, 0.f, hi, lo);
      d[c] = static_cast<uint16_t>(hi);
      d[p.dimp + c] = static_cast<uint16_t>(lo);
    }
  }
}

// The same (and the bf16 form, which needs no scale) for long rows, which come through shared memory: a block has the next rows under way by bulk copies while it looks for
// the largest entry of one and converts it.  (Held in registers, a row's loads and stores took turns: 10,000 x 20,000 in 603 us,
// 290 now.  With Y both rows come; if only one such pair fits, its stores at least drain beside the next loads.)
constexpr int kPackRoom = 208 << 10, kPackThreads = 512, kPackBufs = 4;
template <bool F16>
__global__ void __launch_bounds__(kPackThreads, 1) pack_long_kernel(const __grid_constant__ Pack16 p, int bufs, uint32_t* status) {
  extern __shared__ __align__(128) uint8_t rows_smem[];
  __shared__ __align__(8) uint64_t full[kPackBufs];
  __shared__ float sh[2 * kPackThreads / 32];
  __shared__ uint32_t abort_word;
  pdl_launch_dependents();
  const int t = threadIdx.x, quads = static_cast<int>(p.dim / 4);
  const uint32_t bytes = static_cast<uint32_t>(p.dim) * 4, buf_bytes = (p.Y ? 2 : 1) * bytes;
  if (t == 0) {
    for (int i = 0; i < kPackBufs; ++i) mbar_init(&full[i], 1);
    abort_word = 0;
    fence_barrier_init();
  }
  __syncthreads();
  pdl_wait();
  stamp_begin(p.stamp);
  auto ask = [&](int64_t r, int b) {
    mbar_expect_tx(&full[b], buf_bytes);
    bulk_load(smem_u32(rows_smem) + b * buf_bytes, p.F + r * p.ld, bytes, &full[b]);
    if (p.Y) bulk_load(smem_u32(rows_smem) + b * buf_bytes + bytes, p.Y + r * p.ld, bytes, &full[b]);
  };
  const int64_t step = gridDim.x;
  if (t == 0)
    for (int b = 0; b < bufs && blockIdx.x + b * step < p.n; ++b) ask(blockIdx.x + b * step, b);
  int b = 0;
  uint32_t ph = 0;
  for (int64_t r = blockIdx.x; r < p.n; r += step) {
    if (!__syncthreads_and(mbar_wait(&full[b], ph, &abort_word))) {
      if (t == 0) atomicOr(status, SFB_STATUS_TIMEOUT);
      for (int i = 0; i < 64; ++i) __nanosleep(1000);  // for copies in flight
      return;
    }
    float4* row = reinterpret_cast<float4*>(rows_smem + b * buf_bytes);
    const float4* sub = row + quads;
    float s = 1.f;
    if constexpr (F16) {
      float m = 0.f, ss = 0.f;
      for (int q = t; q < quads; q += kPackThreads) {
        float4 v = row[q];
        if (p.Y) {
          const float4 y = sub[q];
          v = make_float4(v.x - y.x, v.y - y.y, v.z - y.z, v.w - y.w);
          row[q] = v;                                    // (this thread reads it again)
        }
        m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
        if (p.res) ss = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, ss))));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        ss += __shfl_xor_sync(0xffffffffu, ss, o);
      }
      constexpr int kWarps = kPackThreads / 32;
      if ((t & 31) == 0) { sh[t >> 5] = m; sh[kWarps + (t >> 5)] = ss; }
      __syncthreads();
      m = sh[0]; ss = sh[kWarps];
#pragma unroll
      for (int w = 1; w < kWarps; ++w) { m = fmaxf(m, sh[w]); ss += sh[kWarps + w]; }
      s = pow2_scale(m, 13);
      if (t == 0) row_scales(p, r, s, ss);
    }
    uint16_t* d = p.dst + r * 2 * p.dimp;
    float4* v4 = p.V ? reinterpret_cast<float4*>(p.V + r * p.dim) : nullptr;
    for (int q = t; q < quads; q += kPackThreads) {
      float4 v = row[q];
      if (!F16 && p.Y) {
        const float4 y = sub[q];
        v = make_float4(v.x - y.x, v.y - y.y, v.z - y.z, v.w - y.w);
      }
      if (v4) v4[q] = v;
      put_pair4<F16>(d + 4 * q, p.dimp, F16 ? scale4(v, s) : v);
    }
    if (F16 && p.Y) fence_proxy_async_smem();                 // (written to, and to be overwritten by a copy)
    __syncthreads();                                   // the row (and sh) has been read
    if (t == 0 && r + bufs * step < p.n) ask(r + bufs * step, b);
    if (++b == bufs) { b = 0; ph ^= 1; }
  }
}

// fp16 form, sparse coding: one scale for W^T (the smallest of W's rows).  iw: inverse scales of W's rows.
__global__ void __launch_bounds__(1024) sc_scales_kernel(const float* __restrict__ iw, int rows, Scalars* sc) {
  pdl_launch_dependents();
  pdl_wait(iw);
  __shared__ float sh[32];
  float m = 0.f;
  for (int r = threadIdx.x; r < rows; r += 1024) m = fmaxf(m, iw[r]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 32; ++w) m = fmaxf(m, sh[w]);
    sc->iWT = m;
    sc->iWT2 = m * m;
  }
}

// q[i] = inv[i] * max_j |U[i][j]|, one block per pair.
__global__ void __launch_bounds__(256) row_most_kernel(const float* __restrict__ U, int64_t ldu, int64_t rows,
                                                       const float* __restrict__ inv, float* __restrict__ q) {
  pdl_launch_dependents();
  pdl_wait(U, inv, q);
  __shared__ float sh[8];
  const float* u = U + static_cast<int64_t>(blockIdx.x) * ldu;
  float m = 0.f;
  for (int64_t j = threadIdx.x; j < rows; j += 256) m = fmaxf(m, fabsf(u[j]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) m = fmaxf(m, sh[w]);
    q[blockIdx.x] = m * inv[blockIdx.x];
  }
}

// fp16 form: the gathered factors U [K x ldu] as the operand of the update.  The update contracts over the pairs, so the
// scale of u_i is the inverse of v_i's times one factor for all, which brings the largest q[i] = max_j |u_ij| * inv_v[i] to
// 2^13; its inverse to sc->iU.
__global__ void __launch_bounds__(256) pack_u_kernel(const float* __restrict__ U, int64_t ldu, int64_t K, int64_t rows,
                                                     const float* __restrict__ q, const float* __restrict__ inv_v,
                                                     uint16_t* __restrict__ dst, int64_t rowsp, Scalars* sc, const Stamp stamp) {
  pdl_launch_dependents();
  pdl_wait(U, q, inv_v, dst);
  stamp_begin(stamp);
  __shared__ float sh[8];
  float m = 0.f;
  for (int64_t i = threadIdx.x; i < K; i += 256) m = fmaxf(m, q[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  for (int w = 0; w < 8; ++w) m = fmaxf(m, sh[w]);
  const float a = pow2_scale(m, 13);
  if (blockIdx.x == 0 && threadIdx.x == 0) sc->iU = 1.f / a;
  const int64_t quads = (rows + 3) / 4, total = K * quads, stride = static_cast<int64_t>(gridDim.x) * 256;
  for (int64_t t = blockIdx.x * 256ll + threadIdx.x; t < total; t += stride) {
    const int64_t i = t / quads, c = (t - i * quads) * 4;
    // (the pitch is a multiple of 4; the operand's padding stays zero: the coder contracts over the same buffer in the next step,
    // and nothing ever writes the padding of U)
    float4 u = *reinterpret_cast<const float4*>(U + i * ldu + c);
    if (c + 1 >= rows) u.y = 0.f;
    if (c + 2 >= rows) u.z = 0.f;
    if (c + 3 >= rows) u.w = 0.f;
    put_pair4<true>(dst + i * 2 * rowsp + c, rowsp, scale4(u, fminf(a * inv_v[i], 1e36f)));
  }
}

// ---------------------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------------------
#define CKC(call)                                       \
  do {                                                  \
    cudaError_t e__ = (call);                           \
    if (e__ != cudaSuccess) {                           \
      ctx->last_cuda = static_cast<int>(e__);           \
      return SFB_ERR_CUDA;                              \
    }                                                   \
  } while (0)

// Tile width of a product, whether its contraction is cut, and its SM cycles.  A k-block takes the longer of its MMAs (6 cycles per
// column by their rate, 7.2 as measured at 256 columns: 1,838) and of its bytes from L2 at 38 a cycle and SM (192 columns: 1,485;
// 160: 1,395; 64: 1,100).  12,000 cycles from the start to the first MMA and from the last one to the results; 4,000 and, a part, 1,500
// and 12 a column to leave and to take over the parts of a tile, whose adding up waits for one copy after another: a product of fewer
// tiles than pairs is cut into as many parts a tile as that pays for, and not into parts of less than four k-blocks.  (Of 900 drawn
// calls whose plan matters, against all pairs taking part, factors of metric learning, regression in fp32 and sparse coding take 0.74, 0.82
// and 0.82 times as long, in fp32 0.92 times; with 4,500 cycles a part whatever the width 0.76, 0.82, 0.83 and 0.99, 28 of 609 more than 3 %
// longer than with all pairs, and 214 of 504 in fp32 sparse coding: 1,041 x 900 with 54 samples 413 -> 572 us.  Cutting only the last of
// several rounds took fewer cycles at a lower clock: 908 -> 1013 us.)
// flat: cycles with all pairs taking part, at 8,000 for the parts (see split_form_cost).
struct ProductPlan { int bn; int64_t tiles, pairs; bool cut; double cost, flat; };
// fine: drained at every k-block, 21 cycles a column that the MMAs do not hide (7 in W^T W, sym, whose width alone they decide).
ProductPlan plan_width(int64_t M, int64_t N, int64_t Kc, bool sym, bool fine, int bn, int64_t max_pairs) {
  ProductPlan p{};
  p.bn = bn;
  const int tm = static_cast<int>((M + PM - 1) / PM), tn = static_cast<int>((N + bn - 1) / bn);
  p.tiles = sym ? sym_tiles(tm, tn, bn) : static_cast<int64_t>(tm) * tn;
  const double per_kb = std::max(7.2 * bn, (2.0 * kBytesA + bn * BK * 2.0) / 38.0) + (fine ? (sym ? 7.0 : 21.0) * bn : 0.0);
  const int64_t kseg = (Kc + BK - 1) / BK, rounds = (p.tiles + max_pairs - 1) / max_pairs;
  p.pairs = std::min(p.tiles, max_pairs);
  double kb = static_cast<double>(rounds * kseg);
  const double rate = fine ? std::max(7.2 * bn, (2.0 * kBytesA + bn * BK * 2.0) / 38.0) + 7.0 * bn : per_kb;
  p.flat = kb * rate;
  if (!sym && p.tiles < max_pairs) {
    const int64_t most = std::max<int64_t>(1, std::min(max_pairs, p.tiles * kseg / 4));
    const double all = static_cast<double>((p.tiles * kseg + most - 1) / most) * rate + 8000.0;
    p.flat = std::min(p.flat, all);
    double least = kb * per_kb;
    for (int64_t parts = 2; (parts - 1) * p.tiles < most; ++parts) {          // of a tile
      const int64_t pairs = std::min(most, parts * p.tiles);
      const double shared = static_cast<double>((p.tiles * kseg + pairs - 1) / pairs), extra = 4000.0 + (1500.0 + 12.0 * bn) * static_cast<double>(parts);
      if (shared * per_kb + extra < least) {
        least = shared * per_kb + extra;
        p.cut = true;
        p.pairs = pairs;
      }
    }
    kb = least / per_kb;
  }
  const double rest = 12000.0 + static_cast<double>(p.tiles / max_pairs) * 1500.0;
  p.cost = kb * per_kb + rest;
  p.flat += rest;
  return p;
}
ProductPlan plan_product(int64_t M, int64_t N, int64_t Kc, bool sym, bool fine, int64_t max_pairs) {
  if (N <= 64) return plan_width(M, N, Kc, sym, fine, static_cast<int>(round_up(N, 32)), max_pairs);
  ProductPlan best{};
  for (int bn = kMaxN; bn >= 64; bn -= 32) {
    const ProductPlan p = plan_width(M, N, Kc, sym, fine, bn, max_pairs);
    if (bn == kMaxN || p.cost < best.cost) best = p;
  }
  return best;
}

// D[off..off+n) = A * B^T  with A = [*, 2*Cp] and B = [N x 2*Cp] (hi | lo) operands over a contraction of Cp.
template <int EPI, bool F16>
int split_product(sfb_ctx* ctx, int64_t off, int64_t n, const uint16_t* A, const uint16_t* B, int64_t N, int64_t Cp,
                  SplitParams p) {
  TcState* st = static_cast<TcState*>(ctx->tc);
  const ProductPlan plan = plan_product(n, N, Cp, EPI == F_GRAM, kDrain<EPI, F16> == 1, std::min<int64_t>(st->max_pairs, std::min(sm_count(), kModelSms) / 2));
  p.bn = plan.bn;
  p.cut = plan.cut;
  p.partial = ctx->at<float>(ctx->lay.partial);
  p.ready = ctx->at<uint32_t>(ctx->lay.ready);
  p.stages = ring_stages(p.bn);
  p.a_rows = static_cast<int32_t>(std::min<int64_t>(BM, round_up(n, 8)));
  CUtensorMap ma, mb;
  if (!make_map(st, &ma, CU_TENSOR_MAP_DATA_TYPE_UINT16, const_cast<uint16_t*>(A), 2 * Cp, off + n, 2 * Cp * 2, BK, p.a_rows) ||
      !make_map(st, &mb, CU_TENSOR_MAP_DATA_TYPE_UINT16, const_cast<uint16_t*>(B), 2 * Cp, N, 2 * Cp * 2, BK, p.bn / 2))
    return SFB_ERR_CUDA;
  // aux ends with the last sample of this call; C2 covers all of them
  CUtensorMap mx = ma, my = ma;
  p.copies = p.aux && ((reinterpret_cast<uintptr_t>(p.aux + p.aux_row0 * p.ldaux) | static_cast<uintptr_t>(p.ldaux * 4)) & 15u) == 0;
  if (p.copies && !make_map(st, &mx, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, const_cast<float*>(p.aux + p.aux_row0 * p.ldaux), N,
                            off + n - p.aux_row0, p.ldaux * 4, kChunk, 32))
    return SFB_ERR_CUDA;
  if (EPI == F_ISTAG && !make_map(st, &my, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, p.C2, N, off + n, p.ldc * 4, kChunk, 32)) return SFB_ERR_CUDA;
  p.M = static_cast<int32_t>(off + n); p.N = static_cast<int32_t>(N);
  p.m_off = static_cast<int32_t>(off);
  p.tilesM = static_cast<int32_t>((n + PM - 1) / PM);
  p.tilesN = static_cast<int32_t>((N + p.bn - 1) / p.bn);
  p.kseg = static_cast<int32_t>(Cp / BK);
  p.a_lo = p.b_lo = static_cast<int32_t>(Cp);
  p.status = ctx->at<uint32_t>(ctx->lay.status);
  if (plan.tiles <= 0) return SFB_OK;
  CKC((allow_smem<split_product_kernel<EPI, F16>>(kSmem)));
  CKC(launch_kernel_if(plan.tiles <= st->max_pairs, split_product_kernel<EPI, F16>, dim3(static_cast<unsigned>(2 * plan.pairs)),
                       dim3(kThreads), kSmem, ctx->stream, 2, ma, mb, mx, my, p));
  ctx->stats.flops += (EPI == F_GRAM ? 3.0 : 6.0) * n * N * Cp;
  return SFB_OK;
}

// Long rows with 16-byte pieces; false: the caller has to take another kernel.
template <bool F16>
bool pack_long(sfb_ctx* ctx, const Pack16& p, cudaError_t& e) {
  const int64_t buf = p.dim * (p.Y ? 8 : 4);
  const int bufs = static_cast<int>(std::min<int64_t>(kPackBufs, kPackRoom / buf));
  if (p.dim <= 2048 || bufs < (p.Y ? 1 : 2) || p.dim % 4 != 0 || p.ld % 4 != 0) return false;
  if ((e = allow_smem<pack_long_kernel<F16>>(kPackRoom)) == cudaSuccess)
    e = launch_kernel(pack_long_kernel<F16>, dim3(static_cast<unsigned>(std::min<int64_t>(p.n, sm_count()))), dim3(kPackThreads),
                      static_cast<int>(bufs * buf), ctx->stream, 1, p, bufs, ctx->at<uint32_t>(ctx->lay.status));
  return true;
}
cudaError_t pack16(sfb_ctx* ctx, const Pack16& p) {
  cudaStream_t s = ctx->stream;
  cudaError_t e = cudaSuccess;
  if (p.n <= 0) return cudaSuccess;
  if (p.dim <= 2048) return launch_kernel(pack16_kernel<32>, dim3(static_cast<unsigned>((p.n + 7) / 8)), dim3(256), 0, s, 1, p);
  if (pack_long<true>(ctx, p, e)) return e;
  return launch_kernel(pack16_kernel<256>, dim3(static_cast<unsigned>(p.n)), dim3(256), 0, s, 1, p);
}

// bf16 form; Y: subtracted, the difference also to V.
cudaError_t pack_rows(sfb_ctx* ctx, const float* F, const float* Y, int64_t n, int64_t dim, int64_t ld, float* V, uint16_t* dst,
                      int64_t dimp, const Stamp& stamp) {
  cudaStream_t s = ctx->stream;
  cudaError_t e = cudaSuccess;
  if (n <= 0) return cudaSuccess;
  Pack16 p{};
  p.F = F; p.Y = Y; p.n = n; p.dim = dim; p.ld = ld; p.V = V; p.dst = dst; p.dimp = dimp; p.stamp = stamp;
  if (pack_long<false>(ctx, p, e)) return e;
  auto go = [&](auto kernel, int tpr) {
    return launch_kernel(kernel, dim3(static_cast<unsigned>((n + 256 / tpr - 1) / (256 / tpr))), dim3(256), 0, s, 1, F, Y, n,
                         static_cast<int>(dim), ld, V, dst, dimp, stamp);
  };
  if (dim <= 512) return Y ? go(pack_rows_kernel<32, true>, 32) : go(pack_rows_kernel<32, false>, 32);
  return Y ? go(pack_rows_kernel<256, true>, 256) : go(pack_rows_kernel<256, false>, 256);
}

// Features up to which the coder on W^T W forms W^T x by fp32 FMAs and W^T W with its fourth term in the bf16 form.  Every
// iterate carries their error, and for short contractions the rounding of the operands to pairs is most of it.  Error of the
// codes with / without: 700 x 400: 3.7e-6 / 9.1e-6; 1,501 x 1,400: 5.1e-6 / 9.9e-6.
constexpr int64_t kPreciseRows = 2048;

// Sparse coding: ISTA from a = 0, then u = W a - x, v = a.  The first iterate is soft(W^T x / L).
template <bool F16>
int factors_sc(sfb_ctx* ctx, int64_t off, int64_t n, const float* X) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t rows = c.rows, cols = c.cols;
  cudaStream_t s = ctx->stream;
  const int T = c.sc_ista_iters;
  const bool gram = L.Gs != 0;
  float* V = ctx->at<float>(L.V);
  uint16_t* Ws = ctx->at<uint16_t>(L.Ws);
  uint16_t* WTs = ctx->at<uint16_t>(L.WTs);
  uint16_t* Rs = ctx->at<uint16_t>(L.Rs);
  Scalars* sc = ctx->at<Scalars>(L.scalars);
  // the iterates as operands: with the Gram matrix a product reads one and writes the next, so two buffers in turn
  uint16_t* as[2] = {ctx->at<uint16_t>(L.As), ctx->at<uint16_t>(gram ? L.As2 : L.As)};
  const int64_t K = ctx->K;
  const float* iX = F16 ? ctx->at<float>(L.iA) : nullptr;
  float* iR = F16 ? ctx->at<float>(L.iR) : nullptr;
  float* iC = F16 ? ctx->at<float>(L.iC) : nullptr;                  // [2][K]: of odd and even iterations
  float* mR = F16 ? ctx->at<float>(L.mR) : nullptr;                  // [2][K], as mC
  float* mC = F16 ? ctx->at<float>(L.mC) : nullptr;
  auto ista = [&](int t, const float* ia, const float* iab) {
    SplitParams q{};
    q.C = V; q.ldc = cols;
    q.aux = V; q.ldaux = cols;
    q.C2 = gram ? ctx->at<float>(L.Bx) : nullptr;
    q.sc = sc; q.lam = c.sc_lambda;
    q.split = as[t & 1]; q.ld_split = 2 * L.colsp; q.split_half = static_cast<int32_t>(L.colsp);
    if (F16) { q.ia = ia; q.iab = iab; q.most_in = mC + ((t + 1) & 1) * K; q.most_out = mC + (t & 1) * K; q.io = iC + (t & 1) * K; }
    return q;
  };
  auto residual = [&](int t) {                                                          // r = W a_t - x
    uint16_t* a = as[gram ? t & 1 : 0];
    SplitParams q{};
    q.C = ctx->at<float>(L.U); q.ldc = L.ldu;
    q.aux = X - off * rows; q.ldaux = rows; q.aux_row0 = static_cast<int32_t>(off);          // X holds this worker's samples: index it by the global row
    q.split = Rs; q.ld_split = 2 * L.rowsp; q.split_half = static_cast<int32_t>(L.rowsp);
    if (F16) {
      q.ia = iC + (t & 1) * K; q.ib = ctx->at<float>(L.iW);
      q.most_in = mR + ((t + 1) & 1) * K; q.most_out = mR + (t & 1) * K; q.io = iR;
    }
    return split_product<F_SUB, F16>(ctx, off, n, a, Ws, rows, L.colsp, q);
  };
  int rc = SFB_OK;
  if (F16) {
    Pack16 p{};
    p.F = X; p.n = n; p.dim = p.ld = rows; p.dst = Rs + off * 2 * L.rowsp; p.dimp = L.rowsp;
    p.inv = ctx->at<float>(L.iA) + off;
    p.res = mR + off; p.code = mC + off; p.inv_code = iC + off; p.samples = K;
    p.sc = sc;
    CKC(pack16(ctx, p));
  }
  if (T == 0) {
    CKC(cudaMemsetAsync(V + off * cols, 0, static_cast<size_t>(n) * cols * 4, s));
    CKC(cudaMemsetAsync(as[0] + off * 2 * L.colsp, 0, static_cast<size_t>(n) * 2 * L.colsp * 2, s));
  } else if (!F16 && gram && rows <= kPreciseRows) {                                    // W^T x, a_1
    EpiArgs e{};
    e.C = V + off * cols; e.ldc = cols; e.C2 = ctx->at<float>(L.Bx) + off * cols; e.ldc2 = cols;
    e.sc = sc; e.lam = c.sc_lambda;
    CKC(sgemm(s, true, false, EPI_ISTA0, n, cols, rows, X, rows, ctx->W, cols, e, ctx->K));
    ctx->stats.flops += 2.0 * n * rows * cols;
    CKC(pack_rows(ctx, V + off * cols, nullptr, n, cols, cols, nullptr, as[1] + off * 2 * L.colsp, L.colsp, Stamp{}));
  } else {
    if (!F16)
      CKC(pack_rows(ctx, X, nullptr, n, rows, rows, nullptr, Rs + off * 2 * L.rowsp, L.rowsp, Stamp{}));
    if ((rc = split_product<F_ISTA0, F16>(ctx, off, n, Rs, WTs, cols, L.rowsp, ista(1, iX, &sc->iWT))) != SFB_OK) return rc;
  }
  for (int t = 2; t <= T; ++t) {
    if (gram) {
      if constexpr (!F16) rc = split_product<F_ISTAG, F16>(ctx, off, n, as[(t - 1) & 1], ctx->at<uint16_t>(L.Gs), cols, L.colsp, ista(t, nullptr, nullptr));
    } else {
      if ((rc = residual(t - 1)) != SFB_OK) return rc;
      rc = split_product<F_ISTA, F16>(ctx, off, n, Rs, WTs, cols, L.rowsp, ista(t, iR, &sc->iWT));  // a <- soft(a - W^T r / L)
    }
    if (rc) return rc;
  }
  return residual(T);                                                                   // u = W a - x
}

template <bool F16>
int begin_operands(sfb_ctx* ctx) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t rows = c.rows, cols = c.cols;
  cudaStream_t s = ctx->stream;
  uint16_t* Ws = ctx->at<uint16_t>(L.Ws);
  Scalars* sc = ctx->at<Scalars>(L.scalars);
  if (F16) {
    Pack16 p{};
    p.F = ctx->W; p.n = rows; p.dim = p.ld = cols; p.dst = Ws; p.dimp = L.colsp; p.inv = ctx->at<float>(L.iW);
    p.stamp = take_stamp(ctx);
    CKC(pack16(ctx, p));
  } else if (c.model != SFB_SC) {
    CKC(pack_rows(ctx, ctx->W, nullptr, rows, cols, cols, nullptr, Ws, L.colsp, take_stamp(ctx)));
  }
  if (c.model != SFB_SC) return SFB_OK;
  uint16_t* WTs = ctx->at<uint16_t>(L.WTs);
  if (F16) CKC(launch_kernel(sc_scales_kernel, dim3(1), dim3(1024), 0, s, 1, ctx->at<float>(L.iW), static_cast<int>(rows), sc));
  const int64_t blocks = ((cols + 63) / 64) * (L.rowsp / 64);
  if (blocks > 0x7fffffffLL) return SFB_ERR_SHAPE;
  CKC(launch_kernel(pack_t_kernel<F16>, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, s, 1, ctx->W, rows, cols, cols, WTs, L.rowsp, &sc->iWT,
                    Ws, L.colsp, F16 ? Stamp{} : take_stamp(ctx)));
  if (!(F16 ? L.G : L.Gs)) return SFB_OK;
  SplitParams p{};
  p.four = rows <= kPreciseRows;
  p.C = c.sc_lipschitz > 0.f ? nullptr : ctx->at<float>(L.G);
  p.ldc = cols;
  if (F16) {
    p.iab = &sc->iWT2;
  } else {
    p.split = ctx->at<uint16_t>(L.Gs); p.ld_split = 2 * L.colsp; p.split_half = static_cast<int32_t>(L.colsp);
  }
  return split_product<F_GRAM, F16>(ctx, 0, cols, WTs, WTs, cols, L.rowsp, p);
}

}  // namespace

double split_product_cost(int64_t M, int64_t N, int64_t Kc, bool sym, bool fine) {
  return plan_product(M, N, Kc, sym, fine, kModelSms / 2).cost;
}
double split_form_cost(int64_t M, int64_t N, int64_t Kc, bool sym, bool fine) {
  if (N <= 64) return plan_width(M, N, Kc, sym, fine, static_cast<int>(round_up(N, 32)), kModelSms / 2).flat;
  double best = 0.0;
  for (int bn = kMaxN; bn >= 64; bn -= 32) {
    const double c = plan_width(M, N, Kc, sym, fine, bn, kModelSms / 2).flat;
    if (bn == kMaxN || c < best) best = c;
  }
  return best;
}

int split_product_parts(int64_t M, int64_t N, int64_t Kc, bool fine) {
  const ProductPlan p = plan_product(M, N, Kc, false, fine, kModelSms / 2);
  return p.cut ? std::max(2, static_cast<int>((p.pairs + p.tiles - 1) / p.tiles)) : 1;
}

void split_extend_layout(const sfb_config& c, Layout& L, size_t& off) {
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + kAlign - 1) / kAlign * kAlign; return o; };
  const size_t K = static_cast<size_t>(c.workers) * c.batch;
  const bool f16 = c.precision != SFB_PREC_BF16;
  L.colsp = round_up(c.cols, 64);
  L.rowsp = round_up(c.rows, 64);
  L.ldu = round_up(c.rows, 4);                                        // 16-byte row pitch
  L.V = take(K * static_cast<size_t>(c.cols) * 4);                    // the factors in fp32
  L.U = take(K * static_cast<size_t>(L.ldu) * 4);
  L.Rs = take(K * 2 * static_cast<size_t>(L.rowsp) * 2);              // u (SC: first x, then the residuals)
  L.Ws = take(static_cast<size_t>(c.rows) * 2 * L.colsp * 2);         // W, rows x (hi | lo)
  L.As = take(K * 2 * static_cast<size_t>(L.colsp) * 2);              // v (MLR, DML) or the codes a (SC)
  L.partial = take(static_cast<size_t>(kModelSms / 2) * 2 * kEpi * 4 * kSlot);      // parts of tiles (see split_product_kernel)
  L.ready = take(static_cast<size_t>(kModelSms / 2) * 2 * kEpi * 4);
  if (f16) {
    L.iW = take((static_cast<size_t>(c.rows) + 32) * 4);              // inverse scales: rows of W, pairs
    L.iA = take(K * 4);
    L.q = take(K * 4);
  }
  if (c.model != SFB_SC) return;
  if (f16) {
    L.iR = take(K * 4);
    L.iC = take(2 * K * 4);
    L.mR = take(2 * K * 4);
    L.mC = take(2 * K * 4);
  }
  L.WTs = take(static_cast<size_t>(c.cols) * 2 * L.rowsp * 2);        // W^T, atoms x (hi | lo)
  if (f16 && sc_estimate_on_gram(c, split_product_cost(c.cols, c.cols, c.rows, true, true))) L.G = take(static_cast<size_t>(c.cols) * c.cols * 4);
  if (sc_use_gram(c)) {
    L.Gs = take(static_cast<size_t>(c.cols) * 2 * L.colsp * 2);       // W^T W, atoms x (hi | lo)
    L.G = take(c.sc_lipschitz > 0.f ? 0 : static_cast<size_t>(c.cols) * c.cols * 4);   // in fp32 for the power iteration
    L.Bx = take(K * static_cast<size_t>(c.cols) * 4);                 // W^T x
    L.As2 = take(K * 2 * static_cast<size_t>(L.colsp) * 2);           // the codes of every other iteration
  }
}

// A launch that ran into a wait limit may have left flags set.
cudaError_t split_reset(sfb_ctx* ctx) {
  return cudaMemsetAsync(ctx->at<char>(ctx->lay.ready), 0, static_cast<size_t>(kModelSms / 2) * 2 * kEpi * 4, ctx->stream);
}

// Pad columns of the operands are never written by the kernels: cleared once.
int split_init(sfb_ctx* ctx) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const size_t K = static_cast<size_t>(ctx->K);
  CKC(split_reset(ctx));
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

int split_begin_step(sfb_ctx* ctx) { return ctx->h16 ? begin_operands<true>(ctx) : begin_operands<false>(ctx); }

int split_logits(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const float* Y) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t cols = c.cols;
  float* V = ctx->at<float>(L.V) + off * cols;
  uint16_t* As = ctx->at<uint16_t>(L.As);
  SplitParams p{};
  p.C = ctx->at<float>(L.U); p.ldc = L.ldu;
  if (!ctx->h16) {
    CKC(pack_rows(ctx, X, Y, n, cols, cols, V, As + off * 2 * L.colsp, L.colsp, Stamp{}));
    return split_product<F_STORE, false>(ctx, off, n, As, ctx->at<uint16_t>(L.Ws), c.rows, L.colsp, p);
  }
  Pack16 k{};
  k.F = X; k.Y = Y; k.n = n; k.dim = k.ld = cols; k.V = V; k.dst = As + off * 2 * L.colsp; k.dimp = L.colsp;
  k.inv = ctx->at<float>(L.iA) + off;
  k.inv2 = ctx->at<float>(L.q) + off;                  // of u: |u| <= 1 for the logistic models; others set theirs later
  CKC(pack16(ctx, k));
  p.ia = ctx->at<float>(L.iA); p.ib = ctx->at<float>(L.iW);
  return split_product<F_STORE, true>(ctx, off, n, As, ctx->at<uint16_t>(L.Ws), c.rows, L.colsp, p);
}

int split_factors_sc(sfb_ctx* ctx, int64_t off, int64_t n, const float* X) {
  return ctx->h16 ? factors_sc<true>(ctx, off, n, X) : factors_sc<false>(ctx, off, n, X);
}

const uint16_t* split_v(const sfb_ctx* ctx) {
  const Layout& L = ctx->lay;
  const bool odd = ctx->cfg.model == SFB_SC && L.Gs != 0 && (ctx->cfg.sc_ista_iters & 1);     // which buffer the last iterate is in
  return ctx->at<uint16_t>(odd ? L.As2 : L.As);
}
static float* inv_v(const sfb_ctx* ctx) {
  if (ctx->cfg.model != SFB_SC) return ctx->at<float>(ctx->lay.iA);
  return ctx->at<float>(ctx->lay.iC) + (ctx->cfg.sc_ista_iters & 1) * ctx->K;
}

int split_pack_received(sfb_ctx* ctx, int64_t off, int64_t n) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  cudaStream_t s = ctx->stream;
  const float* U = ctx->at<float>(L.U) + off * L.ldu;
  const float* V = ctx->at<float>(L.V) + off * c.cols;
  uint16_t* dst = const_cast<uint16_t*>(split_v(ctx)) + off * 2 * L.colsp;
  if (!ctx->h16) {
    CKC(pack_rows(ctx, U, nullptr, n, c.rows, L.ldu, nullptr, ctx->at<uint16_t>(L.Rs) + off * 2 * L.rowsp, L.rowsp, Stamp{}));
    CKC(pack_rows(ctx, V, nullptr, n, c.cols, c.cols, nullptr, dst, L.colsp, Stamp{}));
    return SFB_OK;
  }
  Pack16 k{};
  k.F = V; k.n = n; k.dim = k.ld = c.cols; k.dst = dst; k.dimp = L.colsp; k.inv = inv_v(ctx) + off;
  CKC(pack16(ctx, k));
  CKC(launch_kernel(row_most_kernel, dim3(static_cast<unsigned>(n)), dim3(256), 0, s, 1, U, L.ldu, c.rows, inv_v(ctx) + off,
                    ctx->at<float>(L.q) + off));
  return SFB_OK;
}

int split_gather(sfb_ctx* ctx) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  if (!ctx->h16) return SFB_OK;                        // every worker wrote its part of the operands
  const Stamp st = take_stamp(ctx);
  if (c.model == SFB_SC)
    CKC(launch_kernel(row_most_kernel, dim3(static_cast<unsigned>(ctx->K)), dim3(256), 0, ctx->stream, 1, ctx->at<float>(L.U), L.ldu,
                      c.rows, inv_v(ctx), ctx->at<float>(L.q)));
  CKC(launch_kernel(pack_u_kernel, dim3(grid1d(ctx->K * ((c.rows + 3) / 4), 256)), dim3(256), 0, ctx->stream, 1, ctx->at<float>(L.U),
                    L.ldu, ctx->K, c.rows, ctx->at<float>(L.q), inv_v(ctx), ctx->at<uint16_t>(L.Rs), L.rowsp,
                    ctx->at<Scalars>(L.scalars), st));
  return SFB_OK;
}

}  // namespace sfb
