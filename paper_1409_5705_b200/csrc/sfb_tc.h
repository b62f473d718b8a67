// Tensor-core (bf16 operand) path of the SFB step: hooks called by the C ABI layer, and the host-side helpers
// the tensor-core translation units share (sfb_tc.cu: factors and forward product; sfb_update.cu: the update).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>

#include "sfb_internal.h"

namespace sfb {

// Appends the bf16-mode buffers to the workspace layout.
void tc_extend_layout(const sfb_config& c, Layout& L, size_t& off);
// fp32 mode on the tensor cores (MLR and its SDCA form): layout, factors, operand packing of the gathered pairs, update.
void tc32_extend_layout(const sfb_config& c, Layout& L, size_t& off);
int tc32_factors(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const int32_t* labels, const int32_t* sdca_ids,
                 float inv_lam_n);
int tc32_forward_partials(sfb_ctx* ctx, const float* X, const int32_t* labels, float* part_out);
int tc32_finish_factors(sfb_ctx* ctx, const float* parts, int shards);
int tc32_gather(sfb_ctx* ctx);
int tc32_update(sfb_ctx* ctx);
int tc_init(sfb_ctx* ctx);
void tc_destroy(sfb_ctx* ctx);
// Rebuilds the bf16 operand copy of W from the caller's fp32 W (MLR; the other models rebuild theirs every step).
int tc_refresh_operands(sfb_ctx* ctx);
// dml_norm_out (DML, row-sharded form; may be null): receives ||z_i||^2 of this context's rows and z stays unscaled.
// fused: the call is part of one that goes on to the update, so X stays as it is until then.
int tc_factors(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const float* Y, const int32_t* labels, bool fused,
               float* dml_norm_out = nullptr);
// Row-sharded MLR: logits and softmax partials of all K samples against this context's rows; then the factors from
// the partials of all shards.
// Parts in which sfb_step_host had better copy the K samples of MLR in bf16 mode (their logits follow part by part).
int tc_host_parts(const sfb_ctx* ctx);
int tc_forward_partials(sfb_ctx* ctx, const float* X, const int32_t* labels, float* part_out);
int tc_finish_factors(sfb_ctx* ctx, const float* parts, int shards);
int tc_sdca_factors(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const int32_t* labels, const int32_t* ids,
                    float inv_lam_n, bool fused);
// MLR in bf16 mode: the fp32 label entries of all K samples into W and the mean loss, unless the factors call has done that
// (fused); before the update.
int tc_labels(sfb_ctx* ctx);
// MLR, bf16 mode: a worker's factors in fp32 as they are sent, and received fp32 factors put into the bf16 layout.
int tc_export_factors(sfb_ctx* ctx, int64_t off, int64_t n, float* U_out, float* V_out);
int tc_import_factors(sfb_ctx* ctx, int64_t off, int64_t n, const float* U_in, const float* V_in);
// Products of (hi | lo) pairs (sfb_split.cu): metric learning and sparse coding in bf16 mode, every model in fp32 mode
// (ctx->h16).  Layout and set-up; what a step's factors share, formed from W before the first of them; v and z = W v of n
// pairs (v = x, or x - y with Y) into the fp32 factor buffers; the factors of sparse coding; fp32 factors that the caller has
// put into the U and V buffers as operands; the rest of the update's operands once all pairs are there; the operand V.
void split_extend_layout(const sfb_config& c, Layout& L, size_t& off);
cudaError_t split_reset(sfb_ctx* ctx);
int split_init(sfb_ctx* ctx);
int split_begin_step(sfb_ctx* ctx);
int split_logits(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const float* Y);
int split_factors_sc(sfb_ctx* ctx, int64_t off, int64_t n, const float* X);
int split_pack_received(sfb_ctx* ctx, int64_t off, int64_t n);
int split_gather(sfb_ctx* ctx);
const uint16_t* split_v(const sfb_ctx* ctx);
double split_product_cost(int64_t M, int64_t N, int64_t Kc, bool sym, bool fine = false);     // fine: sparse coding in fp32 mode
// The same as the forms of the coder are chosen by: the line between forms that round differently does not move with the plans.
double split_form_cost(int64_t M, int64_t N, int64_t Kc, bool sym, bool fine = false);
int split_product_parts(int64_t M, int64_t N, int64_t Kc, bool fine);                         // that a tile is cut into, at most
// MLR, bf16 mode: the kernel of the logits of n samples (see sfb_get_plan) and the parts of a tile; whether the softmax is merged in one launch.
int tc_logits_plan(const sfb_config& c, const Layout& L, int64_t n, bool step, int* parts, bool* merged);
int tc_update(sfb_ctx* ctx);
int tc_get_factors(sfb_ctx* ctx, const void** U, const void** V, int32_t* dtype, int32_t* layout, int64_t* ldu,
                   int64_t* ldv);

// The forward product on pairs of CTAs (sfb_forward.cu): its cycles; its buffers (parts of tiles, their flags); the logits of n packed
// samples at pair offset off, *pw: classes per softmax partial.
double forward_pair_cost(int64_t n, int64_t rows, int64_t cols);
bool forward_pair_pays(int64_t n, int64_t rows, int64_t cols, double other, int64_t other_groups, int* parts);
int64_t forward_pair_groups(int64_t rows);           // most softmax partials of a sample
int64_t forward_pair_cut(int64_t n, int64_t rows, int64_t cols);      // pairs that leave parts of tiles
size_t forward_pair_partial_bytes(int64_t pairs);
size_t forward_pair_ready_bytes();
cudaError_t forward_pair_prepare(int* max_pairs);
cudaError_t forward_pair(sfb_ctx* ctx, int64_t off, int64_t n, int* pw);

// The same for up to 64 samples (forward_few_kernel): whether it takes these sizes; softmax partials, of 32 classes; most resident
// clusters of 1 to 4 CTAs.
bool forward_few_fits(int64_t n, int64_t rows, int64_t cols, bool step);      // step: in a call that goes on to the update
int64_t forward_few_groups(int64_t rows);
cudaError_t forward_few_prepare(int (&most)[5]);
cudaError_t forward_few(sfb_ctx* ctx, int64_t off, int64_t n);

constexpr int32_t kNoSlot = 0x7f7f7f7f;              // a label-row slot that no sample has: above every index (K <= 2^20)

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct MapKey {
  void* base;
  int64_t inner, outer, pitch;
  int32_t dt, box_inner, box_outer;
  bool operator==(const MapKey& o) const {
    return base == o.base && inner == o.inner && outer == o.outer && pitch == o.pitch && dt == o.dt && box_inner == o.box_inner &&
           box_outer == o.box_outer;
  }
};

struct TcState {
  // tensor maps made so far: the buffers of a context stay where they are, so a step finds all of its maps here
  static constexpr int kMaps = 256;
  MapKey key[kMaps];
  CUtensorMap map[kMaps];
  EncodeTiledFn encode;      // cuTensorMapEncodeTiled, obtained through the runtime's driver entry point query
  int sms;                   // multiprocessors of the device
  int few[5];                // resident clusters of 1 to 4 CTAs of forward_few_kernel
  int max_pairs;             // CTA pairs (clusters of 2) of the update kernel that can be resident at once
};

// 2-D row-major tensor [outer x inner] with row pitch `pitch_bytes`, box [box_outer x box_inner], 128-byte swizzle.
inline bool make_map(TcState* st, CUtensorMap* m, CUtensorMapDataType dt, void* base, int64_t inner,
                     int64_t outer, int64_t pitch_bytes, int box_inner, int box_outer) {
  if (inner <= 0 || outer <= 0) return false;
  const MapKey k{base, inner, outer, pitch_bytes, static_cast<int32_t>(dt), box_inner, box_outer};
  uint64_t h = reinterpret_cast<uintptr_t>(base) / 1024 * 31 + static_cast<uint64_t>(outer) * 7 + static_cast<uint64_t>(inner) * 3 +
               static_cast<uint64_t>(box_outer);
  const int slot = static_cast<int>((h ^ (h >> 17)) % TcState::kMaps);
  if (!(st->key[slot] == k)) {
    cuuint64_t dims[2] = {static_cast<cuuint64_t>(inner), static_cast<cuuint64_t>(outer)};
    cuuint64_t strides[1] = {static_cast<cuuint64_t>(pitch_bytes)};
    cuuint32_t box[2] = {static_cast<cuuint32_t>(box_inner), static_cast<cuuint32_t>(box_outer)};
    cuuint32_t estr[2] = {1, 1};
    if (st->encode(&st->map[slot], dt, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
      st->key[slot] = MapKey{};
      return false;
    }
    st->key[slot] = k;
  }
  *m = st->map[slot];
  return true;
}

// Fills st->max_pairs (occupancy query of the update kernel); defined beside that kernel.
int tc_update_init(sfb_ctx* ctx, TcState* st);

}  // namespace sfb
