// Internal declarations shared by the translation units of libsfb (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include <atomic>
#include <stdint.h>

#include "sfb.h"

namespace sfb {

extern std::atomic<int64_t> g_kernel_launches;     // kernels launched by this library in this process
inline void count_launch(int n = 1) { g_kernel_launches.fetch_add(n, std::memory_order_relaxed); }

// Multiprocessors of the current device (looked up once per device ordinal).
int sm_count();
constexpr int kModelSms = 148;        // what the cost models, hence the layout of a workspace, count with: no CUDA call

// ---------------------------------------------------------------------------------------------------------
// Launches.  A step is a chain of dependent kernels, several of them only microseconds long: each is launched with
// programmatic stream serialisation, so that its blocks are scheduled and its set-up runs while the kernel before it
// drains.  Every kernel launched this way calls pdl_wait() before it touches memory (it returns when the kernels before it
// have completed and their writes are visible) and pdl_launch_dependents() early (the next kernel may then start its own
// set-up once all blocks of this one are running).  The tile kernels are launched this way only when they have at most one
// tile per SM: started while the SMs fall free one by one, their blocks land on them in that order, neighbours apart, and the
// operands that neighbours share are read across the dies (3-4 % of a step at 325,000 x 10,000).
// ---------------------------------------------------------------------------------------------------------
struct Stamp {                        // the first block stores the time to at[0] .. at[n - 1]
  unsigned long long* at;
  int32_t n;
};
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// ... with all of the kernel's `__restrict__` parameters: nothing the wait may touch can alias those, so the compiler may move their
// loads and stores above it (a load of a scalar was), unless their addresses come from something that it learns after the wait.
template <typename... P>
__device__ __forceinline__ void pdl_wait(P&... p) {
  pdl_wait();
  int64_t zero = 0;
  asm volatile("" : "+l"(zero) :: "memory");
  ((p += zero), ...);
}
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Time stamps of the phases of a step (sfb_stats.ms_*), written by the kernels themselves: events between them would keep a
// kernel from being scheduled before the one ahead of it has drained.
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void stamp_begin(const Stamp& s) {
  if (s.n > 0 && threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0) {
    const unsigned long long t = global_ns();
    for (int i = 0; i < s.n; ++i) s.at[i] = t;
  }
}
__device__ __forceinline__ void stamp_end(unsigned long long* at) {      // the latest block's time stays
  if (at && threadIdx.x == 0) atomicMax(at, global_ns());
}

template <typename... KArgs, typename... Args>
cudaError_t launch_kernel_if(bool early, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                             int cluster, const Args&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2]{};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = static_cast<unsigned>(cluster);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, int cluster,
                          const Args&... args) {
  return launch_kernel_if(true, kernel, grid, block, smem, s, cluster, args...);
}

// The shared-memory opt-in of a kernel, once per device.
template <auto Kernel>
cudaError_t allow_smem(int bytes) {
  static std::atomic<uint64_t> done{0};                // one bit per device ordinal
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = 1ull << (dev & 63);
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
  return e;
}
#endif

// ---------------------------------------------------------------------------------------------------------
// Workspace carve-up.  Every offset is a multiple of 1024 bytes so that any sub-buffer can be a TMA base.
// ---------------------------------------------------------------------------------------------------------
constexpr size_t kAlign = 1024;
constexpr int kProxSlabs = 64;        // row slabs of the deterministic column reductions

struct Layout {
  size_t status, scalars, loss, V, U, colpart, stageX, stageY, stageL;
  // bf16 tensor-core mode
  size_t Wb, Xb, VT, ZT, UT, P, part, Xf, labels, coef, lse, slot, dL;   // VT, UT: tf32 words only; P: probabilities [K x ldp]; slot, dL: label rows
  // (hi | lo) operands of the split products
  size_t Ws, WTs, As, Rs;             // W by rows, W transposed, the A operand (v or the codes), the residual
  size_t partial, ready;              // parts of the tiles of a split product
  size_t iW, iA, iR, iC, q, mR, mC;   // fp32 mode: inverse scales of the rows of W, of the pairs, what they are taken from; see sfb_split.cu
  // sparse factors (MLR, csr_nnz_max > 0): the step's (sample, column, value) triples and their column-major form
  size_t coo_i, coo_c, coo_x, coo_cx, row_beg, row_end, csc_cnt, csc_cur, csc_ptr, csc_tmp, csc_ent;
  // sparse coding: the dictionary's Gram matrix (when the coder iterates on it), W^T x, the codes of odd iterations, and
  // the scratch of the power iteration
  size_t G, Gs, Bx, V2, As2, pi;
  size_t Wd, Gd, Xd, Bd, Ad;          // in fp64: W, W^T W, the samples, W^T x and the codes, transposed (see sfb_gram64.cu)
  int64_t ldu;                        // row pitch of the fp32 U buffer (rows rounded up to 4; rows itself with tf32 pairs)
  int64_t colsp, rowsp;               // cols, rows rounded up to 64
  int64_t Kp;                         // K rounded up to the contraction block of the update product
  int32_t split;                      // parts that the bf16 forward product of MLR cuts its contraction into
  int32_t pw;                         // columns per softmax partial of the bf16 forward product
  bool on_pairs;                      // some call's logits take the kernel of CTA pairs
  int32_t cut_pairs;                  //   and of those, pairs that leave parts of tiles, at most
  int64_t ldp;                        // row pitch of P: rows rounded up to 64
  int64_t colsb;                      // cols rounded up to the contraction block of the forward product
  size_t total;
};

Layout make_layout(const sfb_config& c);
bool sc_use_gram(const sfb_config& c);        // the coder on W^T W: bf16 mode;
bool sc_use_gram64(const sfb_config& c);      //   FMA kernels of the fp32 mode, in fp64
bool sc_on_pairs(const sfb_config& c);
bool sc_estimate_on_gram(const sfb_config& c, double form);     // L estimated on a W^T W that costs `form` cycles
inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// Which kernels the products of an fp32 mode run on.  Pairs of tf32 words when asked for (logistic models).  SFB_PREC_FP32 runs
// on pairs of fp16 words with fp32 scales (sfb_split.cu) where the products are large enough to repay the packing of their
// operands (W once per step, as much work as 24 more pairs), else on the FMA kernels.  Sparse coding by the
// costs of its forms (sc_on_pairs).  us per step, fp16 pairs / FMAs: sparse coding 814 x 1,252 K = 620 1311 / 2240, 2,422 x 760 K = 209
// 1201 / 723; metric learning 300 x 1,000 K = 500 55 / 49,
// 500 x 4,000 K = 100 66 / 77; regression 2,000 x 5,000 K = 16 128 / 90, 3,000 x 600 K = 130 50 / 64, 10,000 x 20,000 K = 16
// 1306 / 1583, 50,000 x 64 K = 256 192 / 148 (bound by u, which is packed too).
inline bool use_tf32(const sfb_config& c) {
  return c.precision == SFB_PREC_TF32X3 && (c.model == SFB_MLR || c.model == SFB_L2MLR);
}
// Whether W and operands derived from it of `per_entry` bytes an entry leave room in the 180 GB of a GPU for samples and factors; the
// FMA kernels need none (1,000,000 x 20,000: W 80 GB, its pairs as much again, those of W^T for sparse coding 80 more).
inline bool derived_fit(const sfb_config& c, double per_entry) {
  return (4.0 + per_entry) * static_cast<double>(c.rows) * static_cast<double>(c.cols) <= 150e9;
}
inline bool use_h16(const sfb_config& c) {
  if (c.precision != SFB_PREC_FP32 || c.rows < 64 || c.cols < 64) return false;
  if (!derived_fit(c, c.model == SFB_SC ? 8.0 : 4.0)) return false;
  const double K = static_cast<double>(c.workers) * c.batch, macs = K * static_cast<double>(c.rows) * static_cast<double>(c.cols);
  if (c.model == SFB_SC) return sc_on_pairs(c);
  return c.cols >= 256 && (macs >= 1e9 || macs * (1.0 - 24.0 / K) >= 1.8e8);
}

bool sparse_on_fma(const sfb_config& c);      // sparse samples of such a context: on the FMA kernels all the same (see sfb_sparse.cu)

struct Scalars {                      // device-resident scalars
  float loss_mean;
  float L;                            // ||W||_2^2 used by the coder
  float invL;
  float iWT, iWT2, iU;                // inverse scales: W^T and its square, u (see sfb_split.cu)
  unsigned long long copy_pieces;     // 64-byte row pieces of the bf16 operand copy the update passes went over ...
  unsigned long long copy_written;    // ... and how many of them they had to rewrite (the others already held bf16(W))
  unsigned long long ns[4];           // global time at the start of the step, of its gather and of its update, and at its end
};

}  // namespace sfb

namespace sfb {
// For sfb_step_host, made by its first call: a stream for the copies of the mini-batch's parts, an event per part (and one for the
// work ahead of the call), page-locked memory for what is read back.
struct HostSide {
  static constexpr int kParts = 8;
  cudaStream_t copies;
  cudaEvent_t ahead, part[kParts];
  char* back;
  int parts;                          // of the call that is being enqueued (0: none, the samples are there)
};
}  // namespace sfb

struct sfb_ctx {
  sfb::HostSide* host;
  sfb_config cfg;
  sfb::Layout lay;
  float* W;
  char* ws;
  cudaStream_t stream;
  int64_t K;
  int64_t in_dim;
  int64_t row_offset;                 // row-sharded MLR: this context's W holds rows [row_offset, row_offset + rows)
  int64_t global_rows;                //   of a matrix with global_rows rows (class ids are global); 0, rows when unsharded
  bool partials_ready;                // sfb_forward_partials has run since the last update
  bool tf32, h16;                     // fp32 modes with their products on the tensor cores (see use_tf32, use_h16)
  bool sparse_fma;                    // h16, but sparse samples take the FMA kernels; bit p of fma_mask: worker p's of this step did
  uint64_t fma_mask;
  bool update_fma;                    // the gathered factors are not all there as pairs: the update takes the FMA kernels
  bool sdca;                          // SFB_L2MLR: the factors are dual changes; cfg.model is kept as SFB_MLR internally
  float* dualQ;                       // SDCA dual state [dual_n x rows], caller-owned
  int64_t dual_n;
  float step;                         // multiplier of sum u v^T in the update: eta, or eta / (lam N) for SDCA
  int32_t prox_kind;                  // entry-wise prox of the update pass and its parameter (threshold or factor)
  float prox_a;
  uint64_t committed;                 // bit p set: worker p has written its factors since the last update
  bool begun;                         // what the workers' factors of this step share has been derived from W
  uint64_t sparse_mask;               // bit p set: worker p's samples of this step came in compressed-sparse-row form
  int64_t csr_fill;                   // triples staged so far in this step
  int64_t last_stage_nnz;             // entries of the last staged block of samples
  bool sparse_v;                      // the gathered v are in column-major sparse form: the update sums only the non-zeros
  bool gathered;
  bool packed;                        // the samples of the call at hand are operands already, their labels and slots set (see sparse_stage_packed)
  int last_cuda;
  // MLR, bf16 mode: the label entries of the step's factors are not in W; in W by the factors call; were in a past update,
  // their sums kept
  enum Labels : int8_t { kLabelsNone, kLabelsApplied, kLabelsKept } labels;
  sfb::Stamp pending;                 // phases whose beginning the next kernel that can will stamp
  sfb_stats stats;
  void* tc;                           // tensor-core path state (tensor maps), owned

  // the stamps that the next kernel takes along (their phases begin with it)
  sfb::Stamp take_pending() { const sfb::Stamp s = pending; pending = sfb::Stamp{}; return s; }

  template <typename T>
  T* at(size_t off) const { return reinterpret_cast<T*>(ws + off); }
};

namespace sfb {

inline Stamp take_stamp(sfb_ctx* ctx) { return ctx->take_pending(); }

// ---------------------------------------------------------------------------------------------------------
// fp32 FMA matrix products:  C (M x N) = sum_k A(m,k) * B(n,k)  followed by an epilogue.
// A_KC: A(m,k) at A[m*lda + k] (k contiguous), else at A[k*lda + m].  Same for B with n.
//   EPI_STORE  C = acc                                     EPI_SUB    C = acc - aux
//   EPI_RMW    C = prox(C + alpha acc)
//   EPI_ISTA   C = soft(cur - acc / L, lam / L)            EPI_ISTA0  C = soft(acc / L, lam / L), C2 = acc
// ---------------------------------------------------------------------------------------------------------
enum Epilogue { EPI_STORE = 0, EPI_SUB = 1, EPI_RMW = 2, EPI_ISTA = 3, EPI_ISTA0 = 4 };

// Entry-wise proximal operator fused into the update: kind 1 soft-threshold by a, kind 2 multiply by a.
__host__ __device__ __forceinline__ float prox_entry(float w, int kind, float a) {
  if (kind == 1) {
    const float m = fabsf(w) - a;
    return m > 0.f ? copysignf(m, w) : 0.f;
  }
  return kind == 2 ? w * a : w;
}

struct EpiArgs {
  int32_t prox_kind;   // EPI_RMW: entry-wise prox applied to the updated value (0 none)
  float prox_a;
  float alpha;         // EPI_RMW
  float lam;           // EPI_ISTA, EPI_ISTA0
  Stamp begin;         // EPI_RMW: time stamps
  unsigned long long* end;
  float* C;            // output, row-major [M x ldc]
  int64_t ldc;
  float* C2;           // EPI_ISTA0 (may be null)
  int64_t ldc2;
  const float* aux;    // EPI_SUB
  int64_t ldaux;
  const float* cur;    // EPI_ISTA
  int64_t ldcur;
  const Scalars* sc;   // EPI_ISTA, EPI_ISTA0: reads invL
};

struct GemmShape { int tile, split; };               // tile edge; parts the contraction is cut into
double gemm_cost(int tile, int split, int64_t M, int64_t N, int64_t Kc);
GemmShape pick_gemm_shape(int64_t M, int64_t N, int64_t Kc);
double gemm_cycles(int64_t M, int64_t N, int64_t Kc);               // in the better tile

// M_split (0: M): the row count that decides how the contraction is split; callers that compute a product in slices of
// rows pass the whole product's, so that a row has the same bits whichever slice it is computed in.
cudaError_t sgemm(cudaStream_t s, bool a_kc, bool b_kc, Epilogue epi, int64_t M, int64_t N, int64_t Kc,
                  const float* A, int64_t lda, const float* B, int64_t ldb, const EpiArgs& e, int64_t M_split = 0);

// The coder of the fp32 mode on W^T W in fp64 (sfb_gram64.cu): cycles of a product, and of W^T W with W widened; buffers (of W^T W
// alone without coder); W^T W (G32, may be null: also in fp32); the codes of n samples to V.
double gram64_cost(int64_t N, int64_t M, int64_t Kc);
double gram64_form_cost(int64_t D, int64_t A);
void gram64_extend_layout(const sfb_config& c, bool coder, Layout& L, size_t& off);
cudaError_t gram64_begin(sfb_ctx* ctx, float* G32);
cudaError_t gram64_codes(sfb_ctx* ctx, int64_t n, const float* X, float* V);

// ---------------------------------------------------------------------------------------------------------
// Factor kernels (pack, softmax, pair residual, prox, power iteration)
// ---------------------------------------------------------------------------------------------------------
cudaError_t stamp(cudaStream_t s, const Stamp& st);
cudaError_t pack_copy(cudaStream_t s, float* dst, const float* x, const float* y_or_null, int64_t n, const Stamp& st);
cudaError_t fill_zero(cudaStream_t s, float* dst, int64_t n);
cudaError_t mlr_softmax_rows(cudaStream_t s, float* Z, int64_t nsamp, int64_t rows, int64_t ldz, const int32_t* labels,
                             float* loss_per_sample, uint32_t* status);
// Row-sharded MLR: per-sample softmax partials (max, sum exp, label logit, owner flag) of a shard, and the finish with
// the partials of all shards ([shards][nsamp] float4).
cudaError_t mlr_shard_partials(cudaStream_t s, const float* Z, int64_t nsamp, int64_t rows, int64_t ldz,
                               const int32_t* labels, int64_t row_off, float* part);
cudaError_t mlr_shard_finish(cudaStream_t s, float* Z, int64_t nsamp, int64_t rows, int64_t ldz, const int32_t* labels,
                             int64_t row_off, const float* parts, int shards, float* loss, uint32_t* status);
// SDCA (l2-regularised MLR): per sample, from its logits z, its dual row of Q (advanced by gamma * du) and its features x:
// the change du of the dual vector that minimises the dual objective, written in fp32 to out (row pitch ldo; may be Z) or in
// bf16 to P with a 0 at the label entry and -du there to coef.  slot (may be null): the smallest index, from off on, of a
// sample of each class.
struct SdcaArgs {
  const float* Z;
  int64_t n, rows, ldz;
  const float* X;
  int64_t cols;
  const int32_t* labels;
  const int32_t* ids;
  float* Q;
  int64_t n_samples;
  float inv_lam_n, gamma;
  float* out;
  int64_t ldo;
  void* P;
  int64_t ldp;
  float* coef;
  float* loss;
  uint32_t* status;
  int32_t* slot;
  int64_t off;
};
cudaError_t sdca_dual_rows(cudaStream_t s, const SdcaArgs& a);
SdcaArgs sdca_args(const sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const int32_t* labels, const int32_t* ids,
                   float inv_lam_n);               // all but the logits and where du goes
// Row-sharded form: norm_out (may be null) receives the shard's ||z_i||^2 and z is left unscaled; norms_all (may be null),
// [shards][nstride], supplies ||z_i||^2 as the sum over the shards instead of this context's own.
// split (may be null): the scaled rows also as (hi | lo) bf16 pairs, row pitch 2 * split_half.  most (may be null): receives
// inv_v[i] * max_j |u_ij|.
cudaError_t dml_scale_rows(cudaStream_t s, float* Z, int64_t nsamp, int64_t rows, int64_t ld,
                           const int32_t* similar, float margin, void* split = nullptr, int64_t split_half = 0,
                           const float* inv_v = nullptr, float* most = nullptr, float* norm_out = nullptr,
                           const float* norms_all = nullptr, int shards = 0, int64_t nstride = 0);
cudaError_t mean_of(cudaStream_t s, const float* v, int64_t n, float* out, const Stamp& st);
cudaError_t prox_unit_columns(cudaStream_t s, float* W, int64_t rows, int64_t cols, float* colpart, unsigned long long* end);
// L = ||W||_2^2 by power iterations from the normalised all-ones vector, on W^T W itself when G is given, else on W.
// scratch: power_scratch_bytes(cols).
cudaError_t estimate_lipschitz(cudaStream_t s, const float* W, const float* G, int64_t rows, int64_t cols, void* scratch,
                               Scalars* sc, uint32_t* status, int iters);
size_t power_scratch_bytes(int64_t cols);
cudaError_t set_lipschitz(cudaStream_t s, Scalars* sc, float L);
cudaError_t axpy(cudaStream_t s, float* y, const float* x, float alpha, int64_t n);  // y += alpha*x
cudaError_t prox_entries(cudaStream_t s, float* w, int64_t n, int kind, float a);      // w <- prox(w), entry-wise

// ---------------------------------------------------------------------------------------------------------
// Sparse sufficient factors (MLR): staging of compressed-sparse-row samples, their column-major form, the update
// ---------------------------------------------------------------------------------------------------------
void sparse_extend_layout(const sfb_config& c, Layout& L, size_t& off);
// The step's sparse samples take the sparse update: its factor slab of K samples fits the shared memory of a block and,
// unless the config forces either, the cost model prefers it to the tensor-core update over the scattered samples.
bool sparse_update_wanted(const sfb_ctx* ctx);
int sparse_stage(sfb_ctx* ctx, int64_t off, int64_t n, const int64_t* indptr, const int32_t* idx, const float* val,
                 int64_t nnz);
// bf16 mode, rows that fit shared memory: staged and packed in one kernel, in fp32 to Xd [K x cols].
bool sparse_stage_packs(const sfb_ctx* ctx);
int sparse_stage_packed(sfb_ctx* ctx, int64_t off, int64_t n, const int64_t* indptr, const int32_t* idx, const float* val, int64_t nnz,
                        const int32_t* labels, float* Xd);
// fp32 FMA mode: rows of W per block of the row-wise forward over sparse samples (0: the rows do not fit), and that product
bool sparse_forward_wanted(const sfb_ctx* ctx, int64_t n);
int sparse_forward(sfb_ctx* ctx, int64_t off, int64_t n, float* Z, int64_t ldz);
int sparse_build_csc(sfb_ctx* ctx);
int sparse_update(sfb_ctx* ctx);

}  // namespace sfb
