// C ABI of libsfb: argument checking, workspace carve-up, and the sequencing of one SFB step
// (Section 3, Figure 1: compute factors -> broadcast/gather -> reconstruct and apply -> prox).
#include <algorithm>
#include <new>

#include "sfb_internal.h"
#include "sfb_tc.h"

namespace sfb {

std::atomic<int64_t> g_kernel_launches{0};

int sm_count() {
  constexpr int kMaxDevices = 64;
  static std::atomic<int> cache[kMaxDevices];          // zero-initialised: 0 = not looked up yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 148;
  int n = cache[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
    cache[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

static size_t up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

// The coder's iterations a <- soft(a - W^T (W a - x) / L) either take two products with W each, or one with the Gram matrix
// W^T W, formed once per step (half of it: it is symmetric), and W^T x.  The Gram form wins when the mini-batch is large enough
// to repay W^T W; decided by the cost of the products themselves (10,000 x 5,000, K = 512, 20 iterations, bf16: 5.0 -> 2.2 ms
// for the coder).  In bf16 mode it is kept to dictionaries with no more atoms than features: the residual of an overcomplete one
// becomes small against x, and the two-product form then rounds relative to it where W^T W a - W^T x rounds relative to W^T x
// (500 x 1,400: 4.8e-6 against 1.2e-5).  The fp32 mode has it in fp64 only, on the FMA kernels, for the same reason (see
// sfb_gram64.cu).
static double sc_iterations(const sfb_config& c) { return c.sc_ista_iters - 1; }
constexpr int64_t kMostAtoms = 32 << 10;     // (the power iteration keeps a vector of them on chip)

bool sc_use_gram(const sfb_config& c) {
  const int64_t K = static_cast<int64_t>(c.workers) * c.batch, D = c.rows, A = c.cols;
  const double it = sc_iterations(c);
  if (c.precision != SFB_PREC_BF16 || it < 1 || A > D || A > kMostAtoms) return false;
  return split_form_cost(A, A, D, true) + it * split_form_cost(K, A, A, false) <
         it * (split_form_cost(K, D, A, false) + split_form_cost(K, A, D, false));
}

// The power iteration on W^T W, whose rows stay on chip, or on W, which comes from L2 or memory twice an iteration, with a barrier
// between (2,500 x 1,000: 2.6 us an iteration against 21).
bool sc_estimate_on_gram(const sfb_config& c, double form) {
  if (c.sc_lipschitz > 0.f || c.cols > kMostAtoms || !derived_fit(c, 8.0)) return false;
  const double D = static_cast<double>(c.rows), A = static_cast<double>(c.cols);
  return form + 50.0 * (4000.0 + A * A * 4.0 / 3000.0) < 50.0 * (10000.0 + D * A * 8.0 / 640.0);
}

// SM cycles of the coder's products on the FMA kernels, in the cheaper of the two forms; W^T W is there where L is estimated on it.
static double sc_fma_cost(const sfb_config& c, bool& gram64) {
  const int64_t K = static_cast<int64_t>(c.workers) * c.batch, D = c.rows, A = c.cols;
  const double it = sc_iterations(c), last = gemm_cycles(K, D, A), form = gram64_form_cost(D, A);
  const double there = sc_estimate_on_gram(c, form) ? form : 0.0;
  gram64 = false;
  if (it < 0) return last + there;
  const double two = gemm_cycles(K, A, D) + it * (gemm_cycles(K, D, A) + gemm_cycles(K, A, D)) + last + there;
  if (it < 1 || A > kMostAtoms || !derived_fit(c, 8.0)) return two;
  const double one = form + gram64_cost(A, K, D) + it * gram64_cost(A, K, A) + last + 10000.0;
  gram64 = one < two;
  return std::min(one, two);
}
bool sc_use_gram64(const sfb_config& c) {
  bool gram64 = false;
  sc_fma_cost(c, gram64);
  return gram64;
}
// Whether the products of sparse coding in fp32 mode are better off as pairs of fp16 words: the packing of W and W^T at 4.5 TB/s, two
// products an iteration.  Against W^T W in fp64 by the plans' cost: 88 drawn dictionaries on this side of the line that lay on the other
// by split_form_cost take 0.64 times as long in fp64, and their codes are 0.12 times as far from 64 bits.  Against two products of FMAs by
// split_form_cost: 199 on the other side of that line take 0.99 times as long, 97 of them more than 3 % longer, and their codes are up to 2.1
// times as far off (4,960 x 820, 5 iterations: 2.3e-7 on pairs, 4.6e-7).
bool sc_on_pairs(const sfb_config& c) {
  const int64_t K = static_cast<int64_t>(c.workers) * c.batch, D = c.rows, A = c.cols;
  bool gram64;
  const double fma = sc_fma_cost(c, gram64);
  auto product = [&](int64_t N, int64_t Kc) { return gram64 ? split_product_cost(K, N, Kc, false, true) : split_form_cost(K, N, Kc, false, true); };
  const double it = sc_iterations(c), size = static_cast<double>(D) * static_cast<double>(A), form = split_product_cost(A, A, D, true, true);
  const double toD = product(D, A), toA = product(A, D);
  const double pairs = toD + size * 16.0 / 4.5e12 * 1.9e9 + 20000.0 + (it >= 0 ? toA + it * (toD + toA) : 0.0) + (sc_estimate_on_gram(c, form) ? form : 0.0);
  return pairs < fma;
}

Layout make_layout(const sfb_config& cfg) {
  sfb_config c = cfg;
  if (c.model == SFB_L2MLR) c.model = SFB_MLR;        // same buffers: the factors differ, the products do not
  Layout L{};
  const size_t K = static_cast<size_t>(c.workers) * c.batch;
  const size_t rows = c.rows, cols = c.cols;
  const size_t in_dim = c.model == SFB_SC ? rows : cols;
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += up(bytes); return o; };
  L.status = take(sizeof(uint32_t));
  L.scalars = take(sizeof(Scalars));
  L.loss = take(K * 4);
  L.stageX = take(K * in_dim * 4);
  L.stageY = take(c.model == SFB_DML ? K * cols * 4 : 0);
  L.stageL = take(K * 4);
  L.colpart = take(c.model == SFB_SC ? static_cast<size_t>(kProxSlabs) * cols * 8 : 0);
  L.pi = take(c.model == SFB_SC && !(c.sc_lipschitz > 0.f) ? power_scratch_bytes(c.cols) : 0);
  L.Kp = static_cast<int64_t>(K);
  L.colsb = static_cast<int64_t>(cols);
  L.ldu = static_cast<int64_t>(rows);
  if (use_tf32(cfg)) {
    tc32_extend_layout(c, L, off);
  } else if (use_h16(cfg)) {
    split_extend_layout(c, L, off);
  } else if (c.precision != SFB_PREC_BF16) {
    L.ldu = round_up(c.rows, 4);                      // 16-byte row pitch
    L.V = take(K * cols * 4);
    L.U = take(K * static_cast<size_t>(L.ldu) * 4);
    if (c.model == SFB_SC) {
      const bool coder = sc_use_gram64(c), estimate = sc_estimate_on_gram(c, gram64_form_cost(c.rows, c.cols));
      if (coder || estimate) gram64_extend_layout(c, coder, L, off);
      if (estimate || (coder && !(c.sc_lipschitz > 0.f))) L.G = take(cols * cols * 4);      // in fp32 for the power iteration
    }
    if (c.model == SFB_SC) L.V2 = take(K * cols * 4);
  } else {
    tc_extend_layout(c, L, off);
  }
  if (c.csr_nnz_max > 0 && c.model == SFB_MLR) sparse_extend_layout(c, L, off);
  L.total = off;
  return L;
}

}  // namespace sfb

using namespace sfb;

#define CK(call)                                        \
  do {                                                  \
    cudaError_t e__ = (call);                           \
    if (e__ != cudaSuccess) {                           \
      ctx->last_cuda = static_cast<int>(e__);           \
      return SFB_ERR_CUDA;                              \
    }                                                   \
  } while (0)

// The phase that begins now (0 the step, 1 its gather, 2 its update) takes the time of the next kernel that can stamp it.
static void begin_phase(sfb_ctx* ctx, int phase) {
  unsigned long long* at = &ctx->at<Scalars>(ctx->lay.scalars)->ns[phase];
  if (ctx->pending.n > 0 && ctx->pending.at + ctx->pending.n == at) ctx->pending.n += 1;     // nothing ran in between
  else ctx->pending = Stamp{at, 1};
}

static bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

static int check_config(const sfb_config* c) {
  if (!c) return SFB_ERR_ARG;
  if (c->model < SFB_MLR || c->model > SFB_L2MLR) return SFB_ERR_ARG;
  if (c->model == SFB_L2MLR && (!(c->sdca_lambda > 0.f) || c->sdca_n < 1)) return SFB_ERR_ARG;
  if (c->precision < SFB_PREC_BF16 || c->precision > SFB_PREC_FP32_FFMA) return SFB_ERR_ARG;
  if (c->precision == SFB_PREC_TF32X3 && c->model != SFB_MLR && c->model != SFB_L2MLR) return SFB_ERR_UNSUPPORTED;
  if (c->rows <= 0 || c->cols <= 0 || c->workers <= 0 || c->batch <= 0) return SFB_ERR_ARG;
  if (c->workers > 64) return SFB_ERR_SHAPE;
  if (c->cols % 4 != 0) return SFB_ERR_SHAPE;
  if (c->rows > (1LL << 30) || c->cols > (1LL << 30)) return SFB_ERR_SHAPE;
  if (static_cast<int64_t>(c->workers) * c->batch > (1 << 20)) return SFB_ERR_SHAPE;
  if (c->model == SFB_SC && c->sc_ista_iters < 0) return SFB_ERR_ARG;
  if (c->model == SFB_SC && !(c->sc_lambda >= 0.f)) return SFB_ERR_ARG;
  if (c->sc_prox < 0 || c->sc_prox > 1) return SFB_ERR_ARG;
  if (c->prox_kind < 0 || c->prox_kind > 2 || !(c->prox_weight >= 0.f)) return SFB_ERR_ARG;
  if (c->model == SFB_L2MLR && c->prox_kind != 0) return SFB_ERR_UNSUPPORTED;
  if (c->csr_nnz_max < 0 || c->csr_nnz_max + c->cols > (1LL << 31) - 64) return SFB_ERR_SHAPE;
  if (c->csr_update < 0 || c->csr_update > 2) return SFB_ERR_ARG;
  return SFB_OK;
}

extern "C" int sfb_workspace_bytes(const sfb_config* cfg, size_t* out_bytes) {
  if (!out_bytes) return SFB_ERR_ARG;
  int rc = check_config(cfg);
  if (rc) return rc;
  *out_bytes = make_layout(*cfg).total;
  return SFB_OK;
}

extern "C" int sfb_init(const sfb_config* cfg, float* W_dev, void* workspace_dev, size_t workspace_bytes,
                        sfb_ctx** out) {
  if (!out) return SFB_ERR_ARG;
  *out = nullptr;
  int rc = check_config(cfg);
  if (rc) return rc;
  if (!W_dev || !workspace_dev) return SFB_ERR_ARG;
  if (!al16(W_dev) || (reinterpret_cast<uintptr_t>(workspace_dev) & (kAlign - 1)) != 0) return SFB_ERR_ALIGN;
  Layout lay = make_layout(*cfg);
  if (workspace_bytes < lay.total) return SFB_ERR_WORKSPACE;
  int dev = 0, major = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return SFB_ERR_CUDA;
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess) return SFB_ERR_CUDA;
  if (major != 10) return SFB_ERR_ARCH;

  sfb_ctx* ctx = new (std::nothrow) sfb_ctx();
  if (!ctx) return SFB_ERR_ARG;
  ctx->cfg = *cfg;
  ctx->tf32 = use_tf32(*cfg);
  ctx->h16 = use_h16(*cfg);
  if (cfg->precision != SFB_PREC_BF16) ctx->cfg.precision = SFB_PREC_FP32;      // one fp32 family; tf32, h16 say which kernels
  ctx->sparse_fma = ctx->h16 && sparse_on_fma(*cfg);
  ctx->fma_mask = 0;
  ctx->update_fma = false;
  ctx->sdca = cfg->model == SFB_L2MLR;
  if (ctx->sdca) ctx->cfg.model = SFB_MLR;            // the products, buffers and the update are those of MLR
  ctx->dualQ = nullptr;
  ctx->dual_n = 0;
  ctx->step = ctx->sdca ? static_cast<float>(static_cast<double>(cfg->eta) / (static_cast<double>(cfg->sdca_lambda) *
                                                                            static_cast<double>(cfg->sdca_n)))
                        : cfg->eta;
  // prox_{eta h}: threshold eta*w for the l1 norm, factor 1 / (1 + eta*w) for the squared l2 norm
  ctx->prox_kind = cfg->prox_kind;
  ctx->prox_a = cfg->prox_kind == 1 ? cfg->eta * cfg->prox_weight
              : cfg->prox_kind == 2 ? static_cast<float>(1.0 / (1.0 + static_cast<double>(cfg->eta) * cfg->prox_weight)) : 0.f;
  ctx->lay = lay;
  ctx->W = W_dev;
  ctx->ws = static_cast<char*>(workspace_dev);
  ctx->stream = static_cast<cudaStream_t>(cfg->stream);
  ctx->K = static_cast<int64_t>(cfg->workers) * cfg->batch;
  ctx->in_dim = cfg->model == SFB_SC ? cfg->rows : cfg->cols;
  ctx->committed = 0;
  ctx->begun = false;
  ctx->sparse_mask = 0;
  ctx->csr_fill = 0;
  ctx->sparse_v = false;
  ctx->gathered = false;
  ctx->row_offset = 0;
  ctx->global_rows = cfg->rows;
  ctx->partials_ready = false;
  ctx->last_cuda = 0;
  ctx->stats = sfb_stats{};
  ctx->tc = nullptr;
  ctx->host = nullptr;
  ctx->packed = false;
  ctx->labels = sfb_ctx::kLabelsNone;
  ctx->pending = Stamp{};
  // status word, scalars and per-sample losses are the first three (contiguous) regions
  cudaError_t ce = cudaMemsetAsync(ctx->ws + lay.status, 0, lay.stageX - lay.status, ctx->stream);
  if (ce != cudaSuccess) { sfb_destroy(ctx); return SFB_ERR_CUDA; }
  if (cfg->model == SFB_SC && cfg->sc_lipschitz > 0.f) {
    ce = set_lipschitz(ctx->stream, ctx->at<Scalars>(lay.scalars), cfg->sc_lipschitz);
    if (ce != cudaSuccess) { sfb_destroy(ctx); return SFB_ERR_CUDA; }
  }
  if (cfg->precision == SFB_PREC_BF16 || ctx->tf32 || ctx->h16) {
    rc = tc_init(ctx);
    if (rc) { sfb_destroy(ctx); return rc; }
  }
  *out = ctx;
  return SFB_OK;
}

static void free_host_side(HostSide* h) {
  if (!h) return;
  if (h->copies) cudaStreamDestroy(h->copies);
  if (h->ahead) cudaEventDestroy(h->ahead);
  for (cudaEvent_t e : h->part)
    if (e) cudaEventDestroy(e);
  if (h->back) cudaFreeHost(h->back);
  delete h;
}
static cudaError_t make_host_side(sfb_ctx* ctx) {
  HostSide* h = new (std::nothrow) HostSide{};
  if (!h) return cudaErrorMemoryAllocation;
  cudaError_t e = cudaStreamCreateWithFlags(&h->copies, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&h->ahead, cudaEventDisableTiming);
  for (cudaEvent_t& ev : h->part)
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaHostAlloc(reinterpret_cast<void**>(&h->back), ctx->lay.loss - ctx->lay.status, cudaHostAllocDefault);
  if (e == cudaSuccess) ctx->host = h;
  else free_host_side(h);
  return e;
}

extern "C" int sfb_destroy(sfb_ctx* ctx) {
  if (!ctx) return SFB_ERR_ARG;
  tc_destroy(ctx);
  free_host_side(ctx->host);
  delete ctx;
  return SFB_OK;
}

// ---------------------------------------------------------------------------------------------------------
// fp32-operand path
// ---------------------------------------------------------------------------------------------------------
// v = x (or x - y) of n pairs at offset off, and z = W v into U.
static int logits_fp32(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const float* Y, bool pairs) {
  if (pairs) return split_logits(ctx, off, n, X, Y);
  const sfb_config& c = ctx->cfg;
  float* V = ctx->at<float>(ctx->lay.V) + off * c.cols;
  CK(pack_copy(ctx->stream, V, X, Y, n * c.cols, take_stamp(ctx)));
  EpiArgs e{};
  e.C = ctx->at<float>(ctx->lay.U) + off * ctx->lay.ldu; e.ldc = ctx->lay.ldu;
  CK(sgemm(ctx->stream, true, true, EPI_STORE, n, c.rows, c.cols, V, c.cols, ctx->W, c.cols, e, ctx->K));
  ctx->stats.flops += 2.0 * n * c.rows * c.cols;
  return SFB_OK;
}

static int factors_fp32(sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const float* Y,
                        const int32_t* labels, bool pairs, bool sparse_fwd = false, float* dml_norm_out = nullptr) {
  const sfb_config& c = ctx->cfg;
  const int64_t rows = c.rows, cols = c.cols, ldu = ctx->lay.ldu, K = ctx->K;
  float* V = ctx->at<float>(ctx->lay.V) + off * cols;
  float* U = ctx->at<float>(ctx->lay.U) + off * ldu;
  Scalars* sc = ctx->at<Scalars>(ctx->lay.scalars);
  uint32_t* status = ctx->at<uint32_t>(ctx->lay.status);
  cudaStream_t s = ctx->stream;
  EpiArgs e{};
  if (c.model == SFB_MLR || c.model == SFB_DML) {
    if (sparse_fwd) {                                                                   // z_i = W v_i over the non-zeros of v_i
      CK(pack_copy(s, V, X, nullptr, n * cols, take_stamp(ctx)));
      const int rc = sparse_forward(ctx, off, n, ctx->at<float>(ctx->lay.U), ldu);
      if (rc) return rc;
    } else {
      const int rc = logits_fp32(ctx, off, n, X, c.model == SFB_DML ? Y : nullptr, pairs);
      if (rc) return rc;
    }
    if (c.model == SFB_MLR)
      CK(mlr_softmax_rows(s, U, n, rows, ldu, labels, ctx->at<float>(ctx->lay.loss) + off, status));
    else
      CK(dml_scale_rows(s, U, n, rows, ldu, labels, c.dml_margin, nullptr, 0, ctx->h16 ? ctx->at<float>(ctx->lay.iA) + off : nullptr,
                        ctx->h16 ? ctx->at<float>(ctx->lay.q) + off : nullptr, dml_norm_out));
    return SFB_OK;
  }
  if (ctx->h16) return split_factors_sc(ctx, off, n, X);
  // Sparse coding: ISTA from a = 0, then u = W a - x, v = a.  The first iterate is soft(W^T x / L).
  const int T = c.sc_ista_iters;
  float* V2 = ctx->at<float>(ctx->lay.V2) + off * cols;
  auto iterate = [&](int t) { return ((T - t) & 1) == 0 ? V : V2; };                    // where a_t goes: a_T to V
  if (T == 0) {
    CK(fill_zero(s, V, n * cols));
  } else if (ctx->lay.Xd) {
    CK(gram64_codes(ctx, n, X, V));
  } else {
    e.C = iterate(1); e.ldc = cols; e.sc = sc; e.lam = c.sc_lambda;
    CK(sgemm(s, true, false, EPI_ISTA0, n, cols, rows, X, rows, ctx->W, cols, e, K));   // a_1
    ctx->stats.flops += 2.0 * n * rows * cols;
    for (int t = 2; t <= T; ++t) {
      e = EpiArgs{};
      e.C = U; e.ldc = ldu; e.aux = X; e.ldaux = rows;
      CK(sgemm(s, true, true, EPI_SUB, n, rows, cols, iterate(t - 1), cols, ctx->W, cols, e, K));    // r = W a - x
      e = EpiArgs{};
      e.C = iterate(t); e.ldc = cols; e.cur = iterate(t - 1); e.ldcur = cols; e.sc = sc; e.lam = c.sc_lambda;
      CK(sgemm(s, true, false, EPI_ISTA, n, cols, rows, U, ldu, ctx->W, cols, e, K));   // a <- soft(a - W^T r / L)
      ctx->stats.flops += 4.0 * n * rows * cols;
    }
  }
  e = EpiArgs{};
  e.C = U; e.ldc = ldu; e.aux = X; e.ldaux = rows;
  CK(sgemm(s, true, true, EPI_SUB, n, rows, cols, V, cols, ctx->W, cols, e, K));        // u = W a - x
  ctx->stats.flops += 2.0 * n * rows * cols;
  return SFB_OK;
}

// A factors call with which the step begins, or begins anew: the first one, one for all workers, and one for a worker that has
// its factors already (they are computed again, against the W of now).
static bool starts_over(const sfb_ctx* ctx, int32_t worker) {
  return ctx->committed == 0 || worker < 0 || ((ctx->committed >> worker) & 1u) != 0;
}

// What the factors of every worker of a step share, formed from the W that they all see (bulk-synchronous consistency):
// the coder's Gram matrix and its step size.
static int begin_step(sfb_ctx* ctx) {
  const sfb_config& c = ctx->cfg;
  if (ctx->h16 || (c.precision == SFB_PREC_BF16 && c.model != SFB_MLR)) {
    const int rc = split_begin_step(ctx);
    if (rc) return rc;
  }
  if (c.model != SFB_SC) return SFB_OK;
  CK(stamp(ctx->stream, take_stamp(ctx)));
  float* G = ctx->lay.G && !(c.sc_lipschitz > 0.f) ? ctx->at<float>(ctx->lay.G) : nullptr;
  if (ctx->lay.Gd) CK(gram64_begin(ctx, G));
  if (!(c.sc_lipschitz > 0.f))
    CK(estimate_lipschitz(ctx->stream, ctx->W, G, c.rows, c.cols, ctx->at<char>(ctx->lay.pi),
                          ctx->at<Scalars>(ctx->lay.scalars), ctx->at<uint32_t>(ctx->lay.status), 50));
  return SFB_OK;
}

static int update_fp32(sfb_ctx* ctx) {
  const sfb_config& c = ctx->cfg;
  if (ctx->sparse_v) return sparse_update(ctx);
  if (ctx->h16 && !ctx->update_fma) return tc_update(ctx);
  EpiArgs e{};
  e.C = ctx->W; e.ldc = c.cols; e.alpha = -ctx->step;
  e.prox_kind = ctx->prox_kind; e.prox_a = ctx->prox_a;
  e.begin = take_stamp(ctx); e.end = &ctx->at<Scalars>(ctx->lay.scalars)->ns[3];
  CK(sgemm(ctx->stream, false, false, EPI_RMW, c.rows, c.cols, ctx->K, ctx->at<float>(ctx->lay.U), ctx->lay.ldu,
           ctx->at<float>(ctx->lay.V), c.cols, e));
  return SFB_OK;
}

// ---------------------------------------------------------------------------------------------------------
static int check_inputs(sfb_ctx* ctx, const float* X, const float* Y, const int32_t* labels) {
  if (!ctx || !X) return SFB_ERR_ARG;
  if (ctx->cfg.model == SFB_DML && (!Y || !labels)) return SFB_ERR_ARG;
  if (ctx->cfg.model == SFB_MLR && !labels) return SFB_ERR_ARG;
  if (!al16(X) || (Y && !al16(Y))) return SFB_ERR_ALIGN;
  return SFB_OK;
}

// fused: the call belongs to one that goes on to the update.
static int compute_factors(sfb_ctx* ctx, int32_t worker, const float* X_dev, const float* Y_dev, const int32_t* labels_dev,
                           bool fused) {
  int rc = check_inputs(ctx, X_dev, Y_dev, labels_dev);
  if (rc) return rc;
  const sfb_config& c = ctx->cfg;
  if (ctx->sdca) return SFB_ERR_UNSUPPORTED;          // the dual step needs the samples' ids: sfb_sdca_compute_factors
  if (worker < -1 || worker >= c.workers) return SFB_ERR_SHAPE;
  const int64_t off = worker < 0 ? 0 : static_cast<int64_t>(worker) * c.batch;
  const int64_t n = worker < 0 ? ctx->K : c.batch;
  if (ctx->committed == 0) {
    ctx->sparse_mask = ctx->fma_mask = 0;
    ctx->csr_fill = 0;
    begin_phase(ctx, 0);
  }
  if (starts_over(ctx, worker)) ctx->begun = false;
  if (!ctx->begun) {
    if ((rc = begin_step(ctx)) != SFB_OK) return rc;
    ctx->begun = true;
  }
  // bf16 mode: every product runs on the tensor cores; DML and SC, whose u comes from a cancelling residual,
  // carry each value as a (hi, lo) pair of bf16 (fp32-class products)
  rc = ctx->tf32 ? tc32_factors(ctx, off, n, X_dev, labels_dev, nullptr, 0.f)
       : c.precision == SFB_PREC_FP32 ? factors_fp32(ctx, off, n, X_dev, Y_dev, labels_dev, ctx->h16)
                                      : tc_factors(ctx, off, n, X_dev, Y_dev, labels_dev, fused);
  if (rc) return rc;
  const uint64_t all = c.workers == 64 ? ~0ull : ((1ull << c.workers) - 1);
  ctx->committed |= worker < 0 ? all : (1ull << worker);
  ctx->sparse_mask &= ~(worker < 0 ? all : (1ull << worker));       // these samples are dense
  ctx->fma_mask &= ~(worker < 0 ? all : (1ull << worker));
  ctx->gathered = false;
  return SFB_OK;
}

extern "C" int sfb_compute_factors(sfb_ctx* ctx, int32_t worker, const float* X_dev, const float* Y_dev,
                                   const int32_t* labels_dev) {
  return compute_factors(ctx, worker, X_dev, Y_dev, labels_dev, false);
}

// ---------------------------------------------------------------------------------------------------------
// Samples in compressed-sparse-row form (MLR): scattered for the dense forward product, and kept as triples for the
// column-major form that the update reads
// ---------------------------------------------------------------------------------------------------------
static int compute_factors_csr(sfb_ctx* ctx, int32_t worker, const int64_t* indptr_dev, const int32_t* indices_dev,
                               const float* values_dev, int64_t nnz, const int32_t* labels_dev, bool fused) {
  if (!ctx || !indptr_dev || !labels_dev || nnz < 0) return SFB_ERR_ARG;
  if (nnz > 0 && (!indices_dev || !values_dev)) return SFB_ERR_ARG;
  const sfb_config& c = ctx->cfg;
  if (c.model != SFB_MLR || ctx->sdca || c.csr_nnz_max <= 0) return SFB_ERR_UNSUPPORTED;
  if (worker < -1 || worker >= c.workers) return SFB_ERR_SHAPE;
  if (ctx->partials_ready) return SFB_ERR_STATE;
  const uint64_t all = c.workers == 64 ? ~0ull : ((1ull << c.workers) - 1);
  const uint64_t bits = worker < 0 ? all : (1ull << worker);
  if (ctx->committed == 0) {
    ctx->sparse_mask = ctx->fma_mask = 0;
    ctx->csr_fill = 0;
  }
  if (ctx->sparse_mask & bits) return SFB_ERR_STATE;                // its triples are already in the step's list
  if (ctx->csr_fill + nnz > c.csr_nnz_max) return SFB_ERR_SHAPE;
  const int64_t off = worker < 0 ? 0 : static_cast<int64_t>(worker) * c.batch;
  const int64_t n = worker < 0 ? ctx->K : c.batch;
  if (ctx->committed == 0) begin_phase(ctx, 0);
  if (starts_over(ctx, worker)) ctx->begun = false;
  int rc = SFB_OK;
  const bool pairs = ctx->h16 && !ctx->sparse_fma;
  if (!ctx->begun && (pairs || !ctx->h16)) {              // (on the FMA kernels these samples need no pairs of W)
    if ((rc = begin_step(ctx)) != SFB_OK) return rc;
    ctx->begun = true;
  }
  // (in a call that goes on to the update the label rows read the samples from the staging buffer, else from their fp32 copy)
  const bool packed = sparse_stage_packs(ctx);
  float* Xd = ctx->at<float>(packed && !fused ? ctx->lay.Xf : ctx->lay.stageX);
  rc = packed ? sparse_stage_packed(ctx, off, n, indptr_dev, indices_dev, values_dev, nnz, labels_dev, Xd)
              : sparse_stage(ctx, off, n, indptr_dev, indices_dev, values_dev, nnz);
  if (rc) return rc;
  const float* X = Xd + off * c.cols;
  ctx->packed = packed;
  rc = ctx->tf32 ? tc32_factors(ctx, off, n, X, labels_dev, nullptr, 0.f)
       : c.precision == SFB_PREC_FP32 ? factors_fp32(ctx, off, n, X, nullptr, labels_dev, pairs, sparse_forward_wanted(ctx, n))
                                      : tc_factors(ctx, off, n, X, nullptr, labels_dev, fused);
  ctx->packed = false;
  if (rc) return rc;
  ctx->csr_fill += nnz;
  ctx->sparse_mask |= bits;
  if (ctx->sparse_fma) ctx->fma_mask |= bits;
  ctx->committed |= bits;
  ctx->gathered = false;
  return SFB_OK;
}

extern "C" int sfb_compute_factors_csr(sfb_ctx* ctx, int32_t worker, const int64_t* indptr_dev, const int32_t* indices_dev,
                                       const float* values_dev, int64_t nnz, const int32_t* labels_dev) {
  return compute_factors_csr(ctx, worker, indptr_dev, indices_dev, values_dev, nnz, labels_dev, false);
}

extern "C" int sfb_step_csr(sfb_ctx* ctx, const int64_t* indptr_dev, const int32_t* indices_dev, const float* values_dev,
                            int64_t nnz, const int32_t* labels_dev) {
  if (!ctx) return SFB_ERR_ARG;
  ctx->committed = 0;
  int rc = compute_factors_csr(ctx, -1, indptr_dev, indices_dev, values_dev, nnz, labels_dev, true);
  if (rc) return rc;
  rc = sfb_gather_factors(ctx);
  if (rc) return rc;
  return sfb_apply_update(ctx);
}

// ---------------------------------------------------------------------------------------------------------
// Row-sharded MLR: the parameter matrix partitioned by rows over several contexts (one per GPU)
// ---------------------------------------------------------------------------------------------------------
extern "C" int sfb_set_row_shard(sfb_ctx* ctx, int64_t row_offset, int64_t global_rows) {
  if (!ctx) return SFB_ERR_ARG;
  if ((ctx->cfg.model != SFB_MLR && ctx->cfg.model != SFB_DML) || ctx->sdca) return SFB_ERR_UNSUPPORTED;
  if (row_offset < 0 || global_rows < row_offset + ctx->cfg.rows || global_rows > (1LL << 31) - 1) return SFB_ERR_SHAPE;
  if (ctx->committed != 0 || ctx->partials_ready) return SFB_ERR_STATE;
  ctx->row_offset = row_offset;
  ctx->global_rows = global_rows;
  return SFB_OK;
}

extern "C" int sfb_forward_partials(sfb_ctx* ctx, const float* X_dev, const int32_t* labels_dev, float* partials_dev) {
  int rc = check_inputs(ctx, X_dev, nullptr, labels_dev);
  if (rc) return rc;
  if (ctx->cfg.model != SFB_MLR || ctx->sdca) return SFB_ERR_UNSUPPORTED;
  if (!partials_dev) return SFB_ERR_ARG;
  if (!al16(partials_dev)) return SFB_ERR_ALIGN;
  const sfb_config& c = ctx->cfg;
  ctx->committed = 0;
  ctx->sparse_mask = ctx->fma_mask = 0;
  ctx->csr_fill = 0;
  ctx->gathered = false;
  begin_phase(ctx, 0);
  if (c.precision == SFB_PREC_BF16 || ctx->tf32) {
    rc = ctx->tf32 ? tc32_forward_partials(ctx, X_dev, labels_dev, partials_dev)
                   : tc_forward_partials(ctx, X_dev, labels_dev, partials_dev);
    if (rc) return rc;
  } else {
    const int64_t K = ctx->K, ldu = ctx->lay.ldu;
    float* U = ctx->at<float>(ctx->lay.U);
    if ((rc = begin_step(ctx)) != SFB_OK || (rc = logits_fp32(ctx, 0, K, X_dev, nullptr, ctx->h16)) != SFB_OK) return rc;    // z_i = W_shard x_i
    // the class ids are kept for the finish (the caller's buffer may change before it)
    CK(cudaMemcpyAsync(ctx->at<int32_t>(ctx->lay.stageL), labels_dev, static_cast<size_t>(K) * 4, cudaMemcpyDeviceToDevice,
                       ctx->stream));
    CK(mlr_shard_partials(ctx->stream, U, K, c.rows, ldu, ctx->at<int32_t>(ctx->lay.stageL), ctx->row_offset,
                          partials_dev));
  }
  ctx->partials_ready = true;
  return SFB_OK;
}

// DML by rows: z = W v splits over the shards, the hinge needs ||z||^2 = sum over the shards of ||z_shard||^2.
extern "C" int sfb_forward_partials_pairs(sfb_ctx* ctx, const float* X_dev, const float* Y_dev, const int32_t* similar_dev,
                                          float* partials_dev) {
  int rc = check_inputs(ctx, X_dev, Y_dev, similar_dev);
  if (rc) return rc;
  if (ctx->cfg.model != SFB_DML) return SFB_ERR_UNSUPPORTED;
  if (!partials_dev) return SFB_ERR_ARG;
  const sfb_config& c = ctx->cfg;
  ctx->committed = 0;
  ctx->sparse_mask = ctx->fma_mask = 0;
  ctx->csr_fill = 0;
  ctx->gathered = false;
  begin_phase(ctx, 0);
  // the flags are kept for the finish (the caller's buffer may change before it)
  CK(cudaMemcpyAsync(ctx->at<int32_t>(ctx->lay.stageL), similar_dev, static_cast<size_t>(ctx->K) * 4, cudaMemcpyDeviceToDevice,
                     ctx->stream));
  if ((rc = begin_step(ctx)) != SFB_OK) return rc;
  rc = c.precision == SFB_PREC_FP32 ? factors_fp32(ctx, 0, ctx->K, X_dev, Y_dev, similar_dev, ctx->h16, false, partials_dev)
                                    : tc_factors(ctx, 0, ctx->K, X_dev, Y_dev, similar_dev, false, partials_dev);
  if (rc) return rc;
  ctx->partials_ready = true;
  return SFB_OK;
}

extern "C" int sfb_finish_factors(sfb_ctx* ctx, const float* partials_all_dev, int32_t shards) {
  if (!ctx || !partials_all_dev) return SFB_ERR_ARG;
  if (ctx->cfg.model != SFB_MLR && ctx->cfg.model != SFB_DML) return SFB_ERR_UNSUPPORTED;
  if (shards < 1 || shards > 4096) return SFB_ERR_ARG;
  if (!al16(partials_all_dev)) return SFB_ERR_ALIGN;
  if (!ctx->partials_ready) return SFB_ERR_STATE;
  const sfb_config& c = ctx->cfg;
  if (c.model == SFB_DML) {
    const int64_t ldu = ctx->lay.ldu;
    CK(dml_scale_rows(ctx->stream, ctx->at<float>(ctx->lay.U), ctx->K, c.rows, ldu, ctx->at<int32_t>(ctx->lay.stageL),
                      c.dml_margin, c.precision == SFB_PREC_BF16 ? ctx->at<char>(ctx->lay.Rs) : nullptr, ctx->lay.rowsp,
                      ctx->h16 ? ctx->at<float>(ctx->lay.iA) : nullptr, ctx->h16 ? ctx->at<float>(ctx->lay.q) : nullptr, nullptr,
                      partials_all_dev, shards, ctx->K));
    ctx->partials_ready = false;
    ctx->committed = c.workers == 64 ? ~0ull : ((1ull << c.workers) - 1);
    ctx->gathered = false;
    return SFB_OK;
  }
  if (c.precision == SFB_PREC_BF16 || ctx->tf32) {
    const int rc = ctx->tf32 ? tc32_finish_factors(ctx, partials_all_dev, shards)
                             : tc_finish_factors(ctx, partials_all_dev, shards);
    if (rc) return rc;
  } else {
    CK(mlr_shard_finish(ctx->stream, ctx->at<float>(ctx->lay.U), ctx->K, c.rows, ctx->lay.ldu, ctx->at<int32_t>(ctx->lay.stageL),
                        ctx->row_offset, partials_all_dev, shards, ctx->at<float>(ctx->lay.loss),
                        ctx->at<uint32_t>(ctx->lay.status)));
  }
  ctx->partials_ready = false;
  ctx->committed = c.workers == 64 ? ~0ull : ((1ull << c.workers) - 1);
  ctx->gathered = false;
  return SFB_OK;
}

// Sufficient factors computed elsewhere (another replica, another machine) take the place of a worker's own:
// the receiving side of the broadcast of Section 3.
extern "C" int sfb_set_factors(sfb_ctx* ctx, int32_t worker, const float* U_dev, const float* V_dev) {
  if (!ctx || !U_dev || !V_dev) return SFB_ERR_ARG;
  const sfb_config& c = ctx->cfg;
  if (worker < 0 || worker >= c.workers) return SFB_ERR_SHAPE;
  if (ctx->sdca) return SFB_ERR_UNSUPPORTED;
  if (ctx->partials_ready) return SFB_ERR_STATE;
  if (ctx->committed == 0) begin_phase(ctx, 0);
  const int64_t off = static_cast<int64_t>(worker) * c.batch;
  if (c.precision == SFB_PREC_BF16 && c.model == SFB_MLR) {
    const int rc = tc_import_factors(ctx, off, c.batch, U_dev, V_dev);
    if (rc) return rc;
    ctx->committed |= 1ull << worker;
    ctx->sparse_mask &= ~(1ull << worker);
    ctx->gathered = false;
    return SFB_OK;
  }
  const int64_t ldu = ctx->lay.ldu;
  float* U = ctx->at<float>(ctx->lay.U) + off * ldu;
  float* V = ctx->at<float>(ctx->lay.V) + off * c.cols;
  CK(cudaMemcpy2DAsync(U, static_cast<size_t>(ldu) * 4, U_dev, static_cast<size_t>(c.rows) * 4, static_cast<size_t>(c.rows) * 4,
                       static_cast<size_t>(c.batch), cudaMemcpyDeviceToDevice, ctx->stream));
  CK(cudaMemcpyAsync(V, V_dev, static_cast<size_t>(c.batch) * c.cols * 4, cudaMemcpyDeviceToDevice, ctx->stream));
  if (c.precision == SFB_PREC_BF16 || ctx->h16) {
    const int rc = split_pack_received(ctx, off, c.batch);
    if (rc) return rc;
  }
  ctx->committed |= 1ull << worker;
  ctx->sparse_mask &= ~(1ull << worker);             // received factors are dense
  ctx->fma_mask &= ~(1ull << worker);
  ctx->gathered = false;
  return SFB_OK;
}

extern "C" int sfb_export_factors(sfb_ctx* ctx, int32_t worker, float* U_out_dev, float* V_out_dev) {
  if (!ctx || !U_out_dev || !V_out_dev) return SFB_ERR_ARG;
  const sfb_config& c = ctx->cfg;
  if (worker < 0 || worker >= c.workers) return SFB_ERR_SHAPE;
  if (ctx->sdca) return SFB_ERR_UNSUPPORTED;
  if (!(ctx->committed & (1ull << worker))) return SFB_ERR_STATE;
  const int64_t off = static_cast<int64_t>(worker) * c.batch;
  if (c.precision == SFB_PREC_BF16 && c.model == SFB_MLR) return tc_export_factors(ctx, off, c.batch, U_out_dev, V_out_dev);
  const int64_t ldu = ctx->lay.ldu;
  CK(cudaMemcpy2DAsync(U_out_dev, static_cast<size_t>(c.rows) * 4, ctx->at<float>(ctx->lay.U) + off * ldu,
                       static_cast<size_t>(ldu) * 4, static_cast<size_t>(c.rows) * 4, static_cast<size_t>(c.batch),
                       cudaMemcpyDeviceToDevice, ctx->stream));
  CK(cudaMemcpyAsync(V_out_dev, ctx->at<float>(ctx->lay.V) + off * c.cols, static_cast<size_t>(c.batch) * c.cols * 4,
                     cudaMemcpyDeviceToDevice, ctx->stream));
  return SFB_OK;
}

extern "C" int sfb_set_eta(sfb_ctx* ctx, float eta) {
  if (!ctx || !(eta >= 0.f)) return SFB_ERR_ARG;
  if (ctx->committed != 0 || ctx->partials_ready) return SFB_ERR_STATE;       // not between the factors and their update
  ctx->cfg.eta = eta;
  ctx->step = ctx->sdca ? static_cast<float>(static_cast<double>(eta) / (static_cast<double>(ctx->cfg.sdca_lambda) *
                                                                        static_cast<double>(ctx->cfg.sdca_n)))
                        : eta;
  ctx->prox_a = ctx->prox_kind == 1 ? eta * ctx->cfg.prox_weight
              : ctx->prox_kind == 2 ? static_cast<float>(1.0 / (1.0 + static_cast<double>(eta) * ctx->cfg.prox_weight)) : 0.f;
  return SFB_OK;
}

extern "C" int sfb_gather_factors(sfb_ctx* ctx) {
  if (!ctx) return SFB_ERR_ARG;
  const sfb_config& c = ctx->cfg;
  const uint64_t all = c.workers == 64 ? ~0ull : ((1ull << c.workers) - 1);
  if (ctx->committed != all) return SFB_ERR_STATE;
  begin_phase(ctx, 1);
  // Every worker wrote its pairs at row offset p*B of the shared buffers, so the gathered operands are
  // complete; what remains is the per-step read-out over all K pairs.
  // all K samples sparse: the v become their column-major form (and the dense update operands are not needed)
  ctx->update_fma = ctx->fma_mask != 0;
  ctx->sparse_v = c.model == SFB_MLR && c.csr_nnz_max > 0 && ctx->sparse_mask == all && sparse_update_wanted(ctx);
  if (ctx->sparse_v) {
    CK(stamp(ctx->stream, take_stamp(ctx)));
    int rc = sparse_build_csc(ctx);
    if (rc) return rc;
  } else if (ctx->tf32) {
    CK(stamp(ctx->stream, take_stamp(ctx)));
    int rc = tc32_gather(ctx);
    if (rc) return rc;
  } else if (ctx->h16 && !ctx->update_fma) {
    const int rc = split_gather(ctx);
    if (rc) return rc;
  }
  if (c.model == SFB_MLR && c.precision == SFB_PREC_FP32) {        // (bf16 mode: with the label rows)
    CK(mean_of(ctx->stream, ctx->at<float>(ctx->lay.loss), ctx->K,
               &ctx->at<Scalars>(ctx->lay.scalars)->loss_mean, take_stamp(ctx)));
  }
  // bytes per gathered value: fp32, bf16, or a (hi, lo) pair of bf16 for the split operands of DML and SC
  const double esz = (c.precision == SFB_PREC_FP32 || c.model != SFB_MLR) ? 4.0 : 2.0;
  // sparse v: 8 bytes (index, value) per non-zero instead of cols values per sample
  const double pair = ctx->sparse_v ? static_cast<double>(c.rows) * esz + 8.0 * static_cast<double>(ctx->csr_fill) / ctx->K
                                    : static_cast<double>(c.rows + c.cols) * esz;
  ctx->stats.gather_bytes += static_cast<double>(ctx->K) * pair;
  ctx->stats.gather_bytes_p2p += static_cast<double>(c.workers) * (c.workers - 1) * c.batch * pair;
  ctx->stats.dense_sync_bytes += static_cast<double>(c.workers) * c.rows * c.cols * 4.0;
  ctx->gathered = true;
  begin_phase(ctx, 2);
  return SFB_OK;
}

static int apply_prox(sfb_ctx* ctx) {
  const sfb_config& c = ctx->cfg;
  if (c.model == SFB_SC && c.sc_prox == 1)
    CK(prox_unit_columns(ctx->stream, ctx->W, c.rows, c.cols, ctx->at<float>(ctx->lay.colpart),
                         &ctx->at<Scalars>(ctx->lay.scalars)->ns[3]));
  return SFB_OK;
}

extern "C" int sfb_apply_update(sfb_ctx* ctx) {
  if (!ctx) return SFB_ERR_ARG;
  if (!ctx->gathered) return SFB_ERR_STATE;
  const sfb_config& c = ctx->cfg;
  int rc = ctx->tf32 ? tc32_update(ctx) : c.precision == SFB_PREC_FP32 ? update_fp32(ctx) : tc_update(ctx);
  if (rc) return rc;
  ctx->stats.flops += 2.0 * c.rows * c.cols * ctx->K;
  rc = apply_prox(ctx);
  if (rc) return rc;
  ctx->committed = 0;
  ctx->begun = false;
  ctx->sparse_mask = ctx->fma_mask = 0;               // the next step starts with no sparse samples staged
  ctx->csr_fill = 0;
  ctx->gathered = false;
  ctx->stats.steps += 1;
  ctx->stats.samples += ctx->K;
  if (ctx->sparse_v) ctx->stats.sparse_updates += 1;
  return SFB_OK;
}

// ---------------------------------------------------------------------------------------------------------
// l2-regularised MLR by stochastic dual coordinate ascent
// ---------------------------------------------------------------------------------------------------------
extern "C" int sfb_sdca_set_dual(sfb_ctx* ctx, float* Q_dev, int64_t n_samples) {
  if (!ctx || !Q_dev) return SFB_ERR_ARG;
  if (!ctx->sdca) return SFB_ERR_UNSUPPORTED;
  if (n_samples != ctx->cfg.sdca_n) return SFB_ERR_SHAPE;
  if (!al16(Q_dev)) return SFB_ERR_ALIGN;
  ctx->dualQ = Q_dev;
  ctx->dual_n = n_samples;
  return SFB_OK;
}

namespace sfb {
SdcaArgs sdca_args(const sfb_ctx* ctx, int64_t off, int64_t n, const float* X, const int32_t* labels, const int32_t* ids,
                   float inv_lam_n) {
  SdcaArgs a{};
  a.n = n; a.rows = ctx->cfg.rows; a.X = X; a.cols = ctx->cfg.cols; a.labels = labels; a.ids = ids;
  a.Q = ctx->dualQ; a.n_samples = ctx->dual_n; a.inv_lam_n = inv_lam_n; a.gamma = ctx->cfg.eta;
  a.loss = ctx->at<float>(ctx->lay.loss) + off; a.status = ctx->at<uint32_t>(ctx->lay.status); a.off = off;
  return a;
}
}  // namespace sfb

static int sdca_compute_factors(sfb_ctx* ctx, int32_t worker, const float* X_dev, const int32_t* labels_dev,
                                const int32_t* sample_ids_dev, bool fused) {
  if (!ctx || !X_dev || !labels_dev || !sample_ids_dev) return SFB_ERR_ARG;
  if (!ctx->sdca) return SFB_ERR_UNSUPPORTED;
  if (!ctx->dualQ) return SFB_ERR_STATE;
  if (!al16(X_dev)) return SFB_ERR_ALIGN;
  const sfb_config& c = ctx->cfg;
  if (worker < -1 || worker >= c.workers) return SFB_ERR_SHAPE;
  const int64_t off = worker < 0 ? 0 : static_cast<int64_t>(worker) * c.batch;
  const int64_t n = worker < 0 ? ctx->K : c.batch;
  if (ctx->committed == 0) begin_phase(ctx, 0);
  if (starts_over(ctx, worker)) ctx->begun = false;
  const float inv_lam_n = static_cast<float>(1.0 / (static_cast<double>(c.sdca_lambda) * static_cast<double>(c.sdca_n)));
  if (ctx->tf32) {
    const int rc = tc32_factors(ctx, off, n, X_dev, labels_dev, sample_ids_dev, inv_lam_n);
    if (rc) return rc;
  } else if (c.precision == SFB_PREC_FP32) {
    const int64_t ldu = ctx->lay.ldu;
    float* U = ctx->at<float>(ctx->lay.U) + off * ldu;
    if (!ctx->begun) {
      const int rc = begin_step(ctx);
      if (rc) return rc;
      ctx->begun = true;
    }
    const int rc = logits_fp32(ctx, off, n, X_dev, nullptr, ctx->h16);                                       // z_i = W a_i
    if (rc) return rc;
    SdcaArgs a = sdca_args(ctx, off, n, X_dev, labels_dev, sample_ids_dev, inv_lam_n);
    a.Z = U; a.ldz = ldu; a.out = U; a.ldo = ldu;                                                     // u_i = du_i
    CK(sdca_dual_rows(ctx->stream, a));
  } else {
    const int rc = tc_sdca_factors(ctx, off, n, X_dev, labels_dev, sample_ids_dev, inv_lam_n, fused);
    if (rc) return rc;
  }
  const uint64_t all = c.workers == 64 ? ~0ull : ((1ull << c.workers) - 1);
  ctx->committed |= worker < 0 ? all : (1ull << worker);
  ctx->gathered = false;
  return SFB_OK;
}

extern "C" int sfb_sdca_compute_factors(sfb_ctx* ctx, int32_t worker, const float* X_dev, const int32_t* labels_dev,
                                        const int32_t* sample_ids_dev) {
  return sdca_compute_factors(ctx, worker, X_dev, labels_dev, sample_ids_dev, false);
}

extern "C" int sfb_sdca_step(sfb_ctx* ctx, const float* X_dev, const int32_t* labels_dev, const int32_t* sample_ids_dev) {
  if (!ctx) return SFB_ERR_ARG;
  ctx->committed = 0;
  int rc = sdca_compute_factors(ctx, -1, X_dev, labels_dev, sample_ids_dev, true);
  if (rc) return rc;
  rc = sfb_gather_factors(ctx);
  if (rc) return rc;
  return sfb_apply_update(ctx);
}

extern "C" int sfb_refresh_operands(sfb_ctx* ctx) {
  if (!ctx) return SFB_ERR_ARG;
  if (ctx->committed != 0 || ctx->partials_ready) return SFB_ERR_STATE;      // not in the middle of a step
  if (ctx->cfg.precision != SFB_PREC_BF16 && !ctx->tf32) return SFB_OK;       // the FFMA kernels read W itself
  return tc_refresh_operands(ctx);
}

extern "C" int sfb_replay_update(sfb_ctx* ctx) {
  if (!ctx) return SFB_ERR_ARG;
  if (ctx->stats.steps < 1 || ctx->committed != 0 || ctx->partials_ready) return SFB_ERR_STATE;
  const sfb_config& c = ctx->cfg;
  begin_phase(ctx, 2);
  int rc = ctx->tf32 ? tc32_update(ctx) : c.precision == SFB_PREC_FP32 ? update_fp32(ctx) : tc_update(ctx);
  if (rc) return rc;
  ctx->stats.flops += 2.0 * c.rows * c.cols * ctx->K;
  rc = apply_prox(ctx);
  if (rc) return rc;
  return SFB_OK;
}

extern "C" int sfb_step(sfb_ctx* ctx, const float* X_dev, const float* Y_dev, const int32_t* labels_dev) {
  if (!ctx) return SFB_ERR_ARG;
  ctx->committed = 0;
  int rc = compute_factors(ctx, -1, X_dev, Y_dev, labels_dev, true);
  if (rc) return rc;
  rc = sfb_gather_factors(ctx);
  if (rc) return rc;
  return sfb_apply_update(ctx);
}

// The copies in, the step and the copy of what is read back, all enqueued.
static int enqueue_host_step(sfb_ctx* ctx, const float* X_host, const float* Y_host, const int32_t* labels_host) {
  const sfb_config& c = ctx->cfg;
  HostSide& h = *ctx->host;
  float* Xs = ctx->at<float>(ctx->lay.stageX);
  float* Ys = ctx->at<float>(ctx->lay.stageY);
  int32_t* Ls = ctx->at<int32_t>(ctx->lay.stageL);
  // MLR in bf16 mode: the logits of a part of the samples are formed while the next part is copied (20,000 x 4,000, K = 512: the
  // copy's 178 us in line with the step's 330 before).
  const int parts = c.precision == SFB_PREC_BF16 ? tc_host_parts(ctx) : 1;
  const size_t bytes = static_cast<size_t>(ctx->K) * ctx->in_dim * 4;
  if (parts > 1) {
    CK(cudaEventRecord(h.ahead, ctx->stream));           // what the stream still reads of the staging buffer
    CK(cudaStreamWaitEvent(h.copies, h.ahead, 0));
    for (int i = 0; i < parts; ++i) {
      CK(cudaMemcpyAsync(reinterpret_cast<char*>(Xs) + i * (bytes / parts), reinterpret_cast<const char*>(X_host) + i * (bytes / parts),
                         bytes / parts, cudaMemcpyHostToDevice, h.copies));
      CK(cudaEventRecord(h.part[i], h.copies));
    }
  } else {
    CK(cudaMemcpyAsync(Xs, X_host, bytes, cudaMemcpyHostToDevice, ctx->stream));
  }
  if (c.model == SFB_DML)
    CK(cudaMemcpyAsync(Ys, Y_host, static_cast<size_t>(ctx->K) * c.cols * 4, cudaMemcpyHostToDevice, ctx->stream));
  if (c.model != SFB_SC)
    CK(cudaMemcpyAsync(Ls, labels_host, static_cast<size_t>(ctx->K) * 4, cudaMemcpyHostToDevice, ctx->stream));
  h.parts = parts;
  const int rc = sfb_step(ctx, Xs, c.model == SFB_DML ? Ys : nullptr, c.model != SFB_SC ? Ls : nullptr);
  h.parts = 0;
  if (rc) return rc;
  // status word and scalars lie side by side: one copy, to page-locked memory
  CK(cudaMemcpyAsync(h.back, ctx->at<char>(ctx->lay.status), ctx->lay.loss - ctx->lay.status, cudaMemcpyDeviceToHost, ctx->stream));
  return SFB_OK;
}

extern "C" int sfb_step_host(sfb_ctx* ctx, const float* X_host, const float* Y_host, const int32_t* labels_host,
                             float* loss_out, uint32_t* status_out) {
  if (!ctx || !X_host) return SFB_ERR_ARG;
  if (ctx->sdca) return SFB_ERR_UNSUPPORTED;
  const sfb_config& c = ctx->cfg;
  if (c.model == SFB_DML && (!Y_host || !labels_host)) return SFB_ERR_ARG;
  if (c.model == SFB_MLR && !labels_host) return SFB_ERR_ARG;
  if (!ctx->host) CK(make_host_side(ctx));
  HostSide& h = *ctx->host;
  const int rc = enqueue_host_step(ctx, X_host, Y_host, labels_host);
  if (rc) {                                              // whatever failed: the caller's buffers are not read after the return
    cudaStreamSynchronize(h.copies);
    cudaStreamSynchronize(ctx->stream);
    return rc;
  }
  CK(cudaStreamSynchronize(ctx->stream));
  const Scalars* sc = reinterpret_cast<const Scalars*>(h.back + (ctx->lay.scalars - ctx->lay.status));
  if (loss_out) *loss_out = sc->loss_mean;
  if (status_out) *status_out = *reinterpret_cast<const uint32_t*>(h.back);
  return SFB_OK;
}

extern "C" int sfb_dense_sync_step(sfb_ctx* ctx, const float* X_dev, const float* Y_dev, const int32_t* labels_dev,
                                   float* scratch_dev, size_t scratch_bytes) {
  if (!ctx || !scratch_dev) return SFB_ERR_ARG;
  const sfb_config& c = ctx->cfg;
  if (c.precision != SFB_PREC_FP32) return SFB_ERR_UNSUPPORTED;
  if (!al16(scratch_dev)) return SFB_ERR_ALIGN;
  const size_t mat = static_cast<size_t>(c.rows) * c.cols;
  if (scratch_bytes < 2 * mat * 4) return SFB_ERR_WORKSPACE;
  ctx->committed = 0;
  int rc = sfb_compute_factors(ctx, -1, X_dev, Y_dev, labels_dev);
  if (rc) return rc;
  rc = sfb_gather_factors(ctx);   // loss read-out and byte accounting; the factors stay per worker below
  if (rc) return rc;
  float* sum = scratch_dev;
  float* one = scratch_dev + mat;
  const float* U = ctx->at<float>(ctx->lay.U);
  const float* V = ctx->at<float>(ctx->lay.V);
  CK(stamp(ctx->stream, take_stamp(ctx)));
  for (int p = 0; p < c.workers; ++p) {
    // worker p's dense update matrix, as it would be sent to the server
    EpiArgs e{};
    e.C = p == 0 ? sum : one; e.ldc = c.cols;
    CK(sgemm(ctx->stream, false, false, EPI_STORE, c.rows, c.cols, c.batch, U + static_cast<int64_t>(p) * c.batch * ctx->lay.ldu,
             ctx->lay.ldu, V + static_cast<int64_t>(p) * c.batch * c.cols, c.cols, e));
    if (p > 0) CK(axpy(ctx->stream, sum, one, 1.f, static_cast<int64_t>(mat)));          // server-side aggregation
  }
  CK(axpy(ctx->stream, ctx->W, sum, -c.eta, static_cast<int64_t>(mat)));                 // W <- W - eta * sum_p dW_p
  CK(prox_entries(ctx->stream, ctx->W, static_cast<int64_t>(mat), ctx->prox_kind, ctx->prox_a));
  CK(stamp(ctx->stream, Stamp{&ctx->at<Scalars>(ctx->lay.scalars)->ns[3], 1}));
  ctx->stats.flops += 2.0 * c.rows * c.cols * ctx->K;
  rc = apply_prox(ctx);
  if (rc) return rc;
  ctx->committed = 0;
  ctx->begun = false;
  ctx->gathered = false;
  ctx->stats.steps += 1;
  ctx->stats.samples += ctx->K;
  return SFB_OK;
}

extern "C" int sfb_get_factors(sfb_ctx* ctx, const void** U_dev, const void** V_dev, int32_t* dtype, int32_t* layout,
                               int64_t* ldu, int64_t* ldv) {
  if (!ctx) return SFB_ERR_ARG;
  if (ctx->cfg.precision == SFB_PREC_FP32) {
    if (U_dev) *U_dev = ctx->at<float>(ctx->lay.U);
    if (V_dev) *V_dev = ctx->at<float>(ctx->lay.V);
    if (dtype) *dtype = 0;
    if (layout) *layout = 0;
    if (ldu) *ldu = ctx->lay.ldu;
    if (ldv) *ldv = ctx->cfg.cols;
    return SFB_OK;
  }
  return tc_get_factors(ctx, U_dev, V_dev, dtype, layout, ldu, ldv);
}

extern "C" int sfb_get_operand_copy(sfb_ctx* ctx, const void** copy_dev, int32_t* dtype, int64_t* ld) {
  if (!ctx || !copy_dev) return SFB_ERR_ARG;
  if (ctx->cfg.model != SFB_MLR) return SFB_ERR_UNSUPPORTED;
  if (ctx->tf32) {
    *copy_dev = ctx->at<float>(ctx->lay.Ws);
    if (dtype) *dtype = 2;
    if (ld) *ld = 2 * ctx->lay.colsp;
    return SFB_OK;
  }
  if (ctx->cfg.precision != SFB_PREC_BF16) return SFB_ERR_UNSUPPORTED;
  *copy_dev = ctx->at<char>(ctx->lay.Wb);
  if (dtype) *dtype = 1;
  if (ld) *ld = ctx->lay.colsb;
  return SFB_OK;
}

extern "C" int sfb_get_update_form(sfb_ctx* ctx, int32_t* form) {
  if (!ctx || !form) return SFB_ERR_ARG;
  if (ctx->stats.gather_bytes == 0.0) return SFB_ERR_STATE;
  const sfb_config& c = ctx->cfg;
  *form = ctx->sparse_v ? 5 : ctx->tf32 ? 4 : c.precision == SFB_PREC_BF16 ? (c.model == SFB_MLR ? 1 : 2) : ctx->h16 && !ctx->update_fma ? 3 : 0;
  return SFB_OK;
}

extern "C" int sfb_get_plan(const sfb_config* cfg, int64_t samples, int32_t* product, int32_t* parts, int32_t* merged) {
  const int rc = check_config(cfg);
  if (rc) return rc;
  if (!product || !parts || !merged) return SFB_ERR_ARG;
  sfb_config c = *cfg;
  if (samples < 1 || samples > static_cast<int64_t>(c.workers) * c.batch) return SFB_ERR_SHAPE;
  if (c.model == SFB_L2MLR) c.model = SFB_MLR;
  int form = 0, cut = 1;
  bool one = false;
  if (use_tf32(c)) {
    form = 4;
  } else if (c.model == SFB_SC && !use_h16(c) && c.precision != SFB_PREC_BF16) {
    form = sc_use_gram64(c) ? 7 : 0;
  } else if (c.model == SFB_SC) {
    form = sc_use_gram(c) ? 6 : 5;
    cut = split_product_parts(samples, form == 6 ? c.cols : c.rows, c.cols, c.precision != SFB_PREC_BF16);
  } else if (use_h16(c) || (c.precision == SFB_PREC_BF16 && c.model == SFB_DML)) {
    form = 5;
    cut = split_product_parts(samples, c.rows, c.cols, false);
  } else if (c.precision == SFB_PREC_BF16) {
    const bool step = samples == static_cast<int64_t>(c.workers) * c.batch;
    form = tc_logits_plan(c, make_layout(*cfg), samples, step, &cut, &one);
    one = one && step && cfg->model == SFB_MLR;
  }
  *product = form;
  *parts = cut;
  *merged = one;
  return SFB_OK;
}

extern "C" int sfb_get_stats(sfb_ctx* ctx, sfb_stats* out) {
  if (!ctx || !out) return SFB_ERR_ARG;
  const sfb_config& c = ctx->cfg;
  // MLR in bf16 mode forms the mean loss with the label rows, in the update: asked for after the gather already, here
  if (ctx->gathered && c.model == SFB_MLR && c.precision == SFB_PREC_BF16 && ctx->labels == sfb_ctx::kLabelsNone)
    CK(mean_of(ctx->stream, ctx->at<float>(ctx->lay.loss), ctx->K, &ctx->at<Scalars>(ctx->lay.scalars)->loss_mean, Stamp{}));
  CK(cudaStreamSynchronize(ctx->stream));
  if (ctx->stats.steps > 0) {
    Scalars h{};
    CK(cudaMemcpy(&h, ctx->at<Scalars>(ctx->lay.scalars), sizeof(h), cudaMemcpyDeviceToHost));
    auto ms = [&](int from, int to) { return h.ns[to] > h.ns[from] ? static_cast<float>(h.ns[to] - h.ns[from]) * 1e-6f : 0.f; };
    ctx->stats.ms_factors = ms(0, 1);
    ctx->stats.ms_gather = ms(1, 2);
    ctx->stats.ms_update = ms(2, 3);
    ctx->stats.last_loss = h.loss_mean;
    ctx->stats.sc_lipschitz = h.L;
    ctx->stats.copy_pieces = static_cast<int64_t>(h.copy_pieces);
    ctx->stats.copy_written = static_cast<int64_t>(h.copy_written);
  }
  ctx->stats.kernel_launches = g_kernel_launches.load(std::memory_order_relaxed);
  *out = ctx->stats;
  return SFB_OK;
}

extern "C" int sfb_get_status(sfb_ctx* ctx, uint32_t* status_out) {
  if (!ctx || !status_out) return SFB_ERR_ARG;
  CK(cudaMemcpyAsync(status_out, ctx->at<uint32_t>(ctx->lay.status), 4, cudaMemcpyDeviceToHost, ctx->stream));
  CK(cudaMemsetAsync(ctx->at<uint32_t>(ctx->lay.status), 0, 4, ctx->stream));
  CK(cudaStreamSynchronize(ctx->stream));
  if ((*status_out & SFB_STATUS_TIMEOUT) && ctx->lay.ready) CK(split_reset(ctx));
  return SFB_OK;
}

extern "C" int sfb_last_cuda_error(sfb_ctx* ctx) { return ctx ? ctx->last_cuda : 0; }

extern "C" const char* sfb_strerror(int code) {
  switch (code) {
    case SFB_OK: return "ok";
    case SFB_ERR_ARG: return "invalid argument";
    case SFB_ERR_ALIGN: return "pointer not 16-byte aligned";
    case SFB_ERR_SHAPE: return "unsupported shape";
    case SFB_ERR_WORKSPACE: return "workspace or scratch too small";
    case SFB_ERR_CUDA: return "CUDA runtime error";
    case SFB_ERR_ARCH: return "device is not compute capability 10.x";
    case SFB_ERR_TIMEOUT: return "a bounded device-side wait gave up";
    case SFB_ERR_LABEL_RANGE: return "class id out of range";
    case SFB_ERR_STATE: return "call out of order";
    case SFB_ERR_UNSUPPORTED: return "model/precision combination not built";
    case SFB_ERR_STATIC_LIMIT: return "size beyond the library's built-in scratch array";
    default: return "unknown error";
  }
}
