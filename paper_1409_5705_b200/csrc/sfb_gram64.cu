// The sparse coder of the fp32 mode on W^T W:  a <- soft(a - (W^T W a - W^T x) / L)  in fp64 (see sc_use_gram64).
//
// Why fp64: the two products of an iteration become one of half the size or less, but W^T W a and W^T x cancel, so an error of
// 2^-24 of either is one of the gradient, where W^T (W a - x) has it relative to the residual.  In fp32 the codes were 2 to 8 times
// further from the exact iterates than with two products (2,232 x 616, 20 iterations, x in the span of 20 atoms: 4e-7 against
// 1e-7).  In fp64 they are exact to the rounding of the result, and the chip has half its fp32 rate in fp64 (36 TFLOP/s measured).
//
// All operands lie with the contraction outermost (samples and codes transposed), so that a slice of either is a set of 16-byte
// pieces: D[n][m] = sum_k P[k][n] Q[k][m] with P = W or W^T W (n: atoms) and Q the samples or the codes (m: samples).  Eight warps
// per 64 x 64 tile, 32 x 16 each on the fp64 matrix instruction (with FMAs on 4 x 4 outputs a thread the loads from shared memory
// took twice the time of the arithmetic: W^T W of 2,000 x 1,000 140 us against 100, an iteration of 128 samples 24 against 19),
// four stages of 16 k by cp.async.  As in the fp32 products a contraction is cut over a cluster where the tiles leave SMs idle, the
// parts added in rank order.
#include <algorithm>

#include "sfb_internal.h"

namespace sfb {
namespace {

constexpr int NT = 256, BT = 64, BK = 16, STG = 4;
constexpr int PT = BT + 4;                            // row pitch in shared memory: four k of a fragment lie in different banks
constexpr int kSlice = BK * PT;                       // doubles per operand and stage
constexpr int kSmem = STG * 2 * kSlice * 8;
static_assert(kSmem >= BT * BT * 8, "the partial tile of a split contraction takes the ring's memory");

enum Epi { E_GRAM = 0, E_FIRST = 1, E_STEP = 2 };

struct Params {
  int32_t N, M, Kc, split;     // atoms; samples (E_GRAM: atoms); contraction; CTAs that share a tile's contraction
  const double* P;
  const double* Q;
  int64_t ldp, ldq;
  int32_t tilesN;
  double* out;                 // E_GRAM: [N x N]; else the new codes [N x ldq]
  const double* cur;           // E_STEP: the codes
  double* b;                   // W^T x: written by E_FIRST, read by E_STEP
  float* f32;                  // E_GRAM: the same in fp32 (or null)
  const Scalars* sc;
  double lam;
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void cp16(uint32_t dst, const double* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
// k [k0, kend) x columns [c0, width) of an operand into a stage [BK][PT]; the rest reads as zeros.  width is even.
__device__ __forceinline__ void load_slice(uint32_t dst, const double* p, int64_t ld, int k0, int kend, int c0, int width, int t) {
#pragma unroll
  for (int v = 0; v < BK * BT / 2 / NT; ++v) {
    const int idx = t + v * NT, k = idx / (BT / 2), c = (idx % (BT / 2)) * 2;
    const bool in = k0 + k < kend && c0 + c < width;
    cp16(dst + (k * PT + c) * 8, in ? p + static_cast<int64_t>(k0 + k) * ld + c0 + c : p, in ? 16 : 0);
  }
}

// acc (16 x 8) += a (16 x 8) b (8 x 8) in fp64.  Lane 4 g + q: a rows g, g + 8 of columns q, then of q + 4; b column g of rows q, q + 4;
// acc columns 2 q, 2 q + 1 of row g, then of g + 8.
__device__ __forceinline__ void mma(double (&acc)[4], const double (&a)[4], const double (&b)[2]) {
  asm("mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+d"(acc[0]), "+d"(acc[1]), "+d"(acc[2]), "+d"(acc[3])
      : "d"(a[0]), "d"(a[1]), "d"(a[2]), "d"(a[3]), "d"(b[0]), "d"(b[1]));
}

__device__ __forceinline__ double soft(double w, double t) {
  const double a = fabs(w) - t;
  return a > 0. ? copysign(a, w) : 0.;
}

// two neighbouring outputs of row n (m even)
template <int EPI>
__device__ __forceinline__ void finish2(const Params& p, int n, int m, double2 v, double invL, double thr, bool mirror) {
  if (n >= p.N || m >= p.M) return;
  if (EPI == E_GRAM) {                                  // (N is a multiple of 4)
    const int64_t at = static_cast<int64_t>(n) * p.N + m;
    *reinterpret_cast<double2*>(p.out + at) = v;
    if (p.f32) *reinterpret_cast<float2*>(p.f32 + at) = make_float2(static_cast<float>(v.x), static_cast<float>(v.y));
    if (mirror) {
      const int64_t to = static_cast<int64_t>(m) * p.N + n;
      p.out[to] = v.x;
      p.out[to + p.N] = v.y;
      if (p.f32) { p.f32[to] = static_cast<float>(v.x); p.f32[to + p.N] = static_cast<float>(v.y); }
    }
  } else {                                              // (the pitch is even: the last pair of an odd M has room)
    const int64_t at = static_cast<int64_t>(n) * p.ldq + m;
    if (EPI == E_FIRST) {
      *reinterpret_cast<double2*>(p.b + at) = v;
      v = make_double2(soft(v.x * invL, thr), soft(v.y * invL, thr));
    } else {
      const double2 c = *reinterpret_cast<const double2*>(p.cur + at), b = *reinterpret_cast<const double2*>(p.b + at);
      v = make_double2(soft(fma(b.x - v.x, invL, c.x), thr), soft(fma(b.y - v.y, invL, c.y), thr));
    }
    *reinterpret_cast<double2*>(p.out + at) = v;
  }
}

template <int EPI>
__global__ void __launch_bounds__(NT, 2) gram64_kernel(const __grid_constant__ Params p) {
  extern __shared__ __align__(16) double sm[];
  const int t = threadIdx.x;
  const int S = p.split, tile = blockIdx.x / S, part = blockIdx.x % S;
  const int n0 = (tile % p.tilesN) * BT, m0 = (tile / p.tilesN) * BT;
  pdl_launch_dependents();
  pdl_wait();
  if (EPI == E_GRAM && m0 < n0) return;                 // the mirror image of another tile: uniform over the cluster
  const int units = (p.Kc + BK - 1) / BK;
  const int kbeg = static_cast<int>(static_cast<int64_t>(part) * units / S) * BK;
  const int kend = min(p.Kc, static_cast<int>(static_cast<int64_t>(part + 1) * units / S) * BK);
  const int nkb = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;
  const uint32_t base = smem_addr(sm);
  const int widthQ = static_cast<int>(EPI == E_GRAM ? p.N : p.ldq);

  // warp w: rows 32 (w & 1) .., columns 16 (w >> 1) .. of the tile, as 2 x 2 fragments of 16 x 8
  const int lane = t & 31, g = lane >> 2, q = lane & 3, wr = (t >> 5 & 1) * 32, wc = (t >> 6) * 16;
  double acc[2][2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.;
  auto issue = [&](int kb) {
    if (kb < nkb) {
      const uint32_t st = base + (kb % STG) * (2 * kSlice * 8);
      load_slice(st, p.P, p.ldp, kbeg + kb * BK, kend, n0, p.N, t);
      load_slice(st + kSlice * 8, p.Q, p.ldq, kbeg + kb * BK, kend, m0, widthQ, t);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int s = 0; s < STG - 1; ++s) issue(s);
  for (int kb = 0; kb < nkb; ++kb) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STG - 2) : "memory");
    __syncthreads();                                    // stage kb has landed for everyone; stage kb - 1 is free
    issue(kb + STG - 1);
    const double* Ps = sm + (kb % STG) * (2 * kSlice) + q * PT + wr + g;
    const double* Qs = sm + (kb % STG) * (2 * kSlice) + kSlice + q * PT + wc + g;
#pragma unroll
    for (int k = 0; k < BK; k += 8) {
      double a[2][4], c[2][2];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) a[i][e] = Ps[(k + 4 * (e >> 1)) * PT + 16 * i + 8 * (e & 1)];
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) c[j][e] = Qs[(k + 4 * e) * PT + 8 * j];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) mma(acc[i][j], a[i], c[j]);
    }
  }
  double invL = 0., thr = 0.;
  if (EPI != E_GRAM) { invL = 1. / static_cast<double>(p.sc->L); thr = p.lam * invL; }
  const bool mirror = m0 > n0;
  auto each = [&](auto&& put) {                         // of this thread's pairs of outputs: row and column in the tile, values
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) put(wr + 16 * i + 8 * e + g, wc + 8 * j + 2 * q, make_double2(acc[i][j][2 * e], acc[i][j][2 * e + 1]));
  };
  if (S == 1) {
    each([&](int r, int c, double2 v) { finish2<EPI>(p, n0 + r, m0 + c, v, invL, thr, mirror); });
    return;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  each([&](int r, int c, double2 v) { *reinterpret_cast<double2*>(sm + r * BT + c) = v; });
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  const int rows_here = BT / S, rbeg = part * rows_here;
  for (int i = t; i < rows_here * (BT / 2); i += NT) {
    const int r = rbeg + i / (BT / 2), c = (i % (BT / 2)) * 2;
    double2 v = make_double2(0., 0.);
    const uint32_t own = smem_addr(sm + r * BT + c);
    for (int s = 0; s < S; ++s) {
      uint32_t peer;
      double2 w;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(own), "r"(s));
      asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(w.x), "=d"(w.y) : "r"(peer));
      v.x += w.x; v.y += w.y;
    }
    finish2<EPI>(p, n0 + r, m0 + c, v, invL, thr, mirror);
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");      // no CTA leaves while a peer still reads its tile
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __launch_bounds__(256) widen_kernel(const float* src, double* dst, int64_t n4) {
  pdl_launch_dependents();
  pdl_wait();
  const int64_t stride = static_cast<int64_t>(gridDim.x) * 256;
  for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < n4; i += stride) {
    const float4 v = reinterpret_cast<const float4*>(src)[i];
    reinterpret_cast<double2*>(dst)[2 * i] = make_double2(v.x, v.y);
    reinterpret_cast<double2*>(dst)[2 * i + 1] = make_double2(v.z, v.w);
  }
}

// dst[c][r] = src[r][c] for a rows x cols source, 32 x 32 tiles through shared memory; numbered along the rows first.
template <typename From, typename To>
__global__ void __launch_bounds__(256) transpose_kernel(const From* src, int64_t rows, int64_t cols, int64_t lds, To* dst, int64_t ldd) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ To tile[32][33];
  const int64_t blocks = (rows + 31) / 32, r0 = (blockIdx.x % blocks) * 32, c0 = (blockIdx.x / blocks) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
  for (int i = ty; i < 32; i += 8)
    if (r0 + i < rows && c0 + tx < cols) tile[i][tx] = static_cast<To>(src[(r0 + i) * lds + c0 + tx]);
  __syncthreads();
#pragma unroll
  for (int i = ty; i < 32; i += 8)
    if (c0 + i < cols && r0 + tx < rows) dst[(c0 + i) * ldd + r0 + tx] = tile[tx][i];
}
template <typename From, typename To>
cudaError_t transpose(cudaStream_t s, const From* src, int64_t rows, int64_t cols, int64_t lds, To* dst, int64_t ldd) {
  const int64_t blocks = ((rows + 31) / 32) * ((cols + 31) / 32);
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  return launch_kernel(transpose_kernel<From, To>, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, s, 1, src, rows, cols, lds, dst, ldd);
}

// SM cycles with the contraction in `split` parts: a pair of tiles on an SM takes 165 cycles per k (78 % of its fp64 rate), a tile
// alone 95; a part also fills its ring, and the parts are exchanged.
double cost_of(int64_t N, int64_t M, int64_t Kc, bool sym, int split) {
  const double tn = static_cast<double>((N + BT - 1) / BT), tm = static_cast<double>((M + BT - 1) / BT);
  const double tiles = (sym ? 0.5 * tn * (tn + 1.) : tn * tm) * split;
  const int64_t per_sm = static_cast<int64_t>((tiles + kModelSms - 1.) / kModelSms);
  const double pairs = static_cast<double>(per_sm / 2), single = static_cast<double>(per_sm % 2);
  return static_cast<double>(Kc) / split * (165. * pairs + 95. * single) + (pairs + single) * 3500. + (split > 1 ? 3000. : 0.) + 5000.;
}
int pick_split(int64_t N, int64_t M, int64_t Kc, bool sym) {
  int best = 1;
  for (int s = 2; s <= 8 && Kc >= 2 * BK * s; s *= 2)
    if (cost_of(N, M, Kc, sym, s) < 0.97 * cost_of(N, M, Kc, sym, best)) best = s;
  return best;
}

// samples: what the split is chosen for, whichever slice of them a call has
template <int EPI>
cudaError_t product(cudaStream_t s, Params p, int64_t samples) {
  p.split = pick_split(p.N, samples, p.Kc, EPI == E_GRAM);
  p.tilesN = (p.N + BT - 1) / BT;
  const int64_t tiles = static_cast<int64_t>(p.tilesN) * ((p.M + BT - 1) / BT) * p.split;
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  const cudaError_t e = allow_smem<gram64_kernel<EPI>>(kSmem);
  if (e != cudaSuccess) return e;
  return launch_kernel(gram64_kernel<EPI>, dim3(static_cast<unsigned>(tiles)), dim3(NT), kSmem, s, p.split, p);
}

int64_t pitch(int64_t n) { return round_up(n, 2); }

}  // namespace

double gram64_cost(int64_t N, int64_t M, int64_t Kc) { return cost_of(N, M, Kc, false, pick_split(N, M, Kc, false)); }
double gram64_form_cost(int64_t D, int64_t A) {
  return cost_of(A, A, D, true, pick_split(A, A, D, true)) + static_cast<double>(D) * static_cast<double>(A) * 12.0 / 2000.0 + 5000.0;
}

void gram64_extend_layout(const sfb_config& c, bool coder, Layout& L, size_t& off) {
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + kAlign - 1) / kAlign * kAlign; return o; };
  const size_t Kp = static_cast<size_t>(pitch(static_cast<int64_t>(c.workers) * c.batch)), D = c.rows, A = c.cols;
  L.Wd = take(D * A * 8);
  L.Gd = take(A * A * 8);
  if (!coder) return;
  L.Xd = take(D * Kp * 8);
  L.Bd = take(A * Kp * 8);
  L.Ad = take(2 * A * Kp * 8);
}

cudaError_t gram64_begin(sfb_ctx* ctx, float* G32) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t n4 = c.rows * c.cols / 4;
  double* Wd = ctx->at<double>(L.Wd);
  const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((n4 + 255) / 256, static_cast<int64_t>(sm_count()) * 8));
  cudaError_t e = launch_kernel(widen_kernel, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, ctx->stream, 1, ctx->W, Wd, n4);
  if (e != cudaSuccess) return e;
  Params p{};
  p.N = p.M = static_cast<int32_t>(c.cols); p.Kc = static_cast<int32_t>(c.rows);
  p.P = p.Q = Wd; p.ldp = p.ldq = c.cols;
  p.out = ctx->at<double>(L.Gd); p.f32 = G32;
  ctx->stats.flops += static_cast<double>(c.cols) * c.cols * c.rows;
  return product<E_GRAM>(ctx->stream, p, c.cols);
}

cudaError_t gram64_codes(sfb_ctx* ctx, int64_t n, const float* X, float* V) {
  const sfb_config& c = ctx->cfg;
  const Layout& L = ctx->lay;
  const int64_t ld = pitch(n);
  double* a[2] = {ctx->at<double>(L.Ad), ctx->at<double>(L.Ad) + c.cols * pitch(ctx->K)};
  double* Xd = ctx->at<double>(L.Xd);
  cudaError_t e = transpose(ctx->stream, X, n, c.rows, c.rows, Xd, ld);
  if (e != cudaSuccess) return e;
  Params p{};
  p.N = static_cast<int32_t>(c.cols); p.M = static_cast<int32_t>(n); p.Kc = static_cast<int32_t>(c.rows);
  p.P = ctx->at<double>(L.Wd); p.Q = Xd; p.ldp = c.cols; p.ldq = ld;
  p.b = ctx->at<double>(L.Bd); p.sc = ctx->at<Scalars>(L.scalars); p.lam = static_cast<double>(c.sc_lambda);
  p.out = a[0];
  if ((e = product<E_FIRST>(ctx->stream, p, ctx->K)) != cudaSuccess) return e;
  p.P = ctx->at<double>(L.Gd); p.Kc = p.N;
  for (int t = 1; t < c.sc_ista_iters; ++t) {
    p.Q = p.cur = a[(t - 1) & 1];
    p.out = a[t & 1];
    if ((e = product<E_STEP>(ctx->stream, p, ctx->K)) != cudaSuccess) return e;
  }
  ctx->stats.flops += 2.0 * n * c.cols * (static_cast<double>(c.rows) + static_cast<double>(c.sc_ista_iters - 1) * c.cols);
  return transpose(ctx->stream, static_cast<const double*>(a[(c.sc_ista_iters - 1) & 1]), c.cols, n, ld, V, c.cols);
}

}  // namespace sfb
