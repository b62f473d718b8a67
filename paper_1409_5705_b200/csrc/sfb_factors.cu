// Bandwidth-bound kernels of the SFB step in fp32: factor packing, the row softmax of multiclass logistic
// regression, the pair residual of distance metric learning, the column-norm prox of sparse coding and the
// power iteration that estimates the coder's step size.
#include <algorithm>

#include <cuda_bf16.h>

#include "sfb_internal.h"

#define SFB_TRY(call)                         \
  do {                                        \
    const cudaError_t e__ = (call);           \
    if (e__ != cudaSuccess) return e__;       \
  } while (0)

namespace sfb {
namespace {

constexpr int kThreads = 256;

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

// Block-wide sum in a fixed order (warp shuffles, then warp 0 over the per-warp values).
template <int NTHREADS>
__device__ __forceinline__ float block_sum(float v, float* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  float r = (threadIdx.x < NTHREADS / 32) ? sh[threadIdx.x] : 0.f;
  if (w == 0) r = warp_sum(r);
  if (threadIdx.x == 0) sh[0] = r;
  __syncthreads();
  return sh[0];
}
template <int NTHREADS>
__device__ __forceinline__ float block_max(float v, float* sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = warp_max(v);
  __syncthreads();
  if (lane == 0) sh[w] = v;
  __syncthreads();
  float r = (threadIdx.x < NTHREADS / 32) ? sh[threadIdx.x] : -INFINITY;
  if (w == 0) r = warp_max(r);
  if (threadIdx.x == 0) sh[0] = r;
  __syncthreads();
  return sh[0];
}

// v = x (MLR) or v = x - y (DML pair difference, Section 2), 16-byte vectors with a scalar tail.
__global__ void pack_kernel(float* __restrict__ dst, const float* __restrict__ x, const float* __restrict__ y,
                            int64_t n4, int64_t n, const Stamp st) {
  pdl_launch_dependents();
  pdl_wait(dst, x, y);
  stamp_begin(st);
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n4; i += stride) {
    float4 a = reinterpret_cast<const float4*>(x)[i];
    if (y) {
      const float4 b = reinterpret_cast<const float4*>(y)[i];
      a.x -= b.x; a.y -= b.y; a.z -= b.z; a.w -= b.w;
    }
    reinterpret_cast<float4*>(dst)[i] = a;
  }
  for (int64_t i = n4 * 4 + blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride)
    dst[i] = y ? x[i] - y[i] : x[i];
}

__global__ void zero_kernel(float* __restrict__ dst, int64_t n) {
  pdl_launch_dependents();
  pdl_wait(dst);
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride) dst[i] = 0.f;
}

__global__ void prox_entries_kernel(float* __restrict__ w, int64_t n, int kind, float a) {
  pdl_launch_dependents();
  pdl_wait(w);
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride)
    w[i] = prox_entry(w[i], kind, a);
}

__global__ void axpy_kernel(float* __restrict__ y, const float* __restrict__ x, float alpha, int64_t n) {
  pdl_launch_dependents();
  pdl_wait(y, x);
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n; i += stride)
    y[i] = fmaf(alpha, x[i], y[i]);
}

// One block per sample: u = softmax(z) - onehot(y) in place over the sample's row of Z [nsamp x rows]
// (Section 1: u is the prediction vector; Section 2.1: u = d f / d (W a)).  A class id outside [0, rows)
// sets a status bit and subtracts nothing.  loss = log sum exp z - z_y.
template <int NTHREADS>
__global__ void __launch_bounds__(NTHREADS) mlr_softmax_kernel(float* __restrict__ Z, int64_t rows, int64_t ldz,
                                                               const int32_t* __restrict__ labels,
                                                               float* __restrict__ loss, uint32_t* status) {
  pdl_launch_dependents();
  pdl_wait(Z, labels, loss);
  __shared__ float sh[32];
  float* z = Z + static_cast<int64_t>(blockIdx.x) * ldz;
  float m = -INFINITY;
  for (int64_t j = threadIdx.x; j < rows; j += NTHREADS) m = fmaxf(m, z[j]);
  m = block_max<NTHREADS>(m, sh);
  float s = 0.f;
  for (int64_t j = threadIdx.x; j < rows; j += NTHREADS) s += expf(z[j] - m);
  s = block_sum<NTHREADS>(s, sh);
  const float inv = 1.f / s;
  const int32_t y = labels[blockIdx.x];
  const bool ok = y >= 0 && y < rows;
  if (threadIdx.x == 0) {
    if (!ok) atomicOr(status, SFB_STATUS_LABEL_RANGE);
    loss[blockIdx.x] = ok ? (m + logf(s)) - z[y] : 0.f;
  }
  __syncthreads();
  for (int64_t j = threadIdx.x; j < rows; j += NTHREADS) {
    float u = expf(z[j] - m) * inv;
    if (ok && j == y) u -= 1.f;
    z[j] = u;
  }
}

// Row-sharded form of the same factor (the parameter matrix partitioned by rows; every shard holds all K samples'
// logits against its own rows only).  First half, one block per sample: the shard's softmax partial
//   part[i] = (m_i, s_i, zy_i, has_i):  m_i = max_j z_ij,  s_i = sum_j exp(z_ij - m_i)  over the shard's rows j,
//   zy_i = z_{i,y_i} and has_i = 1 when class y_i is one of the shard's rows, else 0 and 0.
// labels are global class ids; the shard holds rows [row_off, row_off + rows).
template <int NTHREADS>
__global__ void __launch_bounds__(NTHREADS) mlr_shard_partials_kernel(const float* __restrict__ Z, int64_t rows, int64_t ldz,
                                                                      const int32_t* __restrict__ labels, int64_t row_off,
                                                                      float4* __restrict__ part) {
  pdl_launch_dependents();
  pdl_wait(Z, labels, part);
  __shared__ float sh[32];
  const float* z = Z + static_cast<int64_t>(blockIdx.x) * ldz;
  float m = -INFINITY;
  for (int64_t j = threadIdx.x; j < rows; j += NTHREADS) m = fmaxf(m, z[j]);
  m = block_max<NTHREADS>(m, sh);
  float s = 0.f;
  for (int64_t j = threadIdx.x; j < rows; j += NTHREADS) s += expf(z[j] - m);
  s = block_sum<NTHREADS>(s, sh);
  if (threadIdx.x == 0) {
    const int64_t yl = static_cast<int64_t>(labels[blockIdx.x]) - row_off;
    const bool mine = yl >= 0 && yl < rows;
    part[blockIdx.x] = make_float4(m, s, mine ? z[yl] : 0.f, mine ? 1.f : 0.f);
  }
}

// Merge of the shards' partials of one sample, in shard order:  lse = M + log sum_g s_g exp(m_g - M),  M = max_g m_g;
// zy = sum_g zy_g (only the owning shard contributes).  parts is [shards][K].
__device__ __forceinline__ void merge_shard_partials(const float4* __restrict__ parts, int shards, int64_t K, int64_t i,
                                                     float& lse, float& zy, float& has) {
  float M = -INFINITY;
  for (int g = 0; g < shards; ++g) M = fmaxf(M, parts[static_cast<int64_t>(g) * K + i].x);
  float S = 0.f;
  zy = 0.f; has = 0.f;
  for (int g = 0; g < shards; ++g) {
    const float4 v = parts[static_cast<int64_t>(g) * K + i];
    S += v.y * expf(v.x - M);
    zy += v.z;
    has += v.w;
  }
  lse = M + logf(S);
}

// Second half, one block per sample: with the global log-partition, u_ij = exp(z_ij - lse_i) - [j is y_i's row] in
// place over the shard's rows; loss_i = lse_i - z_{i,y_i} (the same on every shard).  A class id that no shard owns
// sets the status bit and subtracts nothing.
template <int NTHREADS>
__global__ void __launch_bounds__(NTHREADS) mlr_shard_finish_kernel(float* __restrict__ Z, int64_t rows, int64_t ldz,
                                                                    const int32_t* __restrict__ labels, int64_t row_off,
                                                                    const float4* __restrict__ parts, int shards, int64_t K,
                                                                    float* __restrict__ loss, uint32_t* status) {
  pdl_launch_dependents();
  pdl_wait(Z, labels, parts, loss);
  __shared__ float sh_lse;
  float* z = Z + static_cast<int64_t>(blockIdx.x) * ldz;
  if (threadIdx.x == 0) {
    float lse, zy, has;
    merge_shard_partials(parts, shards, K, blockIdx.x, lse, zy, has);
    const bool ok = has > 0.5f;
    if (!ok) atomicOr(status, SFB_STATUS_LABEL_RANGE);
    loss[blockIdx.x] = ok ? lse - zy : 0.f;
    sh_lse = lse;
  }
  __syncthreads();
  const float lse = sh_lse;
  const int64_t yl = static_cast<int64_t>(labels[blockIdx.x]) - row_off;
  for (int64_t j = threadIdx.x; j < rows; j += NTHREADS) {
    float u = expf(z[j] - lse);
    if (j == yl) u -= 1.f;
    z[j] = u;
  }
}

// SDCA for l2-regularised multiclass logistic regression (Section 2.1, "Stochastic DCA").  One block per sample:
// the new dual row q minimises  sum_j q_j log q_j - q.(z + kappa q_old) + kappa/2 ||q||^2  over the simplex, kappa =
// ||x||^2 / (lam N).  Stationarity: log q_j + kappa q_j = t_j - nu with t = z + kappa q_old, and nu such that the q_j sum
// to 1; nu lies in [lse(t) - kappa, lse(t)].
// q_j(nu) with c = t_j - nu: kappa q = W(kappa e^c), W the Lambert function.  Nearly every class has kappa e^c << 1, where four
// terms of its series at 0 (Corless et al., "On the Lambert W function", 1996) are exact to 5 e^4 < 1e-11; else Newton on
// y = log q for  y + kappa e^y = c  (increasing and convex in y, so monotone from the right of the root, where it starts).
__device__ __forceinline__ float sdca_coordinate(float c, float kappa) {
  const float ec = expf(c), e = kappa * ec;
  if (e < 1e-3f) return ec * fmaf(e, fmaf(e, fmaf(e, -8.f / 3.f, 1.5f), -1.f), 1.f);
  float y = c;                                       // y + kappa e^y - c = kappa e^c >= 0 here: right of the root
  if (c > 0.f) y = fminf(c, logf((c + 1.f) / kappa));
#pragma unroll 1
  for (int it = 0; it < 24; ++it) {
    const float f = kappa * expf(y);
    const float d = (y + f - c) / (1.f + f);
    y -= d;
    if (fabsf(d) <= 1e-7f * fmaxf(1.f, fabsf(y))) break;
  }
  return expf(y);
}

// Sums of three values over the block in a fixed order, in every thread.
template <int NTHREADS>
__device__ __forceinline__ float3 block_sum3(float a, float b, float c, float3* sh) {
  a = warp_sum(a); b = warp_sum(b); c = warp_sum(c);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = make_float3(a, b, c);
  __syncthreads();
  float3 r = make_float3(0.f, 0.f, 0.f);
#pragma unroll
  for (int w = 0; w < NTHREADS / 32; ++w) { r.x += sh[w].x; r.y += sh[w].y; r.z += sh[w].z; }
  return r;
}

struct SdcaParams {
  const float* Z;              // logits [n x ldz]
  int64_t rows, ldz;
  const float* X;
  int64_t cols;
  const int32_t* labels;
  const int32_t* ids;
  float* Q;
  int64_t n_samples;
  float inv_lam_n, gamma;
  float* out;                  // du in fp32 [n x ldo] (may be Z itself), or null with
  int64_t ldo;
  __nv_bfloat16* P;            //   du in bf16 [n x ldp], 0 at the label entry, whose value goes to coef
  int64_t ldp;
  float* coef;
  float* loss;
  uint32_t* status;
  int32_t* slot;               // may be null
  int64_t off;                 // first sample's index (slot)
};

// What bounds it: the exponentials, one per class and pass over a sample's classes.  The passes: t and its maximum; the sums
// behind lse(t), lse(z) and the first step of nu; two or three of the outer Newton; the write-out.  t - lse stays in shared
// memory (KEEP; up to 50,000 classes), and nu is carried as its distance from lse(t): as a number near lse(t) its own spacing
// (1e-6) is above the tolerance of the sum, and the iteration ran to its limit of twelve passes.
// 512 samples x 10,000 classes: 76 us; 420 us with a Newton solve per class and pass and those twelve passes.
template <int NTHREADS, bool KEEP>
__global__ void __launch_bounds__(NTHREADS) sdca_dual_kernel(const __grid_constant__ SdcaParams p) {
  pdl_launch_dependents();
  pdl_wait();
  extern __shared__ float base[];                    // KEEP: t_j, then t_j - lse(t)
  __shared__ float sh[32];
  __shared__ float3 sh3[NTHREADS / 32];
  const int t = threadIdx.x, rows = static_cast<int>(p.rows);
  const int64_t i = blockIdx.x;
  const float* z = p.Z + i * p.ldz;
  float* out = p.out ? p.out + i * p.ldo : nullptr;
  __nv_bfloat16* P = p.P ? p.P + i * p.ldp : nullptr;
  const int64_t id = p.ids[i];
  const int32_t y = p.labels[i];
  const bool ok = id >= 0 && id < p.n_samples && y >= 0 && y < rows;
  if (!ok) {                                         // uniform over the block: skip the sample, contribute nothing
    if (t == 0) {
      atomicOr(p.status, (id >= 0 && id < p.n_samples) ? SFB_STATUS_LABEL_RANGE : SFB_STATUS_SAMPLE_RANGE);
      if (p.coef) p.coef[i] = 0.f;
      p.loss[i] = 0.f;
    }
    for (int j = t; j < rows; j += NTHREADS) {
      if (out) out[j] = 0.f;
      if (P) P[j] = __float2bfloat16_rn(0.f);
    }
    return;
  }
  float* q = p.Q + id * p.rows;
  const float4* x = reinterpret_cast<const float4*>(p.X + i * p.cols);
  float ss = 0.f;
  for (int d = t; d < p.cols / 4; d += NTHREADS) {
    const float4 v = x[d];
    ss = fmaf(v.x, v.x, ss); ss = fmaf(v.y, v.y, ss); ss = fmaf(v.z, v.z, ss); ss = fmaf(v.w, v.w, ss);
  }
  const float kappa = block_sum<NTHREADS>(ss, sh) * p.inv_lam_n;
  float m = -INFINITY, mz = -INFINITY;
#pragma unroll 4
  for (int j = t; j < rows; j += NTHREADS) {
    const float zj = z[j], tj = fmaf(kappa, q[j], zj);
    if (KEEP) base[j] = tj;
    m = fmaxf(m, tj);
    mz = fmaxf(mz, zj);
  }
  m = block_max<NTHREADS>(m, sh);
  mz = block_max<NTHREADS>(mz, sh);
  float s1 = 0.f, s2 = 0.f, sz = 0.f;
#pragma unroll 4
  for (int j = t; j < rows; j += NTHREADS) {
    const float zj = z[j], e = expf((KEEP ? base[j] : fmaf(kappa, q[j], zj)) - m);
    s1 += e;
    s2 = fmaf(e, e, s2);
    sz += expf(zj - mz);
  }
  const float3 r = block_sum3<NTHREADS>(s1, s2, sz, sh3);
  const float lse = m + logf(r.x);
  if (t == 0) {
    p.loss[i] = (mz + logf(r.z)) - z[y];             // the sample's logistic loss at the W of this step
    if (p.slot) atomicMin(&p.slot[y], static_cast<int32_t>(p.off + i));
  }
  if (KEEP)
    for (int j = t; j < rows; j += NTHREADS) base[j] -= lse;
  auto dist = [&](int j) { return KEEP ? base[j] : fmaf(kappa, q[j], z[j]) - lse; };
  // safeguarded Newton on d = nu - lse(t): G(d) = sum_j q_j is decreasing and convex, G(-kappa) >= 1 >= G(0); to first order
  // in kappa G(d) = 1 - kappa sum p^2 - d with p = softmax(t)
  float lo = -kappa, hi = 0.f, d = -kappa * r.y / (r.x * r.x), S = 1.f;
#pragma unroll 1
  for (int it = 0; it < 12; ++it) {
    float G = 0.f, Dv = 0.f;
#pragma unroll 4
    for (int j = t; j < rows; j += NTHREADS) {
      const float qj = sdca_coordinate(dist(j) - d, kappa);
      G += qj;
      Dv += __fdividef(qj, fmaf(kappa, qj, 1.f));    // (only steers the iteration)
    }
    const float3 v = block_sum3<NTHREADS>(G, Dv, 0.f, sh3);
    S = v.x;
    const float g = S - 1.f;
    // the write-out divides by S: what is left of an error g in the sum is g kappa q_j / (1 + kappa q_j) of an entry
    if (fabsf(g) <= 2e-7f || (fabsf(g) <= 1e-4f && fabsf(g) * kappa <= 5e-8f)) break;   // uniform over the block
    if (it == 11) break;
    if (g > 0.f) lo = fmaxf(lo, d); else hi = fminf(hi, d);
    float next = d + g / v.y;
    if (!(next > lo && next < hi)) next = 0.5f * (lo + hi);
    if (next == d) break;
    d = next;
  }
  const float invS = 1.f / S;
#pragma unroll 4
  for (int j = t; j < rows; j += NTHREADS) {
    const float qo = q[j];
    const float du = fmaf(sdca_coordinate(dist(j) - d, kappa), invS, -qo);      // du = q_new - q_old
    if (out) out[j] = du;
    if (P) P[j] = __float2bfloat16_rn(j == y ? 0.f : du);
    q[j] = fmaf(p.gamma, du, qo);
    if (p.coef && j == y) p.coef[i] = -du;
  }
}

// One block per pair: q = ||z||^2; similar: u = 2z; dissimilar: u = -2z if q < margin else 0 (Section 2, DML).
// Row-sharded form: with norm_out the block only stores its shard's q and leaves z as it is; with
// norms_all it takes q as the sum, in shard order, of the shards' values and scales.
template <int NTHREADS>
__global__ void __launch_bounds__(NTHREADS) dml_scale_kernel(float* __restrict__ Z, int64_t rows, int64_t ld,
                                                             const int32_t* __restrict__ similar, float margin,
                                                             float* __restrict__ norm_out,
                                                             const float* __restrict__ norms_all,
                                                             int shards, int64_t nstride, __nv_bfloat16* __restrict__ split,
                                                             int64_t split_half, const float* __restrict__ inv_v,
                                                             float* __restrict__ most) {
  pdl_launch_dependents();
  pdl_wait(Z, similar, norm_out, norms_all, split, inv_v, most);
  __shared__ float sh[32];
  float* z = Z + static_cast<int64_t>(blockIdx.x) * ld;
  float q = 0.f;
  if (norms_all) {
    for (int g = 0; g < shards; ++g) q += norms_all[g * nstride + blockIdx.x];
  } else {
    for (int64_t j = threadIdx.x; j < rows; j += NTHREADS) q = fmaf(z[j], z[j], q);
    q = block_sum<NTHREADS>(q, sh);
  }
  if (norm_out) {
    if (threadIdx.x == 0) norm_out[blockIdx.x] = q;
    return;
  }
  const float c = similar[blockIdx.x] != 0 ? 2.f : (q < margin ? -2.f : 0.f);
  float m = 0.f;
  __nv_bfloat16* hp = split ? split + static_cast<int64_t>(blockIdx.x) * 2 * split_half : nullptr;
  for (int64_t j = threadIdx.x; j < rows; j += NTHREADS) {
    const float u = c * z[j];
    z[j] = u;
    m = fmaxf(m, fabsf(u));
    if (hp) {
      const __nv_bfloat16 hi = __float2bfloat16_rn(u);
      hp[j] = hi;
      hp[split_half + j] = __float2bfloat16_rn(u - __bfloat162float(hi));
    }
  }
  if (most) {
    m = block_max<NTHREADS>(m, sh);
    if (threadIdx.x == 0) most[blockIdx.x] = m * inv_v[blockIdx.x];
  }
}

__global__ void mean_kernel(const float* __restrict__ v, int64_t n, float* out, const Stamp st) {
  pdl_launch_dependents();
  pdl_wait(v);
  stamp_begin(st);
  __shared__ float sh[32];
  float s = 0.f;
  for (int64_t i = threadIdx.x; i < n; i += 256) s += v[i];
  s = block_sum<256>(s, sh);
  if (threadIdx.x == 0) *out = s / static_cast<float>(n);
}

// Column sums of squares in fp64 (the prox must resolve norms to far better than fp32's 6e-8, because the
// rescaling multiplies every entry of W while the step's update is ~1e-3 of ||W||).
constexpr int kProxLoads = 4;         // rows that a thread of the two passes has under way: 10,000 x 5,000, the scaling 95 us with one, 84 with four
__global__ void __launch_bounds__(kThreads) col_sumsq_kernel(const float* __restrict__ W, int64_t rows, int64_t cols,
                                                             double* __restrict__ part, int64_t slab_rows) {
  pdl_launch_dependents();
  pdl_wait(W, part);
  __shared__ double sh[8][128];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t c0 = static_cast<int64_t>(blockIdx.x) * 128 + tx * 4;
  const int64_t r0 = static_cast<int64_t>(blockIdx.y) * slab_rows;
  const int64_t r1 = min(rows, r0 + slab_rows);
  double a0 = 0., a1 = 0., a2 = 0., a3 = 0.;
  if (c0 < cols) {
    for (int64_t r = r0 + ty; r < r1; r += 8 * kProxLoads) {
      float4 w[kProxLoads];
#pragma unroll
      for (int k = 0; k < kProxLoads; ++k)
        w[k] = r + 8 * k < r1 ? *reinterpret_cast<const float4*>(W + (r + 8 * k) * cols + c0) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < kProxLoads; ++k) {
        a0 = fma(static_cast<double>(w[k].x), static_cast<double>(w[k].x), a0);
        a1 = fma(static_cast<double>(w[k].y), static_cast<double>(w[k].y), a1);
        a2 = fma(static_cast<double>(w[k].z), static_cast<double>(w[k].z), a2);
        a3 = fma(static_cast<double>(w[k].w), static_cast<double>(w[k].w), a3);
      }
    }
  }
  sh[ty][tx * 4 + 0] = a0; sh[ty][tx * 4 + 1] = a1; sh[ty][tx * 4 + 2] = a2; sh[ty][tx * 4 + 3] = a3;
  __syncthreads();
  if (threadIdx.x < 128) {
    const int64_t c = static_cast<int64_t>(blockIdx.x) * 128 + threadIdx.x;
    if (c < cols) {
      double s = 0.;
#pragma unroll
      for (int k = 0; k < 8; ++k) s += sh[k][threadIdx.x];
      part[static_cast<int64_t>(blockIdx.y) * cols + c] = s;
    }
  }
}

// Prox of Figure 3: b <- b / ||b|| for the columns with ||b|| > 1, others untouched (bit-identical).
__global__ void __launch_bounds__(kThreads) prox_scale_kernel(float* __restrict__ W, int64_t rows, int64_t cols,
                                                              const double* __restrict__ part, int nslabs,
                                                              int64_t slab_rows, unsigned long long* end) {
  pdl_launch_dependents();
  pdl_wait(W, part);
  __shared__ double scale[128];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  if (threadIdx.x < 128) {
    const int64_t c = static_cast<int64_t>(blockIdx.x) * 128 + threadIdx.x;
    double s = 0.;
    if (c < cols)
      for (int k = 0; k < nslabs; ++k) s += part[static_cast<int64_t>(k) * cols + c];
    scale[threadIdx.x] = s > 1. ? 1. / sqrt(s) : 1.;
  }
  __syncthreads();
  const int64_t c0 = static_cast<int64_t>(blockIdx.x) * 128 + tx * 4;
  stamp_end(end);                     // (the kernel is a single wave of short blocks)
  if (c0 >= cols) return;
  const double s0 = scale[tx * 4], s1 = scale[tx * 4 + 1], s2 = scale[tx * 4 + 2], s3 = scale[tx * 4 + 3];
  if (s0 == 1. && s1 == 1. && s2 == 1. && s3 == 1.) return;
  const int64_t r0 = static_cast<int64_t>(blockIdx.y) * slab_rows;
  const int64_t r1 = min(rows, r0 + slab_rows);
  for (int64_t r = r0 + ty; r < r1; r += 8 * kProxLoads) {
    float4 w[kProxLoads];
#pragma unroll
    for (int k = 0; k < kProxLoads; ++k)
      if (r + 8 * k < r1) w[k] = *reinterpret_cast<const float4*>(W + (r + 8 * k) * cols + c0);
#pragma unroll
    for (int k = 0; k < kProxLoads; ++k) {
      if (r + 8 * k >= r1) break;
      if (s0 != 1.) w[k].x = static_cast<float>(static_cast<double>(w[k].x) * s0);
      if (s1 != 1.) w[k].y = static_cast<float>(static_cast<double>(w[k].y) * s1);
      if (s2 != 1.) w[k].z = static_cast<float>(static_cast<double>(w[k].z) * s2);
      if (s3 != 1.) w[k].w = static_cast<float>(static_cast<double>(w[k].w) * s3);
      *reinterpret_cast<float4*>(W + (r + 8 * k) * cols + c0) = w[k];
    }
  }
}

// ---------------------------------------------------------------------------------------------------------
// Power iteration for the coder's step size: one cooperative kernel runs all iterations, one block per SM, with a barrier
// over the grid where an iteration needs the others' results (separate launches, three per iteration, cost more than the
// arithmetic: 640 us for a 2,000 x 1,000 dictionary).  Sums are in a fixed order.
// An iteration costs little more than the way of the vector from all blocks to all blocks.  With a barrier that way is a store,
// a fence, an atomic, a poll and a load one after the other (4 us an iteration); here every value of the vector carries the
// number of its iteration in the same 8 bytes, and who needs the vector reads it until it is all there.  Two buffers are enough:
// a block writes iteration i + 2 when it has all of i + 1, which the others wrote when they had read all of i.
// The norm is not waited for either: it is known one iteration later.  With rho_i = ||G v_i|| / ||v_i||, which settles, an iteration
// scales by what rho_(i-2) says the next vector's length will be, so that lengths stay at rho_i rho_(i-1) / rho_(i-2)^2, near 1
// whatever the norm of G (scaled by the length before alone they swing between 1 and ||G||^2, and their squares overflow from
// ||W|| = 6e4 on).  Only the first vector, of length ||G v_0||, and the last are scaled by their own norm.
// 2,000 x 1,000: 200 -> 166 -> 125 us.
// ---------------------------------------------------------------------------------------------------------
constexpr int kPiThreads = 512, kPiWarps = kPiThreads / 32;
constexpr int kPiBlocks = 148;                        // most blocks of the grid (the scratch is sized for it)
constexpr int kPiSmem = 200 << 10;

struct PowerParams {
  const float* W;                                     // [rows x cols]; with GRAM the symmetric [cols x cols] W^T W, rows = cols
  int64_t rows, cols;
  unsigned long long* vec;                            // [2][cols]: (iteration, value) of the unnormalised vectors of odd and even ones
  float* part;                                        // [blocks][cols]: column sums over a block's rows (not GRAM)
  double* norms;                                      // [blocks]
  unsigned long long* barrier;
  Scalars* sc;
  uint32_t* status;
  int iters;
  int smem_rows;                                      // GRAM: rows of G a block keeps in shared memory
  int vec_fits;                                       // the vector is kept in shared memory
};

// All blocks of a cooperative launch.  Gives up after about two seconds (the others then do the same).
__device__ __forceinline__ bool grid_barrier(unsigned long long* count, uint32_t* status) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned long long n = gridDim.x, old = atomicAdd(count, 1ull), target = (old / n + 1) * n;
    const long long t0 = clock64();
    ok = 1;
    while (*reinterpret_cast<volatile unsigned long long*>(count) < target)
      if (clock64() - t0 > 4000000000ll) { ok = 0; atomicOr(status, SFB_STATUS_TIMEOUT); break; }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// sum of v over the block, in every thread
__device__ __forceinline__ double block_sum_d(double v, double* sh) {
  v = warp_sum_d(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.;
  for (int w = 0; w < kPiWarps; ++w) s += sh[w];
  return s;
}
__device__ __forceinline__ float block_sum_f(float v, float* sh) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  return warp_sum(sh[threadIdx.x & (kPiWarps - 1)]) * (kPiWarps / 32.f);
}
__device__ __forceinline__ float dot4(const float4 a, const float4 b, float s) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, s))));
}

__device__ __forceinline__ ulonglong2 ld_pair(const unsigned long long* p) {
  ulonglong2 v;
  asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long tagged(float v, int it) {
  return static_cast<unsigned long long>(static_cast<uint32_t>(it)) << 32 | __float_as_uint(v);
}
__device__ __forceinline__ float4 untagged(const ulonglong2 a, const ulonglong2 b) {
  return make_float4(__uint_as_float(static_cast<uint32_t>(a.x)), __uint_as_float(static_cast<uint32_t>(a.y)),
                     __uint_as_float(static_cast<uint32_t>(b.x)), __uint_as_float(static_cast<uint32_t>(b.y)));
}
// The vector of iteration `it` (vs: into shared memory) and a thread's part of the sum of its squares; false after two seconds.
__device__ __forceinline__ bool get_vector(const unsigned long long* vec, int quads, int it, float4* vs, uint32_t* status, float& ss) {
  const long long t0 = clock64();
  const auto want = static_cast<uint32_t>(it);
  bool ok = true;
  ss = 0.f;
  for (int q = threadIdx.x; q < quads && ok; q += kPiThreads) {
    ulonglong2 a, b;
    while (true) {
      a = ld_pair(vec + 4 * q);
      b = ld_pair(vec + 4 * q + 2);
      if (a.x >> 32 == want && a.y >> 32 == want && b.x >> 32 == want && b.y >> 32 == want) break;
      if (clock64() - t0 > 4000000000ll) { ok = false; atomicOr(status, SFB_STATUS_TIMEOUT); break; }
    }
    const float4 v = untagged(a, b);
    if (vs) vs[q] = v;
    ss = dot4(v, v, ss);
  }
  return __syncthreads_and(ok);
}

// GRAM: v <- G v.  A block keeps its rows of G in shared memory for all iterations if they fit (smem_rows).  Otherwise
// v <- W^T (W v): a block takes its rows of W once per iteration for both products and leaves its column sums, which a second
// phase adds after a barrier.
template <bool GRAM>
__global__ void __launch_bounds__(kPiThreads) power_kernel(const PowerParams p) {
  extern __shared__ __align__(16) float pi_smem[];     // [cols] vector (where it fits), GRAM: then [smem_rows][cols] rows of G
  __shared__ double sh[kPiWarps];
  __shared__ float yrow[kPiWarps], shf[kPiWarps];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, nb = gridDim.x, blk = blockIdx.x;
  const int64_t r0 = p.rows * blk / nb, r1 = p.rows * (blk + 1) / nb;
  const int quads = static_cast<int>(p.cols / 4);
  const float start = rsqrtf(static_cast<float>(p.cols));
  float4* vs = GRAM || p.vec_fits ? reinterpret_cast<float4*>(pi_smem) : nullptr;
  float4* gs = vs + quads;
  const int keep = static_cast<int>(r1 - r0 < p.smem_rows ? r1 - r0 : p.smem_rows);
  if (GRAM)
    for (int q = t; q < keep * quads; q += kPiThreads) gs[q] = reinterpret_cast<const float4*>(p.W + r0 * p.cols)[q];
  float scale = 1.f;                                   // of G v in this iteration (1 / ||v|| in the last pass)
  float iscale = 1.f, scale1 = 1.f, len1 = 1.f;        // its inverse; scale and ||v|| of the iteration before
  for (int it = 0; it <= p.iters; ++it) {              // the last pass only forms ||W v||^2
    const unsigned long long* in = p.vec + static_cast<int64_t>(it & 1) * p.cols;
    unsigned long long* out = p.vec + static_cast<int64_t>((it + 1) & 1) * p.cols;
    const bool last = it == p.iters;
    float ss = 0.f;
    if (it == 0) {
      if (vs)
        for (int q = t; q < quads; q += kPiThreads) vs[q] = make_float4(start, start, start, start);
      __syncthreads();
    } else {
      if (!get_vector(in, quads, it, vs, p.status, ss)) return;
    }
    float unit = 1.f;                                  // of a vector that is not in shared memory
    auto vat = [&](int q) {
      if (GRAM || vs) return vs[q];
      if (it == 0) return make_float4(start, start, start, start);
      const float4 v = untagged(ld_pair(in + 4 * q), ld_pair(in + 4 * q + 2));
      return make_float4(v.x * unit, v.y * unit, v.z * unit, v.w * unit);
    };
    if (it > 0 && (last || it == 1)) {
      double s = 0.;
      for (int q = t; q < quads; q += kPiThreads) {
        const float4 v = vat(q);
        s += static_cast<double>(v.x) * v.x + static_cast<double>(v.y) * v.y + static_cast<double>(v.z) * v.z + static_cast<double>(v.w) * v.w;
      }
      const double n = sqrt(block_sum_d(s, sh));
      if (last) {
        scale = static_cast<float>(1. / n);
      } else {                                         // v_1 / ||v_1||, as if v_0 had been scaled by it; rho_0 = ||v_1||
        unit = static_cast<float>(1. / n);
        if (vs) {
          for (int q = t; q < quads; q += kPiThreads) {
            const float4 v = vs[q];
            vs[q] = make_float4(v.x * unit, v.y * unit, v.z * unit, v.w * unit);
          }
          unit = 1.f;
        }
        __syncthreads();
        scale1 = scale = static_cast<float>(1. / n);
        iscale = static_cast<float>(n);
      }
    }
    auto dot_row = [&](const float4* w4) {             // in every lane
      float s0 = 0.f, s1 = 0.f;
      int q = lane;
      for (; q + 32 < quads; q += 64) { s0 = dot4(w4[q], vat(q), s0); s1 = dot4(w4[q + 32], vat(q + 32), s1); }
      if (q < quads) s0 = dot4(w4[q], vat(q), s0);
      return warp_sum(s0 + s1) * scale;
    };
    double acc = 0.;
    if (GRAM) {
      for (int64_t r = r0 + warp; r < r1; r += kPiWarps) {
        const int k = static_cast<int>(r - r0);
        const float y = dot_row(k < keep ? gs + static_cast<int64_t>(k) * quads : reinterpret_cast<const float4*>(p.W + r * p.cols));
        if (lane == 0) {
          if (last) acc += static_cast<double>(y) * static_cast<double>(pi_smem[r] * scale);
          else reinterpret_cast<volatile unsigned long long*>(out)[r] = tagged(y, it + 1);
        }
      }
    } else {
      // rows in groups of one per warp: y_r = W[r] v, then the group's contribution to the column sums
      float* part = p.part + static_cast<int64_t>(blk) * p.cols;
      for (int64_t g = r0; g < r1 || g == r0; g += kPiWarps) {
        const int64_t r = g + warp;
        float y = 0.f;
        if (r < r1) y = dot_row(reinterpret_cast<const float4*>(p.W + r * p.cols));
        if (last) {
          if (lane == 0) acc += static_cast<double>(y) * y;
          continue;
        }
        __syncthreads();
        if (lane == 0) yrow[warp] = y;
        __syncthreads();
        const int n = static_cast<int>(r1 - g < kPiWarps ? r1 - g : kPiWarps);
        for (int q = t; q < quads; q += kPiThreads) {
          float4 z = g == r0 ? make_float4(0.f, 0.f, 0.f, 0.f) : *reinterpret_cast<float4*>(part + 4 * q);
          for (int k = 0; k < n; ++k) {
            const float4 w = *reinterpret_cast<const float4*>(p.W + (g + k) * p.cols + 4 * q);
            z.x = fmaf(w.x, yrow[k], z.x); z.y = fmaf(w.y, yrow[k], z.y);
            z.z = fmaf(w.z, yrow[k], z.z); z.w = fmaf(w.w, yrow[k], z.w);
          }
          *reinterpret_cast<float4*>(part + 4 * q) = z;
        }
      }
      if (!last) {
        if (!grid_barrier(p.barrier, p.status)) return;
        // this block's columns: the sum over the blocks' parts, one warp per quad of columns
        const int q0 = static_cast<int>(static_cast<int64_t>(quads) * blk / nb), q1 = static_cast<int>(static_cast<int64_t>(quads) * (blk + 1) / nb);
        for (int q = q0 + warp; q < q1; q += kPiWarps) {
          float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int b = lane; b < nb; b += 32) {
            const float4 w = __ldcg(reinterpret_cast<const float4*>(p.part + static_cast<int64_t>(b) * p.cols + 4 * q));
            z.x += w.x; z.y += w.y; z.z += w.z; z.w += w.w;
          }
          z.x = warp_sum(z.x); z.y = warp_sum(z.y); z.z = warp_sum(z.z); z.w = warp_sum(z.w);
          if (lane < 4)
            reinterpret_cast<volatile unsigned long long*>(out)[4 * q + lane] =
                tagged(lane == 0 ? z.x : lane == 1 ? z.y : lane == 2 ? z.z : z.w, it + 1);
        }
      }
    }
    // (any scale does but in the last pass; the vector has been read by everyone, too)
    if (it > 1 && !last) {
      const float sq = block_sum_f(ss, shf), ilen = rsqrtf(sq);
      const float irho = len1 * scale1 * ilen;         // of the iteration before
      scale1 = scale;
      len1 = sq * ilen;
      scale = irho * (irho * iscale) * ilen;           // 1 / (rho * (rho * len * scale))
      iscale = 1.f / scale;
    } else if (!last) {
      __syncthreads();
    }
    if (last) {
      acc = block_sum_d(acc, sh);
      if (t == 0) p.norms[blk] = acc;
      if (!grid_barrier(p.barrier, p.status)) return;
    }
  }
  if (blk == 0 && warp == 0) {
    double s = 0.;
    for (int b = lane; b < nb; b += 32) s += __ldcg(p.norms + b);
    s = warp_sum_d(s);
    if (lane == 0) {
      const float L = static_cast<float>(s);
      p.sc->L = L;
      p.sc->invL = 1.f / L;
    }
  }
}

__global__ void set_L_kernel(Scalars* sc, float L) { pdl_launch_dependents(); pdl_wait(); sc->L = L; sc->invL = 1.f / L; }

inline unsigned grid_for(int64_t n, int per_block) {
  int64_t g = (n + per_block - 1) / per_block;
  if (g < 1) g = 1;
  const int64_t cap = static_cast<int64_t>(sm_count()) * 16;
  return static_cast<unsigned>(g > cap ? cap : g);
}

inline int64_t slab_rows_for(int64_t rows) { return (rows + kProxSlabs - 1) / kProxSlabs; }

}  // namespace

__global__ void stamp_kernel(const Stamp st) {
  pdl_launch_dependents();
  pdl_wait();
  stamp_begin(st);
}

cudaError_t stamp(cudaStream_t s, const Stamp& st) {
  if (st.n <= 0) return cudaSuccess;
  return launch_kernel(stamp_kernel, dim3(1), dim3(32), 0, s, 1, st);
}

cudaError_t pack_copy(cudaStream_t s, float* dst, const float* x, const float* y, int64_t n, const Stamp& st) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(pack_kernel, dim3(grid_for(n / 4 + 1, kThreads)), dim3(kThreads), 0, s, 1, dst, x, y, n / 4, n, st);
}

cudaError_t fill_zero(cudaStream_t s, float* dst, int64_t n) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(zero_kernel, dim3(grid_for(n, kThreads)), dim3(kThreads), 0, s, 1, dst, n);
}

cudaError_t axpy(cudaStream_t s, float* y, const float* x, float alpha, int64_t n) {
  if (n <= 0) return cudaSuccess;
  return launch_kernel(axpy_kernel, dim3(grid_for(n, kThreads)), dim3(kThreads), 0, s, 1, y, x, alpha, n);
}

cudaError_t mlr_softmax_rows(cudaStream_t s, float* Z, int64_t nsamp, int64_t rows, int64_t ldz, const int32_t* labels,
                             float* loss, uint32_t* status) {
  if (nsamp <= 0) return cudaSuccess;
  return launch_kernel(mlr_softmax_kernel<512>, dim3(static_cast<unsigned>(nsamp)), dim3(512), 0, s, 1, Z, rows, ldz,
                       labels, loss, status);
}

cudaError_t prox_entries(cudaStream_t s, float* w, int64_t n, int kind, float a) {
  if (n <= 0 || kind == 0) return cudaSuccess;
  return launch_kernel(prox_entries_kernel, dim3(grid_for(n, kThreads)), dim3(kThreads), 0, s, 1, w, n, kind, a);
}

cudaError_t mlr_shard_partials(cudaStream_t s, const float* Z, int64_t nsamp, int64_t rows, int64_t ldz,
                               const int32_t* labels, int64_t row_off, float* part) {
  if (nsamp <= 0) return cudaSuccess;
  return launch_kernel(mlr_shard_partials_kernel<512>, dim3(static_cast<unsigned>(nsamp)), dim3(512), 0, s, 1, Z, rows,
                       ldz, labels, row_off, reinterpret_cast<float4*>(part));
}

cudaError_t mlr_shard_finish(cudaStream_t s, float* Z, int64_t nsamp, int64_t rows, int64_t ldz, const int32_t* labels,
                             int64_t row_off, const float* parts, int shards, float* loss, uint32_t* status) {
  if (nsamp <= 0) return cudaSuccess;
  return launch_kernel(mlr_shard_finish_kernel<512>, dim3(static_cast<unsigned>(nsamp)), dim3(512), 0, s, 1,  Z, rows,
                       ldz, labels, row_off, reinterpret_cast<const float4*>(parts), shards, nsamp, loss, status);
}

cudaError_t sdca_dual_rows(cudaStream_t s, const SdcaArgs& a) {
  if (a.n <= 0) return cudaSuccess;
  SdcaParams p{};
  p.Z = a.Z; p.rows = a.rows; p.ldz = a.ldz; p.X = a.X; p.cols = a.cols; p.labels = a.labels; p.ids = a.ids;
  p.Q = a.Q; p.n_samples = a.n_samples; p.inv_lam_n = a.inv_lam_n; p.gamma = a.gamma;
  p.out = a.out; p.ldo = a.ldo; p.P = static_cast<__nv_bfloat16*>(a.P); p.ldp = a.ldp;
  p.coef = a.coef; p.loss = a.loss; p.status = a.status; p.slot = a.slot; p.off = a.off;
  constexpr int kKeep = 200 << 10;
  const dim3 grid(static_cast<unsigned>(a.n)), block(512);
  if (a.rows * 4 > kKeep) return launch_kernel(sdca_dual_kernel<512, false>, grid, block, 0, s, 1, p);
  const cudaError_t e = allow_smem<sdca_dual_kernel<512, true>>(kKeep);
  if (e != cudaSuccess) return e;
  return launch_kernel(sdca_dual_kernel<512, true>, grid, block, static_cast<size_t>(a.rows) * 4, s, 1, p);
}

cudaError_t dml_scale_rows(cudaStream_t s, float* Z, int64_t nsamp, int64_t rows, int64_t ld,
                           const int32_t* similar, float margin, void* split, int64_t split_half, const float* inv_v,
                           float* most, float* norm_out, const float* norms_all,
                           int shards, int64_t nstride) {
  if (nsamp <= 0) return cudaSuccess;
  return launch_kernel(dml_scale_kernel<256>, dim3(static_cast<unsigned>(nsamp)), dim3(256), 0, s, 1, Z, rows, ld,
                       similar, margin, norm_out, norms_all, shards, nstride, static_cast<__nv_bfloat16*>(split),
                       split_half, inv_v, most);
}

cudaError_t mean_of(cudaStream_t s, const float* v, int64_t n, float* out, const Stamp& st) {
  return launch_kernel(mean_kernel, dim3(1), dim3(256), 0, s, 1, v, n, out, st);
}

cudaError_t prox_unit_columns(cudaStream_t s, float* W, int64_t rows, int64_t cols, float* colpart, unsigned long long* end) {
  const int64_t sr = slab_rows_for(rows);
  dim3 grid(static_cast<unsigned>((cols + 127) / 128), kProxSlabs);
  double* part = reinterpret_cast<double*>(colpart);
  SFB_TRY(launch_kernel(col_sumsq_kernel, grid, dim3(kThreads), 0, s, 1, W, rows, cols, part, sr));
  return launch_kernel(prox_scale_kernel, grid, dim3(kThreads), 0, s, 1, W, rows, cols, part, kProxSlabs, sr, end);
}

size_t power_scratch_bytes(int64_t cols) {
  return 1024 + static_cast<size_t>(kPiBlocks) * 8 + static_cast<size_t>(cols) * 4 * (4 + kPiBlocks);
}

cudaError_t estimate_lipschitz(cudaStream_t s, const float* W, const float* G, int64_t rows, int64_t cols, void* scratch,
                               Scalars* sc, uint32_t* status, int iters) {
  PowerParams p{};
  char* base = static_cast<char*>(scratch);
  p.barrier = reinterpret_cast<unsigned long long*>(base);
  p.vec = reinterpret_cast<unsigned long long*>(base + 1024);
  p.part = reinterpret_cast<float*>(p.vec + 2 * cols);
  p.norms = reinterpret_cast<double*>(p.part + static_cast<int64_t>(kPiBlocks) * cols);
  p.W = G ? G : W;
  p.rows = G ? cols : rows;
  p.cols = cols;
  p.sc = sc; p.status = status; p.iters = iters;
  cudaError_t e = cudaMemsetAsync(base, 0, 1024 + static_cast<size_t>(cols) * 16, s);     // the barrier, the tags
  if (e != cudaSuccess) return e;
  // a row per warp and block: small dictionaries synchronise fewer blocks
  const int64_t want = (p.rows + kPiWarps - 1) / kPiWarps, most = std::min(sm_count(), kPiBlocks);
  const int64_t row = cols * 4, room = kPiSmem - row;
  const int blocks = static_cast<int>(std::max<int64_t>(1, std::min(want, most)));
  if (G && room < 0) return cudaErrorInvalidValue;    // the vector has to fit: the callers form no Gram matrix that wide
  p.smem_rows = G ? static_cast<int>(std::min<int64_t>((p.rows + blocks - 1) / blocks, room / row)) : 0;
  p.vec_fits = room >= 0;
  const size_t smem = p.vec_fits ? static_cast<size_t>(row * (1 + p.smem_rows)) : 0;
  if ((e = allow_smem<power_kernel<true>>(kPiSmem)) != cudaSuccess || (e = allow_smem<power_kernel<false>>(kPiSmem)) != cudaSuccess) return e;
  void* args[] = {&p};
  const dim3 grid(static_cast<unsigned>(blocks)), block(kPiThreads);
  e = G ? cudaLaunchCooperativeKernel(power_kernel<true>, grid, block, args, smem, s)
        : cudaLaunchCooperativeKernel(power_kernel<false>, grid, block, args, smem, s);
  count_launch();
  return e;
}

cudaError_t set_lipschitz(cudaStream_t s, Scalars* sc, float L) {
  return launch_kernel(set_L_kernel, dim3(1), dim3(1), 0, s, 1, sc, L);
}

}  // namespace sfb

// ---------------------------------------------------------------------------------------------------------
// Column prox without any allocation (sfb_prox_columns_noalloc in sfb.h)
// ---------------------------------------------------------------------------------------------------------
#include <mutex>

namespace {

constexpr int64_t kNoAllocMaxCols = SFB_NOALLOC_MAX_COLS;
constexpr int kNoAllocMaxDevices = 64;

// Per-slab column sums of squares of the no-allocation prox: kProxSlabs x kNoAllocMaxCols doubles (8 MB), resident
// on every device that loads the library until the process exits.  Shared by all calls.
static __device__ __align__(256) double g_noalloc_colpart[static_cast<size_t>(sfb::kProxSlabs) * kNoAllocMaxCols];

std::mutex g_noalloc_mutex;
double* g_noalloc_ptr[kNoAllocMaxDevices] = {};   // device address of the array above, per device ordinal

// The array's name is only a handle on the host; the address a kernel can use comes from the runtime, and it
// differs per device.  Looked up once per device, with that device current.
cudaError_t noalloc_scratch(double** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kNoAllocMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (g_noalloc_ptr[dev] == nullptr) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_colpart);
    if (e != cudaSuccess) return e;
    g_noalloc_ptr[dev] = static_cast<double*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return cudaSuccess;
}

}  // namespace

extern "C" int sfb_prox_columns_noalloc(float* W_dev, int64_t rows, int64_t cols, void* stream) {
  if (!W_dev || rows <= 0 || cols <= 0) return SFB_ERR_ARG;
  if ((reinterpret_cast<uintptr_t>(W_dev) & 15u) != 0) return SFB_ERR_ALIGN;
  if (cols % 4 != 0 || rows > (1LL << 30)) return SFB_ERR_SHAPE;
  if (cols > kNoAllocMaxCols) return SFB_ERR_STATIC_LIMIT;
  // The scratch array looked up below belongs to the current device: W must live there too.
  {
    int dev = -1;
    cudaPointerAttributes attr{};
    if (cudaGetDevice(&dev) != cudaSuccess) return SFB_ERR_CUDA;
    if (cudaPointerGetAttributes(&attr, W_dev) != cudaSuccess) { cudaGetLastError(); return SFB_ERR_ARG; }
    if (attr.type != cudaMemoryTypeDevice || attr.device != dev) return SFB_ERR_ARG;
  }
  double* part = nullptr;
  if (noalloc_scratch(&part) != cudaSuccess) return SFB_ERR_CUDA;
  // Every partial that the second kernel reads is written by the first one in this call, so nothing has to start
  // at zero and what an earlier call left in the array does not matter.
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t sr = sfb::slab_rows_for(rows);
  dim3 grid(static_cast<unsigned>((cols + 127) / 128), sfb::kProxSlabs);
  if (sfb::launch_kernel(sfb::col_sumsq_kernel, grid, dim3(sfb::kThreads), 0, s, 1, W_dev, rows, cols, part,
                         sr) != cudaSuccess)
    return SFB_ERR_CUDA;
  const cudaError_t e = sfb::launch_kernel(sfb::prox_scale_kernel, grid, dim3(sfb::kThreads), 0, s, 1, W_dev, rows, cols,
                                           part, sfb::kProxSlabs, sr,
                                           nullptr);
  return e == cudaSuccess ? SFB_OK : SFB_ERR_CUDA;
}
