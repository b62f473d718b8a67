// fp32 FMA matrix products for the fp32-operand mode of the SFB step:
//   forward  z_i = W v_i            (Section 2: the matrix-vector product W a_i, batched over the K samples)
//   update   W  -= eta * U^T V      (Section 3, Figure 1: reconstruction of the K rank-1 updates)
//   coder    the products of the ISTA iterations of the sparse coder (Figure 3's compute_sparse_code)
//
// One register-tiled kernel, 256 threads, a 128 x 128 tile (8 x 8 outputs per thread) or a 64 x 64 one (4 x 4), operands
// brought to shared memory by cp.async in a four-stage ring.  Bound: the FMA pipe (148 SMs x 128 lanes).  What the design
// does about it:
//  * FMAs are issued in pairs of neighbouring output columns (fma.rn.f32x2: two independent fp32 FMAs in one instruction,
//    each rounded as an fma.f32), so half of the issue slots are left for the loads from shared memory.
//  * B sits in shared memory with the contraction outermost; where it has it innermost in memory it is transposed on the
//    way in by 4-byte cp.async.  So is A in the large tile; in the small one its rows stay as they are and are read four k at
//    a time (the large one has no registers left for that).  Pairing neighbouring k instead when both operands have the contraction innermost
//    needs two accumulators per output: 239 registers, two warps per scheduler, and 63 % of the FMA rate.
//  * A product with too few tiles for the SMs is cut along its contraction over a cluster of 2, 4 or 8 CTAs; the partial
//    tiles are added over distributed shared memory in rank order (deterministic, no scratch in memory, no second launch).
#include "sfb_internal.h"

namespace sfb {
namespace {

constexpr int NT = 256;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void cp16(uint32_t dst, const float* src, int bytes) {        // bytes not read are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp4(uint32_t dst, const float* src, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// two fp32 FMAs
__device__ __forceinline__ void ffma2(uint64_t& d, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t dup2(float a) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// The BK x R slice of an operand (element (r, k) at p[r*ld + k] if KC, else at p[k*ld + r]) into a stage: laid out [r][k] if
// KC and not TRANSPOSE, else [k][r], with row pitch P.  Rows >= nrows and k >= kend read as zeros.  vec: 16-byte pieces
// (pointer and pitch allow them).
template <bool KC, bool TRANSPOSE, int R, int BK, int P>
__device__ __forceinline__ void load_slice(uint32_t dst, const float* __restrict__ p, int64_t ld, int r0, int nrows, int k0,
                                           int kend, bool vec, int t) {
  if (KC && TRANSPOSE) {
#pragma unroll
    for (int v = 0; v < R * BK / NT; ++v) {
      const int idx = t + v * NT, k = idx % BK, r = idx / BK;
      const bool in = r0 + r < nrows && k0 + k < kend;
      cp4(dst + (k * P + r) * 4, in ? p + static_cast<int64_t>(r0 + r) * ld + k0 + k : p, in ? 4 : 0);
    }
  } else {
#pragma unroll
    for (int v = 0; v < R * BK / 4 / NT; ++v) {
      const int idx = t + v * NT;
      const int k = KC ? (idx % (BK / 4)) * 4 : idx / (R / 4), r = KC ? idx / (BK / 4) : (idx % (R / 4)) * 4;
      int left = KC ? (r0 + r < nrows ? kend - k0 - k : 0) : (k0 + k < kend ? nrows - r0 - r : 0);
      left = left < 0 ? 0 : left > 4 ? 4 : left;
      const float* src = left <= 0 ? p : KC ? p + static_cast<int64_t>(r0 + r) * ld + k0 + k : p + static_cast<int64_t>(k0 + k) * ld + r0 + r;
      const uint32_t d = dst + (KC ? r * P + k : k * P + r) * 4;
      if (vec) {
        cp16(d, src, left * 4);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) cp4(d + e * 4, e < left ? src + e : p, e < left ? 4 : 0);
      }
    }
  }
}

__device__ __forceinline__ float soft(float w, float t) {
  const float a = fabsf(w) - t;
  return a > 0.f ? copysignf(a, w) : 0.f;
}

struct GemmParams {
  int32_t M, N, Kc;
  const float* A;
  const float* B;
  int64_t lda, ldb;
  int32_t tilesM, split;        // split: CTAs of a cluster that share one tile's contraction
  bool a_vec, b_vec, c_vec;
  EpiArgs e;
};

template <int EPI>
__device__ __forceinline__ float epi_one(float acc, float cur, float aux, const EpiArgs& e, float invL) {
  if (EPI == EPI_STORE) return acc;
  if (EPI == EPI_SUB) return acc - aux;
  if (EPI == EPI_RMW) return prox_entry(fmaf(e.alpha, acc, cur), e.prox_kind, e.prox_a);
  if (EPI == EPI_ISTA0) return soft(acc * invL, e.lam * invL);
  return soft(fmaf(-acc, invL, cur), e.lam * invL);               // EPI_ISTA
}
template <int EPI>
constexpr bool kReadsCur = EPI == EPI_RMW || EPI == EPI_ISTA;

// four neighbouring outputs of row m (n a multiple of 4) or one output
template <int EPI>
__device__ __forceinline__ void epilogue4(const GemmParams& p, int m, int n, float4 acc, float invL) {
  const EpiArgs& e = p.e;
  float* c = e.C + m * e.ldc + n;
  const float* x = EPI == EPI_SUB ? e.aux + m * e.ldaux + n : nullptr;
  const float* q = EPI == EPI_RMW ? c : kReadsCur<EPI> ? e.cur + m * e.ldcur + n : nullptr;
  if (p.c_vec && n + 3 < p.N) {
    float4 cur = make_float4(0.f, 0.f, 0.f, 0.f), aux = cur, out;
    if (kReadsCur<EPI>) cur = *reinterpret_cast<const float4*>(q);
    if (EPI == EPI_SUB) aux = *reinterpret_cast<const float4*>(x);
    out.x = epi_one<EPI>(acc.x, cur.x, aux.x, e, invL);
    out.y = epi_one<EPI>(acc.y, cur.y, aux.y, e, invL);
    out.z = epi_one<EPI>(acc.z, cur.z, aux.z, e, invL);
    out.w = epi_one<EPI>(acc.w, cur.w, aux.w, e, invL);
    *reinterpret_cast<float4*>(c) = out;
    if (EPI == EPI_ISTA0 && e.C2) *reinterpret_cast<float4*>(e.C2 + m * e.ldc2 + n) = acc;
  } else {
    const float a[4] = {acc.x, acc.y, acc.z, acc.w};
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (n + j < p.N) {
        const float cur = kReadsCur<EPI> ? q[j] : 0.f;
        const float aux = EPI == EPI_SUB ? x[j] : 0.f;
        c[j] = epi_one<EPI>(a[j], cur, aux, e, invL);
        if (EPI == EPI_ISTA0 && e.C2) e.C2[m * e.ldc2 + n + j] = a[j];
      }
  }
}

// Outputs of thread (ty, tx in 0..15): groups of four neighbouring columns, 64 apart; rows the same, or 16 apart where A is
// kept by rows.
template <bool BY_ROWS>
__device__ __forceinline__ int lane_row(int t, int i) { return BY_ROWS ? t + 16 * i : (i >> 2) * 64 + t * 4 + (i & 3); }

template <bool A_KC, bool B_KC, int BT, int EPI>
__global__ void __launch_bounds__(NT, 2) sgemm_kernel(const __grid_constant__ GemmParams p) {
  constexpr int T = BT / 16;                          // outputs per thread and direction
  constexpr int BK = BT == 128 ? 16 : 32;
  constexpr int STG = 4;
  constexpr bool BY_ROWS = A_KC && BT == 64;
  constexpr int PA = BY_ROWS ? BK + 4 : A_KC ? BT + 4 : BT, PB = B_KC ? BT + 4 : BT;    // row pitches: [BT][PA] or [BK][PA]; [BK][PB]
  constexpr int FA = (BY_ROWS ? BT : BK) * PA, FB = BK * PB;          // floats per stage
  extern __shared__ __align__(16) float sm[];
  const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
  const int S = p.split;
  const int tile = blockIdx.x / S, part = blockIdx.x % S;   // clusters are consecutive blocks: part = rank in the cluster
  const int tm = tile % p.tilesM, tn = tile / p.tilesM;
  pdl_launch_dependents();
  pdl_wait();
  if (EPI == EPI_RMW) stamp_begin(p.e.begin);
  const int m0 = tm * BT, n0 = tn * BT;
  // parts of the contraction end at multiples of 32 whatever the tile, so that a product has one summation order
  const int units = (p.Kc + 31) / 32;
  const int kbeg = static_cast<int>(static_cast<int64_t>(part) * units / S) * 32;
  const int kend = min(p.Kc, static_cast<int>(static_cast<int64_t>(part + 1) * units / S) * 32);
  const int nkb = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;
  const uint32_t sbase = smem_addr(sm);

  uint64_t acc[T][T / 2];
#pragma unroll
  for (int i = 0; i < T; ++i)
#pragma unroll
    for (int j = 0; j < T / 2; ++j) acc[i][j] = 0ull;

  auto issue = [&](int kb) {
    if (kb < nkb) {
      const uint32_t st = sbase + (kb % STG) * (FA + FB) * 4;
      load_slice<A_KC, !BY_ROWS, BT, BK, PA>(st, p.A, p.lda, m0, p.M, kbeg + kb * BK, kend, p.a_vec, t);
      load_slice<B_KC, true, BT, BK, PB>(st + FA * 4, p.B, p.ldb, n0, p.N, kbeg + kb * BK, kend, p.b_vec, t);
    }
    cp_commit();
  };
#pragma unroll
  for (int s = 0; s < STG - 1; ++s) issue(s);
  for (int kb = 0; kb < nkb; ++kb) {
    cp_wait<STG - 2>();
    __syncthreads();                                  // stage kb has landed for everyone; stage kb-1 is free
    issue(kb + STG - 1);
    const float* As = sm + (kb % STG) * (FA + FB);
    const float* Bs = As + FA;
    float4 a[BY_ROWS ? T : T / 4];                       // rows of A at four k, or at one
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      ulonglong2 b[T / 4];
      if (BY_ROWS && (k & 3) == 0) {
#pragma unroll
        for (int i = 0; i < T; ++i) a[i] = *reinterpret_cast<const float4*>(As + (ty + 16 * i) * PA + k);
      }
#pragma unroll
      for (int h = 0; h < T / 4; ++h) {
        if (!BY_ROWS) a[h] = *reinterpret_cast<const float4*>(As + k * PA + h * 64 + ty * 4);
        b[h] = *reinterpret_cast<const ulonglong2*>(Bs + k * PB + h * 64 + tx * 4);
      }
#pragma unroll
      for (int i = 0; i < T; ++i) {
        const float4 q = a[BY_ROWS ? i : i >> 2];
        const int c = (BY_ROWS ? k : i) & 3;
        const uint64_t d = dup2(c == 0 ? q.x : c == 1 ? q.y : c == 2 ? q.z : q.w);
#pragma unroll
        for (int h = 0; h < T / 4; ++h) { ffma2(acc[i][2 * h], d, b[h].x); ffma2(acc[i][2 * h + 1], d, b[h].y); }
      }
    }
  }

  float invL = 0.f;
  if (EPI == EPI_ISTA || EPI == EPI_ISTA0) invL = p.e.sc->invL;
  if (S == 1) {
#pragma unroll
    for (int i = 0; i < T; ++i) {
      const int m = m0 + lane_row<BY_ROWS>(ty, i);
      if (m >= p.M) continue;
#pragma unroll
      for (int h = 0; h < T / 4; ++h) {
        const int n = n0 + h * 64 + tx * 4;
        const float2 lo = unpack2(acc[i][2 * h]), hi = unpack2(acc[i][2 * h + 1]);
        if (n < p.N) epilogue4<EPI>(p, m, n, make_float4(lo.x, lo.y, hi.x, hi.y), invL);
      }
    }
    if (EPI == EPI_RMW) stamp_end(p.e.end);
    return;
  }
  // The parts of a split contraction: every CTA of the cluster puts its partial tile into its shared memory, then adds up
  // (in rank order) and finishes its share of the rows.
  cp_wait<0>();
  __syncthreads();
#pragma unroll
  for (int i = 0; i < T; ++i)
#pragma unroll
    for (int h = 0; h < T / 4; ++h) {
      const float2 lo = unpack2(acc[i][2 * h]), hi = unpack2(acc[i][2 * h + 1]);
      *reinterpret_cast<float4*>(sm + lane_row<BY_ROWS>(ty, i) * BT + h * 64 + tx * 4) = make_float4(lo.x, lo.y, hi.x, hi.y);
    }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  const int rows_here = BT / S, rbeg = part * rows_here;
  for (int q = t; q < rows_here * (BT / 4); q += NT) {
    const int r = rbeg + q / (BT / 4), c = (q % (BT / 4)) * 4;
    const int m = m0 + r, n = n0 + c;
    if (m >= p.M || n >= p.N) continue;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t own = smem_addr(sm + r * BT + c);
    for (int g = 0; g < S; ++g) {
      uint32_t peer;
      float4 w;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(own), "r"(g));
      asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(w.x), "=f"(w.y), "=f"(w.z), "=f"(w.w) : "r"(peer));
      v.x += w.x; v.y += w.y; v.z += w.z; v.w += w.w;
    }
    epilogue4<EPI>(p, m, n, v, invL);
  }
  if (EPI == EPI_RMW) stamp_end(p.e.end);
  // no CTA leaves while a peer still reads its tile
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

template <bool A_KC, bool B_KC, int BT>
constexpr int smem_bytes() {
  constexpr int BK = BT == 128 ? 16 : 32;
  constexpr int f = (A_KC && BT == 64 ? BT * (BK + 4) : BK * (A_KC ? BT + 4 : BT)) + BK * (B_KC ? BT + 4 : BT);
  constexpr int ring = 4 * f * 4, out = BT * BT * 4;
  return ring > out ? ring : out;
}

template <bool A_KC, bool B_KC, int BT, int EPI>
cudaError_t launch_one(cudaStream_t s, const GemmParams& p, int64_t tiles) {
  constexpr int smem = smem_bytes<A_KC, B_KC, BT>();
  const cudaError_t e = allow_smem<sgemm_kernel<A_KC, B_KC, BT, EPI>>(smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(sgemm_kernel<A_KC, B_KC, BT, EPI>, dim3(static_cast<unsigned>(tiles * p.split)), dim3(NT), smem, s,
                       p.split, p);
}

template <bool A_KC, bool B_KC, int EPI>
cudaError_t launch(cudaStream_t s, int64_t M, int64_t N, int64_t Kc, const float* A, int64_t lda, const float* B,
                   int64_t ldb, const EpiArgs& e, int64_t M_split) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  GemmParams p{};
  p.M = static_cast<int32_t>(M); p.N = static_cast<int32_t>(N); p.Kc = static_cast<int32_t>(Kc);
  p.A = A; p.B = B; p.lda = lda; p.ldb = ldb; p.e = e;
  p.a_vec = aligned16(A) && lda % 4 == 0;
  p.b_vec = aligned16(B) && ldb % 4 == 0;
  p.c_vec = aligned16(e.C) && e.ldc % 4 == 0 && (!e.aux || (aligned16(e.aux) && e.ldaux % 4 == 0)) &&
            (!e.cur || (aligned16(e.cur) && e.ldcur % 4 == 0)) && (!e.C2 || (aligned16(e.C2) && e.ldc2 % 4 == 0));
  const GemmShape g = pick_gemm_shape(M_split > 0 ? M_split : M, N, Kc);
  p.split = g.split;
  // the split belongs to the product (it fixes the summation order); the tile follows the rows of this call
  const bool big = gemm_cost(128, g.split, M, N, Kc) <= gemm_cost(64, g.split, M, N, Kc);
  const int BT = big ? 128 : 64;
  const int64_t tilesM = (M + BT - 1) / BT, tilesN = (N + BT - 1) / BT, tiles = tilesM * tilesN;
  if (tiles * p.split > 0x7fffffffLL) return cudaErrorInvalidValue;
  p.tilesM = static_cast<int32_t>(tilesM);
  return big ? launch_one<A_KC, B_KC, 128, EPI>(s, p, tiles) : launch_one<A_KC, B_KC, 64, EPI>(s, p, tiles);
}

}  // namespace

// SM cycles of a product with BT x BT tiles and its contraction in `split` parts: rounds of tiles over the SMs (two CTAs of
// either tile per SM) times the cycles of a part.  A pair of 128-wide tiles takes about 300 cycles per k on an SM (85 % of
// its FMA rate), a pair of 64-wide ones 100; a tile that has its SM to itself 185 and 65.  A part also pays for filling its
// ring and for the exchange.
double gemm_cost(int BT, int split, int64_t M, int64_t N, int64_t Kc) {
  const double tm = static_cast<double>((M + BT - 1) / BT), tn = static_cast<double>((N + BT - 1) / BT);
  const double tiles = tm * tn * split;
  const double sms = kModelSms;
  const double k = static_cast<double>(Kc) / split;
  const int64_t per_sm = static_cast<int64_t>((tiles + sms - 1.0) / sms);       // tiles of the busiest SM
  const double pairs = static_cast<double>(per_sm / 2), single = static_cast<double>(per_sm % 2);
  const double per_k = BT == 128 ? 300.0 * pairs + 185.0 * single : 100.0 * pairs + 65.0 * single;
  return k * per_k + (pairs + single) * (BT == 128 ? 4000.0 : 2000.0) + (split > 1 ? 2500.0 : 0.0);
}

GemmShape pick_gemm_shape(int64_t M, int64_t N, int64_t Kc) {
  GemmShape best{128, 1};
  double cost = gemm_cost(128, 1, M, N, Kc);
  for (int bt = 128; bt >= 64; bt -= 64)
    for (int s = 1; s <= 8; s *= 2) {
      if (s > 1 && Kc < 64 * s) break;                // at least two 32-deep blocks per part
      const double c = gemm_cost(bt, s, M, N, Kc);
      if (c < 0.97 * cost) { cost = c; best = {bt, s}; }
    }
  return best;
}

double gemm_cycles(int64_t M, int64_t N, int64_t Kc) {
  const GemmShape g = pick_gemm_shape(M, N, Kc);
  return std::min(gemm_cost(128, g.split, M, N, Kc), gemm_cost(64, g.split, M, N, Kc));
}

cudaError_t sgemm(cudaStream_t s, bool a_kc, bool b_kc, Epilogue epi, int64_t M, int64_t N, int64_t Kc,
                  const float* A, int64_t lda, const float* B, int64_t ldb, const EpiArgs& e, int64_t M_split) {
#define SFB_GO(AK, BK_, E) return launch<AK, BK_, E>(s, M, N, Kc, A, lda, B, ldb, e, M_split)
  if (a_kc && b_kc) {
    if (epi == EPI_STORE) SFB_GO(true, true, EPI_STORE);
    if (epi == EPI_SUB) SFB_GO(true, true, EPI_SUB);
  } else if (a_kc) {
    if (epi == EPI_ISTA) SFB_GO(true, false, EPI_ISTA);
    if (epi == EPI_ISTA0) SFB_GO(true, false, EPI_ISTA0);
  } else if (!b_kc) {
    if (epi == EPI_STORE) SFB_GO(false, false, EPI_STORE);
    if (epi == EPI_RMW) SFB_GO(false, false, EPI_RMW);
  }
#undef SFB_GO
  return cudaErrorInvalidValue;                       // a combination no step uses
}

}  // namespace sfb
