// The linear head gamma_n of Eq. 2 and the loss of Eq. 3 for LARGE batches (late blocks train at tens of
// thousands of samples, and with 256 auxiliary filters the head input has 1024 features): then
//   logits = p Wf^T + bf,   dp = dlogits Wf,   gWf = dlogits^T p
// are matrix products worth tiling.  fp32 on the CUDA cores (the fp32 configuration's tolerance rules out
// reduced-precision operands); every output element is produced by one thread that adds its products in
// index order, the reduction over the batch in gWf is cut into a fixed number of ranges whose partial results
// are added in range order: results do not depend on scheduling.
#include <algorithm>

#include "nf_internal.h"
#include "nf_ldst.cuh"

namespace {

// C[i][j] (+ z * M * Nn when split) = sum_{k in the z-th range} A[i*sai + k*sak] * B[k*sbk + j*sbj]
// BM x 64 tile per block of 64 threads, BM / 8 x 8 outputs per thread, each ONE fp32 chain in k order.  HK-deep shared-memory steps,
// two buffers: the next step's loads fly while this one is multiplied, one barrier of two warps per step.  Operands whose
// contiguous index is aligned are fetched four values at a time.  A thread's 64 products per four 16-byte reads keep the FMA pipes
// ahead of shared memory; with 256 threads of 4 x 4 or 2 x 4 outputs the reads and barriers set the pace (the head of
// 6366 images with 1024 inputs and 100 classes: 366 -> 309 us, three products).  Two columns share a packed multiply-add, which rounds each
// as fmaf does (the three products 198 -> 188 us; what is left is the latency of the loads, a few warps per SM).

// Fetches an HK x R tile (R rows of index i, HK of k) of `src` into registers and puts it to sm[k][i].
template <int R, int HK>
struct HeadTile {
  static constexpr int kN = R * HK / 4 / 64;  // groups of four per thread
  float v[kN][4];
  __device__ __forceinline__ void fetch(const float* src, long si, long sk, bool vec, int i0, int I, int k0, int k1) {
#pragma unroll
    for (int r = 0; r < kN; ++r) {
      const int e = threadIdx.x + 64 * r;
      // along i: consecutive threads walk i; along k: HK / 4 threads per row of i
      const int i = i0 + (si == 1 ? (e % (R / 4)) * 4 : e / (HK / 4)), k = k0 + (si == 1 ? e / (R / 4) : (e % (HK / 4)) * 4);
      const float* p = src + (long)i * si + (long)k * sk;
      const int left = si == 1 ? I - i : k1 - k;
      const bool in = si == 1 ? k < k1 : i < I;
      if (in && vec && left >= 4) {
        const float4 q = *reinterpret_cast<const float4*>(p);
        v[r][0] = q.x; v[r][1] = q.y; v[r][2] = q.z; v[r][3] = q.w;
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) v[r][u] = in && u < left ? p[(long)u * (si == 1 ? si : sk)] : 0.f;
      }
    }
  }
  __device__ __forceinline__ void put(float (*sm)[R + 4], long si) const {
#pragma unroll
    for (int r = 0; r < kN; ++r) {
      const int e = threadIdx.x + 64 * r;
      if (si == 1) {
        *reinterpret_cast<float4*>(&sm[e / (R / 4)][(e % (R / 4)) * 4]) = make_float4(v[r][0], v[r][1], v[r][2], v[r][3]);
      } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) sm[(e % (HK / 4)) * 4 + u][e / (HK / 4)] = v[r][u];
      }
    }
  }
};

template <int BM>
__global__ void __launch_bounds__(64) head_gemm_kernel(const float* __restrict__ A, long sai, long sak, const float* __restrict__ B,
                                                       long sbk, long sbj, int M, int Nn, int Kd, float* __restrict__ C) {
  nf_pdl_begin();
  constexpr int TM = BM / 8, HK = BM == 64 ? 16 : 32;
  __shared__ __align__(16) float As[2][HK][BM + 4];
  __shared__ __align__(16) float Bs[2][HK][64 + 4];
  const int t = threadIdx.x, tx = t & 7, ty = t >> 3;
  const int i0 = blockIdx.y * BM, j0 = blockIdx.x * 64;
  const int Z = gridDim.z, z = blockIdx.z;
  const int k_lo = (int)((long)Kd * z / Z), k_hi = (int)((long)Kd * (z + 1) / Z);
  const bool va = (((uintptr_t)A & 15) == 0) && (sai == 1 ? sak % 4 == 0 : sak == 1 && sai % 4 == 0 && k_lo % 4 == 0);
  const bool vb = (((uintptr_t)B & 15) == 0) && (sbj == 1 ? sbk % 4 == 0 : sbk == 1 && sbj % 4 == 0 && k_lo % 4 == 0);
  f32x2 acc[TM][4];  // columns 2v and 2v + 1
#pragma unroll
  for (int a = 0; a < TM; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0;
  HeadTile<BM, HK> ta;
  HeadTile<64, HK> tb;
  ta.fetch(A, sai, sak, va, i0, M, k_lo, k_hi);
  tb.fetch(B, sbj, sbk, vb, j0, Nn, k_lo, k_hi);
  ta.put(As[0], sai);
  tb.put(Bs[0], sbj);
  __syncthreads();
  int buf = 0;
  for (int k0 = k_lo; k0 < k_hi; k0 += HK) {
    const bool more = k0 + HK < k_hi;
    if (more) {
      ta.fetch(A, sai, sak, va, i0, M, k0 + HK, k_hi);
      tb.fetch(B, sbj, sbk, vb, j0, Nn, k0 + HK, k_hi);
    }
#pragma unroll 4
    for (int kk = 0; kk < HK; ++kk) {
      float a[TM];
      f32x2 b[4];
#pragma unroll
      for (int u = 0; u < TM; u += 4) {
        const float4 q = *reinterpret_cast<const float4*>(&As[buf][kk][ty * TM + u]);
        a[u] = q.x; a[u + 1] = q.y; a[u + 2] = q.z; a[u + 3] = q.w;
      }
#pragma unroll
      for (int v = 0; v < 8; v += 4) {  // columns tx * 4 .. + 3 and 32 more
        const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][v * 8 + tx * 4]);
        b[v / 2] = q.x; b[v / 2 + 1] = q.y;
      }
#pragma unroll
      for (int u = 0; u < TM; ++u) {
        const f32x2 aa = nf_pack2(a[u], a[u]);
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[u][v] = nf_fma2(aa, b[v], acc[u][v]);
      }
    }
    if (more) {
      ta.put(As[buf ^ 1], sai);
      tb.put(Bs[buf ^ 1], sbj);
    }
    __syncthreads();
    buf ^= 1;
  }
  float* out = C + (size_t)z * M * Nn;
  const bool vo = Nn % 4 == 0 && ((uintptr_t)out & 15) == 0;
#pragma unroll
  for (int u = 0; u < TM; ++u) {
    const int i = i0 + ty * TM + u;
    float r[8];
#pragma unroll
    for (int v = 0; v < 4; ++v) nf_unpack2(acc[u][v], r[2 * v], r[2 * v + 1]);
#pragma unroll
    for (int v = 0; v < 8; v += 4) {
      const int j = j0 + v * 8 + tx * 4;
      float* o = out + (size_t)i * Nn + j;
      if (i < M && vo && j < Nn) {
        *reinterpret_cast<float4*>(o) = make_float4(r[v], r[v + 1], r[v + 2], r[v + 3]);
      } else if (i < M) {
#pragma unroll
        for (int w = 0; w < 4; ++w)
          if (j + w < Nn) o[w] = r[v + w];
      }
    }
  }
}

// out[e] = (bias ? bias[e % Nn] : 0) + part[0][e] + part[1][e] + ... in range order
__global__ void head_finish_kernel(const float* __restrict__ part, int Z, size_t mn, int Nn, const float* __restrict__ bias,
                                   float* __restrict__ out) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= mn) return;
  float s = bias ? bias[e % Nn] : 0.f;
  for (int z = 0; z < Z; ++z) s += part[(size_t)z * mn + e];
  out[e] = s;
}

// One warp per sample: the loss of Eq. 3 on a row of logits, its derivative dlogits, the per-sample loss.
__global__ void __launch_bounds__(256) head_loss_rows_kernel(const float* __restrict__ logits, const int32_t* __restrict__ labels, int N,
                                                             int K, int loss_kind, float* __restrict__ dlogits,
                                                             float* __restrict__ lossn, int32_t* status, int n_scale) {
  nf_pdl_begin();
  const int n = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (n >= N) return;
  const float* l = logits + (size_t)n * K;
  float* g = dlogits + (size_t)n * K;
  int lab = labels[n];
  if (lab < 0 || lab >= K) {
    if (lane == 0) atomicOr(status, NF_ELABEL);
    lab = lab < 0 ? 0 : K - 1;
  }
  if (loss_kind == 1) {
    float se = 0.f;
    const float sc = 2.f / ((float)n_scale * (float)K);
    for (int k = lane; k < K; k += 32) {
      const float e = l[k] - (k == lab ? 1.f : 0.f);
      se = fmaf(e, e, se);
      g[k] = e * sc;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
    if (lane == 0) lossn[n] = se / (float)K;
    return;
  }
  float mx = -INFINITY;
  for (int k = lane; k < K; k += 32) mx = fmaxf(mx, l[k]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  float se = 0.f;
  for (int k = lane; k < K; k += 32) se += expf(l[k] - mx);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
  const float lse = mx + logf(se);
  if (lane == 0) lossn[n] = lse - l[lab];
  const float invN = 1.f / (float)n_scale;
  for (int k = lane; k < K; k += 32) g[k] = (expf(l[k] - lse) - (k == lab ? 1.f : 0.f)) * invN;
}

// part[rb][k] = sum over the rb-th of gridDim.y row ranges of dlogits[n][k] (32 columns x 8 row lanes per block, lanes added in
// order; the ranges are added in range order by head_finish_kernel: with tens of thousands of rows and a few hundred columns
// a single block per 32 columns was the slowest kernel of the head).  Block (0, 0) also reduces the per-sample losses in
// fp64 (256 lanes, then a fixed tree).
__global__ void __launch_bounds__(256) head_colsum_loss_kernel(const float* __restrict__ dl, const float* __restrict__ lossn, int N, int K,
                                                               float* __restrict__ part, float* __restrict__ loss_out, int32_t* status,
                                                               int n_scale) {
  nf_pdl_begin();
  __shared__ float sm[8][33];
  __shared__ double sd[256];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int k = blockIdx.x * 32 + tx;
  const int n0 = (int)((long)N * blockIdx.y / gridDim.y), n1 = (int)((long)N * (blockIdx.y + 1) / gridDim.y);
  float s = 0.f;
  if (k < K)
    for (int n = n0 + ty; n < n1; n += 8) s += dl[(size_t)n * K + k];
  sm[ty][tx] = s;
  __syncthreads();
  if (ty == 0 && k < K) {
    float tsum = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) tsum += sm[j][tx];
    part[(size_t)blockIdx.y * K + k] = tsum;
  }
  if (blockIdx.x == 0 && blockIdx.y == 0) {
    double a = 0.0;
    for (int n = threadIdx.x; n < N; n += 256) a += (double)lossn[n];
    sd[threadIdx.x] = a;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
      if (threadIdx.x < o) sd[threadIdx.x] += sd[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      const float L = (float)(sd[0] / (double)n_scale);
      *loss_out = L;
      if (!isfinite(L)) atomicOr(status, NF_ENONFINITE);
    }
  }
}

// first arg-max of each row of logits, one warp per sample
__global__ void __launch_bounds__(256) head_argmax_rows_kernel(const float* __restrict__ logits, int N, int K, int32_t* __restrict__ pred) {
  nf_pdl_begin();
  const int n = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (n >= N) return;
  const float* l = logits + (size_t)n * K;
  float best = -INFINITY;
  int arg = 0x7fffffff;
  for (int k = lane; k < K; k += 32)
    if (l[k] > best) { best = l[k]; arg = k; }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oa = __shfl_xor_sync(0xffffffffu, arg, o);
    if (ob > best || (ob == best && oa < arg)) { best = ob; arg = oa; }
  }
  if (lane == 0) pred[n] = arg;
}

int gemm(const float* A, long sai, long sak, const float* B, long sbk, long sbj, int M, int Nn, int Kd, int Z, float* C) {
  // tiles of 64 rows where they fill the chip three times over, else of 32
  const long big = (long)((Nn + 63) / 64) * ((M + 63) / 64) * Z;
  if (big >= 444)
    nf_launch(head_gemm_kernel<64>, dim3((Nn + 63) / 64, (M + 63) / 64, Z), 64, 0, A, sai, sak, B, sbk, sbj, M, Nn, Kd, C);
  else
    nf_launch(head_gemm_kernel<32>, dim3((Nn + 63) / 64, (M + 31) / 32, Z), 64, 0, A, sai, sak, B, sbk, sbj, M, Nn, Kd, C);
  NF_LAUNCHED();
  return NF_OK;
}

}  // namespace

bool nf_head_is_large(int N, int D, int K) { return (double)N * D * K >= (double)(1 << 24); }

int nf_head_logits(const float* p, int N, int D, int K, const float* Wf, const float* bf, float* logits, float* scratch) {
  // logits[n][k] = bf[k] + sum_d p[n][d] Wf[k][d]
  int rc = gemm(p, D, 1, Wf, 1, D, N, K, D, 1, scratch);
  if (rc != NF_OK) return rc;
  const size_t mn = (size_t)N * K;
  nf_launch(head_finish_kernel, (unsigned)((mn + 255) / 256), 256, 0, scratch, 1, mn, K, bf, logits);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_head_predict(const float* logits, int N, int K, int32_t* pred) {
  nf_launch(head_argmax_rows_kernel, (N + 7) / 8, 256, 0, logits, N, K, pred);
  NF_LAUNCHED();
  return NF_OK;
}

size_t nf_head_scratch_floats(int N, int D, int K) {
  const size_t a = (size_t)N * K, b = (size_t)K * D;  // logits before the bias; at least one range of gWf
  return a > b ? a : b;
}

int nf_head_step(const float* p, const int32_t* labels, int N, int D, int K, const float* Wf, const float* bf, float* logits,
                 float* dlogits, float* dp, float* lossn, int32_t* status, int loss_kind, float* gWf, float* gbf, float* loss_out,
                 float* scratch, size_t scratch_floats, int n_scale) {
  if (scratch_floats < nf_head_scratch_floats(N, D, K)) return NF_ENOWS;
  int rc = nf_head_logits(p, N, D, K, Wf, bf, logits, scratch);
  if (rc != NF_OK) return rc;
  nf_launch(head_loss_rows_kernel, (N + 7) / 8, 256, 0, logits, labels, N, K, loss_kind, dlogits, lossn, status, n_scale);
  NF_LAUNCHED();
  // dp[n][d] = sum_k dlogits[n][k] Wf[k][d]
  if ((rc = gemm(dlogits, K, 1, Wf, D, 1, N, D, K, 1, dp)) != NF_OK) return rc;
  // gWf[k][d] = sum_n dlogits[n][k] p[n][d], the batch cut into Z ranges
  const size_t kd = (size_t)K * D;
  int Z = (int)std::min<size_t>(scratch_floats / kd, 64);
  const int tiles = ((D + 63) / 64) * ((K + 63) / 64);
  Z = std::min(Z, std::max(1, 592 / tiles));  // about four blocks per SM
  Z = std::min(Z, std::max(1, N / 256));
  if (Z < 1) Z = 1;
  if ((rc = gemm(dlogits, 1, K, p, D, 1, K, D, N, Z, scratch)) != NF_OK) return rc;
  nf_launch(head_finish_kernel, (unsigned)((kd + 255) / 256), 256, 0, scratch, Z, kd, D, nullptr, gWf);
  NF_LAUNCHED();
  // gbf[k] = sum_n dlogits[n][k]: row ranges in parallel (the scratch is free again), then the ranges in order
  int RB = std::max(1, std::min(64, N / 128));
  if ((size_t)RB * K > scratch_floats) RB = 1;
  nf_launch(head_colsum_loss_kernel, dim3((K + 31) / 32, RB), 256, 0, dlogits, lossn, N, K, scratch, loss_out, status, n_scale);
  NF_LAUNCHED();
  nf_launch(head_finish_kernel, (unsigned)((K + 255) / 256), 256, 0, scratch, RB, (size_t)K, K, nullptr, gbf);
  NF_LAUNCHED();
  return NF_OK;
}
