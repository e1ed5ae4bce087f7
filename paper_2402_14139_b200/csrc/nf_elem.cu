// Memory-bound kernels of the local-layer step: BatchNorm statistics / apply / backward, pooling,
// the linear + softmax cross-entropy head, momentum SGD and the cache gather.  Storage fp32 or
// bf16, arithmetic fp32, cross-block sums finished in fp64 in a fixed order (deterministic).
#include <algorithm>
#include <type_traits>
#include "nf_internal.h"
#include "nf_ldst.cuh"

namespace {

__host__ __device__ inline int pow2ceil_cap256(int c) {
  int l = 1;
  while (l < c && l < 256) l <<= 1;
  return l;
}

// dz at full-resolution pixel p = ((n*Ho)+i)*Wo+j, channel c: gradient that reaches the BatchNorm
// output through ReLU and the optional 2x2 max-pool (first maximum in scan order wins).
template <typename T>
__device__ __forceinline__ float dz_at(const T* __restrict__ y, const T* __restrict__ da, size_t p, int c, int C,
                                       int Ho, int Wo, int pool, float sc, float sh, const T* __restrict__ skip = nullptr) {
  const float z = fmaf(ldf(y, p * C + c), sc, sh) + (skip ? ldf(skip, p * C + c) : 0.f);
  if (!(z > 0.f)) return 0.f;
  if (!pool) return ldf(da, p * C + c);
  const int j = (int)(p % Wo), i = (int)((p / Wo) % Ho);
  const size_t n = p / ((size_t)Wo * Ho);
  const int i0 = i & ~1, j0 = j & ~1;
  float best = -1.f;
  int arg = 0;
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    const size_t q = ((n * Ho + i0 + (d >> 1)) * Wo + j0 + (d & 1)) * C + c;
    const float r = rnd<T>(fmaxf(fmaf(ldf(y, q), sc, sh) + (skip ? ldf(skip, q) : 0.f), 0.f));
    if (r > best) { best = r; arg = d; }
  }
  if (arg != (i - i0) * 2 + (j - j0)) return 0.f;
  return ldf(da, ((n * (Ho / 2) + i / 2) * (Wo / 2) + j / 2) * C + c);
}

struct StatsFn {  // (v, v^2) of a stored tensor
  template <typename T>
  __device__ __forceinline__ void operator()(const T* src, const T*, size_t p, int c, int C, float& a, float& b) const {
    const float v = ldf(src, p * C + c);
    a = v;
    b = v * v;
  }
};

struct BnBwdFn {  // (dz, dz*xhat)
  int Ho, Wo, pool;
  const float *scale, *shift, *mu, *invstd;
  const void* skip;  // identity shortcut added before the ReLU, or NULL
  template <typename T>
  __device__ __forceinline__ void operator()(const T* y, const T* da, size_t p, int c, int C, float& a, float& b) const {
    const float dz = dz_at(y, da, p, c, C, Ho, Wo, pool, scale[c], shift[c], (const T*)skip);
    a = dz;
    b = dz * (ldf(y, p * C + c) - mu[c]) * invstd[c];
  }
};

// red[(block*2 + k)*C + c] = sum over the block's pixel range of value k at channel c
template <typename T, typename Fn>
__global__ void __launch_bounds__(256) channel_reduce_kernel(const T* __restrict__ s0, const T* __restrict__ s1, size_t P,
                                                             int C, Fn fn, float* __restrict__ red) {
  nf_pdl_begin();
  __shared__ float sm[2][256];
  const int lanes = pow2ceil_cap256(C), planes = 256 / lanes;
  const int lc = threadIdx.x % lanes, pl = threadIdx.x / lanes;
  const size_t p0 = P * blockIdx.x / gridDim.x, p1 = P * (blockIdx.x + 1) / gridDim.x;
  for (int c0 = 0; c0 < C; c0 += lanes) {
    const int c = c0 + lc;
    float a = 0.f, b = 0.f;
    if (c < C)
      for (size_t p = p0 + pl; p < p1; p += planes) {
        float u, v;
        fn(s0, s1, p, c, C, u, v);
        a += u;
        b += v;
      }
    sm[0][threadIdx.x] = a;
    sm[1][threadIdx.x] = b;
    __syncthreads();
    if (pl == 0 && c < C) {
      float ta = 0.f, tb = 0.f;
      for (int q = 0; q < planes; ++q) {
        ta += sm[0][q * lanes + lc];
        tb += sm[1][q * lanes + lc];
      }
      red[((size_t)blockIdx.x * 2 + 0) * C + c] = ta;
      red[((size_t)blockIdx.x * 2 + 1) * C + c] = tb;
    }
    __syncthreads();
  }
}


// Sums the per-block partials of 8 consecutive channels in fp64, in a fixed order: block of 1024 threads = 8 channels x 128 lanes
// over the partials.  Returns the two totals to one thread per channel (t = 32 * channel of the block).
// These kernels are one dependent chain: the start-up, a trip to L2, a reduction, and the fetch of their own cold instructions.
// So the code is kept short (an 8-fold unrolled form with predicated loads ran 3 us slower than it is now) and the lanes many.
constexpr int kRedCh = 8, kRedThreads = 1024;
__device__ __forceinline__ void reduce_partials8(const float* __restrict__ red, int nb, int C, double& S, double& Q) {
  __shared__ double sm[2][32][kRedCh + 1];
  const int t = threadIdx.x, ch = t & 7;
  const int c = blockIdx.x * kRedCh + ch;
  double a = 0.0, b = 0.0;
  if (c < C) {
    const float* r = red + (size_t)(t >> 3) * 2 * C + c;
#pragma unroll 1
    for (int k = t >> 3; k < nb; k += 2 * 128, r += (size_t)2 * 128 * 2 * C) {
      const bool two = k + 128 < nb;
      const float u0 = r[0], v0 = r[C], u1 = two ? r[(size_t)128 * 2 * C] : 0.f, v1 = two ? r[(size_t)128 * 2 * C + C] : 0.f;
      a += (double)u0 + (double)u1;
      b += (double)v0 + (double)v1;
    }
  }
#pragma unroll 1
  for (int o = 8; o < 32; o <<= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if ((t & 31) < 8) {
    sm[0][t >> 5][ch] = a;
    sm[1][t >> 5][ch] = b;
  }
  __syncthreads();
  S = 0.0;
  Q = 0.0;
  if (t < 32 * kRedCh) {
    S = sm[0][t & 31][t >> 5];
    Q = sm[1][t & 31][t >> 5];
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
      S += __shfl_xor_sync(0xffffffffu, S, o);
      Q += __shfl_xor_sync(0xffffffffu, Q, o);
    }
  }
}
// channel whose totals thread t holds, or C
__device__ __forceinline__ int reduced_channel(int C) {
  const int c = blockIdx.x * kRedCh + (int)(threadIdx.x >> 5);
  return (threadIdx.x & 31) == 0 && threadIdx.x < 32 * kRedCh && c < C ? c : C;
}

__global__ void bn_finalize_kernel(const float* __restrict__ red, int nb, int C, double M, const float* __restrict__ gamma,
                                   const float* __restrict__ beta, float eps, float bnm, float* scale, float* shift,
                                   float* mu, float* invstd, float* rmean, float* rvar) {
  nf_pdl_begin();
  double S, Q;
  reduce_partials8(red, nb, C, S, Q);
  const int c = reduced_channel(C);
  if (c >= C) return;
  const double m = S / M;
  double v = Q / M - m * m;
  if (v < 0.0) v = 0.0;
  const double is = 1.0 / sqrt(v + (double)eps);
  const float sc = (float)((double)gamma[c] * is);
  scale[c] = sc;
  shift[c] = (float)((double)beta[c] - m * (double)gamma[c] * is);
  mu[c] = (float)m;
  invstd[c] = (float)is;
  if (rmean) {
    rmean[c] = (float)((1.0 - bnm) * (double)rmean[c] + (double)bnm * m);
    const double unb = M > 1.0 ? v * M / (M - 1.0) : v;
    rvar[c] = (float)((1.0 - bnm) * (double)rvar[c] + (double)bnm * unb);
  }
}

// Data-parallel BatchNorm: a rank turns its per-block partials into per-channel totals (fp64, [2][C]) that the
// ranks add up; the statistics and the backward sums are then finished from the totals of the whole batch.
__global__ void partial_totals_kernel(const float* __restrict__ red, int nb, int C, double* __restrict__ tot) {
  nf_pdl_begin();
  double S, Q;
  reduce_partials8(red, nb, C, S, Q);
  const int c = reduced_channel(C);
  if (c >= C) return;
  tot[c] = S;
  tot[C + c] = Q;
}

__global__ void bn_finalize_tot_kernel(const double* __restrict__ tot, int C, double M, const float* __restrict__ gamma,
                                       const float* __restrict__ beta, float eps, float bnm, float* scale, float* shift, float* mu,
                                       float* invstd, float* rmean, float* rvar) {
  nf_pdl_begin();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= C) return;
  const double m = tot[c] / M;
  double v = tot[C + c] / M - m * m;
  if (v < 0.0) v = 0.0;
  const double is = 1.0 / sqrt(v + (double)eps);
  scale[c] = (float)((double)gamma[c] * is);
  shift[c] = (float)((double)beta[c] - m * (double)gamma[c] * is);
  mu[c] = (float)m;
  invstd[c] = (float)is;
  rmean[c] = (float)((1.0 - bnm) * (double)rmean[c] + (double)bnm * m);
  const double unb = M > 1.0 ? v * M / (M - 1.0) : v;
  rvar[c] = (float)((1.0 - bnm) * (double)rvar[c] + (double)bnm * unb);
}

// the gradients of gamma and beta are divided by the number of ranks: the sum over ranks that follows restores them
__global__ void bn_bwd_finalize_tot_kernel(const double* __restrict__ tot, int C, double inv_world, float* sdz, float* sdzx, float* gg,
                                           float* gb) {
  nf_pdl_begin();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= C) return;
  sdz[c] = (float)tot[c];
  sdzx[c] = (float)tot[C + c];
  gb[c] = (float)(tot[c] * inv_world);
  gg[c] = (float)(tot[C + c] * inv_world);
}

__global__ void bn_eval_coeffs_kernel(int C, const float* gamma, const float* beta, float eps, const float* rmean,
                                      const float* rvar, float* scale, float* shift) {
  nf_pdl_begin();
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= C) return;
  const double is = 1.0 / sqrt((double)rvar[c] + (double)eps);
  scale[c] = (float)((double)gamma[c] * is);
  shift[c] = (float)((double)beta[c] - (double)rmean[c] * (double)gamma[c] * is);
}

// out[n,ia,ja,c] = max over the pool window (or the single pixel) of ReLU(y*scale+shift)
template <typename T>
__global__ void bn_apply_kernel(const T* __restrict__ y, int Ho, int Wo, int C, int pool, const float* __restrict__ scale,
                                const float* __restrict__ shift, size_t total, T* __restrict__ out, const T* __restrict__ skip) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int c = (int)(e % C);
  const size_t q = e / C;
  const float sc = scale[c], sh = shift[c];
  if (!pool) {
    stf(out, e, fmaxf(fmaf(ldf(y, e), sc, sh) + (skip ? ldf(skip, e) : 0.f), 0.f));
    return;
  }
  const int Wa = Wo / 2, Ha = Ho / 2;
  const int ja = (int)(q % Wa), ia = (int)((q / Wa) % Ha);
  const size_t n = q / ((size_t)Wa * Ha);
  float best = 0.f;
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    const size_t src = ((n * Ho + 2 * ia + (d >> 1)) * Wo + 2 * ja + (d & 1)) * C + c;
    best = fmaxf(best, fmaf(ldf(y, src), sc, sh) + (skip ? ldf(skip, src) : 0.f));
  }
  stf(out, e, best);
}

__device__ __forceinline__ void bin_range(int u, int H, int& lo, int& hi) {
  lo = (u * H) / 2;
  hi = ((u + 1) * H + 1) / 2;
}

// p[n][f*4 + u*2 + v] = mean of h over bin (u,v);  one block per (n, bin)
// the same for bins of at most 16 pixels: one thread per output p[n][f*4 + bin] (consecutive threads = consecutive channels)
template <typename T>
__global__ void avgpool_small_kernel(const T* __restrict__ h, int Ha, int Wa, int F, size_t total, float* __restrict__ p) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int f = (int)(e % F), bin = (int)((e / F) % 4);
  const size_t n = e / ((size_t)4 * F);
  int i0, i1, j0, j1;
  bin_range(bin / 2, Ha, i0, i1);
  bin_range(bin % 2, Wa, j0, j1);
  float a = 0.f;
  for (int i = i0; i < i1; ++i)
    for (int j = j0; j < j1; ++j) a += ldf(h, ((n * Ha + i) * Wa + j) * F + f);
  p[n * 4 * F + (size_t)f * 4 + bin] = a / (float)((i1 - i0) * (j1 - j0));
}

template <typename T>
__global__ void __launch_bounds__(256) avgpool_kernel(const T* __restrict__ h, int Ha, int Wa, int F, float* __restrict__ p) {
  nf_pdl_begin();
  __shared__ float sm[256];
  const int n = blockIdx.x / 4, bin = blockIdx.x % 4, u = bin / 2, v = bin % 2;
  int i0, i1, j0, j1;
  bin_range(u, Ha, i0, i1);
  bin_range(v, Wa, j0, j1);
  const int bw = j1 - j0, cnt = (i1 - i0) * bw;
  const int lanes = pow2ceil_cap256(F), planes = 256 / lanes;
  const int lf = threadIdx.x % lanes, pl = threadIdx.x / lanes;
  for (int f0 = 0; f0 < F; f0 += lanes) {
    const int f = f0 + lf;
    float a = 0.f;
    if (f < F)
      for (int k = pl; k < cnt; k += planes) {
        const int i = i0 + k / bw, j = j0 + k % bw;
        a += ldf(h, (((size_t)n * Ha + i) * Wa + j) * F + f);
      }
    sm[threadIdx.x] = a;
    __syncthreads();
    if (pl == 0 && f < F) {
      float t = 0.f;
      for (int q = 0; q < planes; ++q) t += sm[q * lanes + lf];
      p[(size_t)n * 4 * F + f * 4 + bin] = t / (float)cnt;
    }
    __syncthreads();
  }
}

// Max-pool down-sampling: p[n][f*4 + bin] = max of h over bin (u,v), parg = position i*Wa+j of the FIRST maximum in
// row-major order; one block per (n, bin).  A thread scans its pixels in increasing order and keeps the first
// maximum; the lanes of a filter are then combined preferring the larger value, the smaller position on ties.
template <typename T>
__global__ void __launch_bounds__(256) auxmax_kernel(const T* __restrict__ h, int Ha, int Wa, int F, float* __restrict__ p,
                                                     int32_t* __restrict__ parg) {
  nf_pdl_begin();
  __shared__ float sv[256];
  __shared__ int si[256];
  const int n = blockIdx.x / 4, bin = blockIdx.x % 4, u = bin / 2, v = bin % 2;
  int i0, i1, j0, j1;
  bin_range(u, Ha, i0, i1);
  bin_range(v, Wa, j0, j1);
  const int bw = j1 - j0, cnt = (i1 - i0) * bw;
  const int lanes = pow2ceil_cap256(F), planes = 256 / lanes;
  const int lf = threadIdx.x % lanes, pl = threadIdx.x / lanes;
  for (int f0 = 0; f0 < F; f0 += lanes) {
    const int f = f0 + lf;
    float best = -INFINITY;
    int at = 0x7fffffff;
    if (f < F)
      for (int k = pl; k < cnt; k += planes) {
        const int i = i0 + k / bw, j = j0 + k % bw;
        const float t = ldf(h, (((size_t)n * Ha + i) * Wa + j) * F + f);
        if (t > best) { best = t; at = i * Wa + j; }
      }
    sv[threadIdx.x] = best;
    si[threadIdx.x] = at;
    __syncthreads();
    if (pl == 0 && f < F) {
      float b = sv[lf];
      int a = si[lf];
      for (int q = 1; q < planes; ++q) {
        const float t = sv[q * lanes + lf];
        const int ti = si[q * lanes + lf];
        if (t > b || (t == b && ti < a)) { b = t; a = ti; }
      }
      p[(size_t)n * 4 * F + f * 4 + bin] = b;
      parg[(size_t)n * 4 * F + f * 4 + bin] = a;
    }
    __syncthreads();
  }
}

// dh[n,i,j,f] = 1[h>0] * sum over the bins whose maximum sits at (i,j) of dp[n][f*4+bin]
template <typename T>
__global__ void dh_max_kernel(const T* __restrict__ h, const float* __restrict__ dp, const int32_t* __restrict__ parg, int Ha, int Wa,
                              int F, size_t total, T* __restrict__ dh) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int f = (int)(e % F);
  const size_t q = e / F;
  const int j = (int)(q % Wa), i = (int)((q / Wa) % Ha);
  const size_t n = q / ((size_t)Wa * Ha);
  float g = 0.f;
  if (ldf(h, e) > 0.f) {
    const int pos = i * Wa + j;
#pragma unroll
    for (int b = 0; b < 4; ++b)
      if (parg[n * 4 * F + f * 4 + b] == pos) g += dp[n * 4 * F + f * 4 + b];
  }
  stf(dh, e, g);
}

__device__ __forceinline__ float block_reduce(float v, float* sm, bool is_max) {
  const int t = threadIdx.x;
  sm[t] = v;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (t < s) sm[t] = is_max ? fmaxf(sm[t], sm[t + s]) : sm[t] + sm[t + s];
    __syncthreads();
  }
  const float r = sm[0];
  __syncthreads();
  return r;
}

// one block per sample: logits, softmax cross-entropy, dlogits = (softmax-onehot)/N, dp = dlogits * Wf
__global__ void __launch_bounds__(256) fc_ce_kernel(const float* __restrict__ p, const int32_t* __restrict__ labels, int N,
                                                    int D, int K, const float* __restrict__ Wf, const float* __restrict__ bf,
                                                    float* __restrict__ logits, float* __restrict__ dlogits,
                                                    float* __restrict__ dp, float* __restrict__ lossn, int32_t* status,
                                                    int loss_kind, int n_scale) {
  nf_pdl_begin();
  extern __shared__ float dyn[];
  float* ps = dyn;          // [D]
  float* ls = dyn + D;      // [K]
  __shared__ float red[256];
  const int n = blockIdx.x, t = threadIdx.x;
  for (int d = t; d < D; d += 256) ps[d] = p[(size_t)n * D + d];
  __syncthreads();
  float mx = -INFINITY;
  for (int k = t; k < K; k += 256) {
    float s = bf[k];
    const float* w = Wf + (size_t)k * D;
    for (int d = 0; d < D; ++d) s = fmaf(w[d], ps[d], s);
    ls[k] = s;
    logits[(size_t)n * K + k] = s;
    mx = fmaxf(mx, s);
  }
  mx = block_reduce(mx, red, true);
  int lab = labels[n];
  if (lab < 0 || lab >= K) {
    if (t == 0) atomicOr(status, NF_ELABEL);
    lab = lab < 0 ? 0 : K - 1;
  }
  if (loss_kind == 1) {
    // mean squared error against the one-hot target: lossn = sum_k e^2 / K, dlogits = 2 e / (N K)
    float se = 0.f;
    const float sc = 2.f / ((float)n_scale * (float)K);
    for (int k = t; k < K; k += 256) {
      const float e = ls[k] - (k == lab ? 1.f : 0.f);
      se = fmaf(e, e, se);
      ls[k] = e * sc;
      dlogits[(size_t)n * K + k] = e * sc;
    }
    se = block_reduce(se, red, false);
    if (t == 0) lossn[n] = se / (float)K;
  } else {
    float se = 0.f;
    for (int k = t; k < K; k += 256) se += expf(ls[k] - mx);
    se = block_reduce(se, red, false);
    const float lse = mx + logf(se);
    if (t == 0) lossn[n] = lse - ls[lab];
    const float invN = 1.f / (float)n_scale;
    for (int k = t; k < K; k += 256) {
      const float g = (expf(ls[k] - lse) - (k == lab ? 1.f : 0.f)) * invN;
      ls[k] = g;
      dlogits[(size_t)n * K + k] = g;
    }
  }
  __syncthreads();
  // dp[d] = sum_k g[k] Wf[k][d]: the classes are cut into G contiguous ranges (G = 256 / D lanes per d when D <= 128),
  // every range is summed in index order and the G range sums are added in range order
  const int G = D <= 128 ? 256 / D : 1;
  if (G > 1) {
    const int d = t % D, kg = t / D;
    float s = 0.f;
    if (kg < G) {
      const int per = (K + G - 1) / G, k0 = kg * per, k1 = min(K, k0 + per);
      int k = k0;
      for (; k + 3 < k1; k += 4) {
        const float w0 = Wf[(size_t)k * D + d], w1 = Wf[(size_t)(k + 1) * D + d], w2 = Wf[(size_t)(k + 2) * D + d],
                    w3 = Wf[(size_t)(k + 3) * D + d];
        s = fmaf(ls[k], w0, s);
        s = fmaf(ls[k + 1], w1, s);
        s = fmaf(ls[k + 2], w2, s);
        s = fmaf(ls[k + 3], w3, s);
      }
      for (; k < k1; ++k) s = fmaf(ls[k], Wf[(size_t)k * D + d], s);
    }
    red[t] = s;
    __syncthreads();
    if (t < D) {
      float tot = 0.f;
      for (int g = 0; g < G; ++g) tot += red[g * D + t];
      dp[(size_t)n * D + t] = tot;
    }
  } else {
    for (int d = t; d < D; d += 256) {
      float s = 0.f;
      for (int k = 0; k < K; ++k) s = fmaf(ls[k], Wf[(size_t)k * D + d], s);
      dp[(size_t)n * D + d] = s;
    }
  }
}


// one block per sample: logits = Wf p + bf (optionally stored) and the class = first arg-max
__global__ void __launch_bounds__(256) fc_predict_kernel(const float* __restrict__ p, int D, int K, const float* __restrict__ Wf,
                                                         const float* __restrict__ bf, float* __restrict__ logits,
                                                         int32_t* __restrict__ pred) {
  nf_pdl_begin();
  extern __shared__ float dyn[];
  float* ps = dyn;
  __shared__ float bv[256];
  __shared__ int bi[256];
  const int n = blockIdx.x, t = threadIdx.x;
  for (int d = t; d < D; d += 256) ps[d] = p[(size_t)n * D + d];
  __syncthreads();
  float best = -INFINITY;
  int arg = 0x7fffffff;
  for (int k = t; k < K; k += 256) {
    float s = bf[k];
    const float* w = Wf + (size_t)k * D;
    for (int d = 0; d < D; ++d) s = fmaf(w[d], ps[d], s);
    if (logits) logits[(size_t)n * K + k] = s;
    if (s > best) { best = s; arg = k; }   // k ascending within a thread: keeps the first maximum
  }
  bv[t] = best;
  bi[t] = arg;
  __syncthreads();
  for (int s2 = 128; s2 > 0; s2 >>= 1) {
    if (t < s2 && (bv[t + s2] > bv[t] || (bv[t + s2] == bv[t] && bi[t + s2] < bi[t]))) {
      bv[t] = bv[t + s2];
      bi[t] = bi[t + s2];
    }
    __syncthreads();
  }
  if (t == 0) pred[n] = bi[0];
}

// dh[n,i,j,f] = 1[h>0] * sum over bins containing (i,j) of dp[n][f*4+bin] / |bin|
template <typename T>
__global__ void dh_kernel(const T* __restrict__ h, const float* __restrict__ dp, int Ha, int Wa, int F, size_t total,
                          T* __restrict__ dh) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int f = (int)(e % F);
  const size_t q = e / F;
  const int j = (int)(q % Wa), i = (int)((q / Wa) % Ha);
  const size_t n = q / ((size_t)Wa * Ha);
  float g = 0.f;
  if (ldf(h, e) > 0.f) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      int i0, i1;
      bin_range(u, Ha, i0, i1);
      if (i < i0 || i >= i1) continue;
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        int j0, j1;
        bin_range(v, Wa, j0, j1);
        if (j < j0 || j >= j1) continue;
        g += dp[n * 4 * F + f * 4 + u * 2 + v] / (float)((i1 - i0) * (j1 - j0));
      }
    }
  }
  stf(dh, e, g);
}

__global__ void sum_partials_kernel(const float* __restrict__ red, int nb, int C, float* __restrict__ out) {
  nf_pdl_begin();
  double S, Q;
  reduce_partials8(red, nb, C, S, Q);
  const int c = reduced_channel(C);
  if (c >= C) return;
  out[c] = (float)S;
}

__global__ void bn_bwd_finalize_kernel(const float* __restrict__ red, int nb, int C, float* sdz, float* sdzx, float* gg,
                                       float* gb) {
  nf_pdl_begin();
  double a, b;
  reduce_partials8(red, nb, C, a, b);
  const int c = reduced_channel(C);
  if (c >= C) return;
  sdz[c] = (float)a;
  sdzx[c] = (float)b;
  gb[c] = (float)a;
  gg[c] = (float)b;
}

// dy = gamma*invstd * (dz - sum(dz)/M - xhat * sum(dz*xhat)/M)
template <typename T>
__global__ void bn_bwd_apply_kernel(const T* __restrict__ y, const T* __restrict__ da, int Ho, int Wo, int C, int pool,
                                    const float* __restrict__ scale, const float* __restrict__ shift,
                                    const float* __restrict__ mu, const float* __restrict__ invstd,
                                    const float* __restrict__ sdz, const float* __restrict__ sdzx, float invM,
                                    size_t total, T* __restrict__ dy, const T* __restrict__ skip) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int c = (int)(e % C);
  const size_t p = e / C;
  const float dz = dz_at(y, da, p, c, C, Ho, Wo, pool, scale[c], shift[c], skip);
  const float xh = (ldf(y, e) - mu[c]) * invstd[c];
  stf(dy, e, scale[c] * (dz - sdz[c] * invM - xh * sdzx[c] * invM));
}

// dz = da * 1[BN(y) + skip > 0], routed through the optional max-pool: the gradient at the layer's BatchNorm output, which is
// also the gradient at a trainable shortcut added there
template <typename T>
__global__ void write_dz_kernel(const T* __restrict__ y, const T* __restrict__ da, int Ho, int Wo, int C, int pool,
                                const float* __restrict__ scale, const float* __restrict__ shift, const T* __restrict__ skip,
                                size_t total, T* __restrict__ dz) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const int c = (int)(e % C);
  stf(dz, e, dz_at(y, da, e / C, c, C, Ho, Wo, pool, scale[c], shift[c], skip));
}

// xpad[p][0..Cp) = (x[p][0..C), 0, ...): one thread per 8-channel chunk (16 bytes) of the padded pixel, C <= 8
__global__ void pad_channels_kernel(const bf16* __restrict__ x, size_t P, int C, int Cp8, uint4* __restrict__ xpad) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= P * Cp8) return;
  const size_t p = e / Cp8;
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  if (e % Cp8 == 0) {
    unsigned short h[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int c = 0; c < C; ++c) h[c] = __bfloat16_as_ushort(x[p * C + c]);
    v = make_uint4(h[0] | ((uint32_t)h[1] << 16), h[2] | ((uint32_t)h[3] << 16), h[4] | ((uint32_t)h[5] << 16), h[6] | ((uint32_t)h[7] << 16));
  }
  xpad[e] = v;
}
__global__ void pad_weights_kernel(const bf16* __restrict__ w, size_t rows, int C, int Cp, bf16* __restrict__ wpad) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= rows * Cp) return;
  const int c = (int)(e % Cp);
  wpad[e] = c < C ? w[(e / Cp) * C + c] : __float2bfloat16(0.f);
}
__global__ void unpad_grad_kernel(const float* __restrict__ gwpad, size_t rows, int C, int Cp, float* __restrict__ gw) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= rows * C) return;
  gw[e] = gwpad[(e / C) * Cp + e % C];
}

// out[i] = sum over the splits of part[k][i]: eight chains (split k in chain k % 8) in index order, the chains added in order.  V
// consecutive elements per thread (4: 16-byte loads); LN = 8: a thread per chain, for many splits of few elements (148 of
// 36 864); LN = 1: one thread runs all chains, for fewer than 16 splits (at most two terms each) of many elements.  A: type of the
// chains (double: partials whose own error is below a rounding of the sum).
template <int V, int LN, typename A>
__global__ void __launch_bounds__(256) sum_parts_kernel(const float* __restrict__ part, int splits, size_t n, float* __restrict__ out) {
  nf_pdl_begin();
  constexpr int kCols = 256 / LN;
  __shared__ A sm[LN][kCols * V];
  const int tx = threadIdx.x % kCols, ty = threadIdx.x / kCols;
  const size_t i = ((size_t)blockIdx.x * kCols + tx) * V;
  A s[V];
#pragma unroll
  for (int e = 0; e < V; ++e) s[e] = 0;
  auto term = [&](int k, float(&v)[V]) {
    const float* src = part + (size_t)k * n + i;
    if constexpr (V == 4) {
      const float4 w = *reinterpret_cast<const float4*>(src);
      v[0] = w.x; v[1] = w.y; v[2] = w.z; v[3] = w.w;
    } else {
      v[0] = *src;
    }
  };
  if constexpr (LN > 1) {
    if (i < n) {
#pragma unroll 8
      for (int k = ty; k < splits; k += LN) {
        float v[V];
        term(k, v);
#pragma unroll
        for (int e = 0; e < V; ++e) s[e] += v[e];
      }
    }
#pragma unroll
    for (int e = 0; e < V; ++e) sm[ty][tx * V + e] = s[e];
    __syncthreads();
    if (threadIdx.x < kCols * V) {  // one thread per element
      A v = sm[0][threadIdx.x];
#pragma unroll
      for (int l = 1; l < LN; ++l) v += sm[l][threadIdx.x];
      const size_t o = (size_t)blockIdx.x * kCols * V + threadIdx.x;
      if (o < n) out[o] = (float)v;
    }
  } else if (i < n) {
    const int heads = splits < 8 ? splits : 8;
#pragma unroll 4
    for (int k = 0; k < heads; ++k) {
      float v[V], w[V];
      term(k, v);
#pragma unroll
      for (int e = 0; e < V; ++e) w[e] = 0.f;
      if (k + 8 < splits) term(k + 8, w);
#pragma unroll
      for (int e = 0; e < V; ++e) s[e] += (A)v[e] + (A)w[e];
    }
    if constexpr (V == 4) {
      *reinterpret_cast<float4*>(out + i) = make_float4((float)s[0], (float)s[1], (float)s[2], (float)s[3]);
    } else {
      out[i] = (float)s[0];
    }
  }
}

__global__ void unpad_grad_mirrored_kernel(const float* __restrict__ gwpad, int Co, int C, int Cp, float* __restrict__ gw) {
  nf_pdl_begin();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= 9 * Co * C) return;
  const int c = e % C, co = (e / C) % Co, tap = e / (C * Co);
  gw[e] = gwpad[((size_t)(8 - tap) * Cp + c) * Co + co];
}

// Momentum SGD over up to kSgdMaxArenas parameter arenas in one launch (all layers of a block).  An arena is a multiple
// of 64 floats and 256-byte aligned, so every thread owns four consecutive elements: 16-byte loads of value, momentum and
// gradient, 16-byte stores of value and momentum, one 8-byte store of the four bf16 copies.  Blocks are dealt to arenas
// through the table of first-block indices.
__global__ void __launch_bounds__(256) sgd_multi_kernel(const SgdTable tb, float lr, float mu) {
  nf_pdl_begin();
  int a = 0;
  while (a + 1 < tb.count && (int)blockIdx.x >= tb.first_block[a + 1]) ++a;
  const size_t i4 = (size_t)(blockIdx.x - tb.first_block[a]) * blockDim.x + threadIdx.x;
  if (i4 * 4 >= tb.n[a]) return;
  const float4 g = reinterpret_cast<const float4*>(tb.grad[a])[i4];
  float4 m = reinterpret_cast<const float4*>(tb.mom[a])[i4];
  float4 t = reinterpret_cast<const float4*>(tb.val[a])[i4];
  m.x = fmaf(mu, m.x, g.x); m.y = fmaf(mu, m.y, g.y); m.z = fmaf(mu, m.z, g.z); m.w = fmaf(mu, m.w, g.w);
  t.x = fmaf(-lr, m.x, t.x); t.y = fmaf(-lr, m.y, t.y); t.z = fmaf(-lr, m.z, t.z); t.w = fmaf(-lr, m.w, t.w);
  reinterpret_cast<float4*>(tb.mom[a])[i4] = m;
  reinterpret_cast<float4*>(tb.val[a])[i4] = t;
  const __nv_bfloat162 lo = __floats2bfloat162_rn(t.x, t.y), hi = __floats2bfloat162_rn(t.z, t.w);
  reinterpret_cast<uint2*>(tb.shadow[a])[i4] =
      make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}

__global__ void shadow_kernel(const float* __restrict__ val, bf16* __restrict__ shadow, size_t n) {
  nf_pdl_begin();
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) shadow[i] = __float2bfloat16_rn(val[i]);
}

// out row r = cache row idx[r], 16 bytes per thread
// An index outside [0, cache_rows) reads nothing: its output row is zero-filled, its label set to -1 and NF_EINDEX raised.
__global__ void gather_kernel(const uint4* __restrict__ cache, const int32_t* __restrict__ cache_labels, int cache_rows,
                              const int32_t* __restrict__ idx, int count, size_t row16, uint4* __restrict__ out,
                              int32_t* __restrict__ out_labels, int32_t* __restrict__ status) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (size_t)count * row16) return;
  const size_t r = e / row16, k = e % row16;
  const int32_t src = idx[r];
  const bool ok = src >= 0 && src < cache_rows;
  out[e] = ok ? cache[(size_t)src * row16 + k] : make_uint4(0u, 0u, 0u, 0u);
  if (k == 0) {
    if (out_labels) out_labels[r] = ok ? cache_labels[src] : -1;
    if (!ok) atomicOr(status, NF_EINDEX);
  }
}


// ------------------------------------------------------------------ vectorised bf16 paths (C % 8 == 0, no pool)
// One thread owns 8 consecutive channels of a pixel: 16-byte loads and stores, coalesced along channels.
struct bf16x8 { uint4 u; };
__device__ __forceinline__ void unpack8(const uint4& u, float (&f)[8]) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 t = __bfloat1622float2(h[i]);
    f[2 * i] = t.x;
    f[2 * i + 1] = t.y;
  }
}
__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
  uint4 u;
  __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
  return u;
}

// Eight consecutive values of either storage type, loaded but not yet unpacked
template <typename T> struct Vec8;
template <> struct Vec8<bf16> {
  uint4 u;
  __device__ __forceinline__ void load(const bf16* p, size_t e) { u = __ldg(reinterpret_cast<const uint4*>(p) + e); }
  __device__ __forceinline__ void get(float (&f)[8]) const { unpack8(u, f); }
};
template <> struct Vec8<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p, size_t e) {
    a = __ldg(reinterpret_cast<const float4*>(p) + 2 * e);
    b = __ldg(reinterpret_cast<const float4*>(p) + 2 * e + 1);
  }
  __device__ __forceinline__ void get(float (&f)[8]) const {
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w; f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
  }
};

// The totals of one pixel range: out[k*C + c] = sum over the range's chains of value k at channel c, sm[k*8 + c%8][base + chain*C8 + c/8],
// by the range's thr threads (lt: the thread among them).  TREE (fp32, a range per block): in fp64, the 256 / C8 chains sixteen at a
// time; one serial fp32 sum over 128 chains of two pixels was less exact than the generic kernel's 16 chains of 16 (16 channels, 8
// images of 32x32: sum(dz*xhat) off by 1.3e-7 against 7.4e-8).  bf16 keeps the serial order, on which bits hang.
template <bool TREE>
__device__ __forceinline__ void range_totals(const float (*sm)[256], int base, int lt, int thr, int C8, int planes, bool on, float* out) {
  const int C = C8 * 8;
  if constexpr (TREE) {
    __shared__ double part[256];
    if (planes > 16) {
      const int o = lt % (2 * C), q0 = lt / (2 * C) * 16, c = o % C;
      double s = 0.0;
      for (int q = q0; q < q0 + 16; ++q) s += (double)sm[o / C * 8 + c % 8][q * C8 + c / 8];
      part[lt] = s;
      __syncthreads();
      if (lt < 2 * C) {
        for (int j = 1; j < planes / 16; ++j) s += part[j * 2 * C + lt];
        if (on) out[lt] = (float)s;
      }
      return;
    }
  }
  if (!on) return;
  for (int t = lt; t < 2 * C; t += thr) {  // value k = t / C of channel c = t % C, one thread each
    const int k = t / C, c = t % C, gg = c / 8, i = c % 8;
    std::conditional_t<TREE, double, float> s = 0;
    for (int q = 0; q < planes; ++q) s += sm[k * 8 + i][base + q * C8 + gg];
    out[t] = (float)s;
  }
}

// out = ReLU(y*scale+shift); grid-stride over (pixel, channel group)
__global__ void __launch_bounds__(256) bn_apply_vec_kernel(const uint4* __restrict__ y, int C8, const float* __restrict__ scale,
                                                           const float* __restrict__ shift, size_t total8,
                                                           uint4* __restrict__ out) {
  nf_pdl_begin();
  extern __shared__ float cs[];  // scale[C], shift[C]
  const int C = C8 * 8;
  for (int i = threadIdx.x; i < C; i += 256) {
    cs[i] = scale[i];
    cs[C + i] = shift[i];
  }
  __syncthreads();
  for (size_t e = (size_t)blockIdx.x * 256 + threadIdx.x; e < total8; e += (size_t)gridDim.x * 256) {
    const int c0 = (int)(e % C8) * 8;
    float v[8];
    unpack8(__ldg(y + e), v);
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = fmaxf(fmaf(v[i], cs[c0 + i], cs[C + c0 + i]), 0.f);
    out[e] = pack8(v);
  }
}


// per-thread constants variant (256 % C8 == 0)
// MODE of this and the two backward kernels below: 0 = ReLU, 1 = a shortcut tensor of y's shape is added before the ReLU, 2 = no
// activation (a projection shortcut).  One element per thread took 18 us where 16-byte accesses take 5 (33 MB).
template <typename T, int MODE>
__global__ void __launch_bounds__(256) bn_apply_vec2_kernel(const T* __restrict__ y, int C8, const float* __restrict__ scale,
                                                            const float* __restrict__ shift, size_t total8, T* __restrict__ out,
                                                            const T* __restrict__ skip) {
  nf_pdl_begin();
  const int c0 = (threadIdx.x % C8) * 8;
  float A[8], B[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    A[i] = scale[c0 + i];
    B[i] = shift[c0 + i];
  }
  const size_t stride = (size_t)gridDim.x * 256;
  for (size_t e0 = (size_t)blockIdx.x * 256 + threadIdx.x; e0 < total8; e0 += 2 * stride) {
    Vec8<T> yq[2], sq[2];
    const int m = e0 + stride < total8 ? 2 : 1;
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (u < m) {
        yq[u].load(y, e0 + u * stride);
        if constexpr (MODE == 1) sq[u].load(skip, e0 + u * stride);
      }
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (u < m) {
        float v[8], k[8];
        yq[u].get(v);
        if constexpr (MODE == 1) sq[u].get(k);
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = MODE == 2 ? fmaf(v[i], A[i], B[i]) : fmaxf(fmaf(v[i], A[i], B[i]) + (MODE == 1 ? k[i] : 0.f), 0.f);
        st8(out + (e0 + u * stride) * 8, v);
      }
  }
}

// partial sums of (dz, dz*xhat) with dz = da * 1[y*scale+shift (+ skip) > 0]; red[(range*2+k)*C + c] over `ranges` pixel ranges.
// MODE 1 also writes dz where a trainable shortcut wants it (dz_out not NULL).  A range has `planes` interleaved chains per
// channel, added in order; a thread runs 8 channels of a chain, so a range takes C / 8 * planes threads and a block several
// ranges where that is less than 256.  Four pixels per trip: eight (with a shortcut twelve) 16-byte loads in flight.  With 118 registers
// two blocks fit an SM: more blocks than that take their ranges in turn instead of waiting for a place and loading the channels'
// constants again (256 channels on 61 maps of 14x14, 748 ranges: 15.4 -> 12 us).
template <typename T, int MODE>
__global__ void __launch_bounds__(256) bn_bwd_reduce_vec_kernel(const T* __restrict__ y, const T* __restrict__ da,
                                                                size_t P, int C8, int planes, int ranges, const float* __restrict__ scale,
                                                                const float* __restrict__ shift, const float* __restrict__ mu,
                                                                const float* __restrict__ invstd, float* __restrict__ red,
                                                                const T* __restrict__ skip, T* __restrict__ dz_out) {
  nf_pdl_begin();
  __shared__ float sm[16][256];
  const int C = C8 * 8, thr = C8 * planes;  // threads per range: a divisor of 256
  const int lt = threadIdx.x % thr, g = lt % C8, pl = lt / C8;
  const int c0 = g * 8;
  float sc[8], sh[8], m[8], is[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    sc[i] = scale[c0 + i]; sh[i] = shift[c0 + i]; m[i] = mu[c0 + i]; is[i] = invstd[c0 + i];
  }
  for (int blk = blockIdx.x; blk * (256 / thr) < ranges; blk += gridDim.x) {
    const int rng = blk * (256 / thr) + threadIdx.x / thr;
    float a[8], b[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = b[i] = 0.f;
    const size_t p0 = rng < ranges ? P * rng / ranges : P, p1 = rng < ranges ? P * (rng + 1) / ranges : P;
    constexpr int kU = 4;
    for (size_t p = p0 + pl; p < p1; p += (size_t)kU * planes) {
      Vec8<T> yq[kU], dq[kU], sq[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const size_t q = p + (size_t)u * planes;
        if (q < p1) {
          yq[u].load(y, q * C8 + g);
          dq[u].load(da, q * C8 + g);
          if constexpr (MODE == 1) sq[u].load(skip, q * C8 + g);
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const size_t q = p + (size_t)u * planes;
        if (q < p1) {
          float yv[8], dv[8], kv[8];
          yq[u].get(yv);
          dq[u].get(dv);
          if constexpr (MODE == 1) sq[u].get(kv);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float dz = MODE == 2 || fmaf(yv[i], sc[i], sh[i]) + (MODE == 1 ? kv[i] : 0.f) > 0.f ? dv[i] : 0.f;
            a[i] += dz;
            b[i] = MODE == 1 || (MODE == 0 && sizeof(T) == 4) ? fmaf(dz * (yv[i] - m[i]), is[i], b[i]) : fmaf(dz, (yv[i] - m[i]) * is[i], b[i]);
            dv[i] = dz;
          }
          if (MODE == 1 && dz_out) st8(dz_out + (q * C8 + g) * 8, dv);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      sm[i][threadIdx.x] = a[i];
      sm[8 + i][threadIdx.x] = b[i];
    }
    __syncthreads();
    range_totals<sizeof(T) == 4 && MODE != 1>(sm, threadIdx.x / thr * thr, lt, thr, C8, planes, rng < ranges, red + (size_t)rng * 2 * C);
    __syncthreads();  // the totals are read before the next ranges are stored
  }
}

// dy = scale * (dz - sum(dz)/M - xhat * sum(dz*xhat)/M)
__global__ void __launch_bounds__(256) bn_bwd_apply_vec_kernel(const uint4* __restrict__ y, const uint4* __restrict__ da, int C8,
                                                               const float* __restrict__ scale, const float* __restrict__ shift,
                                                               const float* __restrict__ mu, const float* __restrict__ invstd,
                                                               const float* __restrict__ sdz, const float* __restrict__ sdzx,
                                                               float invM, size_t total8, uint4* __restrict__ dy) {
  nf_pdl_begin();
  extern __shared__ float cs[];  // per channel: scale, shift, mu, invstd, sdz/M, sdzx/M
  const int C = C8 * 8;
  for (int i = threadIdx.x; i < C; i += 256) {
    cs[i] = scale[i];
    cs[C + i] = shift[i];
    cs[2 * C + i] = mu[i];
    cs[3 * C + i] = invstd[i];
    cs[4 * C + i] = sdz[i] * invM;
    cs[5 * C + i] = sdzx[i] * invM;
  }
  __syncthreads();
  const size_t stride = (size_t)gridDim.x * 256;
  for (size_t e0 = (size_t)blockIdx.x * 256 + threadIdx.x; e0 < total8; e0 += 2 * stride) {  // two vectors per iteration
    const size_t e1 = e0 + stride;
    const bool two = e1 < total8;
    const uint4 ya = __ldg(y + e0), da0 = __ldg(da + e0);
    uint4 yb = ya, db = da0;
    if (two) {
      yb = __ldg(y + e1);
      db = __ldg(da + e1);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (h == 1 && !two) break;
      const size_t e = h ? e1 : e0;
      const int c0 = (int)(e % C8) * 8;
      float yv[8], dv[8], o[8];
      unpack8(h ? yb : ya, yv);
      unpack8(h ? db : da0, dv);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int c = c0 + i;
        const float dz = fmaf(yv[i], cs[c], cs[C + c]) > 0.f ? dv[i] : 0.f;
        const float xh = (yv[i] - cs[2 * C + c]) * cs[3 * C + c];
        o[i] = cs[c] * (dz - cs[4 * C + c] - xh * cs[5 * C + c]);
      }
      dy[e] = pack8(o);
    }
  }
}


// Same result with per-thread constants: when 256 % C8 == 0 a thread keeps its 8 channels over the whole
// grid-stride loop, and dy = s*dz + k1*y + k0 with k1 = -s*m2*invstd, k0 = s*(m2*invstd*mu - m1),
// m1 = sum(dz)/M, m2 = sum(dz*xhat)/M: five instructions per element.
// FORM 0: that.  k1*y and k0 cancel where |mu| is large against sigma (fp32, |mu| = 30 sigma: four times the error in a channel's
// sum of dy), so it is for bf16 without a shortcut, whose rounding hides that.  FORM 1: dy = s*dz + (k1*(y - mu) - s*m1).
// FORM 2: the generic kernel's form term by term.
template <typename T, int MODE, int FORM>
__global__ void __launch_bounds__(256) bn_bwd_apply_vec2_kernel(const T* __restrict__ y, const T* __restrict__ da, int C8,
                                                                const float* __restrict__ scale, const float* __restrict__ shift,
                                                                const float* __restrict__ mu, const float* __restrict__ invstd,
                                                                const float* __restrict__ sdz, const float* __restrict__ sdzx,
                                                                float invM, size_t total8, T* __restrict__ dy, const T* __restrict__ skip) {
  nf_pdl_begin();
  const int c0 = (threadIdx.x % C8) * 8;
  float A[8], B[8], K1[8], K0[8], M1[8], IS[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float s = scale[c0 + i], m1 = sdz[c0 + i] * invM, m2 = sdzx[c0 + i] * invM, is = invstd[c0 + i];
    A[i] = s;
    B[i] = shift[c0 + i];
    if constexpr (FORM == 2) {
      M1[i] = mu[c0 + i]; IS[i] = is; K1[i] = sdzx[c0 + i]; K0[i] = sdz[c0 + i];
    } else if constexpr (FORM == 1) {
      M1[i] = mu[c0 + i]; K1[i] = -s * m2 * is; K0[i] = -s * m1;
    } else {
      K1[i] = -s * m2 * is;
      K0[i] = s * (m2 * is * mu[c0 + i] - m1);
    }
  }
  const size_t stride = (size_t)gridDim.x * 256;
  for (size_t e0 = (size_t)blockIdx.x * 256 + threadIdx.x; e0 < total8; e0 += 2 * stride) {
    Vec8<T> yq[2], dq[2], sq[2];
    const int m = e0 + stride < total8 ? 2 : 1;
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (u < m) {
        yq[u].load(y, e0 + u * stride);
        dq[u].load(da, e0 + u * stride);
        if constexpr (MODE == 1) sq[u].load(skip, e0 + u * stride);
      }
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (u < m) {
        float yv[8], dv[8], kv[8], o[8];
        yq[u].get(yv);
        dq[u].get(dv);
        if constexpr (MODE == 1) sq[u].get(kv);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float dz = MODE == 2 || fmaf(yv[i], A[i], B[i]) + (MODE == 1 ? kv[i] : 0.f) > 0.f ? dv[i] : 0.f;
          if constexpr (FORM == 2) {
            const float xh = (yv[i] - M1[i]) * IS[i];
            o[i] = A[i] * (dz - K0[i] * invM - xh * K1[i] * invM);
          } else if constexpr (FORM == 1) {
            o[i] = fmaf(A[i], dz, fmaf(K1[i], yv[i] - M1[i], K0[i]));
          } else {
            o[i] = fmaf(A[i], dz, fmaf(K1[i], yv[i], K0[i]));
          }
        }
        st8(dy + (e0 + u * stride) * 8, o);
      }
  }
}

// partial sums of (v, v^2); same layout of partials as channel_reduce_kernel
template <typename T>
__global__ void __launch_bounds__(256) channel_sums_vec_kernel(const T* __restrict__ src, size_t P, int C8,
                                                               float* __restrict__ red) {
  nf_pdl_begin();
  __shared__ float sm[16][256];
  const int C = C8 * 8;
  const int planes = 256 / C8, g = threadIdx.x % C8, pl = threadIdx.x / C8;
  float a[8], b[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = b[i] = 0.f;
  const size_t p0 = P * blockIdx.x / gridDim.x, p1 = P * (blockIdx.x + 1) / gridDim.x;
  for (size_t p = p0 + pl; p < p1; p += 4 * (size_t)planes) {  // four loads in flight, added in index order
    Vec8<T> q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (p + (size_t)u * planes < p1) q[u].load(src, (p + (size_t)u * planes) * C8 + g);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (p + (size_t)u * planes < p1) {
        float v[8];
        q[u].get(v);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          a[i] += v[i];
          b[i] = fmaf(v[i], v[i], b[i]);
        }
      }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    sm[i][threadIdx.x] = a[i];
    sm[8 + i][threadIdx.x] = b[i];
  }
  __syncthreads();
  range_totals<sizeof(T) == 4>(sm, 0, threadIdx.x, 256, C8, planes, true, red + (size_t)blockIdx.x * 2 * C);
}


// dh = 1[h>0] * dp[n][f*4+bin]/|bin| for even sizes (every pixel lies in exactly one bin), 8 filters per
// thread, fused with the per-filter sum of dh (the aux bias gradient): red[(block*2+0)*F + f].
// CACHE: the image's 8 x 4 gradients of a thread's channels stay in registers (from 128 filters on: few pixels per block and step,
// where eight strided loads a pixel cost more than the 32 registers; 6366 maps of 8 x 8 x 256: 198 -> 130 us).
template <bool CACHE>
__global__ void __launch_bounds__(256) dh_vec_kernel(const uint4* __restrict__ h, const float* __restrict__ dp, int Ha, int Wa,
                                                     int F8, size_t P, uint4* __restrict__ dh, float* __restrict__ red) {
  nf_pdl_begin();
  __shared__ float sm[8][256];
  const int F = F8 * 8;
  const int planes = 256 / F8, g = threadIdx.x % F8, pl = threadIdx.x / F8;
  const float inv_bin = 1.f / (float)((Ha / 2) * (Wa / 2));
  float a[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = 0.f;
  const size_t p0 = P * blockIdx.x / gridDim.x, p1 = P * (blockIdx.x + 1) / gridDim.x;
  float4 dv[CACHE ? 8 : 1];
  size_t cur = ~(size_t)0;
  auto one = [&](size_t p, const uint4 hq) {
    int i, j;
    size_t n;
    if (p <= 0xffffffffull) {  // 32-bit index arithmetic where it fits
      const uint32_t p32 = (uint32_t)p, row = p32 / (uint32_t)Wa;
      j = (int)(p32 - row * (uint32_t)Wa);
      n = row / (uint32_t)Ha;
      i = (int)(row - (uint32_t)n * (uint32_t)Ha);
    } else {
      j = (int)(p % Wa);
      i = (int)((p / Wa) % Ha);
      n = p / ((size_t)Wa * Ha);
    }
    const int bin = (i >= Ha / 2 ? 2 : 0) + (j >= Wa / 2 ? 1 : 0);
    float hv[8], o[8];
    unpack8(hq, hv);
    if constexpr (CACHE) {
      if (n != cur) {
        cur = n;
        const float4* d = reinterpret_cast<const float4*>(dp + n * 4 * F) + g * 8;
#pragma unroll
        for (int e = 0; e < 8; ++e) dv[e] = __ldg(d + e);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float top = bin & 1 ? dv[e].y : dv[e].x, bot = bin & 1 ? dv[e].w : dv[e].z;
        o[e] = hv[e] > 0.f ? (bin & 2 ? bot : top) * inv_bin : 0.f;
      }
    } else {
      const float* d = dp + n * 4 * F + (size_t)(g * 8) * 4 + bin;
#pragma unroll
      for (int e = 0; e < 8; ++e) o[e] = hv[e] > 0.f ? d[e * 4] * inv_bin : 0.f;
    }
    const uint4 packed = pack8(o);
    dh[p * F8 + g] = packed;
    float r[8];
    unpack8(packed, r);  // the bias gradient sums the values as stored
#pragma unroll
    for (int e = 0; e < 8; ++e) a[e] += r[e];
  };
  size_t p = p0 + pl;
  for (; p + 3 * (size_t)planes < p1; p += 4 * (size_t)planes) {  // four loads in flight, handled in index order
    uint4 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) q[u] = __ldg(h + (p + (size_t)u * planes) * F8 + g);
#pragma unroll
    for (int u = 0; u < 4; ++u) one(p + (size_t)u * planes, q[u]);
  }
  for (; p < p1; p += planes) one(p, __ldg(h + p * F8 + g));
#pragma unroll
  for (int e = 0; e < 8; ++e) sm[e][threadIdx.x] = a[e];
  __syncthreads();
  for (int t = threadIdx.x; t < F; t += 256) {
    const int gg = t / 8, e = t % 8;
    float s = 0.f;
    for (int q = 0; q < planes; ++q) s += sm[e][q * F8 + gg];
    red[((size_t)blockIdx.x * 2 + 0) * F + t] = s;
    red[((size_t)blockIdx.x * 2 + 1) * F + t] = 0.f;
  }
}

// avgpool_small for bf16, eight channels and all four bins per thread: 16-byte loads and stores, the same sums.  (One 2-byte load at
// a time took 185 us on 6366 maps of 8 x 8 x 256, 208 MB.)
__global__ void __launch_bounds__(256) avgpool_small_vec_kernel(const uint4* __restrict__ h, int Ha, int Wa, int F8, size_t total,
                                                                float4* __restrict__ p) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (e >= total) return;
  const size_t n = e / F8;
  const uint4* hn = h + n * Ha * Wa * F8 + e % F8;
  float o[4][8];
#pragma unroll
  for (int bin = 0; bin < 4; ++bin) {
    int i0, i1, j0, j1;
    bin_range(bin / 2, Ha, i0, i1);
    bin_range(bin % 2, Wa, j0, j1);
    float a[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) a[c] = 0.f;
    for (int i = i0; i < i1; ++i) {
      for (int j = j0; j < j1; j += 4) {
        uint4 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] = __ldg(hn + (size_t)(i * Wa + min(j + u, j1 - 1)) * F8);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float v[8];
          unpack8(q[u], v);
#pragma unroll
          for (int c = 0; c < 8; ++c) a[c] = j + u < j1 ? a[c] + v[c] : a[c];
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) o[bin][c] = a[c] / (float)((i1 - i0) * (j1 - j0));
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) p[e * 8 + c] = make_float4(o[0][c], o[1][c], o[2][c], o[3][c]);
}

// Average pool of even maps in one pass: a thread per (image, eight channels, bin), sixteen loads in flight.  The sums are those of the
// kernels around it: M = 1, the bin's pixels in order; M > 1, `planes` chains of M pixels each, planes apart, the chains added in order.
// Many images: 16x16 maps with 16 filters, 1777 of them, 37 + 3 -> 5 us (there half the threads of a block per bin had nothing to do and
// sixteen added 128 sums one by one); 8x8 with 256, 6366 of them, 61 -> 45 (a thread for all four bins left a second wave nearly empty).
// Blocks of 64 threads, so that a few thousand of them reach every SM (exits of two layers at 16x16, 1777 images: 891 -> 881 us).
template <int M>
__global__ void __launch_bounds__(64) avgpool_vec_kernel(const uint4* __restrict__ h, int Ha, int Wa, int F8, int cnt, int planes,
                                                          uint32_t bw_mul, bool divide, size_t total, float* __restrict__ p) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * 64 + threadIdx.x;
  if (e >= total) return;
  const int bin = (int)(e & 3), g = (int)((e >> 2) % F8), bw = Wa / 2;
  const size_t n = (e >> 2) / F8;
  const uint4* hb = h + ((n * Ha + (bin & 2 ? Ha / 2 : 0)) * Wa + (bin & 1 ? bw : 0)) * F8 + g;
  const int chains = M == 1 ? cnt : planes;
  constexpr int B = 16 / M;
  float s[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) s[c] = 0.f;
#pragma unroll 1
  for (int q0 = 0; q0 < chains; q0 += B) {
    uint4 v[B][M];
#pragma unroll
    for (int u = 0; u < B; ++u)
#pragma unroll
      for (int r = 0; r < M; ++r) {
        const uint32_t k = (uint32_t)(min(q0 + u, chains - 1) + r * planes), row = __umulhi(k, bw_mul);  // k / bw
        v[u][r] = __ldg(hb + ((size_t)row * Wa + (k - row * bw)) * F8);
      }
#pragma unroll
    for (int u = 0; u < B; ++u) {
      float a[8];
      unpack8(v[u][0], a);
#pragma unroll
      for (int r = 1; r < M; ++r) {
        float b[8];
        unpack8(v[u][r], b);
#pragma unroll
        for (int c = 0; c < 8; ++c) a[c] += b[c];
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) s[c] = q0 + u < chains ? s[c] + a[c] : s[c];
    }
  }
  float* o = p + (n * F8 + g) * 32 + bin;
  const float inv = 1.f / (float)cnt;
#pragma unroll
  for (int c = 0; c < 8; ++c) o[c * 4] = divide ? s[c] / (float)cnt : s[c] * inv;
}

// average pool, stage 1: partial bin sums over a slice of rows; part[(n*4+bin)*S + s][F]
__global__ void __launch_bounds__(256) avgpool_part_vec_kernel(const uint4* __restrict__ h, int Ha, int Wa, int F8, int S,
                                                               float* __restrict__ part) {
  nf_pdl_begin();
  __shared__ float sm[8][256];
  const int F = F8 * 8;
  const int planes = 256 / F8, g = threadIdx.x % F8, pl = threadIdx.x / F8;
  const int sidx = blockIdx.x % S, bin = (blockIdx.x / S) % 4, n = blockIdx.x / (4 * S);
  const int bh = Ha / 2, bw = Wa / 2, i0 = (bin >> 1) * bh, j0 = (bin & 1) * bw;
  const int cnt = bh * bw, k0 = (int)((long)cnt * sidx / S), k1 = (int)((long)cnt * (sidx + 1) / S);
  float a[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = 0.f;
  const uint4* hn = h + (size_t)n * Ha * Wa * F8 + g;
  int k = k0 + pl;
  for (; k + 3 * planes < k1; k += 4 * planes) {  // four loads in flight, added in index order
    uint4 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int kk = k + u * planes;
      q[u] = __ldg(hn + ((size_t)(i0 + kk / bw) * Wa + j0 + kk % bw) * F8);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float v[8];
      unpack8(q[u], v);
#pragma unroll
      for (int e = 0; e < 8; ++e) a[e] += v[e];
    }
  }
  for (; k < k1; k += planes) {
    float v[8];
    unpack8(__ldg(hn + ((size_t)(i0 + k / bw) * Wa + j0 + k % bw) * F8), v);
#pragma unroll
    for (int e = 0; e < 8; ++e) a[e] += v[e];
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) sm[e][threadIdx.x] = a[e];
  __syncthreads();
  for (int t = threadIdx.x; t < F; t += 256) {
    const int gg = t / 8, e = t % 8;
    float s = 0.f;
    for (int q = 0; q < planes; ++q) s += sm[e][q * F8 + gg];
    part[(size_t)blockIdx.x * F + t] = s;
  }
}
// stage 2: p[n][f*4+bin] = sum over slices / |bin|
// Average pool to 2 x 2 from the partials the fused aux forward leaves: part[tile][4][F] holds, per 14 x 8-pixel tile (tiles in
// row-major order per image, th x tw of them) and epilogue warp, the channel sums over the warp's pixels.  One block per
// (image, quadrant); thread (f, lane) adds every `lanes`-th of the quadrant's th/2 * tw/2 * 4 partials in index order, the lane
// sums are added in lane order.
__global__ void __launch_bounds__(256) pool_finish_kernel(const float* __restrict__ part, int th, int tw, int F, float inv_cnt,
                                                          float* __restrict__ p) {
  nf_pdl_begin();
  __shared__ float sm[256];
  const int n = blockIdx.x >> 2, bin = blockIdx.x & 3, u = bin >> 1, v = bin & 1;
  const int lanes = 256 / F, f = threadIdx.x % F, ln = threadIdx.x / F;
  const int qh = th / 2, qw = tw / 2, cnt = qh * qw * 4;
  float s = 0.f;
  if (ln < lanes) {
    auto at = [&](int k) {
      const int w4 = k & 3, tq = k >> 2, ty = u * qh + tq / qw, tx = v * qw + tq % qw;
      return part[(((size_t)n * th + ty) * tw + tx) * 4 * F + (size_t)w4 * F + f];
    };
    int k = ln;
    for (; k + 3 * lanes < cnt; k += 4 * lanes) {  // four loads in flight, added in index order
      const float a0 = at(k), a1 = at(k + lanes), a2 = at(k + 2 * lanes), a3 = at(k + 3 * lanes);
      s += a0;
      s += a1;
      s += a2;
      s += a3;
    }
    for (; k < cnt; k += lanes) s += at(k);
  }
  sm[threadIdx.x] = s;
  __syncthreads();
  if (ln == 0) {
    float t = 0.f;
    for (int l = 0; l < lanes; ++l) t += sm[l * F + f];
    p[(size_t)n * 4 * F + f * 4 + bin] = t * inv_cnt;
  }
}

// dh from the sign mask of h (one bit per element, byte g of a pixel = channels 8g .. 8g+7): dh = bit ? dp[n][f*4+bin] / |bin| : 0,
// stored in bf16; per-block partial sums of the stored values for the bias gradient, laid out as dh_vec_kernel does.
__global__ void __launch_bounds__(256) dh_mask_vec_kernel(const uint8_t* __restrict__ mask, const float* __restrict__ dp, int Ha, int Wa,
                                                          int F8, size_t P, uint4* __restrict__ dh, float* __restrict__ red) {
  nf_pdl_begin();
  __shared__ float sm[8][256];
  __shared__ __align__(16) float tab[4][4][64];  // dp / |bin| of up to four images, [image][bin][channel]: 16-byte reads per thread
  const int F = F8 * 8;
  const int planes = 256 / F8, g = threadIdx.x % F8, pl = threadIdx.x / F8;
  const float inv_bin = 1.f / (float)((Ha / 2) * (Wa / 2));
  float a[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) a[i] = 0.f;
  const size_t p0 = P * blockIdx.x / gridDim.x, p1 = P * (blockIdx.x + 1) / gridDim.x;
  const size_t img = (size_t)Wa * Ha;
  const size_t n_lo = p0 / img, n_hi = p1 > p0 ? (p1 - 1) / img : n_lo;
  const bool tabled = F <= 64 && n_hi - n_lo < 4;  // the block's pixel range touches few images: their dp rows fit the table
  if (tabled)
    for (int i = threadIdx.x; i < (int)(n_hi - n_lo + 1) * 4 * F; i += 256) {
      const int f = i % F, bin = (i / F) % 4, ni = i / (4 * F);
      tab[ni][bin][f] = dp[(n_lo + ni) * 4 * F + (size_t)f * 4 + bin] * inv_bin;
    }
  __syncthreads();
  auto one = [&](size_t p, uint32_t m) {
    // 32-bit index arithmetic (the host keeps P below 2^31): three 64-bit divisions per pixel had made this kernel compute-bound
    const uint32_t p32 = (uint32_t)p, row = p32 / (uint32_t)Wa;
    const int j = (int)(p32 - row * (uint32_t)Wa), i = (int)(row % (uint32_t)Ha);
    const size_t n = row / (uint32_t)Ha;
    const int bin = (i >= Ha / 2 ? 2 : 0) + (j >= Wa / 2 ? 1 : 0);
    float o[8];
    if (tabled) {
      const float4 t0 = *reinterpret_cast<const float4*>(&tab[n - n_lo][bin][g * 8]);
      const float4 t1 = *reinterpret_cast<const float4*>(&tab[n - n_lo][bin][g * 8 + 4]);
      const float tv[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
#pragma unroll
      for (int e = 0; e < 8; ++e) o[e] = (m >> e) & 1u ? tv[e] : 0.f;
    } else {
      const float* d = dp + n * 4 * F + (size_t)(g * 8) * 4 + bin;
#pragma unroll
      for (int e = 0; e < 8; ++e) o[e] = (m >> e) & 1u ? d[e * 4] * inv_bin : 0.f;
    }
    const uint4 packed = pack8(o);
    dh[p * F8 + g] = packed;
    float r[8];
    unpack8(packed, r);  // the bias gradient sums the values as stored
#pragma unroll
    for (int e = 0; e < 8; ++e) a[e] += r[e];
  };
  if (pl < planes) {  // threads beyond planes * F8 (F8 not a divisor of 256) idle
    size_t p = p0 + pl;
    for (; p + 3 * (size_t)planes < p1; p += 4 * (size_t)planes) {  // four mask bytes in flight, handled in index order
      uint32_t m[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) m[u] = mask[(p + (size_t)u * planes) * F8 + g];
#pragma unroll
      for (int u = 0; u < 4; ++u) one(p + (size_t)u * planes, m[u]);
    }
    for (; p < p1; p += planes) one(p, mask[p * F8 + g]);
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) sm[e][threadIdx.x] = a[e];
  __syncthreads();
  for (int t = threadIdx.x; t < F; t += 256) {
    const int gg = t / 8, e = t % 8;
    float s = 0.f;
    for (int q = 0; q < planes; ++q) s += sm[e][q * F8 + gg];
    red[((size_t)blockIdx.x * 2 + 0) * F + t] = s;
    red[((size_t)blockIdx.x * 2 + 1) * F + t] = 0.f;
  }
}

__global__ void avgpool_finish_kernel(const float* __restrict__ part, int N, int F, int S, float inv_cnt, float* __restrict__ p) {
  nf_pdl_begin();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= N * 4 * F) return;
  const int f = e % F, bin = (e / F) % 4, n = e / (4 * F);
  float s = 0.f;
  for (int k = 0; k < S; ++k) s += part[((size_t)(n * 4 + bin) * S + k) * F + f];
  p[(size_t)n * 4 * F + f * 4 + bin] = s * inv_cnt;
}


// ------------------------------------------------------------------ vectorised bf16 paths for pooled layers
// One thread owns 8 channels of one POOLED pixel: it reads the four conv outputs of the 2x2 window.
__device__ __forceinline__ size_t div_small(size_t e, int d) {  // e / d in 32 bits where e fits
  return e <= 0xffffffffull ? (size_t)((uint32_t)e / (uint32_t)d) : e / (size_t)d;
}
__device__ __forceinline__ size_t win_base(size_t q, int Ho, int Wo, int C8) {  // q = pooled pixel index
  const int Wa = Wo / 2, Ha = Ho / 2;
  if (q <= 0xffffffffull) {  // 32-bit index arithmetic where it fits: three 64-bit divisions per window made these kernels compute-bound
    const uint32_t q32 = (uint32_t)q, row = q32 / (uint32_t)Wa;
    const uint32_t ja = q32 - row * (uint32_t)Wa, n = row / (uint32_t)Ha, ia = row - n * (uint32_t)Ha;
    return (((size_t)n * Ho + 2 * ia) * Wo + 2 * ja) * C8;
  }
  const int ja = (int)(q % Wa), ia = (int)((q / Wa) % Ha);
  const size_t n = q / ((size_t)Wa * Ha);
  return ((n * Ho + 2 * ia) * Wo + 2 * ja) * C8;
}

// Which of the four window positions of a channel pair (packed bf16 y in w[0..3]) receives the gradient: all-ones halves in keep[d]
// where position d is the first maximum, in scan order, of the bf16-rounded ReLU outputs and that maximum is positive; returns that
// maximum.  Two channels per instruction from the conversion on: with one channel at a time the two kernels below were bound by these
// instructions.
__device__ __forceinline__ __nv_bfloat162 pool_winner2(const uint32_t (&w)[4], float A0, float A1, float B0, float B1, uint32_t (&keep)[4]) {
  __nv_bfloat162 r[4];
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    const float z0 = fmaf(__uint_as_float(w[d] << 16), A0, B0), z1 = fmaf(__uint_as_float(w[d] & 0xffff0000u), A1, B1);
    uint32_t u;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(u) : "f"(z1), "f"(z0));
    r[d] = *reinterpret_cast<const __nv_bfloat162*>(&u);
  }
  const __nv_bfloat162 m = __hmax2(__hmax2(r[0], r[1]), __hmax2(r[2], r[3]));
  const uint32_t pos = __hgt2_mask(m, __floats2bfloat162_rn(0.f, 0.f));
  const uint32_t e0 = __heq2_mask(r[0], m), e1 = __heq2_mask(r[1], m), e2 = __heq2_mask(r[2], m);
  keep[0] = pos & e0;
  keep[1] = pos & e1 & ~e0;
  keep[2] = pos & e2 & ~(e0 | e1);
  keep[3] = pos & ~(e0 | e1 | e2);
  return m;
}

// BatchNorm + ReLU + 2x2 max-pool.  WIN: a step also keeps, per window and channel, the y that its backward pass will want (the winner's,
// or where nothing is positive the first one, whose own test then says so): a quarter of y, so that the sums of the backward pass need
// not read y again and find the winners once more.  1904 maps of 64x64x64: this kernel 200 -> 234 us, the sums 264 -> 96.
template <bool WIN>
__global__ void __launch_bounds__(256) bn_apply_pool_vec_kernel(const uint4* __restrict__ y, int Ho, int Wo, int C8,
                                                                const float* __restrict__ scale,
                                                                const float* __restrict__ shift,
                                                                size_t total8, uint4* __restrict__ out, uint4* __restrict__ ywin) {
  nf_pdl_begin();
  const int c0 = (threadIdx.x % C8) * 8;
  float A[8], B[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) { A[i] = scale[c0 + i]; B[i] = shift[c0 + i]; }
  for (size_t e = (size_t)blockIdx.x * 256 + threadIdx.x; e < total8; e += (size_t)gridDim.x * 256) {
    const size_t b = win_base(div_small(e, C8), Ho, Wo, C8) + threadIdx.x % C8;  // 256 % C8 == 0: the chunk of a thread is fixed
    const uint4 v4[4] = {__ldg(y + b), __ldg(y + b + C8), __ldg(y + b + (size_t)Wo * C8), __ldg(y + b + (size_t)Wo * C8 + C8)};
    if constexpr (WIN) {
      const uint32_t* yw = reinterpret_cast<const uint32_t*>(v4);  // [window position][channel pair]
      uint32_t o[4], w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t p[4] = {yw[i], yw[4 + i], yw[8 + i], yw[12 + i]};
        uint32_t k[4];
        const __nv_bfloat162 m = pool_winner2(p, A[2 * i], A[2 * i + 1], B[2 * i], B[2 * i + 1], k);
        const __nv_bfloat162 z = __hmax2(m, __floats2bfloat162_rn(0.f, 0.f));  // NaN counts as zero, as in fmaxf
        o[i] = *reinterpret_cast<const uint32_t*>(&z);
        w[i] = (p[1] & k[1]) | (p[2] & k[2]) | (p[3] & k[3]) | (p[0] & ~(k[1] | k[2] | k[3]));
      }
      out[e] = make_uint4(o[0], o[1], o[2], o[3]);
      ywin[e] = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
      float best[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) best[i] = 0.f;
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        float v[8];
        unpack8(v4[d], v);
#pragma unroll
        for (int i = 0; i < 8; ++i) best[i] = fmaxf(best[i], fmaf(v[i], A[i], B[i]));
      }
      out[e] = pack8(best);
    }
  }
}

// Partial sums of (dz, dz*xhat) of a pooled layer from the winners that its forward pass kept: ywin and da have the pooled shape.  The
// ranges, chains and order are those of the kernels that read y itself.
__global__ void __launch_bounds__(256) bn_bwd_reduce_win_vec_kernel(const uint4* __restrict__ ywin, const uint4* __restrict__ da, size_t Pq,
                                                                    int C8, const float* __restrict__ scale,
                                                                    const float* __restrict__ shift, const float* __restrict__ mu,
                                                                    const float* __restrict__ invstd, float* __restrict__ red) {
  nf_pdl_begin();
  __shared__ float sm[16][256];
  const int C = C8 * 8;
  const int planes = 256 / C8, g = threadIdx.x % C8, pl = threadIdx.x / C8;
  const int c0 = g * 8;
  float A[8], B[8], m[8], is[8], a[8], b[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    A[i] = scale[c0 + i]; B[i] = shift[c0 + i]; m[i] = mu[c0 + i]; is[i] = invstd[c0 + i];
    a[i] = 0.f; b[i] = 0.f;
  }
  const size_t q0 = Pq * blockIdx.x / gridDim.x, q1 = Pq * (blockIdx.x + 1) / gridDim.x;
  constexpr int kU = 4;  // windows in flight, added in index order
  for (size_t q = q0 + pl; q < q1; q += (size_t)kU * planes) {
    uint4 yv[kU], dv[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const size_t e = q + (size_t)u * planes;
      if (e < q1) {
        yv[u] = __ldg(ywin + e * C8 + g);
        dv[u] = __ldg(da + e * C8 + g);
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      if (q + (size_t)u * planes >= q1) break;
      const uint32_t yw[4] = {yv[u].x, yv[u].y, yv[u].z, yv[u].w}, dw[4] = {dv[u].x, dv[u].y, dv[u].z, dv[u].w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float z0 = fmaf(__uint_as_float(yw[i] << 16), A[2 * i], B[2 * i]), z1 = fmaf(__uint_as_float(yw[i] & 0xffff0000u), A[2 * i + 1], B[2 * i + 1]);
        const __nv_bfloat162 r = __floats2bfloat162_rn(z0, z1);
        const uint32_t pos = __hgt2_mask(r, __floats2bfloat162_rn(0.f, 0.f));
        const uint32_t dd = dw[i] & pos, yy = yw[i] & pos;
        const float d0 = __uint_as_float(dd << 16), d1 = __uint_as_float(dd & 0xffff0000u);
        a[2 * i] += d0;
        a[2 * i + 1] += d1;
        b[2 * i] = fmaf(d0, (__uint_as_float(yy << 16) - m[2 * i]) * is[2 * i], b[2 * i]);
        b[2 * i + 1] = fmaf(d1, (__uint_as_float(yy & 0xffff0000u) - m[2 * i + 1]) * is[2 * i + 1], b[2 * i + 1]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    sm[i][threadIdx.x] = a[i];
    sm[8 + i][threadIdx.x] = b[i];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 2 * C; t += 256) {
    const int k = t / C, c = t % C, gg = c / 8, i = c % 8;
    float s = 0.f;
    for (int qq = 0; qq < planes; ++qq) s += sm[k * 8 + i][qq * C8 + gg];
    red[((size_t)blockIdx.x * 2 + k) * C + c] = s;
  }
}

__global__ void __launch_bounds__(256, 2) bn_bwd_apply_pool_vec_kernel(const uint4* __restrict__ y, const uint4* __restrict__ da, int Ho,
                                                                    int Wo, int C8, const float* __restrict__ scale,
                                                                    const float* __restrict__ shift, const float* __restrict__ mu,
                                                                    const float* __restrict__ invstd, const float* __restrict__ sdz,
                                                                    const float* __restrict__ sdzx, float invM, size_t total8,
                                                                    uint4* __restrict__ dy) {
  nf_pdl_begin();
  const int c0 = (threadIdx.x % C8) * 8;
  float A[8], B[8], K1[8], K0[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float s = scale[c0 + i], m1 = sdz[c0 + i] * invM, m2 = sdzx[c0 + i] * invM, is = invstd[c0 + i];
    A[i] = s; B[i] = shift[c0 + i];
    K1[i] = -s * m2 * is;
    K0[i] = s * (m2 * is * mu[c0 + i] - m1);
  }
  const size_t off[4] = {0, (size_t)C8, (size_t)Wo * C8, (size_t)Wo * C8 + C8}, step = (size_t)gridDim.x * 256;
  size_t e = (size_t)blockIdx.x * 256 + threadIdx.x, nb = 0;
  uint4 nx[5];
  auto fetch = [&](size_t i) {  // as in the reduction
    nb = win_base(div_small(i, C8), Ho, Wo, C8) + threadIdx.x % C8;
#pragma unroll
    for (int d = 0; d < 4; ++d) nx[d] = __ldg(y + nb + off[d]);
    nx[4] = __ldg(da + i);
  };
  if (e < total8) fetch(e);
  for (; e < total8; e += step) {  // e over pooled vectors
    const size_t bb = nb;
    const uint4 v4[5] = {nx[0], nx[1], nx[2], nx[3], nx[4]};
    if (e + step < total8) fetch(e + step);
    const uint32_t* yw = reinterpret_cast<const uint32_t*>(v4);
    uint32_t ow[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t w[4] = {yw[i], yw[4 + i], yw[8 + i], yw[12 + i]};
      uint32_t k[4];
      pool_winner2(w, A[2 * i], A[2 * i + 1], B[2 * i], B[2 * i + 1], k);
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        const uint32_t dd = yw[16 + i] & k[d];
        const float o0 = fmaf(A[2 * i], __uint_as_float(dd << 16), fmaf(K1[2 * i], __uint_as_float(w[d] << 16), K0[2 * i]));
        const float o1 = fmaf(A[2 * i + 1], __uint_as_float(dd & 0xffff0000u), fmaf(K1[2 * i + 1], __uint_as_float(w[d] & 0xffff0000u), K0[2 * i + 1]));
        const __nv_bfloat162 q = __floats2bfloat162_rn(o0, o1);
        ow[d][i] = *reinterpret_cast<const uint32_t*>(&q);
      }
    }
#pragma unroll
    for (int d = 0; d < 4; ++d) dy[bb + off[d]] = make_uint4(ow[d][0], ow[d][1], ow[d][2], ow[d][3]);
  }
}

inline bool vec_ok(int dtype, int C, int pool) { return dtype == NF_BF16 && C % 8 == 0 && C <= 1024 && !pool; }
// either storage type: a thread keeps its eight channels over its whole loop
inline bool vec2_ok(int C, int pool) { return C % 8 == 0 && C <= 2048 && 256 % (C / 8) == 0 && !pool; }
inline int vec_blocks(size_t work_items) {
  size_t b = (work_items + 256 * 8 - 1) / (256 * 8);
  if (b < 1) b = 1;
  if (b > 148 * 16) b = 148 * 16;
  return (int)b;
}

inline unsigned nblk(size_t n, int per) { return (unsigned)((n + per - 1) / per); }

}  // namespace

#define DISPATCH(dtype, CALL_F32, CALL_BF16) \
  do {                                       \
    if ((dtype) == NF_F32) { CALL_F32; } else { CALL_BF16; } \
  } while (0)

int nf_k_channel_blocks(size_t P, int C) {
  const int planes = 256 / pow2ceil_cap256(C);
  size_t nb = (P + (size_t)planes * 16 - 1) / ((size_t)planes * 16);
  if (nb < 1) nb = 1;
  if (nb > 1184) nb = 1184;
  return (int)nb;
}

int nf_k_channel_sums(int dtype, const void* src, size_t P, int C, float* red, size_t red_floats, int* nblocks) {
  const int nb = nf_k_channel_blocks(P, C);
  if ((size_t)nb * 2 * C > red_floats) return NF_ENOWS;
  if (vec2_ok(C, 0)) {
    DISPATCH(dtype, (nf_launch(channel_sums_vec_kernel<float>, nb, 256, 0, (const float*)src, P, C / 8, red)),
             (nf_launch(channel_sums_vec_kernel<bf16>, nb, 256, 0, (const bf16*)src, P, C / 8, red)));
    NF_LAUNCHED();
    *nblocks = nb;
    return NF_OK;
  }
  DISPATCH(dtype,
           (nf_launch(channel_reduce_kernel<float, StatsFn>, nb, 256, 0, (const float*)src, nullptr, P, C, StatsFn(), red)),
           (nf_launch(channel_reduce_kernel<bf16, StatsFn>, nb, 256, 0, (const bf16*)src, nullptr, P, C, StatsFn(), red)));
  NF_LAUNCHED();
  *nblocks = nb;
  return NF_OK;
}

int nf_k_bn_finalize(const float* red, int nblocks, int C, double M, const float* gamma, const float* beta,
                       float eps, float bn_momentum, float* scale, float* shift, float* mu, float* invstd,
                       float* rmean, float* rvar) {
  nf_launch(bn_finalize_kernel, nblk(C, kRedCh), kRedThreads, 0, red, nblocks, C, M, gamma, beta, eps, bn_momentum, scale,
                                                            shift, mu, invstd, rmean, rvar);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_partial_totals(const float* red, int nblocks, int C, double* tot) {
  nf_launch(partial_totals_kernel, nblk(C, kRedCh), kRedThreads, 0, red, nblocks, C, tot);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_bn_finalize_tot(const double* tot, int C, double M, const float* gamma, const float* beta, float eps, float bn_momentum,
                           float* scale, float* shift, float* mu, float* invstd, float* rmean, float* rvar) {
  nf_launch(bn_finalize_tot_kernel, nblk(C, 128), 128, 0, tot, C, M, gamma, beta, eps, bn_momentum, scale, shift, mu, invstd,
                                                                rmean, rvar);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_bn_bwd_finalize_tot(const double* tot, int C, int world, float* sdz, float* sdzx, float* ggamma, float* gbeta) {
  nf_launch(bn_bwd_finalize_tot_kernel, nblk(C, 128), 128, 0, tot, C, 1.0 / (double)world, sdz, sdzx, ggamma, gbeta);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_bn_eval_coeffs(int C, const float* gamma, const float* beta, float eps, const float* rmean,
                          const float* rvar, float* scale, float* shift) {
  nf_launch(bn_eval_coeffs_kernel, nblk(C, 128), 128, 0, C, gamma, beta, eps, rmean, rvar, scale, shift);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_bn_apply(int dtype, const void* y, int N, int Ho, int Wo, int C, int pool, const float* scale,
                    const float* shift, void* out, const void* skip, void* ywin) {
  const size_t total = (size_t)N * (pool ? Ho / 2 : Ho) * (pool ? Wo / 2 : Wo) * C;
  if (vec2_ok(C, pool)) {
#define NF_APPLY(T, M) \
  nf_launch(bn_apply_vec2_kernel<T, M>, vec_blocks(total / 8), 256, 0, (const T*)y, C / 8, scale, shift, total / 8, (T*)out, (const T*)skip)
    DISPATCH(dtype, (skip ? NF_APPLY(float, 1) : NF_APPLY(float, 0)), (skip ? NF_APPLY(bf16, 1) : NF_APPLY(bf16, 0)));
#undef NF_APPLY
    NF_LAUNCHED();
    return NF_OK;
  }
  if (skip) {  // residual layers with a pool or odd channel counts take the generic kernels
    DISPATCH(dtype,
             (nf_launch(bn_apply_kernel<float>, nblk(total, 256), 256, 0, (const float*)y, Ho, Wo, C, pool, scale, shift, total, (float*)out, (const float*)skip)),
             (nf_launch(bn_apply_kernel<bf16>, nblk(total, 256), 256, 0, (const bf16*)y, Ho, Wo, C, pool, scale, shift, total, (bf16*)out, (const bf16*)skip)));
    NF_LAUNCHED();
    return NF_OK;
  }
  if (pool && vec_ok(dtype, C, 0) && 256 % (C / 8) == 0) {
    nf_launch(ywin ? bn_apply_pool_vec_kernel<true> : bn_apply_pool_vec_kernel<false>, vec_blocks(total / 8), 256, 0, (const uint4*)y, Ho, Wo, C / 8,
              scale, shift, total / 8, (uint4*)out, (uint4*)ywin);
    NF_LAUNCHED();
    return NF_OK;
  }
  if (vec_ok(dtype, C, pool)) {
    nf_launch(bn_apply_vec_kernel, vec_blocks(total / 8), 256, 2 * C * sizeof(float), (const uint4*)y, C / 8, scale, shift,
                                                                                         total / 8, (uint4*)out);
    NF_LAUNCHED();
    return NF_OK;
  }
  DISPATCH(dtype,
           (nf_launch(bn_apply_kernel<float>, nblk(total, 256), 256, 0, (const float*)y, Ho, Wo, C, pool, scale, shift, total, (float*)out, nullptr)),
           (nf_launch(bn_apply_kernel<bf16>, nblk(total, 256), 256, 0, (const bf16*)y, Ho, Wo, C, pool, scale, shift, total, (bf16*)out, nullptr)));
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_avgpool_slices(int N, int Ha, int Wa) {
  const long cnt = (long)(Ha / 2) * (Wa / 2);
  long S = 1184 / ((long)N * 4);
  if (S > cnt / 64) S = cnt / 64;
  if (S < 1) S = 1;
  return (int)S;
}

// k / bw as the upper half of k * ceil(2^32 / bw): exact for k * bw < 2^32
static uint32_t recip(int bw) { return (uint32_t)((((uint64_t)1 << 32) + bw - 1) / bw); }

int nf_k_avgpool_fast(const void* h, int N, int Ha, int Wa, int F, float* part, size_t part_floats, float* p) {
  if (F % 8 || 256 % (F / 8) || (Ha & 1) || (Wa & 1)) return NF_EUNSUPPORTED;
  if ((long)(Ha / 2) * (Wa / 2) <= 16) return NF_EUNSUPPORTED;  // tiny maps: the caller's generic path has a kernel for them
  const int S = nf_k_avgpool_slices(N, Ha, Wa);
  // One pass where no slices are cut, the chains are whole and there are threads enough for their length.  One pass against the two kernels
  // behind it, in us, operands in L2 where they fit.  Chains of one pixel, up to 64 of them: 16x16x16, 8 images 4.9 / 4.6, 256 images 5.1 /
  // 10.4, 4096 images 7.8 / 70.  More of them: 32x32x8, 1024 threads 17.5 / 16.2, 4096 18 / 38, 16 384 21 / 129; 20x20x16, 7.8 / 6.3, 7.9 /
  // 14, 9.2 / 38: the line lies on the safe side.  Longer chains: 32x32x64, 32 768 threads 43 / 35, 49 152 50 / 49, 65 536 56 / 63, which
  // draws the line; the others there (32x32x32 43 / 61, 16x16x64 13 / 25, 16x16x256 8.4 / 15) would gain from 16 384 on.
  const int cnt = (Ha / 2) * (Wa / 2), planes = 256 / (F / 8), m = cnt <= planes ? 1 : cnt % planes ? 0 : cnt / planes;
  const size_t total = (size_t)N * 4 * (F / 8);
  if (S == 1 && Wa >= 4 && (m == 1 || m == 2 || m == 4 || m == 8) && cnt < 65536 && (m > 1 ? total >= 49152 : cnt <= 64 || total >= 16384)) {
    auto* k = m == 1 ? avgpool_vec_kernel<1> : m == 2 ? avgpool_vec_kernel<2> : m == 4 ? avgpool_vec_kernel<4> : avgpool_vec_kernel<8>;
    nf_launch(k, nblk(total, 64), 64, 0, (const uint4*)h, Ha, Wa, F / 8, cnt, planes, recip(Wa / 2), false, total, p);
    NF_LAUNCHED();
    return NF_OK;
  }
  if ((size_t)N * 4 * S * F > part_floats) return NF_EUNSUPPORTED;
  nf_launch(avgpool_part_vec_kernel, N * 4 * S, 256, 0, (const uint4*)h, Ha, Wa, F / 8, S, part);
  NF_LAUNCHED();
  nf_launch(avgpool_finish_kernel, nblk((size_t)N * 4 * F, 256), 256, 0, part, N, F, S, 1.f / (float)((Ha / 2) * (Wa / 2)), p);
  NF_LAUNCHED();
  return NF_OK;
}

// dh with the fused aux-bias gradient partials (bf16, F % 8 == 0, even sizes); nblocks partials in red
int nf_k_pool_finish(const float* part, int N, int th, int tw, int F, float inv_cnt, float* p) {
  if (F < 1 || F > 256) return NF_EUNSUPPORTED;
  nf_launch(pool_finish_kernel, N * 4, 256, 0, part, th, tw, F, inv_cnt, p);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_dh_mask(const uint8_t* mask, const float* dp, int N, int Ha, int Wa, int F, void* dh, float* red, size_t red_floats,
                 int* nblocks) {
  if (F % 8 || F > 2048 || (Ha & 1) || (Wa & 1)) return NF_EUNSUPPORTED;
  const size_t P = (size_t)N * Ha * Wa;
  if (P >= ((size_t)1 << 31)) return NF_EUNSUPPORTED;
  const int nb = nf_k_channel_blocks(P, F);
  if ((size_t)nb * 2 * F > red_floats) return NF_ENOWS;
  nf_launch(dh_mask_vec_kernel, nb, 256, 0, mask, dp, Ha, Wa, F / 8, P, (uint4*)dh, red);
  NF_LAUNCHED();
  *nblocks = nb;
  return NF_OK;
}

int nf_k_dh_fast(const void* h, const float* dp, int N, int Ha, int Wa, int F, void* dh, float* red, size_t red_floats,
                   int* nblocks) {
  if (F % 8 || 256 % (F / 8) || (Ha & 1) || (Wa & 1)) return NF_EUNSUPPORTED;
  const size_t P = (size_t)N * Ha * Wa;
  const int nb = nf_k_channel_blocks(P, F);
  if ((size_t)nb * 2 * F > red_floats) return NF_EUNSUPPORTED;
  nf_launch(F >= 128 ? dh_vec_kernel<true> : dh_vec_kernel<false>, nb, 256, 0, (const uint4*)h, dp, Ha, Wa, F / 8, P, (uint4*)dh, red);
  NF_LAUNCHED();
  *nblocks = nb;
  return NF_OK;
}

int nf_k_avgpool(int dtype, const void* h, int N, int Ha, int Wa, int F, float* p) {
  if ((long)((Ha + 1) / 2) * ((Wa + 1) / 2) <= 16) {  // tiny maps (late blocks train at thousands of samples): a thread per output
    // (bf16: 32 outputs per thread where one each would not fit the chip at once, or is one pixel; one image of 7 x 7: 15 against 6 us)
    if (dtype == NF_BF16 && F % 8 == 0 && ((size_t)N * 4 * F > (size_t)148 * 2048 || Ha * Wa <= 4)) {
      const size_t groups = (size_t)N * (F / 8);
      if (Ha % 2 == 0 && Wa % 2 == 0 && Wa >= 4) {
        nf_launch(avgpool_vec_kernel<1>, nblk(groups * 4, 64), 64, 0, (const uint4*)h, Ha, Wa, F / 8, (Ha / 2) * (Wa / 2), 1, recip(Wa / 2), true,
                  groups * 4, p);
        NF_LAUNCHED();
        return NF_OK;
      }
      nf_launch(avgpool_small_vec_kernel, nblk(groups, 256), 256, 0, (const uint4*)h, Ha, Wa, F / 8, groups, (float4*)p);
      NF_LAUNCHED();
      return NF_OK;
    }
    const size_t total = (size_t)N * 4 * F;
    DISPATCH(dtype, (nf_launch(avgpool_small_kernel<float>, nblk(total, 256), 256, 0, (const float*)h, Ha, Wa, F, total, p)),
             (nf_launch(avgpool_small_kernel<bf16>, nblk(total, 256), 256, 0, (const bf16*)h, Ha, Wa, F, total, p)));
    NF_LAUNCHED();
    return NF_OK;
  }
  DISPATCH(dtype, (nf_launch(avgpool_kernel<float>, N * 4, 256, 0, (const float*)h, Ha, Wa, F, p)),
           (nf_launch(avgpool_kernel<bf16>, N * 4, 256, 0, (const bf16*)h, Ha, Wa, F, p)));
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_fc_ce(const float* p, const int32_t* labels, int N, int D, int K, const float* Wf, const float* bf,
                 float* logits, float* dlogits, float* dp, float* lossn, int32_t* status, int loss_kind, int n_scale) {
  const size_t smem = (size_t)(D + K) * sizeof(float);
  if (smem > 40000) return NF_EUNSUPPORTED;
  nf_launch(fc_ce_kernel, N, 256, smem, p, labels, N, D, K, Wf, bf, logits, dlogits, dp, lossn, status, loss_kind, n_scale);
  NF_LAUNCHED();
  return NF_OK;
}

__global__ void __launch_bounds__(256) count_equal_kernel(const int32_t* __restrict__ a, const int32_t* __restrict__ b, long long n,
                                                          unsigned long long* __restrict__ count) {
  nf_pdl_begin();
  unsigned c = 0;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += 256LL * gridDim.x) c += a[i] == b[i];
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(count, (unsigned long long)c);   // integer sum: order-independent
}

int nf_k_count_equal(const int32_t* a, const int32_t* b, long long n, unsigned long long* count) {
  const int blocks = (int)std::min<long long>((n + 255) / 256, 1184);
  nf_launch(count_equal_kernel, blocks, 256, 0, a, b, n, count);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_fc_predict(const float* p, int N, int D, int K, const float* Wf, const float* bf, float* logits, int32_t* pred) {
  const size_t smem = (size_t)D * sizeof(float);
  if (smem > 40000) return NF_EUNSUPPORTED;
  nf_launch(fc_predict_kernel, N, 256, smem, p, D, K, Wf, bf, logits, pred);
  NF_LAUNCHED();
  return NF_OK;
}

// out[8 - tap][c][f] = w[tap][f][c]: the weights of the input-gradient convolution written as a forward convolution
__global__ void flip_weights_kernel(const bf16* __restrict__ w, int F, int C, bf16* __restrict__ out) {
  nf_pdl_begin();
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (size_t)9 * F * C) return;
  const int f = (int)(e % F), c = (int)((e / F) % C), tap = (int)(e / ((size_t)F * C));
  out[e] = w[((size_t)(8 - tap) * F + f) * C + c];
}

int nf_k_flip_weights(const bf16* w, int F, int C, bf16* out) {
  nf_launch(flip_weights_kernel, nblk((size_t)9 * F * C, 256), 256, 0, w, F, C, out);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_auxmax(int dtype, const void* h, int N, int Ha, int Wa, int F, float* p, int32_t* parg) {
  DISPATCH(dtype, (nf_launch(auxmax_kernel<float>, N * 4, 256, 0, (const float*)h, Ha, Wa, F, p, parg)),
           (nf_launch(auxmax_kernel<bf16>, N * 4, 256, 0, (const bf16*)h, Ha, Wa, F, p, parg)));
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_dh_max(int dtype, const void* h, const float* dp, const int32_t* parg, int N, int Ha, int Wa, int F, void* dh) {
  const size_t total = (size_t)N * Ha * Wa * F;
  DISPATCH(dtype, (nf_launch(dh_max_kernel<float>, nblk(total, 256), 256, 0, (const float*)h, dp, parg, Ha, Wa, F, total, (float*)dh)),
           (nf_launch(dh_max_kernel<bf16>, nblk(total, 256), 256, 0, (const bf16*)h, dp, parg, Ha, Wa, F, total, (bf16*)dh)));
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_dh(int dtype, const void* h, const float* dp, int N, int Ha, int Wa, int F, void* dh) {
  const size_t total = (size_t)N * Ha * Wa * F;
  DISPATCH(dtype, (nf_launch(dh_kernel<float>, nblk(total, 256), 256, 0, (const float*)h, dp, Ha, Wa, F, total, (float*)dh)),
           (nf_launch(dh_kernel<bf16>, nblk(total, 256), 256, 0, (const bf16*)h, dp, Ha, Wa, F, total, (bf16*)dh)));
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_sum_partials(const float* red, int nblocks, int C, float* out) {
  nf_launch(sum_partials_kernel, nblk(C, kRedCh), kRedThreads, 0, red, nblocks, C, out);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_bn_bwd_reduce(int dtype, const void* y, const void* da, int N, int Ho, int Wo, int C, int pool,
                         const float* scale, const float* shift, const float* mu, const float* invstd, float* red,
                         size_t red_floats, int* nblocks, const void* skip, void* dz_out, const void* ywin) {
  const size_t P = (size_t)N * Ho * Wo;
  const int nb = nf_k_channel_blocks(P, C);
  if ((size_t)nb * 2 * C > red_floats) return NF_ENOWS;
  const bool vec = vec2_ok(C, pool);
  if (!skip && pool && vec_ok(dtype, C, 0) && 256 % (C / 8) == 0) {
    if (!ywin) return NF_EINVAL;
    nf_launch(bn_bwd_reduce_win_vec_kernel, nb, 256, 0, (const uint4*)ywin, (const uint4*)da, P / 4, C / 8, scale, shift, mu, invstd, red);
    NF_LAUNCHED();
    *nblocks = nb;
    // behind the sums: dz may lie over the winners
    return dz_out ? nf_k_write_dz(dtype, y, da, N, Ho, Wo, C, pool, scale, shift, skip, dz_out) : NF_OK;
  }
  if (dz_out && !(skip && vec)) {  // else the reduction below writes it
    const int rc = nf_k_write_dz(dtype, y, da, N, Ho, Wo, C, pool, scale, shift, skip, dz_out);
    if (rc != NF_OK) return rc;
  }
  if (vec) {
    // without a shortcut a range is a block's 256 / (C / 8) chains; with one, the generic kernel's (256 channels and chains)
    const int planes = skip ? 256 / pow2ceil_cap256(C) : 256 / (C / 8), per = 256 / (C / 8 * planes);
#define NF_REDUCE(T, M)                                                                                                                  \
  nf_launch(bn_bwd_reduce_vec_kernel<T, M>, std::min(nblk(nb, per), 296u), 256, 0, (const T*)y, (const T*)da, P, C / 8, planes, nb, scale, shift, mu, invstd, red, \
            (const T*)skip, (T*)dz_out)
    DISPATCH(dtype, (skip ? NF_REDUCE(float, 1) : NF_REDUCE(float, 0)), (skip ? NF_REDUCE(bf16, 1) : NF_REDUCE(bf16, 0)));
#undef NF_REDUCE
    NF_LAUNCHED();
    *nblocks = nb;
    return NF_OK;
  }
  BnBwdFn fn{Ho, Wo, pool, scale, shift, mu, invstd, skip};
  DISPATCH(dtype,
           (nf_launch(channel_reduce_kernel<float, BnBwdFn>, nb, 256, 0, (const float*)y, (const float*)da, P, C, fn, red)),
           (nf_launch(channel_reduce_kernel<bf16, BnBwdFn>, nb, 256, 0, (const bf16*)y, (const bf16*)da, P, C, fn, red)));
  NF_LAUNCHED();
  *nblocks = nb;
  return NF_OK;
}

int nf_k_write_dz(int dtype, const void* y, const void* da, int N, int Ho, int Wo, int C, int pool, const float* scale,
                  const float* shift, const void* skip, void* dz) {
  const size_t total = (size_t)N * Ho * Wo * C;
  DISPATCH(dtype,
           (nf_launch(write_dz_kernel<float>, nblk(total, 256), 256, 0, (const float*)y, (const float*)da, Ho, Wo, C, pool, scale, shift, (const float*)skip, total, (float*)dz)),
           (nf_launch(write_dz_kernel<bf16>, nblk(total, 256), 256, 0, (const bf16*)y, (const bf16*)da, Ho, Wo, C, pool, scale, shift, (const bf16*)skip, total, (bf16*)dz)));
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_bn_bwd_finalize(const float* red, int nblocks, int C, float* sdz, float* sdzx, float* ggamma,
                           float* gbeta) {
  nf_launch(bn_bwd_finalize_kernel, nblk(C, kRedCh), kRedThreads, 0, red, nblocks, C, sdz, sdzx, ggamma, gbeta);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_bn_bwd_apply(int dtype, const void* y, const void* da, int N, int Ho, int Wo, int C, int pool,
                        const float* scale, const float* shift, const float* mu, const float* invstd,
                        const float* sdz, const float* sdzx, double M, void* dy, const void* skip) {
  const size_t total = (size_t)N * Ho * Wo * C;
  const float invM = (float)(1.0 / M);
  if (vec2_ok(C, pool)) {
#define NF_APPLY(T, M, FM)                                                                                                                       \
  nf_launch(bn_bwd_apply_vec2_kernel<T, M, FM>, vec_blocks(total / 8), 256, 0, (const T*)y, (const T*)da, C / 8, scale, shift, mu, invstd, sdz, sdzx, \
            invM, total / 8, (T*)dy, (const T*)skip)
    // form 0 in bf16 up to 1024 channels: where it has always been
    DISPATCH(dtype, (skip ? NF_APPLY(float, 1, 2) : NF_APPLY(float, 0, 1)),
             (skip ? NF_APPLY(bf16, 1, 2) : C <= 1024 ? NF_APPLY(bf16, 0, 0) : NF_APPLY(bf16, 0, 1)));
#undef NF_APPLY
    NF_LAUNCHED();
    return NF_OK;
  }
  if (skip) {
    DISPATCH(dtype,
             (nf_launch(bn_bwd_apply_kernel<float>, nblk(total, 256), 256, 0, (const float*)y, (const float*)da, Ho, Wo, C, pool, scale, shift, mu, invstd, sdz, sdzx, invM, total, (float*)dy, (const float*)skip)),
             (nf_launch(bn_bwd_apply_kernel<bf16>, nblk(total, 256), 256, 0, (const bf16*)y, (const bf16*)da, Ho, Wo, C, pool, scale, shift, mu, invstd, sdz, sdzx, invM, total, (bf16*)dy, (const bf16*)skip)));
    NF_LAUNCHED();
    return NF_OK;
  }
  if (pool && vec_ok(dtype, C, 0) && 256 % (C / 8) == 0) {
    nf_launch(bn_bwd_apply_pool_vec_kernel, vec_blocks(total / 32), 256, 0, (const uint4*)y, (const uint4*)da, Ho, Wo, C / 8, scale,
                                                                                 shift, mu, invstd, sdz, sdzx, invM, total / 32, (uint4*)dy);
    NF_LAUNCHED();
    return NF_OK;
  }
  if (vec_ok(dtype, C, pool)) {
    nf_launch(bn_bwd_apply_vec_kernel, vec_blocks(total / 8), 256, 6 * C * sizeof(float), 
        (const uint4*)y, (const uint4*)da, C / 8, scale, shift, mu, invstd, sdz, sdzx, invM, total / 8, (uint4*)dy);
    NF_LAUNCHED();
    return NF_OK;
  }
  DISPATCH(dtype,
           (nf_launch(bn_bwd_apply_kernel<float>, nblk(total, 256), 256, 0, (const float*)y, (const float*)da, Ho, Wo, C, pool, scale, shift, mu, invstd, sdz, sdzx, invM, total, (float*)dy, nullptr)),
           (nf_launch(bn_bwd_apply_kernel<bf16>, nblk(total, 256), 256, 0, (const bf16*)y, (const bf16*)da, Ho, Wo, C, pool, scale, shift, mu, invstd, sdz, sdzx, invM, total, (bf16*)dy, nullptr)));
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_pad_channels(const void* x, size_t P, int C, int Cp, void* xpad) {
  if (C < 1 || C > 8 || Cp % 8) return NF_EUNSUPPORTED;
  nf_launch(pad_channels_kernel, nblk(P * (Cp / 8), 256), 256, 0, (const bf16*)x, P, C, Cp / 8, (uint4*)xpad);
  NF_LAUNCHED();
  return NF_OK;
}
int nf_k_pad_weights(const bf16* w, size_t rows, int C, int Cp, bf16* wpad) {
  nf_launch(pad_weights_kernel, nblk(rows * Cp, 256), 256, 0, w, rows, C, Cp, wpad);
  NF_LAUNCHED();
  return NF_OK;
}
int nf_k_unpad_grad_mirrored(const float* gwpad, int Co, int C, int Cp, float* gw) {
  nf_launch(unpad_grad_mirrored_kernel, nblk((size_t)9 * Co * C, 256), 256, 0, gwpad, Co, C, Cp, gw);
  NF_LAUNCHED();
  return NF_OK;
}
int nf_k_unpad_grad(const float* gwpad, size_t rows, int C, int Cp, float* gw) {
  nf_launch(unpad_grad_kernel, nblk(rows * C, 256), 256, 0, gwpad, rows, C, Cp, gw);
  NF_LAUNCHED();
  return NF_OK;
}

template <typename A>
static void sum_parts(const float* part, int splits, size_t n, float* out) {
  const bool vec = n % 4 == 0 && (((uintptr_t)part | (uintptr_t)out) & 15) == 0;
  if (splits >= 16) {
    if (vec) nf_launch(sum_parts_kernel<4, 8, A>, nblk(n, 128), 256, 0, part, splits, n, out);
    else nf_launch(sum_parts_kernel<1, 8, A>, nblk(n, 32), 256, 0, part, splits, n, out);
  } else {
    if (vec) nf_launch(sum_parts_kernel<4, 1, A>, nblk(n, 1024), 256, 0, part, splits, n, out);
    else nf_launch(sum_parts_kernel<1, 1, A>, nblk(n, 256), 256, 0, part, splits, n, out);
  }
}

int nf_k_sum_parts(const float* part, int splits, size_t n, float* out, bool fp64) {
  if (fp64) sum_parts<double>(part, splits, n, out);
  else sum_parts<float>(part, splits, n, out);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_sgd_multi(const SgdTable& tb_in, float lr, float momentum) {
  if (tb_in.count < 1 || tb_in.count > kSgdMaxArenas) return NF_EINVAL;
  SgdTable tb = tb_in;
  int blocks = 0;
  for (int a = 0; a < tb.count; ++a) {
    if (tb.n[a] % 4) return NF_EINVAL;
    tb.first_block[a] = blocks;
    blocks += (int)nblk(tb.n[a] / 4, 256);
  }
  nf_launch(sgd_multi_kernel, blocks, 256, 0, tb, lr, momentum);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_sgd(float* val, float* mom, const float* grad, bf16* shadow, size_t n, float lr, float momentum) {
  SgdTable tb{};
  tb.count = 1;
  tb.val[0] = val; tb.mom[0] = mom; tb.grad[0] = grad; tb.shadow[0] = shadow; tb.n[0] = n;
  return nf_k_sgd_multi(tb, lr, momentum);
}

int nf_k_shadow(const float* val, bf16* shadow, size_t n) {
  nf_launch(shadow_kernel, nblk(n, 256), 256, 0, val, shadow, n);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_k_gather(const void* cache, const int32_t* cache_labels, int cache_rows, const int32_t* idx, int count, size_t row_bytes,
                  void* out, int32_t* out_labels, int32_t* status) {
  const size_t row16 = row_bytes / 16;
  nf_launch(gather_kernel, nblk((size_t)count * row16, 256), 256, 0, (const uint4*)cache, cache_labels, cache_rows, idx,
                                                                         count, row16, (uint4*)out, out_labels, status);
  NF_LAUNCHED();
  return NF_OK;
}

// ---- BatchNorm without an activation (projection shortcut); NF_EUNSUPPORTED for channel counts the kernels above do not take
int nf_k_bn_plain_apply(int dtype, const void* y, size_t P, int C, const float* scale, const float* shift, void* out) {
  if (!vec2_ok(C, 0)) return NF_EUNSUPPORTED;
  const size_t n8 = P * C / 8;
  DISPATCH(dtype, (nf_launch(bn_apply_vec2_kernel<float, 2>, vec_blocks(n8), 256, 0, (const float*)y, C / 8, scale, shift, n8, (float*)out, nullptr)),
           (nf_launch(bn_apply_vec2_kernel<bf16, 2>, vec_blocks(n8), 256, 0, (const bf16*)y, C / 8, scale, shift, n8, (bf16*)out, nullptr)));
  NF_LAUNCHED();
  return NF_OK;
}
int nf_k_bn_plain_bwd_reduce(int dtype, const void* y, const void* dz, size_t P, int C, const float* mu, const float* invstd, float* red,
                             size_t red_floats, int* nblocks) {
  if (!vec2_ok(C, 0)) return NF_EUNSUPPORTED;
  const int nb = std::min(nf_k_channel_blocks(P, C), 296);  // two blocks per SM: each pays for its channel constants and its reduction
  if ((size_t)nb * 2 * C > red_floats) return NF_ENOWS;
  const int planes = 256 / (C / 8);
  DISPATCH(dtype, (nf_launch(bn_bwd_reduce_vec_kernel<float, 2>, nb, 256, 0, (const float*)y, (const float*)dz, P, C / 8, planes, nb, mu, mu, mu, invstd, red, nullptr, nullptr)),
           (nf_launch(bn_bwd_reduce_vec_kernel<bf16, 2>, nb, 256, 0, (const bf16*)y, (const bf16*)dz, P, C / 8, planes, nb, mu, mu, mu, invstd, red, nullptr, nullptr)));
  NF_LAUNCHED();
  *nblocks = nb;
  return NF_OK;
}
int nf_k_bn_plain_bwd_apply(int dtype, const void* y, const void* dz, size_t P, int C, const float* scale, const float* mu,
                            const float* invstd, const float* sdz, const float* sdzx, double M, void* dy) {
  if (!vec2_ok(C, 0)) return NF_EUNSUPPORTED;
  const size_t n8 = P * C / 8;
  const float invM = (float)(1.0 / M);
  DISPATCH(dtype, (nf_launch(bn_bwd_apply_vec2_kernel<float, 2, 1>, vec_blocks(n8), 256, 0, (const float*)y, (const float*)dz, C / 8, scale, mu, mu, invstd, sdz, sdzx, invM, n8, (float*)dy, nullptr)),
           (nf_launch(bn_bwd_apply_vec2_kernel<bf16, 2, 1>, vec_blocks(n8), 256, 0, (const bf16*)y, (const bf16*)dz, C / 8, scale, mu, mu, invstd, sdz, sdzx, invM, n8, (bf16*)dy, nullptr)));
  NF_LAUNCHED();
  return NF_OK;
}
