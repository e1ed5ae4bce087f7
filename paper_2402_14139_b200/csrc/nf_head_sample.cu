// The head of a step, one block per sample: average pool of h to 2 x 2, linear layer, loss, and the gradients back to h, in one
// kernel; the gradients that sum over the batch (linear weights and bias, auxiliary conv bias) and the mean loss in a second.
//
// These heads are pure latency (64 to 512 samples, at most a few million multiply-adds): as separate pool, pool-finish, loss,
// weight-gradient, dh and bias kernels they took 55 of 215 us of a 32 x 32-pixel layer at 128 samples, each kernel a launch and a
// few dependent trips to L2 (the weight gradient with one block per class and one load at a time alone 20 us).  Here a sample's
// h is read once, kept in shared memory until dh is written, and every loop has several independent loads in flight.
// fp32 throughout, every sum in a fixed order.
#include <math.h>

#include "nf_internal.h"
#include "nf_ldst.cuh"

namespace {

constexpr int kHT = 512;  // threads of the per-sample kernel: with at most one block per SM the most that still share a barrier cheaply
constexpr int kWarps = kHT / 32;

struct HeadArgs {
  const void* h;        // [N][Ha][Wa][F], or NULL when the pooled inputs come from `part`
  const float* part;    // pooling partials of the fused aux forward: [N][th][tw][4][F] (14 x 8-pixel tiles, four warps each)
  int th, tw;
  int N, Ha, Wa, F, K;
  const int32_t* labels;
  const float *Wf, *bf;
  float *p, *logits, *dlogits, *dp, *lossn;
  int32_t* status;
  void* dh;             // NULL: dh is written elsewhere
  float* bred;          // [N][F] sums of the stored dh over the sample's pixels (with dh)
  int loss_kind, n_scale;
};

// reduction over the block; every thread gets the result
__device__ __forceinline__ float block_all(float v, float* sm, bool is_max) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float u = __shfl_xor_sync(0xffffffffu, v, o);
    v = is_max ? fmaxf(v, u) : v + u;
  }
  __syncthreads();  // sm may still be read from the reduction before
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  v = sm[0];
#pragma unroll
  for (int w = 1; w < kWarps; ++w) v = is_max ? fmaxf(v, sm[w]) : v + sm[w];
  return v;
}

// F8 = F / 8 in {1, 2, 4, 8}: a warp covers whole pixels, and its lanes with equal lane % F8 hold the same channels.
template <typename T, int F8>
__global__ void __launch_bounds__(kHT) head_sample_kernel(const HeadArgs a) {
  nf_pdl_begin();
  constexpr int F = F8 * 8, D = 4 * F;
  extern __shared__ __align__(16) uint8_t dyn[];
  float* ps = reinterpret_cast<float*>(dyn);  // [D] pooled inputs, then their gradient
  float* ls = ps + D;                         // [K] logits, then dlogits
  float* rd = ls + ((a.K + 3) & ~3);          // [kWarps][D] reductions
  float* tab = rd + kWarps * D;               // [9][F] dh of a positive h, by row class and column class of its pixel
  T* hs = reinterpret_cast<T*>(tab + 9 * F);  // the sample's h
  const int n = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int px = a.Ha * a.Wa, g = t % F8;
  // rows [0, r1) belong to the upper bins, [r0, Ha) to the lower ones: the middle row of an odd height to both; columns likewise
  const int r0 = a.Ha / 2, r1 = (a.Ha + 1) / 2, c0 = a.Wa / 2, c1 = (a.Wa + 1) / 2;

  if (a.h) {
    float s[4][8];
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int e = 0; e < 8; ++e) s[b][e] = 0.f;
    const T* hn = reinterpret_cast<const T*>(a.h) + (size_t)n * px * F;
    constexpr int kStep = kHT / F8;
    for (int q0 = t / F8; q0 < px; q0 += 4 * kStep) {  // four loads in flight
      float v[4][8];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (q0 + u * kStep < px) ld8(hn + (size_t)(q0 + u * kStep) * F + g * 8, v[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int q = q0 + u * kStep;
        if (q < px) {
          if (a.dh) st8(hs + (size_t)q * F + g * 8, v[u]);
          const int i = q / a.Wa, j = q - i * a.Wa;
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const bool in = (b & 2 ? i >= r0 : i < r1) && (b & 1 ? j >= c0 : j < c1);
#pragma unroll
            for (int e = 0; e < 8; ++e) s[b][e] += in ? v[u][e] : 0.f;
          }
        }
      }
    }
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int e = 0; e < 8; ++e) {
#pragma unroll
        for (int o = 16; o >= F8; o >>= 1) s[b][e] += __shfl_xor_sync(0xffffffffu, s[b][e], o);
        if (lane < F8) rd[warp * D + (lane * 8 + e) * 4 + b] = s[b][e];
      }
    __syncthreads();
    for (int d = t; d < D; d += kHT) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) v += rd[w * D + d];
      const int b = d & 3;
      v /= (float)((b & 2 ? a.Ha - r0 : r1) * (b & 1 ? a.Wa - c0 : c1));
      ps[d] = v;
      a.p[(size_t)n * D + d] = v;
    }
  } else {
    // a warp per bin and quarter of the bin's partials; lanes run over the channels
    const int qh = a.th / 2, qw = a.tw / 2, cnt = qh * qw * 4, b = warp & 3, sub = warp >> 2;
    constexpr int kSub = kWarps / 4;
    for (int f = lane; f < F; f += 32) {
      float v = 0.f;
      int k = sub;
      const float* base = a.part + (((size_t)n * a.th + (b >> 1) * qh) * a.tw + (b & 1) * qw) * 4 * F + f;
      auto at = [&](int kk) { return base[((size_t)((kk >> 2) / qw) * a.tw + (kk >> 2) % qw) * 4 * F + (size_t)(kk & 3) * F]; };
      for (; k + 7 * kSub < cnt; k += 8 * kSub) {
        float u[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) u[e] = at(k + e * kSub);
#pragma unroll
        for (int e = 0; e < 8; ++e) v += u[e];
      }
      for (; k < cnt; k += kSub) v += at(k);
      rd[sub * D + f * 4 + b] = v;
    }
    __syncthreads();
    for (int d = t; d < D; d += kHT) {
      float v = 0.f;
#pragma unroll
      for (int w = 0; w < kSub; ++w) v += rd[w * D + d];
      v *= 1.f / (float)(r0 * c0);
      ps[d] = v;
      a.p[(size_t)n * D + d] = v;
    }
  }
  __syncthreads();

  // logits: kLpc lanes per class, each with 4 (or 8) of the inputs in registers; four classes at a time per lane group
  constexpr int kLpc = F < 32 ? F : 32, kVec = F / kLpc, kGroups = kHT / kLpc;
  {
    const int l = t % kLpc, grp = t / kLpc;
    float4 x[kVec];
#pragma unroll
    for (int v = 0; v < kVec; ++v) x[v] = *reinterpret_cast<const float4*>(ps + (l + v * kLpc) * 4);
    for (int kb = 0; kb < a.K; kb += 4 * kGroups) {  // the same trips for every thread: whole warps in the shuffles
      const int k0 = kb + grp;
      float s[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int k = k0 + u * kGroups;
        s[u] = 0.f;
        if (k < a.K) {
#pragma unroll
          for (int v = 0; v < kVec; ++v) {
            const float4 w = *reinterpret_cast<const float4*>(a.Wf + (size_t)k * D + (l + v * kLpc) * 4);
            s[u] = fmaf(w.x, x[v].x, s[u]);
            s[u] = fmaf(w.y, x[v].y, s[u]);
            s[u] = fmaf(w.z, x[v].z, s[u]);
            s[u] = fmaf(w.w, x[v].w, s[u]);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
#pragma unroll
        for (int o = kLpc / 2; o > 0; o >>= 1) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
        const int k = k0 + u * kGroups;
        if (l == 0 && k < a.K) ls[k] = s[u] + a.bf[k];
      }
    }
  }
  __syncthreads();
  int lab = a.labels[n];
  if (lab < 0 || lab >= a.K) {
    if (t == 0) atomicOr(a.status, NF_ELABEL);
    lab = lab < 0 ? 0 : a.K - 1;
  }
  float* lrow = a.logits + (size_t)n * a.K;
  float* grow = a.dlogits + (size_t)n * a.K;
  if (a.loss_kind == 1) {  // mean squared error against the one-hot target
    float se = 0.f;
    const float sc = 2.f / ((float)a.n_scale * (float)a.K);
    for (int k = t; k < a.K; k += kHT) {
      const float l = ls[k], e = l - (k == lab ? 1.f : 0.f);
      se = fmaf(e, e, se);
      lrow[k] = l;
      grow[k] = e * sc;
      ls[k] = e * sc;
    }
    se = block_all(se, rd, false);
    if (t == 0) a.lossn[n] = se / (float)a.K;
  } else {
    float mx = -INFINITY;
    for (int k = t; k < a.K; k += kHT) mx = fmaxf(mx, ls[k]);
    mx = block_all(mx, rd, true);
    float se = 0.f;
    for (int k = t; k < a.K; k += kHT) se += expf(ls[k] - mx);
    se = block_all(se, rd, false);
    const float lse = mx + logf(se);
    if (t == 0) a.lossn[n] = lse - ls[lab];
    __syncthreads();
    const float invN = 1.f / (float)a.n_scale;
    for (int k = t; k < a.K; k += kHT) {
      const float l = ls[k], gr = (expf(l - lse) - (k == lab ? 1.f : 0.f)) * invN;
      lrow[k] = l;
      grow[k] = gr;
      ls[k] = gr;
    }
  }
  __syncthreads();

  // dp[d] = sum_k dlogits[k] Wf[k][d]: the classes in kG contiguous ranges, the range sums added in order
  constexpr int kG = kHT / D;
  {
    const int d = t % D, kg = t / D, per = (a.K + kG - 1) / kG, ka = kg * per, kb = min(a.K, ka + per);
    float s = 0.f;
    int k = ka;
    for (; k + 7 < kb; k += 8) {
      float w[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) w[u] = a.Wf[(size_t)(k + u) * D + d];
#pragma unroll
      for (int u = 0; u < 8; ++u) s = fmaf(ls[k + u], w[u], s);
    }
    for (; k < kb; ++k) s = fmaf(ls[k], a.Wf[(size_t)k * D + d], s);
    rd[kg * D + d] = s;
  }
  __syncthreads();
  for (int d = t; d < D; d += kHT) {
    float v = 0.f;
#pragma unroll
    for (int q = 0; q < kG; ++q) v += rd[q * D + d];
    a.dp[(size_t)n * D + d] = v;
    ps[d] = v;
  }
  if (!a.dh) return;
  __syncthreads();
  for (int i = t; i < 9 * F; i += kHT) {  // class 0: first bin only, 1: second bin only, 2: both
    const int f = i % F, cc = (i / F) % 3, rc = i / (3 * F);
    float v = 0.f;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int u = b >> 1, w = b & 1;
      if ((rc == 2 || rc == u) && (cc == 2 || cc == w)) v += ps[f * 4 + b] / (float)((u ? a.Ha - r0 : r1) * (w ? a.Wa - c0 : c1));
    }
    tab[i] = v;
  }
  __syncthreads();
  float bs[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) bs[e] = 0.f;
  T* dhn = reinterpret_cast<T*>(a.dh) + (size_t)n * px * F;
  for (int q = t / F8; q < px; q += kHT / F8) {
    const int i = q / a.Wa, j = q - i * a.Wa;
    const int rc = i < r0 ? 0 : i >= r1 ? 1 : 2, cc = j < c0 ? 0 : j >= c1 ? 1 : 2;
    float v[8], o[8];
    ld8(hs + (size_t)q * F + g * 8, v);
    ld8(tab + (rc * 3 + cc) * F + g * 8, o);
#pragma unroll
    for (int e = 0; e < 8; ++e) o[e] = v[e] > 0.f ? o[e] : 0.f;
    st8(dhn + (size_t)q * F + g * 8, o);
#pragma unroll
    for (int e = 0; e < 8; ++e) bs[e] += o[e];  // the bias gradient sums the values as stored
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) {
#pragma unroll
    for (int o = 16; o >= F8; o >>= 1) bs[e] += __shfl_xor_sync(0xffffffffu, bs[e], o);
    if (lane < F8) rd[warp * F + lane * 8 + e] = bs[e];
  }
  __syncthreads();
  for (int f = t; f < F; f += kHT) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) v += rd[w * F + f];
    a.bred[(size_t)n * F + f] = v;
  }
}

// Sums over the batch.  Blocks [0, K * DT): class k = b / DT, inputs 32 (b % DT) ..: gWf, and gbf where b % DT == 0; 32 inputs x
// 8 sample lanes, eight samples in flight per lane, lanes added in order.  Then FT blocks of 32 filters: gba from the per-sample
// sums of dh (fp64, none when bred is NULL); the last block: the mean loss (fp64).
__global__ void __launch_bounds__(256) head_batch_kernel(const float* __restrict__ p, const float* __restrict__ dl,
                                                         const float* __restrict__ lossn, const float* __restrict__ bred, int N, int D,
                                                         int K, int DT, int FT, int F, float* __restrict__ gWf, float* __restrict__ gbf,
                                                         float* __restrict__ gba, float* __restrict__ loss_out,
                                                         int32_t* __restrict__ status, int n_scale) {
  nf_pdl_begin();
  __shared__ double sd[8][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, b = blockIdx.x;
  if (b < K * DT) {
    float(*sf)[33] = reinterpret_cast<float(*)[33]>(sd);
    const int k = b / DT, d = (b % DT) * 32 + tx;
    float s = 0.f, sb = 0.f;
    int n = ty;
    for (; n + 56 < N; n += 64) {
      float u[8], v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        u[e] = dl[(size_t)(n + 8 * e) * K + k];
        v[e] = d < D ? p[(size_t)(n + 8 * e) * D + d] : 0.f;
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        s = fmaf(u[e], v[e], s);
        sb += u[e];
      }
    }
    for (; n < N; n += 8) {
      const float u = dl[(size_t)n * K + k];
      s = fmaf(u, d < D ? p[(size_t)n * D + d] : 0.f, s);
      sb += u;
    }
    sf[ty][tx] = s;
    if (tx == 0) sf[ty][32] = sb;
    __syncthreads();
    if (ty == 0) {
      float v = 0.f;
#pragma unroll
      for (int q = 0; q < 8; ++q) v += sf[q][tx];
      if (d < D) gWf[(size_t)k * D + d] = v;
      if (tx == 0 && b % DT == 0) {
        float c = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) c += sf[q][32];
        gbf[k] = c;
      }
    }
    return;
  }
  const bool loss = b == K * DT + FT;
  const int f = (b - K * DT) * 32 + tx;
  double s = 0.0;
  if (loss) {
    for (int n = threadIdx.x; n < N; n += 256) s += (double)lossn[n];
  } else if (f < F) {
#pragma unroll 8
    for (int n = ty; n < N; n += 8) s += (double)bred[(size_t)n * F + f];
  }
  sd[ty][tx] = s;
  __syncthreads();
  if (loss && ty == 0) {
    double v = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) v += sd[q][tx];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (tx == 0) {
      const float L = (float)(v / (double)n_scale);
      *loss_out = L;
      if (!isfinite(L)) atomicOr(status, NF_ENONFINITE);
    }
  } else if (!loss && ty == 0 && f < F) {
    double v = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) v += sd[q][tx];
    gba[f] = (float)v;
  }
}

constexpr size_t kSmemMax = 200 * 1024;

size_t fixed_smem(int F, int K) { return ((size_t)4 * F + ((K + 3) & ~3) + (size_t)kWarps * 4 * F + 9 * F) * 4; }

template <typename T, int F8>
int run_sample(const HeadArgs& a, size_t smem) {
  static bool done[64];  // function attributes belong to a device's context: set once per device
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!done[dev]) {
    NF_CUDA(cudaFuncSetAttribute(head_sample_kernel<T, F8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
    done[dev] = true;
  }
  nf_launch(head_sample_kernel<T, F8>, a.N, kHT, smem, a);
  NF_LAUNCHED();
  return NF_OK;
}

}  // namespace

// 0: not covered; 1: everything but dh; 2: dh as well.  Filters in 8, 16, 32, 64; dh where the sample's h fits beside the tables.
int nf_head_sample_mode(int dtype, int Ha, int Wa, int F, int K) {
  if ((F != 8 && F != 16 && F != 32 && F != 64) || K > 16384 || Ha < 2 || Wa < 2) return 0;
  if (fixed_smem(F, K) > kSmemMax) return 0;
  return fixed_smem(F, K) + (size_t)Ha * Wa * F * nf_esize(dtype) <= kSmemMax ? 2 : 1;
}

int nf_head_sample_step(const NfHeadIo& io, int dtype, int N, int Ha, int Wa, int F, int K, int loss_kind, int n_scale) {
  HeadArgs a{};
  a.h = io.h; a.part = io.part; a.th = Ha / 8; a.tw = Wa / 14;
  a.N = N; a.Ha = Ha; a.Wa = Wa; a.F = F; a.K = K;
  a.labels = io.labels; a.Wf = io.Wf; a.bf = io.bf;
  a.p = io.p; a.logits = io.logits; a.dlogits = io.dlogits; a.dp = io.dp; a.lossn = io.lossn; a.status = io.status;
  a.dh = io.dh; a.bred = io.bred; a.loss_kind = loss_kind; a.n_scale = n_scale;
  const size_t smem = fixed_smem(F, K) + (io.dh ? (size_t)Ha * Wa * F * nf_esize(dtype) : 0);
  int rc;
  if (dtype == NF_F32)
    rc = F == 8 ? run_sample<float, 1>(a, smem) : F == 16 ? run_sample<float, 2>(a, smem)
       : F == 32 ? run_sample<float, 4>(a, smem) : run_sample<float, 8>(a, smem);
  else
    rc = F == 8 ? run_sample<bf16, 1>(a, smem) : F == 16 ? run_sample<bf16, 2>(a, smem)
       : F == 32 ? run_sample<bf16, 4>(a, smem) : run_sample<bf16, 8>(a, smem);
  if (rc != NF_OK) return rc;
  const int D = 4 * F, DT = (D + 31) / 32, FT = io.dh ? (F + 31) / 32 : 0;
  nf_launch(head_batch_kernel, (unsigned)(K * DT + FT + 1), 256, 0, io.p, io.dlogits, io.lossn, io.bred, N, D, K, DT, FT, F, io.gWf, io.gbf, io.gba,
            io.loss_out, io.status, n_scale);
  NF_LAUNCHED();
  return NF_OK;
}
