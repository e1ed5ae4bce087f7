// The head of a step, one block per sample: average pool of h to 2 x 2, linear layer, loss, and the gradients back to h, in one
// kernel; the gradients that sum over the batch (linear weights and bias, auxiliary conv bias) and the mean loss in a second.
//
// These heads are pure latency (64 to 512 samples, at most a few million multiply-adds): as separate pool, pool-finish, loss,
// weight-gradient, dh and bias kernels they took 55 of 215 us of a 32 x 32-pixel layer at 128 samples, each kernel a launch and a
// few dependent trips to L2 (the weight gradient with one block per class and one load at a time alone 20 us); now 12 + 3 us.
// A sample's h is read once; its sign bits stay in shared memory until dh is written, the linear weights take h's place there.
// Loads come in batches whose indexes are clamped instead of guarded, so that no branch separates them, and loops stay rolled:
// at this size the fetch of unrolled code costs more than it saves.
// fp32 throughout, every sum in a fixed order: the order of the kernels for other sizes (nf_elem.cu, nf_head_small.cu), so that a
// layer computes the same bits whichever of them its size selects.
#include <math.h>

#include <algorithm>

#include "nf_internal.h"
#include "nf_ldst.cuh"

namespace {

constexpr int kHT = 512;  // threads of the per-sample kernel: with at most one block per SM the most that still share a barrier cheaply
constexpr int kWarps = kHT / 32;

struct HeadArgs {
  const void* h;        // [N][Ha][Wa][F], or NULL when the pooled inputs come from `part` or, where that is NULL too, are in p
  const float* part;    // pooling partials of the fused aux forward: [N][th][tw][4][F] (14 x 8-pixel tiles, four warps each)
  int slices, planes;   // order of a bin's sum: `slices` ranges of its pixels, `planes` interleaved chains in each
  int even, dh_even;    // the mean as a product with 1 / |bin| (else a quotient), in the pool and in dh
  int th, tw;
  int N, Ha, Wa, F, K;
  const int32_t* labels;
  const float *Wf, *bf;
  float *p, *logits, *dlogits, *dp, *lossn;
  int32_t* status;
  void* dh;             // with h; else dh is written elsewhere
  float* bred;          // [N][F] sums of the stored dh over the sample's pixels (with dh)
  int loss_kind, n_scale;
  int groups;           // class ranges of the sums in dp
  int KS, S, parts;     // SL: classes per slice, slices, ranges their shares are folded in
  int chunk;            // classes whose weights fit shared memory at a time
  size_t off;           // where the offsets and the sign bits lie in shared memory
};

// eight values as they are in memory
template <typename T> struct Raw8;
template <> struct Raw8<bf16> {
  uint4 u;
  __device__ __forceinline__ void load(const bf16* p) { u = *reinterpret_cast<const uint4*>(p); }
  __device__ __forceinline__ void store(bf16* p) const { *reinterpret_cast<uint4*>(p) = u; }
  __device__ __forceinline__ uint32_t positive() const {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
    uint32_t b = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      b |= (__uint_as_float(w[i] << 16) > 0.f ? 1u : 0u) << (2 * i);
      b |= (__uint_as_float(w[i] & 0xffff0000u) > 0.f ? 1u : 0u) << (2 * i + 1);
    }
    return b;
  }
};
template <> struct Raw8<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p) {
    a = *reinterpret_cast<const float4*>(p);
    b = *reinterpret_cast<const float4*>(p + 4);
  }
  __device__ __forceinline__ void store(float* p) const {
    *reinterpret_cast<float4*>(p) = a;
    *reinterpret_cast<float4*>(p + 4) = b;
  }
  __device__ __forceinline__ uint32_t positive() const {
    const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint32_t r = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) r |= (v[i] > 0.f ? 1u : 0u) << i;
    return r;
  }
};
__device__ __forceinline__ float2 pair(const bf16* p) {
  const uint32_t u = *reinterpret_cast<const uint32_t*>(p);
  return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}
__device__ __forceinline__ float2 pair(const float* p) { return *reinterpret_cast<const float2*>(p); }

// maximum over the block, for every thread
__device__ __forceinline__ float block_max(float v, float* sm) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  v = sm[0];
#pragma unroll
  for (int w = 1; w < kWarps; ++w) v = fmaxf(v, sm[w]);
  __syncthreads();
  return v;
}
// sum of the values of the first 256 threads as a binary tree (t with t + 128, + 64, ...), for every thread
__device__ __forceinline__ float tree_sum256(float v, float* sm) {
  const int t = threadIdx.x;
  if (t < 256) sm[t] = v;
  __syncthreads();
  if (t < 32) {
    float q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = sm[t + 32 * i] + sm[t + 32 * i + 128];
    v = (q[0] + q[2]) + (q[1] + q[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (t == 0) sm[256] = v;
  }
  __syncthreads();
  v = sm[256];
  __syncthreads();
  return v;
}

template <int F8> constexpr int kRd = kWarps * 32 * F8 < 1024 ? 1024 : kWarps * 32 * F8;

// F8 = F / 8 in {1, 2, 4, 8}: a warp covers whole pixels, and its lanes with equal lane % F8 hold the same channels.
// STAGE: the linear weights fit shared memory.  SL: many classes per sample, sums by class slices as in nf_head_small.cu.
template <typename T, int F8, bool STAGE, bool SL>
__global__ void __launch_bounds__(kHT) head_sample_kernel(const HeadArgs a) {
  nf_pdl_begin();
  constexpr int F = F8 * 8, D = 4 * F;
  extern __shared__ __align__(16) uint8_t dyn[];
  float* ps = reinterpret_cast<float*>(dyn);  // [D] pooled inputs, then their gradient
  float* ls = ps + D;                         // [K] bias, logits, dlogits
  float* rd = ls + ((a.K + 3) & ~3);          // reductions: [kWarps][D] or [4][256]
  float* tab = rd + kRd<F8>;                  // [9][F] dh of a positive h, by row class and column class of its pixel
  T* hs = reinterpret_cast<T*>(tab + 9 * F);  // the sample's h
  uint32_t* off = reinterpret_cast<uint32_t*>(dyn + a.off);  // byte offset in the image of a bin's k-th pixel
  uint8_t* mask = reinterpret_cast<uint8_t*>(off + (((a.Ha + 1) / 2) * ((a.Wa + 1) / 2) + 3) / 4 * 4);  // bit e of [unit]: h > 0
  const int n = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int px = a.Ha * a.Wa, g = t % F8;
  // rows [0, r1) belong to the upper bins, [r0, Ha) to the lower ones: the middle row of an odd height to both; columns likewise
  const int r0 = a.Ha / 2, r1 = (a.Ha + 1) / 2, c0 = a.Wa / 2, c1 = (a.Wa + 1) / 2;
  int lab = a.labels[n];
  for (int k = t; k < a.K; k += kHT) ls[k] = a.bf[k];

  if (a.h) {
    {
      const T* src = reinterpret_cast<const T*>(a.h) + (size_t)n * px * F;
      const int units = px * F8;  // of eight values
#pragma unroll 1
      for (int i0 = t; i0 < units; i0 += 8 * kHT) {
        Raw8<T> q[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) q[j].load(src + (size_t)min(i0 + j * kHT, units - 1) * 8);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (i0 + j * kHT < units) {
            q[j].store(hs + (size_t)(i0 + j * kHT) * 8);
            mask[i0 + j * kHT] = (uint8_t)q[j].positive();
          }
      }
    }
    const int bw = c1, cnt = r1 * c1;  // all four bins have this size
    for (int k = t; k < cnt; k += kHT) off[k] = (uint32_t)((k / bw) * a.Wa + k % bw) * F * sizeof(T);
    __syncthreads();
    // a thread per (bin, slice, channel pair): sixteen chains at a time, each in pixel order, added in chain order
    for (int i = t; i < 2 * a.slices * F; i += kHT) {
      const int f = (i % (F / 2)) * 2, sl = (i / (F / 2)) % a.slices, bin = i / (F / 2 * a.slices);
      const uint8_t* hb = reinterpret_cast<const uint8_t*>(hs + ((size_t)(bin & 2 ? r0 : 0) * a.Wa + (bin & 1 ? c0 : 0)) * F + f);
      const int k0 = cnt * sl / a.slices, k1 = cnt * (sl + 1) / a.slices;
      float ta = 0.f, tb = 0.f;
      const int planes = min(a.planes, k1 - k0);
      const bool whole = planes % 16 == 0 && (k1 - k0) % a.planes == 0 && k0 % 4 == 0;
#pragma unroll 1
      for (int pl = 0; pl < planes; pl += 16) {
        float ca[16], cb[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) ca[u] = cb[u] = 0.f;
#pragma unroll 1
        for (int k = k0 + pl; k < k1; k += a.planes) {
          uint32_t o[16];
          if (whole) {
#pragma unroll
            for (int u = 0; u < 16; u += 4) {
              const uint4 x = *reinterpret_cast<const uint4*>(off + k + u);
              o[u] = x.x; o[u + 1] = x.y; o[u + 2] = x.z; o[u + 3] = x.w;
            }
          } else {
#pragma unroll
            for (int u = 0; u < 16; ++u) o[u] = off[min(k + u, cnt - 1)];
          }
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const float2 v = pair(reinterpret_cast<const T*>(hb + o[u]));
            const bool in = whole || (k + u < k1 && pl + u < planes);
            ca[u] += in ? v.x : 0.f;
            cb[u] += in ? v.y : 0.f;
          }
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          ta += ca[u];
          tb += cb[u];
        }
      }
      rd[sl * D + f * 4 + bin] = ta;
      rd[sl * D + f * 4 + 4 + bin] = tb;
    }
    __syncthreads();
    for (int d = t; d < D; d += kHT) {
      float v = 0.f;
      for (int sl = 0; sl < a.slices; ++sl) v += rd[sl * D + d];
      v = a.even ? v * (1.f / (float)cnt) : v / (float)cnt;
      ps[d] = v;
      a.p[(size_t)n * D + d] = v;
    }
  } else if (!a.part) {
    for (int d = t; d < D; d += kHT) ps[d] = a.p[(size_t)n * D + d];
  } else {
    // per bin 256 / F chains over its partials, added in order; eight loads in flight
    const int qh = a.th / 2, qw = a.tw / 2, cnt = qh * qw * 4;
    constexpr int kLn = 256 / F;
    for (int i = t; i < 1024; i += kHT) {
      const int f = i % F, ln = (i % 256) / F, b = i / 256;
      const float* base = a.part + (((size_t)n * a.th + (b >> 1) * qh) * a.tw + (b & 1) * qw) * 4 * F + f;
      float v = 0.f;
#pragma unroll 1
      for (int k = ln; k < cnt; k += 8 * kLn) {
        float u[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int kk = min(k + e * kLn, cnt - 1), tq = kk >> 2;
          u[e] = base[((size_t)(tq / qw) * a.tw + tq % qw) * 4 * F + (size_t)(kk & 3) * F];
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) v += k + e * kLn < cnt ? u[e] : 0.f;
      }
      rd[i] = v;
    }
    __syncthreads();
    for (int d = t; d < D; d += kHT) {
      float v = 0.f;
#pragma unroll 4
      for (int l = 0; l < kLn; ++l) v += rd[(d & 3) * 256 + l * F + (d >> 2)];
      v *= 1.f / (float)(r0 * c0);
      ps[d] = v;
      a.p[(size_t)n * D + d] = v;
    }
  }
  __syncthreads();

  // The linear weights are read twice, by rows and by columns: by rows through shared memory, in h's place, `chunk` classes at a
  // time (padded against bank conflicts); by columns from there where all of them fit, else from L2.
  constexpr int kRow = D + 4;
  float* ws = reinterpret_cast<float*>(hs);
#pragma unroll 1
  for (int kc = 0; kc < a.K; kc += a.chunk) {
    const int kn = min(a.chunk, a.K - kc), units = kn * (D / 4);
    const float4* src = reinterpret_cast<const float4*>(a.Wf + (size_t)kc * D);
    if (kc) __syncthreads();
#pragma unroll 1
    for (int i0 = t; i0 < units; i0 += 8 * kHT) {
      float4 q[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) q[j] = src[min(i0 + j * kHT, units - 1)];
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (i0 + j * kHT < units) {
          const int i = i0 + j * kHT;
          *reinterpret_cast<float4*>(ws + (size_t)(i / (D / 4)) * kRow + (i % (D / 4)) * 4) = q[j];
        }
    }
    __syncthreads();
    // logits: a thread per class, inputs in order
    for (int k = t; k < kn; k += kHT) {
      float v = ls[kc + k];  // the bias
      const float4* w = reinterpret_cast<const float4*>(ws + (size_t)k * kRow);
      const float4* x = reinterpret_cast<const float4*>(ps);
#pragma unroll 8
      for (int d = 0; d < D / 4; ++d) {
        const float4 wv = w[d], xv = x[d];
        v = fmaf(wv.x, xv.x, v);
        v = fmaf(wv.y, xv.y, v);
        v = fmaf(wv.z, xv.z, v);
        v = fmaf(wv.w, xv.w, v);
      }
      ls[kc + k] = v;
    }
  }
  const float* wrow = STAGE ? ws : a.Wf;
  constexpr int pitch = STAGE ? kRow : D;
  __syncthreads();
  if (lab < 0 || lab >= a.K) {
    if (t == 0) atomicOr(a.status, NF_ELABEL);
    lab = lab < 0 ? 0 : a.K - 1;
  }
  float* lrow = a.logits + (size_t)n * a.K;
  float* grow = a.dlogits + (size_t)n * a.K;
  if constexpr (SL) {
    // shares of the slices (maximum and sum of exponentials, or the squared error), folded in `parts` ranges, then those in order
    float* sh = rd;  // [S][2]
    for (int j = t; j < a.S; j += kHT) {
      const int k0 = j * a.KS, k1 = min(a.K, k0 + a.KS);
      float m = 0.f, q = 0.f;
      if (a.loss_kind == 1) {
        for (int k = k0; k < k1; ++k) {
          const float e = ls[k] - (k == lab ? 1.f : 0.f);
          q = fmaf(e, e, q);
        }
      } else {
        m = -INFINITY;
        for (int k = k0; k < k1; ++k) m = fmaxf(m, ls[k]);
#pragma unroll 4
        for (int k = k0; k < k1; ++k) q += expf(ls[k] - m);
      }
      sh[2 * j] = m;
      sh[2 * j + 1] = q;
    }
    __syncthreads();
    auto fold = [&](float& m, float& q, float mj, float qj) {
      if (a.loss_kind == 1) {
        q += qj;
      } else {
        const float mm = fmaxf(m, mj);
        q = q * expf(m - mm) + qj * expf(mj - mm);
        m = mm;
      }
    };
    float* fp = sh + 2 * a.S;  // [parts][2]
    if (t < a.parts) {
      float m = -INFINITY, q = 0.f;
      for (int j = t; j < a.S; j += a.parts) fold(m, q, sh[2 * j], sh[2 * j + 1]);
      fp[2 * t] = m;
      fp[2 * t + 1] = q;
    }
    __syncthreads();
    if (t == 0) {
      float m = fp[0], q = fp[1];
      for (int i = 1; i < a.parts; ++i)
        if (a.loss_kind == 1 || fp[2 * i] > -INFINITY) fold(m, q, fp[2 * i], fp[2 * i + 1]);
      const float lse = a.loss_kind == 1 ? q : m + logf(q);
      fp[0] = lse;
      a.lossn[n] = a.loss_kind == 1 ? q / (float)a.K : lse - ls[lab];
    }
    __syncthreads();
    const float lse = fp[0], invN = 1.f / (float)a.n_scale, sc = 2.f / ((float)a.n_scale * (float)a.K);
    for (int k = t; k < a.K; k += kHT) {
      const float l = ls[k], hit = k == lab ? 1.f : 0.f;
      const float gr = a.loss_kind == 1 ? (l - hit) * sc : (expf(l - lse) - hit) * invN;
      lrow[k] = l;
      grow[k] = gr;
      ls[k] = gr;
    }
  } else if (a.loss_kind == 1) {  // mean squared error against the one-hot target
    float se = 0.f;
    const float sc = 2.f / ((float)a.n_scale * (float)a.K);
    if (t < 256)
      for (int k = t; k < a.K; k += 256) {
        const float l = ls[k], e = l - (k == lab ? 1.f : 0.f);
        se = fmaf(e, e, se);
        lrow[k] = l;
        grow[k] = e * sc;
        ls[k] = e * sc;
      }
    se = tree_sum256(se, rd);
    if (t == 0) a.lossn[n] = se / (float)a.K;
  } else {
    float mx = -INFINITY;
    for (int k = t; k < a.K; k += kHT) mx = fmaxf(mx, ls[k]);
    mx = block_max(mx, rd);
    float se = 0.f;
    if (t < 256)
      for (int k = t; k < a.K; k += 256) se += expf(ls[k] - mx);
    se = tree_sum256(se, rd);
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

  // dp[d] = sum_k dlogits[k] Wf[k][d]: the classes in contiguous ranges, each in order.  The range sums are added in order, or (SL:
  // the ranges are the slices) as four interleaved chains, (0 + 1) + (2 + 3).
  const int kG = SL ? a.S : a.groups, per = SL ? a.KS : (a.K + kG - 1) / kG;
  float* sums = SL ? ws : rd;  // [kG][D]
  for (int i = t; i < kG * D; i += kHT) {
    const int d = i % D, ka = i / D * per, kb = min(a.K, ka + per);
    float s = 0.f;
#pragma unroll 1
    for (int k = ka; k < kb; k += 16) {
      float w[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) w[u] = wrow[(size_t)min(k + u, kb - 1) * pitch + d];
#pragma unroll
      for (int u = 0; u < 16; ++u)
        if (k + u < kb) s = fmaf(ls[k + u], w[u], s);
    }
    sums[i] = s;
  }
  __syncthreads();
  for (int d = t; d < D; d += kHT) {
    float v = 0.f;
    if constexpr (SL) {
      float c[4] = {0.f, 0.f, 0.f, 0.f};
      const int S4 = kG & ~3;
#pragma unroll 4
      for (int q = 0; q < S4; ++q) c[q & 3] += sums[q * D + d];
      for (int q = S4; q < kG; ++q) c[0] += sums[q * D + d];
      v = (c[0] + c[1]) + (c[2] + c[3]);
    } else {
      for (int q = 0; q < kG; ++q) v += sums[q * D + d];
    }
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
      if ((rc == 2 || rc == u) && (cc == 2 || cc == w)) v += a.dh_even ? ps[f * 4 + b] * (1.f / (float)(r1 * c1)) : ps[f * 4 + b] / (float)(r1 * c1);
    }
    tab[i] = v;
  }
  __syncthreads();
  float bs[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) bs[e] = 0.f;
  T* dhn = reinterpret_cast<T*>(a.dh) + (size_t)n * px * F;
#pragma unroll 2
  for (int i = t; i < px * F8; i += kHT) {  // kHT is a multiple of F8: the thread's channels stay
    const int q = i / F8, ii = q / a.Wa, jj = q - ii * a.Wa;
    const int rc = ii < r0 ? 0 : ii >= r1 ? 1 : 2, cc = jj < c0 ? 0 : jj >= c1 ? 1 : 2;
    const uint32_t bits = mask[i];
    float o[8];
    ld8(tab + (rc * 3 + cc) * F + g * 8, o);
#pragma unroll
    for (int e = 0; e < 8; ++e) o[e] = (bits >> e) & 1u ? o[e] : 0.f;
    st8(dhn + (size_t)i * 8, o);
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

// Sums over the batch.  Blocks [0, KT * DT): gWf of 64 inputs from 64 (b % DT) on, and gbf where b % DT == 0.  SL 0: class b / DT, four
// interleaved chains over the samples combined as (0 + 1) + (2 + 3); SL 1: four classes from 4 (b / DT) on, one chain each.  Then FT
// blocks of 32 filters: gba from the per-sample sums of dh (fp64); the last block: the mean loss (fp64).
template <bool SL>
__global__ void __launch_bounds__(256) head_batch_kernel(const float* __restrict__ p, const float* __restrict__ dl,
                                                         const float* __restrict__ lossn, const float* __restrict__ bred, int N, int D,
                                                         int K, int KT, int DT, int FT, int F, float* __restrict__ gWf,
                                                         float* __restrict__ gbf, float* __restrict__ gba, float* __restrict__ loss_out,
                                                         int32_t* __restrict__ status, int n_scale) {
  nf_pdl_begin();
  __shared__ double sd[8][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, b = blockIdx.x;
  if (b < KT * DT) {
    float(*sf)[64] = reinterpret_cast<float(*)[64]>(sd);
    const int dx = threadIdx.x & 63, ch = threadIdx.x >> 6, d = (b % DT) * 64 + dx;
    const int k = SL ? (b / DT) * 4 + ch : b / DT;
    float s = 0.f, sb = 0.f;
    if (d < D && k < K) {
      // samples ch, ch + 4, ... below N4; chain 0 goes on with the last one to three.  SL: all samples
      const int N4 = SL ? 0 : N & ~3, cnt = N4 / 4, all = SL ? N : cnt + (ch == 0 ? N - N4 : 0);
#pragma unroll 1
      for (int j = 0; j < all; j += 16) {
        float u[16], v[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int q = min(j + e, all - 1), n = q < cnt ? ch + 4 * q : N4 + q - cnt;
          v[e] = p[(size_t)n * D + d];
          u[e] = dl[(size_t)n * K + k];
        }
#pragma unroll
        for (int e = 0; e < 16; ++e)
          if (j + e < all) {
            s = fmaf(u[e], v[e], s);
            sb += u[e];
          }
      }
    }
    if constexpr (SL) {
      if (d < D && k < K) gWf[(size_t)k * D + d] = s;
      if (b % DT == 0 && dx == 0 && k < K) gbf[k] = sb;
    } else {
      sf[ch][dx] = s;
      __syncthreads();
      if (ch == 0 && d < D) gWf[(size_t)k * D + d] = (sf[0][dx] + sf[1][dx]) + (sf[2][dx] + sf[3][dx]);
      if (b % DT == 0 && ty == 7) {
        float c = 0.f;
#pragma unroll 1
        for (int n0 = tx; n0 < N; n0 += 128) {
          float u[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) u[e] = dl[(size_t)min(n0 + 32 * e, N - 1) * K + k];
#pragma unroll
          for (int e = 0; e < 4; ++e) c += n0 + 32 * e < N ? u[e] : 0.f;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if (tx == 0) gbf[k] = c;
      }
    }
    return;
  }
  const bool loss = b == KT * DT + FT;
  const int f = (b - KT * DT) * 32 + tx;
  double s = 0.0;
  if (loss) {
    if (ty == 0) {
#pragma unroll 4
      for (int n = tx; n < N; n += 32) s += (double)lossn[n];
    }
  } else if (f < F) {
#pragma unroll 8
    for (int n = ty; n < N; n += 8) s += (double)bred[(size_t)n * F + f];
  }
  sd[ty][tx] = s;
  __syncthreads();
  if (loss && ty == 0) {
    double v = s;
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

// Summation order of the average pool, as the stand-alone pool kernels have it (nf_k_avgpool_fast, nf_k_avgpool)
struct PoolOrder {
  int slices, planes, even;
};
PoolOrder pool_order(int dtype, int N, int Ha, int Wa, int F) {
  const bool even = Ha % 2 == 0 && Wa % 2 == 0;
  if (dtype == NF_BF16 && even && (Ha / 2) * (Wa / 2) > 16) return {nf_k_avgpool_slices(N, Ha, Wa), 256 / (F / 8), 1};
  const int cnt = ((Ha + 1) / 2) * ((Wa + 1) / 2);
  if (dtype == NF_F32) return {std::max(1, std::min(kWarps, cnt / 16)), 16, 0};  // fp32 follows no other kernel's bits
  return {1, cnt <= 16 ? 1 : 256 / F, 0};
}
size_t h_smem(int dtype, int Ha, int Wa, int F) { return (size_t)Ha * Wa * F * nf_esize(dtype); }
size_t off_smem(int Ha, int Wa, int F) {  // offsets and sign bits
  return (size_t)((((Ha + 1) / 2) * ((Wa + 1) / 2) + 3) / 4 * 4) * 4 + (size_t)Ha * Wa * (F / 8);
}
size_t fixed_smem(int F, int K) {
  const int rd = std::max(kWarps * 4 * F, 1024);
  return ((size_t)4 * F + ((K + 3) & ~3) + rd + 9 * F) * 4;
}

template <typename T, int F8, bool STAGE, bool SL>
int launch_sample(const HeadArgs& a, size_t smem) {
  static bool done[64];  // function attributes belong to a device's context: set once per device
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!done[dev]) {
    NF_CUDA(cudaFuncSetAttribute(head_sample_kernel<T, F8, STAGE, SL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax + 1024));
    done[dev] = true;
  }
  nf_launch(head_sample_kernel<T, F8, STAGE, SL>, a.N, kHT, smem, a);
  NF_LAUNCHED();
  return NF_OK;
}
template <typename T, int F8>
int run_sample(const HeadArgs& a, size_t smem, bool stage) {
  if (a.S) return launch_sample<T, F8, false, true>(a, smem);
  return stage ? launch_sample<T, F8, true, false>(a, smem) : launch_sample<T, F8, false, false>(a, smem);
}

}  // namespace

// 0: not covered; 1: from pooled inputs (p, or the fused aux forward's partials); 2: from h, with dh, where the sample's h fits
// beside the tables.  Filters in 8, 16, 32, 64.
int nf_head_sample_mode(int dtype, int N, int Ha, int Wa, int F, int K) {
  if ((F != 8 && F != 16 && F != 32 && F != 64) || K > 16384 || Ha < 2 || Wa < 2) return 0;
  if (fixed_smem(F, K) > kSmemMax) return 0;
  const PoolOrder o = pool_order(dtype, N, Ha, Wa, F);
  int KS, S, parts;
  if (nf_head_slice_order(N, 4 * F, K, &KS, &S, &parts) &&
      (2 * (S + parts) > std::max(kWarps * 4 * F, 1024) || fixed_smem(F, K) + (size_t)S * 16 * F + off_smem(Ha, Wa, F) > kSmemMax))
    return 0;
  if (fixed_smem(F, K) + 16 * (4 * F + 4) * 4 > kSmemMax) return 0;
  const size_t need = fixed_smem(F, K) + std::max(h_smem(dtype, Ha, Wa, F), (size_t)16 * (4 * F + 4) * 4) + off_smem(Ha, Wa, F);
  return o.slices <= kWarps && need <= kSmemMax ? 2 : 1;
}

int nf_head_sample_step(const NfHeadIo& io, int dtype, int N, int Ha, int Wa, int F, int K, int loss_kind, int n_scale) {
  HeadArgs a{};
  a.h = io.h; a.part = io.part; a.th = Ha / 8; a.tw = Wa / 14;
  a.N = N; a.Ha = Ha; a.Wa = Wa; a.F = F; a.K = K;
  a.labels = io.labels; a.Wf = io.Wf; a.bf = io.bf;
  a.p = io.p; a.logits = io.logits; a.dlogits = io.dlogits; a.dp = io.dp; a.lossn = io.lossn; a.status = io.status;
  a.dh = io.dh; a.bred = io.bred; a.loss_kind = loss_kind; a.n_scale = n_scale;
  const PoolOrder o = pool_order(dtype, N, Ha, Wa, F);
  a.slices = o.slices; a.planes = o.planes; a.even = o.even;
  a.dh_even = dtype == NF_BF16 && Ha % 2 == 0 && Wa % 2 == 0;
  const int D = 4 * F;
  // fixed tables, then h or the weights, then (with h) offsets and sign bits
  const size_t tail = io.h ? off_smem(Ha, Wa, F) : 0;
  const size_t fixed = fixed_smem(F, K), row = (size_t)(D + 4) * 4;
  size_t smem = fixed + (io.h ? h_smem(dtype, Ha, Wa, F) : 0);
  const bool sliced = nf_head_slice_order(N, D, K, &a.KS, &a.S, &a.parts);
  if (!sliced) a.S = 0;
  a.chunk = (int)std::min<size_t>(K, (kSmemMax - fixed - tail) / row);
  const bool stage = a.chunk == K && !sliced;
  smem = std::max(smem, fixed + a.chunk * row);
  if (sliced) smem = std::max(smem, fixed + (size_t)a.S * D * 4);
  smem = (smem + 15) & ~(size_t)15;
  a.off = smem;
  smem += tail;
  a.groups = D <= 128 ? 256 / D : 1;
  int rc;
  if (dtype == NF_F32)
    rc = F == 8 ? run_sample<float, 1>(a, smem, stage) : F == 16 ? run_sample<float, 2>(a, smem, stage)
       : F == 32 ? run_sample<float, 4>(a, smem, stage) : run_sample<float, 8>(a, smem, stage);
  else
    rc = F == 8 ? run_sample<bf16, 1>(a, smem, stage) : F == 16 ? run_sample<bf16, 2>(a, smem, stage)
       : F == 32 ? run_sample<bf16, 4>(a, smem, stage) : run_sample<bf16, 8>(a, smem, stage);
  return rc;
}

int nf_head_sample_sums(const NfHeadIo& io, int N, int F, int K, int n_scale) {
  int KS, S, parts;
  const int D = 4 * F;
  const bool sliced = nf_head_slice_order(N, D, K, &KS, &S, &parts);
  const int DT = (D + 63) / 64, FT = io.dh ? (F + 31) / 32 : 0;
  const int KT = sliced ? (K + 3) / 4 : K;
  nf_launch(sliced ? head_batch_kernel<true> : head_batch_kernel<false>, (unsigned)(KT * DT + FT + 1), 256, 0, io.p, io.dlogits, io.lossn, io.bred, N, D,
            K, KT, DT, FT, F, io.gWf, io.gbf, io.gba, io.loss_out, io.status, n_scale);
  NF_LAUNCHED();
  return NF_OK;
}

// One block per class with a thread per input, as this once was, took twice as long (8000 samples of 1 x 1 maps, 8 filters, 10
// classes: the step 763 -> 262 us).
int nf_head_batch_sums(const float* p, const float* dlogits, const float* lossn, int N, int D, int K, float* gWf, float* gbf, float* loss_out,
                       int32_t* status, int n_scale) {
  const int DT = (D + 63) / 64;
  nf_launch(head_batch_kernel<false>, (unsigned)(K * DT + 1), 256, 0, p, dlogits, lossn, nullptr, N, D, K, K, DT, 0, 0, gWf, gbf, nullptr, loss_out,
            status, n_scale);
  NF_LAUNCHED();
  return NF_OK;
}
