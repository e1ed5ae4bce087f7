// Generic CUDA-core kernels of the local-layer step: any shape, fp32 or bf16 storage, fp32
// accumulation, deterministic reductions (fixed-order partials, no floating-point atomics).
// They carry the fp32 configuration and every shape the tensor-core kernels do not cover.
#include <algorithm>

#include "nf_internal.h"
#include "nf_ldst.cuh"

namespace {

// ------------------------------------------------------------------ direct convolution, 3x3 with pad 1 or 1x1
// y[n,i,j,co] = act(bias[co] + sum_{kh,kw,ci} w(tap,co,ci) * x[n, i*s+kh-pad, j*s+kw-pad, ci]).
// Weight element (tap,co,ci) sits at w[t*ws_tap + co*ws_co + ci*ws_ci] with t = tap, or 8-tap when
// flip is set (flip + swapped strides turn the same kernel into the input-gradient convolution).
//
// A block owns PX output pixels (of any images) x CO channels, a thread TP x TC of them; per step (chunk of CK input channels, tap)
// the operands go to shared memory transposed, the next step's loads fly meanwhile, one barrier per step.  Every output is ONE
// fp32 chain over chunk, tap, channel, whatever the tile, so the tile is chosen by size alone: 64 x 64 where that fills the
// chip, 32 x 32 below, 64 x 16 for few output channels.  (The earlier kernel gave each block 16 pixels of one row and 16 channels
// and each thread one output: 2 loads per multiply-add, 7 TFLOP/s; 16 -> 8 channels on 8 images of 32x32 20 us.)
struct ConvArgs {
  const void* x;
  const void* w;
  void* y;
  const float* bias;
  long ws_tap, ws_co, ws_ci;
  int H, W, Ci, Co, Ho, Wo, stride, taps, flip, relu;
  uint32_t P;     // output pixels of the launch
  uint32_t row0;  // the first one's row, where a launch takes some rows of one image (else 0)
};

template <int T> __device__ __forceinline__ void ld_tile(const float* p, float (&v)[T]) {
  if constexpr (T == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else if constexpr (T == 2) {
    const float2 q = *reinterpret_cast<const float2*>(p);
    v[0] = q.x; v[1] = q.y;
  } else {
    v[0] = *p;
  }
}

// WCO: 1 = eight consecutive output channels of the weights are contiguous, 0 = eight input channels.  VEC: rows of eight are
// whole and aligned; otherwise elements are fetched one by one.
template <typename T, int PX, int CO, int CK, int TP, int TC, int SPB, int WCO, int VEC>
__global__ void __launch_bounds__((PX / TP) * (CO / TC)) conv_direct_kernel(const ConvArgs a) {
  nf_pdl_begin();
  constexpr int kThr = (PX / TP) * (CO / TC), kXU = PX * CK / 8, kWU = CO * CK / 8;  // units of eight values per step
  constexpr int kXN = (kXU + kThr - 1) / kThr, kWN = (kWU + kThr - 1) / kThr;
  constexpr int kW0 = kThr >= kXU + kWU ? kXU : 0;  // first thread that fetches weights: others than fetch pixels where there are enough
  // column q of row c is kept at q ^ (8 * (c / 8)) (mod the row): the transposing stores then hit different banks
  constexpr int kXM = PX >= 32 ? 24 : 8, kWM = CO >= 32 ? 24 : 8;
  constexpr int kBuf = SPB == 9 ? 1 : 2;  // nine taps: one buffer, the next chunk waits in registers
  __shared__ __align__(16) float xs[kBuf][SPB][CK][PX];
  __shared__ __align__(16) float ws[kBuf][SPB][CK][CO];
  const T* __restrict__ x = reinterpret_cast<const T*>(a.x);
  const T* __restrict__ w = reinterpret_cast<const T*>(a.w);
  const int t = threadIdx.x, tc = t % (CO / TC), tp = t / (CO / TC);
  const uint32_t p0 = blockIdx.x * PX;
  const int co0 = (blockIdx.y + gridDim.y * blockIdx.z) * CO, pad = a.taps == 9 ? 1 : 0;

  int xi[kXN], xj[kXN];   // input row and column of the unit's pixel at tap (0, 0)
  size_t xb[kXN];         // its image's first element; pixels past the end: marked by a row far outside
#pragma unroll
  for (int u = 0; u < kXN; ++u) {
    const int e = t + u * kThr;
    const uint32_t p = p0 + e / (CK / 8);
    const uint32_t q = p / a.Wo, r = q + a.row0, n = r / a.Ho;
    xj[u] = (int)(p - q * a.Wo) * a.stride - pad;
    xi[u] = p < a.P && e < kXU ? (int)(r - n * a.Ho) * a.stride - pad : -1000000;
    xb[u] = (size_t)n * a.H * a.W * a.Ci;
  }
  float xr_[SPB][kXN][8], wr_[SPB][kWN][8];
  auto fetch = [&](int c0, int tap, float(&xr)[kXN][8], float(&wr)[kWN][8]) {
    const int kh = tap / 3, kw = tap - kh * 3;
#pragma unroll
    for (int u = 0; u < kXN; ++u) {
      const int e = t + u * kThr, ci = c0 + (e % (CK / 8)) * 8;
      const int ii = xi[u] + kh, jj = xj[u] + kw;
#pragma unroll
      for (int q = 0; q < 8; ++q) xr[u][q] = 0.f;
      if (ii >= 0 && ii < a.H && jj >= 0 && jj < a.W && ci < a.Ci) {
        const T* src = x + xb[u] + ((size_t)ii * a.W + jj) * a.Ci + ci;
        if constexpr (VEC) {
          ld8(src, xr[u]);
        } else {
          for (int q = 0; q < 8 && ci + q < a.Ci; ++q) xr[u][q] = ldf(src, q);
        }
      }
    }
    const size_t tb = (size_t)(a.flip ? 8 - tap : tap) * a.ws_tap;
#pragma unroll
    for (int u = 0; u < kWN; ++u) {
      const int e = t - kW0 + u * kThr;
      const int ci = c0 + (WCO ? e / (CO / 8) : (e % (CK / 8)) * 8), co = co0 + (WCO ? (e % (CO / 8)) * 8 : e / (CK / 8));
#pragma unroll
      for (int q = 0; q < 8; ++q) wr[u][q] = 0.f;
      if (e >= 0 && e < kWU && ci < a.Ci && co < a.Co) {
        const T* src = w + tb + (size_t)co * a.ws_co + (size_t)ci * a.ws_ci;
        if constexpr (VEC) {
          ld8(src, wr[u]);
        } else {
          for (int q = 0; q < 8 && (WCO ? co + q < a.Co : ci + q < a.Ci); ++q) wr[u][q] = ldf(src, (size_t)q * (WCO ? a.ws_co : a.ws_ci));
        }
      }
    }
  };
  auto put = [&](float(&xs)[CK][PX], float(&ws)[CK][CO], const float(&xr)[kXN][8], const float(&wr)[kWN][8]) {
#pragma unroll
    for (int u = 0; u < kXN; ++u) {
      const int e = t + u * kThr;
      if (e < kXU) {
        const int cc = e % (CK / 8), px = e / (CK / 8);
#pragma unroll
        for (int q = 0; q < 8; ++q) xs[cc * 8 + q][px ^ ((cc * 8) & kXM)] = xr[u][q];
      }
    }
#pragma unroll
    for (int u = 0; u < kWN; ++u) {
      const int e = t - kW0 + u * kThr;
      if (e >= 0 && e < kWU) {
        if constexpr (WCO) {
          const int c = e / (CO / 8), q0 = (e % (CO / 8)) * 8;
          float* dst = &ws[c][q0 ^ (c & ~7 & kWM)];
          *reinterpret_cast<float4*>(dst) = make_float4(wr[u][0], wr[u][1], wr[u][2], wr[u][3]);
          *reinterpret_cast<float4*>(dst + 4) = make_float4(wr[u][4], wr[u][5], wr[u][6], wr[u][7]);
        } else {
          const int cc = e % (CK / 8), co = e / (CK / 8);
#pragma unroll
          for (int q = 0; q < 8; ++q) ws[cc * 8 + q][co ^ ((cc * 8) & kWM)] = wr[u][q];
        }
      }
    }
  };

  float acc[TP][TC];
#pragma unroll
  for (int i = 0; i < TP; ++i)
#pragma unroll
    for (int j = 0; j < TC; ++j) acc[i][j] = 0.f;
  // steps (chunk, tap) go SPB at a time; `taps` is a multiple of SPB wherever SPB > 1
#pragma unroll
  for (int i = 0; i < SPB; ++i) fetch(0, i, xr_[i], wr_[i]);
#pragma unroll
  for (int i = 0; i < SPB; ++i) put(xs[0][i], ws[0][i], xr_[i], wr_[i]);
  __syncthreads();
  int c0 = 0, tap = 0, b = 0;
  while (true) {
    int nc = c0, nt = tap + SPB;
    if (nt == a.taps) {
      nt = 0;
      nc += CK;
    }
    const bool more = nc < a.Ci;
    if (more)
#pragma unroll
      for (int i = 0; i < SPB; ++i) fetch(nc, nt + i, xr_[i], wr_[i]);
    if constexpr (SPB == 9) {
      // eight channels of operands on their way at once: alone on its SM, a block of this small tile otherwise waits for shared memory
      // on every channel; the larger tiles hide that with other warps and are faster as the compiler orders them
#pragma unroll 1
      for (int st = 0; st < SPB; ++st)
#pragma unroll 1
        for (int c = 0; c < CK; c += 8) {
          float xv[8][TP], wv[8][TC];
          const int sx = (tp * TP) ^ (c & kXM), sw = (tc * TC) ^ (c & kWM);
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            ld_tile<TP>(&xs[b][st][c + u][sx], xv[u]);
            ld_tile<TC>(&ws[b][st][c + u][sw], wv[u]);
          }
#pragma unroll
          for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int i = 0; i < TP; ++i)
#pragma unroll
              for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(xv[u][i], wv[u][j], acc[i][j]);
        }
    } else {
#pragma unroll 1
      for (int st = 0; st < SPB; ++st)
#pragma unroll 8
        for (int c = 0; c < CK; ++c) {
          float xv[TP], wv[TC];
          const float* xp = &xs[b][st][c][(tp * TP) ^ (c & ~7 & kXM)];
          const float* wp = &ws[b][st][c][(tc * TC) ^ (c & ~7 & kWM)];
          ld_tile<TP>(xp, xv);
          ld_tile<TC>(wp, wv);
#pragma unroll
          for (int i = 0; i < TP; ++i)
#pragma unroll
            for (int j = 0; j < TC; ++j) acc[i][j] = fmaf(xv[i], wv[j], acc[i][j]);
        }
    }
    if (!more) break;
    if constexpr (kBuf == 1) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < SPB; ++i) put(xs[0][i], ws[0][i], xr_[i], wr_[i]);
      __syncthreads();
    } else {
#pragma unroll
      for (int i = 0; i < SPB; ++i) put(xs[b ^ 1][i], ws[b ^ 1][i], xr_[i], wr_[i]);
      __syncthreads();
      b ^= 1;
    }
    c0 = nc;
    tap = nt;
  }
  T* y = reinterpret_cast<T*>(a.y);
#pragma unroll
  for (int i = 0; i < TP; ++i) {
    const uint32_t p = p0 + tp * TP + i;
    if (p >= a.P) break;
#pragma unroll
    for (int j = 0; j < TC; ++j) {
      const int co = co0 + tc * TC + j;
      if (co < a.Co) {
        float v = acc[i][j];
        if (a.bias) v += a.bias[co];
        if (a.relu) v = fmaxf(v, 0.f);
        stf(y, (size_t)p * a.Co + co, v);
      }
    }
  }
}

template <typename T, int PX, int CO, int CK, int TP, int TC, int SPB>
int launch_direct(const ConvArgs& a) {
  const unsigned cols = (unsigned)((a.Co + CO - 1) / CO), y = cols < 65535 ? cols : 65535;
  const dim3 grid((unsigned)((a.P + PX - 1) / PX), y, (cols + y - 1) / y);  // channel tiles beyond Co do nothing
  const int thr = (PX / TP) * (CO / TC);
  const bool wco = a.ws_co == 1 && a.ws_ci != 1;
  const bool vec = a.Ci % 8 == 0 && (((uintptr_t)a.x | (uintptr_t)a.w) & 15) == 0 && (wco ? a.Co % 8 == 0 && a.ws_ci % 8 == 0 : a.ws_ci == 1 && a.ws_co % 8 == 0) &&
                   a.ws_tap % 8 == 0;
  if (wco)
    vec ? nf_launch(conv_direct_kernel<T, PX, CO, CK, TP, TC, SPB, 1, 1>, grid, thr, 0, a)
        : nf_launch(conv_direct_kernel<T, PX, CO, CK, TP, TC, SPB, 1, 0>, grid, thr, 0, a);
  else
    vec ? nf_launch(conv_direct_kernel<T, PX, CO, CK, TP, TC, SPB, 0, 1>, grid, thr, 0, a)
        : nf_launch(conv_direct_kernel<T, PX, CO, CK, TP, TC, SPB, 0, 0>, grid, thr, 0, a);
  NF_LAUNCHED();
  return NF_OK;
}

template <typename T>
int run_direct(const ConvArgs& a) {
  // Few output channels: 64 x 16 tiles; with at most 16 input channels (chunks of 16: the same chain, half the shared memory work)
  // a step is so short that the trip to L2 shows, so three taps share one (16 -> 8 channels on 8 images of 32x32: 10.7 -> 6 us)
  if (a.Co <= 16 && a.Ci <= 16)
    return a.taps == 9 ? launch_direct<T, 64, 16, 16, 2, 2, 3>(a) : launch_direct<T, 64, 16, 16, 2, 2, 1>(a);
  // 64 x 64 tiles from one block per SM on (148): below that, four times as many blocks of 32 x 32 finish sooner.  Where even those
  // (or blocks of 64 x 16) leave SMs idle, 16 x 16 with all nine taps per step, a chain of a ninth as many trips to L2: evaluation of one
  // image, 512 channels at 7x7 382 -> 225 us, 256 at 14x14 213 -> 139 (229 and 152 with a block per 16 pixels of a row, one output
  // per thread, as all sizes once had)
  const long big = (long)((a.P + 63) / 64) * ((a.Co + 63) / 64), mid = a.Co <= 16 ? (a.P + 63) / 64 : (long)((a.P + 31) / 32) * ((a.Co + 31) / 32);
  if (mid < 148) return a.taps == 9 ? launch_direct<T, 16, 16, 32, 2, 1, 9>(a) : launch_direct<T, 16, 16, 32, 2, 1, 1>(a);
  if (a.Co <= 16) return launch_direct<T, 64, 16, 32, 2, 2, 1>(a);
  if (big >= 148) return launch_direct<T, 64, 64, 32, 4, 4, 1>(a);
  return launch_direct<T, 32, 32, 32, 2, 2, 1>(a);
}

// ------------------------------------------------------------------ direct weight gradient
// part[split][tap][co][ci] = sum over the split's (n,i) rows and all j of g[n,i,j,co] * x[n,i*s+kh-1,j*s+kw-1,ci]
constexpr int WG_J = 64;

template <typename T>
__global__ void __launch_bounds__(256) wgrad_direct_kernel(const T* __restrict__ x, int N, int H, int W, int Ci,
                                                           const T* __restrict__ g, int Co, int s, int Ho, int Wo,
                                                           int splits, float* __restrict__ part) {
  nf_pdl_begin();
  __shared__ float gs[WG_J][16];
  __shared__ float xs[3][WG_J * 2 + 2][16];
  const int cit = (Ci + 15) / 16, cot = (Co + 15) / 16;
  int b = blockIdx.x;
  const int ti = b % cit; b /= cit;
  const int to = b % cot; b /= cot;
  const int sp = b;
  const int tid = threadIdx.x, ci_l = tid % 16, co_l = tid / 16;
  const int ci0 = ti * 16, co0 = to * 16;
  const long rows = (long)N * Ho;
  const long r0 = rows * sp / splits, r1 = rows * (sp + 1) / splits;
  float acc[9];
#pragma unroll
  for (int t = 0; t < 9; ++t) acc[t] = 0.f;
  for (long r = r0; r < r1; ++r) {
    const int n = (int)(r / Ho), i = (int)(r % Ho);
    for (int j0 = 0; j0 < Wo; j0 += WG_J) {
      const int jn = min(WG_J, Wo - j0);
      const int cols = (jn - 1) * s + 3;
      for (int e = tid; e < jn * 16; e += 256) {
        const int c = e % 16, j = e / 16;
        gs[j][c] = (co0 + c < Co) ? ldf(g, (((size_t)n * Ho + i) * Wo + j0 + j) * Co + co0 + c) : 0.f;
      }
      for (int e = tid; e < 3 * cols * 16; e += 256) {
        const int c = e % 16, col = (e / 16) % cols, rr = e / (16 * cols);
        const int ii = i * s + rr - 1, jj = j0 * s + col - 1;
        float v = 0.f;
        if (ci0 + c < Ci && ii >= 0 && ii < H && jj >= 0 && jj < W)
          v = ldf(x, (((size_t)n * H + ii) * W + jj) * Ci + ci0 + c);
        xs[rr][col][c] = v;
      }
      __syncthreads();
      for (int j = 0; j < jn; ++j) {
        const float gv = gs[j][co_l];
#pragma unroll
        for (int kh = 0; kh < 3; ++kh)
#pragma unroll
          for (int kw = 0; kw < 3; ++kw) acc[kh * 3 + kw] = fmaf(gv, xs[kh][j * s + kw][ci_l], acc[kh * 3 + kw]);
      }
      __syncthreads();
    }
  }
  if (co0 + co_l < Co && ci0 + ci_l < Ci)
#pragma unroll
    for (int t = 0; t < 9; ++t) part[(((size_t)sp * 9 + t) * Co + co0 + co_l) * Ci + ci0 + ci_l] = acc[t];
}

// ------------------------------------------------------------------ first-layer kernels (Cin <= 4)
// An RGB input gives a K dimension of only 27: too thin for the tensor cores and, with 6-byte pixels,
// not addressable by TMA.  One thread computes 16 output channels of one pixel from its 3x3xCin patch held
// in registers; weights sit in shared memory and are read as warp-wide broadcasts.
template <typename T> __device__ __forceinline__ void store16(T* dst, const float (&v)[16]);
template <> __device__ __forceinline__ void store16<float>(float* dst, const float (&v)[16]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) reinterpret_cast<float4*>(dst)[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
}
template <> __device__ __forceinline__ void store16<bf16>(bf16* dst, const float (&v)[16]) {
  uint32_t w[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const __nv_bfloat162 b2 = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
    w[k] = *reinterpret_cast<const uint32_t*>(&b2);
  }
  reinterpret_cast<uint4*>(dst)[0] = make_uint4(w[0], w[1], w[2], w[3]);
  reinterpret_cast<uint4*>(dst)[1] = make_uint4(w[4], w[5], w[6], w[7]);
}

template <typename T>
__global__ void __launch_bounds__(256) conv_smallc_kernel(const T* __restrict__ x, int N, int H, int W, int Ci,
                                                          const T* __restrict__ w, int s, int Co, int Ho, int Wo,
                                                          T* __restrict__ y) {
  nf_pdl_begin();
  extern __shared__ float wsm[];  // [tap][ci][co]
  for (int e = threadIdx.y * 32 + threadIdx.x; e < 9 * Ci * Co; e += blockDim.x * blockDim.y) {
    const int co = e % Co, ci = (e / Co) % Ci, t = e / (Co * Ci);
    wsm[e] = ldf(w, ((size_t)t * Co + co) * Ci + ci);
  }
  __syncthreads();
  const size_t P = (size_t)N * Ho * Wo;
  const int co0 = threadIdx.y * 16;
  for (size_t pix = (size_t)blockIdx.x * 32 + threadIdx.x; pix < P; pix += (size_t)gridDim.x * 32) {  // weights loaded once per block
    const int j = (int)(pix % Wo), i = (int)((pix / Wo) % Ho);
    const size_t n = pix / ((size_t)Wo * Ho);
    float patch[36];
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      const int ii = i * s + t / 3 - 1, jj = j * s + t % 3 - 1;
      const bool in = ii >= 0 && ii < H && jj >= 0 && jj < W;
#pragma unroll
      for (int c = 0; c < 4; ++c) patch[t * 4 + c] = (in && c < Ci) ? ldf(x, ((n * H + ii) * W + jj) * Ci + c) : 0.f;
    }
    float acc[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) acc[k] = 0.f;
#pragma unroll
    for (int t = 0; t < 9; ++t)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (c < Ci) {
          const float xv = patch[t * 4 + c];
          const float4* wr = reinterpret_cast<const float4*>(wsm + (t * Ci + c) * Co + co0);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float4 wv = wr[k];
            acc[4 * k] = fmaf(xv, wv.x, acc[4 * k]);
            acc[4 * k + 1] = fmaf(xv, wv.y, acc[4 * k + 1]);
            acc[4 * k + 2] = fmaf(xv, wv.z, acc[4 * k + 2]);
            acc[4 * k + 3] = fmaf(xv, wv.w, acc[4 * k + 3]);
          }
        }
    store16(y + pix * Co + co0, acc);
  }
}

// part[split][tap][co][ci]: thread (co, lane) sums its 9*Ci products over the pixels lane, lane+4, ... of the
// split's rows; the 3 input rows of an output row are staged in shared memory and read as broadcasts.
template <typename T>
__global__ void __launch_bounds__(512) wgrad_smallc_kernel(const T* __restrict__ x, int N, int H, int W, int Ci,
                                                           const T* __restrict__ g, int Co, int s, int Ho, int Wo,
                                                           int splits, float* __restrict__ part) {
  nf_pdl_begin();
  extern __shared__ float sm[];           // xrow[(R-1)*s + 3][W + 2][4]  then  red[4][Co][36]
  constexpr int R = 4;                    // output rows staged per synchronisation
  const int xr = (R - 1) * s + 3;
  float* xrow = sm;
  float* red = sm + xr * (W + 2) * 4;
  const int co = threadIdx.x, ln = threadIdx.y, tid = ln * blockDim.x + co, nthr = blockDim.x * 4;
  const long rows = (long)N * Ho;
  const long r0 = rows * blockIdx.x / splits, r1 = rows * (blockIdx.x + 1) / splits;
  float acc[36];
#pragma unroll
  for (int k = 0; k < 36; ++k) acc[k] = 0.f;
  for (long r = r0; r < r1;) {
    const int n = (int)(r / Ho), i = (int)(r % Ho);
    int nr = R;
    if (nr > r1 - r) nr = (int)(r1 - r);
    if (nr > Ho - i) nr = Ho - i;          // stay inside one image
    const int need = (nr - 1) * s + 3;
    __syncthreads();
    for (int e = tid; e < need * (W + 2) * 4; e += nthr) {
      const int c = e & 3, col = (e >> 2) % (W + 2), rr = (e >> 2) / (W + 2);
      const int ii = i * s + rr - 1, jj = col - 1;
      xrow[e] = (c < Ci && ii >= 0 && ii < H && jj >= 0 && jj < W) ? ldf(x, (((size_t)n * H + ii) * W + jj) * Ci + c) : 0.f;
    }
    __syncthreads();
    for (int q = 0; q < nr; ++q)
      for (int j = ln; j < Wo; j += 4) {
        const float gv = ldf(g, (((size_t)n * Ho + i + q) * Wo + j) * Co + co);
#pragma unroll
        for (int t = 0; t < 9; ++t) {
          const float4 xv = *reinterpret_cast<const float4*>(xrow + ((q * s + t / 3) * (W + 2) + j * s + t % 3) * 4);
          acc[t * 4 + 0] = fmaf(gv, xv.x, acc[t * 4 + 0]);
          acc[t * 4 + 1] = fmaf(gv, xv.y, acc[t * 4 + 1]);
          acc[t * 4 + 2] = fmaf(gv, xv.z, acc[t * 4 + 2]);
          acc[t * 4 + 3] = fmaf(gv, xv.w, acc[t * 4 + 3]);
        }
      }
    r += nr;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 36; ++k) red[(ln * Co + co) * 36 + k] = acc[k];
  __syncthreads();
  if (ln == 0)
    for (int t = 0; t < 9; ++t)
      for (int c = 0; c < Ci; ++c) {
        float v = 0.f;
        for (int q = 0; q < 4; ++q) v += red[(q * Co + co) * 36 + t * 4 + c];
        part[(((size_t)blockIdx.x * 9 + t) * Co + co) * Ci + c] = v;
      }
}

inline bool smallc_ok(int Ci, int Co, int W) { return Ci <= 4 && Co % 16 == 0 && Co <= 128 && W <= 512; }

}  // namespace

int nf_k_conv(int dtype, const void* x, int N, int H, int W, int Ci, const void* w, long ws_tap, long ws_co,
                long ws_ci, int flip, const float* bias, int relu, int stride, int Co, void* y) {
  const int Ho = (H - 1) / stride + 1, Wo = (W - 1) / stride + 1;
  if (smallc_ok(Ci, Co, W) && !flip && !bias && !relu && ws_ci == 1 && ws_co == Ci && ws_tap == (long)Co * Ci) {
    const size_t P = (size_t)N * Ho * Wo;
    const dim3 blk(32, Co / 16);
    const size_t sm = (size_t)9 * Ci * Co * sizeof(float);
    size_t nblk_ = (P + 31) / 32;
    if (nblk_ > 148 * 16) nblk_ = 148 * 16;
    const unsigned grid = (unsigned)nblk_;
    if (dtype == NF_F32)
      nf_launch(conv_smallc_kernel<float>, grid, blk, sm, (const float*)x, N, H, W, Ci, (const float*)w,
                                                                                   stride, Co, Ho, Wo, (float*)y);
    else
      nf_launch(conv_smallc_kernel<bf16>, grid, blk, sm, (const bf16*)x, N, H, W, Ci, (const bf16*)w,
                                                                                  stride, Co, Ho, Wo, (bf16*)y);
    NF_LAUNCHED();
    return NF_OK;
  }
  if ((long)N * Ho * ((Wo + 15) / 16) * ((Co + 15) / 16) > 0x7fffffffL) return NF_EUNSUPPORTED;
  return nf_k_conv_taps(dtype, x, N, H, W, Ci, w, 9, ws_tap, ws_co, ws_ci, flip, bias, relu, stride, Co, y);
}

int nf_k_conv_taps(int dtype, const void* x, int N, int H, int W, int Ci, const void* w, int taps, long ws_tap, long ws_co, long ws_ci,
                   int flip, const float* bias, int relu, int stride, int Co, void* y) {
  const int Ho = (H - 1) / stride + 1, Wo = (W - 1) / stride + 1;
  // A launch numbers its pixels in 32 bits: as many images as that holds, or rows of one image where that is more.
  constexpr long kMaxPixels = 0x7fffffffL;
  const long map = (long)Ho * Wo, imgs = std::max(1L, kMaxPixels / map), rows = map > kMaxPixels ? kMaxPixels / Wo : Ho;
  const size_t es = nf_esize(dtype);
  for (long n0 = 0; n0 < N; n0 += imgs)
    for (long r0 = 0; r0 < Ho; r0 += rows) {
      const long P = std::min(imgs, N - n0) * std::min(rows, Ho - r0) * Wo;
      const ConvArgs a{(const char*)x + (size_t)n0 * H * W * Ci * es, w, (char*)y + (size_t)(n0 * map + r0 * Wo) * Co * es, bias, ws_tap, ws_co, ws_ci,
                       H, W, Ci, Co, Ho, Wo, stride, taps, flip, relu, (uint32_t)P, (uint32_t)r0};
      const int rc = dtype == NF_F32 ? run_direct<float>(a) : run_direct<bf16>(a);
      if (rc != NF_OK) return rc;
    }
  return NF_OK;
}

int nf_k_wgrad_splits(int N, int Ho, int Ci, int Co) {
  if (Ci <= 4 && Co % 16 == 0 && Co <= 128) {  // first-layer kernel: one block per slice of rows
    long sp = (long)N * Ho;
    return (int)(sp > 1184 ? 1184 : sp);
  }
  const long tiles = (long)((Ci + 15) / 16) * ((Co + 15) / 16);
  long s = 2368 / tiles;
  if (s < 1) s = 1;
  if (s > (long)N * Ho) s = (long)N * Ho;
  return (int)s;
}

int nf_k_wgrad(int dtype, const void* x, int N, int H, int W, int Ci, const void* g, int Co, int stride,
                 float* part, size_t part_floats, float* dw) {
  const int Ho = (H - 1) / stride + 1, Wo = (W - 1) / stride + 1;
  const int splits = nf_k_wgrad_splits(N, Ho, Ci, Co);
  const size_t n = (size_t)9 * Co * Ci;
  if ((size_t)splits * n > part_floats) return NF_ENOWS;
  if (smallc_ok(Ci, Co, W)) {
    const dim3 blk(Co, 4);
    const size_t sm = ((size_t)(3 * stride + 3) * (W + 2) * 4 + (size_t)4 * Co * 36) * sizeof(float);
    static bool attr_done = false;
    if (!attr_done) {
      NF_CUDA(cudaFuncSetAttribute(wgrad_smallc_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024));
      NF_CUDA(cudaFuncSetAttribute(wgrad_smallc_kernel<bf16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024));
      attr_done = true;
    }
    if (dtype == NF_F32)
      nf_launch(wgrad_smallc_kernel<float>, splits, blk, sm, (const float*)x, N, H, W, Ci, (const float*)g, Co, stride, Ho, Wo,
                                                                 splits, part);
    else
      nf_launch(wgrad_smallc_kernel<bf16>, splits, blk, sm, (const bf16*)x, N, H, W, Ci, (const bf16*)g, Co, stride, Ho, Wo,
                                                                splits, part);
    NF_LAUNCHED();
    return nf_k_sum_parts(part, splits, n, dw);
  }
  const unsigned blocks = (unsigned)(((Ci + 15) / 16) * ((Co + 15) / 16) * splits);
  if (dtype == NF_F32)
    nf_launch(wgrad_direct_kernel<float>, blocks, 256, 0, (const float*)x, N, H, W, Ci, (const float*)g, Co,
                                                                stride, Ho, Wo, splits, part);
  else
    nf_launch(wgrad_direct_kernel<bf16>, blocks, 256, 0, (const bf16*)x, N, H, W, Ci, (const bf16*)g, Co,
                                                               stride, Ho, Wo, splits, part);
  NF_LAUNCHED();
  return nf_k_sum_parts(part, splits, n, dw);
}
