// Evaluation of a first layer (3 -> 64 channels, 3x3, stride 1): convolution, BatchNorm with running statistics and ReLU in one kernel
// that reads the images as they are.
//
// A contraction over 27 products is nothing for the tensor cores; what the layer costs is the memory traffic of its output and the
// instructions around it.  On the folded kernel it cost a copy of the images with 32-byte pixels and an epilogue that handled every output
// three times (shift-add of the column taps).  Here the operand [128 pixels][27 products] is gathered by ordinary loads straight into the
// swizzled layout the tensor core reads: 9 values of an image row are 18 consecutive bytes, five 32-bit words and at most one shift by half
// a word.  K = 32: the three kernel rows take ten places each, the tenth and the last two are zero.  Two instructions per tile, the epilogue
// reads each output once.  A block needs 62 KB and 128 tensor-memory columns, so three share an SM and hide each other's latencies; no
// deeper pipeline inside one was needed.
#include <cuda.h>

#include <algorithm>

#include "nf_ptx.cuh"
#include "nf_tc.h"
#include "nf_tiles.cuh"

namespace {

constexpr int kThreads = 288;  // warps 0-3 gather, 4-7 epilogue, 8 issues
constexpr int kStages = 3;
constexpr int kBlocksPerSm = 3;
constexpr int kA = 128 * 64, kW = 64 * 64, kOut = 128 * 128;
constexpr int kSmem = 1024 + kStages * kA + kW + 2 * kOut + 64 * 8 + 256;

struct FirstParams {
  const bf16* x;  // [N][H][W][3]
  const bf16* w;  // [9][64][3]
  const float *scale, *shift;
  int32_t* status;
  int H, W, bw_log, bh, total;
  TileGrid tg;
};

// Words 0..4 of v: the nine values of pixels (h, w - 1 .. w + 1), zero outside the image, and a zero.  W is even, so a row starts on a
// word; the first value of an even w lies in the upper half of its word.
__device__ __forceinline__ void gather_row(const uint32_t* __restrict__ x, size_t row, int W, int w, bool in, uint32_t* v) {
  const uint32_t* p = x + (row * W + w) * 3 / 2 - ((w & 1) ? 1 : 2);  // 3 (w - 1) / 2 rounded down, in words of the row
  uint32_t q[6];
#pragma unroll
  for (int i = 0; i < 5; ++i) q[i] = in && (i >= 2 || w > 0) && (i < 3 || w < W - 1) ? __ldg(p + i) : 0u;
  q[5] = 0u;
  const uint32_t sh = (w & 1) ? 0u : 16u;
#pragma unroll
  for (int i = 0; i < 5; ++i) v[i] = __funnelshift_r(q[i], q[i + 1], sh);
  v[4] &= 0xffffu;
}

__device__ __forceinline__ uint32_t bn_relu2(uint32_t y, float4 c) {  // c: scale and shift of two channels
  const __nv_bfloat162 b = __floats2bfloat162_rn(fmaxf(fmaf(__uint_as_float(y << 16), c.x, c.z), 0.f),
                                                 fmaxf(fmaf(__uint_as_float(y & 0xffff0000u), c.y, c.w), 0.f));
  return *reinterpret_cast<const uint32_t*>(&b);
}

__global__ void __launch_bounds__(kThreads, kBlocksPerSm) first_eval_kernel(const __grid_constant__ CUtensorMap tm_out, const FirstParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* wsm = smem + kStages * kA;
  uint8_t* stg = wsm + kW;
  float4* coef = reinterpret_cast<float4*>(stg + 2 * kOut);  // [32]: scale, scale, shift, shift of two channels
  uint64_t* full = reinterpret_cast<uint64_t*>(coef + 32);
  uint64_t* empty = full + kStages;
  uint64_t* tfull = empty + kStages;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* epi_go = reinterpret_cast<volatile int*>(tmem_slot + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(&full[s], 128);
      ptx::mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&tfull[a], 1);
      ptx::mbar_init(&tempty[a], 128);
    }
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(&tm_out);
  }
  if (warp == 8) {
    ptx::tmem_alloc(tmem_slot, 128);
    ptx::tmem_relinquish();
  }
  // The block has its columns before it lets the next kernel's blocks in: those allocate theirs and hold them while they wait for this grid,
  // and the wait for columns knows no limit.
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  nf_pdl_begin();
  for (int i = threadIdx.x; i < 256; i += kThreads) {  // weights: row co, places 8c .. 8c+7
    const int co = i >> 2, c = i & 3;
    uint32_t v[4];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int k = c * 8 + e, kh = k / 10, j = k % 10;
      const uint32_t b = kh < 3 && j < 9 ? __bfloat16_as_ushort(p.w[((kh * 3 + j / 3) * 64 + co) * 3 + j % 3]) : 0u;
      v[e >> 1] = e & 1 ? v[e >> 1] | b << 16 : b;
    }
    *reinterpret_cast<uint4*>(wsm + co * 64 + ((c ^ ((co >> 1) & 3)) * 16)) = make_uint4(v[0], v[1], v[2], v[3]);
  }
  if (threadIdx.x < 32) {
    const int c = threadIdx.x * 2;
    coef[threadIdx.x] = make_float4(p.scale[c], p.scale[c + 1], p.shift[c], p.shift[c + 1]);
  }
  ptx::fence_async_smem();
  __syncthreads();
  const uint32_t tmem_base = *tmem_slot;

  if (warp < 4) {
    const int r = threadIdx.x, dw = r & ((1 << p.bw_log) - 1), dh = r >> p.bw_log;
    uint32_t s = 0, ph = 0;
    for (int t = blockIdx.x; t < p.total; t += gridDim.x) {
      const TileAt at = tile_at(t, p.tg);
      const int w = (at.w << p.bw_log) + dw, h = at.h * p.bh + dh;
      uint32_t v[16];
#pragma unroll
      for (int kh = 0; kh < 3; ++kh) {
        const int hh = h + kh - 1;
        gather_row(reinterpret_cast<const uint32_t*>(p.x), (size_t)at.n * p.H + hh, p.W, w, hh >= 0 && hh < p.H, v + kh * 5);
      }
      v[15] = 0u;
      if (!ptx::mbar_wait(&empty[s], ph ^ 1, abort_flag)) break;
      uint8_t* row = smem + s * kA + r * 64;
#pragma unroll
      for (int c = 0; c < 4; ++c) *reinterpret_cast<uint4*>(row + ((c ^ ((r >> 1) & 3)) * 16)) = make_uint4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
      ptx::fence_async_smem();
      ptx::mbar_arrive(&full[s]);
      if (++s == kStages) {
        s = 0;
        ph ^= 1;
      }
    }
  } else if (warp == 8) {
    if (ptx::elect_one()) {
      constexpr uint32_t idesc = ptx::idesc_bf16(128, 64, 0, 0);
      const uint64_t hi = ptx::sdesc(0, 16, 512, 4);
      const uint32_t a16 = ptx::smem_u32(smem) >> 4, b16 = ptx::smem_u32(wsm) >> 4;
      uint32_t s = 0, ph = 0, tl = 0;
      for (int t = blockIdx.x; t < p.total; t += gridDim.x, ++tl) {
        const uint32_t acc = tl & 1;
        if (!ptx::mbar_wait(&tempty[acc], ((tl >> 1) & 1) ^ 1, abort_flag)) break;
        if (!ptx::mbar_wait(&full[s], ph, abort_flag)) break;
        ptx::tc_fence_after();
#pragma unroll
        for (int k = 0; k < 2; ++k)
          ptx::mma_f16(tmem_base + acc * 64, hi | (uint64_t)(a16 + s * (kA >> 4) + k * 2), hi | (uint64_t)(b16 + k * 2), idesc, k);
        ptx::mma_commit(&empty[s]);
        ptx::mma_commit(&tfull[acc]);
        if (++s == kStages) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    __syncwarp();
  } else {
    // Accumulators are read as matrix fragments: a thread holds 16 channels of every eighth pixel, so that its coefficients stay in
    // registers, and matrix stores write a pixel's 8 channels as 16 bytes.  With a thread per pixel the coefficients came from shared
    // memory, 32 loads of 16 bytes per tile, and kept the load-store unit busy 82 % of the time.
    const int et = threadIdx.x - 128, lg = warp & 3;
    const int mrow = (lane & 7) + (lane >> 3 & 1) * 8, mchunk = lane >> 4;  // the row and 8-channel chunk this thread addresses
    float4 cf[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) cf[i] = coef[i * 4 + (lane & 3)];  // channels 8 i + 2 (lane % 4) and the next
    uint32_t tl = 0;
    for (int t = blockIdx.x; t < p.total; t += gridDim.x, ++tl) {
      const TileAt at = tile_at(t, p.tg);
      const uint32_t acc = tl & 1;
      ptx::mbar_wait(&tfull[acc], (tl >> 1) & 1, abort_flag);  // sets the abort flag itself when it gives up
      ptx::tc_fence_after();
      if (et == 0) {
        ptx::tma_store_wait_read_but_one();  // the store before the last one has read the staging tile that comes next
        *epi_go = *abort_flag ? 0 : 1;       // one thread decides for all 128
      }
      ptx::named_barrier(1, 128);
      if (!*epi_go) break;
      uint8_t* const out = stg + acc * kOut;
      const uint32_t tbase = tmem_base + acc * 64, obase = ptx::smem_u32(out);
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {  // 16 pixels of the warp's 32
        const uint32_t px = (uint32_t)(lg * 32 + hf * 16 + mrow);
        uint32_t v[4][8];
#pragma unroll
        for (int j = 0; j < 4; ++j) ptx::tmem_ld_16x256b_x2(tbase + ((uint32_t)(lg * 32 + hf * 16) << 16) + j * 16, v[j]);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uint32_t o[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {  // rounded for storage, as where y is stored, then normalised
            const __nv_bfloat162 y = __floats2bfloat162_rn(__uint_as_float(v[j][2 * q]), __uint_as_float(v[j][2 * q + 1]));
            o[q] = bn_relu2(*reinterpret_cast<const uint32_t*>(&y), cf[2 * j + q / 2]);
          }
          ptx::stmatrix_x4(obase + px * 128 + (((2 * j + mchunk) ^ (px & 7)) * 16), o[0], o[1], o[2], o[3]);
        }
      }
      ptx::tc_fence_before();
      ptx::mbar_arrive(&tempty[acc]);
      ptx::fence_async_smem();
      ptx::named_barrier(1, 128);
      if (et == 0) {
        ptx::tma_store_4d(&tm_out, out, 0, (int)at.w << p.bw_log, (int)at.h * p.bh, (int)at.n);
        ptx::tma_store_commit();
      }
    }
    if (et == 0) ptx::tma_store_wait_all();
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(p.status, NF_ETIMEOUT);
    const unsigned long long t0 = ptx::globaltimer();
    while (ptx::globaltimer() - t0 < 2000000ull) __nanosleep(1000);
  }
  if (warp == 8) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, 128);
  }
}

}  // namespace

// RGB images on maps that the folded kernel would otherwise take (cin_pad 16) and 128-pixel tiles divide, with an even width.  Not where
// the output overlaps the images: a block would overwrite pixels that others still gather; there the padded copy stays in use.
bool nf_first_eval_ok(const nf_layer* L, const void* x, int count, const void* act) {
  int BW, BH;
  if (L->cin_pad != 16 || L->Cin != 3 || L->Cout != 64 || L->o.stride != 1 || L->W % 2 || !nf_tc_tile(L->H, L->W, &BW, &BH)) return false;
  const char *in0 = (const char*)x, *in1 = in0 + (size_t)count * L->H * L->W * 3 * 2;
  const char *out0 = (const char*)act, *out1 = out0 + (size_t)count * L->H * L->W * 64 * 2;
  return (in1 <= out0 || out1 <= in0) && (long long)count * (L->H / BH) * (L->W / BW) < (1ll << 30);
}

int nf_first_eval(nf_layer* L, const void* x, int count, void* act) {
  static bool done[64];  // function attributes belong to a device's context: set once per device
  int dev = 0, BW, BH;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!done[dev]) {
    NF_CUDA(cudaFuncSetAttribute(first_eval_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
    done[dev] = true;
  }
  nf_tc_tile(L->H, L->W, &BW, &BH);
  CUtensorMap tm;
  const int rc = nf_tc_out_map(&tm, act, count, L->H, L->W, 64, BW, BH);
  if (rc != NF_OK) return rc;
  FirstParams p{};
  p.x = (const bf16*)x;
  p.w = L->shadow + L->off[NF_P_W];
  p.scale = L->scale; p.shift = L->shift; p.status = L->status;
  p.H = L->H; p.W = L->W; p.bh = BH;
  while ((1 << p.bw_log) < BW) ++p.bw_log;
  p.tg = tile_grid(1, L->W / BW, L->H / BH);
  p.total = count * (L->H / BH) * (L->W / BW);
  nf_launch(first_eval_kernel, std::min(p.total, kBlocksPerSm * nf_tc_sm_count()), kThreads, kSmem, tm, p);
  NF_LAUNCHED();
  return NF_OK;
}
