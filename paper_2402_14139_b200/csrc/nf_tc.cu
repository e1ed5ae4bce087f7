// Tensor-core convolution kernels for sm_100a: implicit GEMM on tcgen05.mma with accumulators in
// tensor memory, operands staged in shared memory by TMA, warp-specialised persistent CTAs.
//
// Forward (Eq. 1's theta_n x_n, stride 1, Cin and Cout multiples of 64):
//   GEMM view  D[pixel, co] = sum_{tap, ci} X[pixel shifted by tap, ci] * W[tap][co][ci]
//   M tile = 128 output pixels = a BW x BH patch of one image, N tile = BN output channels,
//   K loop  = (Cin/64 channel chunks) x (3 column taps kw); for each such step ONE TMA box of
//   (BH+2) rows x BW pixels x 64 channels lands in shared memory (zero fill outside the image is
//   the padding) and serves the three row taps kh = 0,1,2 by advancing the operand descriptor by
//   kh rows, so the input is fetched 3(BH+2)/BH times from L2 instead of 9 times.
//   Epilogue: TMEM -> registers -> bf16 -> swizzled shared tile -> TMA store of y; the per-channel
//   sum and sum of squares of the stored (rounded) values are accumulated per CTA for BatchNorm.
#include <cuda.h>

#include <algorithm>
#include <utility>

#include "nf_ptx.cuh"
#include "nf_tc.h"
#include "nf_tiles.cuh"

namespace {

constexpr int kThreads = 192;  // warp 0: TMA producer, warp 1: MMA issuer + TMEM owner, warps 2-5: epilogue
constexpr int kMaxStages = 8;
// normalisation threads of the fused BatchNorm + aux forward: two groups of 128 that take the stages in turn.  A single group
// was the slowest role of the kernel (busy 2350 of every 2450 cycles per tile while the issuer waited 520 on it: one warp per
// scheduler cannot hide the latency of its load - arithmetic - store - fence chain).  Splitting the ten rows of ONE box over
// two groups had measured slower (0.25 -> 0.27 ms); alternating whole stages gives each group twice the time per box.  Three
// groups measured slower again (aux forward 0.637 -> 0.681 ms over the c4 block): the tensor-core instructions stretch with
// every warp that works on shared memory.
constexpr int kXfGroups = 2;
constexpr int kXfThreads = 128 * kXfGroups;
constexpr int kFoldThreads = 320;  // folded-tap forward: producer, MMA issuer and two epilogue groups of four warps
// Tiles of y2 (the conv output read beside the input gradient, stats >= 2) in flight per CTA.  A slot turns over once per
// load latency plus epilogue time, so with the earlier two slots per epilogue group the kernel ran at the pace of these loads
// (about four tiles per HBM round trip) whatever else it did; with five the loads run as far ahead as the operand stages.
constexpr int kYSlots = 5;

// Position in a ring of `stages` buffers: index and the parity a waiter for "full" expects in this round
struct Ring {
  uint32_t s = 0, ph = 0;
  __device__ __forceinline__ void next(uint32_t stages) {
    if (++s == stages) {
      s = 0;
      ph ^= 1;
    }
  }
};

// a second group of four epilogue warps in the input gradient of tiles of several images, and for 256 channels without sums
constexpr int fwd_threads(int epi, int pt, int ns = 0) { return (epi == 0 && pt == 2) || ns ? kThreads + 128 : kThreads; }

struct FwdParams {
  int N, H, W, Cin, Cout;
  int BW, BH, tiles_w, tiles_h, n_tiles, total_tiles, kchunks, stages;
  int stride, BI;     // PT mode: conv stride and images per tile (BW*BH*BI = 128)
  int seg_steps;      // SEG: k-steps per accumulator
  TileGrid tg;
  int stats, yslots;  // yslots: buffers for the tiles of y2
  float* red;         // [grid / n_tiles * parts][2][Cout] channel partials
  int32_t* status;    // device status word
  const float* bias;  // EPI 1: per-channel bias added before the ReLU
  bf16* out;          // EPI 1: destination [N][H][W][Cout], written straight from registers
  // stats == 2 (EPI 0): the output is the gradient da at a BatchNorm+ReLU output of the same shape; the partial sums are
  // (dz, dz * xhat) with dz = da * 1[y2*scale+shift > 0], and the tiles of y2 come through tm_y2
  const float *bn_scale, *bn_shift, *bn_mu, *bn_invstd;
  CUtensorMap tm_y2;
};

struct TcPlan {
  int ok, BW, BH, BI, PT, BN, KC, RW, SEG, SB, NS, stages, grid, parts, yslots;
  size_t smem;
};

// POST = 1 (stats == 0): the forward writes ReLU(y * scale + shift) of the bf16-rounded y instead of y: BatchNorm with
// running statistics, whose coefficients are known beforehand (cache fill, exits).  Two channels, packed:
__device__ __forceinline__ uint32_t bn_relu2(uint32_t y, float2 sc, float2 sh) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(fmaxf(fmaf(__uint_as_float(y << 16), sc.x, sh.x), 0.f),
                                                 fmaxf(fmaf(__uint_as_float(y & 0xffff0000u), sc.y, sh.y), 0.f));
  return *reinterpret_cast<const uint32_t*>(&b);
}

// Sum of the next `n` segment accumulators (of four taken in turn; `taken` counts them) for one thread's row of BN columns.
template <int BN>
__device__ __forceinline__ void add_segments(uint32_t tbase, int n, uint32_t& taken, uint64_t* tfull, uint64_t* tempty,
                                             volatile int* abort_flag, float (&sum)[BN]) {
  for (int i = 0; i < n; ++i, ++taken) {
    const uint32_t acc = taken & 3;
    ptx::mbar_wait(&tfull[acc], (taken >> 2) & 1, abort_flag);  // sets the abort flag itself when it gives up
    ptx::tc_fence_after();
#pragma unroll
    for (int j = 0; j < BN / 16; ++j) {
      uint32_t v[16];
      ptx::tmem_ld16(tbase + acc * BN + j * 16, v);
      ptx::tmem_ld_wait();
#pragma unroll
      for (int e = 0; e < 16; ++e) sum[j * 16 + e] = i ? sum[j * 16 + e] + __uint_as_float(v[e]) : __uint_as_float(v[e]);
    }
    ptx::tc_fence_before();
    ptx::mbar_arrive(&tempty[acc]);
  }
}

// EPI 0: y in bf16 through a TMA store plus BatchNorm partial sums (BN = 64 or 128).
// EPI 1: bias + ReLU, channels [0, Cout) of a BN-wide tile written directly (aux conv; Cout <= BN <= 64,
//        weight rows beyond Cout are zero-filled by TMA).
// KC  : channels per K chunk of the activation box (64, or 16/32 for the narrow dh tensor of the aux
//       input gradient; rows of 2*KC bytes with the matching TMA swizzle).
// BMN : 0 = weights [tap][co][ci] read K-major (forward); 1 = weights [tap][f][c] read MN-major with the
//       taps mirrored, which makes the same kernel the input-gradient convolution da = dh (*) Wa^T.
// PT  : 1 = one TMA box per tap: stride-2 convolutions (the box is gathered with element stride 2, so the
//       three row taps cannot share a box), feature maps smaller than a tile, where a tile spans BI whole
//       images (8x8x2, 4x4x8, 2x2x32), and maps that no tile divides; p.H, p.W are the OUTPUT sizes.
//       2 (HN) = tiles of several images for narrow auxiliary convolutions: the box's dimensions run (channel, column, image, row),
//       so that a row tap is a constant offset for all images and THREE boxes per chunk serve the nine taps, in one stage with
//       all the weights.  The per-tap form is bound by its TMA rows (nine boxes of 128) and L2 fill: 512 channels, 8 filters,
//       8602 maps of 8x8, forward 352 -> 297 us; input gradient of a pooled 256-channel layer at 16x16 198 -> 126 us.
// RW  : 1 = all nine weight tiles of the CTA's channel tile stay resident in shared memory for the whole
//       kernel (single 64-channel K chunk, 9*BN*128 bytes); the pipeline then carries activations only.
// SEG : 1 (PT) = a new accumulator every seg_steps k-steps, the segments added in fp32 by the epilogue.  The tensor
//       core's running sum drops low bits on every instruction: over 2304 products 0.07 % of the bf16 outputs came out one unit
//       off the nearest value, against 0.016 % of an fp32 chain.  Maps that no tile divides had such chains (they ran on the CUDA
//       cores), and their layers are small enough for that to show; seg_steps (run_fwd) keeps the error below theirs.
// SB  : 1 (PT 0) = ONE box per chunk for the nine taps.  A tile is 8 columns x 16 rows, its box has a column more on either side, and an
//       image row of the tile is one 8-row group of the operand: a tap is a start address kh rows and kw pixels into the box, the groups
//       lie 10 pixels apart (the swizzle is a function of the address, so TMA and the tensor core agree wherever a tap starts).  The
//       products come in the order of the three-box form, so every bit stays.  For tiles of several images it gained nothing: there
//       the narrow instructions are the limit (512 channels, 8 filters, 8x8: 264 us with three boxes, 264 to 281 with one).
// NS  : 1 (EPI 0, no sums) = two epilogue groups with a staging tile of 64 channels each.  256 channels: they take the quarters of a
//       tile in turn; 64 and 128: every second tile.  One group was the slowest role: 16 000 to 20 000 cycles for a tile of 256
//       channels whose products take 9200 with 128 input channels (evaluation, 1777 maps of 16x16: 257 -> 190 us).
template <int BN, int EPI, int KC = 64, int BMN = 0, int PT = 0, int RW = 0, int SEG = 0, int POST = 0, int SB = 0, int NS = 0>
__global__ void __launch_bounds__(fwd_threads(EPI, PT, NS), 1)
conv_fwd_tc_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                   const __grid_constant__ CUtensorMap tm_y, const __grid_constant__ FwdParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int kARow = KC * 2;  // bytes of one pixel row of the activation box
  constexpr uint32_t kALayout = KC == 64 ? 2 : KC == 32 ? 4 : 6;
  constexpr bool HN = PT == 2, SG = HN && EPI == 0;  // SG: the sums of stats 2 are taken by a warp group of their own
  const int a_box = (p.BH + 2) * (SB ? 10 : p.BW) * p.BI * kARow;  // HN: one of the three column-shifted boxes, a multiple of 1024
  const int a_bytes = SB ? a_box : HN ? 3 * a_box : PT ? 128 * kARow : a_box;
  const int a_stride = (a_bytes + 1023) & ~1023;  // keeps the weight tiles 1024-byte aligned
  static_assert(!HN || RW == BMN, "forward: weights in the stages; input gradient: resident");
  static_assert(!SB || (PT == 0 && !SEG && (!BMN || RW)), "one box: tiles of one image; input gradient: weights resident");
  static_assert(!NS || (EPI == 0 && !SEG && PT != 2), "two groups: no sums");
  constexpr bool NINE = HN || SB;  // all nine taps of a chunk in one stage
  constexpr int b_bytes = RW ? 0 : NINE ? 9 * BN * 128 : PT ? (BMN ? (BN / 64) * KC * 128 : BN * 128) : BMN ? (BN / 64) * 3 * KC * 128 : 3 * BN * 128;
  // resident weights [kw][kh][BN][64] (SB: [chunk][kh][kw][BN][64], BMN: [half][kh][kw][KC][64])
  const int w_bytes = !RW ? 0 : BMN ? 9 * (BN / 64) * KC * 128 : (SB ? p.kchunks : 1) * 9 * BN * 128;
  const int stage_bytes = a_stride + b_bytes;
  // 256 channels leave through staging (and y2) tiles of 128, one half after the other: with 32 KB instead of 64 the ring gets four
  // stages of 48 KB for three, three for two beside y2 tiles (a stage is multiplied in 512 cycles, a fill takes over 1000)
  constexpr int kHalf = BN == 256 ? 2 : 1;
  constexpr int kSub = EPI == 0 ? BN / 64 / kHalf : 0;  // 64-channel sub-tiles of the output staging
  uint8_t* wres = smem + (size_t)p.stages * stage_bytes;
  uint8_t* stg = wres + w_bytes;
  constexpr int kStg = SG ? 2 : 1;              // staging tiles
  uint8_t* ybuf = stg + (NS ? 2 : kStg * kSub) * 16384;  // stats 2: the y2 tile of the tile in the epilogue (kSub sub-tiles)
  uint64_t* bars = reinterpret_cast<uint64_t*>(ybuf + (p.stats == 2 ? p.yslots : 0) * kSub * 16384);
  uint64_t* full = bars;
  uint64_t* empty = bars + kMaxStages;
  uint64_t* tfull = bars + 2 * kMaxStages;
  constexpr uint32_t kAccs = SEG ? 4 : 2;
  uint64_t* tempty = tfull + kAccs;
  uint64_t* wfull = tempty + kAccs;
  uint64_t* yfull = wfull + 1;
  uint64_t* yempty = yfull + 2;
  uint64_t* sfull = yempty + 2;  // SG: staging tile written / its sums taken
  uint64_t* sfree = sfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sfree + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* epi_go = reinterpret_cast<volatile int*>(tmem_slot + 2);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < (int)kAccs; ++a) {
      ptx::mbar_init(&tfull[a], 1);
      ptx::mbar_init(&tempty[a], NS && BN == 256 ? 256 : 128);
    }
    ptx::mbar_init(wfull, 1);
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&yfull[i], 1);
      ptx::mbar_init(&yempty[i], 128);
      ptx::mbar_init(&sfull[i], 128);
      ptx::mbar_init(&sfree[i], 128);
    }
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(&tm_x);
    ptx::prefetch_tmap(&tm_w);
    ptx::prefetch_tmap(&tm_y);
  }
  static_assert(!SEG || (PT == 1 && BN <= 128), "segmented accumulation: per-tap form");
  constexpr uint32_t kTmemCols = kAccs * BN < 32 ? 32 : kAccs * BN;
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  nf_pdl_begin();  // everything above touches only this CTA and overlaps the previous kernel

  if (warp == 0) {
    // ---------------- producer: one TMA box of activations + three weight tiles per k-step.  One thread runs the whole loop:
    // with a warp vote, a ring index by division and a reconvergence per step the producer and the issuer each spent about
    // 650 cycles per step whatever its size (measured with clock counters), more than a 256-wide step's arithmetic (512).
    if (ptx::elect_one()) {
      if constexpr (RW) {
        if (blockIdx.x < p.total_tiles) {
          ptx::mbar_expect_tx(wfull, (uint32_t)w_bytes);
          if constexpr (BMN) {
#pragma unroll
            for (int hf = 0; hf < BN / 64; ++hf)
              ptx::tma_load_4d(wres + hf * 9 * KC * 128, &tm_w, wfull, (blockIdx.x % p.n_tiles) * BN + hf * 64, 0, 0, 0);
          } else if constexpr (SB) {
            for (int ck = 0; ck < p.kchunks; ++ck) ptx::tma_load_4d(wres + ck * 9 * BN * 128, &tm_w, wfull, ck * 64, 0, 0, 0);
          } else {
#pragma unroll
            for (int kw = 0; kw < 3; ++kw) ptx::tma_load_4d(wres + kw * 3 * BN * 128, &tm_w, wfull, 0, (blockIdx.x % p.n_tiles) * BN, kw, 0);
          }
        }
      }
      Ring rg;
      uint32_t ptl = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < p.total_tiles; t += gridDim.x, ++ptl) {
        const TileAt at = tile_at(t, p.tg);
        const int co0 = at.nt * BN, w0 = at.w * p.BW, h0 = at.h * p.BH, n = at.n * p.BI;
        for (int ck = 0; ok && ck < p.kchunks; ++ck) {
#pragma unroll
          for (int tap = 0; tap < (NINE ? 1 : PT ? 9 : 3); ++tap, rg.next(p.stages)) {
            if (!ptx::mbar_wait(&empty[rg.s], rg.ph ^ 1, abort_flag)) { ok = false; break; }
            uint64_t* fb = &full[rg.s];
            uint8_t* a_s = smem + (size_t)rg.s * stage_bytes;
            ptx::mbar_expect_tx(fb, (uint32_t)(a_bytes + b_bytes));
            if constexpr (NINE) {
              if constexpr (SB) {
                ptx::tma_load_4d(a_s, &tm_x, fb, ck * KC, w0 - 1, h0 - 1, n);
              } else {
#pragma unroll
                for (int kw = 0; kw < 3; ++kw) ptx::tma_load_4d(a_s + kw * a_box, &tm_x, fb, ck * KC, w0 + kw - 1, n, h0 - 1);
              }
              if constexpr (!RW) {
                ptx::tma_load_4d(a_s + a_stride, &tm_w, fb, ck * 64, co0, 0, 0);  // [kh][kw][BN][64]
              }
            } else if constexpr (PT) {
              const int kh = tap / 3, kw = tap % 3;
              ptx::tma_load_4d(a_s, &tm_x, fb, ck * KC, p.stride * w0 + kw - 1, p.stride * h0 + kh - 1, n);
              if constexpr (BMN) {
#pragma unroll
                for (int hf = 0; hf < BN / 64; ++hf)  // [half][KC rows of f][64 channels], both taps mirrored
                  ptx::tma_load_4d(a_s + a_stride + hf * KC * 128, &tm_w, fb, co0 + hf * 64, 0, 2 - kw, 2 - kh);
              } else {
                ptx::tma_load_4d(a_s + a_stride, &tm_w, fb, ck * 64, co0, kw, kh);
              }
            } else {
              ptx::tma_load_4d(a_s, &tm_x, fb, ck * KC, w0 + tap - 1, h0 - 1, n);
              if constexpr (BMN) {
#pragma unroll
                for (int hf = 0; hf < BN / 64; ++hf)  // [half][kh][KC rows of f][64 channels], mirrored column tap
                  ptx::tma_load_4d(a_s + a_stride + hf * 3 * KC * 128, &tm_w, fb, co0 + hf * 64, 0, 2 - tap, 0);
              } else if constexpr (!RW) {
                ptx::tma_load_4d(a_s + a_stride, &tm_w, fb, ck * 64, co0, tap, 0);
              }
            }
          }
        }
        if constexpr (EPI == 0) {
          // the y2 tile of this output tile goes out after its operand loads: its buffer is free once the epilogue has finished
          // the statistics of the previous tile (of the one before with two buffers), which it does while this tile is multiplied
          if (kHalf == 1 && ok && p.stats == 2) {
            const uint32_t ys = p.yslots == 2 ? ptl & 1 : 0, yph = p.yslots == 2 ? (ptl >> 1) & 1 : ptl & 1;
            if (!ptx::mbar_wait(&yempty[ys], yph ^ 1, abort_flag)) break;
            ptx::mbar_expect_tx(&yfull[ys], (uint32_t)(kSub * 16384));
#pragma unroll
            for (int sb = 0; sb < kSub; ++sb) ptx::tma_load_4d(ybuf + (ys * kSub + sb) * 16384, &p.tm_y2, &yfull[ys], co0 + sb * 64, w0, h0, n);
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (one thread, as above)
    constexpr uint32_t idesc = ptx::idesc_bf16(128, BN, 0, BMN);
    // descriptors differ only in their 14-bit address field: constant upper parts, address added per use
    const uint64_t a_hi = ptx::sdesc(0, 16, (SB ? 10 : 8) * kARow, kALayout);
    const uint64_t b_hi = BMN ? ptx::sdesc(0, (NINE ? 9 : PT ? 1 : 3) * KC * 128, 1024, 2) : ptx::sdesc(0, 16, 1024, 2);
    const uint32_t a_row16 = (uint32_t)((HN ? p.BI : 1) * (SB ? 10 : p.BW) * kARow) >> 4;  // one image row of the box, in 16-byte units
    if (ptx::elect_one()) {
      Ring rg;
      uint32_t tl = 0;
      bool ok = true;
      if constexpr (RW) {
        if (blockIdx.x < p.total_tiles) ok = ptx::mbar_wait(wfull, 0, abort_flag);
      }
      const int steps = (NINE ? 1 : PT ? 9 : 3) * p.kchunks, seg = SEG ? p.seg_steps : steps;
      for (int t = blockIdx.x; ok && t < p.total_tiles; t += gridDim.x) {
        uint32_t acc = 0, d = 0, accumulate = 0;
        int step = 0, in_seg = 0;  // in_seg: k-steps of the segment so far
        for (int ck = 0; ok && ck < p.kchunks; ++ck) {
#pragma unroll
          for (int tap = 0; tap < (NINE ? 1 : PT ? 9 : 3); ++tap, rg.next(p.stages)) {
            if (in_seg == 0) {
              acc = tl % kAccs;
              if (!ptx::mbar_wait(&tempty[acc], ((tl / kAccs) & 1) ^ 1, abort_flag)) { ok = false; break; }
              ++tl;
              d = tmem_base + acc * BN;
              accumulate = 0;
            }
            ++step;
            ++in_seg;
            if (!ptx::mbar_wait(&full[rg.s], rg.ph, abort_flag)) { ok = false; break; }
            ptx::tc_fence_after();
            const uint32_t a_base = ptx::smem_u32(smem) + rg.s * stage_bytes;
            const uint32_t a16 = a_base >> 4;
            const uint32_t b16 = RW ? (ptx::smem_u32(wres) + (SB && !BMN ? ck * 9 : tap * 3) * BN * 128) >> 4 : (a_base + a_stride) >> 4;
            if constexpr (NINE) {  // all nine taps of the chunk, in the order of the per-tap form (HN) or of the three-box form
              const uint32_t col16 = SB ? kARow >> 4 : (uint32_t)a_box >> 4;  // one column tap on
#pragma unroll
              for (int t9 = 0; t9 < 9; ++t9)
#pragma unroll
                for (int k = 0; k < KC / 16; ++k) {
                  const int kh = HN ? t9 / 3 : t9 % 3, kw = HN ? t9 % 3 : t9 / 3, tw = kh * 3 + kw;
                  const uint64_t ad = a_hi | (uint64_t)(a16 + kw * col16 + kh * a_row16 + k * 2);
                  const uint64_t bd = b_hi | (uint64_t)(BMN ? b16 + (((8 - tw) * KC * 128 + k * 16 * 128) >> 4) : b16 + ((tw * BN * 128 + k * 32) >> 4));
                  ptx::mma_f16(d, ad, bd, idesc, accumulate);
                  accumulate = 1;
                }
            } else
#pragma unroll
            for (int kh = 0; kh < (PT ? 1 : 3); ++kh)
#pragma unroll
              for (int k = 0; k < KC / 16; ++k) {
                const uint64_t ad = a_hi | (uint64_t)(a16 + kh * a_row16 + k * 2);
                const uint64_t bd = b_hi | (uint64_t)(BMN ? b16 + (((PT ? 0 : (2 - kh) * KC * 128) + k * 16 * 128) >> 4)
                                                          : b16 + ((kh * BN * 128 + k * 32) >> 4));
                ptx::mma_f16(d, ad, bd, idesc, accumulate);
                accumulate = 1;
              }
            ptx::mma_commit(&empty[rg.s]);
            if (step == steps || in_seg == seg) {
              ptx::mma_commit(&tfull[acc]);
              in_seg = 0;
            }
          }
        }
      }
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: 128 threads, thread <-> output pixel (TMEM lane)
    if constexpr (NS) {
      const int grp = warp >= 6 ? 1 : 0, et = (threadIdx.x - 64) & 127, lg = warp & 3, r = lg * 32 + lane;
      const bool affine = POST, biased = !POST && p.bias;
      uint8_t* const stile = stg + grp * 16384;
      constexpr bool kShare = BN == 256;  // both groups work on every tile
      constexpr int kQ = kShare ? 2 : BN / 64;
      uint32_t tl = kShare ? 0 : grp;
      bool go = true;
      for (int t = blockIdx.x + tl * gridDim.x; go && t < p.total_tiles; t += (kShare ? 1 : 2) * gridDim.x, tl += kShare ? 1 : 2) {
        const TileAt at = tile_at(t, p.tg);
        const uint32_t acc = tl & 1;
        ptx::mbar_wait(&tfull[acc], (tl >> 1) & 1, abort_flag);  // sets the abort flag itself when it gives up
        ptx::tc_fence_after();
#pragma unroll
        for (int qi = 0; qi < kQ; ++qi) {
          const int cq = (kShare ? 2 * qi + grp : qi) * 64, ch0 = at.nt * BN + cq;  // first column and channel of these 64
          if (et == 0) {
            ptx::tma_store_wait_read();  // the last store out of this group's staging tile has finished reading it
            epi_go[grp] = *abort_flag ? 0 : 1;
          }
          ptx::named_barrier(1 + grp, 128);
          if (!epi_go[grp]) {
            go = false;
            break;
          }
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            uint32_t v[32];
            ptx::tmem_ld32(tmem_base + ((uint32_t)(lg * 32) << 16) + acc * BN + cq + j * 32, v);
            ptx::tmem_ld_wait();
            const float4* c0 = reinterpret_cast<const float4*>((POST ? p.bn_scale : p.bias) + ch0 + j * 32);
            const float4* c1 = reinterpret_cast<const float4*>(p.bn_shift + ch0 + j * 32);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t w[4];
#pragma unroll
              for (int e = 0; e < 4; e += 2) {
                float o[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) o[i] = __uint_as_float(v[q * 8 + 2 * e + i]);
                if (biased) {  // bias and ReLU before the value is rounded for storage
                  const float4 b = __ldg(c0 + q * 2 + e / 2);
                  o[0] = fmaxf(o[0] + b.x, 0.f); o[1] = fmaxf(o[1] + b.y, 0.f); o[2] = fmaxf(o[2] + b.z, 0.f); o[3] = fmaxf(o[3] + b.w, 0.f);
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                  const __nv_bfloat162 b2 = __floats2bfloat162_rn(o[2 * i], o[2 * i + 1]);
                  w[e + i] = *reinterpret_cast<const uint32_t*>(&b2);
                }
                if (affine) {
                  const float4 sc = __ldg(c0 + q * 2 + e / 2), sh = __ldg(c1 + q * 2 + e / 2);
                  w[e] = bn_relu2(w[e], make_float2(sc.x, sc.y), make_float2(sh.x, sh.y));
                  w[e + 1] = bn_relu2(w[e + 1], make_float2(sc.z, sc.w), make_float2(sh.z, sh.w));
                }
              }
              *reinterpret_cast<uint4*>(stile + r * 128 + (((j * 4 + q) ^ (r & 7)) * 16)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
          }
          if (qi == kQ - 1) {
            ptx::tc_fence_before();
            ptx::mbar_arrive(&tempty[acc]);
          }
          ptx::fence_async_smem();
          ptx::named_barrier(1 + grp, 128);
          if (et == 0) {
            ptx::tma_store_4d(&tm_y, stile, ch0, (int)at.w * p.BW, (int)at.h * p.BH, (int)at.n * p.BI);
            ptx::tma_store_commit();
          }
        }
      }
      if (et == 0) ptx::tma_store_wait_all();
    } else if constexpr (EPI == 0) {
    const int et = threadIdx.x - 64;
    const int lg = warp & 3;          // TMEM lane group this warp may read
    const int r = lg * 32 + lane;     // row of the tile = pixel (r % BW, r / BW)
    constexpr int kRowsPer = BN >= 128 ? 128 : 64;  // rows each thread sums for its channel
    const int sc = et % BN, shalf = et / BN;        // stats: channel and row half of this thread
    // place of the thread's pixel in its tile; HN: rows of the accumulator run over (row, image, column)
    const int rw = r % p.BW, rh = HN ? r / (p.BW * p.BI) : (r / p.BW) % p.BH;
    const int sr = HN ? (((r / p.BW) % p.BI) * p.BH + rh) * p.BW + rw : r;  // its row of the staging tile (image, row, column)
    uint32_t sg = 0;                                  // SEG: segments taken so far
    float ssum = 0.f, ssq = 0.f;
    float ssum2 = 0.f, ssq2 = 0.f;                  // BN = 256: the thread's second channel, sc + 128
    uint32_t tl = 0;
    int my_nt = blockIdx.x % p.n_tiles;
    float bsc = 0.f, bsh = 0.f, bsc2 = 0.f, bsh2 = 0.f;  // stats 2: BatchNorm scale / shift of the thread's channel(s)
    if (p.stats == 2) {
      const int ch = my_nt * BN + sc;
      bsc = p.bn_scale[ch];
      bsh = p.bn_shift[ch];
      if constexpr (BN == 256) {
        bsc2 = p.bn_scale[ch + 128];
        bsh2 = p.bn_shift[ch + 128];
      }
    }
    const bool sums = SG && warp >= 6;
    if constexpr (SG) {
      if (sums && p.stats == 2) {
        // sums of (dz, dz * y2), one channel per thread in row order as below, while the other group stages the next tile (that
        // work in one group took 8000 cycles per 128 x 128 tile whose products take 600)
        const int st = threadIdx.x - 192, c = st % BN, half = st / BN;
        const float fsc = p.bn_scale[my_nt * BN + c], fsh = p.bn_shift[my_nt * BN + c];
        for (int t = blockIdx.x; t < p.total_tiles; t += gridDim.x, ++tl) {
          const uint32_t bsel = tl & 1, ph = (tl >> 1) & 1;
          if (!ptx::mbar_wait(&yfull[bsel], ph, abort_flag) || !ptx::mbar_wait(&sfull[bsel], ph, abort_flag)) break;
          const uint8_t* dcol = stg + bsel * kSub * 16384 + (c / 64) * 16384 + (c % 8) * 2 + half * kRowsPer * 128;
          const uint8_t* ycol = ybuf + bsel * kSub * 16384 + (c / 64) * 16384 + (c % 8) * 2 + half * kRowsPer * 128;
          const int u = (c % 64) / 8;
#pragma unroll 16
          for (int row = 0; row < kRowsPer; ++row) {
            const int off = row * 128 + ((u ^ (row & 7)) * 16);
            const float d = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(dcol + off));
            const float yv = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(ycol + off));
            const float dz = fmaf(yv, fsc, fsh) > 0.f ? d : 0.f;
            ssum += dz;
            ssq = fmaf(dz, yv, ssq);
          }
          ptx::mbar_release_read(&yempty[bsel]);
          ptx::mbar_arrive(&sfree[bsel]);
        }
        const int ch = my_nt * BN + c;
        ssq = (float)((double)p.bn_invstd[ch] * ((double)ssq - (double)p.bn_mu[ch] * (double)ssum));
        const size_t row = (size_t)(blockIdx.x / p.n_tiles) * (128 / BN) + half;
        p.red[(row * 2 + 0) * p.Cout + ch] = ssum;
        p.red[(row * 2 + 1) * p.Cout + ch] = ssq;
      }
    }
    for (int t = sums ? p.total_tiles : blockIdx.x; t < p.total_tiles; t += gridDim.x, ++tl) {
      const TileAt at = tile_at(t, p.tg);
      const int nt = at.nt, w0 = at.w * p.BW, h0 = at.h * p.BH, n = at.n * p.BI;
      const uint32_t acc = tl & 1, aph = (tl >> 1) & 1;
      float seg[SEG ? BN : 1];
      if constexpr (SEG) {
        add_segments<BN>(tmem_base + ((uint32_t)(lg * 32) << 16), (9 * p.kchunks + p.seg_steps - 1) / p.seg_steps, sg, tfull, tempty, abort_flag, seg);
      } else {
        ptx::mbar_wait(&tfull[acc], aph, abort_flag);  // sets the abort flag itself when it gives up
        ptx::tc_fence_after();
      }
      bool go = true;
#pragma unroll
      for (int hf = 0; hf < kHalf; ++hf) {
        const int ch0 = nt * BN + hf * 128;  // first channel of the half
        uint8_t* const stile = stg + (SG ? (tl & 1) * kSub * 16384 : 0);
        if constexpr (SG) {
          if (p.stats == 2) ptx::mbar_wait(&sfree[tl & 1], ((tl >> 1) & 1) ^ 1, abort_flag);
        }
        if (et == 0) {
          // the last store out of this staging tile has finished reading it
          if constexpr (SG) ptx::tma_store_wait_read_but_one(); else ptx::tma_store_wait_read();
          *epi_go = *abort_flag ? 0 : 1;  // one thread decides for all 128, so nobody is left alone at a barrier
        }
        ptx::named_barrier(1, 128);
        if (!*epi_go) {
          go = false;
          break;
        }
        if constexpr (kHalf == 2) {
          if (et == 0 && p.stats == 2) {  // every thread has passed the last half's sums
            ptx::mbar_expect_tx(yfull, (uint32_t)(kSub * 16384));
#pragma unroll
            for (int sb = 0; sb < kSub; ++sb) ptx::tma_load_4d(ybuf + sb * 16384, &p.tm_y2, yfull, ch0 + sb * 64, w0, h0, n);
          }
        }
        const bool inside = w0 + rw < p.W && h0 + rh < p.H;  // a pixel over the edge is staged as zero: it adds nothing to the sums
#pragma unroll
        for (int j = 0; j < BN / kHalf / 32; ++j) {
          uint32_t v[32];
          if constexpr (SEG) {
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(seg[j * 32 + e]);
          } else {
            ptx::tmem_ld32(tmem_base + ((uint32_t)(lg * 32) << 16) + acc * BN + hf * 128 + j * 32, v);
            ptx::tmem_ld_wait();
          }
          uint8_t* sub = stile + ((j * 32) / 64) * 16384 + sr * 128;
          const int u0 = ((j * 32) % 64) / 8;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float o0 = __uint_as_float(v[q * 8 + 2 * e]), o1 = __uint_as_float(v[q * 8 + 2 * e + 1]);
              if (p.bias) {  // wide aux forward: bias and ReLU before the value is rounded for storage
                const float* bch = p.bias + ch0 + j * 32 + q * 8 + 2 * e;
                o0 = fmaxf(o0 + __ldg(bch), 0.f);
                o1 = fmaxf(o1 + __ldg(bch + 1), 0.f);
              }
              const __nv_bfloat162 b2 = __floats2bfloat162_rn(o0, o1);
              w[e] = *reinterpret_cast<const uint32_t*>(&b2);
            }
            if constexpr (POST) {
              const float* ps = p.bn_scale + ch0 + j * 32 + q * 8;
              const float* ph = p.bn_shift + ch0 + j * 32 + q * 8;
#pragma unroll
              for (int e = 0; e < 4; ++e)
                w[e] = bn_relu2(w[e], __ldg(reinterpret_cast<const float2*>(ps) + e), __ldg(reinterpret_cast<const float2*>(ph) + e));
            }
            *reinterpret_cast<uint4*>(sub + (((u0 + q) ^ (sr & 7)) * 16)) = inside ? make_uint4(w[0], w[1], w[2], w[3]) : make_uint4(0u, 0u, 0u, 0u);
          }
        }
        if (!SEG && hf == kHalf - 1) {
          ptx::tc_fence_before();
          ptx::mbar_arrive(&tempty[acc]);
        }
        ptx::fence_async_smem();
        ptx::named_barrier(1, 128);
        if (et == 0) {
#pragma unroll
          for (int sb = 0; sb < kSub; ++sb) ptx::tma_store_4d(&tm_y, stile + sb * 16384, ch0 + sb * 64, w0, h0, n);
          ptx::tma_store_commit();
        }
        if constexpr (SG) {
          if (p.stats == 2) ptx::mbar_arrive(&sfull[tl & 1]);
          continue;
        }
        if (p.stats == 2) {
          // sums of dz and dz*y2 (the last step turns them into sum dz*xhat = invstd * (sum dz*y2 - mu * sum dz))
          const uint32_t ys = p.yslots == 2 ? tl & 1 : 0;
          const uint8_t* yb = ybuf + ys * kSub * 16384;
          ptx::mbar_wait(&yfull[ys], kHalf == 2 ? hf : p.yslots == 2 ? (tl >> 1) & 1 : tl & 1, abort_flag);
          const float csc = hf ? bsc2 : bsc, csh = hf ? bsh2 : bsh;
          float &sum = hf ? ssum2 : ssum, &sq = hf ? ssq2 : ssq;
          const int coff = (sc / 64) * 16384 + (sc % 8) * 2;
          const int u = (sc % 64) / 8;
          const int rb = shalf * kRowsPer;
#pragma unroll 8
          for (int rr = 0; rr < kRowsPer; ++rr) {
            const int row = rb + rr;
            const int off = coff + row * 128 + ((u ^ (row & 7)) * 16);
            const float d = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(stg + off));
            const float yv = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(yb + off));
            const float dz = fmaf(yv, csc, csh) > 0.f ? d : 0.f;
            sum += dz;
            sq = fmaf(dz, yv, sq);
          }
          ptx::mbar_release_read(&yempty[ys]);
        } else if (p.stats) {
          float &sum = hf ? ssum2 : ssum, &sq = hf ? ssq2 : ssq;
          const uint8_t* col = stg + (sc / 64) * 16384 + (sc % 8) * 2;
          const int u = (sc % 64) / 8;
          const int rb = shalf * kRowsPer;
#pragma unroll 8
          for (int rr = 0; rr < kRowsPer; ++rr) {
            const int row = rb + rr;
            const float v = __bfloat162float(*reinterpret_cast<const __nv_bfloat16*>(col + row * 128 + ((u ^ (row & 7)) * 16)));
            sum += v;
            sq = fmaf(v, v, sq);
          }
        }
      }
      if (!go) break;
    }
    if (et == 0) ptx::tma_store_wait_all();
    if (!SG && p.stats) {
      constexpr int parts = 128 / BN > 0 ? 128 / BN : 1;
      const size_t b = (size_t)(blockIdx.x / p.n_tiles) * parts + shalf;  // the CTAs of one pixel range fill one row of partials
      if (p.stats == 2) {
        const int ch = my_nt * BN + sc;
        ssq = (float)((double)p.bn_invstd[ch] * ((double)ssq - (double)p.bn_mu[ch] * (double)ssum));
        if constexpr (BN == 256) ssq2 = (float)((double)p.bn_invstd[ch + 128] * ((double)ssq2 - (double)p.bn_mu[ch + 128] * (double)ssum2));
      }
      p.red[(b * 2 + 0) * p.Cout + my_nt * BN + sc] = ssum;
      p.red[(b * 2 + 1) * p.Cout + my_nt * BN + sc] = ssq;
      if constexpr (BN == 256) {
        p.red[(b * 2 + 0) * p.Cout + my_nt * BN + 128 + sc] = ssum2;
        p.red[(b * 2 + 1) * p.Cout + my_nt * BN + 128 + sc] = ssq2;
      }
    }
    } else {
      const int et = threadIdx.x - 64;
      const int lg = warp & 3;
      const int r = lg * 32 + lane;
      // place of the thread's pixel in its tile
      const int rw = r % p.BW, rh = HN ? r / (p.BW * p.BI) : (r / p.BW) % p.BH, img = HN ? (r / p.BW) % p.BI : r / (p.BW * p.BH);
      uint32_t sg = 0;
      uint32_t tl = 0;
      for (int t = blockIdx.x; t < p.total_tiles; t += gridDim.x, ++tl) {
        const TileAt at = tile_at(t, p.tg);
        const int w0 = at.w * p.BW, h0 = at.h * p.BH, n = at.n * p.BI;
        const uint32_t acc = tl & 1, aph = (tl >> 1) & 1;
        float seg[SEG ? BN : 1];
        if constexpr (SEG) {
          add_segments<BN>(tmem_base + ((uint32_t)(lg * 32) << 16), (9 * p.kchunks + p.seg_steps - 1) / p.seg_steps, sg, tfull, tempty, abort_flag, seg);
        } else {
          ptx::mbar_wait(&tfull[acc], aph, abort_flag);
          ptx::tc_fence_after();
        }
        if (et == 0) *epi_go = *abort_flag ? 0 : 1;
        ptx::named_barrier(1, 128);
        if (!*epi_go) break;
        const bool img_ok = n + img < p.N && w0 + rw < p.W && h0 + rh < p.H;
        bf16* dst = p.out + (((size_t)(n + img) * p.H + h0 + rh) * p.W + w0 + rw) * p.Cout;
#pragma unroll
        for (int j = 0; j < BN / 16; ++j) {
          uint32_t v[16];
          if constexpr (SEG) {
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = __float_as_uint(seg[j * 16 + e]);
          } else {
            ptx::tmem_ld16(tmem_base + ((uint32_t)(lg * 32) << 16) + acc * BN + j * 16, v);
            ptx::tmem_ld_wait();
          }
          if (j * 16 < p.Cout && img_ok) {
            uint32_t w[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const int c = j * 16 + 2 * e;
              const float a0 = c < p.Cout ? fmaxf(__uint_as_float(v[2 * e]) + p.bias[c], 0.f) : 0.f;
              const float a1 = c + 1 < p.Cout ? fmaxf(__uint_as_float(v[2 * e + 1]) + p.bias[c + 1], 0.f) : 0.f;
              const __nv_bfloat162 b2 = __floats2bfloat162_rn(a0, a1);
              w[e] = *reinterpret_cast<const uint32_t*>(&b2);
            }
            const int c0 = j * 16;
            if ((p.Cout & 7) == 0) {
              *reinterpret_cast<uint4*>(dst + c0) = make_uint4(w[0], w[1], w[2], w[3]);
              if (c0 + 8 < p.Cout) *reinterpret_cast<uint4*>(dst + c0 + 8) = make_uint4(w[4], w[5], w[6], w[7]);
            } else if ((p.Cout & 3) == 0) {
#pragma unroll
              for (int g4 = 0; g4 < 4; ++g4)
                if (c0 + 4 * g4 < p.Cout) *reinterpret_cast<uint2*>(dst + c0 + 4 * g4) = make_uint2(w[2 * g4], w[2 * g4 + 1]);
            } else {
              for (int e = 0; e < 16 && c0 + e < p.Cout; ++e)
                dst[c0 + e] = __ushort_as_bfloat16((unsigned short)((w[e >> 1] >> ((e & 1) * 16)) & 0xffffu));
            }
          }
        }
        if constexpr (!SEG) {
          ptx::tc_fence_before();
          ptx::mbar_arrive(&tempty[acc]);
        }
      }
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(p.status, NF_ETIMEOUT);
    // give copies still in flight time to land before the shared memory is released
    const unsigned long long t0 = ptx::globaltimer();
    while (ptx::globaltimer() - t0 < 2000000ull) __nanosleep(1000);
  }
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, kTmemCols);
  }
}


// ---------------------------------------------------------------- forward, 64 -> 64 channels, column taps folded into N
// With a 64-wide N tile an MMA is bound by the bytes of its operands, not by its arithmetic.  This
// variant widens N to 192: D'[pixel, (kw, co)] = sum_{kh, ci} X[pixel shifted by kh rows, ci] * W[kh][kw][co][ci],
// i.e. the three column taps become three 64-column groups of one accumulator and only the three row
// taps remain in the K loop (12 instructions of N = 192 per tile instead of 36 of N = 64, one
// activation box per tile instead of three).  The output is the shift-add
//   y[h, w, co] = D'[(h, w-1), kw=0, co] + D'[(h, w), kw=1, co] + D'[(h, w+1), kw=2, co],
// done in the epilogue with warp shuffles: a tile is 16 columns x 8 rows of pixels of which the outer
// two columns are halo, so the left/right neighbours of every output pixel are adjacent TMEM lanes of the
// same warp.  14 x 8 output pixels per tile; needs W % 14 == 0 and H % 8 == 0.
// Per-channel partial sums of one epilogue group (128 threads = 4 warps; a thread holds 8 channels, lane & 7 selects which):
// shuffles add the lanes of a warp, the warps are added through `scratch` (2 KB of shared memory the group owns) in warp order,
// and lanes 0..7 of the group's first warp write the 64 channel totals: red[0][c0 + ..] the first sums, red[1][..] the second
// (bn_second: turned into sum(dz * xhat) = invstd * (sum(dz * y) - mu * sum(dz)) in fp64).
__device__ __forceinline__ void fold_group_partial(float (&s1)[8], float (&s2)[8], float* scratch, int grp, int lg, int lane,
                                                   bool bn_second, const float* mu, const float* invstd, int c0, float* red, int C) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    s1[i] += __shfl_xor_sync(0xffffffffu, s1[i], 8);
    s2[i] += __shfl_xor_sync(0xffffffffu, s2[i], 8);
    s1[i] += __shfl_xor_sync(0xffffffffu, s1[i], 16);
    s2[i] += __shfl_xor_sync(0xffffffffu, s2[i], 16);
  }
  ptx::named_barrier(1 + grp, 128);  // the group's last TMA store has read the staging tile (its issuer waited before this)
  if (lane < 8) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      scratch[(lg * 2 + 0) * 64 + lane * 8 + i] = s1[i];
      scratch[(lg * 2 + 1) * 64 + lane * 8 + i] = s2[i];
    }
  }
  ptx::named_barrier(1 + grp, 128);
  if (lg == 0 && lane < 8) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int c = lane * 8 + i;
      const float a = ((scratch[0 * 64 + c] + scratch[2 * 64 + c]) + scratch[4 * 64 + c]) + scratch[6 * 64 + c];
      float b = ((scratch[1 * 64 + c] + scratch[3 * 64 + c]) + scratch[5 * 64 + c]) + scratch[7 * 64 + c];
      if (bn_second) b = (float)((double)invstd[c0 + c] * ((double)b - (double)mu[c0 + c] * (double)a));
      red[c0 + c] = a;
      red[C + c0 + c] = b;
    }
  }
}

struct FoldParams {
  int N, H, W, Cout, kchunks, n_tiles, tiles_w, tiles_h, total_tiles, stages, stats;
  TileGrid tg;
  float* red;         // EPI 0, stats != 0: [grid / n_tiles * 8][2][Cout]
  int32_t* status;
  const float *bn_scale, *bn_shift, *bn_mu, *bn_invstd;  // stats >= 2
  const float *bn_sdz, *bn_sdzx;                         // stats == 4: the reduced sums of the whole batch
  float inv_m;                                           // stats == 4: 1 / (elements per channel)
  const float* bias;  // EPI 1
  bf16* out;          // EPI 1: [N][H][W][Cout]
  // XF: the input map is the conv output y; a = ReLU(y*scale + shift) is formed in shared memory and written to xf_a
  const float *xf_scale, *xf_shift;
  bf16* xf_a;         // [N][H][W][64 * kchunks]
  // EPI 1 with pool_part != nullptr: h itself is not written.  What the rest of the step needs of it leaves the epilogue
  // directly: per tile and epilogue warp the per-channel sums of h over the warp's pixels (the average pool to 2 x 2 adds
  // them up; a tile never straddles a quadrant: H/2 % 8 == 0, W/2 % 14 == 0), and one bit per element, h > 0.
  float* pool_part;   // [total_tiles][4][Cout]
  uint8_t* mask;      // [N][H][W][Cout / 8], bit f % 8 of byte f / 8
};

// G   : width of one column-tap group of the accumulator (N = 3*G): 64 for the main conv, 16/32/64 for the
//       aux conv with F <= G filters (weight rows beyond F are zero-filled by TMA).
// EPI : 0 = y in bf16 through a TMA store + BatchNorm partial sums (G = 64, Cout = 64);
//       1 = bias + ReLU, F channels written straight from registers (aux conv forward).
// Cin = 64 * kchunks; all 9 * kchunks weight tiles stay resident in shared memory.
// stats (EPI 0): 1 = per-channel sums of (y, y^2) of the stored values (BatchNorm forward statistics);
//       2 = the output is the gradient da at a BatchNorm+ReLU output of the same shape: per-channel sums of
//       (dz, dz * xhat) with dz = da * 1[y2*scale+shift > 0], xhat = (y2 - mu) * invstd, where the tile of the
//       pre-normalisation values y2 is fetched through tm_y2 (BatchNorm backward reduction fused into the producer of da);
//       3 = the same sums, but da is not written at all; 4 = the second pass of that pair: da is formed again, turned
//       into dy = scale * (dz - sum(dz)/M - xhat * sum(dz*xhat)/M) in the staging tile with the sums of pass 3, and dy is
//       what the TMA store writes.  Passes 3 + 4 replace "write da; read y and da; write dy" by one more read of the
//       narrow dh tensor: da never reaches memory.
// KC / MIR: KC = channels of the activation box (64; 16 or 32 for the aux input gradient whose input dh has F
// channels), MIR = 1 reads the weights [tap][f][c] MN-major with both taps mirrored (input-gradient convolution;
// the CTA's 64-channel output tile is blockIdx.x % n_tiles).
// UF = 1 (input gradient with KC <= 32 only): the column taps are NOT folded.  With so few input channels a tile needs
// only nine instructions (one per tap, N = 64) even unfolded, and the epilogue is what bounds the kernel: three
// column-shifted activation boxes per stage replace the shift-add, the accumulator is 64 columns wide and all 16 x 8
// pixels of a tile are outputs (W % 16 == 0).
// XF = 1 (aux forward only): BatchNorm + ReLU of the layer are applied on the way in.  The boxes are loaded from the
// conv output y; four more warps turn each box into a = ReLU(y*scale + shift) in place (zero outside the image, as the
// padding of a must be), write the tile's own 14 x 8 pixels of a to global memory (the layer's output activation) and
// only then hand the stage to the issuer.  The separate normalisation pass (read y, write a) and this kernel's read of
// a disappear; the halo pixels are normalised by both neighbours.
template <int G, int EPI, int KC = 64, int MIR = 0, int UF = 0, int XF = 0, int POST = 0>
__global__ void __launch_bounds__(kFoldThreads + kXfThreads * XF, 1)
conv_fwd_fold_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                     const __grid_constant__ CUtensorMap tm_y, const __grid_constant__ CUtensorMap tm_y2, const FoldParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int kARow = KC * 2;               // bytes of one pixel of the activation box
  constexpr uint32_t kALayout = KC == 64 ? 2 : KC == 32 ? 4 : 6;
  static_assert(!UF || (MIR && EPI == 0 && G == 64 && KC <= 32), "unfolded form: input gradient with few input channels");
  static_assert(!XF || (EPI == 1 && KC == 64 && !MIR && !UF), "fused normalisation: aux forward only");
  // UF = 2: tiles of 8 columns x 16 rows fed by ONE box of 10 x 18 pixels.  An image row of the tile is then exactly one
  // 8-row group of the operand, so the nine taps are nine start addresses (kh * 10 + kw pixels into the box) with a constant
  // pitch of 10 pixels between groups: a third of the TMA rows of the three-box form, whose narrow 32-byte rows made the
  // producer the slowest role of the kernel.  The shared-memory swizzle is a function of the address, so TMA and the tensor
  // core agree wherever a tap starts.
  constexpr int kBox = UF == 2 ? 18 * 10 * kARow : 10 * 16 * kARow;  // (8+2) rows x 16 pixels x KC channels
  constexpr int kABytes = UF == 2 ? (kBox + 1023) / 1024 * 1024 : (UF ? 3 : 1) * kBox;  // UF 1: one box per column tap
  constexpr int kTW = UF == 2 ? 8 : UF ? 16 : 14;  // output columns of a tile
  constexpr int kTH = UF == 2 ? 16 : 8;            // output rows of a tile
  constexpr int kStatIters = UF ? 8 : 7;           // 16-row slices of the staged tile (128 or 112 pixels)
  constexpr int kWTile = MIR ? 3 * KC * 128 : 3 * G * kARow;  // one kernel row: [kw*G + co][64 ci], or mirrored [kw][f][64 c]
  const int w_bytes = 3 * p.kchunks * kWTile; // [chunk][kh][kw*G + co][64 ci]
  uint8_t* wres = smem + (size_t)p.stages * kABytes;
  uint8_t* stg = wres + w_bytes;              // EPI 0: 112 (UF: 128) output pixels x 128 bytes
  uint8_t* ybuf = stg + 2 * 16384;            // EPI 0, stats >= 2: kYSlots tiles of y2, taken in turn by the CTA's tiles
  constexpr int kAStg = 112 * 128;            // XF: one 14 x 8-pixel tile of a on its way to global memory (three in rotation per group)
  // one staging tile per epilogue group (EPI 0), or the three tiles of a (XF)
  uint64_t* bars = reinterpret_cast<uint64_t*>(stg + (EPI == 0 ? (p.stats >= 2 ? 2 + kYSlots : 2) * 16384 : XF ? 3 * kXfGroups * kAStg : 0));
  uint64_t* full = bars;
  uint64_t* empty = bars + kMaxStages;
  uint64_t* tfull = bars + 2 * kMaxStages;
  uint64_t* tempty = tfull + 4;
  uint64_t* wfull = tempty + 4;
  uint64_t* yfull = wfull + 1;
  uint64_t* yempty = yfull + kYSlots;
  uint64_t* xfull = yempty + kYSlots;  // XF: stage normalised, ready for the issuer
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(xfull + kMaxStages);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* epi_go = reinterpret_cast<volatile int*>(tmem_slot + 2);  // [2], one per epilogue group
  volatile int* xf_go = reinterpret_cast<volatile int*>(tmem_slot + 4);   // [2 per group], alternating between a group's iterations
  // Accumulators in tensor memory.  The unfolded form needs 64 columns each and keeps four, so that the issuer can run two
  // tiles ahead of each epilogue group (group g takes the tiles tl = g, g + 2, ... and so alternates between two of them);
  // the folded forms need up to 192 columns each and keep two, one per group.
  constexpr uint32_t kAccs = UF ? 4 : 2;
  constexpr uint32_t kAccStride = UF ? 128 : G == 64 ? 256 : 128;  // columns between two accumulators
  constexpr uint32_t kTmemCols = kAccs * kAccStride;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
      ptx::mbar_init(&xfull[s], 128);
    }
    for (int a = 0; a < (int)kAccs; ++a) {
      ptx::mbar_init(&tfull[a], 1);
      ptx::mbar_init(&tempty[a], 128);
    }
    for (int a = 0; a < kYSlots; ++a) {
      ptx::mbar_init(&yfull[a], 1);
      ptx::mbar_init(&yempty[a], 128);
    }
    ptx::mbar_init(wfull, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(&tm_x);
    ptx::prefetch_tmap(&tm_w);
    ptx::prefetch_tmap(&tm_y);
    ptx::prefetch_tmap(&tm_y2);
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  nf_pdl_begin();  // everything above touches only this CTA and overlaps the previous kernel

  if (warp == 0) {
    if (ptx::elect_one()) {  // one thread runs the whole loop, as in the generic kernel
      if (blockIdx.x < p.total_tiles) {
        ptx::mbar_expect_tx(wfull, (uint32_t)w_bytes);
        for (int ck = 0; ck < p.kchunks; ++ck)
#pragma unroll
          for (int kh = 0; kh < 3; ++kh)
            ptx::tma_load_4d(wres + (ck * 3 + kh) * kWTile, &tm_w, wfull, MIR ? (int)(blockIdx.x % p.n_tiles) * 64 : ck * 64, 0, 0, kh);
      }
      Ring rg, yr;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < p.total_tiles; t += gridDim.x) {
        const TileAt at = tile_at(t, p.tg);
        const int w0 = at.w * kTW, h0 = at.h * kTH, n = at.n;
        for (int ck = 0; ck < p.kchunks; ++ck, rg.next(p.stages)) {
          if (!ptx::mbar_wait(&empty[rg.s], rg.ph ^ 1, abort_flag)) { ok = false; break; }
          uint64_t* fb = &full[rg.s];
          uint8_t* st = smem + (size_t)rg.s * kABytes;
          ptx::mbar_expect_tx(fb, (uint32_t)(UF == 2 ? kBox : kABytes));
          if constexpr (UF == 1) {
#pragma unroll
            for (int kw = 0; kw < 3; ++kw) ptx::tma_load_4d(st + kw * kBox, &tm_x, fb, ck * KC, w0 - 1 + kw, h0 - 1, n);
          } else {
            ptx::tma_load_4d(st, &tm_x, fb, ck * KC, w0 - 1, h0 - 1, n);
          }
        }
        if constexpr (EPI == 0) {
          if (ok && p.stats >= 2) {  // the y2 tile of this output tile, for the epilogue group that owns it
            if (!ptx::mbar_wait(&yempty[yr.s], yr.ph ^ 1, abort_flag)) break;
            ptx::mbar_expect_tx(&yfull[yr.s], kTW * kTH * 128);
            ptx::tma_load_4d(ybuf + yr.s * 16384, &tm_y2, &yfull[yr.s], (int)at.nt * 64, w0, h0, n);
            yr.next(kYSlots);
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    constexpr uint32_t idesc = ptx::idesc_bf16(128, UF ? G : 3 * G, 0, MIR);
    const uint64_t a_hi = ptx::sdesc(0, 16, (UF == 2 ? 10 : 8) * kARow, kALayout);  // UF 2: next 8-pixel group = next box row
    const uint64_t b_hi = MIR ? ptx::sdesc(0, KC * 128, 1024, 2) : ptx::sdesc(0, 16, 8 * kARow, kALayout);
    const uint32_t w16 = ptx::smem_u32(wres) >> 4;
    if (ptx::elect_one()) {
      Ring rg;
      uint32_t tl = 0;
      bool ok = blockIdx.x >= p.total_tiles || ptx::mbar_wait(wfull, 0, abort_flag);
      for (int t = blockIdx.x; ok && t < p.total_tiles; t += gridDim.x, ++tl) {
        const uint32_t acc = tl % kAccs, aph = (tl / kAccs) & 1;
        if (!ptx::mbar_wait(&tempty[acc], aph ^ 1, abort_flag)) break;
        ptx::tc_fence_after();
        const uint32_t d = tmem_base + acc * kAccStride;
        for (int ck = 0; ck < p.kchunks; ++ck, rg.next(p.stages)) {
          if (!ptx::mbar_wait(XF ? &xfull[rg.s] : &full[rg.s], rg.ph, abort_flag)) { ok = false; break; }
          ptx::tc_fence_after();
          const uint32_t a16 = (ptx::smem_u32(smem) + rg.s * kABytes) >> 4;
          if constexpr (UF) {  // one instruction per tap and 16 input channels; tap (kh, kw) reads the mirrored weight tile
#pragma unroll
            for (int kh = 0; kh < 3; ++kh)
#pragma unroll
              for (int kw = 0; kw < 3; ++kw)
#pragma unroll
                for (int k = 0; k < KC / 16; ++k) {
                  const uint64_t ad = UF == 2 ? a_hi | (uint64_t)(a16 + ((kh * 10 + kw) * kARow >> 4) + k * 2)
                                              : a_hi | (uint64_t)(a16 + kw * (kBox >> 4) + kh * (16 * kARow >> 4) + k * 2);
                  const uint64_t bd = b_hi | (uint64_t)(w16 + (2 - kh) * (kWTile >> 4) + (2 - kw) * (KC * 128 >> 4) + k * 128);
                  ptx::mma_f16(d, ad, bd, idesc, (kh | kw | k) != 0);
                }
          } else {
#pragma unroll
            for (int kh = 0; kh < 3; ++kh)
#pragma unroll
              for (int k = 0; k < KC / 16; ++k) {
                const uint64_t ad = a_hi | (uint64_t)(a16 + kh * (16 * kARow >> 4) + k * 2);
                const uint64_t bd = MIR ? b_hi | (uint64_t)(w16 + (2 - kh) * (kWTile >> 4) + k * 128)   // mirrored row tap, 16 f rows on
                                        : b_hi | (uint64_t)(w16 + (ck * 3 + kh) * (kWTile >> 4) + k * 2);
                ptx::mma_f16(d, ad, bd, idesc, (ck | kh | k) != 0);
              }
          }
          ptx::mma_commit(&empty[rg.s]);
        }
        if (ok) ptx::mma_commit(&tfull[acc]);
      }
    }
    __syncwarp();
  } else if (XF && warp >= kFoldThreads / 32) {
    // normalisation warps: a thread owns one 16-byte channel chunk (8 channels) of one box column and walks the 10 rows.
    // The tile's own 14 x 8 pixels of a leave through a TMA store: the threads copy them from registers into a dense staging
    // tile (three in rotation) and one thread issues the store, so no global store instruction runs in these warps.
    const int xt = (threadIdx.x - kFoldThreads) & 127, xgrp = (threadIdx.x - kFoldThreads) >> 7;  // group xgrp takes the stages it % kXfGroups == xgrp
    constexpr int kXg = 1, kRows = 10, xg = 0;
    uint8_t* const stg_x = stg + xgrp * 3 * kAStg;
    const int j = xt & 7, col = xt >> 3;                   // logical chunk, box column (0..15)
    const uint32_t off0 = (uint32_t)col * 128 + (uint32_t)((j ^ (col & 7)) * 16);  // 128-byte swizzle: the row's low bits are col's
    uint32_t it = 0;
    Ring rg;
    float sc[8], sh[8];
    int coef_ck = -1;  // channel chunk whose coefficients the registers hold
    bool go = true;
    for (int t = blockIdx.x; go && t < p.total_tiles; t += gridDim.x) {
      const TileAt at = tile_at(t, p.tg);
      const int w0 = at.w * 14, h0 = at.h * 8, n = at.n;
      const int w = w0 - 1 + col;
      const bool w_in = w >= 0 && w < p.W, w_own = col >= 1 && col <= 14;
      for (int ck = 0; ck < p.kchunks; ++ck, ++it, rg.next(p.stages)) {
        if ((int)(it % kXfGroups) != xgrp) continue;
        const uint32_t jt = it / kXfGroups;  // this group's iteration count
        const int s = rg.s;
        const uint32_t ph = rg.ph;
        if (ck != coef_ck) {
          coef_ck = ck;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            sc[i] = __ldg(p.xf_scale + ck * 64 + j * 8 + i);
            sh[i] = __ldg(p.xf_shift + ck * 64 + j * 8 + i);
          }
        }
        const bool ok = ptx::mbar_wait(&full[s], ph, abort_flag);
        const uint32_t astg = ptx::smem_u32(stg_x) + (jt % 3) * kAStg;
        if (ok) {
          const uint32_t box = ptx::smem_u32(smem + (size_t)s * kABytes) + off0 + xg * 2048;
          // all rows are loaded first, then normalised, then stored: the loads overlap instead of queueing behind stores
          uint4 q[kRows];
#pragma unroll
          for (int i = 0; i < kRows; ++i) q[i] = ptx::lds128(box + i * kXg * 2048);
#pragma unroll
          for (int i = 0; i < kRows; ++i) {
            const int h = h0 - 1 + i * kXg + xg;
            const uint32_t qw[4] = {q[i].x, q[i].y, q[i].z, q[i].w};
            uint32_t ow[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float a0 = fmaxf(fmaf(__uint_as_float(qw[e] << 16), sc[2 * e], sh[2 * e]), 0.f);
              const float a1 = fmaxf(fmaf(__uint_as_float(qw[e] & 0xffff0000u), sc[2 * e + 1], sh[2 * e + 1]), 0.f);
              const __nv_bfloat162 b2 = __floats2bfloat162_rn(a0, a1);
              ow[e] = *reinterpret_cast<const uint32_t*>(&b2);
            }
            const bool in = w_in && h >= 0 && h < p.H;
            q[i] = in ? make_uint4(ow[0], ow[1], ow[2], ow[3]) : make_uint4(0u, 0u, 0u, 0u);
            ptx::sts128(box + i * kXg * 2048, q[i]);
          }
          if (w_own) {  // box rows 1..8 x columns 1..14 are the tile's own pixels: dense rows of the staging tile, same swizzle
#pragma unroll
            for (int i = 1; i <= 8; ++i) {
              const uint32_t orow = (uint32_t)((i - 1) * 14 + col - 1);
              ptx::sts128(astg + orow * 128 + ((j ^ (orow & 7)) * 16), q[i]);
            }
          }
          ptx::fence_async_smem();  // the tensor core and the TMA store read shared memory through the async proxy
          ptx::mbar_arrive(&xfull[s]);
        }
        // one thread decides for all 128 whether to go on, so nobody is left alone at the barrier
        if (xt == 0) xf_go[xgrp * 2 + (jt & 1)] = ok && !*abort_flag ? 1 : 0;
        ptx::named_barrier(3 + xgrp, 128);
        if (!xf_go[xgrp * 2 + (jt & 1)]) { go = false; break; }
        if (xt == 0) {
          ptx::tma_store_4d(&tm_y, reinterpret_cast<const void*>(stg_x + (jt % 3) * kAStg), ck * 64, w0, h0, n);
          ptx::tma_store_commit();
          ptx::tma_store_wait_read_but_one();  // the store before this one has read its tile: the tile after next may be written
        }
      }
    }
    if (xt == 0) ptx::tma_store_wait_all();
  } else {
    // two epilogue groups of 128 threads; group g owns accumulator g and takes every second tile of the CTA
    const int grp = (threadIdx.x - 64) >> 7;
    const int et = (threadIdx.x - 64) & 127;
    uint8_t* const stg_g = stg + grp * 16384;
    const int lg = warp & 3;
    const int r = lg * 32 + lane;            // TMEM lane = extended-tile pixel (we = r % 16, h = r / 16)
    const int we = r & 15, hh = r >> 4;
    const bool valid = UF || (we >= 1 && we <= 14);
    const int orow = UF ? r : (we - 1) + 14 * hh;  // row of the output staging tile
    // statistics: a thread owns 8 channels (one 16-byte chunk of a pixel row) and the 7 rows rg, rg+16, ...
    const int schunk = et & 7, srg = et >> 3;
    float s1[8], s2[8], bsc[8], bsh[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) s1[i] = s2[i] = bsc[i] = bsh[i] = 0.f;
    if constexpr (EPI == 0) {
      if (p.stats >= 2) {
        const int ch = (int)(blockIdx.x % p.n_tiles) * 64 + schunk * 8;
#pragma unroll
        for (int i = 0; i < 8; ++i) { bsc[i] = p.bn_scale[ch + i]; bsh[i] = p.bn_shift[ch + i]; }
        if (p.stats == 4) {  // s1, s2 hold the per-channel constants of dy = scale*dz + s1*y + s2 instead of running sums
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float sc = bsc[i], m1 = p.bn_sdz[ch + i] * p.inv_m, m2 = p.bn_sdzx[ch + i] * p.inv_m, is = p.bn_invstd[ch + i];
            s1[i] = -sc * m2 * is;
            s2[i] = sc * (m2 * is * p.bn_mu[ch + i] - m1);
          }
        }
      }
    }
    uint32_t tl = grp;
    for (int t = blockIdx.x + grp * gridDim.x; t < p.total_tiles; t += 2 * gridDim.x, tl += 2) {
      const TileAt at = tile_at(t, p.tg);
      const int nt = at.nt, w0 = at.w * kTW, h0 = at.h * kTH, n = at.n;
      const uint32_t acc = tl % kAccs, aph = (tl / kAccs) & 1;
      ptx::mbar_wait(&tfull[acc], aph, abort_flag);
      ptx::tc_fence_after();
      if (et == 0) {
        if constexpr (EPI == 0) ptx::tma_store_wait_read();
        epi_go[grp] = *abort_flag ? 0 : 1;
      }
      ptx::named_barrier(1 + grp, 128);
      if (!epi_go[grp]) break;
      // a last tile column may reach beyond the image (widths that are not multiples of 14): those pixels are stored as
      // zeros in the staging tile (they add nothing to the statistics; the TMA store clips them) and never written directly
      const bool vcol = valid && (UF || w0 + we - 1 < p.W);
      const uint32_t tbase = tmem_base + ((uint32_t)(lg * 32) << 16) + acc * kAccStride;
      bf16* gdst = EPI == 1 ? p.out + (((size_t)n * p.H + h0 + hh) * p.W + w0 + we - 1) * p.Cout : nullptr;
      // 16 output channels at a time; the next 16 are on their way from tensor memory while these are added and stored
      uint32_t t0[2][16], t1[2][16], t2[2][16];
      auto fetch = [&](int q, uint32_t (&a0)[16], uint32_t (&a1)[16], uint32_t (&a2)[16]) {
        if constexpr (UF) {
          ptx::tmem_ld16(tbase + q * 16, a1);
        } else {
          ptx::tmem_ld16(tbase + (MIR ? 2 * G : 0) + q * 16, a0);  // group feeding the pixel on the left
          ptx::tmem_ld16(tbase + G + q * 16, a1);
          ptx::tmem_ld16(tbase + (MIR ? 0 : 2 * G) + q * 16, a2);  // group feeding the pixel on the right
        }
      };
      fetch(0, t0[0], t1[0], t2[0]);
#pragma unroll
      for (int q = 0; q < G / 16; ++q) {
        uint32_t (&v0)[16] = t0[q & 1];
        uint32_t (&v1)[16] = t1[q & 1];
        uint32_t (&v2)[16] = t2[q & 1];
        ptx::tmem_ld_wait();
        if (q + 1 < G / 16) fetch(q + 1, t0[(q + 1) & 1], t1[(q + 1) & 1], t2[(q + 1) & 1]);
        uint32_t w[8];
        if constexpr (UF) {
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(v1[2 * e]), __uint_as_float(v1[2 * e + 1]));
            w[e] = *reinterpret_cast<const uint32_t*>(&b2);
          }
        } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          float o[2];
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2) {
            const int c = 2 * e + h2;
            const float left = __shfl_up_sync(0xffffffffu, __uint_as_float(v0[c]), 1);     // kw = 0 term of pixel w-1
            const float right = __shfl_down_sync(0xffffffffu, __uint_as_float(v2[c]), 1);  // kw = 2 term of pixel w+1
            o[h2] = left + __uint_as_float(v1[c]) + right;
            if constexpr (EPI == 1) {
              const int ch = q * 16 + c;
              o[h2] = ch < p.Cout ? fmaxf(o[h2] + p.bias[ch], 0.f) : 0.f;
            } else {
              if (p.bias) o[h2] = fmaxf(o[h2] + __ldg(p.bias + nt * 64 + q * 16 + c), 0.f);
            }
          }
          const __nv_bfloat162 b2 = __floats2bfloat162_rn(o[0], o[1]);
          w[e] = *reinterpret_cast<const uint32_t*>(&b2);
        }
        }
        if constexpr (EPI == 0) {
          if constexpr (POST) {
            const float2* ps = reinterpret_cast<const float2*>(p.bn_scale + nt * 64 + q * 16);
            const float2* ph = reinterpret_cast<const float2*>(p.bn_shift + nt * 64 + q * 16);
#pragma unroll
            for (int e = 0; e < 8; ++e) w[e] = bn_relu2(w[e], __ldg(ps + e), __ldg(ph + e));
          }
          if (valid) {
            uint8_t* dst = stg_g + orow * 128;
            *reinterpret_cast<uint4*>(dst + (((2 * q) ^ (orow & 7)) * 16)) = vcol ? make_uint4(w[0], w[1], w[2], w[3]) : make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4*>(dst + (((2 * q + 1) ^ (orow & 7)) * 16)) = vcol ? make_uint4(w[4], w[5], w[6], w[7]) : make_uint4(0u, 0u, 0u, 0u);
          }
        } else if (p.pool_part) {
          // h stays in registers: its sign bits go to the mask, its sum over the warp's 32 pixels (halo pixels count as
          // zero) to the pooling partials.  The 16 channel sums are formed by a reduce-scatter over the lanes: each step
          // halves the channels a lane carries and doubles the pixels its sums cover (16 shuffles for 16 channels); the
          // lane pair (2j, 2j+1) ends with the sum of channel j's bit pattern below.
          const int c0 = q * 16;
          float ov[16];
          uint32_t bits = 0;
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float lo = __uint_as_float(w[e] << 16), hi = __uint_as_float(w[e] & 0xffff0000u);
            ov[2 * e] = vcol ? lo : 0.f;
            ov[2 * e + 1] = vcol ? hi : 0.f;
            bits |= (lo > 0.f ? 1u : 0u) << (2 * e);
            bits |= (hi > 0.f ? 1u : 0u) << (2 * e + 1);
          }
          if (vcol && c0 < p.Cout) {
            uint8_t* mdst = p.mask + ((((size_t)n * p.H + h0 + hh) * p.W + w0 + we - 1) * (size_t)(p.Cout >> 3)) + (c0 >> 3);
            mdst[0] = (uint8_t)(bits & 0xffu);
            if (c0 + 8 < p.Cout) mdst[1] = (uint8_t)(bits >> 8);
          }
          float r8[8], r4[4], r2[2];
          const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float send = b4 ? ov[i] : ov[8 + i], keep = b4 ? ov[8 + i] : ov[i];
            r8[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float send = b3 ? r8[i] : r8[4 + i], keep = b3 ? r8[4 + i] : r8[i];
            r4[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float send = b2 ? r4[i] : r4[2 + i], keep = b2 ? r4[2 + i] : r4[i];
            r2[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
          }
          float r1 = (b1 ? r2[1] : r2[0]) + __shfl_xor_sync(0xffffffffu, b1 ? r2[0] : r2[1], 2);
          r1 += __shfl_xor_sync(0xffffffffu, r1, 1);
          const int ch = c0 + (b4 ? 8 : 0) + (b3 ? 4 : 0) + (b2 ? 2 : 0) + (b1 ? 1 : 0);
          if ((lane & 1) == 0 && ch < p.Cout) p.pool_part[((size_t)t * 4 + lg) * p.Cout + ch] = r1;
        } else {
          const int c0 = q * 16;             // Cout is a multiple of 8 here
          if (vcol && c0 < p.Cout) {
            *reinterpret_cast<uint4*>(gdst + c0) = make_uint4(w[0], w[1], w[2], w[3]);
            if (c0 + 8 < p.Cout) *reinterpret_cast<uint4*>(gdst + c0 + 8) = make_uint4(w[4], w[5], w[6], w[7]);
          }
        }
      }
      ptx::tc_fence_before();
      ptx::mbar_arrive(&tempty[acc]);
      if constexpr (EPI == 0) {
        ptx::fence_async_smem();
        ptx::named_barrier(1 + grp, 128);
        if (p.stats == 4) {
          // second pass: the staged da tile becomes dy in place (thread <-> 8 channels x 7 or 8 rows, as for the sums)
          const uint32_t slot = tl % kYSlots;
          ptx::mbar_wait(&yfull[slot], (tl / kYSlots) & 1, abort_flag);
          const uint8_t* yb = ybuf + slot * 16384;
#pragma unroll
          for (int rr = 0; rr < kStatIters; ++rr) {
            const int row = srg + 16 * rr;
            const int off = row * 128 + ((schunk ^ (row & 7)) * 16);
            const uint4 dq = *reinterpret_cast<const uint4*>(stg_g + off);
            const uint4 yq = *reinterpret_cast<const uint4*>(yb + off);
            const uint32_t dw[4] = {dq.x, dq.y, dq.z, dq.w}, yw[4] = {yq.x, yq.y, yq.z, yq.w};
            uint32_t ow[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float d0 = __uint_as_float(dw[e] << 16), d1 = __uint_as_float(dw[e] & 0xffff0000u);
              const float y0 = __uint_as_float(yw[e] << 16), y1 = __uint_as_float(yw[e] & 0xffff0000u);
              const float z0 = fmaf(y0, bsc[2 * e], bsh[2 * e]) > 0.f ? d0 : 0.f;
              const float z1 = fmaf(y1, bsc[2 * e + 1], bsh[2 * e + 1]) > 0.f ? d1 : 0.f;
              const float o0 = fmaf(bsc[2 * e], z0, fmaf(s1[2 * e], y0, s2[2 * e]));
              const float o1 = fmaf(bsc[2 * e + 1], z1, fmaf(s1[2 * e + 1], y1, s2[2 * e + 1]));
              const __nv_bfloat162 b2 = __floats2bfloat162_rn(o0, o1);
              ow[e] = *reinterpret_cast<const uint32_t*>(&b2);
            }
            *reinterpret_cast<uint4*>(stg_g + off) = make_uint4(ow[0], ow[1], ow[2], ow[3]);
          }
          ptx::mbar_release_read(&yempty[slot]);
          ptx::fence_async_smem();
          ptx::named_barrier(1 + grp, 128);
        }
        if (et == 0 && p.stats != 3) {
          ptx::tma_store_4d(&tm_y, stg_g, nt * 64, w0, h0, n);
          ptx::tma_store_commit();
        }
        if (p.stats == 2 || p.stats == 3) {
          // sums of dz and dz*y2 (the caller of the kernel gets sum dz*xhat = invstd * (sum dz*y2 - mu * sum dz))
          const uint32_t slot = tl % kYSlots;
          ptx::mbar_wait(&yfull[slot], (tl / kYSlots) & 1, abort_flag);
          const uint8_t* yb = ybuf + slot * 16384;
#pragma unroll
          for (int rr = 0; rr < kStatIters; ++rr) {
            const int row = srg + 16 * rr;
            const int off = row * 128 + ((schunk ^ (row & 7)) * 16);
            const uint4 dq = *reinterpret_cast<const uint4*>(stg_g + off);
            const uint4 yq = *reinterpret_cast<const uint4*>(yb + off);
            const uint32_t dw[4] = {dq.x, dq.y, dq.z, dq.w}, yw[4] = {yq.x, yq.y, yq.z, yq.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float d0 = __uint_as_float(dw[e] << 16), d1 = __uint_as_float(dw[e] & 0xffff0000u);
              const float y0 = __uint_as_float(yw[e] << 16), y1 = __uint_as_float(yw[e] & 0xffff0000u);
              const float z0 = fmaf(y0, bsc[2 * e], bsh[2 * e]) > 0.f ? d0 : 0.f;
              const float z1 = fmaf(y1, bsc[2 * e + 1], bsh[2 * e + 1]) > 0.f ? d1 : 0.f;
              s1[2 * e] += z0;
              s1[2 * e + 1] += z1;
              s2[2 * e] = fmaf(z0, y0, s2[2 * e]);
              s2[2 * e + 1] = fmaf(z1, y1, s2[2 * e + 1]);
            }
          }
          ptx::mbar_release_read(&yempty[slot]);
        } else if (p.stats == 1) {
#pragma unroll
          for (int rr = 0; rr < kStatIters; ++rr) {
            const int row = srg + 16 * rr;
            const uint4 vq = *reinterpret_cast<const uint4*>(stg_g + row * 128 + ((schunk ^ (row & 7)) * 16));
            const uint32_t vw[4] = {vq.x, vq.y, vq.z, vq.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float v0 = __uint_as_float(vw[e] << 16), v1 = __uint_as_float(vw[e] & 0xffff0000u);
              s1[2 * e] += v0;
              s1[2 * e + 1] += v1;
              s2[2 * e] = fmaf(v0, v0, s2[2 * e]);
              s2[2 * e + 1] = fmaf(v1, v1, s2[2 * e + 1]);
            }
          }
        }
      }
    }
    if constexpr (EPI == 0) {
      if (et == 0) ptx::tma_store_wait_all();
      if (p.stats && p.stats != 4) {
        // one partial per epilogue group: lanes with the same chunk (lane & 7) are added by shuffles, the group's four warps
        // through the (now idle) staging tile, all in a fixed order
        fold_group_partial(s1, s2, reinterpret_cast<float*>(stg_g), grp, lg, lane, p.stats >= 2, p.bn_mu, p.bn_invstd,
                           (int)(blockIdx.x % p.n_tiles) * 64, p.red + ((size_t)(blockIdx.x / p.n_tiles) * 2 + grp) * 2 * p.Cout, p.Cout);
      }
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(p.status, NF_ETIMEOUT);
    const unsigned long long t0 = ptx::globaltimer();
    while (ptx::globaltimer() - t0 < 2000000ull) __nanosleep(1000);
  }
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, kTmemCols);
  }
}

// ---------------------------------------------------------------- aux input gradient, 256 pixels per instruction
// The narrow input gradient da = dh (*) Wa^T (K = F <= 32 per tap) is bound by the NUMBER of its K = 16 instructions: up to 64 columns
// an instruction takes about 40 cycles, the time to read its operands, whatever its width.  With the pixels on the M side an instruction covers
// 128 of them; here the operands are swapped: A = the mirrored weight tile of a tap, [64 output channels] x [16 f] (M = 64,
// MN-major as stored), B = 256 pixels x [16 f] of the dh box (N = 256, K-major), so the nine taps of a 256-pixel tile are nine
// instructions instead of eighteen.  A tile is 8 columns x 32 rows; ONE 10 x 34-pixel box feeds all taps (a tap is a start
// address kh * 10 + kw pixels into the box, an image row of the tile is one 8-row group, pitch 10 pixels: the swizzle is a
// function of the address).  The accumulator holds D[channel][pixel]: with M = 64, channel c sits in lane 32 * (c / 16) + c % 16,
// so warp q of an epilogue group reads channels 16q .. 16q+15 in lanes 0..15 of its quadrant as accumulator fragments and
// transposes them into the pixel-major staging tile with transposing matrix stores (16 bytes = 8 channels per pixel and store row).
// From there on everything is as in the folded kernel: BatchNorm-backward sums (stats 2, 3), the second pass that turns the
// tile into dy (stats 4), TMA store (not for stats 3).  Needs W % 8 == 0 and H % 16 == 0 (a last tile row of 16 image rows: the
// box rows below the image load as zeros, the store is clipped, the sums skip them); one 64-channel output tile per CTA.
constexpr int kWideThreads = 320;
constexpr int kWideYSlots = 3;

template <int KC>
__global__ void __launch_bounds__(kWideThreads, 1)
aux_dgrad_wide_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                      const __grid_constant__ CUtensorMap tm_y, const __grid_constant__ CUtensorMap tm_y2, const FoldParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr int kARow = KC * 2;                                    // bytes of one pixel of the dh box
  constexpr uint32_t kALayout = KC == 32 ? 4 : 6;
  constexpr int kBox = 34 * 10 * kARow;                            // (32+2) rows x (8+2) pixels
  constexpr int kStage = (kBox + 1023) / 1024 * 1024;
  constexpr int kWTile = 3 * KC * 128;                             // one kernel row: [kw][f][64 c]
  constexpr int kTile = 256 * 128;                                 // 256 pixels x 64 channels bf16
  uint8_t* wres = smem + (size_t)p.stages * kStage;
  uint8_t* stg = wres + 3 * kWTile;                                // one staging tile per epilogue group
  uint8_t* ybuf = stg + 2 * kTile;                                 // stats >= 2: kWideYSlots tiles of y2
  uint64_t* bars = reinterpret_cast<uint64_t*>(ybuf + (p.stats >= 2 ? kWideYSlots : 0) * kTile);
  uint64_t* full = bars;
  uint64_t* empty = bars + kMaxStages;
  uint64_t* tfull = bars + 2 * kMaxStages;
  uint64_t* tempty = tfull + 2;
  uint64_t* wfull = tempty + 2;
  uint64_t* yfull = wfull + 1;
  uint64_t* yempty = yfull + kWideYSlots;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(yempty + kWideYSlots);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* epi_go = reinterpret_cast<volatile int*>(tmem_slot + 2);
  constexpr uint32_t kTmemCols = 512;                              // two accumulators of 256 columns

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      ptx::mbar_init(&tfull[a], 1);
      ptx::mbar_init(&tempty[a], 128);
    }
    for (int a = 0; a < kWideYSlots; ++a) {
      ptx::mbar_init(&yfull[a], 1);
      ptx::mbar_init(&yempty[a], 128);
    }
    ptx::mbar_init(wfull, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(&tm_x);
    ptx::prefetch_tmap(&tm_w);
    ptx::prefetch_tmap(&tm_y);
    ptx::prefetch_tmap(&tm_y2);
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  nf_pdl_begin();  // everything above touches only this CTA and overlaps the previous kernel

  if (warp == 0) {
    // ---------------- producer: the CTA's weights once, then per tile one dh box and (stats >= 2) the y2 tile
    if (ptx::elect_one()) {
      if (blockIdx.x < p.total_tiles) {
        ptx::mbar_expect_tx(wfull, (uint32_t)(3 * kWTile));
#pragma unroll
        for (int kh = 0; kh < 3; ++kh) ptx::tma_load_4d(wres + kh * kWTile, &tm_w, wfull, (int)(blockIdx.x % p.n_tiles) * 64, 0, 0, kh);
      }
      Ring rg, yr;
      for (int t = blockIdx.x; t < p.total_tiles; t += gridDim.x, rg.next(p.stages)) {
        const TileAt at = tile_at(t, p.tg);
        const int w0 = at.w * 8, h0 = at.h * 32, n = at.n;
        if (!ptx::mbar_wait(&empty[rg.s], rg.ph ^ 1, abort_flag)) break;
        ptx::mbar_expect_tx(&full[rg.s], (uint32_t)kBox);
        ptx::tma_load_4d(smem + (size_t)rg.s * kStage, &tm_x, &full[rg.s], 0, w0 - 1, h0 - 1, n);
        if (p.stats >= 2) {
          if (!ptx::mbar_wait(&yempty[yr.s], yr.ph ^ 1, abort_flag)) break;
          ptx::mbar_expect_tx(&yfull[yr.s], (uint32_t)kTile);
          ptx::tma_load_4d(ybuf + yr.s * kTile, &tm_y2, &yfull[yr.s], (int)at.nt * 64, w0, h0, n);
          yr.next(kWideYSlots);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- issuer: nine instructions per tile, D[channel][pixel] += Wa_mirrored(tap)[channel][f] * dh[pixel + tap][f]
    constexpr uint32_t idesc = ptx::idesc_bf16(64, 256, 1, 0);
    const uint64_t a_hi = ptx::sdesc(0, KC * 128, 1024, 2);          // weight tile of a tap: [f][64 c], MN-major
    const uint64_t b_hi = ptx::sdesc(0, 16, 10 * kARow, kALayout);   // pixels: next 8-pixel group = next box row
    const uint32_t w16 = ptx::smem_u32(wres) >> 4;
    if (ptx::elect_one()) {
      Ring rg;
      uint32_t tl = 0;
      const bool ok = blockIdx.x >= p.total_tiles || ptx::mbar_wait(wfull, 0, abort_flag);
      for (int t = blockIdx.x; ok && t < p.total_tiles; t += gridDim.x, ++tl, rg.next(p.stages)) {
        const uint32_t acc = tl & 1, aph = (tl >> 1) & 1;
        if (!ptx::mbar_wait(&tempty[acc], aph ^ 1, abort_flag)) break;
        ptx::tc_fence_after();
        if (!ptx::mbar_wait(&full[rg.s], rg.ph, abort_flag)) break;
        ptx::tc_fence_after();
        const uint32_t d = tmem_base + acc * 256;
        const uint32_t x16 = (ptx::smem_u32(smem) + rg.s * kStage) >> 4;
#pragma unroll
        for (int kh = 0; kh < 3; ++kh)
#pragma unroll
          for (int kw = 0; kw < 3; ++kw)
#pragma unroll
            for (int k = 0; k < KC / 16; ++k) {
              const uint64_t ad = a_hi | (uint64_t)(w16 + (2 - kh) * (kWTile >> 4) + (2 - kw) * (KC * 128 >> 4) + k * 128);
              const uint64_t bd = b_hi | (uint64_t)(x16 + ((kh * 10 + kw) * kARow >> 4) + k * 2);
              ptx::mma_f16(d, ad, bd, idesc, (kh | kw | k) != 0);
            }
        ptx::mma_commit(&empty[rg.s]);
        ptx::mma_commit(&tfull[acc]);
      }
    }
    __syncwarp();
  } else {
    // ---------------- two epilogue groups of 128 threads; group g takes the tiles tl = g, g + 2, ... (accumulator g)
    const int grp = (threadIdx.x - 64) >> 7;
    const int et = (threadIdx.x - 64) & 127;
    uint8_t* const stg_g = stg + grp * kTile;
    const int lg = warp & 3;                     // lane quadrant of tensor memory: channels 16*lg .. 16*lg + 15 in lanes 0..15
    // sums / second pass: a thread owns 8 channels (one 16-byte chunk) and the 16 rows srg, srg + 16, ... of the 256
    const int schunk = et & 7, srg = et >> 3;
    float s1[8], s2[8], bsc[8], bsh[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) s1[i] = s2[i] = bsc[i] = bsh[i] = 0.f;
    if (p.stats >= 2) {
      const int c0 = (int)(blockIdx.x % p.n_tiles) * 64 + schunk * 8;
#pragma unroll
      for (int i = 0; i < 8; ++i) { bsc[i] = p.bn_scale[c0 + i]; bsh[i] = p.bn_shift[c0 + i]; }
      if (p.stats == 4) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float sc = bsc[i], m1 = p.bn_sdz[c0 + i] * p.inv_m, m2 = p.bn_sdzx[c0 + i] * p.inv_m, is = p.bn_invstd[c0 + i];
          s1[i] = -sc * m2 * is;
          s2[i] = sc * (m2 * is * p.bn_mu[c0 + i] - m1);
        }
      }
    }
    uint32_t tl = grp;
    for (int t = blockIdx.x + grp * gridDim.x; t < p.total_tiles; t += 2 * gridDim.x, tl += 2) {
      const TileAt at = tile_at(t, p.tg);
      const int nt = at.nt, w0 = at.w * 8, h0 = at.h * 32, n = at.n;
      const uint32_t acc = grp, aph = (tl >> 1) & 1;
      ptx::mbar_wait(&tfull[acc], aph, abort_flag);
      ptx::tc_fence_after();
      if (et == 0) {
        ptx::tma_store_wait_read();              // the previous store of this group has read the staging tile
        epi_go[grp] = *abort_flag ? 0 : 1;
      }
      ptx::named_barrier(1 + grp, 128);
      if (!epi_go[grp]) break;
      const uint32_t tbase = tmem_base + ((uint32_t)(lg * 32) << 16) + acc * 256;
      // Transpose through the matrix-store instruction: a fragment load hands thread i channel i / 4 (and i / 4 + 8) of the
      // warp's 16 with two neighbouring pixels; as bfloat16 pairs these are the column fragments of 8 x 8 matrices whose
      // transposed store writes, per pixel, the 8 channels of a chunk as 16 contiguous bytes of the pixel-major tile.
      const uint32_t sbase = ptx::smem_u32(stg_g);
      const int mrow = lane & 7, mat = lane >> 3;                       // this thread addresses row mrow of matrix mat
      const uint32_t mchunk = (uint32_t)(2 * lg + (mat & 1));           // matrices 0, 2: channels 16 lg + 0..7; 1, 3: + 8..15
#pragma unroll 4
      for (int j = 0; j < 16; ++j) {             // 16 pixels at a time
        uint32_t v[8];
        ptx::tmem_ld_16x256b_x2(tbase + j * 16, v);
        ptx::tmem_ld_wait();
        uint32_t r[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {            // r[0]: ch 0-7, px 0-7; r[1]: ch 8-15, px 0-7; r[2], r[3]: px 8-15
          const __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(v[2 * q]), __uint_as_float(v[2 * q + 1]));
          r[q] = *reinterpret_cast<const uint32_t*>(&b2);
        }
        const uint32_t px = (uint32_t)(j * 16 + (mat >> 1) * 8 + mrow);
        ptx::stmatrix_x4_trans(sbase + px * 128 + ((mchunk ^ (px & 7)) * 16), r[0], r[1], r[2], r[3]);
      }
      ptx::tc_fence_before();
      ptx::mbar_arrive(&tempty[acc]);
      ptx::fence_async_smem();
      ptx::named_barrier(1 + grp, 128);
      const uint32_t slot = tl % kWideYSlots;
      if (p.stats == 4) {
        ptx::mbar_wait(&yfull[slot], (tl / kWideYSlots) & 1, abort_flag);
        const uint8_t* yb = ybuf + slot * kTile;
#pragma unroll 4
        for (int rr = 0; rr < 16; ++rr) {
          const int row = srg + 16 * rr;
          const int off = row * 128 + ((schunk ^ (row & 7)) * 16);
          const uint4 dq = *reinterpret_cast<const uint4*>(stg_g + off);
          const uint4 yq = *reinterpret_cast<const uint4*>(yb + off);
          const uint32_t dw[4] = {dq.x, dq.y, dq.z, dq.w}, yw[4] = {yq.x, yq.y, yq.z, yq.w};
          uint32_t ow[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float d0 = __uint_as_float(dw[e] << 16), d1 = __uint_as_float(dw[e] & 0xffff0000u);
            const float y0 = __uint_as_float(yw[e] << 16), y1 = __uint_as_float(yw[e] & 0xffff0000u);
            const float z0 = fmaf(y0, bsc[2 * e], bsh[2 * e]) > 0.f ? d0 : 0.f;
            const float z1 = fmaf(y1, bsc[2 * e + 1], bsh[2 * e + 1]) > 0.f ? d1 : 0.f;
            const float o0 = fmaf(bsc[2 * e], z0, fmaf(s1[2 * e], y0, s2[2 * e]));
            const float o1 = fmaf(bsc[2 * e + 1], z1, fmaf(s1[2 * e + 1], y1, s2[2 * e + 1]));
            const __nv_bfloat162 b2 = __floats2bfloat162_rn(o0, o1);
            ow[e] = *reinterpret_cast<const uint32_t*>(&b2);
          }
          *reinterpret_cast<uint4*>(stg_g + off) = make_uint4(ow[0], ow[1], ow[2], ow[3]);
        }
        ptx::mbar_release_read(&yempty[slot]);
        ptx::fence_async_smem();
        ptx::named_barrier(1 + grp, 128);
      }
      if (et == 0 && p.stats != 3) {
        ptx::tma_store_4d(&tm_y, stg_g, nt * 64, w0, h0, n);
        ptx::tma_store_commit();
      }
      if (p.stats == 2 || p.stats == 3) {
        ptx::mbar_wait(&yfull[slot], (tl / kWideYSlots) & 1, abort_flag);
        const uint8_t* yb = ybuf + slot * kTile;
#pragma unroll 4
        for (int rr = 0; rr < 16; ++rr) {
          const int row = srg + 16 * rr;
          const bool rv = h0 + (row >> 3) < p.H;  // a last tile row may reach below the image: those pixels count for nothing
          const int off = row * 128 + ((schunk ^ (row & 7)) * 16);
          const uint4 dq = *reinterpret_cast<const uint4*>(stg_g + off);
          const uint4 yq = *reinterpret_cast<const uint4*>(yb + off);
          const uint32_t dw[4] = {dq.x, dq.y, dq.z, dq.w}, yw[4] = {yq.x, yq.y, yq.z, yq.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float d0 = __uint_as_float(dw[e] << 16), d1 = __uint_as_float(dw[e] & 0xffff0000u);
            const float y0 = __uint_as_float(yw[e] << 16), y1 = __uint_as_float(yw[e] & 0xffff0000u);
            const float z0 = rv && fmaf(y0, bsc[2 * e], bsh[2 * e]) > 0.f ? d0 : 0.f;
            const float z1 = rv && fmaf(y1, bsc[2 * e + 1], bsh[2 * e + 1]) > 0.f ? d1 : 0.f;
            s1[2 * e] += z0;
            s1[2 * e + 1] += z1;
            s2[2 * e] = fmaf(z0, y0, s2[2 * e]);
            s2[2 * e + 1] = fmaf(z1, y1, s2[2 * e + 1]);
          }
        }
        ptx::mbar_release_read(&yempty[slot]);
      }
    }
    if (et == 0) ptx::tma_store_wait_all();
    if (p.stats == 2 || p.stats == 3)  // one partial per epilogue group, as in the folded kernel
      fold_group_partial(s1, s2, reinterpret_cast<float*>(stg_g), grp, lg, lane, true, p.bn_mu, p.bn_invstd,
                         (int)(blockIdx.x % p.n_tiles) * 64, p.red + ((size_t)(blockIdx.x / p.n_tiles) * 2 + grp) * 2 * p.Cout, p.Cout);
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(p.status, NF_ETIMEOUT);
    const unsigned long long t0 = ptx::globaltimer();
    while (ptx::globaltimer() - t0 < 2000000ull) __nanosleep(1000);
  }
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, kTmemCols);
  }
}

// ---------------------------------------------------------------- weight gradient
// dW[tap][co][ci] = sum over pixels of dy[pixel, co] * x[pixel shifted by tap, ci].  The K dimension of the
// GEMM is the pixel index, so both operands are MN-major in shared memory exactly as TMA delivers the
// channels-last tiles.  Work is split over (64-input-channel chunk, output-channel chunk) pairs and over
// the pixel tiles (split-K): accumulators stay in tensor memory over a CTA's whole pixel range and are
// written as per-CTA partials that a second kernel sums in a fixed order.  Two kernels: the per-tap form
// below (stride 2 and small feature maps) and conv_wgrad_kw_kernel (stride 1).
struct WgParams {
  int N, H, W, Cin, Cout;
  int BW, BH, tiles_w, tiles_h, pix_tiles, ci_chunks, co_chunks, splits, stages, stride, BI;
  TileGrid tg;
  int dy_shift;     // row form: the column tap moves the gradient (as in conv_wgrad_kw_kernel) instead of the activation
  float* part;      // [splits][9][Cout][Cin]
  int32_t* status;
};

// NB = width of the output-gradient tile in channels (64: main conv, one 64-channel chunk per CTA;
// 16/32/64: aux conv with F <= NB filters, rows of 2*NB bytes with the matching TMA swizzle).
// Per-tap form: stride-2 convolutions, and feature maps smaller than a tile where a tile
// spans BI whole images.  The shifted activation tiles are gathered by TMA, with element stride 2 for
// stride 2, one 128-pixel tile per tap; a CTA then owns one kernel row kh (grid dimension) with its three column
// taps: taps (kh,0) and (kh,1) stacked in one instruction, tap (kh,2) in a second, half-empty one.
// SEG = 1, 2 (maps that no tile divides, NB <= 64): a new pair of accumulators every SEG instructions of 16 pixels, added outside the
// tensor core, two segments to one term of a compensated fp32 sum, so that the error is one segment's and not the whole pixel
// range's.  The running sum of the tensor core loses about 2^-27 per instruction, always towards zero: over the 80 instructions of a
// CTA's range the weight gradient of 256 -> 256 channels on 61 maps of 14x14 was off by 1.9e-6 of its size, the auxiliary one by
// 5.5e-7, where the fp32 chains that such maps had before gave 8.5e-7 and 6.6e-8.  A thread holds one row's 64 sums and 64
// corrections: warps 0-3 the first accumulator of the pair, warps 4 and 5 the filled half of the second; warps 6 and 7 produce
// and issue (with 256 threads all of that stays in registers).  The sums bound this form: that stage of two layers 281 -> 342 us,
// the two gradients now off by 1.1e-7 and 6.0e-8.
// HB = 1 (maps 8 pixels wide, stride 1, no segments): the three column taps are one box of ten columns.  An image row of the tile is one
// group of eight pixels, groups lie ten pixels apart, and the second stacked tap starts one pixel further.  Same products in the same
// order as three boxes, 24 KB a tile for 52: the auxiliary gradient of 512 channels, 8 filters, 8602 maps of 8x8, which the fill of shared
// memory bound, 384 -> 324 us.
constexpr int kSegSets = 4;
constexpr int wgrad_threads(int seg) { return seg ? 256 : kThreads; }

template <int NB, int SEG, int HB>
__global__ void __launch_bounds__(wgrad_threads(SEG), 1)
conv_wgrad_tc_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_dy, const WgParams p) {
  constexpr int kAtoms = NB > 64 ? NB / 64 : 1;                // 64-channel atoms of the dy tile (NB = 128, 256: main conv only)
  constexpr int kBRow = (NB > 64 ? 64 : NB) * 2;               // bytes of one pixel row of one atom
  constexpr uint32_t kBLayout = NB >= 64 ? 2 : NB == 32 ? 4 : 6;  // swizzle of that tile
  constexpr int kBTile = 128 * kBRow;                          // one atom
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  static_assert(!SEG || NB <= 64, "a thread holds the sums of one accumulator");
  static_assert(!HB || (!SEG && NB <= 64), "one box: no segments");
  constexpr int kStages = NB > 64 ? 2 : HB ? 5 : 3;
  constexpr int kJobs = 2;  // instructions (accumulators) per 16 pixels
  constexpr int copy_bytes = HB ? 128 : 16384;  // from one column tap to the next: one pixel of the box, or a 128-pixel tile
  constexpr int x_bytes = HB ? 160 * 128 : 3 * copy_bytes;
  const int stage_bytes = x_bytes + kAtoms * 16384;  // a dy atom always gets 16 KB so the unused rows read by the
                                                            // half-empty last instruction stay inside the stage
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)kStages * stage_bytes);
  uint64_t* full = bars;
  uint64_t* empty = bars + kStages;
  uint64_t* done = bars + 2 * kStages;
  uint64_t* tfull = done + 1;    // SEG: pair of accumulators complete / taken
  uint64_t* tempty = tfull + kSegSets;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + kSegSets);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  constexpr uint32_t kNeed = kJobs * NB * (SEG ? kSegSets : 1);
  constexpr uint32_t kCols = kNeed <= 32 ? 32 : kNeed <= 64 ? 64 : kNeed <= 128 ? 128 : kNeed <= 256 ? 256 : 512;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kProducer = SEG ? 6 : 0, kIssuer = SEG ? 7 : 1;
  const int blocks = p.ci_chunks * p.co_chunks;
  const int blk = blockIdx.x % blocks;
  const int rest = blockIdx.x / blocks;
  const int khg = rest % 3;  // kernel row owned by this CTA
  const int sp = rest / 3;
  const int cic = blk % p.ci_chunks, coc = blk / p.ci_chunks;
  const int t0 = (int)((long)p.pix_tiles * sp / p.splits), t1 = (int)((long)p.pix_tiles * (sp + 1) / p.splits);

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    ptx::mbar_init(done, 1);
    for (int a = 0; a < kSegSets; ++a) {
      ptx::mbar_init(&tfull[a], 1);
      ptx::mbar_init(&tempty[a], 192);
    }
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(&tm_x);
    ptx::prefetch_tmap(&tm_dy);
  }
  if (warp == kIssuer) {
    ptx::tmem_alloc(tmem_slot, kCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  nf_pdl_begin();  // everything above touches only this CTA and overlaps the previous kernel

  if (warp == kProducer) {
    if (ptx::elect_one()) {  // producer and issuer: one thread runs the whole loop, as in the forward kernels
      Ring rg;
      for (int t = t0; t < t1; ++t, rg.next(kStages)) {
        const TileAt at = tile_at(t, p.tg);
        const int w0 = at.w * p.BW, h0 = at.h * p.BH, n = at.n * p.BI;
        if (!ptx::mbar_wait(&empty[rg.s], rg.ph ^ 1, abort_flag)) break;
        uint64_t* fb = &full[rg.s];
        uint8_t* st = smem + (size_t)rg.s * stage_bytes;
        ptx::mbar_expect_tx(fb, (uint32_t)(x_bytes + kAtoms * kBTile));
#pragma unroll
        for (int kw = 0; kw < (HB ? 1 : 3); ++kw)
          ptx::tma_load_4d(st + kw * copy_bytes, &tm_x, fb, cic * 64, p.stride * w0 + kw - 1, p.stride * h0 + khg - 1, n);
#pragma unroll
        for (int a = 0; a < kAtoms; ++a) ptx::tma_load_4d(st + x_bytes + a * 16384, &tm_dy, fb, coc * NB + a * 64, w0, h0, n);
      }
    }
    __syncwarp();
  } else if (warp == kIssuer) {
    constexpr uint32_t idesc = ptx::idesc_bf16(128, NB, 1, 1);
    // descriptors differ only in the address field; the second stacked chunk sits one tap tile further
    const uint64_t a_copy_hi = ptx::sdesc(0, copy_bytes, HB ? 1280 : 1024, 2);
    const uint64_t b_hi = ptx::sdesc(0, 16384, 8 * kBRow, kBLayout);  // next 64-channel atom: 16 KB further
    constexpr uint32_t copy16 = (uint32_t)copy_bytes >> 4;
    if (ptx::elect_one()) {
      Ring rg;
      bool ok = true;
      uint32_t sg = 0;  // SEG: segments started
      for (int t = t0; ok && t < t1; ++t, rg.next(kStages)) {
        if (!ptx::mbar_wait(&full[rg.s], rg.ph, abort_flag)) { ok = false; break; }
        ptx::tc_fence_after();
        const uint32_t xb = ptx::smem_u32(smem) + rg.s * stage_bytes;
        const uint32_t x16 = xb >> 4, g16 = (xb + x_bytes) >> 4;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const uint32_t k16 = k * (HB ? 160 : 128);  // 16 pixels (HB: two rows of the box) x 128 bytes, in 16-byte units
          const uint64_t bd = b_hi | (uint64_t)(g16 + k * kBRow);
          uint32_t acc = t > t0 || k != 0, d = tmem_base;
          if constexpr (SEG) {
            if (k % SEG == 0) {
              if (!ptx::mbar_wait(&tempty[sg % kSegSets], ((sg / kSegSets) & 1) ^ 1, abort_flag)) { ok = false; break; }
              ptx::tc_fence_after();
            }
            d += (sg % kSegSets) * kJobs * NB;
            acc = k % SEG != 0;
          }
          // taps (kh,0) and (kh,1): second chunk one tile further; tap (kh,2): rows 64..127 unused
          ptx::mma_f16(d, a_copy_hi | (uint64_t)(x16 + k16), bd, idesc, acc);
          ptx::mma_f16(d + NB, a_copy_hi | (uint64_t)(x16 + 2 * copy16 + k16), bd, idesc, acc);
          if constexpr (SEG) {
            if (k % SEG == SEG - 1) {
              if (k == 7) ptx::mma_commit(&empty[rg.s]);  // before the last arrival that somebody waits for
              ptx::mma_commit(&tfull[sg % kSegSets]);
              ++sg;
            }
          }
        }
        if constexpr (!SEG) ptx::mma_commit(&empty[rg.s]);
      }
      if (!SEG && ok) ptx::mma_commit(done);
    }
    __syncwarp();
  } else if constexpr (SEG) {
    // the sums of accumulator j over the segments; lane m of tensor memory = row m of the stacked (tap, ci) chunks
    const int lg = warp & 3, m = lg * 32 + lane, j = warp >> 2;
    const int tap = khg * 3 + (j == 0 ? (m < 64 ? 0 : 1) : 2);
    float s[NB], c[NB];
#pragma unroll
    for (int e = 0; e < NB; ++e) s[e] = c[e] = 0.f;
    const int pairs = (t1 - t0) * (8 / SEG / 2);
    const uint32_t row = tmem_base + ((uint32_t)(lg * 32) << 16) + j * NB;
#pragma unroll 1
    for (int i = 0; i < pairs; ++i) {
      const uint32_t a0 = 2 * i % kSegSets, ph = (2 * i / kSegSets) & 1;  // both sets of a pair are in the same round
      ptx::mbar_wait(&tfull[a0], ph, abort_flag);  // sets the abort flag itself when it gives up
      ptx::mbar_wait(&tfull[a0 + 1], ph, abort_flag);
      ptx::tc_fence_after();
#pragma unroll
      for (int q = 0; q < NB / 16; ++q) {
        uint32_t u[16], v[16];
        ptx::tmem_ld16(row + a0 * kJobs * NB + q * 16, u);
        ptx::tmem_ld16(row + (a0 + 1) * kJobs * NB + q * 16, v);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 16; ++e) {  // Kahan's sum
          float &se = s[q * 16 + e], &ce = c[q * 16 + e];
          const float y = (__uint_as_float(u[e]) + __uint_as_float(v[e])) - ce, t = se + y;
          ce = fmaxf((t - se) - y, -1e32f);  // NaN after an infinite t: the sum stays infinite (a true correction is below 2^104)
          se = t;
        }
      }
      ptx::tc_fence_before();
      ptx::mbar_arrive(&tempty[a0]);
      ptx::mbar_arrive(&tempty[a0 + 1]);
    }
    if (!*abort_flag) {
      const size_t plane = (size_t)p.Cout * p.Cin, pitch = p.Cin;
      float* dst = p.part + ((size_t)sp * 9 + tap) * plane + (size_t)(coc * NB) * p.Cin + cic * 64 + (m & 63);
      const int co_left = p.Cout - coc * NB;
#pragma unroll
      for (int e = 0; e < NB; ++e, dst += pitch)
        if (e < co_left) *dst = s[e];
    }
  } else {
    // epilogue: after the last MMA, lane m of tensor memory = row m of the stacked (tap, ci) chunks
    const int lg = warp & 3, m = lg * 32 + lane;
    if (ptx::mbar_wait(done, 0, abort_flag) && t1 > t0) {
      ptx::tc_fence_after();
      const size_t plane = (size_t)p.Cout * p.Cin;
      float* base = p.part + (size_t)sp * 9 * plane + (size_t)(coc * NB) * p.Cin + cic * 64 + (m & 63);
      const int co_left = p.Cout - coc * NB;  // output channels of this chunk that exist (aux: F may be < NB)
#pragma unroll 1
      for (int j = 0; j < kJobs; ++j) {
        // taps of accumulator j: rows 0..63 -> tapA, rows 64..127 -> tapB (kh*3+kw)
        const int tapA = khg * 3 + (j == 0 ? 0 : 2);
        const int tapB = j == 0 ? khg * 3 + 1 : -1;
        const int tap = m < 64 ? tapA : tapB;
#pragma unroll 2
        for (int q = 0; q < NB / 16; ++q) {  // not fully unrolled: 16 column blocks of address arithmetic spill at NB = 256
          uint32_t v[16];
          ptx::tmem_ld16(tmem_base + ((uint32_t)(lg * 32) << 16) + j * NB + q * 16, v);
          ptx::tmem_ld_wait();
          if (tap >= 0) {
            float* dst = base + (size_t)tap * plane + (size_t)(q * 16) * p.Cin;
#pragma unroll
            for (int e = 0; e < 16; ++e)
              if (q * 16 + e < co_left) dst[(size_t)e * p.Cin] = __uint_as_float(v[e]);
          }
        }
      }
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(p.status, NF_ETIMEOUT);
    const unsigned long long tt = ptx::globaltimer();
    while (ptx::globaltimer() - tt < 2000000ull) __nanosleep(1000);
  }
  if (warp == kIssuer) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, kCols);
  }
}

// ---------------------------------------------------------------- weight gradient, stride 1, column shift on the gradient
// dW[kh,kw][co][ci] = sum_{i,j} dy[i,j,co] * x[i+kh-1, j+kw-1, ci].  With j' = j+kw-1 this is
//   sum over the pixels (i,j') of the x grid of  x[i+kh-1, j', ci] * dy[i, j'-kw+1, co]   (dy = 0 outside),
// so the column tap can sit on the gradient operand: ONE activation box (BH+2 rows, no column copies)
// and three column-shifted gradient tiles per stage.  Per 16 pixels two instructions:
//   A (M = 128) = rows kh=0 and kh=1 of the box stacked (second one half empty: kh=2 + unused rows),
//   B (N = 3*NB) = the three shifted gradient tiles side by side (MN-major atoms one tile apart).
// Fewer operand bytes per useful FLOP than stacking all nine taps on the activation side.
template <int NB>
__global__ void __launch_bounds__(kThreads, 1)
conv_wgrad_kw_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_dy, const WgParams p) {
  constexpr int kBRow = NB * 2;
  constexpr uint32_t kBLayout = NB == 64 ? 2 : NB == 32 ? 4 : 6;
  constexpr int kBTile = 128 * kBRow;                 // one shifted gradient tile
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int box_bytes = (p.BH + 2) * p.BW * 128;
  const int g_region = 3 * kBTile < 4096 ? 4096 : 3 * kBTile;  // >= 32 rows after the box for the unused operand rows
  const int stage_bytes = box_bytes + g_region;
  const int stages = p.stages;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)stages * stage_bytes);
  uint64_t* full = bars;
  uint64_t* empty = bars + kMaxStages;
  uint64_t* done = bars + 2 * kMaxStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  constexpr uint32_t kAcc = NB == 64 ? 256 : 3 * NB <= 64 ? 64 : 128;  // columns reserved per accumulator
  constexpr uint32_t kCols = 2 * kAcc;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int blocks = p.ci_chunks * p.co_chunks;
  const int blk = blockIdx.x % blocks, sp = blockIdx.x / blocks;
  const int cic = blk % p.ci_chunks, coc = blk / p.ci_chunks;
  const int t0 = (int)((long)p.pix_tiles * sp / p.splits), t1 = (int)((long)p.pix_tiles * (sp + 1) / p.splits);

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    ptx::mbar_init(done, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(&tm_x);
    ptx::prefetch_tmap(&tm_dy);
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, kCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  nf_pdl_begin();  // everything above touches only this CTA and overlaps the previous kernel

  if (warp == 0) {
    if (ptx::elect_one()) {
      Ring rg;
      for (int t = t0; t < t1; ++t, rg.next(stages)) {
        const TileAt at = tile_at(t, p.tg);
        const int w0 = at.w * p.BW, h0 = at.h * p.BH, n = at.n;
        if (!ptx::mbar_wait(&empty[rg.s], rg.ph ^ 1, abort_flag)) break;
        uint64_t* fb = &full[rg.s];
        uint8_t* st = smem + (size_t)rg.s * stage_bytes;
        ptx::mbar_expect_tx(fb, (uint32_t)(box_bytes + 3 * kBTile));
        ptx::tma_load_4d(st, &tm_x, fb, cic * 64, w0, h0 - 1, n);
#pragma unroll
        for (int kw = 0; kw < 3; ++kw)  // gradient column j = j' - kw + 1
          ptx::tma_load_4d(st + box_bytes + kw * kBTile, &tm_dy, fb, coc * NB, w0 - kw + 1, h0, n);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    constexpr uint32_t idesc = ptx::idesc_bf16(128, 3 * NB, 1, 1);
    const uint64_t a_hi = ptx::sdesc(0, p.BW * 128, 1024, 2);      // second 64 rows: one image row further
    const uint64_t b_hi = ptx::sdesc(0, kBTile, 8 * kBRow, kBLayout);  // next N atom: next shifted tile
    const uint32_t row16 = (uint32_t)(p.BW * 128) >> 4;
    if (ptx::elect_one()) {
      Ring rg;
      bool ok = true;
      for (int t = t0; t < t1; ++t, rg.next(stages)) {
        if (!ptx::mbar_wait(&full[rg.s], rg.ph, abort_flag)) { ok = false; break; }
        ptx::tc_fence_after();
        const uint32_t xb = ptx::smem_u32(smem) + rg.s * stage_bytes;
        const uint32_t x16 = xb >> 4, g16 = (xb + box_bytes) >> 4;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const uint64_t bd = b_hi | (uint64_t)(g16 + k * kBRow);   // 16 pixels x kBRow bytes = k * kBRow sixteen-byte units
          const uint32_t acc = t > t0 || k != 0;
          ptx::mma_f16(tmem_base, a_hi | (uint64_t)(x16 + k * 128), bd, idesc, acc);                      // kh = 0 | 1
          ptx::mma_f16(tmem_base + kAcc, a_hi | (uint64_t)(x16 + 2 * row16 + k * 128), bd, idesc, acc);  // kh = 2 | unused
        }
        ptx::mma_commit(&empty[rg.s]);
      }
      if (ok) ptx::mma_commit(done);
    }
    __syncwarp();
  } else {
    const int lg = warp & 3, m = lg * 32 + lane;
    if (ptx::mbar_wait(done, 0, abort_flag) && t1 > t0) {
      ptx::tc_fence_after();
      const size_t plane = (size_t)p.Cout * p.Cin;
      float* base = p.part + (size_t)sp * 9 * plane + (size_t)(coc * NB) * p.Cin + cic * 64 + (m & 63);
      const int co_left = p.Cout - coc * NB;
#pragma unroll 1
      for (int j = 0; j < 2; ++j) {
        const int kh = j == 0 ? (m < 64 ? 0 : 1) : (m < 64 ? 2 : -1);
#pragma unroll 1
        for (int kw = 0; kw < 3; ++kw)
#pragma unroll
          for (int q = 0; q < NB / 16; ++q) {
            uint32_t v[16];
            ptx::tmem_ld16(tmem_base + ((uint32_t)(lg * 32) << 16) + j * kAcc + kw * NB + q * 16, v);
            ptx::tmem_ld_wait();
            if (kh >= 0) {
              float* dst = base + (size_t)(kh * 3 + kw) * plane + (size_t)(q * 16) * p.Cin;
#pragma unroll
              for (int e = 0; e < 16; ++e)
                if (q * 16 + e < co_left) dst[(size_t)e * p.Cin] = __uint_as_float(v[e]);
            }
          }
      }
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(p.status, NF_ETIMEOUT);
    const unsigned long long tt = ptx::globaltimer();
    while (ptx::globaltimer() - tt < 2000000ull) __nanosleep(1000);
  }
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, kCols);
  }
}

// ---------------------------------------------------------------- weight gradient, stride 1, 128 output channels on the M side
// A CTA owns one column tap kw, 128 output channels and CC chunks of 64 input channels:
//   A (M = 128) = the gradient tile of 128 output channels (two MN-major atoms),
//   B (N = 192) = the three row taps of ONE activation box (rows h0 - 1 .. h0 + BH, columns shifted by kw - 1) as consecutive
//                 64-channel atoms one image row apart (or the box unshifted and the gradient shifted by 1 - kw, the same sum over
//                 the activation's pixels),
// so an instruction per 16 pixels and chunk yields three taps x 64 x 128 with no idle half: the forms with the activation on the M
// side stack taps 0 | 1 and 2 | nothing and waste a quarter of the tensor pipe, and the per-tap one fetches each pixel three times
// (112 KB of shared memory fill per 128 pixels and 3 x 64 x 256 products; here 72 KB for the same with CC = 2).  Tiles of BI images
// (8x8x2, 4x4x8) have a box of BH + 2 rows per image; 16 consecutive pixels of the gradient tile must lie in one image:
// BW * BH a multiple of 16.  The partial sums leave with 16-byte stores, a thread per output channel.
template <int CC>
__global__ void __launch_bounds__(kThreads, 1)
conv_wgrad_row_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_dy, const WgParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int box_bytes = p.BI * (p.BH + 2) * p.BW * 128;
  const int stage_bytes = CC * box_bytes + 2 * 16384;
  const int stages = p.stages;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)stages * stage_bytes);
  uint64_t* full = bars;
  uint64_t* empty = bars + kMaxStages;
  uint64_t* done = bars + 2 * kMaxStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  constexpr uint32_t kCols = CC * 256;  // 192 used of each 256

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int blocks = p.ci_chunks * p.co_chunks;
  const int blk = blockIdx.x % blocks, rest = blockIdx.x / blocks;
  const int kw = rest % 3, sp = rest / 3;
  const int cic = blk % p.ci_chunks, coc = blk / p.ci_chunks;
  const int t0 = (int)((long)p.pix_tiles * sp / p.splits), t1 = (int)((long)p.pix_tiles * (sp + 1) / p.splits);

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    ptx::mbar_init(done, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(&tm_x);
    ptx::prefetch_tmap(&tm_dy);
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, kCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  nf_pdl_begin();  // everything above touches only this CTA and overlaps the previous kernel

  if (warp == 0) {
    if (ptx::elect_one()) {
      Ring rg;
      for (int t = t0; t < t1; ++t, rg.next(stages)) {
        const TileAt at = tile_at(t, p.tg);
        const int w0 = at.w * p.BW, h0 = at.h * p.BH, n = at.n * p.BI;
        if (!ptx::mbar_wait(&empty[rg.s], rg.ph ^ 1, abort_flag)) break;
        uint64_t* fb = &full[rg.s];
        uint8_t* st = smem + (size_t)rg.s * stage_bytes;
        ptx::mbar_expect_tx(fb, (uint32_t)stage_bytes);
#pragma unroll
        for (int a = 0; a < 2; ++a) ptx::tma_load_4d(st + a * 16384, &tm_dy, fb, coc * 128 + a * 64, w0 - (p.dy_shift ? kw - 1 : 0), h0, n);
#pragma unroll
        for (int c = 0; c < CC; ++c)
          ptx::tma_load_4d(st + 32768 + c * box_bytes, &tm_x, fb, (cic * CC + c) * 64, w0 + (p.dy_shift ? 0 : kw - 1), h0 - 1, n);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    constexpr uint32_t idesc = ptx::idesc_bf16(128, 192, 1, 1);
    const uint64_t a_hi = ptx::sdesc(0, 16384, 1024, 2);       // next 64 output channels: next atom
    const uint64_t b_hi = ptx::sdesc(0, p.BW * 128, 1024, 2);  // next row tap: one image row further
    const int per_img = p.BW * p.BH / 16;                      // 16-pixel steps per image of the tile
    const uint32_t gap16 = (uint32_t)(2 * p.BW * 128) >> 4;    // the two halo rows between the images' boxes
    if (ptx::elect_one()) {
      Ring rg;
      bool ok = true;
      for (int t = t0; t < t1; ++t, rg.next(stages)) {
        if (!ptx::mbar_wait(&full[rg.s], rg.ph, abort_flag)) { ok = false; break; }
        ptx::tc_fence_after();
        const uint32_t g16 = (ptx::smem_u32(smem) + rg.s * stage_bytes) >> 4;
        uint32_t x16 = g16 + (32768 >> 4);
        int left = per_img;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (left == 0) {
            x16 += gap16;
            left = per_img;
          }
          --left;
#pragma unroll
          for (int c = 0; c < CC; ++c)
            ptx::mma_f16(tmem_base + c * 256, a_hi | (uint64_t)(g16 + k * 128), b_hi | (uint64_t)(x16 + ((c * box_bytes) >> 4) + k * 128), idesc,
                         t > t0 || k != 0);
        }
        ptx::mma_commit(&empty[rg.s]);
      }
      if (ok) ptx::mma_commit(done);
    }
    __syncwarp();
  } else {
    const int lg = warp & 3, m = lg * 32 + lane;  // m: output channel of the CTA's 128
    if (ptx::mbar_wait(done, 0, abort_flag) && t1 > t0) {
      ptx::tc_fence_after();
      const size_t plane = (size_t)p.Cout * p.Cin;
      float* base = p.part + ((size_t)sp * 9 + kw) * plane + (size_t)(coc * 128 + m) * p.Cin + cic * CC * 64;
#pragma unroll 1
      for (int q = 0; q < CC * 12; ++q) {  // 16 input channels of one row tap at a time
        const int c = q / 12, kh = (q / 4) % 3, b = q % 4;
        uint32_t v[16];
        ptx::tmem_ld16(tmem_base + ((uint32_t)(lg * 32) << 16) + c * 256 + kh * 64 + b * 16, v);
        ptx::tmem_ld_wait();
        float4* dst = reinterpret_cast<float4*>(base + (size_t)(kh * 3) * plane + c * 64 + b * 16);
#pragma unroll
        for (int e = 0; e < 4; ++e)
          dst[e] = make_float4(__uint_as_float(v[4 * e]), __uint_as_float(v[4 * e + 1]), __uint_as_float(v[4 * e + 2]),
                               __uint_as_float(v[4 * e + 3]));
      }
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(p.status, NF_ETIMEOUT);
    const unsigned long long tt = ptx::globaltimer();
    while (ptx::globaltimer() - tt < 2000000ull) __nanosleep(1000);
  }
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, kCols);
  }
}

// ---------------------------------------------------------------- weight gradient, stride 1, few filters: gradient on the M side
// An instruction of up to 64 columns takes about 40 cycles whatever its width, one of 192 takes 96, so for the auxiliary conv
// (F <= 32 filters) the fewest instructions win.  Here the roles of conv_wgrad_kw_kernel are swapped:
//   A (M = 4 * NB rows) = the three column-shifted gradient tiles as consecutive MN-major atoms (kw, f) plus one unused atom,
//   B (N = 192)         = the three row taps of the activation box as consecutive 64-channel atoms (kh, ci),
// so ONE instruction per 16 pixels produces all nine taps: D[(kw, f), (kh, ci)].  NB = 16 uses the 64-row shape
// (row r in TMEM lane 32 * (r / 16) + r % 16), NB = 32 the 128-row shape (row r in lane r); in both, the warp of
// lane quadrant q holds column tap kw = q and lane l holds filter f = l.
template <int NB>
__global__ void __launch_bounds__(kThreads, 1)
conv_wgrad_gx_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_dy, const WgParams p) {
  constexpr int kBRow = NB * 2;
  constexpr uint32_t kGLayout = NB == 32 ? 4 : 6;
  constexpr int kGTile = 128 * kBRow;                 // one shifted gradient tile
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int box_bytes = (p.BH + 2) * p.BW * 128;
  const int stage_bytes = box_bytes + 4 * kGTile;     // the fourth atom is never loaded: its accumulator rows are not read
  const int stages = p.stages;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + (size_t)stages * stage_bytes);
  uint64_t* full = bars;
  uint64_t* empty = bars + kMaxStages;
  uint64_t* done = bars + 2 * kMaxStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  constexpr uint32_t kCols = 256;                     // 192 accumulator columns

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cic = blockIdx.x % p.ci_chunks, sp = blockIdx.x / p.ci_chunks;
  const int t0 = (int)((long)p.pix_tiles * sp / p.splits), t1 = (int)((long)p.pix_tiles * (sp + 1) / p.splits);

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) {
      ptx::mbar_init(&full[s], 1);
      ptx::mbar_init(&empty[s], 1);
    }
    ptx::mbar_init(done, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::prefetch_tmap(&tm_x);
    ptx::prefetch_tmap(&tm_dy);
  }
  if (warp == 1) {
    ptx::tmem_alloc(tmem_slot, kCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  nf_pdl_begin();  // everything above touches only this CTA and overlaps the previous kernel

  if (warp == 0) {
    if (ptx::elect_one()) {
      Ring rg;
      for (int t = t0; t < t1; ++t, rg.next(stages)) {
        const TileAt at = tile_at(t, p.tg);
        const int w0 = at.w * p.BW, h0 = at.h * p.BH, n = at.n;
        if (!ptx::mbar_wait(&empty[rg.s], rg.ph ^ 1, abort_flag)) break;
        uint64_t* fb = &full[rg.s];
        uint8_t* st = smem + (size_t)rg.s * stage_bytes;
        ptx::mbar_expect_tx(fb, (uint32_t)(box_bytes + 3 * kGTile));
        ptx::tma_load_4d(st, &tm_x, fb, cic * 64, w0, h0 - 1, n);
#pragma unroll
        for (int kw = 0; kw < 3; ++kw)  // gradient column j = j' - kw + 1
          ptx::tma_load_4d(st + box_bytes + kw * kGTile, &tm_dy, fb, 0, w0 - kw + 1, h0, n);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    constexpr uint32_t idesc = ptx::idesc_bf16(4 * NB, 192, 1, 1);
    const uint64_t a_hi = ptx::sdesc(0, kGTile, 8 * kBRow, kGLayout);  // next M atom: next shifted tile
    const uint64_t b_hi = ptx::sdesc(0, p.BW * 128, 1024, 2);          // next N atom: one image row further (next kh)
    if (ptx::elect_one()) {
      Ring rg;
      bool ok = true;
      for (int t = t0; t < t1; ++t, rg.next(stages)) {
        if (!ptx::mbar_wait(&full[rg.s], rg.ph, abort_flag)) { ok = false; break; }
        ptx::tc_fence_after();
        const uint32_t xb = ptx::smem_u32(smem) + rg.s * stage_bytes;
        const uint32_t x16 = xb >> 4, g16 = (xb + box_bytes) >> 4;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          ptx::mma_f16(tmem_base, a_hi | (uint64_t)(g16 + k * kBRow), b_hi | (uint64_t)(x16 + k * 128), idesc, t > t0 || k != 0);
        ptx::mma_commit(&empty[rg.s]);
      }
      if (ok) ptx::mma_commit(done);
    }
    __syncwarp();
  } else {
    const int lg = warp & 3;  // = column tap kw of this warp's rows
    if (ptx::mbar_wait(done, 0, abort_flag) && t1 > t0) {
      ptx::tc_fence_after();
      const size_t plane = (size_t)p.Cout * p.Cin;
      const bool mine = lg < 3 && lane < NB && lane < p.Cout;
      float* base = p.part + (size_t)sp * 9 * plane + (size_t)lg * plane + (size_t)lane * p.Cin + cic * 64;
#pragma unroll 1
      for (int kh = 0; kh < 3; ++kh)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t v[16];
          ptx::tmem_ld16(tmem_base + ((uint32_t)(lg * 32) << 16) + kh * 64 + q * 16, v);
          ptx::tmem_ld_wait();
          if (mine) {
            float4* dst = reinterpret_cast<float4*>(base + (size_t)(kh * 3) * plane + q * 16);
#pragma unroll
            for (int e = 0; e < 4; ++e)
              dst[e] = make_float4(__uint_as_float(v[4 * e]), __uint_as_float(v[4 * e + 1]), __uint_as_float(v[4 * e + 2]),
                                   __uint_as_float(v[4 * e + 3]));
          }
        }
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) atomicOr(p.status, NF_ETIMEOUT);
    const unsigned long long tt = ptx::globaltimer();
    while (ptx::globaltimer() - tt < 2000000ull) __nanosleep(1000);
  }
  if (warp == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, kCols);
  }
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// bf16 tensor, 4 dims (innermost first), zero fill outside; the swizzle span equals the inner box (32/64/128 bytes)
// rows_last: the map's dimensions run (channel, column, image, row) instead of (channel, column, row, image); dims and box stay in
// the latter order.
int make_map4(CUtensorMap* m, const void* base, const uint64_t dims[4], const uint32_t box[4], int spatial_stride = 1,
              bool rows_last = false) {
  const CUtensorMapSwizzle sw = box[0] * 2 >= 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                : box[0] * 2 == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
  EncodeTiledFn fn = encode_fn();
  if (!fn) return NF_ECUDA;
  cuuint64_t gdim[4] = {dims[0], dims[1], dims[2], dims[3]};
  cuuint64_t gstr[3] = {dims[0] * 2, dims[0] * dims[1] * 2, dims[0] * dims[1] * dims[2] * 2};
  // with an element stride s along w and h the box spans s*box elements and keeps every s-th one
  const cuuint32_t ss = (cuuint32_t)spatial_stride;
  cuuint32_t bx[4] = {box[0], box[1] * ss, box[2] * ss, box[3]};
  cuuint32_t es[4] = {1, ss, ss, 1};
  if (rows_last) {
    std::swap(gdim[2], gdim[3]);
    std::swap(gstr[1], gstr[2]);
    std::swap(bx[2], bx[3]);
  }
  const CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), gdim, gstr, bx, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? NF_OK : nf_cuda_check(cudaErrorInvalidValue, "cuTensorMapEncodeTiled");
}

// Per-process caches (kernel attributes, SM count, symbol addresses) are kept per device: a process may use several.
constexpr int kMaxDevices = 64;
int current_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
  return dev;
}

int sm_count() {
  static int n_dev[kMaxDevices];
  const int dev = current_device();
  int& n = n_dev[dev];
  if (!n) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 148;
  }
  return n;
}

// mode 0: main forward (y + statistics), 1: aux forward (bias + ReLU, Cout = F), 2: aux input gradient
// (Cin = F <= 64 and a multiple of 8, Cout a multiple of 64, mirrored MN-major weights).
// H, W: OUTPUT size (equal to the input size for stride 1).
// Pixel tile of 128 output pixels: a BW x BH patch of one image, or (per-tap mode only) of BI images at once.
// Sizes that no patch divides (14, 7, 28, odd ones) take the per-tap mode with the powers of two BW * BH * BI = 128 that cover
// the N x H x W pixels with the fewest tiles (7x7 maps: one pixel of 128 images; 14x14: 2x2 pixels of 32): loads beyond an
// edge read zeros, stores are clipped, the epilogue zeroes what hangs over.  Where several cover equally well the one with
// the largest patch is taken: neighbouring taps then find most of their pixels in L2.
// Returns whether the tiles divide the maps (a last tile may still lack images).
bool pick_tile(int N, int H, int W, int* BW, int* BH, int* BI) {
  const int cand[3][2] = {{16, 8}, {32, 4}, {8, 16}};
  for (auto& c : cand)
    if (W % c[0] == 0 && H % c[1] == 0) {
      *BW = c[0]; *BH = c[1]; *BI = 1;
      return true;
    }
  if (W * H <= 64 && 128 % (W * H) == 0 && (W & (W - 1)) == 0) {  // 8x8, 4x4, 2x2, 8x4, 1x1 ...
    *BW = W; *BH = H; *BI = 128 / (W * H);
    return true;
  }
  long best = -1;
  for (int bi = 1; bi <= 128; bi *= 2)
    for (int bw = 1; bw * bi <= 128; bw *= 2) {
      const int bh = 128 / (bi * bw);
      const long tiles = (long)((N + bi - 1) / bi) * ((H + bh - 1) / bh) * ((W + bw - 1) / bw);
      if (best < 0 || tiles < best) {
        best = tiles;
        *BW = bw; *BH = bh; *BI = bi;
      }
    }
  return false;
}
// Whether a convolution whose result is rounded for storage (forward, input gradient) goes to the tensor cores.  Maps that tile
// exactly always do; the others, in segments, from 8192 output pixels on (64 tiles).  Below that a layer's gradients hang on a few
// thousand ReLU decisions, and an output that is rounded the other way moves them by up to several per cent in the next step; the
// CUDA-core kernels give the same bits as they always have there.  The line is drawn by that, not by speed: just below it the
// tensor cores would be several times faster.  The weight gradients stay in fp32, decide nothing and always run here.
bool tc_size_ok(int N, int H, int W) {
  int BW, BH, BI;
  return pick_tile(N, H, W, &BW, &BH, &BI) || (long)N * H * W >= 8192;
}

bool tiles_exactly(int H, int W) {
  int BW, BH, BI;
  return pick_tile(1, H, W, &BW, &BH, &BI);
}

// ybuf = 1 reserves the y2 tile of the fused BatchNorm-backward sums (as large as the output staging)
TcPlan plan_fwd(int H, int W, int Cin, int Cout, int N, int epi = 0, int stride = 1, int ybuf = 0) {
  TcPlan pl{};
  if (stride == 2 && (epi != 0 || Cin % 64)) return pl;
  if (epi == 2 ? (Cin > 64 || Cin % 8 || Cout % 64) : (Cin % 64 != 0)) return pl;
  if (epi == 0 ? (Cout % 64 != 0) : epi == 1 ? (Cout > 64) : false) return pl;
  const bool exact = pick_tile(N, H, W, &pl.BW, &pl.BH, &pl.BI);
  pl.PT = (stride == 2 || pl.BI > 1 || !exact) ? 1 : 0;
  pl.SEG = !exact;  // maps that no tile divides
  if (epi == 0 && Cout % 256 == 0) pl.PT = 1;  // 256-wide instructions need the per-tap form (one tap of weights per stage)
  pl.BN = epi != 1 ? (Cout % 128 == 0 ? 128 : 64) : (Cout <= 16 ? 16 : Cout <= 32 ? 32 : 64);
  if (epi == 0 && pl.PT && !pl.SEG && Cout % 256 == 0) pl.BN = 256;  // per-tap form: weights of one tap and 256 channels are 32 KB a stage
  pl.KC = epi == 2 ? (Cin <= 16 ? 16 : Cin <= 32 ? 32 : 64) : 64;
  size_t a_stride = pl.PT ? (size_t)128 * pl.KC * 2 : ((size_t)(pl.BH + 2) * pl.BW * pl.KC * 2 + 1023) & ~(size_t)1023;
  pl.RW = (!pl.PT && epi != 2 && Cin == 64 && pl.BN <= 64) ? 1 : 0;  // weights resident in shared memory
  size_t b_stage = pl.RW ? 0 : pl.PT ? (epi == 2 ? (size_t)(pl.BN / 64) * pl.KC * 128 : (size_t)pl.BN * 128)
                                           : epi == 2 ? (size_t)(pl.BN / 64) * 3 * pl.KC * 128 : (size_t)3 * pl.BN * 128;
  pl.yslots = ybuf ? 1 : 0;
  size_t extra = pl.RW ? (size_t)9 * pl.BN * 128 : 0;
  // narrow auxiliary convolutions on several images per tile: three boxes per chunk where the swizzle allows it and two stages (and,
  // for the gradient, two y2 tiles) fit; maps of one row gain nothing
  if (pl.PT && stride == 1 && !pl.SEG && pl.BI > 1 && pl.BH > 1 && pl.BI * pl.BW % 8 == 0 && (epi == 1 ? pl.BN <= 32 : epi == 2 && pl.KC == 16)) {
    const size_t a3 = (size_t)3 * (pl.BH + 2) * pl.BW * pl.BI * pl.KC * 2, b9 = (size_t)9 * (epi == 2 ? pl.BN / 64 * pl.KC : pl.BN) * 128;
    const size_t staged = epi == 2 ? (size_t)pl.BN / 64 * 16384 : 0;  // two output tiles, two of y2
    if (a3 % 3072 == 0 && 2 * a3 + (epi == 2 ? 1 : 2) * b9 + 4 * staged + 2048 <= 232448) {
      pl.PT = 2;
      pl.RW = epi == 2;
      a_stride = a3;
      b_stage = epi == 2 ? 0 : b9;
      pl.yslots *= 2;
      extra = staged + (epi == 2 ? b9 : 0);
    }
  }
  // Tiles of one image without sums over them.  64 aux filters: two epilogue groups, outputs through staging tiles (1904 maps of 32x32x64
  // 242 -> 151 us, 64 maps 14.6 -> 11.1).  One box per chunk: up to 32 filters over several chunks (256 channels at 16x16, 1777 maps:
  // 115 -> 107 us; with one chunk the box of a tile is too little to tell); and, with two epilogue groups, the input gradient (of a
  // pooled layer or one with a shortcut), where the weights fit beside three stages (1904 maps of 32x32x64 158 -> 148 us).
  const bool sumless = pl.PT == 0 && stride == 1 && (epi == 1 || (epi == 2 && !ybuf));
  if (sumless && W % 8 == 0 && H % 16 == 0 && (epi == 2 || (Cin > 64 && Cout <= 32))) {
    const size_t a1 = ((size_t)18 * 10 * pl.KC * 2 + 1023) & ~(size_t)1023, b9 = (size_t)9 * (epi == 2 ? pl.BN / 64 * pl.KC : pl.BN) * 128;
    const size_t staged = epi == 2 ? 32768 : 0;
    const bool resident = epi == 2 || Cin / 64 * b9 + staged + 4 * a1 + 2048 <= 232448;
    if (resident ? b9 * (epi == 2 ? 1 : Cin / 64) + staged + 3 * a1 + 2048 <= 232448 : staged + 2 * (a1 + b9) + 2048 <= 232448) {
      pl.SB = 1;
      pl.BW = 8; pl.BH = 16;
      pl.RW = resident;
      a_stride = a1;
      b_stage = resident ? 0 : b9;
      extra = resident ? b9 * (epi == 2 ? 1 : Cin / 64) : 0;
    }
  }
  pl.NS = sumless && !pl.SEG && (epi == 1 ? Cout == 64 : pl.SB);
  const size_t stage = ((a_stride + 1023) & ~(size_t)1023) + b_stage;
  const size_t fixed = (size_t)(pl.NS ? 2 : epi != 1 ? (pl.BN == 256 ? 2 : pl.BN / 64) : 0) * 16384 * (1 + pl.yslots) + extra + 1024 + 1024;
  int st = (int)((232448 - fixed) / stage);
  if (st > kMaxStages) st = kMaxStages;
  if (st < 2) return pl;
  pl.stages = st;
  pl.smem = (size_t)st * stage + fixed;
  pl.parts = pl.BN >= 128 ? 1 : 128 / pl.BN;
  const int n_tiles = epi != 1 ? Cout / pl.BN : 1;
  const long total = (long)((N + pl.BI - 1) / pl.BI) * ((H + pl.BH - 1) / pl.BH) * ((W + pl.BW - 1) / pl.BW) * n_tiles;
  if (total >= (1l << 30)) return pl;
  long g = sm_count();
  g -= g % n_tiles;  // every CTA keeps one channel tile for its whole life
  if (g < n_tiles) g = n_tiles;
  if (g > total) g = total;
  pl.grid = (int)g;
  pl.ok = 1;
  return pl;
}

template <int BN, int EPI, int KC = 64, int BMN = 0, int PT = 0, int RW = 0, int SEG = 0, int POST = 0, int SB = 0, int NS = 0>
int launch_fwd(const TcPlan& pl, const CUtensorMap& mx, const CUtensorMap& mw, const CUtensorMap& my, const FwdParams& p) {
  static bool attr_done_dev[kMaxDevices];  // function attributes belong to a device's context: set once per device
  bool& attr_done = attr_done_dev[current_device()];
  if (!attr_done) {
    NF_CUDA(cudaFuncSetAttribute(conv_fwd_tc_kernel<BN, EPI, KC, BMN, PT, RW, SEG, POST, SB, NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448));
    attr_done = true;
  }
  nf_launch(conv_fwd_tc_kernel<BN, EPI, KC, BMN, PT, RW, SEG, POST, SB, NS>, pl.grid, fwd_threads(EPI, PT, NS), pl.smem, mx, mw, my, p);
  NF_LAUNCHED();
  return NF_OK;
}

// The folded-tap kernel covers, when W % 14 == 0 and H % 8 == 0: the main forward 64 -> 64 (epi 0), the aux
// forward with F <= 64, F % 8 == 0 (epi 1) if all weight tiles fit in shared memory beside >= 3 activation
// stages, and the aux input gradient F -> Cout (epi 2; F <= 32, F % 8 == 0, Cout % 64 == 0).  The input gradient
// also takes widths that tile by 16 instead of 14 (its unfolded form): always with the fused BatchNorm-backward
// sums (stats 2) or 64 output channels; without the sums a wider layer is faster on the generic kernel's
// 128-channel tiles (measured).
int fold_group(int Cout, int epi) { return epi != 1 ? 64 : (Cout <= 16 ? 16 : Cout <= 32 ? 32 : 64); }
// widths the 14-column tiles of the folded forward cover: multiples of 14, and wider maps whose ragged last tile column wastes
// at most a third (32, 48, 64, ...: the zero-filled loads and clipped stores of TMA make the overhang harmless)
bool fold_width_ok(int W) { return W % 14 == 0 || (W >= 28 && ((W + 13) / 14) * 14 * 3 <= W * 4); }

// Maps that no 128-pixel tile divides (56 x 56, 40 x 40) stay with the segmented sums in a layer; the stand-alone forward (any_map)
// takes the folded kernel there too, as it always has.
bool fold_ok(int H, int W, int Cin, int Cout, int epi, int stride, int stats = 0, size_t extra_smem = 0, bool any_map = false) {
  if (stride != 1 || H % 8 || !(any_map || tiles_exactly(H, W))) return false;
  if (epi == 2 && W % 14 && W % 16 == 0 && (stats >= 2 || Cout == 64)) return Cin <= 32 && Cin % 8 == 0 && Cout % 64 == 0;
  if (epi == 2 ? W % 14 != 0 : !fold_width_ok(W)) return false;
  // the plain aux forward (no fused normalisation: extra_smem == 0) stays on the generic kernel for ragged widths: with 64
  // filters at 32 columns the folded form measured slower there (0.33 vs 0.25 ms), the fused form faster everywhere
  if (epi == 1 && W % 14 != 0 && extra_smem == 0) return false;
  if (epi == 2) return Cin <= 32 && Cin % 8 == 0 && Cout % 64 == 0;
  if (Cin == 16 && epi == 0) return Cout == 64;  // first layers, padded to 16 channels
  if (Cin % 64) return false;
  if (epi == 0 ? (Cin != 64 || Cout != 64) : (Cout > 64 || Cout % 8)) return false;
  const size_t wbytes = (size_t)9 * (Cin / 64) * fold_group(Cout, epi) * 128;
  return wbytes + (epi == 0 ? 2 * 16384 : 0) + extra_smem + 2048 + 3 * 20480 <= 232448;
}

template <int G, int EPI, int KC = 64, int MIR = 0, int UF = 0, int XF = 0, int POST = 0>
int launch_fold(int grid, size_t smem, const CUtensorMap& mx, const CUtensorMap& mw, const CUtensorMap& my, const CUtensorMap& my2,
                const FoldParams& p) {
  static bool attr_done_dev[kMaxDevices];  // function attributes belong to a device's context: set once per device
  bool& attr_done = attr_done_dev[current_device()];
  if (!attr_done) {
    NF_CUDA(cudaFuncSetAttribute(conv_fwd_fold_kernel<G, EPI, KC, MIR, UF, XF, POST>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448));
    attr_done = true;
  }
  nf_launch(conv_fwd_fold_kernel<G, EPI, KC, MIR, UF, XF, POST>, grid, kFoldThreads + kXfThreads * XF, smem, mx, mw, my, my2, p);
  NF_LAUNCHED();
  return NF_OK;
}

// BatchNorm-backward inputs of the fused reduction (stats 2): y2 has the shape of the output
struct BnBwdIn {
  const void* y2;
  const float *scale, *shift, *mu, *invstd;
  const float *sdz = nullptr, *sdzx = nullptr;  // second pass (stats 4): the reduced sums and 1 / (elements per channel)
  float inv_m = 0.f;
};

// Normalisation fused into the aux forward (epi 1): x is then the conv output and a = ReLU(x*scale + shift) is written to a
struct XfIn {
  const float *scale, *shift;
  void* a;
  float* pool_part;  // non-null: pooling partials and sign mask instead of h (see FoldParams)
  uint8_t* mask;
};

int run_fold(int N, int H, int W, int Cin, int Cout, const void* x, const void* w, void* y, int stats, float* red,
             size_t red_floats, int32_t* status, int* nb, int epi, const float* bias, const BnBwdIn* bn = nullptr,
             const XfIn* xf = nullptr) {
  const int G = fold_group(Cout, epi);
  const int KC = epi == 2 ? (Cin <= 16 ? 16 : 32) : Cin < 64 ? 16 : 64;
  // input gradient on widths that also tile by 16: the unfolded form (three shifted boxes, no shift-add in the epilogue);
  // where the map tiles by 8 x 16 as well: its single-box form
  const bool uf = epi == 2 && W % 16 == 0;
  const bool uf2 = uf && H % 16 == 0;
  // ... and by 8 x 32 with 16 channels of dh: the form with 256 pixels per instruction
  const bool wide = uf2 && KC == 16;  // H % 16 == 0: the last tile row may be half a tile
  const int TW = uf2 ? 8 : uf ? 16 : 14, TH = wide ? 32 : uf2 ? 16 : 8;
  CUtensorMap mx, mw, my, my2;
  const uint64_t dx[4] = {(uint64_t)Cin, (uint64_t)W, (uint64_t)H, (uint64_t)N};
  const uint32_t bx[4] = {(uint32_t)KC, (uint32_t)(uf2 ? 10 : 16), (uint32_t)(wide ? 34 : uf2 ? 18 : 10), 1};
  // forward: weights [kh][kw][Cout][Cin], box = G rows of co x 64 ci for the three kw of one kh;
  // input gradient: weights [kh][kw][F][Cout], box = KC rows of f x 64 c for the three kw of one kh
  const uint64_t dw[4] = {(uint64_t)(epi == 2 ? Cout : Cin), (uint64_t)(epi == 2 ? Cin : Cout), 3, 3};
  const uint32_t bw[4] = {(uint32_t)(epi == 2 ? 64 : KC), (uint32_t)(epi == 2 ? KC : G), 3, 1};
  const uint64_t dy[4] = {(uint64_t)Cout, (uint64_t)W, (uint64_t)H, (uint64_t)N};
  const uint32_t by[4] = {64, (uint32_t)TW, (uint32_t)TH, 1};
  int rc;
  if ((rc = make_map4(&mx, x, dx, bx)) != NF_OK) return rc;
  if ((rc = make_map4(&mw, w, dw, bw)) != NF_OK) return rc;
  if (epi != 1) {
    if ((rc = make_map4(&my, y, dy, by)) != NF_OK) return rc;
  } else {
    my = mx;
  }
  if (xf) {  // the normalised activation leaves the aux forward through TMA stores of 14 x 8-pixel tiles, 64 channels each
    const uint32_t ba[4] = {64, 14, 8, 1};
    if ((rc = make_map4(&my, xf->a, dx, ba)) != NF_OK) return rc;
  }
  my2 = my;
  if (stats >= 2) {
    if (epi != 2 || !bn || (stats == 4 && (!bn->sdz || !bn->sdzx))) return NF_EINVAL;
    if ((rc = make_map4(&my2, bn->y2, dy, by)) != NF_OK) return rc;
  }
  FoldParams p{};
  if (bn) {
    p.bn_scale = bn->scale; p.bn_shift = bn->shift; p.bn_mu = bn->mu; p.bn_invstd = bn->invstd;
    p.bn_sdz = bn->sdz; p.bn_sdzx = bn->sdzx; p.inv_m = bn->inv_m;
  }
  p.N = N; p.H = H; p.W = W; p.Cout = Cout; p.kchunks = epi == 2 || Cin < 64 ? 1 : Cin / 64; p.n_tiles = epi == 2 ? Cout / 64 : 1;
  p.tiles_w = (W + TW - 1) / TW; p.tiles_h = (H + TH - 1) / TH; p.total_tiles = N * p.tiles_w * p.tiles_h * p.n_tiles;
  if ((long long)N * p.tiles_w * p.tiles_h * p.n_tiles > (1ll << 30)) return NF_EUNSUPPORTED;
  p.stats = stats; p.red = red; p.status = status; p.bias = bias; p.out = (bf16*)y;
  p.tg = tile_grid(p.n_tiles, p.tiles_w, p.tiles_h);
  const size_t a_bytes = wide ? ((size_t)34 * 10 * KC * 2 + 1023) / 1024 * 1024
                         : uf2 ? ((size_t)18 * 10 * KC * 2 + 1023) / 1024 * 1024 : (size_t)(uf ? 3 : 1) * 10 * 16 * KC * 2;
  const size_t wbytes = epi == 2 ? (size_t)9 * KC * 128 : (size_t)9 * p.kchunks * G * KC * 2;
  const size_t fixed = wide ? wbytes + (size_t)(stats >= 2 ? 2 + kWideYSlots : 2) * 32768 + 1024 + 1024
                            : wbytes + (epi != 1 ? (stats >= 2 ? 2 + kYSlots : 2) * 16384 : xf ? 3 * kXfGroups * 112 * 128 : 0) + 1024 + 1024;
  int st = (int)((232448 - fixed) / a_bytes);
  if (st > kMaxStages) st = kMaxStages;
  p.stages = st;
  const size_t smem = (size_t)st * a_bytes + fixed;
  int grid = sm_count();
  grid -= grid % p.n_tiles;  // a CTA keeps one output-channel tile (and its resident weights) for its whole life
  if (grid < p.n_tiles) grid = p.n_tiles;
  if (grid > p.total_tiles) grid = p.total_tiles;
  if (stats && stats != 4) {
    const size_t need = (size_t)(grid / p.n_tiles) * 2 * 2 * Cout;  // every CTA writes its two partials (one per epilogue group)
    if (need > red_floats) return NF_ENOWS;
    *nb = grid / p.n_tiles * 2;
  }
  if (xf) {
    if (epi != 1) return NF_EINVAL;
    p.xf_scale = xf->scale; p.xf_shift = xf->shift; p.xf_a = (bf16*)xf->a;
    p.pool_part = xf->pool_part; p.mask = xf->mask;
    return G == 16 ? launch_fold<16, 1, 64, 0, 0, 1>(grid, smem, mx, mw, my, my2, p)
                   : G == 32 ? launch_fold<32, 1, 64, 0, 0, 1>(grid, smem, mx, mw, my, my2, p)
                             : launch_fold<64, 1, 64, 0, 0, 1>(grid, smem, mx, mw, my, my2, p);
  }
  if (epi == 0 && bn)  // evaluation: normalised in the epilogue
    return KC == 16 ? launch_fold<64, 0, 16, 0, 0, 0, 1>(grid, smem, mx, mw, my, my2, p) : launch_fold<64, 0, 64, 0, 0, 0, 1>(grid, smem, mx, mw, my, my2, p);
  if (epi == 0 && KC == 16) return launch_fold<64, 0, 16>(grid, smem, mx, mw, my, my2, p);
  if (epi == 0) return launch_fold<64, 0>(grid, smem, mx, mw, my, my2, p);
  if (wide) {
    static bool attr_done_dev[kMaxDevices];
    bool& attr_done = attr_done_dev[current_device()];
    if (!attr_done) {
      NF_CUDA(cudaFuncSetAttribute(aux_dgrad_wide_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448));
      attr_done = true;
    }
    nf_launch(aux_dgrad_wide_kernel<16>, grid, kWideThreads, smem, mx, mw, my, my2, p);
    NF_LAUNCHED();
    return NF_OK;
  }
  if (epi == 2 && uf2)
    return KC == 16 ? launch_fold<64, 0, 16, 1, 2>(grid, smem, mx, mw, my, my2, p) : launch_fold<64, 0, 32, 1, 2>(grid, smem, mx, mw, my, my2, p);
  if (epi == 2 && uf)
    return KC == 16 ? launch_fold<64, 0, 16, 1, 1>(grid, smem, mx, mw, my, my2, p) : launch_fold<64, 0, 32, 1, 1>(grid, smem, mx, mw, my, my2, p);
  if (epi == 2)
    return KC == 16 ? launch_fold<64, 0, 16, 1>(grid, smem, mx, mw, my, my2, p) : launch_fold<64, 0, 32, 1>(grid, smem, mx, mw, my, my2, p);
  return G == 16 ? launch_fold<16, 1>(grid, smem, mx, mw, my, my2, p)
                 : G == 32 ? launch_fold<32, 1>(grid, smem, mx, mw, my, my2, p) : launch_fold<64, 1>(grid, smem, mx, mw, my, my2, p);
}

// epi 0: y through TMA + optional statistics.  epi 1: out = ReLU(conv + bias) written directly (y unused).
// H, W are the INPUT size; stride 2 halves them (rounding up) for the output.
int run_fwd(int N, int Hin, int Win, int Cin, int Cout, const void* x, const void* w, void* y, int stats, float* red,
            size_t red_floats, int32_t* status, int* nb, int epi = 0, const float* bias = nullptr, int stride = 1,
            const BnBwdIn* bn = nullptr, bool any_map = false) {
  const int H = (Hin - 1) / stride + 1, W = (Win - 1) / stride + 1;
  if (fold_ok(H, W, Cin, Cout, epi, stride, stats, 0, any_map))
    return run_fold(N, H, W, Cin, Cout, x, w, y, stats, red, red_floats, status, nb, epi, bias, bn);
  if (stats > 2) return NF_EUNSUPPORTED;  // the two-pass input gradient exists in the folded kernel only
  if (stats == 2 && (!bn || epi == 1)) return NF_EINVAL;
  const TcPlan pl = plan_fwd(H, W, Cin, Cout, N, epi, stride, stats == 2);
  if (!pl.ok) return NF_EUNSUPPORTED;
  CUtensorMap mx, mw, my;
  const bool hn = pl.PT == 2;
  const uint64_t dx[4] = {(uint64_t)Cin, (uint64_t)Win, (uint64_t)Hin, (uint64_t)N};
  const uint32_t bx[4] = {(uint32_t)pl.KC, (uint32_t)(pl.SB ? 10 : pl.BW), (uint32_t)(pl.PT == 1 ? pl.BH : pl.BH + 2), (uint32_t)pl.BI};
  // forward: weights [kh][kw][Cout][Cin] -> box of BN rows x 64 ci for three kh; input gradient: weights
  // [kh][kw][F][Cout] -> box of KC rows of f x 64 c for three kh
  const uint64_t dw[4] = {(uint64_t)(epi == 2 ? Cout : Cin), (uint64_t)(epi == 2 ? Cin : Cout), 3, 3};
  const uint32_t bw[4] = {64, (uint32_t)(epi == 2 ? pl.KC : pl.BN), hn || pl.SB ? 3u : 1u, (uint32_t)(pl.PT == 1 ? 1 : 3)};
  const uint64_t dy[4] = {(uint64_t)Cout, (uint64_t)W, (uint64_t)H, (uint64_t)N};
  const uint32_t by[4] = {64, (uint32_t)pl.BW, (uint32_t)pl.BH, (uint32_t)pl.BI};
  int rc;
  if ((rc = make_map4(&mx, x, dx, bx, stride, hn)) != NF_OK) return rc;
  if ((rc = make_map4(&mw, w, dw, bw)) != NF_OK) return rc;
  if (epi != 1 || pl.NS) {
    if ((rc = make_map4(&my, y, dy, by)) != NF_OK) return rc;
  } else {
    my = mx;  // not used by this epilogue
  }
  FwdParams p{};
  p.N = N; p.H = H; p.W = W; p.Cin = Cin; p.Cout = Cout;
  p.BW = pl.BW; p.BH = pl.BH; p.tiles_w = (W + pl.BW - 1) / pl.BW; p.tiles_h = (H + pl.BH - 1) / pl.BH; p.n_tiles = epi != 1 ? Cout / pl.BN : 1;
  p.bias = bias; p.out = (bf16*)y;
  p.total_tiles = ((N + pl.BI - 1) / pl.BI) * p.tiles_h * p.tiles_w * p.n_tiles;
  p.stride = stride; p.BI = pl.BI;
  p.tg = tile_grid(p.n_tiles, p.tiles_w, p.tiles_h);
  p.kchunks = epi == 2 ? 1 : Cin / 64;
  // An fp32 chain over 64 channels has only 576 roundings, one over 16 or 32 filters 144 or 288: segments of 64 (16 filters: 48)
  // products there, of 192 from 128 channels on.  Share of outputs off the nearest bf16 value, chain -> segments: 64 channels
  // 0.0078 -> 0.0064 %, 128 0.0118 -> 0.0105 %, 512 0.022 -> 0.012 %.
  p.seg_steps = pl.KC == 16 ? 3 : pl.KC == 32 ? 2 : p.kchunks == 1 ? 1 : 3;
  p.stages = pl.stages; p.stats = stats; p.red = red; p.status = status;
  p.yslots = pl.yslots;
  p.tm_y2 = my;
  if (stats == 0 && bn) {
    p.bn_scale = bn->scale; p.bn_shift = bn->shift;
  }
  if (stats == 2) {
    if ((rc = make_map4(&p.tm_y2, bn->y2, dy, by)) != NF_OK) return rc;
    p.bn_scale = bn->scale; p.bn_shift = bn->shift; p.bn_mu = bn->mu; p.bn_invstd = bn->invstd;
  }
  if (stats) {
    const int rows = pl.grid / p.n_tiles * pl.parts;
    if ((size_t)rows * 2 * Cout > red_floats) return NF_ENOWS;
    *nb = rows;
  }
  if (epi == 0 && stats == 0 && bn) {  // evaluation: normalised in the epilogue
    if (pl.SEG)
      return pl.BN == 128 ? launch_fwd<128, 0, 64, 0, 1, 0, 1, 1>(pl, mx, mw, my, p) : launch_fwd<64, 0, 64, 0, 1, 0, 1, 1>(pl, mx, mw, my, p);
    if (pl.PT)
      return pl.BN == 256 ? launch_fwd<256, 0, 64, 0, 1, 0, 0, 1, 0, 1>(pl, mx, mw, my, p)
           : pl.BN == 128 ? launch_fwd<128, 0, 64, 0, 1, 0, 0, 1>(pl, mx, mw, my, p) : launch_fwd<64, 0, 64, 0, 1, 0, 0, 1>(pl, mx, mw, my, p);
    if (pl.RW) return launch_fwd<64, 0, 64, 0, 0, 1, 0, 1>(pl, mx, mw, my, p);
    return pl.BN == 128 ? launch_fwd<128, 0, 64, 0, 0, 0, 0, 1>(pl, mx, mw, my, p) : launch_fwd<64, 0, 64, 0, 0, 0, 0, 1>(pl, mx, mw, my, p);
  }
  if (pl.SEG) {  // maps that no tile divides
    if (epi == 0) return pl.BN == 128 ? launch_fwd<128, 0, 64, 0, 1, 0, 1>(pl, mx, mw, my, p) : launch_fwd<64, 0, 64, 0, 1, 0, 1>(pl, mx, mw, my, p);
    if (epi == 2 && pl.BN == 128)
      return pl.KC == 16 ? launch_fwd<128, 0, 16, 1, 1, 0, 1>(pl, mx, mw, my, p)
                         : pl.KC == 32 ? launch_fwd<128, 0, 32, 1, 1, 0, 1>(pl, mx, mw, my, p) : launch_fwd<128, 0, 64, 1, 1, 0, 1>(pl, mx, mw, my, p);
    if (epi == 2)
      return pl.KC == 16 ? launch_fwd<64, 0, 16, 1, 1, 0, 1>(pl, mx, mw, my, p)
                         : pl.KC == 32 ? launch_fwd<64, 0, 32, 1, 1, 0, 1>(pl, mx, mw, my, p) : launch_fwd<64, 0, 64, 1, 1, 0, 1>(pl, mx, mw, my, p);
    return pl.BN == 16 ? launch_fwd<16, 1, 64, 0, 1, 0, 1>(pl, mx, mw, my, p)
                       : pl.BN == 32 ? launch_fwd<32, 1, 64, 0, 1, 0, 1>(pl, mx, mw, my, p) : launch_fwd<64, 1, 64, 0, 1, 0, 1>(pl, mx, mw, my, p);
  }
  if (pl.NS && epi == 1)  // 64 filters: the outputs leave as a main convolution's do
    return pl.RW ? launch_fwd<64, 0, 64, 0, 0, 1, 0, 0, 0, 1>(pl, mx, mw, my, p) : launch_fwd<64, 0, 64, 0, 0, 0, 0, 0, 0, 1>(pl, mx, mw, my, p);
  if (pl.SB && epi == 1) {
    if (pl.BN == 16) return pl.RW ? launch_fwd<16, 1, 64, 0, 0, 1, 0, 0, 1>(pl, mx, mw, my, p) : launch_fwd<16, 1, 64, 0, 0, 0, 0, 0, 1>(pl, mx, mw, my, p);
    return pl.RW ? launch_fwd<32, 1, 64, 0, 0, 1, 0, 0, 1>(pl, mx, mw, my, p) : launch_fwd<32, 1, 64, 0, 0, 0, 0, 0, 1>(pl, mx, mw, my, p);
  }
  if (pl.SB) {
    if (pl.BN == 128)
      return pl.KC == 16 ? launch_fwd<128, 0, 16, 1, 0, 1, 0, 0, 1, 1>(pl, mx, mw, my, p)
                         : pl.KC == 32 ? launch_fwd<128, 0, 32, 1, 0, 1, 0, 0, 1, 1>(pl, mx, mw, my, p) : NF_EUNSUPPORTED;
    return pl.KC == 16 ? launch_fwd<64, 0, 16, 1, 0, 1, 0, 0, 1, 1>(pl, mx, mw, my, p)
                       : pl.KC == 32 ? launch_fwd<64, 0, 32, 1, 0, 1, 0, 0, 1, 1>(pl, mx, mw, my, p) : launch_fwd<64, 0, 64, 1, 0, 1, 0, 0, 1, 1>(pl, mx, mw, my, p);
  }
  if (pl.PT == 2) {
    if (epi == 1) return pl.BN == 16 ? launch_fwd<16, 1, 64, 0, 2>(pl, mx, mw, my, p) : launch_fwd<32, 1, 64, 0, 2>(pl, mx, mw, my, p);
    return pl.BN == 128 ? launch_fwd<128, 0, 16, 1, 2, 1>(pl, mx, mw, my, p) : launch_fwd<64, 0, 16, 1, 2, 1>(pl, mx, mw, my, p);
  }
  if (pl.PT) {  // per-tap boxes: stride 2, or several small images per tile
    if (epi == 0)
      return pl.BN == 256 ? (stats ? launch_fwd<256, 0, 64, 0, 1>(pl, mx, mw, my, p) : launch_fwd<256, 0, 64, 0, 1, 0, 0, 0, 0, 1>(pl, mx, mw, my, p))
                          : pl.BN == 128 ? launch_fwd<128, 0, 64, 0, 1>(pl, mx, mw, my, p) : launch_fwd<64, 0, 64, 0, 1>(pl, mx, mw, my, p);
    if (epi == 1)
      return pl.BN == 16 ? launch_fwd<16, 1, 64, 0, 1>(pl, mx, mw, my, p)
                         : pl.BN == 32 ? launch_fwd<32, 1, 64, 0, 1>(pl, mx, mw, my, p) : launch_fwd<64, 1, 64, 0, 1>(pl, mx, mw, my, p);
    if (pl.BN == 128)
      return pl.KC == 16 ? launch_fwd<128, 0, 16, 1, 1>(pl, mx, mw, my, p)
                         : pl.KC == 32 ? launch_fwd<128, 0, 32, 1, 1>(pl, mx, mw, my, p) : launch_fwd<128, 0, 64, 1, 1>(pl, mx, mw, my, p);
    return pl.KC == 16 ? launch_fwd<64, 0, 16, 1, 1>(pl, mx, mw, my, p)
                       : pl.KC == 32 ? launch_fwd<64, 0, 32, 1, 1>(pl, mx, mw, my, p) : launch_fwd<64, 0, 64, 1, 1>(pl, mx, mw, my, p);
  }
  if (epi == 0 && pl.RW) return launch_fwd<64, 0, 64, 0, 0, 1>(pl, mx, mw, my, p);
  if (epi == 0) return pl.BN == 128 ? launch_fwd<128, 0>(pl, mx, mw, my, p) : launch_fwd<64, 0>(pl, mx, mw, my, p);
  if (epi == 1 && pl.RW)
    return pl.BN == 16 ? launch_fwd<16, 1, 64, 0, 0, 1>(pl, mx, mw, my, p)
                       : pl.BN == 32 ? launch_fwd<32, 1, 64, 0, 0, 1>(pl, mx, mw, my, p) : launch_fwd<64, 1, 64, 0, 0, 1>(pl, mx, mw, my, p);
  if (epi == 2) {
    if (pl.BN == 128)
      return pl.KC == 16 ? launch_fwd<128, 0, 16, 1>(pl, mx, mw, my, p)
                         : pl.KC == 32 ? launch_fwd<128, 0, 32, 1>(pl, mx, mw, my, p) : launch_fwd<128, 0, 64, 1>(pl, mx, mw, my, p);
    return pl.KC == 16 ? launch_fwd<64, 0, 16, 1>(pl, mx, mw, my, p)
                       : pl.KC == 32 ? launch_fwd<64, 0, 32, 1>(pl, mx, mw, my, p) : launch_fwd<64, 0, 64, 1>(pl, mx, mw, my, p);
  }
  return pl.BN == 16 ? launch_fwd<16, 1>(pl, mx, mw, my, p)
                     : pl.BN == 32 ? launch_fwd<32, 1>(pl, mx, mw, my, p) : launch_fwd<64, 1>(pl, mx, mw, my, p);
}

struct WgPlan {
  int ok, exact, BW, BH, BI, PT, SEG, NB, GX, ROW, HB, splits, grid, stages;  // ROW: input-channel chunks per CTA of the row kernel, or 0
  size_t smem, part_floats;
};

// Pixel splits for `units` CTAs per split (channel chunk pairs x kernel rows or columns): the count whose CTAs fill whole waves of
// SMs best (smallest on ties), e.g. 512 -> 512 channels with three row groups: 192 units -> 3 splits = 576 CTAs = 3.9 waves
// instead of 1.3
long wgrad_splits(int units, long pix_tiles) {
  const int sms = sm_count();
  long base = sms / units;
  if (base < 1) base = 1;
  long sp = base;
  double best = 0.0;
  for (long c = 1; c <= (base * 2 > 16 ? base * 2 : 16) && c <= pix_tiles; ++c) {
    const long total = c * units, waves = (total + sms - 1) / sms;
    const double eff = (double)total / (double)(waves * sms);
    if (eff > best + 1e-9) {
      best = eff;
      sp = c;
    }
  }
  return sp > pix_tiles ? pix_tiles : sp;
}

// aux = 0: main conv (Cout a multiple of 64).  aux = 1: aux conv (Cout = F <= 64, a multiple of 8).
// H, W: size of the gradient tensor (the conv OUTPUT; equals the input size for stride 1).
WgPlan plan_wgrad(int H, int W, int Cin, int Cout, int N, int aux = 0, int stride = 1) {
  WgPlan pl{};
  if (Cin % 64 || (stride == 2 && aux)) return pl;
  if (aux ? (Cout > 64 || Cout % 8) : (Cout % 64 != 0)) return pl;
  pl.exact = pick_tile(N, H, W, &pl.BW, &pl.BH, &pl.BI);
  pl.PT = (stride == 2 || pl.BI > 1 || !pl.exact) ? 1 : 0;
  pl.NB = aux ? (Cout <= 16 ? 16 : Cout <= 32 ? 32 : 64) : 64;
  // maps that no tile divides: segments of 32 pixels, of 16 below 8192 pixels, where the chains to compare with are shorter
  pl.SEG = pl.exact ? 0 : (long)N * H * W < 8192 ? 1 : 2;
  if (!aux && pl.PT && !pl.SEG) pl.NB = Cout % 256 == 0 ? 256 : Cout % 128 == 0 ? 128 : 64;  // per-tap form: as wide an instruction as Cout allows
  pl.GX = (aux && !pl.PT && pl.NB <= 32) ? 1 : 0;  // few filters: one instruction per 16 pixels with the gradient on the M side
  const long pix_tiles = (long)((N + pl.BI - 1) / pl.BI) * ((H + pl.BH - 1) / pl.BH) * ((W + pl.BW - 1) / pl.BW);
  if (pix_tiles >= (1l << 30)) return pl;
  int units = (Cin / 64) * (aux ? 1 : Cout / pl.NB) * (pl.PT ? 3 : 1);
  long sp = wgrad_splits(units, pix_tiles);
  pl.part_floats = (size_t)sp * 9 * Cout * Cin;
  // 128 output channels: the form without an idle half, wherever 16 pixels of a tile are consecutive in one image.  The splits are
  // those of the other forms, so that every sum runs over the same pixels in the same order and the bits stay what they were; of one
  // or two chunks of input channels per CTA the one whose CTAs fill their waves better (two on near ties: less to fetch).
  const size_t box = (size_t)pl.BI * (pl.BH + 2) * pl.BW * 128;
  if (!aux && !pl.SEG && stride == 1 && Cout % 128 == 0 && pl.BW >= 4 && pl.BW * pl.BH % 16 == 0) {
    // single-image tiles with one chunk only: the form above has as little to fetch and fills its wave (64 -> 128 channels at 32x32)
    double best = pl.PT || Cin % 128 == 0 ? 0.0 : 0.75;
    for (int cc = Cin % 128 == 0 ? 2 : 1; cc >= 1; --cc) {
      if (2 * (cc * box + 32768) > 232448 - 2048) continue;  // two stages have to fit
      const long u = Cin / 64 / cc * (Cout / 128) * 3, ctas = u * sp, waves = (ctas + sm_count() - 1) / sm_count();
      const double eff = (double)ctas / (double)(waves * sm_count());
      if (eff > best + 0.1) {
        best = eff;
        pl.ROW = cc;
        pl.NB = 128;
        units = (int)u;
      }
    }
  }
  pl.HB = aux && stride == 1 && pl.PT && !pl.SEG && !pl.ROW && pl.BW == 8 && W == 8;  // (a main convolution there takes the row form)
  size_t g_region = (size_t)(pl.GX ? 4 : 3) * 128 * pl.NB * 2;
  if (g_region < 4096) g_region = 4096;
  const size_t stage = pl.ROW ? pl.ROW * box + 32768
                     : pl.HB ? (size_t)20480 + 16384
                     : pl.PT ? (size_t)49152 + (pl.NB > 64 ? pl.NB / 64 : 1) * 16384 : (size_t)(pl.BH + 2) * pl.BW * 128 + g_region;
  pl.stages = pl.PT && !pl.ROW ? (pl.NB > 64 ? 2 : pl.HB ? 5 : 3) : (int)((232448 - 2048) / stage);
  if (pl.stages > kMaxStages) pl.stages = kMaxStages;
  if (pl.stages < 2) return pl;
  pl.smem = (size_t)pl.stages * stage + 1024 + 1024;
  if (pl.smem > 232448) return pl;
  pl.splits = (int)sp;
  pl.grid = (int)(sp * units);
  pl.ok = 1;
  return pl;
}

template <int NB>
int launch_wgrad_kw(const WgPlan& pl, const CUtensorMap& mx, const CUtensorMap& mg, const WgParams& p) {
  static bool attr_done_dev[kMaxDevices];  // function attributes belong to a device's context: set once per device
  bool& attr_done = attr_done_dev[current_device()];
  if (!attr_done) {
    NF_CUDA(cudaFuncSetAttribute(conv_wgrad_kw_kernel<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448));
    attr_done = true;
  }
  nf_launch(conv_wgrad_kw_kernel<NB>, pl.grid, kThreads, pl.smem, mx, mg, p);
  NF_LAUNCHED();
  return NF_OK;
}

template <int CC>
int launch_wgrad_row(const WgPlan& pl, const CUtensorMap& mx, const CUtensorMap& mg, const WgParams& p) {
  static bool attr_done_dev[kMaxDevices];  // function attributes belong to a device's context: set once per device
  bool& attr_done = attr_done_dev[current_device()];
  if (!attr_done) {
    NF_CUDA(cudaFuncSetAttribute(conv_wgrad_row_kernel<CC>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448));
    attr_done = true;
  }
  nf_launch(conv_wgrad_row_kernel<CC>, pl.grid, kThreads, pl.smem, mx, mg, p);
  NF_LAUNCHED();
  return NF_OK;
}

template <int NB>
int launch_wgrad_gx(const WgPlan& pl, const CUtensorMap& mx, const CUtensorMap& mg, const WgParams& p) {
  static bool attr_done_dev[kMaxDevices];  // function attributes belong to a device's context: set once per device
  bool& attr_done = attr_done_dev[current_device()];
  if (!attr_done) {
    NF_CUDA(cudaFuncSetAttribute(conv_wgrad_gx_kernel<NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448));
    attr_done = true;
  }
  nf_launch(conv_wgrad_gx_kernel<NB>, pl.grid, kThreads, pl.smem, mx, mg, p);
  NF_LAUNCHED();
  return NF_OK;
}

template <int NB, int SEG, int HB = 0>
int launch_wgrad(const WgPlan& pl, const CUtensorMap& mx, const CUtensorMap& mg, const WgParams& p) {
  static bool attr_done_dev[kMaxDevices];  // function attributes belong to a device's context: set once per device
  bool& attr_done = attr_done_dev[current_device()];
  if (!attr_done) {
    NF_CUDA(cudaFuncSetAttribute(conv_wgrad_tc_kernel<NB, SEG, HB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448));
    attr_done = true;
  }
  nf_launch(conv_wgrad_tc_kernel<NB, SEG, HB>, pl.grid, wgrad_threads(SEG), pl.smem, mx, mg, p);
  NF_LAUNCHED();
  return NF_OK;
}

// Hin, Win: INPUT size; the gradient tensor has the strided output size.
int run_wgrad(int N, int Hin, int Win, int Cin, int Cout, const void* x, const void* dy, float* part, size_t part_floats,
              float* dw, int32_t* status, int aux = 0, int stride = 1) {
  const int H = (Hin - 1) / stride + 1, W = (Win - 1) / stride + 1;
  const WgPlan pl = plan_wgrad(H, W, Cin, Cout, N, aux, stride);
  if (!pl.ok) return NF_EUNSUPPORTED;
  if (pl.part_floats > part_floats) return NF_ENOWS;
  CUtensorMap mx, mg;
  const uint64_t dx[4] = {(uint64_t)Cin, (uint64_t)Win, (uint64_t)Hin, (uint64_t)N};
  const uint32_t bx[4] = {64, (uint32_t)(pl.HB ? 10 : pl.BW), (uint32_t)(pl.PT && !pl.ROW ? pl.BH : pl.BH + 2), (uint32_t)pl.BI};
  const uint64_t dg[4] = {(uint64_t)Cout, (uint64_t)W, (uint64_t)H, (uint64_t)N};
  const uint32_t bg[4] = {(uint32_t)(pl.NB > 64 ? 64 : pl.NB), (uint32_t)pl.BW, (uint32_t)pl.BH, (uint32_t)pl.BI};
  int rc;
  if ((rc = make_map4(&mx, x, dx, bx, stride)) != NF_OK) return rc;
  if ((rc = make_map4(&mg, dy, dg, bg)) != NF_OK) return rc;
  WgParams p{};
  p.N = N; p.H = H; p.W = W; p.Cin = Cin; p.Cout = Cout; p.BW = pl.BW; p.BH = pl.BH;
  p.tiles_w = (W + pl.BW - 1) / pl.BW; p.tiles_h = (H + pl.BH - 1) / pl.BH; p.pix_tiles = ((N + pl.BI - 1) / pl.BI) * p.tiles_h * p.tiles_w;
  p.stride = stride; p.BI = pl.BI;
  p.tg = tile_grid(1, p.tiles_w, p.tiles_h);
  p.ci_chunks = pl.ROW ? Cin / 64 / pl.ROW : Cin / 64; p.co_chunks = aux ? 1 : Cout / pl.NB; p.splits = pl.splits; p.part = part; p.status = status;
  p.stages = pl.stages;
  p.dy_shift = !pl.PT;
  if (pl.ROW)
    rc = pl.ROW == 2 ? launch_wgrad_row<2>(pl, mx, mg, p) : launch_wgrad_row<1>(pl, mx, mg, p);
  else if (pl.GX)
    rc = pl.NB == 32 ? launch_wgrad_gx<32>(pl, mx, mg, p) : launch_wgrad_gx<16>(pl, mx, mg, p);
  else if (pl.SEG == 1)
    rc = pl.NB == 64 ? launch_wgrad<64, 1>(pl, mx, mg, p) : pl.NB == 32 ? launch_wgrad<32, 1>(pl, mx, mg, p) : launch_wgrad<16, 1>(pl, mx, mg, p);
  else if (pl.SEG)
    rc = pl.NB == 64 ? launch_wgrad<64, 2>(pl, mx, mg, p) : pl.NB == 32 ? launch_wgrad<32, 2>(pl, mx, mg, p) : launch_wgrad<16, 2>(pl, mx, mg, p);
  else if (pl.HB)
    rc = pl.NB == 64 ? launch_wgrad<64, 0, 1>(pl, mx, mg, p) : pl.NB == 32 ? launch_wgrad<32, 0, 1>(pl, mx, mg, p) : launch_wgrad<16, 0, 1>(pl, mx, mg, p);
  else if (pl.PT)
    rc = pl.NB == 256 ? launch_wgrad<256, 0>(pl, mx, mg, p) : pl.NB == 128 ? launch_wgrad<128, 0>(pl, mx, mg, p)
       : pl.NB == 64 ? launch_wgrad<64, 0>(pl, mx, mg, p) : pl.NB == 32 ? launch_wgrad<32, 0>(pl, mx, mg, p) : launch_wgrad<16, 0>(pl, mx, mg, p);
  else
    rc = launch_wgrad_kw<64>(pl, mx, mg, p);  // up to 32 filters take the form above
  if (rc != NF_OK) return rc;
  const size_t n = (size_t)9 * Cout * Cin;
  return nf_k_sum_parts(part, pl.splits, n, dw, pl.SEG != 0);
}

}  // namespace

// The classic local-learning setting (256 auxiliary filters) and the paper's own rule for late layers give F > 64.
// Then the aux conv is as wide as a main conv and uses the same three kernels: forward (bias and ReLU in its epilogue),
// weight gradient, and the input gradient written as a forward conv over a mirrored, transposed weight copy.
static bool wide_aux(const nf_layer* L) { return L->F > 64 && L->F % 64 == 0; }

void nf_tc_select(nf_layer* L) {
  L->fam[0] = L->fam[1] = L->fam[2] = L->fam[3] = L->dgrad_tc = 0;
  L->cin_pad = 0;
  if (L->o.dtype != NF_BF16) return;
  // A first layer with a handful of input channels (RGB) is far too thin a contraction for useful tensor-core work (K = 27),
  // but its CUDA-core kernels reach under a tenth of the memory bandwidth, and the tensor cores are idle anyway: the input
  // batch is copied once per step into a zero-padded tensor whose pixels TMA can address, and the main conv runs on the ordinary
  // kernels.  16 channels where the folded forward and the narrow weight gradient cover the shape (64 output channels; VGG first
  // layer at 64 x 64, 1260 images: copy + forward 636 -> 300 us against 64 channels), else 64.
  const bool main_ok = tc_size_ok(L->o.N, L->Ho, L->Wo), aux_ok = tc_size_ok(L->o.N, L->Ha, L->Wa);
  if (L->Cin <= 8 && main_ok) {
    if (fold_ok(L->Ho, L->Wo, 16, L->Cout, 0, L->o.stride) && plan_wgrad(L->Ho, L->Wo, L->Cout, 16, L->o.N, 1).ok)
      L->cin_pad = 16;
    else if (plan_fwd(L->Ho, L->Wo, 64, L->Cout, L->o.N, 0, L->o.stride).ok && plan_wgrad(L->Ho, L->Wo, 64, L->Cout, L->o.N, 0, L->o.stride).ok)
      L->cin_pad = 64;
  }
  const int Cin = L->cin_pad ? L->cin_pad : L->Cin;
  if (L->cin_pad == 16) L->fam[0] = L->fam[1] = 1;
  if (main_ok && plan_fwd(L->Ho, L->Wo, Cin, L->Cout, L->o.N, 0, L->o.stride).ok) L->fam[0] = 1;
  if (plan_wgrad(L->Ho, L->Wo, Cin, L->Cout, L->o.N, 0, L->o.stride).ok) L->fam[1] = 1;
  if (wide_aux(L)) {  // more than 64 filters: the aux conv runs on the kernels of the main conv
    if (aux_ok && plan_fwd(L->Ha, L->Wa, L->Cout, L->F, L->o.N, 0).ok) L->fam[2] = 1;
    if (plan_wgrad(L->Ha, L->Wa, L->Cout, L->F, L->o.N, 0).ok && plan_fwd(L->Ha, L->Wa, L->F, L->Cout, L->o.N, 0).ok) L->fam[3] = 1;
    L->dgrad_tc = L->fam[3] && aux_ok;
    return;
  }
  if (aux_ok && plan_fwd(L->Ha, L->Wa, L->Cout, L->F, L->o.N, 1).ok) L->fam[2] = 1;
  if (plan_wgrad(L->Ha, L->Wa, L->Cout, L->F, L->o.N, 1).ok && plan_fwd(L->Ha, L->Wa, L->F, L->Cout, L->o.N, 2).ok) L->fam[3] = 1;
  L->dgrad_tc = L->fam[3] && aux_ok;
}

size_t nf_tc_scratch_floats(const nf_layer* L) {
  const size_t a = L->cin_pad == 16 ? plan_wgrad(L->Ho, L->Wo, L->Cout, 16, L->o.N, 1).part_floats : L->fam[1] ? plan_wgrad(L->Ho, L->Wo, L->cin_pad ? L->cin_pad : L->Cin, L->Cout, L->o.N, 0, L->o.stride).part_floats : 0;
  const size_t b = L->fam[3] ? plan_wgrad(L->Ha, L->Wa, L->Cout, L->F, L->o.N, wide_aux(L) ? 0 : 1).part_floats : 0;
  return a > b ? a : b;
}

size_t nf_tc_red_floats(const nf_layer* L) {
  size_t need = 0;
  if (L->fam[3]) need = (size_t)sm_count() * 8 * 2 * L->Cout;  // input-gradient kernel with the fused BatchNorm-backward sums
  if (!L->fam[0]) return need;
  const TcPlan pl = plan_fwd(L->Ho, L->Wo, L->cin_pad ? L->cin_pad : L->Cin, L->Cout, L->o.N, 0, L->o.stride);
  const size_t fwd = (size_t)sm_count() * (pl.parts < 8 ? 8 : pl.parts) * 2 * L->Cout;  // room for 8 partials per CTA; the folded kernel writes 2
  return fwd > need ? fwd : need;
}

// input and operand weights of the main conv: the caller's, or their zero-padded copies of 16 or 64 channels (refreshed here)
static int main_conv_operands(nf_layer* L, const void* x, int count, const void** xin, const void** win, int* Cin) {
  *xin = x;
  *win = L->shadow + L->off[NF_P_W];
  *Cin = L->Cin;
  if (!L->cin_pad) return NF_OK;
  int rc = nf_k_pad_channels(x, (size_t)count * L->H * L->W, L->Cin, L->cin_pad, L->xpad);
  if (rc != NF_OK) return rc;
  if ((rc = nf_k_pad_weights(L->shadow + L->off[NF_P_W], (size_t)9 * L->Cout, L->Cin, L->cin_pad, L->wpad)) != NF_OK) return rc;
  *xin = L->xpad;
  *win = L->wpad;
  *Cin = L->cin_pad;
  return NF_OK;
}

// On maps that no tile divides the statistics (and in the input gradient the BatchNorm-backward sums) are left to the passes of the
// CUDA-core path: the fused sums run in chains of a CTA's whole pixel range, the second ones in the form sum(dz*y) - mu*sum(dz),
// which cost a factor of up to 5 in the error of a normalised activation's rounding and of 2 to 30 in that of sum(dz*xhat).
int nf_tc_conv_fwd(nf_layer* L, const void* x, int& nb) {
  const void *xin, *win;
  int Cin;
  const int rc = main_conv_operands(L, x, L->o.N, &xin, &win, &Cin);
  if (rc != NF_OK) return rc;
  nb = 0;
  return run_fwd(L->o.N, L->H, L->W, Cin, L->Cout, xin, win, L->y, tiles_exactly(L->Ho, L->Wo), L->red, L->red_floats, L->status, &nb, 0,
                 nullptr, L->o.stride);
}

int nf_tc_conv_fwd_eval(nf_layer* L, const void* x, int count, void* act) {
  if (act && nf_first_eval_ok(L, x, count, act)) return nf_first_eval(L, x, count, act);
  int nb = 0, Cin;
  const void *xin, *win;
  const int rc = main_conv_operands(L, x, count, &xin, &win, &Cin);
  if (rc != NF_OK) return rc;
  const BnBwdIn bn{nullptr, L->scale, L->shift, nullptr, nullptr};
  return run_fwd(count, L->H, L->W, Cin, L->Cout, xin, win, act ? act : L->y, 0, nullptr, 0, L->status, &nb, 0, nullptr, L->o.stride,
                 act ? &bn : nullptr);
}

int nf_tc_aux_fwd(nf_layer* L, const void* a, int count) {
  int nb = 0;
  if (wide_aux(L)) {
    return run_fwd(count, L->Ha, L->Wa, L->Cout, L->F, a, L->shadow + L->off[NF_P_WA], L->h, 0, nullptr, 0, L->status, &nb, 0,
                   L->val + L->off[NF_P_BA]);
  }
  return run_fwd(count, L->Ha, L->Wa, L->Cout, L->F, a, L->shadow + L->off[NF_P_WA], L->h, 0, nullptr, 0, L->status, &nb, 1,
                 L->val + L->off[NF_P_BA]);
}

bool nf_tc_bn_aux_fused(const nf_layer* L) {
  // beside the weights and three activation stages the kernel then also holds three staging tiles of a.  On widths that are
  // no multiple of 14 (ragged last tile column) only for up to 32 filters: with 64 the wide shift-add epilogue ate the gain
  // (32 x 32 maps, 64 filters: aux forward + normalisation 0.174 ms separate, 0.197 ms fused).
  if (L->Wa % 14 != 0 && L->F > 32) return false;
  return L->fam[2] && !wide_aux(L) && !L->o.maxpool && fold_ok(L->Ha, L->Wa, L->Cout, L->F, 1, 1, 0, 3 * kXfGroups * 112 * 128);
}

// The fused aux forward can also keep h out of memory when the head pools by averaging and no tile straddles a pooling
// quadrant (14 x 8-pixel tiles: Ha/2 a multiple of 8, Wa/2 of 14): the epilogue then emits pooling partials and a sign mask.
bool nf_tc_aux_pool_fused(const nf_layer* L) {
  return nf_tc_bn_aux_fused(L) && L->o.aux_pool == NF_POOL_AVG && (L->Ha / 2) % 8 == 0 && (L->Wa / 2) % 14 == 0 && L->Ha % 2 == 0 &&
         L->Wa % 2 == 0 && (size_t)L->o.N * L->Ha * L->Wa < ((size_t)1 << 31);
}

size_t nf_tc_pool_part_floats(const nf_layer* L) {
  return (size_t)L->o.N * (L->Wa / 14) * (L->Ha / 8) * 4 * L->F;
}

int nf_tc_bn_aux_fwd(nf_layer* L, void* act_out) {
  if (!nf_tc_bn_aux_fused(L) || L->skip) return NF_EUNSUPPORTED;
  int nb = 0;
  const bool pooled = nf_tc_aux_pool_fused(L);
  // the partials live in the split-K scratch (free until the weight gradients), the mask in the unused h buffer
  const XfIn xf{L->scale, L->shift, act_out, pooled ? L->wpart : nullptr, pooled ? (uint8_t*)L->h : nullptr};
  return run_fold(L->o.N, L->Ha, L->Wa, L->Cout, L->F, L->y, L->shadow + L->off[NF_P_WA], L->h, 0, nullptr, 0, L->status, &nb, 1,
                  L->val + L->off[NF_P_BA], nullptr, &xf);
}

int nf_tc_wgrad(nf_layer* L, const void* x) {
  if (L->cin_pad) {  // the padded copy of this step's input is still in place (the forward made it); x itself is not read again
    // 16 channels: the roles of input and gradient are exchanged, so that the narrow tensor takes the narrow side of the auxiliary
    // weight gradient: with i' = i + kh - 1 the sum runs over the input's pixels and the gradient is shifted by 1 - kh, which gives
    // [8 - tap][ci][co]
    const bool narrow = L->cin_pad == 16;
    const int rc = narrow ? run_wgrad(L->o.N, L->H, L->W, L->Cout, 16, L->dy, L->xpad, L->wpart, L->wpart_floats, L->gwpad, L->status, 1)
                          : run_wgrad(L->o.N, L->H, L->W, L->cin_pad, L->Cout, L->xpad, L->dy, L->wpart, L->wpart_floats, L->gwpad, L->status, 0,
                                      L->o.stride);
    if (rc != NF_OK) return rc;
    return narrow ? nf_k_unpad_grad_mirrored(L->gwpad, L->Cout, L->Cin, 16, L->grad + L->off[NF_P_W])
                  : nf_k_unpad_grad(L->gwpad, (size_t)9 * L->Cout, L->Cin, L->cin_pad, L->grad + L->off[NF_P_W]);
  }
  return run_wgrad(L->o.N, L->H, L->W, L->Cin, L->Cout, x, L->dy, L->wpart, L->wpart_floats, L->grad + L->off[NF_P_W],
                   L->status, 0, L->o.stride);
}

// Two-pass form of the input gradient (folded kernel, no pool, no shortcut, fewer than 64 aux filters): the first pass only
// reduces the BatchNorm-backward sums, the second (nf_tc_aux_dgrad_dy, after the sums have been finished) forms da again and
// writes dy = BatchNorm-backward(da) directly, so da is never stored and the separate apply pass (read y and da, write dy)
// disappears: 1.75 activation-sized tensors less memory traffic per layer step for one more read of the narrow dh.
bool nf_tc_dgrad_two_pass(const nf_layer* L) {
  return L->dgrad_tc && !wide_aux(L) && !L->o.maxpool && fold_ok(L->Ha, L->Wa, L->F, L->Cout, 2, 1, 3) &&
         (size_t)(sm_count() / (L->Cout / 64)) * 8 * 2 * L->Cout <= L->red_floats;
}

int nf_tc_aux_dgrad_dy(nf_layer* L, double M) {
  if (!nf_tc_dgrad_two_pass(L) || L->skip || L->skip_grad) return NF_EUNSUPPORTED;
  int nb = 0;
  BnBwdIn bn{L->y, L->scale, L->shift, L->mu, L->invstd};
  bn.sdz = L->sdz; bn.sdzx = L->sdzx; bn.inv_m = (float)(1.0 / M);
  return run_fwd(L->o.N, L->Ha, L->Wa, L->F, L->Cout, L->dh, L->shadow + L->off[NF_P_WA], L->dy, 4, nullptr, 0, L->status, &nb, 2,
                 nullptr, 1, &bn);
}

int nf_tc_aux_dgrad(nf_layer* L, int* bn_nb) {
  int nb = 0;
  *bn_nb = 0;
  if (nf_tc_dgrad_two_pass(L) && !L->skip && !L->skip_grad) {  // first pass: sums only, nothing stored
    const BnBwdIn bn{L->y, L->scale, L->shift, L->mu, L->invstd};
    return run_fwd(L->o.N, L->Ha, L->Wa, L->F, L->Cout, L->dh, L->shadow + L->off[NF_P_WA], L->da, 3, L->red, L->red_floats, L->status,
                   bn_nb, 2, nullptr, 1, &bn);
  }
  const bool wide = wide_aux(L);
  const void* w = L->shadow + L->off[NF_P_WA];
  if (wide) {
    const int rc = nf_k_flip_weights(L->shadow + L->off[NF_P_WA], L->F, L->Cout, L->wa_t);
    if (rc != NF_OK) return rc;
    w = L->wa_t;
  }
  const int epi = wide ? 0 : 2;
  // Without a pool (and without a shortcut) da has the shape of y, and the kernel that produces it also reduces
  // (dz, dz*xhat) per channel while it holds the tile: the BatchNorm backward then needs no reduction pass.
  if (!L->o.maxpool && !L->skip && tiles_exactly(L->Ha, L->Wa)) {
    const BnBwdIn bn{L->y, L->scale, L->shift, L->mu, L->invstd};
    bool fits;
    if (fold_ok(L->Ha, L->Wa, L->F, L->Cout, epi, 1, 2)) {
      fits = (size_t)(sm_count() / (L->Cout / 64)) * 8 * 2 * L->Cout <= L->red_floats;
    } else {
      const TcPlan pl = plan_fwd(L->Ha, L->Wa, L->F, L->Cout, L->o.N, epi, 1, 1);
      fits = pl.ok && (size_t)pl.grid * pl.parts * 2 * L->Cout <= L->red_floats;
    }
    if (fits)
      return run_fwd(L->o.N, L->Ha, L->Wa, L->F, L->Cout, L->dh, w, L->da, 2, L->red, L->red_floats, L->status, bn_nb, epi, nullptr,
                     1, &bn);
  }
  return run_fwd(L->o.N, L->Ha, L->Wa, L->F, L->Cout, L->dh, w, L->da, 0, nullptr, 0, L->status, &nb, epi);
}

int nf_tc_aux_wgrad(nf_layer* L, const void* a) {
  return run_wgrad(L->o.N, L->Ha, L->Wa, L->Cout, L->F, a, L->dh, L->wpart, L->wpart_floats, L->grad + L->off[NF_P_WA],
                   L->status, wide_aux(L) ? 0 : 1);
}

// The stand-alone weight gradient takes maps that no tile divides only where its split partials need no more scratch than the
// CUDA-core kernel would, or fit the library's own array: what a caller's scratch was enough for stays accepted.
static bool standalone_wgrad_ok(int N, int Ho, int Wo, int Cin, int Cout, const WgPlan& pl) {
  const size_t limit = std::max((size_t)nf_k_wgrad_splits(N, Ho, Cin, Cout) * 9 * Cout * Cin, (size_t)NF_STATIC_SCRATCH_BYTES / sizeof(float));
  return pl.ok && (pl.exact || pl.part_floats <= limit);
}

size_t nf_tc_conv3x3_wgrad_scratch_floats(int N, int H, int W, int Cin, int Cout, int stride) {
  const int Ho = (H - 1) / stride + 1, Wo = (W - 1) / stride + 1;
  const WgPlan pl = plan_wgrad(Ho, Wo, Cin, Cout, N, 0, stride);
  return standalone_wgrad_ok(N, Ho, Wo, Cin, Cout, pl) ? pl.part_floats : 0;
}

int nf_tc_sm_count() { return sm_count(); }
int nf_tc_tile(int H, int W, int* BW, int* BH) {
  int BI;
  return pick_tile(1, H, W, BW, BH, &BI) && BI == 1;
}
int nf_tc_out_map(CUtensorMap* m, void* base, int N, int H, int W, int C, int BW, int BH) {
  const uint64_t d[4] = {(uint64_t)C, (uint64_t)W, (uint64_t)H, (uint64_t)N};
  const uint32_t b[4] = {64, (uint32_t)BW, (uint32_t)BH, 1};
  return make_map4(m, base, d, b);
}

static __device__ int32_t g_op_status;  // status word of the stand-alone operations (one per device that loads the library)

int nf_tc_op_status_ptr(int32_t** out) {
  static int32_t* st_dev[kMaxDevices];
  int32_t*& st = st_dev[current_device()];
  if (!st) NF_CUDA(cudaGetSymbolAddress((void**)&st, g_op_status));
  *out = st;
  return NF_OK;
}

int nf_tc_conv3x3_forward(const void* x, const void* w, int N, int H, int W, int Cin, int Cout, int stride, void* y) {
  const int Ho = (H - 1) / stride + 1, Wo = (W - 1) / stride + 1;
  if (!tc_size_ok(N, Ho, Wo) && !fold_ok(Ho, Wo, Cin, Cout, 0, stride, 0, 0, true)) return NF_EUNSUPPORTED;
  int32_t* st = nullptr;
  if (nf_tc_op_status_ptr(&st) != NF_OK) return NF_ECUDA;
  int nb = 0;
  return run_fwd(N, H, W, Cin, Cout, x, w, y, 0, nullptr, 0, st, &nb, 0, nullptr, stride, nullptr, true);
}

int nf_tc_conv3x3_wgrad(const void* x, const void* g, int N, int H, int W, int Cin, int Cout, int stride, float* part,
                        size_t part_floats, float* dw) {
  const int Ho = (H - 1) / stride + 1, Wo = (W - 1) / stride + 1;
  if (!standalone_wgrad_ok(N, Ho, Wo, Cin, Cout, plan_wgrad(Ho, Wo, Cin, Cout, N, 0, stride))) return NF_EUNSUPPORTED;
  int32_t* st = nullptr;
  if (nf_tc_op_status_ptr(&st) != NF_OK) return NF_ECUDA;
  return run_wgrad(N, H, W, Cin, Cout, x, g, part, part_floats, dw, st, 0, stride);
}

// One CTA of one warp waits, with the bounded wait every tensor-core kernel uses, on a barrier that nobody ever
// arrives at, and then leaves the way those kernels do: abort flag set by the waiter, NF_ETIMEOUT raised in the status
// word, waited time reported.  No TMA, no tensor memory, nothing else in flight.
__global__ void bounded_wait_probe_kernel(unsigned long long limit_ns, int32_t* status, unsigned long long* waited_ns) {
  nf_pdl_begin();
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    ptx::mbar_init(&bar, 1);
    abort_flag = 0;
    ptx::fence_mbar_init();
  }
  __syncthreads();
  const unsigned long long t0 = ptx::globaltimer();
  const bool done = __all_sync(0xffffffffu, ptx::mbar_wait(&bar, 0, &abort_flag, limit_ns));
  const unsigned long long t1 = ptx::globaltimer();
  __syncthreads();
  if (threadIdx.x == 0) {
    if (!done && abort_flag) atomicOr(status, NF_ETIMEOUT);
    *waited_ns = t1 - t0;
  }
}

int nf_tc_bounded_wait_probe(unsigned long long limit_ns, unsigned long long* waited_ns_dev) {
  int32_t* st = nullptr;
  if (nf_tc_op_status_ptr(&st) != NF_OK) return NF_ECUDA;
  nf_launch(bounded_wait_probe_kernel, 1, 32, 0, limit_ns, st, waited_ns_dev);
  NF_LAUNCHED();
  return NF_OK;
}

int nf_tc_op_status(int32_t* out) {
  NF_CUDA(cudaStreamSynchronize(g_nf_stream));
  NF_CUDA(cudaMemcpyFromSymbol(out, g_op_status, sizeof(int32_t)));
  const int32_t zero = 0;
  NF_CUDA(cudaMemcpyToSymbol(g_op_status, &zero, sizeof(int32_t)));
  return NF_OK;
}
