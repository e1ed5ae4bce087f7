// Pixel tiles of the persistent convolution kernels: tile number -> place, without run-time divisions.
#pragma once
#include <stdint.h>

// Division by a number that is fixed for a launch, as a multiplication by a rounded-up reciprocal (Granlund and Montgomery, Division by
// Invariant Integers using Multiplication, 1994; exact for dividends below 2^31).  The role loops decode
// a tile number per tile; a 32-bit division by a run-time value costs a single thread about 100 cycles of dependent instructions.
struct FDiv {
  uint32_t d, mul, shift;
};
static inline FDiv fdiv_of(uint32_t d) {
  FDiv f{d, 0, 0};
  if (d == 1) return f;
  uint32_t lg = 0;
  while ((1ull << lg) < d) ++lg;
  f.mul = (uint32_t)(((1ull << (31 + lg)) + d - 1) / d);
  f.shift = lg - 1;
  return f;
}
__device__ __forceinline__ uint32_t fdiv(uint32_t n, const FDiv& f, uint32_t* rem) {
  const uint32_t q = f.d == 1 ? n : __umulhi(n, f.mul) >> f.shift;
  *rem = n - q * f.d;
  return q;
}

// First pixel and image (group) of pixel tile m: tiles run along the width, then the height, then the images
struct TileGrid {
  FDiv nt, tw, th;  // channel tiles, tile columns, tile rows
};
static inline TileGrid tile_grid(int n_tiles, int tiles_w, int tiles_h) { return {fdiv_of(n_tiles), fdiv_of(tiles_w), fdiv_of(tiles_h)}; }
struct TileAt {
  uint32_t nt, w, h, n;
};
__device__ __forceinline__ TileAt tile_at(uint32_t t, const TileGrid& g) {
  TileAt a;
  const uint32_t m = fdiv(t, g.nt, &a.nt), r = fdiv(m, g.tw, &a.w);
  a.n = fdiv(r, g.th, &a.h);
  return a;
}
