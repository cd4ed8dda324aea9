// Index arithmetic of the 3 x 3 layers' tiles (k_conv3, k_wgrad3).
//
// The cell grid of an image is cut into strips of at most kStripMax columns
// (one strip up to nx = 126).  Within a strip the positions are numbered with
// a zero border column on either side, q = y PW + x', PW = TW + 2, x' = 0 and
// PW - 1 being the neighbouring columns (zero outside the image).  A tile is
// 128 consecutive numbers q; its inputs are the 130 + 2 PW numbers
// q0 - PW - 1 .. q0 + 127 + PW + 1 (rows above and below the image zero), and
// tap (dy, dx) of row q is the input at q + dy PW + dx.
//
// A tile costs a load, an MMA and an epilogue round trip however few of its
// positions are cells, so small grids are stacked: `per` images one below the
// other with one zero row between them, H1 = H + 1 rows each, numbered as one
// tall image.  The line: an eighth fewer tiles that way (at 21 x 32 cells it
// would save 3 %, and the gradient's order of additions would change for it).
// Forward / gradient, us, a tile per image and stacked: 16384 images of one
// cell 285 / 1828 and 60 / 256, 8192 of 2 x 2 183 / 1054 and 79 / 302, 4096 of
// 4 x 6 197 / 819 and 162 / 541; 1024 of 8 x 10 140 / 466 and 139 / 454.
// A stack holds up to 2^17 positions (a thousand tiles), so that its last,
// partly empty tile does not count.
//
// Row and column of a position come from a multiplication by
// floor(2^32 / PW) + 1 in place of a division (two divisions per position cost
// 29.7 us a layer at 256 images of 481x321, 13.9 without).  That is the exact
// quotient of n only while n PW < 2^32, which the numbers q of a tall grid
// exceed (PW = 128 from row 262144 on).  So a tile divides once, for its first
// position, with a correction (below), and its other positions are counted
// from the start of that row: n < PW + 128 + 2 PW + 130 < 2^10.
//
// Plain integer code: the host test suite checks it against divisions.
#pragma once

#include <stdint.h>

#if defined(__CUDACC__)
#define GMMSP_GRID3_FN __host__ __device__ __forceinline__
#else
#define GMMSP_GRID3_FN inline
#endif

namespace gmmsp {
namespace cnn {

constexpr int kStripMax = 126;

GMMSP_GRID3_FN uint32_t mulhi32(uint32_t a, uint32_t b) {
#if defined(__CUDA_ARCH__)
  return __umulhi(a, b);
#else
  return uint32_t((uint64_t(a) * b) >> 32);
#endif
}

struct Grid3 {
  int B, H, W;         // images and their cell grids (B H W <= 2^30)
  int strips, TW, PW;  // strips per image, their columns, the bordered row length
  int per, stacks;     // images per stack (1: not stacked), stacks
  int H1;              // rows from one image of a stack to the next
  int tps;             // tiles per strip of a stack
  int tiles;           // stacks strips tps (< 2^31: at most 3 B H W / 128 full ones and one more per strip)
  int NP, GS;          // inputs of a tile; bytes per channel group of them
  uint32_t rPW, rH1;   // floor(2^32 / PW) + 1; the same of H1, 0 where not stacked
};
constexpr int kStackPositions = 1 << 17;
inline Grid3 grid3_of(int B, int H, int W) {
  Grid3 g{};
  g.B = B;
  g.H = H;
  g.W = W;
  g.strips = (W + kStripMax - 1) / kStripMax;
  g.TW = (W + g.strips - 1) / g.strips;
  g.PW = g.TW + 2;
  g.rPW = uint32_t((1ull << 32) / uint32_t(g.PW)) + 1u;
  g.per = 1;
  g.stacks = B;
  g.H1 = H + 1;
  g.tps = int(((long long)H * g.PW + 127) / 128);
  const long long most = kStackPositions / ((long long)g.H1 * g.PW);  // images of a stack
  if (B > 1 && most > 1) {
    const int stacks = int((B + most - 1) / most), per = int((B + (long long)stacks - 1) / stacks);
    const int tps = ((per * g.H1 - 1) * g.PW + 127) / 128;
    if (8LL * stacks * tps <= 7LL * B * g.tps) {
      g.per = per;
      g.stacks = (B + per - 1) / per;
      g.tps = tps;
      g.rH1 = uint32_t((1ull << 32) / uint32_t(g.H1)) + 1u;
    }
  }
  g.tiles = g.stacks * g.strips * g.tps;
  g.NP = 130 + 2 * g.PW;
  g.GS = (g.NP * 16 + 127) / 128 * 128 + 32;  // 32 mod 128: the four groups of a position fall into other banks
  return g;
}

struct Tile3 {
  int img, end;  // image of the first position; the stack's images end before this one
  int c0;        // first column of the strip
  int y0, x0;    // row (of the image) and bordered column of the first position
};
GMMSP_GRID3_FN Tile3 tile3_at(const Grid3& g, int tile) {
  const int s = tile / g.tps;
  // q0 < 2^31 + 128, and the multiplication is off by less than q0 PW / 2^32 of a
  // position: the quotient is exact or one too large
  const uint32_t q0 = uint32_t(tile - s * g.tps) * 128u;
  uint32_t y = mulhi32(q0, g.rPW);
  if (y * uint32_t(g.PW) > q0) --y;
  const int x0 = int(q0 - y * uint32_t(g.PW)), first = s / g.strips * g.per;
  const int i = int(mulhi32(y, g.rH1));  // image of the stack (y H1 < 2^32 in a stack; else 0)
  return {first + i, first + g.per, (s % g.strips) * g.TW, int(y) - i * g.H1, x0};
}

// Row of the tile's position p (0 .. 127) in the [B H W] arrays, or -1 where it
// is no output (border column, below the image, past the strip or the image).
GMMSP_GRID3_FN int row3(const Grid3& g, const Tile3& t, int p) {
  const int n = t.x0 + p, dy = int(mulhi32(uint32_t(n), g.rPW));
  const int x = n - dy * g.PW, col = t.c0 + x - 1;
  int y = t.y0 + dy;
  const int i = int(mulhi32(uint32_t(y), g.rH1)), img = t.img + i;
  y -= i * g.H1;
  return (y < g.H && x >= 1 && x <= g.TW && col < g.W && img < t.end && img < g.B) ? (img * g.H + y) * g.W + col : -1;
}

// The same of the tile's input p (0 .. NP - 1), position p - PW - 1, or -1 where
// it is zero.  (The row before the first position's belongs to the previous
// image of a stack only where no output reads it.)
GMMSP_GRID3_FN int in3(const Grid3& g, const Tile3& t, int p) {
  const int n = t.x0 + p + g.PW - 1, dy = int(mulhi32(uint32_t(n), g.rPW));  // two rows on: not negative
  const int col = t.c0 + n - dy * g.PW - 1;
  int y = t.y0 + dy - 2;
  const int i = int(mulhi32(uint32_t(y < 0 ? 0 : y), g.rH1)), img = t.img + i;
  y -= i * g.H1;
  return (uint32_t(y) < uint32_t(g.H) && uint32_t(col) < uint32_t(g.W) && img < t.end && img < g.B)
             ? (img * g.H + y) * g.W + col
             : -1;
}

}  // namespace cnn
}  // namespace gmmsp
