// Per-cell helpers shared by the kernels of gmmsp_em.cu:
// the cell's extent and candidate mask, the special-function approximations
// of the E-step, the log2 density of one candidate, and the image lookup of
// a batch.
#pragma once

#include <math.h>

#include "gmmsp_internal.cuh"

namespace gmmsp {

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The largest of three (NaNs are passed over, as by fmaxf).
__device__ __forceinline__ float max3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}
// ... and of nine (four instructions).
__device__ __forceinline__ float max9(const float (&e)[9]) {
  return max3(max3(e[0], e[1], e[2]), max3(e[3], e[4], e[5]), max3(e[6], e[7], e[8]));
}

struct Cell {
  int cx, cy;      // cell coordinates
  int x0, y0;      // first pixel
  int cw, ch;      // extent (v, or the remainder)
  unsigned mask;   // bit s set when slot s is a seed of the grid
};

__device__ __forceinline__ Cell make_cell(const Geom& g, int cell) {
  Cell c;
  c.cy = cell / g.ncx;
  c.cx = cell - c.cy * g.ncx;
  c.x0 = c.cx * g.v;
  c.y0 = c.cy * g.v;
  c.cw = min(g.v, g.W - c.x0);
  c.ch = min(g.v, g.H - c.y0);
  // slot s = 3 r + q is seed (c_x - 1 + q, c_y - 1 + r): the product of a column
  // mask (q) and a row mask (r) of the seeds on the grid
  const unsigned cols = (c.cx >= 1 && c.cx - 1 < g.nx ? 1u : 0u) | (c.cx < g.nx ? 2u : 0u) |
                        (c.cx + 1 < g.nx ? 4u : 0u);
  const unsigned rows = (c.cy >= 1 && c.cy - 1 < g.ny ? 1u : 0u) | (c.cy < g.ny ? 2u : 0u) |
                        (c.cy + 1 < g.ny ? 4u : 0u);
  c.mask = (rows & 1u ? cols : 0u) | (rows & 2u ? cols << 3 : 0u) | (rows & 4u ? cols << 6 : 0u);
  return c;
}

// The colour of pixel (x, y) of image g, read through GMMSP_IN_BOUNDS (a
// checked build yields 0 outside the image and records the event).
template <int CM, class Src>
__device__ __forceinline__ float4 load_pixel(const Src& s, const Geom& g, int x, int y) {
  if (!(GMMSP_IN_BOUNDS(x, g.W, BND_PIXEL_X) && GMMSP_IN_BOUNDS(y, g.H, BND_PIXEL_Y)))
    return make_float4(0.f, 0.f, 0.f, 0.f);
  return load_z<CM>(s, x, y);
}

// One lane's walk over a cell's pixels p, p + step, ... (p = y cw + x, row
// after row): the position as floats (exact small integers) and the pixel's
// offset, advanced by additions -- no division, conversion or address
// product per pixel.
template <class Src>
struct Walk {
  typedef typename Src::Off Off;
  float fx, fy;      // position in the cell
  Off at;            // offset of the pixel
  float cw, dx, dy;  // the cell's width; step = dy cw + dx
  Off inc, wrap;
  __device__ __forceinline__ void start(const Src& s, const Cell& c, int p, int step) {
    const int y = __float2int_rz((float(p) + 0.5f) * (1.f / float(c.cw)));  // exact floor(p / cw)
    const int x = p - y * c.cw;
    const int q = __float2int_rz((float(step) + 0.5f) * (1.f / float(c.cw))), r = step - q * c.cw;
    fx = float(x);
    fy = float(y);
    cw = float(c.cw);
    dx = float(r);
    dy = float(q);
    at = s.at(c.x0 + x, c.y0 + y);
    inc = q * s.row() + r * Src::kStep;
    wrap = s.row() - c.cw * Src::kStep;
  }
  __device__ __forceinline__ void next() {
    fx += dx;
    fy += dy;
    at += inc;
    if (fx >= cw) {
      fx -= cw;
      fy += 1.f;
      at += wrap;
    }
  }
  template <int CM>
  __device__ __forceinline__ float4 load(const Src& s, const Geom& g, const Cell& c) const {
    if (!(GMMSP_IN_BOUNDS(c.x0 + int(fx), g.W, BND_PIXEL_X) && GMMSP_IN_BOUNDS(c.y0 + int(fy), g.H, BND_PIXEL_Y)))
      return make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (CM == kColourGray) return make_float4(s.load_l_at(at), 0.f, 0.f, 0.f);
    else return s.load_at(at);
  }
};

// Two FP32 values in a register pair, and the packed arithmetic on them (one
// instruction for both, each rounded as the scalar operation).
typedef unsigned long long f2;
__device__ __forceinline__ f2 pack_f2(float lo, float hi) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float lo_f2(f2 a) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a));
  return lo;
}
__device__ __forceinline__ float hi_f2(f2 a) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a));
  return hi;
}
__device__ __forceinline__ f2 add_f2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 sub_f2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 mul_f2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 fma_f2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// A pixel as the densities take it: position in the cell and colour.
struct Pix2 {
  f2 xy, La, bb;
};
__device__ __forceinline__ Pix2 pix2(float fx, float fy, float4 z) {
  return {pack_f2(fx, fy), pack_f2(z.x, z.y), pack_f2(z.z, z.z)};
}

// log2 p(z; theta_k) for one candidate: the log normaliser plus the two
// quadratic forms, with -1/2 log2(e) Sigma^{-1} folded into the coefficients.
// The position is relative to the cell origin (the staged mean is relative to
// the same origin).  Operations on two components run as packed FP32: 14
// instructions instead of 19 per candidate of the full model, the same
// operations in the same order for each component.
// DIAG: both blocks diagonal (the Sec. III-C start and the learned start, whose
// packed 2xy, 2La, 2Lb and 2ab coefficients are exactly +-0): the same
// operations without the zero terms, so the same bits, and 12 of the 16
// floats read.
template <int CM, bool DIAG = false>
__device__ __forceinline__ float log2_density(const float4* P, const Pix2& z) {
  const ulonglong2 p0 = *reinterpret_cast<const ulonglong2*>(P), p1 = *reinterpret_cast<const ulonglong2*>(P + 1);
  const f2 d = sub_f2(z.xy, p0.x);
  const float dx = lo_f2(d), dy = hi_f2(d);
  const f2 s = mul_f2(p1.y, d);                      // (xx dx, yy dy)
  if constexpr (DIAG) {
    const float2 p3 = *(reinterpret_cast<const float2*>(P + 3) + 1);  // bb, normaliser
    float q = fmaf(lo_f2(s), dx, p3.y);              // xx dx^2
    q = fmaf(hi_f2(s), dy, q);                       // yy dy^2
    if constexpr (CM != kColourGray) {
      const f2 c = sub_f2(z.La, p0.y);
      const float db = lo_f2(z.bb) - lo_f2(p1.x);
      const f2 t = mul_f2(*reinterpret_cast<const f2*>(P + 2), c);
      q = fmaf(lo_f2(t), lo_f2(c), q);               // LL dL^2
      q = fmaf(hi_f2(t), hi_f2(c), q);               // aa da^2
      q = fmaf(p3.x * db, db, q);                    // bb db^2
    } else {
      const float dL = lo_f2(z.La) - lo_f2(p0.y);
      q = fmaf(P[2].x * dL, dL, q);
    }
    return q;
  }
  const float4 p3 = P[3];                            // 2xy, 2La, bb, normaliser
  float q = fmaf(fmaf(p3.x, dy, lo_f2(s)), dx, p3.w);  // (xx dx + 2xy dy) dx
  q = fmaf(hi_f2(s), dy, q);                         // yy dy^2
  if constexpr (CM == kColourGray) {
    const float dL = lo_f2(z.La) - lo_f2(p0.y);
    q = fmaf(P[2].x * dL, dL, q);                    // LL dL^2
  } else {
    const ulonglong2 p2 = *reinterpret_cast<const ulonglong2*>(P + 2);  // (LL, aa), (2Lb, 2ab)
    const f2 c = sub_f2(z.La, p0.y), bb = sub_f2(z.bb, p1.x);
    const float dL = lo_f2(c), da = hi_f2(c), db = lo_f2(bb);
    f2 t = mul_f2(p2.x, c);                          // (LL dL, aa da)
    if constexpr (CM == kColourFull) {
      t = fma_f2(p2.y, bb, pack_f2(fmaf(p3.y, da, lo_f2(t)), hi_f2(t)));
      q = fmaf(lo_f2(t), dL, q);                     // (LL dL + 2La da + 2Lb db) dL
      q = fmaf(hi_f2(t), da, q);                     // (aa da + 2ab db) da
    } else {
      q = fmaf(lo_f2(t), dL, q);                     // LL dL^2
      q = fmaf(fmaf(hi_f2(p2.y), db, hi_f2(t)), da, q);  // (aa da + 2ab db) da
    }
    q = fmaf(p3.z * db, db, q);                      // bb db^2
  }
  return q;
}

// The batch image owning work item `item` (a cell when which == 0, a
// superpixel when which == 1): binary search over the images' prefix offsets.
__device__ __forceinline__ int find_image(const BatchImage* __restrict__ imgs, int n, int item,
                                          int which /*0 cells, 1 superpixels*/) {
  if (imgs[0].uniform) {  // images of one geometry: a division
    const int i = item / (which == 0 ? imgs[0].g.ncells : imgs[0].g.K);
    return i < n ? i : n - 1;
  }
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    const int off = which == 0 ? imgs[mid].cell_off : imgs[mid].k_off;
    if (off <= item) lo = mid; else hi = mid;
  }
  return lo;
}

}  // namespace gmmsp
