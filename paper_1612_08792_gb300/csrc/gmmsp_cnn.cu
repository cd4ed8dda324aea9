// The learned initialiser (include/gmmsp_cnn.h): a small convolutional
// network that predicts, for every superpixel of a CIELAB image, the offset
// of its fitted mean from the Sec. III-C start and the logarithms of its
// fitted covariance diagonal.  It stands in for Algorithm 1, step 1, so that
// fewer EM iterations reach the same likelihood; the EM steps themselves are
// unchanged.  The paper has no such network.
//
// Kernels (activations and weights BF16, accumulation FP32 in tensor memory,
// every product on the tcgen05 tensor cores):
//   k_pix   x0 -> h1 -> h2 -> c0 fused: one block per group of cells (128
//           rows = 3 x 3 pixel patches), both 1 x 1 layers as 128 x 32 x 32
//           MMAs with the accumulators in TMEM, the average pooling in shared
//           memory.  Reads the CIELAB planes once and writes c0 (and, when
//           training, x0, h1 and h2 for the backward pass).
//   k_conv3 3 x 3 convolution of the cell grid, forward and data gradient: one
//           tile of 128 zero-bordered positions and its halo per step, the
//           taps addressed by shifting the matrix descriptor's start, all 18
//           MMAs issued at once.
//   k_wgrad3 weight and bias gradient of a 3 x 3 layer from the same tiles
//           (one accumulator per tap in tensor memory, kept over the tiles).
//   k_pix_bwd the backward pass of the pixel level fused: pooling and ReLU
//           gradient, data gradient of the second 1 x 1 layer, both weight
//           gradients.
//   k_loss, k_grad_reduce, k_adam, k_targets, k_init_from_net.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include "../../include/gmmsp.h"
#include "../../include/gmmsp_cnn.h"
#include "gmmsp_cnn_internal.cuh"
#include "gmmsp_grid3.cuh"
#include "gmmsp_internal.cuh"
#include "gmmsp_lab.cuh"
#include "gmmsp_math.cuh"
#include "gmmsp_tc.cuh"

namespace gmmsp {
namespace cnn {

constexpr int kC = 32;                     // channels of every hidden layer
constexpr int kOut = GMMSP_NET_CHANNELS;   // output channels of the last layer (16)
constexpr int kUsed = GMMSP_NET_OUTPUTS;   // outputs used per superpixel (10)
constexpr uint32_t kWaitTries = 1u << 22;  // bound on every mbarrier wait
constexpr int kLossBlocks = 128;

constexpr float kInScale = 0.02f;    // L, a, b -> about [-1, 1] (L shifted by 50)
constexpr int kStartCh = 29;         // c0 channels 29-31: the start pixel's scaled colour (not pooled)
constexpr float kColourUnit = 10.f;  // colour mean offsets in units of 10

// Flat parameter vector W1, b1, ..., W6, b6 with W[cout][taps * 32 + cin].
struct ParamLayout {
  int w[6], b[6], taps[6], cout[6];
  int total;
};
inline int pix_params(const ParamLayout& p) { return p.w[2]; }  // of the two 1 x 1 layers, at the front
inline ParamLayout param_layout() {
  ParamLayout p{};
  const int taps[6] = {1, 1, 9, 9, 9, 9};
  const int cout[6] = {kC, kC, kC, kC, kC, kOut};
  int off = 0;
  for (int l = 0; l < 6; ++l) {
    p.taps[l] = taps[l];
    p.cout[l] = cout[l];
    p.w[l] = off;
    off += cout[l] * taps[l] * kC;
    p.b[l] = off;
    off += cout[l];
  }
  p.total = off;
  return p;
}

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// ------------------------------------------------- 3 x 3 layers: tiles
// Tiles, their positions and inputs: gmmsp_grid3.cuh.
//
// In shared memory the inputs lie as channel groups of 8 (16 bytes), position
// after position: group g of input i at g GS + 16 i.  Eight consecutive
// positions of a group are then one 128-byte core matrix wherever they start,
// so a tap is the same tile read from another start address: every input is
// loaded once instead of nine times, and the 18 MMAs of a tile are issued
// together (the gather per tap that this replaced read each activation nine
// times from L2 and paid one MMA round trip per tap).  The same bytes serve as
// a K-major operand (rows = positions: 8-row groups 128 bytes apart, K groups
// GS apart) and as an MN-major one (K = positions).
constexpr int kWLd = 528;                     // bytes between (tap, input group) slices of the staged weights
constexpr int kWBytes = 36 * kWLd;            // 9 taps x 4 groups x 32 output channels x 16 bytes, padded
constexpr int kRowTile = 128 * 16 + 32;       // a group of a 128-position tile without halo (bank offset 32)

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The tile's inputs with their halo, G channel groups per position.
template <int G>
__device__ __forceinline__ void load_halo(const Grid3& g, const Tile3& t, const __nv_bfloat16* __restrict__ x,
                                          uint32_t dst) {
  for (int i = threadIdx.x; i < g.NP * G; i += 128) {
    const int p = i / G, gr = i - p * G;
    const int r = in3(g, t, p);
    cp_async16(dst + gr * g.GS + p * 16, x + (long long)max(r, 0) * (8 * G) + gr * 8, r >= 0);
  }
}

// The staged weights of a 3 x 3 layer: slices (tap, group of 8 input channels),
// output channel co of slice s at s kWLd + 16 co.  K-major for the forward
// pass (rows = output channels), MN-major for the data gradient (rows = input
// channels, K = output channels).  Kept in global memory in this form beside
// the plain BF16 parameters (store_bf16), so that staging is a linear copy.
__device__ __forceinline__ void load_weights3(const unsigned char* __restrict__ w, uint32_t dst) {
#pragma unroll
  for (int i = threadIdx.x; i < kWBytes / 16; i += 128) cp_async16(dst + i * 16, w + i * 16, true);
}

// BF16 copies of parameter i: the flat one and, for the 3 x 3 layers, the
// staged one.
struct BfParams {
  __nv_bfloat16* flat;
  unsigned char* staged;  // kWBytes per 3 x 3 layer
  int w[4], n[4];         // offset and number of each 3 x 3 layer's weights
};
__device__ __forceinline__ void store_bf16(const BfParams& p, int i, float v) {
  const __nv_bfloat16 h = __float2bfloat16(v);
  p.flat[i] = h;
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const int j = i - p.w[l];
    if (j >= 0 && j < p.n[l]) {
      const int co = j / 288, r = j - co * 288;
      reinterpret_cast<__nv_bfloat16*>(p.staged + l * kWBytes + (r >> 3) * kWLd)[co * 8 + (r & 7)] = h;
    }
  }
}

struct Conv3 {
  Grid3 g;
  const __nv_bfloat16* a;     // forward: layer input [B H W][32]; data gradient: gradient of the output [B H W][cout]
  const unsigned char* w;     // staged weights
  const float* bias;          // forward: [cout]
  __nv_bfloat16* y;           // output [B H W][32] BF16 (forward: ReLU(. + bias); data gradient: masked), or ...
  float* y32;                 // ... FP32 [B H W][cout] without ReLU (the last layer's forward)
  const __nv_bfloat16* mask;  // data gradient: zero where mask <= 0 (or null)
};

// 3 x 3 convolution, one tile per step: forward (A = the input, K = (tap,
// input channel)) or data gradient (A = the output's gradient with GC groups
// of 8 channels, K = (tap, output channel), taps mirrored).  K runs in the
// same order of 16-wide MMAs as a tap-by-tap GEMM would, so the FP32 sums are
// the same.
//
// Bound by latency: a tile is one load round trip, 18 MMAs, one epilogue.
// 31.8 KB of shared memory at nx = 32 leave 6 blocks per SM to overlap them,
// and a block takes further tiles with its weights staged once.  Measured
// per 32-channel layer at 481x321, v = 15 (nx = 32), ncu, cold cache: 13.9 us
// on 256 images (30.3 us for the tap-by-tap gather), 6.1 us on 32 (15.2 us);
// index divisions by the row length in place of the multiplications cost
// 29.7 and 10.2 us.
template <bool DGRAD, int GC, int N>
__global__ void __launch_bounds__(128, 6) k_conv3(Conv3 c, int* err) {
  extern __shared__ __align__(128) unsigned char smem3[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_sh;
  const int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t sW = tc::smem_u32(smem3), sX = sW + kWBytes;
  if (warp == 0) {
    tc::tmem_alloc(&tmem_sh, 32);
    tc::tmem_relinquish();
  }
  if (tid == 0) tc::mbar_init(&mbar, 1);
  load_weights3(c.w, sW);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_sh;
  constexpr uint32_t idesc = tc::idesc_bf16_f32(128, N) | (DGRAD ? tc::kTransB : 0u);
  bool ok = true;
  uint32_t phase = 0;
  for (int tile = blockIdx.x; tile < c.g.tiles; tile += gridDim.x) {
    const Tile3 t = tile3_at(c.g, tile);
    load_halo<GC>(c.g, t, c.a, sX);
    cp_async_wait_all();
    tc::fence_async_smem();
    tc::fence_before_sync();  // the previous tile's accumulator has been read
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      // descriptor start addresses count 16 bytes: one input position per unit
      uint64_t ad[GC / 2];
#pragma unroll
      for (int kk = 0; kk < GC / 2; ++kk) ad[kk] = tc::smem_desc(sX + 2 * kk * c.g.GS, c.g.GS, 128) + (c.g.PW + 1);
      const uint64_t bd = DGRAD ? tc::smem_desc(sW, 128, kWLd) : tc::smem_desc(sW, kWLd, 128);
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const int d = (tap / 3 - 1) * c.g.PW + (tap % 3 - 1);
#pragma unroll
        for (int kk = 0; kk < GC / 2; ++kk)
          tc::mma_bf16(tmem, ad[kk] + (DGRAD ? -d : d), bd + (tap * 4 * kWLd + (DGRAD ? kk * 256 : 2 * kk * kWLd)) / 16,
                       idesc, (tap > 0 || kk > 0) ? 1u : 0u);
      }
      tc::mma_commit(&mbar);
    }
    const int row = row3(c.g, t, tid);
    uint4 m[4] = {};
    if (DGRAD && c.mask && row >= 0) {
      const uint4* ms = reinterpret_cast<const uint4*>(c.mask + (long long)row * kC);
#pragma unroll
      for (int j = 0; j < 4; ++j) m[j] = __ldg(ms + j);
    }
    const bool w = tc::mbar_wait(&mbar, phase & 1u, kWaitTries);
    ok = __syncthreads_and(w) != 0;
    if (!ok) break;
    ++phase;
    tc::fence_after_sync();
    float acc[N];
#pragma unroll
    for (int c0 = 0; c0 < N; c0 += 16) {
      float v[16];
      tc::tmem_ld16(tmem + (uint32_t(warp * 32) << 16) + uint32_t(c0), v);
#pragma unroll
      for (int i = 0; i < 16; ++i) acc[c0 + i] = v[i];
    }
    if (row < 0) continue;
    if (!DGRAD && c.y32) {
#pragma unroll
      for (int i = 0; i < N; i += 4)
        *reinterpret_cast<float4*>(c.y32 + (long long)row * N + i) =
            make_float4(acc[i] + __ldg(c.bias + i), acc[i + 1] + __ldg(c.bias + i + 1),
                        acc[i + 2] + __ldg(c.bias + i + 2), acc[i + 3] + __ldg(c.bias + i + 3));
      continue;
    }
    const uint32_t* mw = reinterpret_cast<const uint32_t*>(m);
    uint32_t u[N / 2];
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      float a = acc[i], b = acc[i + 1];
      if (!DGRAD) {
        a = fmaxf(a + __ldg(c.bias + i), 0.f);
        b = fmaxf(b + __ldg(c.bias + i + 1), 0.f);
      } else if (c.mask) {
        if (!(bf_lo(mw[i / 2]) > 0.f)) a = 0.f;
        if (!(bf_hi(mw[i / 2]) > 0.f)) b = 0.f;
      }
      u[i / 2] = pack2(a, b);
    }
    uint4* dst = reinterpret_cast<uint4*>(c.y + (long long)row * N);
#pragma unroll
    for (int j = 0; j < N / 8; ++j) dst[j] = make_uint4(u[4 * j], u[4 * j + 1], u[4 * j + 2], u[4 * j + 3]);
  }
  if (!ok) {
    // give the MMAs in flight one more bounded chance to land before TMEM is freed
    tc::mbar_wait(&mbar, phase & 1u, kWaitTries);
    if (tid == 0) atomicExch(err, 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 32);
}

// 128 zero-bordered positions of [B H W][8 G] without halo, zero where the
// position is no output: a contraction over positions must not see the border.
template <int G>
__device__ __forceinline__ void load_rows3(const Grid3& g, const Tile3& t, const __nv_bfloat16* __restrict__ x,
                                           uint32_t dst) {
  for (int i = threadIdx.x; i < 128 * G; i += 128) {
    const int p = i / G, gr = i - p * G;
    const int r = row3(g, t, p);
    cp_async16(dst + gr * kRowTile + p * 16, x + (long long)max(r, 0) * (8 * G) + gr * 8, r >= 0);
  }
}

// `bytes` of BF16 ones: as the channel group behind an input's four they make
// the bias gradient column 32 of the weight gradient's product (N = 48; the
// columns of the group after that hold any bits and are not read).
__device__ __forceinline__ void fill_ones(unsigned char* p, int bytes) {
  for (int i = threadIdx.x * 16; i < bytes; i += 128 * 16)
    *reinterpret_cast<uint4*>(p + i) = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
}

// The MMAs read 128 rows of an MN-major operand of 16 or 32: rows past the
// channel count come from the shared memory behind it (any bits: they only
// enter accumulator rows that nothing reads), which must exist.
constexpr int kMnSpan = 16 * kRowTile;

// First accumulator column of a tap: 32 each, the centre's last, followed by
// the bias column.
__device__ __forceinline__ int wgrad3_col(int tap) { return tap < 4 ? tap * 32 : (tap > 4 ? (tap - 1) * 32 : 256); }

struct Wgrad3 {
  Grid3 g;
  const __nv_bfloat16* x[4];   // each layer's input [B H W][32]
  const __nv_bfloat16* gy[4];  // gradient of its output before the activation [B H W][32] (the last layer: [16])
  int off[4];                  // its place in a block's sums
  float* part;                 // sums of block b at part + b stride: per layer [cout][288], then [cout] of the bias
  long long stride;
};

// Weight and bias gradients of the 3 x 3 layers (blockIdx.y the layer):
// D_tap[co][cin] += sum over the tile's positions of gy[q][co] x[q + tap][cin],
// both operands MN-major (K = positions), the accumulators and the bias column
// in tensor memory over all tiles of the block, written once at the end.  One
// block per SM (512 TMEM columns), so the four layers share one launch of at
// most one block per SM: a quarter of the partial sums of a launch per layer.
// Bound by latency; it replaces a GEMM whose operands
// were gathered two bytes at a time and which ran few blocks of 64 serial
// steps (1.0-1.2 ms per layer at 32 images of 481x321, v = 15, against 26.5 us
// for the four layers).
template <int GC>
__device__ __forceinline__ void wgrad3_layer(const Wgrad3& c, int layer, int* err) {
  extern __shared__ __align__(128) unsigned char smem3[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_sh;
  const int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t sG = tc::smem_u32(smem3), sX = sG + GC * kRowTile;
  if (warp == 0) {
    tc::tmem_alloc(&tmem_sh, 512);
    tc::tmem_relinquish();
  }
  if (tid == 0) tc::mbar_init(&mbar, 1);
  fill_ones(smem3 + GC * kRowTile + 4 * c.g.GS, c.g.GS);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_sh;
  constexpr uint32_t id32 = tc::idesc_bf16_f32(128, 32) | tc::kTransA | tc::kTransB;
  constexpr uint32_t id48 = tc::idesc_bf16_f32(128, 48) | tc::kTransA | tc::kTransB;
  bool ok = true;
  uint32_t phase = 0;
  for (int tile = blockIdx.x; tile < c.g.tiles; tile += gridDim.x) {
    const Tile3 t = tile3_at(c.g, tile);
    load_rows3<GC>(c.g, t, c.gy[layer], sG);
    load_halo<4>(c.g, t, c.x[layer], sX);
    cp_async_wait_all();
    tc::fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      const bool first = tile == int(blockIdx.x);
      const uint64_t a0 = tc::smem_desc(sG, 128, kRowTile), b0 = tc::smem_desc(sX, 128, c.g.GS) + (c.g.PW + 1);
      for (int kk = 0; kk < 8; ++kk) {
        const uint64_t ad = a0 + kk * 16;
        const uint32_t acc = first && kk == 0 ? 0u : 1u;
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
          const int d = (tap / 3 - 1) * c.g.PW + (tap % 3 - 1);
          tc::mma_bf16(tmem + wgrad3_col(tap), ad, b0 + (d + kk * 16), tap == 4 ? id48 : id32, acc);
        }
      }
      tc::mma_commit(&mbar);
    }
    const bool w = tc::mbar_wait(&mbar, phase & 1u, kWaitTries);  // the tiles are refilled next
    ok = __syncthreads_and(w) != 0;
    if (!ok) break;
    ++phase;
  }
  tc::fence_after_sync();
  if (!ok) {
    tc::mbar_wait(&mbar, phase & 1u, kWaitTries);
    if (tid == 0) atomicExch(err, 1);
  } else if (warp == 0) {  // accumulator row = output channel = lane
    float* out = c.part + blockIdx.x * c.stride + c.off[layer];
    for (int c0 = 0; c0 <= 288; c0 += 16) {
      float v[16];
      tc::tmem_ld16(tmem + uint32_t(c0), v);
      if (tid < 8 * GC) {  // lanes past the channels only load
        if (c0 == 288) {
          out[8 * GC * 288 + tid] = v[0];
        } else {
          const int j = c0 >> 5, tap = j < 4 ? j : (j < 8 ? j + 1 : 4);
          float4* o = reinterpret_cast<float4*>(out + tid * 288 + tap * 32 + (c0 & 16));
#pragma unroll
          for (int i = 0; i < 4; ++i) o[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}
__global__ void __launch_bounds__(128) k_wgrad3(Wgrad3 c, int* err) {
  if (blockIdx.y == 3) wgrad3_layer<2>(c, 3, err);
  else wgrad3_layer<4>(c, blockIdx.y, err);
}

// ------------------------------------------------------------------ k_pix
struct PixArgs {
  const float* lab;  // B images, each three planes of W H floats (L, a, b), consecutive
  // Converting mode (rgb non-null): the cells' pixels are read as sRGB from
  // the batch table's RGB8 rows and their CIELAB values written to lab_out
  // (planes as `lab`) on the way; `lab` is then unused.
  const BatchImage* rgb;
  float* lab_out;
  const float* srgb;  // 256 decoded sRGB code values (k_srgb_table)
  Rgb2LabConst k;
  int W, H, v, f, nx, ny;
  int cells;         // B n_x n_y
  int cpb;           // cells per block: floor(128 / f^2)
  const __nv_bfloat16* w1;
  const float* b1;
  const __nv_bfloat16* w2;
  const float* b2;
  __nv_bfloat16* c0;            // [cells][32]
  __nv_bfloat16 *x0, *h1;       // training: [blocks 128][32]
  uint32_t* h2;                 // training: bit c of row r set where h2 > 0
  int* err;
};

// Row r of block b is patch q = r mod f^2 of cell b cpb + r / f^2; the patch
// covers the pixels (k_x v + 3 (q mod f) + dx, k_y v + 3 (q / f) + dy),
// dx, dy in {0, 1, 2}; input channel (3 dy + dx) 3 + colour.  The inputs are
// gathered by patch rows: thread t takes patch (q mod f = t mod f, q / f =
// t / (cpb f)) of the block's cell (t mod (cpb f)) / f, so that a warp's
// loads run along image rows across the block's cells; the thread writes the
// patch's row of the A tile.  After the MMAs thread t owns row t.
//
// Shared memory: the A tile (8 KB) and both weight tiles (4 KB) while the
// MMAs run; the pooling buffer (128 rows of 16 BF16 pairs, 17 words apart)
// reuses the same bytes once the second MMA has completed.  Both layers
// accumulate into the same 32 TMEM columns (the second MMA is issued after
// every thread has read the first result).  In the converting mode each
// thread converts its patch's 9 pixels in registers (its inputs) and stores
// their CIELAB values to the planes.
constexpr int kPixMinBlocks = 8;
constexpr int kPixSmem = 128 * kC * 2 + 2 * kC * kC * 2;  // A + weight tiles (12 KB)
constexpr int kPoolLd = kC / 2 + 1;                       // words per pooling row
static_assert(128 * kPoolLd * 4 <= kPixSmem, "pooling buffer");

// The sRGB decoding table of the converting mode, once per network (the
// conversion kernels' own table code, so that both give the same bits).
__global__ void k_srgb_table(float* lin) { build_srgb_table(lin); }

// TRAIN: x0, h1 and the signs of h2 are kept for the backward pass.
template <bool TRAIN>
__global__ void __launch_bounds__(128, kPixMinBlocks) k_pix(PixArgs a) {
  __shared__ __align__(1024) unsigned char smem[kPixSmem];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_sh;
  unsigned char* sA = smem;
  unsigned char (*sW)[kC * kC * 2] = reinterpret_cast<unsigned char (*)[kC * kC * 2]>(smem + 128 * kC * 2);
  uint32_t (*sH)[kPoolLd] = reinterpret_cast<uint32_t (*)[kPoolLd]>(smem);
  const int tid = threadIdx.x, warp = tid >> 5;
  if (warp == 0) {
    tc::tmem_alloc(&tmem_sh, 32);
    tc::tmem_relinquish();
  }
  if (tid == 0) tc::mbar_init(&mbar, 1);
  const int ff = a.f * a.f;
  // row tid (after the MMAs)
  const int lc = tid / ff;
  const bool valid = lc < a.cpb && (long long)blockIdx.x * a.cpb + lc < a.cells;
  // the patch this thread gathers (patch-row order) and its row of the A tile
  const int prow = a.cpb * a.f;                  // patches per patch row of the block
  const int qy = tid / prow, qr = tid - qy * prow;
  const int lci = qr / a.f, qx = qr - lci * a.f;
  const bool pad = qy >= a.f;                    // tid >= cpb f^2: a zero row
  const int row_in = pad ? tid : lci * ff + qy * a.f + qx;
  const int cell = blockIdx.x * a.cpb + lci;  // < cells + cpb, an int
  const bool valid_in = !pad && cell < a.cells;
  uint32_t u[16];
  // the Sec. III-C start pixel (k_x v + v/2, k_y v + v/2) lies in patch (qs, qs) at (ds, ds)
  const int qs = (a.v / 2) / 3, ds = (a.v / 2) % 3;
  const bool start_row = valid_in && qy == qs && qx == qs;
  float zs[3] = {0.f, 0.f, 0.f};
  __shared__ float lin[256];  // converting mode: the sRGB table
  if (a.rgb) {
    lin[tid] = __ldg(a.srgb + tid);
    lin[tid + 128] = __ldg(a.srgb + tid + 128);
  }
  {
    float in[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) in[i] = 0.f;
    const int K = a.nx * a.ny;
    const int img = valid_in ? int(cell / K) : 0, k = valid_in ? int(cell - (long long)img * K) : 0;
    const int ky = k / a.nx, kx = k - ky * a.nx;
    const int px0 = kx * a.v + 3 * qx, py0 = ky * a.v + 3 * qy;
    if (a.rgb) {
      // all 27 code values first (independent loads), then the table, then
      // the conversion; each pixel's CIELAB values are stored from registers
      // A patch row is 9 consecutive bytes; they are read as the three aligned
      // 32-bit words that hold them.  The first word holds the row's first
      // byte and the last word its last, so no word reaches past the page of
      // a byte of the image (the bytes after the 9th are not used).
      uint8_t code[27];
      const BatchImage* im = a.rgb + img;
      if (valid_in) {
        const long long pitch = im->pitch;
        const uint8_t* S = static_cast<const uint8_t*>(im->image) + (long long)py0 * pitch + 3LL * px0;
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) {
          const uintptr_t at = reinterpret_cast<uintptr_t>(S + dy * pitch);
          const uint32_t* w = reinterpret_cast<const uint32_t*>(at & ~uintptr_t(3));
          const uint32_t sh = uint32_t(at & 3) * 8;
          const uint32_t w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2);
          const uint32_t lo = __funnelshift_r(w0, w1, sh), hi = __funnelshift_r(w1, w2, sh);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            code[dy * 9 + j] = uint8_t(lo >> (8 * j));
            code[dy * 9 + 4 + j] = uint8_t(hi >> (8 * j));
          }
          code[dy * 9 + 8] = uint8_t(w2 >> sh);
        }
      }
      __syncthreads();  // the table
      const long long N = (long long)a.W * a.H;
      const long long p0 = (long long)py0 * a.W + px0;
      float* T = a.lab_out + 3 * (valid_in ? im->pix_off : 0) + p0;
#pragma unroll
      for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          if (!valid_in) continue;
          const int c = (dy * 3 + dx) * 3;
          float L, A, B;
          srgb8_to_lab(a.k, lin, code + c, L, A, B);
          float* t = T + (long long)dy * a.W + dx;
          if (GMMSP_IN_BOUNDS((t - a.lab_out) + 2 * N, (long long)(a.cells / K) * 3 * N, BND_PIXEL_Y)) {
            t[0] = L;
            t[N] = A;
            t[2 * N] = B;
          }
          in[c + 0] = fmaf(L, kInScale, -1.f);
          in[c + 1] = A * kInScale;
          in[c + 2] = B * kInScale;
          if (start_row && dy == ds && dx == ds) {
            zs[0] = in[c + 0];
            zs[1] = in[c + 1];
            zs[2] = in[c + 2];
          }
        }
    } else if (valid_in) {
      const long long N = (long long)a.W * a.H;
      const float* P = a.lab + (long long)img * 3 * N;
#pragma unroll
      for (int dy = 0; dy < 3; ++dy)
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          const long long i = (long long)(py0 + dy) * a.W + (px0 + dx);
          const int c = (dy * 3 + dx) * 3;
          in[c + 0] = fmaf(__ldg(P + i), kInScale, -1.f);
          in[c + 1] = __ldg(P + N + i) * kInScale;
          in[c + 2] = __ldg(P + 2 * N + i) * kInScale;
          if (start_row && dy == ds && dx == ds) {
            zs[0] = in[c + 0];
            zs[1] = in[c + 1];
            zs[2] = in[c + 2];
          }
        }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) u[i] = pack2(in[2 * i], in[2 * i + 1]);
  }
  if (tid < 64) {
    const uint4* src = reinterpret_cast<const uint4*>((tid < 32 ? a.w1 : a.w2) + (tid & 31) * kC);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<uint4*>(sW[tid >> 5] + tc::tile_offset(tid & 31, 8 * j, kC)) = __ldg(src + j);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint4 v4 = make_uint4(u[4 * j], u[4 * j + 1], u[4 * j + 2], u[4 * j + 3]);
    *reinterpret_cast<uint4*>(sA + tc::tile_offset(row_in, 8 * j, kC)) = v4;
    if (TRAIN) reinterpret_cast<uint4*>(a.x0 + ((long long)blockIdx.x * 128 + row_in) * kC)[j] = v4;
  }
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_sh;
  constexpr uint32_t idesc = tc::idesc_bf16_f32(128, kC);
  const uint32_t a0 = tc::smem_u32(sA);
  bool ok = true;
  int layer = 0;
  for (; layer < 2; ++layer) {
    if (tid == 0) {
      const uint32_t b0 = tc::smem_u32(sW[layer]);
#pragma unroll
      for (int kk = 0; kk < 2; ++kk)
        tc::mma_bf16(tmem, tc::smem_desc(a0 + kk * 256, 128, 512),
                     tc::smem_desc(b0 + kk * 256, 128, 512), idesc, kk > 0 ? 1u : 0u);
      tc::mma_commit(&mbar);
    }
    const bool w = tc::mbar_wait(&mbar, uint32_t(layer), kWaitTries);
    ok = __syncthreads_and(w) != 0;
    tc::fence_after_sync();
    if (!ok) break;
    float acc[32];
#pragma unroll
    for (int c0 = 0; c0 < 32; c0 += 16) {
      float v[16];
      tc::tmem_ld16(tmem + (uint32_t(warp * 32) << 16) + uint32_t(c0), v);
#pragma unroll
      for (int i = 0; i < 16; ++i) acc[c0 + i] = v[i];
    }
    const float* bias = layer == 0 ? a.b1 : a.b2;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float e0 = valid ? fmaxf(acc[2 * i] + __ldg(bias + 2 * i), 0.f) : 0.f;
      const float e1 = valid ? fmaxf(acc[2 * i + 1] + __ldg(bias + 2 * i + 1), 0.f) : 0.f;
      u[i] = pack2(e0, e1);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (layer == 1) break;
      const uint4 v4 = make_uint4(u[4 * j], u[4 * j + 1], u[4 * j + 2], u[4 * j + 3]);
      *reinterpret_cast<uint4*>(sA + tc::tile_offset(tid, 8 * j, kC)) = v4;
      if (TRAIN) reinterpret_cast<uint4*>(a.h1 + ((long long)blockIdx.x * 128 + tid) * kC)[j] = v4;
    }
    if (TRAIN && layer == 1) {  // the backward pass needs only where h2 > 0
      uint32_t m = 0;
#pragma unroll
      for (int i = 0; i < 16; ++i) m |= (bf_lo(u[i]) > 0.f ? 1u : 0u) << (2 * i) | (bf_hi(u[i]) > 0.f ? 1u : 0u) << (2 * i + 1);
      a.h2[(long long)blockIdx.x * 128 + tid] = m;
    }
    if (layer == 0) {
      tc::fence_async_smem();
      tc::fence_before_sync();
      __syncthreads();
      tc::fence_after_sync();
    } else {
      __syncthreads();  // every thread is past the tiles before they are overwritten
#pragma unroll
      for (int i = 0; i < 16; ++i) sH[tid][i] = u[i];
      __syncthreads();
      // pooling: channel pair (2 cp, 2 cp + 1) of cell l, summed over its f^2 rows in order
      for (int idx = tid; idx < a.cpb * (kC / 2); idx += 128) {
        const int l = idx >> 4, cp = idx & 15;
        const long long cl = (long long)blockIdx.x * a.cpb + l;
        if (cl >= a.cells || 2 * cp >= kStartCh) continue;
        float s0 = 0.f, s1 = 0.f;
        for (int p = 0; p < ff; ++p) {
          const uint32_t w = sH[l * ff + p][cp];
          s0 += bf_lo(w);
          s1 += bf_hi(w);
        }
        a.c0[cl * kC + 2 * cp] = __float2bfloat16(s0 / float(ff));
        if (2 * cp + 1 < kStartCh) a.c0[cl * kC + 2 * cp + 1] = __float2bfloat16(s1 / float(ff));
      }
      if (start_row) {
#pragma unroll
        for (int c = 0; c < 3; ++c) a.c0[(long long)cell * kC + kStartCh + c] = __float2bfloat16(zs[c]);
      }
    }
  }
  if (!ok) {
    tc::mbar_wait(&mbar, uint32_t(layer & 1), kWaitTries);
    if (tid == 0) atomicExch(a.err, 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 32);
}

// --------------------------------------------------------------- k_pix_bwd
struct PixBwd {
  const __nv_bfloat16* gc0;           // gradient of c0 [cells][32]
  const __nv_bfloat16 *x0, *h1;       // saved by k_pix: [blocks 128][32]
  const uint32_t* h2;                 // saved by k_pix: bit c of row r set where h2 > 0
  const __nv_bfloat16* w2;            // [32][32]
  int blocks, cells, cpb, ff;         // row blocks of k_pix, superpixels, cells per block, patches per cell
  unsigned rff;                       // floor(2^32 / ff) + 1: p / ff = umulhi(p, rff) for a row p < 128 (ff > 1)
  float* part;                        // block b's sums at part + b stride: W1, b1, W2, b2 as in the parameters
  long long stride;
};
constexpr int kPixTile = 4 * kRowTile;  // 128 rows x 32 channels
// g2, g1, h1 and its ones, x0 and its ones, W2
constexpr int kPixBwdH1 = 2 * kPixTile, kPixBwdX0 = kPixBwdH1 + kPixTile + kRowTile,
              kPixBwdW = kPixBwdX0 + kPixTile + kRowTile;
constexpr int kPixBwdCols = 128;        // accumulators: W2 and b2 48, W1 and b1 48, data gradient 32
constexpr int kPixBwdPerSm = 4;         // resident blocks: 4 x 128 TMEM columns, and no fifth by shared memory
constexpr int kPixBwdSmem = 46 * 1024;
static_assert(kPixBwdW + 4 * kWLd <= kPixBwdSmem && kPixTile + kMnSpan <= kPixBwdSmem, "shared memory");
static_assert(kPixBwdX0 + 6 * kRowTile <= kPixBwdSmem, "shared memory");

// Backward pass of the pixel level over the 128-row blocks of k_pix:
//   g2 = gradient of c0 / f^2 where h2 > 0 (average pooling, ReLU; channels
//        kStartCh.. of c0 are inputs), BF16
//   W2 += g2^T h1, b2 += g2^T 1, g1 = (g2 W2 where h1 > 0), BF16
//   W1 += g1^T x0, b1 += g1^T 1
// with g2 and g1 in shared memory only.  A tile of rows lies as in the 3 x 3
// layers (groups of 8 channels, 16 bytes per row), so that g2 is the K-major
// operand of the data gradient and the MN-major one of the weight gradient.
// The weight gradients stay in tensor memory over the block's tiles.
// Bound by the latency of a tile's steps (load, MMA, mask, MMA) at four blocks
// per SM (128 TMEM columns, 46 KB each); the loads of the next tile are in
// flight, in registers, during the MMAs of this one.  At 32 images of
// 481x321, v = 15: 29 us (48 us without loading ahead), 74 MB read, in place
// of a pooling pass (59 us), a data gradient and two weight-gradient GEMMs
// (2.5 ms) that read g2 and g1 four times from memory.
__global__ void __launch_bounds__(128, kPixBwdPerSm) k_pix_bwd(PixBwd a, int* err) {
  extern __shared__ __align__(128) unsigned char smem3[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_sh;
  const int tid = threadIdx.x, warp = tid >> 5;
  unsigned char *pG2 = smem3, *pG1 = smem3 + kPixTile, *pH1 = smem3 + kPixBwdH1, *pX0 = smem3 + kPixBwdX0;
  const uint32_t sG2 = tc::smem_u32(pG2), sG1 = sG2 + kPixTile, sH1 = sG2 + kPixBwdH1, sX0 = sG2 + kPixBwdX0,
                 sW = sG2 + kPixBwdW;
  if (warp == 0) {
    tc::tmem_alloc(&tmem_sh, kPixBwdCols);
    tc::tmem_relinquish();
  }
  if (tid == 0) tc::mbar_init(&mbar, 1);
  fill_ones(pH1 + kPixTile, kRowTile);
  fill_ones(pX0 + kPixTile, kRowTile);
  cp_async16(sW + (tid & 3) * kWLd + (tid >> 2) * 16, a.w2 + (tid >> 2) * kC + (tid & 3) * 8, true);
  cp_async_wait_all();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tW2 = tmem_sh, tW1 = tW2 + 48, tD = tW2 + 96;
  constexpr uint32_t idD = tc::idesc_bf16_f32(128, 32) | tc::kTransB;
  constexpr uint32_t id48 = tc::idesc_bf16_f32(128, 48) | tc::kTransA | tc::kTransB;
  const float inv = 1.f / float(a.ff);
  bool ok = true;
  uint32_t phase = 0;
  // a tile's loads, held in registers from the previous tile's MMAs on
  uint4 xv[4], hv[4], gv[4];
  uint32_t h2[4];
  auto load = [&](int b) {
    const long long r0 = (long long)b * 128;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = tid + 128 * j, p = i >> 2, gr = i & 3;
      const int lc = a.ff == 1 ? p : int(__umulhi(unsigned(p), a.rff)), cell = b * a.cpb + lc;
      const bool in = lc < a.cpb && cell < a.cells;
      hv[j] = __ldg(reinterpret_cast<const uint4*>(a.h1 + r0 * kC) + i);
      xv[j] = __ldg(reinterpret_cast<const uint4*>(a.x0 + r0 * kC) + i);
      h2[j] = in ? __ldg(a.h2 + r0 + p) : 0u;
      gv[j] = in ? __ldg(reinterpret_cast<const uint4*>(a.gc0 + (long long)cell * kC + gr * 8)) : make_uint4(0, 0, 0, 0);
    }
  };
  load(blockIdx.x);  // blockIdx.x < a.blocks
  for (int b = blockIdx.x; b < a.blocks; b += gridDim.x) {
    const uint32_t acc0 = b == int(blockIdx.x) ? 0u : 1u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = tid + 128 * j, p = i >> 2, gr = i & 3;
      *reinterpret_cast<uint4*>(pH1 + gr * kRowTile + p * 16) = hv[j];
      *reinterpret_cast<uint4*>(pX0 + gr * kRowTile + p * 16) = xv[j];
      uint32_t m = h2[j] >> (gr * 8);
      if (gr == 3) m &= (1u << (kStartCh - 24)) - 1u;  // channels kStartCh.. are inputs
      const uint32_t* gw = reinterpret_cast<const uint32_t*>(&gv[j]);
      uint32_t u[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        u[k] = pack2((m >> (2 * k)) & 1u ? bf_lo(gw[k]) * inv : 0.f, (m >> (2 * k + 1)) & 1u ? bf_hi(gw[k]) * inv : 0.f);
      *reinterpret_cast<uint4*>(pG2 + gr * kRowTile + p * 16) = make_uint4(u[0], u[1], u[2], u[3]);
    }
    if (b + int(gridDim.x) < a.blocks) load(b + gridDim.x);
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
#pragma unroll
      for (int kk = 0; kk < 2; ++kk)
        tc::mma_bf16(tD, tc::smem_desc(sG2 + 2 * kk * kRowTile, kRowTile, 128), tc::smem_desc(sW + kk * 256, 128, kWLd),
                     idD, kk);
      tc::mma_commit(&mbar);
      for (int kk = 0; kk < 8; ++kk) {
        const uint64_t ad = tc::smem_desc(sG2 + kk * 256, 128, kRowTile);
        tc::mma_bf16(tW2, ad, tc::smem_desc(sH1 + kk * 256, 128, kRowTile), id48, kk ? 1u : acc0);
      }
    }
    bool w = tc::mbar_wait(&mbar, phase & 1u, kWaitTries);
    ok = __syncthreads_and(w) != 0;
    if (!ok) break;
    ++phase;
    tc::fence_after_sync();
    // g1 of row tid: the data gradient where h1 > 0
    float d[32];
#pragma unroll
    for (int c0 = 0; c0 < 32; c0 += 16) {
      float v[16];
      tc::tmem_ld16(tD + (uint32_t(warp * 32) << 16) + uint32_t(c0), v);
#pragma unroll
      for (int i = 0; i < 16; ++i) d[c0 + i] = v[i];
    }
#pragma unroll
    for (int gr = 0; gr < 4; ++gr) {
      const uint4 m = *reinterpret_cast<const uint4*>(pH1 + gr * kRowTile + tid * 16);
      const uint32_t* mw = reinterpret_cast<const uint32_t*>(&m);
      uint32_t u[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        u[k] = pack2(bf_lo(mw[k]) > 0.f ? d[gr * 8 + 2 * k] : 0.f, bf_hi(mw[k]) > 0.f ? d[gr * 8 + 2 * k + 1] : 0.f);
      *reinterpret_cast<uint4*>(pG1 + gr * kRowTile + tid * 16) = make_uint4(u[0], u[1], u[2], u[3]);
    }
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      for (int kk = 0; kk < 8; ++kk) {
        const uint64_t ad = tc::smem_desc(sG1 + kk * 256, 128, kRowTile);
        tc::mma_bf16(tW1, ad, tc::smem_desc(sX0 + kk * 256, 128, kRowTile), id48, kk ? 1u : acc0);
      }
      tc::mma_commit(&mbar);
    }
    w = tc::mbar_wait(&mbar, phase & 1u, kWaitTries);  // the tiles are refilled next
    ok = __syncthreads_and(w) != 0;
    if (!ok) break;
    ++phase;
  }
  tc::fence_after_sync();
  if (!ok) {
    tc::mbar_wait(&mbar, phase & 1u, kWaitTries);
    if (tid == 0) atomicExch(err, 1);
  } else if (warp == 0) {  // accumulator row = output channel = lane
    float* out = a.part + blockIdx.x * a.stride;
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      float* o = out + l * (kC * kC + kC);
      for (int c0 = 0; c0 < 32; c0 += 16) {
        float v[16];
        tc::tmem_ld16((l ? tW2 : tW1) + uint32_t(c0), v);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          reinterpret_cast<float4*>(o + tid * kC + c0)[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
      }
      float v[16];
      tc::tmem_ld16((l ? tW2 : tW1) + 32u, v);
      o[kC * kC + tid] = v[0];
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tW2, kPixBwdCols);
}

// ------------------------------------------------------------ elementwise
// Mean squared error over the used outputs: gradient (BF16) into g, per-block
// sums of squares (FP64) into lpart.
__global__ void __launch_bounds__(256) k_loss(const float* __restrict__ out, const float* __restrict__ target,
                                              long long cells, __nv_bfloat16* __restrict__ g,
                                              double* __restrict__ lpart) {
  __shared__ double red[256];
  double s = 0.0;
  const float scale = float(2.0 / double(cells * kUsed));
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < cells * kOut;
       i += (long long)gridDim.x * blockDim.x) {
    const long long cell = i / kOut;
    const int j = int(i - cell * kOut);
    float gv = 0.f;
    if (j < kUsed) {
      const float d = out[i] - target[cell * kUsed + j];
      s += double(d) * double(d);
      gv = scale * d;
    }
    g[i] = __float2bfloat16(gv);
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) lpart[blockIdx.x] = red[0];
}

// Sum of the blocks' weight-gradient partials (rows in parameter order; a
// fixed order: G interleaved sums, then those in turn).  A block of 256
// threads takes 256 / G parameters, thread (g, l) rows g, g + G, ...
template <int G>
__device__ __forceinline__ void reduce_rows(const float* __restrict__ p, int rows, int stride, int i0,
                                            float* __restrict__ out) {
  constexpr int L = 256 / G;
  __shared__ float red[G][L + 1];
  const int l = threadIdx.x % L, g = threadIdx.x / L, i = i0 + l;
  float s = 0.f;
  if (i < stride) {
#pragma unroll 4
    for (int r = g; r < rows; r += G) s += __ldg(p + (long long)r * stride + i);
  }
  red[g][l] = s;
  __syncthreads();
  if (g == 0 && i < stride) {
#pragma unroll
    for (int k = 1; k < G; ++k) s += red[k][l];
    out[i] = s;
  }
}
// The first `split` parameters (the pixel level's) over n0 rows of p0: up to
// 608 of them, whose chain of loads sets the time, so 32 sums per parameter;
// the others over n1 <= 38 rows of p1, 8 sums per parameter.
__global__ void __launch_bounds__(256) k_grad_reduce(const float* __restrict__ p0, int n0, int split,
                                                     const float* __restrict__ p1, int n1, int total,
                                                     float* __restrict__ grad) {
  const int first = (split + 7) / 8;
  if (int(blockIdx.x) < first) reduce_rows<32>(p0, n0, split, blockIdx.x * 8, grad);
  else reduce_rows<8>(p1, n1, total - split, (blockIdx.x - first) * 32, grad + split);
}

// Adam (Kingma and Ba, 2015) on the FP32 master weights; refreshes the BF16 copy.
__global__ void k_adam(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, BfParams wb, int n, float lr, float b1,
                       float b2, float eps, float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    w[i] = wi;
    store_bf16(wb, i, wi);
  }
}

__global__ void k_to_bf16(const float* __restrict__ a, BfParams b, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    store_bf16(b, i, a[i]);
}

// Targets from fitted parameters of B images of geometry g (theta and the
// CIELAB planes laid out image after image); units as the network outputs.
__global__ void k_targets(const double* __restrict__ theta, const float* __restrict__ lab, int B, Geom g,
                          double lambda_c, float* __restrict__ t) {
  const long long total = (long long)B * g.K;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int img = int(i / g.K), k = int(i - (long long)img * g.K);
    const int kx = k % g.nx, ky = k / g.nx;
    const int x = kx * g.v + g.v / 2, y = ky * g.v + g.v / 2;
    const long long N = (long long)g.W * g.H, j = (long long)y * g.W + x;
    const float* P = lab + (long long)img * 3 * N;
    const double* th = theta + i * kTheta;
    float* o = t + i * kUsed;
    const double v = g.v, l2 = lambda_c * lambda_c;
    o[0] = float((th[0] - x) / v);
    o[1] = float((th[1] - y) / v);
    o[2] = float((th[2] - double(P[j])) / kColourUnit);
    o[3] = float((th[3] - double(P[N + j])) / kColourUnit);
    o[4] = float((th[4] - double(P[2 * N + j])) / kColourUnit);
    o[5] = float(log(th[5] / (v * v)));
    o[6] = float(log(th[7] / (v * v)));
    o[7] = float(log(th[8] / l2));
    o[8] = float(log(th[11] / l2));
    o[9] = float(log(th[13] / l2));
  }
}

// theta_0 from the network outputs (the inverse of the target map): spatial
// mean clipped to the three cells around the seed's own, [(k_x - 1) v,
// (k_x + 2) v] x [(k_y - 1) v, (k_y + 2) v] (the span of Eq. Ik's window
// without its clamp to the image), axis-aligned covariances with
// the diagonal (their eigenvalues) floored at eps (Eq. mlams, mlamc); then
// the packed E-step coefficients.  Superpixel i reads its 5 mean offsets at
// dmu + i ds and its 5 log-eigenvalues at logeig + i ls (the network's output
// rows: ds = ls = 16; a caller's arrays: 5).
__global__ void k_init_from_net(const float* __restrict__ dmu, int ds, const float* __restrict__ logeig, int ls,
                                const float* __restrict__ lab, int B, Geom g, double lambda_c, double eps_s,
                                double eps_c, double* __restrict__ theta, float* __restrict__ gp,
                                unsigned long long* __restrict__ counters) {
  const long long total = (long long)B * g.K;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int img = int(i / g.K), k = int(i - (long long)img * g.K);
    const int kx = k % g.nx, ky = k / g.nx;
    const int x = kx * g.v + g.v / 2, y = ky * g.v + g.v / 2;
    const long long N = (long long)g.W * g.H, j = (long long)y * g.W + x;
    const float* P = lab + (long long)img * 3 * N;
    float o[10];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      o[q] = dmu[i * ds + q];
      o[5 + q] = logeig[i * ls + q];
    }
    const double v = g.v, l2 = lambda_c * lambda_c;
    double mu[5] = {x + v * widen(o[0]), y + v * widen(o[1]), widen(P[j]) + kColourUnit * widen(o[2]),
                    widen(P[N + j]) + kColourUnit * widen(o[3]),
                    widen(P[2 * N + j]) + kColourUnit * widen(o[4])};
    mu[0] = fmin(fmax(mu[0], double(kx - 1) * v), double(kx + 2) * v);
    mu[1] = fmin(fmax(mu[1], double(ky - 1) * v), double(ky + 2) * v);
    const float lo = -10.f, hi = 10.f;
    const double cs[3] = {fmax(v * v * exp(widen(fminf(fmaxf(o[5], lo), hi))), eps_s), 0.0,
                          fmax(v * v * exp(widen(fminf(fmaxf(o[6], lo), hi))), eps_s)};
    const double cc[6] = {fmax(l2 * exp(widen(fminf(fmaxf(o[7], lo), hi))), eps_c), 0.0, 0.0,
                          fmax(l2 * exp(widen(fminf(fmaxf(o[8], lo), hi))), eps_c), 0.0,
                          fmax(l2 * exp(widen(fminf(fmaxf(o[9], lo), hi))), eps_c)};
    double* th = theta + i * kTheta;
    bool fin = true;
    for (int q = 0; q < 5; ++q) {
      th[q] = mu[q];
      fin = fin && isfinite(mu[q]);
    }
    for (int q = 0; q < 3; ++q) th[5 + q] = cs[q];
    for (int q = 0; q < 6; ++q) th[8 + q] = cc[q];
    th[14] = th[15] = 0.0;
    fin = pack_gp<double>(mu, cs, cc, double(kx * g.v), double(ky * g.v), gp + i * kGP) && fin;
    if (!fin) atomicAdd(counters + CNT_NONFINITE, 1ull);
  }
}

// Self-test of the bounded waits: allocates TMEM like the network kernels,
// waits on an mbarrier that nothing arrives on for max_tries polls, waits
// once more (bounded), frees the TMEM and records that it gave up.
__global__ void __launch_bounds__(128) k_wait_selftest(uint32_t max_tries, int* gave_up) {
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t tmem_sh;
  const int tid = threadIdx.x, warp = tid >> 5;
  if (warp == 0) {
    tc::tmem_alloc(&tmem_sh, 32);
    tc::tmem_relinquish();
  }
  if (tid == 0) tc::mbar_init(&mbar, 1);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_sh;
  const bool ok = __syncthreads_and(tc::mbar_wait(&mbar, 0, max_tries)) != 0;
  if (!ok) {
    tc::mbar_wait(&mbar, 0, max_tries);
    if (tid == 0) atomicExch(gave_up, 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 32);
}

int grid_for(long long n, int block) {
  long long b = (n + block - 1) / block;
  b = std::min<long long>(b, 152LL * 16);
  return int(std::max<long long>(b, 1));
}

}  // namespace cnn

cudaError_t bounds_take_cnn(unsigned long long* word) {
  *word = 0ull;
#ifdef GMMSP_CHECK_BOUNDS
  cudaError_t e = cudaMemcpyFromSymbol(word, g_bounds_word, sizeof(*word));
  if (e != cudaSuccess) return e;
  const unsigned long long zero = 0ull;
  return cudaMemcpyToSymbol(g_bounds_word, &zero, sizeof(zero));
#else
  return cudaSuccess;
#endif
}

}  // namespace gmmsp

using gmmsp::BatchImage;
using gmmsp::Geom;
using gmmsp::rgb2lab_const;
using namespace gmmsp::cnn;

// --------------------------------------------------------------- the object
struct gmmsp_net_s {
  int v = 0, f = 0, cpb = 0;
  cudaStream_t stream = nullptr;
  ParamLayout pl{};
  void* pslab = nullptr;  // parameters, Adam state, gradients, error word
  float *w32 = nullptr, *m = nullptr, *vv = nullptr, *grad = nullptr;
  __nv_bfloat16* wbf = nullptr;
  unsigned char* wst = nullptr;  // the 3 x 3 layers' weights as the kernels stage them
  int* err = nullptr;
  float* srgb = nullptr;  // the converting mode's sRGB table
  long long adam_t = 0;
  int sms = 152;          // SMs of the device
  // workspace (grown on demand, never during stream capture)
  void* wslab = nullptr;
  long long cap_cells = 0;
  bool cap_train = false;
  long long generation = 0;
  __nv_bfloat16* c[4] = {};
  __nv_bfloat16 *x0 = nullptr, *h1 = nullptr, *gout = nullptr;
  uint32_t* h2 = nullptr;
  __nv_bfloat16* gc[4] = {};
  float *out = nullptr;
  float *wpart0 = nullptr, *wpart1 = nullptr;  // weight-gradient partials per block: layers 0-1, layers 2-5
  double* lpart = nullptr;
  long long last_cells = 0;  // superpixels of the last forward pass
  std::unique_ptr<char[]> back;  // host side of grad_to_host: the gradient, the loss sums and the error word
  std::string msg;
};

namespace {

size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

gmmsp_status nfail(gmmsp_net n, gmmsp_status s, const std::string& m) {
  if (n) n->msg = m;
  return s;
}

#define GN_CHECK(n, call)                                                              \
  do {                                                                                 \
    cudaError_t e_ = (call);                                                           \
    if (e_ != cudaSuccess)                                                             \
      return nfail((n), e_ == cudaErrorMemoryAllocation ? GMMSP_E_NOMEM : GMMSP_E_CUDA, \
                   std::string(#call) + ": " + cudaGetErrorString(e_));                \
  } while (0)

BfParams bf_params(gmmsp_net n) {
  BfParams p{n->wbf, n->wst, {}, {}};
  for (int l = 0; l < 4; ++l) {
    p.w[l] = n->pl.w[l + 2];
    p.n[l] = n->pl.cout[l + 2] * 288;
  }
  return p;
}

long long nblocks_of(gmmsp_net n, long long cells) { return (cells + n->cpb - 1) / n->cpb; }

// The EM seed grid of a W x H image at the network's spacing (Eq. nxyK).
bool net_geom(gmmsp_net n, int W, int H, Geom* g) {
  if (W < n->v || H < n->v) return false;
  g->W = W; g->H = H; g->v = n->v;
  g->nx = W / n->v; g->ny = H / n->v;
  g->K = g->nx * g->ny;
  g->ncx = (W + n->v - 1) / n->v;
  g->ncy = (H + n->v - 1) / n->v;
  g->ncells = g->ncx * g->ncy;
  return true;
}

// Largest batch (in superpixels) the kernels index with 32-bit rows.
bool cells_fit(gmmsp_net n, long long cells) { return nblocks_of(n, cells) * 128 <= (1LL << 30); }

gmmsp_status reserve(gmmsp_net n, long long cells, bool train) {
  if (cells <= n->cap_cells && (!train || n->cap_train)) return GMMSP_OK;
  cells = std::max(cells, n->cap_cells);
  train = train || n->cap_train;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(n->stream, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone)
    return nfail(n, GMMSP_E_STATE, "network workspace must be reserved before stream capture");
  const long long nrows = nblocks_of(n, cells) * 128;
  const size_t act = up256(size_t(cells) * kC * 2);
  const size_t pix = up256(size_t(nrows) * kC * 2);
  size_t off = 0;
  const size_t o_c = off;   off += 4 * act;
  const size_t o_out = off; off += up256(size_t(cells) * kOut * sizeof(float));
  size_t o_x0 = 0, o_gout = 0, o_gc = 0, o_wp0 = 0, o_wp1 = 0;
  if (train) {
    o_x0 = off;   off += 2 * pix + up256(size_t(nrows) * 4);  // x0, h1, the bits of h2
    o_gout = off; off += up256(size_t(cells) * kOut * 2);
    o_gc = off;   off += 4 * act;
    o_wp0 = off;  off += up256(size_t(n->sms) * kPixBwdPerSm * pix_params(n->pl) * sizeof(float));
    o_wp1 = off;  off += up256(size_t(std::max(1, n->sms / 4)) * (n->pl.total - pix_params(n->pl)) * sizeof(float));
  }
  if (n->wslab) {
    GN_CHECK(n, cudaStreamSynchronize(n->stream));
    cudaFree(n->wslab);
    n->wslab = nullptr;
    n->cap_cells = 0;
    n->cap_train = false;
  }
  void* slab = nullptr;
  GN_CHECK(n, cudaMalloc(&slab, off));
  ++n->generation;
  char* b = static_cast<char*>(slab);
  n->wslab = slab;
  for (int i = 0; i < 4; ++i) n->c[i] = reinterpret_cast<__nv_bfloat16*>(b + o_c + i * act);
  n->out = reinterpret_cast<float*>(b + o_out);
  if (train) {
    n->x0 = reinterpret_cast<__nv_bfloat16*>(b + o_x0);
    n->h1 = reinterpret_cast<__nv_bfloat16*>(b + o_x0 + pix);
    n->h2 = reinterpret_cast<uint32_t*>(b + o_x0 + 2 * pix);
    n->gout = reinterpret_cast<__nv_bfloat16*>(b + o_gout);
    for (int i = 0; i < 4; ++i) n->gc[i] = reinterpret_cast<__nv_bfloat16*>(b + o_gc + i * act);
    n->wpart0 = reinterpret_cast<float*>(b + o_wp0);
    n->wpart1 = reinterpret_cast<float*>(b + o_wp1);
  } else {
    n->x0 = n->h1 = n->gout = nullptr;
    for (auto& p : n->gc) p = nullptr;
    n->h2 = nullptr;
    n->wpart0 = n->wpart1 = nullptr;
  }
  n->cap_cells = cells;
  n->cap_train = train;
  return GMMSP_OK;
}

// One tile per step on as many blocks as are resident at once (shared memory
// and the 512 TMEM columns: 16 blocks of 32), so that each stages the weights
// once.
template <bool DGRAD, int GC, int N>
cudaError_t launch_conv3(gmmsp_net n, const Conv3& c, cudaStream_t s) {
  const int smem = kWBytes + GC * c.g.GS;
  const int per = std::max(1, std::min(16, 228 * 1024 / (smem + 2048)));
  const unsigned blocks = unsigned(std::min(c.g.tiles, n->sms * per));
  k_conv3<DGRAD, GC, N><<<blocks, 128, smem, s>>>(c, n->err);
  return cudaGetLastError();
}

// Forward pass; out receives [B K][16] FP32.  Training also stores x0, h1, h2.
// With rgb non-null the first kernel reads the cells' pixels as RGB8 through
// the batch table and writes their CIELAB values to lab_out.
gmmsp_status enqueue_forward(gmmsp_net n, const float* lab, int B, const Geom& g, float* out, bool train,
                             cudaStream_t s, const BatchImage* rgb = nullptr, float* lab_out = nullptr) {
  const long long cells = (long long)B * g.K;
  n->last_cells = cells;
  PixArgs a{};
  a.lab = lab;
  a.rgb = rgb;
  a.lab_out = lab_out;
  a.srgb = n->srgb;
  if (rgb) a.k = rgb2lab_const();
  a.W = g.W; a.H = g.H; a.v = g.v; a.f = n->f; a.nx = g.nx; a.ny = g.ny;
  a.cells = int(cells);
  a.cpb = n->cpb;
  a.w1 = n->wbf + n->pl.w[0];
  a.b1 = n->w32 + n->pl.b[0];
  a.w2 = n->wbf + n->pl.w[1];
  a.b2 = n->w32 + n->pl.b[1];
  a.c0 = n->c[0];
  a.x0 = train ? n->x0 : nullptr;
  a.h1 = train ? n->h1 : nullptr;
  a.h2 = train ? n->h2 : nullptr;
  a.err = n->err;
  const unsigned pblocks = unsigned(nblocks_of(n, cells));
  if (train) k_pix<true><<<pblocks, 128, 0, s>>>(a);
  else k_pix<false><<<pblocks, 128, 0, s>>>(a);
  GN_CHECK(n, cudaGetLastError());
  Conv3 c{};
  c.g = grid3_of(B, g.ny, g.nx);
  for (int l = 2; l < 6; ++l) {
    c.a = n->c[l - 2];
    c.w = n->wst + (l - 2) * kWBytes;
    c.bias = n->w32 + n->pl.b[l];
    if (l < 5) {
      c.y = n->c[l - 1];
      GN_CHECK(n, (launch_conv3<false, 4, 32>(n, c, s)));
    } else {
      c.y32 = out;
      GN_CHECK(n, (launch_conv3<false, 4, 16>(n, c, s)));
    }
  }
  return GMMSP_OK;
}

// Forward, loss, and the gradient of every parameter into n->grad.
gmmsp_status enqueue_grad(gmmsp_net n, const float* lab, int B, const Geom& g, const float* target,
                          cudaStream_t s) {
  gmmsp_status st = enqueue_forward(n, lab, B, g, n->out, true, s);
  if (st != GMMSP_OK) return st;
  const long long cells = (long long)B * g.K;
  k_loss<<<kLossBlocks, 256, 0, s>>>(n->out, target, cells, n->gout, n->lpart);
  GN_CHECK(n, cudaGetLastError());
  // the 3 x 3 layers, last to first
  const int np0 = pix_params(n->pl), np1 = n->pl.total - np0;
  const Grid3 g3 = grid3_of(B, g.ny, g.nx);
  const __nv_bfloat16* gy = n->gout;
  Wgrad3 w{};
  w.g = g3;
  w.part = n->wpart1;
  w.stride = np1;
  for (int l = 5; l >= 2; --l) {
    w.x[l - 2] = n->c[l - 2];
    w.gy[l - 2] = gy;
    w.off[l - 2] = n->pl.w[l] - np0;
    Conv3 c{};
    c.g = g3;
    c.a = gy;
    c.w = n->wst + (l - 2) * kWBytes;
    c.y = n->gc[l - 2];
    c.mask = l > 2 ? n->c[l - 2] : nullptr;  // c0 is a pooled value with no ReLU of its own
    if (l == 5) GN_CHECK(n, (launch_conv3<true, 2, 32>(n, c, s)));
    else GN_CHECK(n, (launch_conv3<true, 4, 32>(n, c, s)));
    gy = c.y;
  }
  const unsigned wblocks = unsigned(std::min(g3.tiles, std::max(1, n->sms / 4)));
  k_wgrad3<<<dim3(wblocks, 4), 128, std::max(kMnSpan, 4 * kRowTile + 6 * g3.GS), s>>>(w, n->err);
  GN_CHECK(n, cudaGetLastError());
  // the pixel level, then the sums over the blocks
  PixBwd p{};
  p.gc0 = gy;
  p.x0 = n->x0;
  p.h1 = n->h1;
  p.h2 = n->h2;
  p.w2 = n->wbf + n->pl.w[1];
  p.blocks = int(nblocks_of(n, cells));
  p.cells = int(cells);
  p.cpb = n->cpb;
  p.ff = n->f * n->f;
  p.rff = unsigned((1ull << 32) / unsigned(p.ff)) + 1u;
  p.part = n->wpart0;
  p.stride = np0;
  const unsigned pblocks = unsigned(std::min(p.blocks, n->sms * kPixBwdPerSm));
  k_pix_bwd<<<pblocks, 128, kPixBwdSmem, s>>>(p, n->err);
  GN_CHECK(n, cudaGetLastError());
  k_grad_reduce<<<unsigned((np0 + 7) / 8 + (np1 + 31) / 32), 256, 0, s>>>(n->wpart0, int(pblocks), np0, n->wpart1,
                                                                 int(wblocks), n->pl.total, n->grad);
  GN_CHECK(n, cudaGetLastError());
  return GMMSP_OK;
}

gmmsp_status check_err(gmmsp_net n) {
  int e = 0;
  GN_CHECK(n, cudaMemcpyAsync(&e, n->err, sizeof(int), cudaMemcpyDeviceToHost, n->stream));
  GN_CHECK(n, cudaStreamSynchronize(n->stream));
  if (e) return nfail(n, GMMSP_E_TIMEOUT, "a tensor-core kernel gave up waiting on its MMA barrier");
  return GMMSP_OK;
}

// The gradient and / or the loss of the last backward pass to the host, and
// the error word: one copy of the memory that holds them side by side.
gmmsp_status grad_to_host(gmmsp_net n, long long cells, float* grad_host, double* loss_host) {
  const char* from = grad_host ? reinterpret_cast<const char*>(n->grad) : reinterpret_cast<const char*>(n->lpart);
  const size_t bytes = size_t(reinterpret_cast<const char*>(n->err + 1) - from);
  GN_CHECK(n, cudaMemcpyAsync(n->back.get(), from, bytes, cudaMemcpyDeviceToHost, n->stream));
  GN_CHECK(n, cudaStreamSynchronize(n->stream));
  auto at = [&](const void* dev) { return n->back.get() + (static_cast<const char*>(dev) - from); };
  int e = 0;
  memcpy(&e, at(n->err), sizeof(int));
  if (grad_host) memcpy(grad_host, at(n->grad), size_t(n->pl.total) * 4);
  if (e) return nfail(n, GMMSP_E_TIMEOUT, "a tensor-core kernel gave up waiting on its MMA barrier");
  if (loss_host) {
    double lp[kLossBlocks];
    memcpy(lp, at(n->lpart), sizeof(lp));
    double s = 0.0;
    for (int i = 0; i < kLossBlocks; ++i) s += lp[i];
    *loss_host = s / double(cells * kUsed);
  }
  return GMMSP_OK;
}

}  // namespace

// ------------------------------------------------ library-internal entry points
namespace gmmsp {

gmmsp_status net_reserve(gmmsp_net n, int B, const Geom& g, std::string* why) {
  if (!n) return GMMSP_E_INVALID;
  if (g.v != n->v) {
    if (why) *why = "the network's spacing differs from the context's";
    return GMMSP_E_INVALID;
  }
  if (!cells_fit(n, (long long)B * g.K)) {
    if (why) *why = "batch too large for the network";
    return GMMSP_E_INVALID;
  }
  const gmmsp_status st = reserve(n, (long long)B * g.K, false);
  if (st != GMMSP_OK && why) *why = n->msg;
  return st;
}

long long net_generation(gmmsp_net n) { return n ? n->generation : -1; }

cudaError_t net_enqueue_init(gmmsp_net n, float* lab, const BatchImage* rgb, int B, const Geom& g,
                             double lambda_c, double eps_s, double eps_c, double* theta, float* gp,
                             unsigned long long* counters, cudaStream_t s) {
  if ((long long)B * g.K > n->cap_cells) return cudaErrorInvalidValue;
  if (enqueue_forward(n, lab, B, g, n->out, false, s, rgb, rgb ? lab : nullptr) != GMMSP_OK)
    return cudaErrorLaunchFailure;
  return launch_init_from_outputs(n->out, kOut, n->out + 5, kOut, lab, B, g, lambda_c, eps_s, eps_c, theta, gp,
                                  counters, s);
}

cudaError_t launch_init_from_outputs(const float* dmu, int ds, const float* logeig, int ls, const float* lab, int B,
                                     const Geom& g, double lambda_c, double eps_s, double eps_c, double* theta,
                                     float* gp, unsigned long long* counters, cudaStream_t s) {
  const long long total = (long long)B * g.K;
  k_init_from_net<<<grid_for(total, 128), 128, 0, s>>>(dmu, ds, logeig, ls, lab, B, g, lambda_c, eps_s, eps_c,
                                                       theta, gp, counters);
  return cudaGetLastError();
}

cudaError_t launch_targets(const double* theta, const float* lab, int B, const Geom& g, double lambda_c,
                           float* target, cudaStream_t s) {
  const long long total = (long long)B * g.K;
  k_targets<<<grid_for(total, 128), 128, 0, s>>>(theta, lab, B, g, lambda_c, target);
  return cudaGetLastError();
}

}  // namespace gmmsp

// --------------------------------------------------------------------- C ABI
extern "C" {

long long gmmsp_net_param_count(void) { return param_layout().total; }

gmmsp_status gmmsp_net_create(gmmsp_net* out, int spacing, void* stream) {
  if (!out) return GMMSP_E_INVALID;
  *out = nullptr;
  if (spacing < 3 || spacing > 33 || spacing % 3 != 0) return GMMSP_E_INVALID;
  gmmsp_net n = new (std::nothrow) gmmsp_net_s();
  if (!n) return GMMSP_E_NOMEM;
  n->v = spacing;
  n->f = spacing / 3;
  n->cpb = 128 / (n->f * n->f);
  n->stream = static_cast<cudaStream_t>(stream);
  n->pl = param_layout();
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&n->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    cudaGetLastError();
    delete n;
    return GMMSP_E_CUDA;
  }
  const size_t np = size_t(n->pl.total);
  size_t off = 0;
  const size_t o_w = off; off += up256(np * 4);
  const size_t o_m = off; off += up256(np * 4);
  const size_t o_v = off; off += up256(np * 4);
  // gradient, loss sums and error word side by side: read back in one copy
  const size_t o_g = off; off += up256(np * 4);
  const size_t o_l = off; off += kLossBlocks * sizeof(double);
  const size_t o_e = off; off += 256;
  const size_t o_b = off; off += up256(np * 2);
  const size_t o_s = off; off += up256(4 * kWBytes);
  const size_t o_t = off; off += 256 * 4;
  n->back.reset(new (std::nothrow) char[o_e + sizeof(int) - o_g]);
  if (!n->back) {
    delete n;
    return GMMSP_E_NOMEM;
  }
  const char* inj = getenv("GMMSP_FAIL_ALLOC");
  cudaError_t e = (inj && inj[0] == '1') ? cudaErrorMemoryAllocation : cudaMalloc(&n->pslab, off);
  if (e != cudaSuccess) {
    cudaGetLastError();
    delete n;
    return e == cudaErrorMemoryAllocation ? GMMSP_E_NOMEM : GMMSP_E_CUDA;
  }
  char* b = static_cast<char*>(n->pslab);
  n->w32 = reinterpret_cast<float*>(b + o_w);
  n->m = reinterpret_cast<float*>(b + o_m);
  n->vv = reinterpret_cast<float*>(b + o_v);
  n->grad = reinterpret_cast<float*>(b + o_g);
  n->wbf = reinterpret_cast<__nv_bfloat16*>(b + o_b);
  n->wst = reinterpret_cast<unsigned char*>(b + o_s);
  n->lpart = reinterpret_cast<double*>(b + o_l);
  n->err = reinterpret_cast<int*>(b + o_e);
  n->srgb = reinterpret_cast<float*>(b + o_t);
  e = cudaMemsetAsync(n->pslab, 0, off, n->stream);
  if (e == cudaSuccess) {
    k_srgb_table<<<1, 256, 0, n->stream>>>(n->srgb);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(n->stream);
  if (e != cudaSuccess) {
    cudaFree(n->pslab);
    delete n;
    return GMMSP_E_CUDA;
  }
  *out = n;
  return GMMSP_OK;
}

gmmsp_status gmmsp_net_set_weights(gmmsp_net n, const float* host, long long count) {
  if (!n) return GMMSP_E_INVALID;
  if (!host || count != n->pl.total) return nfail(n, GMMSP_E_INVALID, "weight count mismatch");
  for (long long i = 0; i < count; ++i)
    if (!isfinite(host[i])) return nfail(n, GMMSP_E_INVALID, "non-finite weight");
  const size_t bytes = size_t(count) * 4;
  GN_CHECK(n, cudaMemcpyAsync(n->w32, host, bytes, cudaMemcpyHostToDevice, n->stream));
  GN_CHECK(n, cudaMemsetAsync(n->m, 0, bytes, n->stream));
  GN_CHECK(n, cudaMemsetAsync(n->vv, 0, bytes, n->stream));
  k_to_bf16<<<grid_for(count, 256), 256, 0, n->stream>>>(n->w32, bf_params(n), int(count));
  GN_CHECK(n, cudaGetLastError());
  GN_CHECK(n, cudaStreamSynchronize(n->stream));
  n->adam_t = 0;
  return GMMSP_OK;
}

gmmsp_status gmmsp_net_get_weights(gmmsp_net n, float* host, long long count) {
  if (!n) return GMMSP_E_INVALID;
  if (!host || count != n->pl.total) return nfail(n, GMMSP_E_INVALID, "weight count mismatch");
  GN_CHECK(n, cudaMemcpyAsync(host, n->w32, size_t(count) * 4, cudaMemcpyDeviceToHost, n->stream));
  GN_CHECK(n, cudaStreamSynchronize(n->stream));
  return GMMSP_OK;
}

gmmsp_status gmmsp_net_get_adam(gmmsp_net n, float* m_host, float* v_host, long long count, long long* step) {
  if (!n) return GMMSP_E_INVALID;
  if (!m_host || !v_host || !step || count != n->pl.total) return nfail(n, GMMSP_E_INVALID, "bad arguments");
  GN_CHECK(n, cudaMemcpyAsync(m_host, n->m, size_t(count) * 4, cudaMemcpyDeviceToHost, n->stream));
  GN_CHECK(n, cudaMemcpyAsync(v_host, n->vv, size_t(count) * 4, cudaMemcpyDeviceToHost, n->stream));
  GN_CHECK(n, cudaStreamSynchronize(n->stream));
  *step = n->adam_t;
  return GMMSP_OK;
}

gmmsp_status gmmsp_net_set_adam(gmmsp_net n, const float* m_host, const float* v_host, long long count,
                                long long step) {
  if (!n) return GMMSP_E_INVALID;
  if (!m_host || !v_host || count != n->pl.total || step < 0) return nfail(n, GMMSP_E_INVALID, "bad arguments");
  for (long long i = 0; i < count; ++i)
    if (!isfinite(m_host[i]) || !(v_host[i] >= 0.f) || !isfinite(v_host[i]))
      return nfail(n, GMMSP_E_INVALID, "non-finite or negative optimiser state");
  GN_CHECK(n, cudaMemcpyAsync(n->m, m_host, size_t(count) * 4, cudaMemcpyHostToDevice, n->stream));
  GN_CHECK(n, cudaMemcpyAsync(n->vv, v_host, size_t(count) * 4, cudaMemcpyHostToDevice, n->stream));
  GN_CHECK(n, cudaStreamSynchronize(n->stream));
  n->adam_t = step;
  return GMMSP_OK;
}

gmmsp_status gmmsp_net_forward(gmmsp_net n, const float* lab_dev, int B, int W, int H, float* out_dev) {
  GMMSP_NVTX("gmmsp_net_forward");
  if (!n) return GMMSP_E_INVALID;
  Geom g;
  if (!lab_dev || !out_dev || B < 1 || !net_geom(n, W, H, &g)) return nfail(n, GMMSP_E_INVALID, "bad arguments");
  if (!cells_fit(n, (long long)B * g.K)) return nfail(n, GMMSP_E_INVALID, "batch too large");
  const gmmsp_status st = reserve(n, (long long)B * g.K, false);
  if (st != GMMSP_OK) return st;
  return enqueue_forward(n, lab_dev, B, g, out_dev, false, n->stream);
}

gmmsp_status gmmsp_net_grad(gmmsp_net n, const float* lab_dev, int B, int W, int H, const float* target_dev,
                            float* grad_host, double* loss_host) {
  GMMSP_NVTX("gmmsp_net_grad");
  if (!n) return GMMSP_E_INVALID;
  Geom g;
  if (!lab_dev || !target_dev || B < 1 || !net_geom(n, W, H, &g))
    return nfail(n, GMMSP_E_INVALID, "bad arguments");
  const long long cells = (long long)B * g.K;
  if (!cells_fit(n, cells)) return nfail(n, GMMSP_E_INVALID, "batch too large");
  gmmsp_status st = reserve(n, cells, true);
  if (st != GMMSP_OK) return st;
  st = enqueue_grad(n, lab_dev, B, g, target_dev, n->stream);
  if (st != GMMSP_OK) return st;
  return grad_host || loss_host ? grad_to_host(n, cells, grad_host, loss_host) : GMMSP_OK;
}

gmmsp_status gmmsp_net_adam(gmmsp_net n, float lr, float beta1, float beta2, float eps) {
  if (!n) return GMMSP_E_INVALID;
  if (!(lr >= 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) || !(eps > 0.f))
    return nfail(n, GMMSP_E_INVALID, "bad Adam hyper-parameters");
  ++n->adam_t;
  const float c1 = float(1.0 / (1.0 - pow(double(beta1), double(n->adam_t))));
  const float c2 = float(1.0 / (1.0 - pow(double(beta2), double(n->adam_t))));
  const int np = n->pl.total;
  k_adam<<<grid_for(np, 256), 256, 0, n->stream>>>(n->w32, n->m, n->vv, n->grad, bf_params(n), np, lr, beta1, beta2,
                                                   eps, c1, c2);
  GN_CHECK(n, cudaGetLastError());
  return GMMSP_OK;
}

gmmsp_status gmmsp_net_train_step(gmmsp_net n, const float* lab_dev, int B, int W, int H,
                                  const float* target_dev, float lr, double* loss_host) {
  GMMSP_NVTX("gmmsp_net_train_step");
  gmmsp_status st = gmmsp_net_grad(n, lab_dev, B, W, H, target_dev, nullptr, nullptr);
  if (st != GMMSP_OK) return st;
  st = gmmsp_net_adam(n, lr, 0.9f, 0.999f, 1e-8f);
  if (st != GMMSP_OK || !loss_host) return st;
  Geom g;
  net_geom(n, W, H, &g);
  return grad_to_host(n, (long long)B * g.K, nullptr, loss_host);
}

gmmsp_status gmmsp_net_get_activation(gmmsp_net n, int layer, float* host, long long count) {
  if (!n) return GMMSP_E_INVALID;
  if (layer < 0 || layer > 3 || !host || count != n->last_cells * kC || n->last_cells == 0)
    return nfail(n, GMMSP_E_INVALID, "bad activation request");
  std::vector<uint16_t> tmp(static_cast<size_t>(count));
  GN_CHECK(n, cudaMemcpyAsync(tmp.data(), n->c[layer], size_t(count) * 2, cudaMemcpyDeviceToHost, n->stream));
  const gmmsp_status st = check_err(n);
  if (st != GMMSP_OK) return st;
  for (long long i = 0; i < count; ++i) {  // a bfloat16 is the top half of a float32
    const uint32_t u = uint32_t(tmp[size_t(i)]) << 16;
    memcpy(host + i, &u, 4);
  }
  return GMMSP_OK;
}

gmmsp_status gmmsp_net_check(gmmsp_net n) {
  if (!n) return GMMSP_E_INVALID;
  return check_err(n);
}

gmmsp_status gmmsp_tc_wait_selftest(int max_tries, void* stream) {
  if (max_tries < 1 || max_tries > (1 << 20)) return GMMSP_E_INVALID;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int* flag = nullptr;
  if (cudaMalloc(&flag, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return GMMSP_E_NOMEM;
  }
  int host = 0;
  cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int), s);
  if (e == cudaSuccess) {
    k_wait_selftest<<<1, 128, 0, s>>>(uint32_t(max_tries), flag);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&host, flag, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(flag);
  if (e != cudaSuccess) return GMMSP_E_CUDA;
  return host ? GMMSP_E_TIMEOUT : GMMSP_OK;
}

const char* gmmsp_net_last_error(gmmsp_net n) { return n ? n->msg.c_str() : "null network"; }

void gmmsp_net_destroy(gmmsp_net n) {
  if (!n) return;
  cudaStreamSynchronize(n->stream);
  if (n->wslab) cudaFree(n->wslab);
  if (n->pslab) cudaFree(n->pslab);
  delete n;
}

}  // extern "C"
