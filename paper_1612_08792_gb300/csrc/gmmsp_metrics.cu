// Accuracy metrics of Sec. IV against a ground-truth segmentation
// (declared in include/gmmsp_metrics.h): boundary recall, the
// under-segmentation error of Eq. (ue) and the achievable segmentation
// accuracy of Eq. (asa).  Everything is integer counting, so the results are
// exact and independent of the order of the atomics:
//   k_tiles  one pass over both maps in tiles of 512 x 32 pixels: the overlap
//            table |s_k & s_g| (dense K x G), the boundary flags of both maps
//            as bit rows in shared memory, and from them the ground-truth
//            boundary pixels and those with a superpixel boundary pixel within
//            the Chebyshev radius
//   k_table  per superpixel |s_k|, max_g |s_k & s_g| and the Eq. (ue) terms,
//            one warp per superpixel, summed per block and added with 64-bit
//            atomics
// Every kernel takes a table of images (blockIdx.z, blockIdx.y), so a batch of
// images is two launches and one synchronisation.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "../../include/gmmsp.h"
#include "../../include/gmmsp_metrics.h"
#include "gmmsp_internal.cuh"

namespace gmmsp {
namespace metrics {

enum : int { C_BAD = 0, C_BR_REC = 1, C_BR_TOT = 2, C_UE = 3, C_ASA = 4, C_N = 5 };

// One image of a call and its scratch.
struct MImg {
  const int32_t* labels;     // W H superpixel labels in [0, K)
  const int32_t* gt;         // W H ground-truth ids in [0, G)
  int W, H, K, G;
  unsigned* table;           // K x G overlap counts
  unsigned long long* cnt;   // C_N counters
};

constexpr int kChunk = 128;                    // pixels a warp takes in a row: four per lane
constexpr int kTileChunks = 4, kTileRows = 32;  // a tile: 512 by 32 pixels, one warp per chunk
constexpr int kMaxRadius = 64;                 // within one chunk
constexpr int kBitRows = kTileRows + 2 * kMaxRadius, kBitCols = (kTileChunks + 2) * 4;

// One map walked down a chunk: the values of the rows above, at and below the
// current one for the lane's four pixels x .. x + 3, and of the pixel left of
// the warp's first lane or right of its last.  Rows outside the image are
// moved to the nearest row inside: a pixel never differs from itself.
struct Quad {
  const int32_t* p;  // pixel x in the row below
  int up[4], v[4], dn[4], e, de;
  // in: bit j set where pixel x + j exists, bit 4 the pixel beside (offset `beside`)
  __device__ __forceinline__ void start(const int32_t* m, long long r0, long long r1, long long r2, unsigned in,
                                        int beside) {
    p = m + r2;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      up[j] = v[j] = dn[j] = 0;
      if ((in >> j) & 1u) {
        up[j] = __ldg(m + r0 + j);
        v[j] = __ldg(m + r1 + j);
        dn[j] = __ldg(p + j);
      }
    }
    e = de = 0;
    if (in & 16u) {
      e = __ldg(m + r1 + beside);
      de = __ldg(p + beside);
    }
  }
  // bits[j]: the lanes whose pixel x + j differs from a 4-neighbour.  lft, rgt: pixel x - 1 (x + 4) exists.
  __device__ __forceinline__ void bits(unsigned in, bool lft, bool rgt, int lane, unsigned (&b)[4]) const {
    const int pl = __shfl_up_sync(0xffffffffu, v[3], 1), pr = __shfl_down_sync(0xffffffffu, v[0], 1);
    const bool d0 = lft && (lane == 0 ? e : pl) != v[0], d4 = rgt && (lane == 31 ? e : pr) != v[3];
    const bool d1 = (in & 2u) && v[0] != v[1], d2 = (in & 4u) && v[1] != v[2], d3 = (in & 8u) && v[2] != v[3];
    b[0] = __ballot_sync(0xffffffffu, (in & 1u) && (d0 || d1 || up[0] != v[0] || dn[0] != v[0]));
    b[1] = __ballot_sync(0xffffffffu, (in & 2u) && (d1 || d2 || up[1] != v[1] || dn[1] != v[1]));
    b[2] = __ballot_sync(0xffffffffu, (in & 4u) && (d2 || d3 || up[2] != v[2] || dn[2] != v[2]));
    b[3] = __ballot_sync(0xffffffffu, (in & 8u) && (d3 || d4 || up[3] != v[3] || dn[3] != v[3]));
  }
  // to the next row; step: from its row below to the one after
  __device__ __forceinline__ void next(int step, unsigned in, int beside) {
    p += step;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      up[j] = v[j];
      v[j] = dn[j];
      if ((in >> j) & 1u) dn[j] = __ldg(p + j);
    }
    e = de;
    if (in & 16u) de = __ldg(p + beside);
  }
};

// One tile of one image (blockIdx.z).  A warp takes a chunk of 128 pixels down
// the tile's rows, four pixels per lane, with the rows above and below in
// registers, so that a label is loaded once and compared without shared
// memory; the rows within the radius above and below the tile and the chunks
// beside it are done for the superpixel map only.  A lane counts its pixels of
// one (k, g) pair, going back and forth along its four pixels, and adds the
// count to the table when the pair changes: about one atomic per eight pixels.
// The boundary flags lie as bit planes: plane j of a chunk holds pixel 4 l + j
// at bit l.  The recall test is then bit arithmetic: the superpixel planes of
// 2 r + 1 rows or'ed, spread by r to either side.
//
// Bound by latency at 28 warps per SM (72 registers; 64 spill and are slower):
// issue 39 %, DRAM 19 %.  175 us at 256 images of 481x321, in place of a pass
// of per-pixel atomics, a pass writing one byte per pixel and a pass scanning
// those bytes around every ground-truth boundary pixel (370 + 231 + 304 us).
// One pixel per lane took twice the instructions and 227 us.
__global__ void __launch_bounds__(kTileChunks * 32, 7) k_tiles(const MImg* __restrict__ imgs, int radius,
                                                           int tile_row0) {
  const MImg im = imgs[blockIdx.z];
  const int x0 = blockIdx.x * kTileChunks * kChunk, y0 = (tile_row0 + int(blockIdx.y)) * kTileRows;
  if (x0 >= im.W || y0 >= im.H) return;  // whole blocks only
  __shared__ __align__(16) unsigned sb[kBitRows][kBitCols];
  __shared__ __align__(16) unsigned gb[kTileRows][kTileChunks * 4];
  __shared__ unsigned long long total[3];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x < 3) total[threadIdx.x] = 0;
  const int halo = radius > 0 ? 1 : 0, rows = min(kTileRows, im.H - y0);
  unsigned bad = 0;
  for (int w = warp; w < kTileChunks + 2 * halo; w += kTileChunks) {
    // sides up to 2^31 - 1: a chunk that would start past the last int wraps to a
    // negative column (outside), and no sum below goes past the image's sides
    const int xw = int(unsigned(x0) + unsigned(kChunk * (w - halo))), x = xw + 4 * lane;
    const bool inner = w >= halo && w < halo + kTileChunks;
    if (xw < 0 || xw >= im.W) {  // no pixel of the chunk lies in the image
      for (int i = lane; i < (rows + 2 * radius) * 4; i += 32) sb[i >> 2][4 * w + (i & 3)] = 0;
      if (inner)
        for (int i = lane; i < rows * 4; i += 32) gb[i >> 2][4 * (w - halo) + (i & 3)] = 0;
      continue;
    }
    const int beside = lane == 0 ? -1 : 4;
    const bool lft = x > 0 && x < im.W, rgt = im.W - x > 4;
    unsigned in = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) in |= x + j < im.W ? 1u << j : 0u;
    if ((lane == 0 && lft) || (lane == 31 && rgt)) in |= 16u;
    auto at = [&](int y) { return (long long)min(max(y, 0), im.H - 1) * im.W + x; };
    int y = y0 - radius;
    Quad L;
    L.start(im.labels, at(y - 1), at(y), at(y + 1), in, beside);
    auto step = [&] {  // no step where the row below stays the first or the last
      if (y < im.H) ++y;
      return y >= 0 && y < im.H - 1 ? im.W : 0;
    };
    unsigned b[4];
    // the rows of the radius above and below the tile: superpixel bits only
    auto border = [&](int i) {
      L.bits(in, lft, rgt, lane, b);
      if (lane < 4) sb[i][4 * w + lane] = y >= 0 && y < im.H ? (lane < 2 ? b[lane & 1] : b[2 + (lane & 1)]) : 0u;
      L.next(step(), in, beside);
    };
    for (int i = 0; i < radius; ++i) border(i);
    if (inner) {
      Quad G;
      G.start(im.gt, at(y - 1), at(y), at(y + 1), in, beside);
      unsigned pair = 0, run = 0, added = 0;
      auto count = [&](int j) {
        const bool ok = ((in >> j) & 1u) && unsigned(L.v[j]) < unsigned(im.K) && unsigned(G.v[j]) < unsigned(im.G);
        const unsigned p = unsigned(L.v[j]) * unsigned(im.G) + unsigned(G.v[j]);  // K G <= 2^31
        if (ok && p != pair) {
          if (run) atomicAdd(im.table + pair, run);
          added += run;
          pair = p;
          run = 0;
        }
        run += ok;
      };
#pragma unroll 2
      for (int t = 0; t < rows; ++t) {
        L.bits(in, lft, rgt, lane, b);
        if (lane == 0) *reinterpret_cast<uint4*>(&sb[radius + t][4 * w]) = make_uint4(b[0], b[1], b[2], b[3]);
        G.bits(in, lft, rgt, lane, b);
        if (lane == 0) *reinterpret_cast<uint4*>(&gb[t][4 * (w - halo)]) = make_uint4(b[0], b[1], b[2], b[3]);
        if (t & 1) {
          count(3); count(2); count(1); count(0);
        } else {
          count(0); count(1); count(2); count(3);
        }
        const int d = step();
        L.next(d, in, beside);
        G.next(d, in, beside);
      }
      if (run) atomicAdd(im.table + pair, run);
      bad += rows * __popc(in & 15u) - (added + run);
    } else {
      for (int t = 0; t < rows; ++t) border(radius + t);
    }
    for (int i = radius + rows; i < rows + 2 * radius; ++i) border(i);
  }
  __syncthreads();
  unsigned rec = 0, tot = 0;
  for (int i = threadIdx.x; i < rows * kTileChunks; i += kTileChunks * 32) {
    const int y = i / kTileChunks, c = i - y * kTileChunks;
    const uint4 g4 = *reinterpret_cast<const uint4*>(&gb[y][4 * c]);
    const unsigned g[4] = {g4.x, g4.y, g4.z, g4.w};
    if (!(g[0] | g[1] | g[2] | g[3])) continue;
    // the planes of this chunk and of its neighbours, the rows within the radius or'ed
    unsigned P[3][4] = {};
    for (int d = 0; d <= 2 * radius; ++d)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (k != 1 && halo == 0) continue;
        const uint4 q = *reinterpret_cast<const uint4*>(&sb[y + d][4 * (c + halo + k - 1)]);
        P[k][0] |= q.x;
        P[k][1] |= q.y;
        P[k][2] |= q.z;
        P[k][3] |= q.w;
      }
    // pixel 4 l + j sees pixel 4 (l + q) + t for |4 q + t - j| <= radius
    unsigned near[4] = {};
    const int qm = (radius + 3) / 4;
    for (int q = -qm; q <= qm; ++q)
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const unsigned s = q >= 0 ? __funnelshift_r(P[1][t], P[2][t], q) : __funnelshift_l(P[0][t], P[1][t], -q);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (abs(4 * q + t - j) <= radius) near[j] |= s;
      }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      tot += __popc(g[j]);
      rec += __popc(g[j] & near[j]);
    }
  }
  rec = __reduce_add_sync(0xffffffffu, rec);
  tot = __reduce_add_sync(0xffffffffu, tot);
  bad = __reduce_add_sync(0xffffffffu, bad);
  if (lane == 0) {
    if (rec) atomicAdd(&total[0], (unsigned long long)rec);
    if (tot) atomicAdd(&total[1], (unsigned long long)tot);
    if (bad) atomicAdd(&total[2], (unsigned long long)bad);
  }
  __syncthreads();
  if (threadIdx.x < 3 && total[threadIdx.x])
    atomicAdd(im.cnt + (threadIdx.x == 0 ? C_BR_REC : (threadIdx.x == 1 ? C_BR_TOT : C_BAD)), total[threadIdx.x]);
}

// One warp per superpixel, the row of the table read along the lanes (twice:
// the size, then the entries above eps times it).  An entry n exceeds
// lim = eps |s_k| (a double >= 0) exactly when n > floor(lim).  47 us for the
// 103 MB of 256 tables of 672 x 150 (one thread per row and an FP64 comparison
// per entry: 148 us).
__global__ void __launch_bounds__(256) k_table(const MImg* __restrict__ imgs, double eps) {
  const MImg im = imgs[blockIdx.y];
  __shared__ unsigned long long total[2];
  if (threadIdx.x < 2) total[threadIdx.x] = 0;
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long ue = 0, asa = 0;
  for (int k = blockIdx.x * 8 + warp; k < im.K; k += gridDim.x * 8) {
    const unsigned* row = im.table + (long long)k * im.G;
    unsigned long long size = 0;
    unsigned best = 0;
    for (int g = lane; g < im.G; g += 32) {
      const unsigned n = row[g];
      size += n;
      best = max(best, n);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) size += __shfl_xor_sync(0xffffffffu, size, o);
    best = __reduce_max_sync(0xffffffffu, best);
    if (size == 0) continue;
    const unsigned long long lim = (unsigned long long)floor(eps * double(size));  // eps < 1: below size
    unsigned above = 0;
    for (int g = lane; g < im.G; g += 32) above += row[g] > lim;
    above = __reduce_add_sync(0xffffffffu, above);
    asa += best;
    ue += above * size;
  }
  if (lane == 0) {
    if (ue) atomicAdd(&total[0], ue);
    if (asa) atomicAdd(&total[1], asa);
  }
  __syncthreads();
  if (threadIdx.x < 2 && total[threadIdx.x]) atomicAdd(im.cnt + (threadIdx.x == 0 ? C_UE : C_ASA), total[threadIdx.x]);
}

}  // namespace metrics
}  // namespace gmmsp

using namespace gmmsp::metrics;

extern "C" gmmsp_status gmmsp_segmentation_metrics_many(int n, const int32_t* const* labels_dev,
                                                        const int32_t* const* gt_dev, const int* W, const int* H,
                                                        const int* K, const int* G, int radius, double eps,
                                                        gmmsp_seg_metrics* out, void* stream) {
  GMMSP_NVTX("gmmsp_segmentation_metrics_many");
  if (n < 1 || n > 65535 || !labels_dev || !gt_dev || !W || !H || !K || !G || !out || radius < 0 || radius > 64 ||
      !(eps >= 0.0 && eps < 1.0))
    return GMMSP_E_INVALID;
  auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
  std::vector<MImg> host(n);
  std::vector<size_t> o_table(n);
  size_t off = up(sizeof(MImg) * n);                      // image table first
  const size_t o_cnt = off;
  off += up(sizeof(unsigned long long) * C_N * n);
  int maxW = 0, maxH = 0, maxK = 0;
  for (int i = 0; i < n; ++i) {
    if (!labels_dev[i] || !gt_dev[i] || W[i] < 1 || H[i] < 1 || K[i] < 1 || G[i] < 1) return GMMSP_E_INVALID;
    const long long cells = (long long)K[i] * G[i];
    if (cells > (1LL << 31)) return GMMSP_E_INVALID;
    o_table[i] = off;
    off += up(size_t(cells) * 4);
    maxW = std::max(maxW, W[i]);
    maxH = std::max(maxH, H[i]);
    maxK = std::max(maxK, K[i]);
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  gmmsp::CallScratch scratch;
  cudaError_t e = scratch.alloc(off, s);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? GMMSP_E_NOMEM : GMMSP_E_CUDA;
  char* b = static_cast<char*>(scratch.ptr);
  unsigned long long* cnt = reinterpret_cast<unsigned long long*>(b + o_cnt);
  for (int i = 0; i < n; ++i)
    host[i] = MImg{labels_dev[i], gt_dev[i], W[i], H[i], K[i], G[i], reinterpret_cast<unsigned*>(b + o_table[i]),
                   cnt + size_t(C_N) * i};
  MImg* table = reinterpret_cast<MImg*>(b);
  std::vector<unsigned long long> hc(size_t(C_N) * n, 0ull);
  const long long tx = (maxW + (kTileChunks * kChunk - 1LL)) / (kTileChunks * kChunk), ty = (maxH + (kTileRows - 1LL)) / kTileRows;
  const unsigned perk = unsigned(std::min<long long>((maxK + 7) / 8, std::max<long long>(1, (152LL * 32 + n - 1) / n)));
  do {
    if ((e = cudaMemcpyAsync(table, host.data(), sizeof(MImg) * n, cudaMemcpyHostToDevice, s)) != cudaSuccess) break;
    if ((e = cudaMemsetAsync(b + o_cnt, 0, off - o_cnt, s)) != cudaSuccess) break;  // counters and tables
    for (long long t0 = 0; t0 < ty; t0 += 65535) {  // grid.y holds at most 65535 rows of tiles
      k_tiles<<<dim3(unsigned(tx), unsigned(std::min<long long>(65535, ty - t0)), n), kTileChunks * 32, 0, s>>>(
          table, radius, int(t0));
    }
    k_table<<<dim3(perk, n), 256, 0, s>>>(table, eps);
    if ((e = cudaGetLastError()) != cudaSuccess) break;
    if ((e = cudaMemcpyAsync(hc.data(), cnt, sizeof(unsigned long long) * C_N * n, cudaMemcpyDeviceToHost, s)) !=
        cudaSuccess)
      break;
    e = cudaStreamSynchronize(s);
  } while (false);
  if (e != cudaSuccess) return GMMSP_E_CUDA;
  gmmsp_status st = GMMSP_OK;
  for (int i = 0; i < n; ++i) {
    const unsigned long long* h = hc.data() + size_t(C_N) * i;
    const double N = double((long long)W[i] * H[i]);
    gmmsp_seg_metrics& o = out[i];
    if (h[C_BAD]) st = GMMSP_E_INVALID;
    o.br_recovered = (long long)h[C_BR_REC];
    o.br_total = (long long)h[C_BR_TOT];
    o.ue_sum = (long long)h[C_UE];
    o.asa_sum = (long long)h[C_ASA];
    o.br = o.br_total ? double(o.br_recovered) / double(o.br_total) : 1.0;
    o.ue = double(o.ue_sum) / N - 1.0;
    o.asa = double(o.asa_sum) / N;
  }
  return st;
}

extern "C" gmmsp_status gmmsp_segmentation_metrics(const int32_t* labels_dev, const int32_t* gt_dev, int W, int H,
                                                   int K, int G, int radius, double eps,
                                                   gmmsp_seg_metrics* out, void* stream) {
  if (!labels_dev || !gt_dev || !out) return GMMSP_E_INVALID;
  return gmmsp_segmentation_metrics_many(1, &labels_dev, &gt_dev, &W, &H, &K, &G, radius, eps, out, stream);
}
