// Connectivity post-processing (Algorithm 1, step 8; Sec. III-D), declared in
// include/gmmsp_conn.h.  The paper sorts the isolated superpixels by size
// and merges, one after the other, those smaller than a quarter of the
// desired size into the neighbouring superpixel nearest in colour, adding
// the source's size to the destination's.  Readings (the same as the
// oracle's): an isolated superpixel is a 4-connected component of one label;
// small means 4 K |c| < N; order (size, smallest pixel index); a group keeps
// the colour of the component that founded it (mean of its fixed-point
// colour sum); nearest = smallest squared CIELAB distance, ties to the
// smaller index; pixels take the label of their group's founder.
//
// Parallel form with the same result.  A large component is never a source,
// so its group and colour never change; two small components therefore only
// influence each other through a chain of adjacent small components.  The
// small components split into clusters (connected sets of the small-small
// adjacency), and the sequential rule restricted to one cluster, in the
// cluster's own (size, index) order, gives exactly what the sequential pass
// over the whole image gives there.  One thread (or one warp) runs each
// cluster.
//
// Data layout.  After the pixel-level labelling every component gets a
// compact index c in the order of its smallest pixel (so ordering by c is
// ordering by that pixel), and every per-component array is indexed by c:
// about 1.6 M entries for 256 images of 481x321, a few MB each, which the
// L2 keeps while the merge reads them at random.
//
// Kernels (all images of a call at once; pixel kernels take blockIdx.y as the
// image, tile loops cover all pixels of the call):
//   k_cc_tile                       labelling of 32 x 32 tiles, parent = the
//                                   tile's root; the list of the tile's roots
//   k_cc_border                     unions across the tiles' borders
//   k_tile_roots / k_root_count / k_root_scan / k_root_assign  the tiles'
//                                   roots point at their component's, a bit per
//                                   component, counts and a scan, compact index
//                                   per tile root
//   k_comp_map                      parent := compact index; sizes and
//                                   fixed-point colour sums (atomics)
//   k_comp_flags                    small flag, mean colour, group state per component
//   k_scan_* (twice)                offsets of the adjacency lists and of the clusters
//   k_edges                         small-small clusters and adjacency lists
//   k_cluster_count / _fill         member lists as (size << 32 | c) keys
//   k_cluster_merge                 one thread per cluster of <= kThreadCluster
//                                   members, one warp per larger cluster (adjacency
//                                   over the lanes)
//   k_group_label / k_relabel       label of the group founder
// One allocation (kept by a context between calls) and one synchronisation
// per call.  Every loop over a parent chain or a retry is bounded; running
// out sets the error word (reported as GMMSP_E_TIMEOUT).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <memory>
#include <new>

#include "../../include/gmmsp.h"
#include "../../include/gmmsp_conn.h"
#include "gmmsp_internal.cuh"

namespace gmmsp {
namespace conn {

constexpr int kMaxHops = 1 << 24;      // bound on any parent-chain walk or union retry
constexpr int kFixedShift = 20;        // colour sums in units of 2^-20
constexpr int kMaxCluster = 1 << 16;   // bound on the members of a cluster
constexpr int kThreadCluster = 2;      // clusters up to this size: one thread; larger: one warp
constexpr int kHugeCluster = 32;       // warp clusters above this size are started first
constexpr int kScanTile = 4096;        // elements per block of the tile kernels (1024 threads x 4)
constexpr int kMergeWarps = 4;
constexpr int kCcTile = 32;            // side of the tiles labelled in shared memory
constexpr int kCcWarps = 4;            // tiles per block
constexpr int kCcAhead = 8;            // rows of labels in flight
constexpr int kChunk = 128;            // pixels a warp walks down at once: four per lane
constexpr int kMapRows = 16, kEdgeRows = 8;  // ... by k_comp_map and k_edges at most; fewer where the call has few pixels
constexpr long long kOneBlockScan = 1 << 18;  // pixels up to which one block scans (64 steps at most)

// One image of a call: pixels [off, off + W H) of the call's arrays.
struct Img {
  int W, H, K;
  long long off;
  const float* lab;   // three FP32 planes of W H values
  int32_t* labels;    // the caller's labels (read, then rewritten by k_relabel)
};

struct Scratch {
  // per pixel of the call
  int* parent;                // union-find, then the compact index
  int* cidr;                  // at the tiles' root pixels: the compact index; then (k_cluster_fill) ...
  int* big;                   // ... in the same memory, roots of clusters above kThreadCluster members: those
                              // above kHugeCluster from the front, the others from the back
  // per component (compact index c < ncomp)
  int* size;                  // pixel count; in the merge, of a small founder's group
  long long* csum;            // 3 fixed-point colour sums, then (k_comp_flags) ...
  double* mean;               // ... the 3 mean colours csum / size, in the same memory
  float4* mean32;             // the means in FP32 and the largest of their magnitudes
  int* cimg;                  // image
  int32_t* clabel;            // its label
  int* cpar;                  // cluster union-find over small components, -1 for the others
  int* deg;                   // entries of its adjacency list
  unsigned* aoff;             // (ncomp + 1) offsets of the lists, each with room for the component's perimeter
  int* adj;                   // adjacency lists (compact indices of neighbouring components)
  int* cl_count;              // members of the cluster it roots, counted down as they are filled in; in the
                              // merge, the order of a large cluster's members
  unsigned* cl_off;           // (ncomp + 1) member offsets
  unsigned long long* cl_key; // members as (size << 32 | c), grouped by cluster
  int* gpar;                  // merge union-find (group founder)
  int* next;                  // the members of a group as a ring (small founders' groups)
  int* tile_sum;              // tile kernels: per tile counts, then their exclusive prefix
  // the tiles' roots (before the per-component arrays that lie in the same memory)
  int* roots;                 // a tile's root pixels, from its place on (tile_place)
  int* nroots;                // at a tile's place: their number
  unsigned* bits;             // a bit per pixel: the root of a component
  unsigned* before;           // per 32 pixels: components of the same kScanTile pixels before them
  unsigned long long* cnt;    // counters: 0 small, 1 merged, 2 components
  int* ncomp;                 // the component count as int (read by later kernels)
  int* nbig;                  // [0] entries at the front of `big`, [1] at the back
  int* err;
};

__device__ __forceinline__ int find_root(const int* p, int x, int* err) {
  for (int h = 0; h < kMaxHops; ++h) {
    const int q = p[x];
    if (q == x) return x;
    x = q;
  }
  atomicExch(err, 1);
  return x;
}

// Root of x with path halving, for the union phases: every visited node is
// re-pointed at its grandparent, an ancestor in the same set, so no set
// changes; a concurrent link that such a store overwrites is redone by that
// link's own retry.
__device__ __forceinline__ int find_halve(int* p, int x, int* err) {
  for (int h = 0; h < kMaxHops; ++h) {
    const int q = p[x];
    if (q == x) return x;
    const int r = p[q];
    if (r == q) return q;
    p[x] = r;
    x = r;
  }
  atomicExch(err, 1);
  return x;
}

// Root of x in the merge union-find, with path compression.  Only the
// thread or warp that owns a cluster calls it, on that cluster's members and
// on large components (their own roots), so the compression writes touch no
// other cluster's nodes; lanes of one warp that compress the same node write
// the same root.
__device__ __forceinline__ int find_group(int* p, int x, int* err) {
  const int r = find_root(p, x, err);
  for (int h = 0; h < kMaxHops && p[x] != r; ++h) {
    const int q = p[x];
    p[x] = r;
    x = q;
  }
  return r;
}

// Lock-free union by the smaller index (atomicMin on the larger root): the
// final root of every set is its smallest member.
__device__ __forceinline__ void unite(int* p, int a, int b, int* err) {
  for (int h = 0; h < kMaxHops; ++h) {
    a = find_halve(p, a, err);
    b = find_halve(p, b, err);
    if (a == b) return;
    if (a < b) {
      const int old = atomicMin(p + b, a);
      if (old == b) return;
      b = old;
    } else {
      const int old = atomicMin(p + a, b);
      if (old == a) return;
      a = old;
    }
  }
  atomicExch(err, 1);
}

// A union or a path halving may be at work on the entry: its sign stays.
__device__ __forceinline__ bool is_small(const Scratch& S, int c) { return S.cpar[c] >= 0; }

__device__ __forceinline__ bool small_size(long long s, int K, long long N) { return 4LL * K * s < N; }

// Loops over the roots q of image im's tiles, a warp per tile (fewer than 2^30
// tiles: 32-bit divisions).
#define FOR_TILE_ROOTS(q)                                                                                      \
  const unsigned tx_ = unsigned(im.W + kCcTile - 1) / kCcTile;                                                 \
  const unsigned tiles_ = tx_ * ((unsigned(im.H) + unsigned(tile_rows) - 1u) / unsigned(tile_rows));           \
  for (unsigned t_ = blockIdx.x * kCcWarps + (threadIdx.x >> 5); t_ < tiles_; t_ += gridDim.x * kCcWarps)      \
    for (int y_ = int(t_ / tx_),                                                                               \
             at_ = int(tile_place(im, int(t_ - unsigned(y_) * tx_) * kCcTile, y_ * tile_rows,                  \
                                  min(tile_rows, im.H - y_ * tile_rows))),                                     \
             i_ = int(threadIdx.x & 31), n_ = S.nroots[at_];                                                   \
         i_ < n_; i_ += 32)                                                                                    \
      if (const int q = S.roots[at_ + i_]; true)

// Per-component loops over c < *S.ncomp.
#define FOR_COMPONENTS(c)      \
  const int ncomp_ = *S.ncomp; \
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncomp_; c += gridDim.x * blockDim.x)

// Where a tile's list starts: the pixels of the tiles before it, tile row after
// tile row (a tile has no more roots than pixels).
__device__ __forceinline__ long long tile_place(const Img& im, int x0, int y0, int rows) {
  return im.off + (long long)y0 * im.W + (long long)x0 * rows;
}

// Labels one tile of 32 x 32 pixels (x tile_rows where the call has few pixels:
// a tile is a serial walk) per warp.  A row's runs of one label come from a
// ballot; a run takes the number of the leftmost run above that it touches,
// carried down in registers, or a fresh one, and only where it touches a run
// above of another number are the two queued for a union in shared memory, 32
// unions at a time.  Numbers are given in the order of the pixels, so a tile's
// root is the smallest pixel of its piece of the component.  Then parent = the
// root's pixel.  (One union per pair of touching runs, nearly all of them
// between runs of one piece already: 150 instructions per row of 32 pixels,
// 308 us on 256 images of 481x321, 170 this way.)  Only the tiles' borders are left to
// global unions: 6 % of the pixels (labelling all of them in global memory
// took 195 + 703 us).
__global__ void __launch_bounds__(kCcWarps * 32) k_cc_tile(const Img* __restrict__ imgs, Scratch S, int nwords,
                                                          int tile_rows) {
  __shared__ int parent[kCcWarps][kCcTile * kCcTile];            // over the numbers given
  __shared__ uint16_t first[kCcWarps][kCcTile * kCcTile];        // a number's first pixel
  __shared__ uint16_t number[kCcWarps][kCcTile * kCcTile];       // of every pixel
  __shared__ unsigned queue[kCcWarps][64];                       // unions to do: two numbers each
  const Img im = imgs[blockIdx.y];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int *p = S.parent, *err = S.err;
  for (int i = int((blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x); i < nwords;
       i += int(gridDim.x * gridDim.y * blockDim.x))
    S.bits[i] = 0u;
  const int tx = (im.W + kCcTile - 1) / kCcTile;
  const long long tiles = (long long)tx * ((im.H + tile_rows - 1) / tile_rows);
  const unsigned below = (1u << lane) - 1u, upto = 0xffffffffu >> (31 - lane);
  int* q = parent[warp];
  uint16_t *F = first[warp], *R = number[warp];
  unsigned* Q = queue[warp];
  for (long long t = (long long)blockIdx.x * kCcWarps + warp; t < tiles; t += (long long)gridDim.x * kCcWarps) {
    const int ty = int(t / tx), x0 = int(t - (long long)ty * tx) * kCcTile, y0 = ty * tile_rows;
    const int rows = min(tile_rows, im.H - y0);
    const bool in = x0 + lane < im.W;
    const long long g0 = (long long)y0 * im.W + x0;
    const int32_t* L = im.labels + g0 + lane;
    int32_t next[kCcAhead], up = 0;  // the labels of the next rows, loaded ahead; of the row above
#pragma unroll
    for (int j = 0; j < kCcAhead; ++j) next[j] = in && j < rows ? L[(long long)j * im.W] : 0;
    int given = 0, queued = 0, nup = 0;  // numbers given, unions queued (below 32 between rows), the number above
    auto work = [&](int at_least) {
      __syncwarp();
      while (queued >= at_least && queued > 0) {
        const int k = min(32, queued);
        queued -= k;
        if (lane < k) unite(q, int(Q[queued + lane] & 0xffffu), int(Q[queued + lane] >> 16), err);
        __syncwarp();
      }
    };
    for (int r0 = 0; r0 < rows; r0 += kCcAhead) {
#pragma unroll
      for (int j = 0; j < kCcAhead; ++j) {
        const int r = r0 + j;
        if (r >= rows) continue;
        const int32_t l = next[j];
        if (in && r + kCcAhead < rows) next[j] = L[(long long)(r + kCcAhead) * im.W];
        const int32_t lprev = __shfl_up_sync(0xffffffffu, l, 1), uprev = __shfl_up_sync(0xffffffffu, up, 1);
        const bool head = !(in && lane > 0 && lprev == l), same = in && r > 0 && l == up;
        const unsigned heads = __ballot_sync(0xffffffffu, head), sames = __ballot_sync(0xffffffffu, same);
        // this lane's run: lanes at .. the one before the next head
        const int at = 31 - __clz(heads & upto);
        const unsigned after = heads & ~upto;
        const unsigned run = (after ? (after & (0u - after)) - 1u : 0xffffffffu) & (0xffffffffu << at);
        const unsigned touch = sames & run;
        const bool fresh = head && in && !touch;
        const unsigned freshs = __ballot_sync(0xffffffffu, fresh);
        const int mine = fresh ? given + __popc(freshs & below) : nup;
        const int num = __shfl_sync(0xffffffffu, mine, touch ? __ffs(touch) - 1 : at);
        if (fresh) {
          q[num] = num;
          F[num] = uint16_t(r * 32 + lane);
        }
        given += __popc(freshs);
        R[r * 32 + lane] = uint16_t(num);
        const bool join = same && nup != num && !(!head && uprev == l);
        const unsigned joins = __ballot_sync(0xffffffffu, join);
        if (joins) {
          if (join) Q[queued + __popc(joins & below)] = unsigned(num) | unsigned(nup) << 16;
          queued += __popc(joins);
          work(32);
        }
        up = l;
        nup = num;
      }
    }
    work(1);
    // every number's root, as a pixel of the tile (F of a root stays); the roots go to the tile's list
    const int at0 = int(im.off + g0);
    const long long place = tile_place(im, x0, y0, rows);
    int listed = 0;
    for (int i = lane; i - lane < given; i += 32) {
      const int root = i < given ? find_root(q, i, err) : -1;
      const unsigned is_root = __ballot_sync(0xffffffffu, root == i);
      if (root == i) S.roots[place + listed + __popc(is_root & below)] = at0 + (F[i] >> 5) * im.W + (F[i] & 31);
      listed += __popc(is_root);
      if (root >= 0) {
        q[i] = root;
        F[i] = F[root];
      }
    }
    if (lane == 0) S.nroots[place] = listed;
    __syncwarp();
    int* P = p + im.off + g0 + lane;
    for (int r = 0; r < rows; ++r, P += im.W) {
      if (!in) continue;
      const int root = F[R[r * 32 + lane]];
      *P = at0 + (root >> 5) * im.W + (root & 31);  // pixel numbers of a call stay below 2^30
    }
    __syncwarp();  // the tile's arrays are refilled
  }
}

// The unions across the tiles' borders: pixels x = 32 k with their left
// neighbour, pixels y = tile_rows k with the one above.  A pair that the previous one
// along the border already joined (both pairs of one label, inside the same
// two tiles) is skipped.
__global__ void k_cc_border(const Img* __restrict__ imgs, int* p, int* err, int tile_rows) {
  const Img im = imgs[blockIdx.y];
  const int nx = (im.W - 1) / kCcTile, ny = (im.H - 1) / tile_rows;
  const long long vertical = (long long)nx * im.H, total = vertical + (long long)ny * im.W;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    int x, y;
    long long other, back;  // offsets of the pixel across the border, of the previous pixel along it
    bool first;             // of its tile's side
    if (i < vertical) {
      const int k = int(i / im.H);
      y = int(i - (long long)k * im.H);
      x = (k + 1) * kCcTile;
      other = -1;
      back = -(long long)im.W;
      first = y % tile_rows == 0;
    } else {
      const long long j = i - vertical;
      const int k = int(j / im.W);
      x = int(j - (long long)k * im.W);
      y = (k + 1) * tile_rows;
      other = -(long long)im.W;
      back = -1;
      first = x % kCcTile == 0;
    }
    const long long g = (long long)y * im.W + x;
    const int32_t l = im.labels[g];
    if (im.labels[g + other] != l) continue;
    if (!first && im.labels[g + back] == l && im.labels[g + back + other] == l) continue;
    unite(p, int(im.off + g), int(im.off + g + other), err);
  }
}

// Exclusive scan of one value per thread over the block; total = the block sum.
__device__ __forceinline__ unsigned block_exclusive_scan(unsigned v, unsigned* warp_sums, unsigned& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    unsigned w = lane < int(blockDim.x >> 5) ? warp_sums[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    warp_sums[lane] = w;  // inclusive prefix of the warp totals
  }
  __syncthreads();
  total = warp_sums[(blockDim.x >> 5) - 1];
  const unsigned before = warp ? warp_sums[warp - 1] : 0u;
  __syncthreads();  // warp_sums is reused by the next call
  return before + x - v;
}

// Image of pixel g of the call (binary search over the images' offsets).
__device__ __forceinline__ int image_of(const Img* __restrict__ imgs, int n, long long g) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (imgs[mid].off <= g) lo = mid; else hi = mid;
  }
  return lo;
}

// After the unions only the tiles' roots are looked at again (a few per cent
// of the pixels; every pixel points at one): each points at its component's
// root, and the components' roots set their bits.  The walks only read, so the
// one store per root cannot be overwritten by another thread's walk (a halving
// store here could leave a non-root behind).  The compact indices of the
// components are in the order of their roots (smallest pixels): bits set
// before, counted and scanned; no counter that every block updates.  (Over all
// pixels, which a second pass read again for the indices: 96 + 116 us on 256
// images of 481x321.)
__global__ void __launch_bounds__(kCcWarps * 32) k_tile_roots(const Img* __restrict__ imgs, Scratch S, int tile_rows) {
  const Img im = imgs[blockIdx.y];
  FOR_TILE_ROOTS(q) {
    const int r = find_root(S.parent, q, S.err);
    S.parent[q] = r;
    if (r == q) atomicOr(S.bits + (q >> 5), 1u << (q & 31));
  }
}

// Components of tile `tile` of kScanTile pixels (the warp's result), and of
// those the ones before each 32 pixels: four words per lane.
__device__ __forceinline__ int count_roots(const Scratch& S, int tile, int nwords, int lane) {
  const int w0 = tile * (kScanTile / 32) + 4 * lane;
  int n[4], sum = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    n[j] = w0 + j < nwords ? __popc(S.bits[w0 + j]) : 0;
    sum += n[j];
  }
  int x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  const int total = __shfl_sync(0xffffffffu, x, 31);
  x -= sum;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (w0 + j < nwords) S.before[w0 + j] = unsigned(x);
    x += n[j];
  }
  return total;
}

__global__ void __launch_bounds__(256) k_root_count(int ntiles, int nwords, Scratch S) {
  const int tile = int(blockIdx.x * 8 + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
  if (tile >= ntiles) return;
  const int n = count_roots(S, tile, nwords, lane);
  if (lane == 0) S.tile_sum[tile] = n;
}

// Exclusive scan of the ntiles tile counts in place (one block); the total
// is the component count.  COUNT: the block counts them first (few tiles).
template <bool COUNT>
__global__ void __launch_bounds__(1024) k_root_scan(int ntiles, int nwords, Scratch S) {
  __shared__ unsigned warp_sums[32];
  if (COUNT) {
    for (int tile = int(threadIdx.x >> 5); tile < ntiles; tile += 32) {
      const int n = count_roots(S, tile, nwords, int(threadIdx.x & 31));
      if ((threadIdx.x & 31) == 0) S.tile_sum[tile] = n;
    }
    __syncthreads();
  }
  int carry = 0;
  for (int c = 0; c < ntiles; c += 1024) {
    const int i = c + threadIdx.x;
    const int v = i < ntiles ? S.tile_sum[i] : 0;
    unsigned total;
    const unsigned ex = block_exclusive_scan(unsigned(v), warp_sums, total);
    if (i < ntiles) S.tile_sum[i] = carry + int(ex);
    carry += int(total);
  }
  if (threadIdx.x == 0) {
    *S.ncomp = carry;
    S.cnt[2] = (unsigned long long)carry;
  }
}

// The compact index at every tile's root; the start of every component, what is
// zero in the order of the components (tile after tile, each 32-byte sector
// of these arrays is written in several pieces: 106 us on 256 images of 481x321).
__global__ void __launch_bounds__(kCcWarps * 32) k_root_assign(const Img* __restrict__ imgs, Scratch S, int tile_rows) {
  const Img im = imgs[blockIdx.y];
  const int ncomp = *S.ncomp, step = int(gridDim.x * gridDim.y * blockDim.x);
  for (int c = int((blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x); c < ncomp; c += step) {
    S.size[c] = 0;
    S.deg[c] = 0;
    S.cl_count[c] = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) S.csum[c + (long long)k * ncomp] = 0;
  }
  FOR_TILE_ROOTS(q) {
    const int r = S.parent[q];
    const int c = S.tile_sum[r / kScanTile] + int(S.before[r >> 5]) + __popc(S.bits[r >> 5] & ((1u << (r & 31)) - 1u));
    S.cidr[q] = c;
    if (r != q) continue;
    S.cimg[c] = int(blockIdx.y);
    S.clabel[c] = im.labels[q - im.off];
  }
}

// parent := compact index of the pixel's component; component sizes and
// fixed-point colour sums.  A warp walks a chunk of 128 pixels down 16 rows,
// four pixels per lane; a lane adds its pixels of one component in registers,
// going back and forth along its four pixels, and updates the component's sums
// when it changes: about one set of atomics per eight pixels.  (A warp-wide
// segmented reduction of 64-bit values per row run took 373 us on 256 images
// of 481x321.)
__global__ void __launch_bounds__(128) k_comp_map(const Img* __restrict__ imgs, Scratch S, int chunk_rows) {
  const Img im = imgs[blockIdx.y];
  const long long N = (long long)im.W * im.H;
  const int lane = threadIdx.x & 31;
  const int cx = (im.W + kChunk - 1) / kChunk;
  const long long chunks = (long long)cx * ((im.H + chunk_rows - 1) / chunk_rows);
  for (long long t = (long long)blockIdx.x * 4 + (threadIdx.x >> 5); t < chunks; t += (long long)gridDim.x * 4) {
    const int cy = int(t / cx), x = int(t - (long long)cy * cx) * kChunk + 4 * lane, y0 = cy * chunk_rows;
    const int n = min(4, im.W - x), rows = min(chunk_rows, im.H - y0);
    if (n <= 0) continue;
    int c = -1, cnt = 0;
    long long s0 = 0, s1 = 0, s2 = 0;
    auto flush = [&] {
      if (!cnt) return;
      atomicAdd(S.size + c, cnt);
      unsigned long long* o = reinterpret_cast<unsigned long long*>(S.csum + 3LL * c);
      atomicAdd(o, (unsigned long long)s0);
      atomicAdd(o + 1, (unsigned long long)s1);
      atomicAdd(o + 2, (unsigned long long)s2);
    };
    int* P = S.parent + im.off + (long long)y0 * im.W + x;
    const float* Z = im.lab + (long long)y0 * im.W + x;
    int qn[4] = {};
    float zn[3][4] = {};  // the next row's
    auto ahead = [&](const int* p, const float* z) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j < n) {
          qn[j] = p[j];
#pragma unroll
          for (int k = 0; k < 3; ++k) zn[k][j] = __ldg(z + k * N + j);
        }
    };
    ahead(P, Z);
    for (int r = 0; r < rows; ++r, P += im.W, Z += im.W) {
      int cq[4];
      float z[3][4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        cq[j] = j < n ? S.cidr[qn[j]] : 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) z[k][j] = zn[k][j];
      }
      if (r + 1 < rows) ahead(P + im.W, Z + im.W);
      auto add = [&](int j) {
        if (j >= n) return;
        if (cq[j] != c) {
          flush();
          c = cq[j];
          cnt = 0;
          s0 = s1 = s2 = 0;
        }
        P[j] = c;
        ++cnt;
        // z 2^20 is exact in FP32 (a power-of-two scaling): round(2^20 z)
        s0 += __float2ll_rn(z[0][j] * float(1 << kFixedShift));
        s1 += __float2ll_rn(z[1][j] * float(1 << kFixedShift));
        s2 += __float2ll_rn(z[2][j] * float(1 << kFixedShift));
      };
      if (r & 1) {
        add(3); add(2); add(1); add(0);
      } else {
        add(0); add(1); add(2); add(3);
      }
    }
    flush();
  }
}

// Small flag, mean colour (the FP64 quotient csum / size, written over the
// sums) and the initial group state of every component (each is its own
// group); the small count takes one atomic per block.
__global__ void __launch_bounds__(256) k_comp_flags(const Img* __restrict__ imgs, Scratch S) {
  const int ncomp = *S.ncomp;
  for (int base = blockIdx.x * blockDim.x; base < ncomp; base += gridDim.x * blockDim.x) {
    const int c = base + threadIdx.x;
    bool sm = false;
    if (c < ncomp) {
      const Img im = imgs[S.cimg[c]];
      const int sz = S.size[c];
      sm = small_size(sz, im.K, (long long)im.W * im.H);
      double m[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) S.mean[3LL * c + k] = m[k] = double(S.csum[3LL * c + k]) / double(sz);
      const float x = float(m[0]), y = float(m[1]), z = float(m[2]);
      S.mean32[c] = make_float4(x, y, z, fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z))));
      S.gpar[c] = c;
      S.cpar[c] = sm ? c : -1;
      S.next[c] = c;
    }
    const int nsm = __syncthreads_count(sm);
    if (threadIdx.x == 0 && nsm) atomicAdd(S.cnt + 0, (unsigned long long)nsm);
  }
}

// One edge between different components i and j: small ones that touch join a
// cluster, and each small side's list gets the other.  A list has room for its
// component's whole perimeter (2 size + 2 edges at most for a 4-connected set
// of pixels), so it is filled in the pass that finds the edges.
__device__ __forceinline__ void add_neighbour(const Scratch& S, int i, int j) {
  const unsigned at = S.aoff[i] + unsigned(atomicAdd(S.deg + i, 1));  // < 4 T < 2^32
  if (at < S.aoff[i + 1]) S.adj[at] = j;
  else atomicExch(S.err, 1);
}
__device__ __forceinline__ void add_edge(const Scratch& S, int i, int j) {
  const bool si = is_small(S, i), sj = is_small(S, j);
  if (si) add_neighbour(S, i, j);
  if (sj) add_neighbour(S, j, i);
  if (si && sj) unite(S.cpar, i, j, S.err);
}

// Walks the 4-neighbour edges between different components (the edge to the
// right and the edge below of every pixel).  An edge whose pair of components
// the previous edge along the same line already gave (the row above for the
// edge to the right, the pixel to the left for the edge below) is skipped: the
// lists are neighbour sets, and most repeats go.  A warp walks a chunk of 128
// pixels down 8 rows, four pixels per lane with the rows above and below in
// registers, so an index is loaded once; the edges found go through a queue in
// shared memory and are worked on 32 at a time, so that their chains of random
// accesses overlap (worked on where they were found: 684 us on 256 images of
// 481x321; one pixel per thread, in a counting and a filling pass: 2 x 390).
__global__ void __launch_bounds__(128, 8) k_edges(const Img* __restrict__ imgs, Scratch S, int chunk_rows) {
  const Img im = imgs[blockIdx.y];
  const int lane = threadIdx.x & 31;
  __shared__ int2 queue[4][32 + 8 * 32];
  int2* Q = queue[threadIdx.x >> 5];
  int queued = 0;  // below 32 between rows; a row adds at most 8 per lane
  auto push = [&](bool has, int i, int j) {
    const unsigned m = __ballot_sync(0xffffffffu, has);
    if (has) Q[queued + __popc(m & ((1u << lane) - 1u))] = make_int2(i, j);
    queued += __popc(m);
  };
  auto work = [&](int at_least) {
    __syncwarp();
    while (queued >= at_least && queued > 0) {
      const int k = min(32, queued);
      queued -= k;
      if (lane < k) {
        const int2 e = Q[queued + lane];
        add_edge(S, e.x, e.y);
      }
      __syncwarp();
    }
  };
  const int cx = (im.W + kChunk - 1) / kChunk;
  const long long chunks = (long long)cx * ((im.H + chunk_rows - 1) / chunk_rows);
  for (long long t = (long long)blockIdx.x * 4 + (threadIdx.x >> 5); t < chunks; t += (long long)gridDim.x * 4) {
    const int cy = int(t / cx), x = int(t - (long long)cy * cx) * kChunk + 4 * lane, y0 = cy * chunk_rows;
    const int n = max(0, min(4, im.W - x)), rows = min(chunk_rows, im.H - y0);
    const bool left = x > 0 && x < im.W, right = x + 4 < im.W;  // pixel x - 1, x + 4 exists
    // the pixel beside the warp's first / last lane
    const int beside = lane == 0 ? -1 : 4;
    const bool e_in = (lane == 0 && left) || (lane == 31 && right);
    const int* P = S.parent + im.off + (long long)y0 * im.W + x;
    int up[4], v[4], dn[4], ue = -1, e = -1, de = -1;
    auto row = [&](const int* q, bool ok, int (&d)[4], int& de_) {
#pragma unroll
      for (int j = 0; j < 4; ++j) d[j] = ok && j < n ? q[j] : -1;
      de_ = ok && e_in ? q[beside] : -1;
    };
    row(P - im.W, y0 > 0, up, ue);
    row(P, true, v, e);
    for (int r = 0; r < rows; ++r, P += im.W) {
      row(P + im.W, y0 + r + 1 < im.H, dn, de);
      // neighbours across the lanes: left of pixel 0 (this row, the row below), right of pixel 3 (this row, above)
      const int lv = __shfl_up_sync(0xffffffffu, v[3], 1), ld = __shfl_up_sync(0xffffffffu, dn[3], 1);
      const int rv = __shfl_down_sync(0xffffffffu, v[0], 1), ru = __shfl_down_sync(0xffffffffu, up[0], 1);
      const int l_v = lane == 0 ? e : lv, l_d = lane == 0 ? de : ld, r_v = lane == 31 ? e : rv, r_u = lane == 31 ? ue : ru;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int ci = v[j];
        const bool has_r = j < n && (j < 3 ? j + 1 < n : right);
        const int cr = j < 3 ? v[j < 3 ? j + 1 : 3] : r_v, cru = j < 3 ? up[j < 3 ? j + 1 : 3] : r_u;
        push(has_r && cr != ci && !(up[j] == ci && cru == cr), ci, cr);
        const int cd = dn[j];
        const bool has_l = j > 0 || left;
        const int cl = j > 0 ? v[j > 0 ? j - 1 : 0] : l_v, cld = j > 0 ? dn[j > 0 ? j - 1 : 0] : l_d;
        push(j < n && cd >= 0 && cd != ci && !(has_l && cl == ci && cld == cd), ci, cd);
      }
      work(32);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        up[j] = v[j];
        v[j] = dn[j];
      }
      ue = e;
      e = de;
    }
  }
  work(1);
}

// What the scans add up: the room of a component's adjacency list (the
// perimeter of a small component, at most 2 size + 2 edges), or the members of
// the cluster it roots.
enum ScanOf : int { kScanLists = 0, kScanClusters = 1 };
template <int OF>
__device__ __forceinline__ unsigned scan_value(const Scratch& S, int c) {
  if (OF == kScanClusters) return unsigned(S.cl_count[c]);
  return is_small(S, c) ? 2u * unsigned(S.size[c]) + 2u : 0u;
}

// Exclusive prefix sum over the n = *S.ncomp components into out[0..n] (out[n]
// = the total), in three kernels: tile scans (kScanTile elements per block), a
// scan of the tile sums (one block), the tile offsets added.  The grids cover
// the largest possible n; blocks past n return at once.  Few pixels: one block
// does it alone (k_scan_one).
template <int OF>
__global__ void __launch_bounds__(1024) k_scan_tiles(Scratch S, unsigned* __restrict__ out) {
  __shared__ unsigned warp_sums[32];
  const int n = *S.ncomp;
  const long long base = (long long)blockIdx.x * kScanTile;
  if (base >= n) return;
  const long long i0 = base + 4LL * threadIdx.x;
  unsigned v[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = (i0 + j < n) ? scan_value<OF>(S, int(i0 + j)) : 0u;
  const unsigned t = v[0] + v[1] + v[2] + v[3];
  unsigned total;
  unsigned run = block_exclusive_scan(t, warp_sums, total);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (i0 + j < n) out[i0 + j] = run;
    run += v[j];
  }
  if (threadIdx.x == 0) S.tile_sum[blockIdx.x] = int(total);
}

template <int OF>
__global__ void __launch_bounds__(1024) k_scan_one(Scratch S, unsigned* __restrict__ out) {
  __shared__ unsigned warp_sums[32];
  const int n = *S.ncomp;
  unsigned carry = 0;
  for (int base = 0; base < n; base += kScanTile) {
    const int i0 = base + 4 * threadIdx.x;
    unsigned v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = (i0 + j < n) ? scan_value<OF>(S, i0 + j) : 0u;
    const unsigned t = v[0] + v[1] + v[2] + v[3];
    unsigned total;
    unsigned run = carry + block_exclusive_scan(t, warp_sums, total);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (i0 + j < n) out[i0 + j] = run;
      run += v[j];
    }
    carry += total;
  }
  if (threadIdx.x == 0) out[n] = carry;
}

__global__ void __launch_bounds__(1024) k_scan_tile_sums(Scratch S, unsigned* __restrict__ out) {
  __shared__ unsigned warp_sums[32];
  const int n = *S.ncomp;
  const int ntiles = (n + kScanTile - 1) / kScanTile;
  unsigned carry = 0;
  for (int c = 0; c < ntiles; c += 1024) {
    const int i = c + threadIdx.x;
    const unsigned v = i < ntiles ? unsigned(S.tile_sum[i]) : 0u;
    unsigned total;
    const unsigned ex = block_exclusive_scan(v, warp_sums, total);
    if (i < ntiles) S.tile_sum[i] = int(carry + ex);
    carry += total;
  }
  if (threadIdx.x == 0) out[n] = carry;
}

__global__ void __launch_bounds__(1024) k_scan_add(Scratch S, unsigned* __restrict__ out) {
  const int n = *S.ncomp;
  const long long base = (long long)blockIdx.x * kScanTile;
  if (base >= n || blockIdx.x == 0) return;
  const unsigned add = unsigned(S.tile_sum[blockIdx.x]);
  const long long i0 = base + 4LL * threadIdx.x;
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (i0 + j < n) out[i0 + j] += add;
}

// Cluster root of every small component, member counts per cluster root.
__global__ void k_cluster_count(Scratch S) {
  FOR_COMPONENTS(c) {
    if (!is_small(S, c)) continue;
    atomicAdd(S.cl_count + find_root(S.cpar, c, S.err), 1);
  }
}

// Members of each cluster as sort keys (size << 32 | c): contiguous per
// cluster, so that the sort reads and writes no scattered data.  The clusters
// for a warp (above kThreadCluster members) go to its list.
__global__ void __launch_bounds__(256) k_cluster_fill(Scratch S) {
  const int ncomp = *S.ncomp;
  __shared__ int n_of[2], at_of[2];  // huge and other clusters of this step: their number, their place in the list
  for (int base = blockIdx.x * 256; base < ncomp; base += gridDim.x * 256) {
    const int c = base + threadIdx.x;
    if (threadIdx.x < 2) n_of[threadIdx.x] = 0;
    __syncthreads();
    int kind = -1, at = 0;
    if (c < ncomp && is_small(S, c)) {
      const int r = find_root(S.cpar, c, S.err);
      const unsigned off = S.cl_off[r];
      if (r == c) {
        const int n = int(S.cl_off[c + 1] - off);
        kind = n > kHugeCluster ? 0 : (n > kThreadCluster ? 1 : -1);
        if (kind >= 0) at = atomicAdd(&n_of[kind], 1);
      }
      S.cl_key[off + unsigned(atomicSub(S.cl_count + r, 1) - 1)] = ((unsigned long long)(unsigned)S.size[c] << 32) | unsigned(c);
    }
    __syncthreads();
    if (threadIdx.x < 2 && n_of[threadIdx.x]) at_of[threadIdx.x] = atomicAdd(S.nbig + threadIdx.x, n_of[threadIdx.x]);
    __syncthreads();
    if (kind == 0) S.big[at_of[0] + at] = c;
    if (kind == 1) S.big[ncomp - 1 - (at_of[1] + at)] = c;
  }
}

// Squared distance of the mean colours of components a and b, in a fixed
// order without contractions.
__device__ __forceinline__ double dist2_of(double a0, double a1, double a2, double b0, double b1, double b2) {
  const double t0 = __dsub_rn(a0, b0), t1 = __dsub_rn(a1, b1), t2 = __dsub_rn(a2, b2);
  return __dadd_rn(__dadd_rn(__dmul_rn(t0, t0), __dmul_rn(t1, t1)), __dmul_rn(t2, t2));
}
__device__ __forceinline__ double dist2(const double* mean, int a, int b) {
  return dist2_of(mean[3LL * a], mean[3LL * a + 1], mean[3LL * a + 2], mean[3LL * b], mean[3LL * b + 1],
                  mean[3LL * b + 2]);
}

// The same distance in FP32, and how far it may be from the FP64 one: with the
// means within 2^-24 M of theirs (M the largest magnitude), each difference is
// off by at most 2^-22 M, its square by 2^-20 M^2, and the rounding of the
// squares and sums (of at most 12 M^2) adds less than 2.3 2^-20 M^2: below
// 5.5 2^-20 M^2 in all, taken as 2^-17 M^2.  FP64 runs at 1/64 of the FP32
// rate here, so a nearest group is found in FP32 and FP64 decides only between
// those that the bound cannot tell apart.
__device__ __forceinline__ float dist2_32(float4 a, float4 b, float& off) {
  const float t0 = a.x - b.x, t1 = a.y - b.y, t2 = a.z - b.z, m = fmaxf(a.w, b.w);
  off = m * m * 0x1p-17f;
  return t0 * t0 + t1 * t1 + t2 * t2;
}

// Merge of small component r (still its group's founder, still small) into
// the nearest group `best` next to its group.  A small destination belongs
// to the same cluster and gets r's size and members; a large destination is
// never a source, and no decision reads its size.
__device__ __forceinline__ void merge_into(Scratch& S, int r, int best) {
  S.gpar[r] = best;
  if (is_small(S, best)) {
    S.size[best] += S.size[r];
    const int n = S.next[best];  // two rings become one
    S.next[best] = S.next[r];
    S.next[r] = n;
  }
  S.size[r] = 0;
}

// Insertion sort of n keys (one thread).
__device__ __forceinline__ void sort_keys(unsigned long long* key, int n) {
  for (int a = 1; a < n; ++a) {
    const unsigned long long v = key[a];
    int b = a - 1;
    while (b >= 0 && key[b] > v) {
      key[b + 1] = key[b];
      --b;
    }
    key[b + 1] = v;
  }
}

// One thread per cluster of at most kThreadCluster members: the sequential
// rule over the members in (size, index) order.
__device__ __forceinline__ unsigned merge_small_clusters(const Img* __restrict__ imgs, Scratch& S, int first, int step) {
  unsigned merged = 0;
  const int ncomp = *S.ncomp;
  for (int c = first; c < ncomp; c += step) {
    if (S.cpar[c] != c) continue;  // not a cluster root
    const int n = int(S.cl_off[c + 1] - S.cl_off[c]);
    if (n > kThreadCluster) continue;
    const Img im = imgs[S.cimg[c]];
    const long long N = (long long)im.W * im.H;
    unsigned long long* key = S.cl_key + S.cl_off[c];
    sort_keys(key, n);
    for (int a = 0; a < n; ++a) {
      const int r = int(unsigned(key[a]));
      if (S.gpar[r] != r || !small_size(S.size[r], im.K, N)) continue;
      const float4 mr = S.mean32[r];
      int best = -1;
      float low = 0.f, high = INFINITY;  // the nearest one's distance lies in [low, high]
      bool close = false;                // another group may be as near
      int hops = 0;
      for (int m = r; (m != r || hops == 0) && hops < kMaxHops; m = S.next[m], ++hops) {
        const unsigned q0 = S.aoff[m], q1 = q0 + unsigned(S.deg[m]);
        for (unsigned q = q0; q < q1; ++q) {
          const int g = find_group(S.gpar, S.adj[q], S.err);
          if (g == r || g == best) continue;
          float off;
          const float d = dist2_32(mr, S.mean32[g], off);
          if (best < 0 || d + off < low) {  // certainly nearer
            best = g;
            low = d - off;
            high = d + off;
            close = false;
          } else if (d - off <= high) {     // not certainly farther
            close = true;
            low = fminf(low, d - off);
            high = fminf(high, d + off);
          }
        }
      }
      if (hops >= kMaxHops) atomicExch(S.err, 1);
      if (best < 0) continue;
      if (close) {
        best = -1;
        double bd = 0.0;
        for (int m = r, h = 0; (m != r || h == 0) && h < kMaxHops; m = S.next[m], ++h) {
          const unsigned q0 = S.aoff[m], q1 = q0 + unsigned(S.deg[m]);
          for (unsigned q = q0; q < q1; ++q) {
            const int g = find_group(S.gpar, S.adj[q], S.err);
            if (g == r) continue;
            float off;
            if (dist2_32(mr, S.mean32[g], off) - off > high) continue;  // certainly not the nearest
            const double d = dist2(S.mean, r, g);
            if (best < 0 || d < bd || (d == bd && g < best)) {
              best = g;
              bd = d;
            }
          }
        }
      }
      merge_into(S, r, best);
      ++merged;
    }
  }
  return merged;
}

// The nearest group over the lanes: the smallest distance (doubles >= 0 order
// like their bits), then the smallest group index; 0x7fffffff where no lane
// has one.
__device__ __forceinline__ int warp_nearest(double bd, int best) {
  const unsigned hi = unsigned(__double2hiint(bd)), lo = unsigned(__double2loint(bd));
  const unsigned mh = __reduce_min_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_min_sync(0xffffffffu, hi == mh ? lo : ~0u);
  return __reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? best : 0x7fffffff);
}

// A member's data that no merge changes, fetched ahead of its turn: its list's
// place, its first 32 neighbours (one per lane), and the mean colours.
struct Member {
  int r = -1;
  unsigned q0 = 0, deg = 0;
  int adj = -1;
  float4 mr, ma;
  __device__ __forceinline__ void list(const Scratch& S, int r_) {
    r = r_;
    q0 = S.aoff[r];
    deg = unsigned(S.deg[r]);
  }
  __device__ __forceinline__ void neighbours(const Scratch& S, int lane) { adj = unsigned(lane) < deg ? S.adj[q0 + lane] : -1; }
  __device__ __forceinline__ void means(const Scratch& S) {
    mr = S.mean32[r];
    ma = adj >= 0 ? S.mean32[adj] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
};

// One warp per cluster above kThreadCluster members.  The members are ordered
// by counting the smaller keys of each (keys are distinct), up to 32 through
// the lanes, more through memory; then they are taken in order as above, with
// the adjacency entries of each member's group spread over the lanes.  The
// chain over the members of the largest cluster sets the time, so what no
// merge changes is fetched one to three members ahead.  __syncwarp orders lane
// 0's merge writes before the next member's reads.
__device__ __forceinline__ unsigned merge_cluster(const Img* __restrict__ imgs, Scratch& S, int c, int* order,
                                                  int lane) {
  unsigned merged = 0;
  const Img im = imgs[S.cimg[c]];
  const long long N = (long long)im.W * im.H;
  const unsigned long long* key = S.cl_key + S.cl_off[c];
  const int n = int(S.cl_off[c + 1] - S.cl_off[c]);
  if (n > kMaxCluster) {
    if (lane == 0) atomicExch(S.err, 1);
    return 0;
  }
  if (n <= 32) {
    const unsigned long long k = lane < n ? key[lane] : ~0ull;
    int rank = 0;
    for (int j = 0; j < n; ++j) rank += __shfl_sync(0xffffffffu, k, j) < k;
    if (lane < n) order[rank] = int(unsigned(k));
  } else {
    order = S.cl_count + S.cl_off[c];  // the counts are done with
    for (int i = lane; i < n; i += 32) {
      const unsigned long long k = key[i];
      int rank = 0;
#pragma unroll 4
      for (int j = 0; j < n; ++j) rank += __ldg(key + j) < k;
      order[rank] = int(unsigned(k));
    }
  }
  __syncwarp();
  const auto member = [&](int a) { return order[a]; };
  Member m0, m1, m2;  // this member, the next, the one after
  m0.list(S, member(0));
  m0.neighbours(S, lane);
  m0.means(S);
  if (n > 1) {
    m1.list(S, member(1));
    m1.neighbours(S, lane);
  }
  if (n > 2) m2.list(S, member(2));
  for (int a = 0; a < n; ++a) {
    const Member me = m0;
    if (a + 1 < n) {
      m0 = m1;
      m0.means(S);
    }
    if (a + 2 < n) {
      m1 = m2;
      m1.neighbours(S, lane);
    }
    if (a + 3 < n) m2.list(S, member(a + 3));
    const int r = me.r;
    if (S.gpar[r] != r || !small_size(S.size[r], im.K, N)) continue;  // warp-uniform
    // this lane's neighbour groups: one that is nearest in FP32, and whether
    // another may be as near
    int best = 0x7fffffff;
    float low = INFINITY, high = INFINITY;
    bool close = false;
    auto consider = [&](int g, float4 mg) {
      if (g == r || g == best) return;
      float off;
      const float d = dist2_32(me.mr, mg, off);
      if (best == 0x7fffffff || d + off < low) {
        best = g;
        low = d - off;
        high = d + off;
        close = false;
      } else if (d - off <= high) {
        close = true;
        low = fminf(low, d - off);
        high = fminf(high, d + off);
      }
    };
    if (me.adj >= 0) {
      const int g = find_group(S.gpar, me.adj, S.err);
      consider(g, g == me.adj ? me.ma : S.mean32[g]);
    }
    int hops = 0;
    for (int m = r; (m != r || hops == 0) && hops < kMaxHops; m = S.next[m], ++hops) {
      const unsigned q0 = m == r ? me.q0 : S.aoff[m], q1 = q0 + (m == r ? me.deg : unsigned(S.deg[m]));
      for (unsigned q = q0 + lane + (m == r ? 32u : 0u); q < q1; q += 32) {
        const int g = find_group(S.gpar, S.adj[q], S.err);
        consider(g, S.mean32[g]);
      }
    }
    if (hops >= kMaxHops && lane == 0) atomicExch(S.err, 1);
    // the smallest upper bound over the lanes: what lies above it is out
    const unsigned hb = __reduce_min_sync(0xffffffffu, high >= 0.f ? __float_as_uint(high) : 0u);
    const float hmin = __uint_as_float(hb);
    const bool in = best != 0x7fffffff && low <= hmin;
    const unsigned lanes = __ballot_sync(0xffffffffu, in);
    if (lanes == 0u) continue;  // no neighbour
    const int first = __shfl_sync(0xffffffffu, best, __ffs(lanes) - 1);
    if (__any_sync(0xffffffffu, in && (close || best != first))) {  // FP64 decides
      best = 0x7fffffff;
      double bd = INFINITY;
      for (int m = r, h = 0; (m != r || h == 0) && h < kMaxHops; m = S.next[m], ++h) {
        const unsigned q0 = S.aoff[m], q1 = q0 + unsigned(S.deg[m]);
        for (unsigned q = q0 + lane; q < q1; q += 32) {
          const int g = find_group(S.gpar, S.adj[q], S.err);
          if (g == r) continue;
          float off;
          if (dist2_32(me.mr, S.mean32[g], off) - off > hmin) continue;
          const double d = dist2(S.mean, r, g);
          if (d < bd || (d == bd && g < best)) {
            best = g;
            bd = d;
          }
        }
      }
      best = warp_nearest(bd, best);
    } else {
      best = first;
    }
    if (best != 0x7fffffff && lane == 0) {
      merge_into(S, r, best);
      ++merged;
    }
    __syncwarp();
  }
  __syncwarp();  // `order` is refilled by the next cluster
  return merged;
}

// All clusters in one launch: the first `warp_blocks` blocks take the list of
// the larger ones, a warp each, those above kHugeCluster members first (the
// longest serial chains start earliest); the other blocks take the clusters of
// one or two members, a thread each, beside them.
__global__ void __launch_bounds__(kMergeWarps * 32, 8) k_cluster_merge(const Img* __restrict__ imgs, Scratch S,
                                                                      int warp_blocks) {
  __shared__ int order[kMergeWarps][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned merged = 0;
  if (int(blockIdx.x) < warp_blocks) {
    const int nhuge = S.nbig[0], nbig = S.nbig[0] + S.nbig[1], ncomp = *S.ncomp;
    for (int b = blockIdx.x * kMergeWarps + warp; b < nbig; b += warp_blocks * kMergeWarps)
      merged += merge_cluster(imgs, S, b < nhuge ? S.big[b] : S.big[ncomp - 1 - (b - nhuge)], order[warp], lane);
  } else {
    const int blocks = int(gridDim.x) - warp_blocks;
    merged = merge_small_clusters(imgs, S, (int(blockIdx.x) - warp_blocks) * int(blockDim.x) + int(threadIdx.x),
                                  blocks * int(blockDim.x));
  }
  merged = __reduce_add_sync(0xffffffffu, merged);
  if (lane == 0 && merged) atomicAdd(S.cnt + 1, (unsigned long long)merged);
}

// The label of every merged component's group founder, in the place of its own
// (a component that is its own group keeps its label).
__global__ void k_group_label(Scratch S) {
  FOR_COMPONENTS(c) {
    const int g = S.gpar[c];
    if (g != c) S.next[c] = S.clabel[find_root(S.gpar, g, S.err)];  // the member lists are done with
  }
}

// Pixels of merged components only: the others have their label already.  A
// thread takes four consecutive pixels of the call.
__global__ void __launch_bounds__(256) k_relabel(const Img* __restrict__ imgs, int n, long long T, Scratch S) {
  __shared__ int first_image;
  const long long base = 4LL * blockIdx.x * 256, g0 = base + 4 * threadIdx.x;
  if (threadIdx.x == 0) first_image = image_of(imgs, n, base);
  __syncthreads();
  int c[4];
  if (g0 + 3 < T) {
    const int4 q = *reinterpret_cast<const int4*>(S.parent + g0);
    c[0] = q.x;
    c[1] = q.y;
    c[2] = q.z;
    c[3] = q.w;
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) c[j] = g0 + j < T ? S.parent[g0 + j] : -1;
  }
  int gp[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) gp[j] = c[j] >= 0 ? __ldg(S.gpar + c[j]) : -1;
  int i = first_image;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (gp[j] == c[j]) continue;
    const long long g = g0 + j;
    while (i + 1 < n && imgs[i + 1].off <= g) ++i;
    imgs[i].labels[g - imgs[i].off] = S.next[c[j]];
  }
}

}  // namespace conn

gmmsp_status enforce_connectivity_many(int n, const int* W, const int* H, const int* K, int32_t* const* labels,
                                       const float* const* lab, gmmsp_conn_stats* stats, cudaStream_t s,
                                       ConnScratch* cache) {
  GMMSP_NVTX("enforce_connectivity_many");
  using namespace conn;
  if (n < 1 || n > 65535) return GMMSP_E_INVALID;
  // the image table and, behind it, the counters (zeros): uploaded in one copy
  const size_t up_bytes = ((sizeof(Img) * n + 255) & ~size_t(255)) + 256;
  const std::unique_ptr<char[]> up_host(new (std::nothrow) char[up_bytes]());
  if (!up_host) return GMMSP_E_NOMEM;
  Img* host = reinterpret_cast<Img*>(up_host.get());
  long long T = 0, maxN = 0;
  for (int i = 0; i < n; ++i) {
    if (W[i] < 1 || H[i] < 1 || K[i] < 1 || !labels[i] || !lab[i]) return GMMSP_E_INVALID;
    host[i] = Img{W[i], H[i], K[i], T, lab[i], labels[i]};
    T += (long long)W[i] * H[i];
    maxN = std::max(maxN, (long long)W[i] * H[i]);
  }
  if (T >= (1LL << 30)) return GMMSP_E_INVALID;
  auto up = [](size_t x) { return (x + 255) & ~size_t(255); };
  // every per-component array has room for T components (one per pixel at most): 112 bytes per pixel in all
  const size_t nI = up(size_t(T) * 4), nI1 = up(size_t(T + 1) * 4);
  const long long ntiles = std::max<long long>(1, (T + kScanTile - 1) / kScanTile);
  enum { A_PARENT, A_CIDR, A_SIZE, A_CIMG, A_CLABEL, A_CPAR, A_DEG, A_CLCOUNT, A_GPAR, A_NEXT, kIntArrays };
  enum { O_AOFF = kIntArrays, O_CLOFF, O_ADJ, O_CSUM, O_MEAN32, O_TABLE, O_CNT, O_KEY, O_TILE, kRegions };
  size_t o[kRegions];
  size_t off = 0;
  for (int j = 0; j < kIntArrays; ++j) { o[j] = off; off += nI; }
  o[O_AOFF] = off; off += nI1;
  o[O_CLOFF] = off; off += nI1;
  o[O_ADJ] = off; off += up(size_t(T) * 16);   // 2 size + 2 <= 4 size entries per small component
  o[O_CSUM] = off; off += up(size_t(T) * 24);
  o[O_MEAN32] = off; off += up(size_t(T) * 16);
  o[O_TABLE] = off; off += up(sizeof(Img) * n);
  o[O_CNT] = off; off += 256;                  // behind the table: uploaded (as zeros) with it
  o[O_KEY] = off; off += up(size_t(T) * 8);
  o[O_TILE] = off; off += up(size_t(ntiles + 1) * 4);
  void* slab = nullptr;
  cudaError_t e = cudaSuccess;
  CallScratch scratch;  // without a context's cache
  if (!cache) {
    e = scratch.alloc(off, s);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? GMMSP_E_NOMEM : GMMSP_E_CUDA;
    slab = scratch.ptr;
  } else if (cache->bytes >= off) {
    slab = cache->ptr;
  } else {
    if (cache->ptr) {
      cudaStreamSynchronize(s);
      cudaFree(cache->ptr);
      cache->ptr = nullptr;
      cache->bytes = 0;
    }
    e = cudaMalloc(&slab, off);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return e == cudaErrorMemoryAllocation ? GMMSP_E_NOMEM : GMMSP_E_CUDA;
    }
    cache->ptr = slab;
    cache->bytes = off;
  }
  char* b = static_cast<char*>(slab);
  auto ia = [&](int j) { return reinterpret_cast<int*>(b + o[j]); };
  Scratch S{};
  S.parent = ia(A_PARENT); S.cidr = ia(A_CIDR); S.size = ia(A_SIZE); S.cimg = ia(A_CIMG);
  S.clabel = reinterpret_cast<int32_t*>(ia(A_CLABEL)); S.cpar = ia(A_CPAR);
  S.deg = ia(A_DEG); S.cl_count = ia(A_CLCOUNT); S.gpar = ia(A_GPAR); S.next = ia(A_NEXT);
  S.big = S.cidr;
  S.aoff = reinterpret_cast<unsigned*>(ia(O_AOFF));
  S.cl_off = reinterpret_cast<unsigned*>(ia(O_CLOFF));
  S.adj = ia(O_ADJ);
  S.csum = reinterpret_cast<long long*>(b + o[O_CSUM]);
  S.mean = reinterpret_cast<double*>(b + o[O_CSUM]);
  S.mean32 = reinterpret_cast<float4*>(b + o[O_MEAN32]);
  Img* table = reinterpret_cast<Img*>(b + o[O_TABLE]);
  S.cnt = reinterpret_cast<unsigned long long*>(b + o[O_CNT]);
  S.ncomp = reinterpret_cast<int*>(b + o[O_CNT] + 64);
  S.err = reinterpret_cast<int*>(b + o[O_CNT] + 128);
  S.nbig = reinterpret_cast<int*>(b + o[O_CNT] + 192);
  S.cl_key = reinterpret_cast<unsigned long long*>(b + o[O_KEY]);
  S.tile_sum = ia(O_TILE);
  // before the adjacency lists, the cluster keys and the member lists are written
  const int nwords = int((T + 31) / 32);
  S.roots = S.adj;
  S.bits = reinterpret_cast<unsigned*>(S.cl_key);
  S.before = S.aoff;
  S.nroots = S.next;
  // blocks per image: enough to fill the machine across the images
  const long long per = std::max<long long>(1, std::min<long long>((maxN + 255) / 256, (152LL * 16 + n - 1) / n));
  const dim3 gp{static_cast<unsigned>(per), static_cast<unsigned>(n)};
  const int gs = 152 * 8;
  const unsigned nt = unsigned(ntiles);
  const bool one = T <= kOneBlockScan;
  // chunks and tiles of an image, four per block, at least enough blocks to fill the machine across the images
  const auto blocks_of = [&](int w, int h) {
    long long most = 1;
    for (int i = 0; i < n; ++i)
      most = std::max(most, ((W[i] + w - 1LL) / w) * ((H[i] + h - 1LL) / h));
    return dim3(unsigned(std::max<long long>(1, std::min<long long>((most + 3) / 4, (152LL * 64 + n - 1) / n))), unsigned(n));
  };
  // rows a warp walks: fewer where the most would leave much of the machine idle (the walk over a chunk is serial).  On
  // 256 images of 481x321 (128-pixel chunks: 11264 warps at 32 rows, 2.3 waves) the sums take 283 / 276 / 291 us and
  // the edges 251 / 229 / 215 us at 32 / 16 / 8 rows.
  long long chunk_cols = 0;
  for (int i = 0; i < n; ++i) chunk_cols += (W[i] + kChunk - 1LL) / kChunk * H[i];
  int rows = kCcTile;
  while (rows > 4 && chunk_cols / rows < 152LL * 32) rows /= 2;
  const int tile_rows = rows < kCcTile ? 8 : kCcTile, map_rows = std::min(rows, kMapRows), edge_rows = std::min(rows, kEdgeRows);
  const dim3 gt = blocks_of(kCcTile, tile_rows), gm = blocks_of(kChunk, map_rows), ge = blocks_of(kChunk, edge_rows);
  // merging: twice as many blocks as fit on the machine for either kind of cluster, so that an SM whose clusters are
  // done early takes more (half of the resident blocks for either kind: 549 us, 2.13 ms for the call on 256 images of
  // 481x321; this many 1.93 ms, and no less with 32 to 128 per SM)
  const int warp_blocks = int(std::max<long long>(1, std::min<long long>(152 * 16, (T + 1023) / 1024)));
  const int thread_blocks = warp_blocks;
  char back[256] = {};
  unsigned long long hc[3] = {};
  int herr = 0;
  do {
    if ((e = cudaMemcpyAsync(table, up_host.get(), up_bytes, cudaMemcpyHostToDevice, s)) != cudaSuccess) break;
    k_cc_tile<<<gt, kCcWarps * 32, 0, s>>>(table, S, nwords, tile_rows);
    k_cc_border<<<gp, 256, 0, s>>>(table, S.parent, S.err, tile_rows);
    k_tile_roots<<<gt, kCcWarps * 32, 0, s>>>(table, S, tile_rows);
    if (one) {
      k_root_scan<true><<<1, 1024, 0, s>>>(int(ntiles), nwords, S);
    } else {
      k_root_count<<<(nt + 7) / 8, 256, 0, s>>>(int(ntiles), nwords, S);
      k_root_scan<false><<<1, 1024, 0, s>>>(int(ntiles), nwords, S);
    }
    k_root_assign<<<gt, kCcWarps * 32, 0, s>>>(table, S, tile_rows);
    k_comp_map<<<gm, 128, 0, s>>>(table, S, map_rows);
    k_comp_flags<<<gs, 256, 0, s>>>(table, S);
    if (one) {
      k_scan_one<kScanLists><<<1, 1024, 0, s>>>(S, S.aoff);
    } else {
      k_scan_tiles<kScanLists><<<nt, 1024, 0, s>>>(S, S.aoff);
      k_scan_tile_sums<<<1, 1024, 0, s>>>(S, S.aoff);
      k_scan_add<<<nt, 1024, 0, s>>>(S, S.aoff);
    }
    k_edges<<<ge, 128, 0, s>>>(table, S, edge_rows);
    k_cluster_count<<<gs, 256, 0, s>>>(S);
    if (one) {
      k_scan_one<kScanClusters><<<1, 1024, 0, s>>>(S, S.cl_off);
    } else {
      k_scan_tiles<kScanClusters><<<nt, 1024, 0, s>>>(S, S.cl_off);
      k_scan_tile_sums<<<1, 1024, 0, s>>>(S, S.cl_off);
      k_scan_add<<<nt, 1024, 0, s>>>(S, S.cl_off);
    }
    k_cluster_fill<<<gs, 256, 0, s>>>(S);
    k_cluster_merge<<<warp_blocks + thread_blocks, kMergeWarps * 32, 0, s>>>(table, S, warp_blocks);
    k_group_label<<<gs, 256, 0, s>>>(S);
    k_relabel<<<unsigned((T + 1023) / 1024), 256, 0, s>>>(table, n, T, S);
    if ((e = cudaGetLastError()) != cudaSuccess) break;
    if ((e = cudaMemcpyAsync(back, S.cnt, sizeof(back), cudaMemcpyDeviceToHost, s)) != cudaSuccess) break;
    e = cudaStreamSynchronize(s);
    memcpy(hc, back, sizeof(hc));
    memcpy(&herr, back + 128, sizeof(herr));
  } while (false);
  if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? GMMSP_E_NOMEM : GMMSP_E_CUDA;
  if (herr) return GMMSP_E_TIMEOUT;
  if (stats) {
    stats->components = (long long)hc[2];
    stats->small = (long long)hc[0];
    stats->merged = (long long)hc[1];
  }
  return GMMSP_OK;
}

gmmsp_status enforce_connectivity(int32_t* labels_dev, const float* lab, int W, int H, int K,
                                  gmmsp_conn_stats* stats, cudaStream_t s, ConnScratch* cache) {
  int32_t* l[1] = {labels_dev};
  const float* c[1] = {lab};
  return enforce_connectivity_many(1, &W, &H, &K, l, c, stats, s, cache);
}

}  // namespace gmmsp

extern "C" gmmsp_status gmmsp_enforce_connectivity(int32_t* labels_dev, const float* lab_planes_dev, int W, int H,
                                                   int K, gmmsp_conn_stats* stats_host, void* stream) {
  if (!labels_dev || !lab_planes_dev || W < 1 || H < 1 || K < 1) return GMMSP_E_INVALID;
  return gmmsp::enforce_connectivity(labels_dev, lab_planes_dev, W, H, K, stats_host,
                                     static_cast<cudaStream_t>(stream), nullptr);
}
