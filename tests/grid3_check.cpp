// Host check of the 3 x 3 layers' index arithmetic (gmmsp_grid3.cuh) against
// 64-bit divisions:
//  * small grids of every kind, few and many images (stacked or not): every
//    cell is the output of exactly one position of one tile, and every tile's
//    inputs are the right cells;
//  * every bordered row length at the most rows a network call accepts
//    (2^30 cells, image sides below 2^31 at a spacing of 3): tiles at the ends,
//    around the rows where the multiplication in place of the division starts
//    to fail, and at random;
//  * as many images of small grids as a call accepts;
//  * many images of any grid take few more tiles than their positions fill.
// Prints "ok <counts>" and exits 0, or prints the first mismatch and exits 1.
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <vector>

#include "gmmsp_grid3.cuh"

using namespace gmmsp::cnn;
typedef long long ll;

static uint64_t state = 0x9e3779b97f4a7c15ull;
static uint64_t next_u64() {  // splitmix64
  uint64_t z = (state += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

// Row of number q of strip `strip` of the stack that begins with image `first`,
// -1 off the cells.  `halo`: the neighbouring strips' columns count too.
static ll want_row(const Grid3& g, ll first, int strip, ll q, bool halo) {
  const ll Y = q >= 0 ? q / g.PW : -((-q + g.PW - 1) / g.PW), x = q - Y * g.PW;
  const ll col = (ll)strip * g.TW + x - 1;
  if (Y < 0 || col < 0 || col >= g.W || (!halo && (x < 1 || x > g.TW))) return -1;
  const ll i = g.per > 1 ? Y / (g.H + 1) : 0, y = Y - i * (g.H + 1);
  if (y >= g.H || i >= g.per || first + i >= g.B) return -1;
  return ((first + i) * g.H + y) * g.W + col;
}

static ll checked = 0;
static bool check_tile(const Grid3& g, ll tile, std::vector<int>* seen) {
  const Tile3 t = tile3_at(g, int(tile));
  const ll s = tile / g.tps, img = s / g.strips * g.per, q0 = (tile - s * g.tps) * 128;
  const int strip = int(s % g.strips);
  for (int p = 0; p < 128; ++p) {
    const ll r = row3(g, t, p), w = want_row(g, img, strip, q0 + p, false);
    if (r != w) {
      printf("output: B %d H %d W %d tile %lld position %d: row %lld, not %lld\n", g.B, g.H, g.W, tile, p, r, w);
      return false;
    }
    if (seen && r >= 0) ++(*seen)[size_t(r)];
  }
  // An input matters where a tap of an output reads it.
  std::vector<char> used(size_t(g.NP), 0);
  for (int p = 0; p < 128; ++p)
    if (want_row(g, img, strip, q0 + p, false) >= 0)
      for (int dy = -1; dy <= 1; ++dy)
        for (int dx = -1; dx <= 1; ++dx) used[size_t(p + g.PW + 1 + dy * g.PW + dx)] = 1;
  for (int p = 0; p < g.NP; ++p) {
    const ll r = in3(g, t, p);
    if (r < -1 || r >= (ll)g.B * g.H * g.W) {
      printf("input out of range: B %d H %d W %d tile %lld input %d: row %lld\n", g.B, g.H, g.W, tile, p, r);
      return false;
    }
    const ll w = want_row(g, img, strip, q0 + p - g.PW - 1, true);
    if (used[size_t(p)] && r != w) {
      printf("input: B %d H %d W %d tile %lld input %d: row %lld, not %lld\n", g.B, g.H, g.W, tile, p, r, w);
      return false;
    }
  }
  ++checked;
  return true;
}

static bool check_all(int B, int H, int W) {
  const Grid3 g = grid3_of(B, H, W);
  std::vector<int> seen(size_t(B) * H * W, 0);
  for (int t = 0; t < g.tiles; ++t)
    if (!check_tile(g, t, &seen)) return false;
  for (size_t i = 0; i < seen.size(); ++i)
    if (seen[i] != 1) {
      printf("B %d H %d W %d: cell %zu is the output of %d positions\n", B, H, W, i, seen[i]);
      return false;
    }
  return true;
}

int main() {
  ll stacked = 0;
  for (int W = 1; W <= 400; W += W < 12 ? 1 : (W < 120 ? 19 : (W < 131 ? 1 : 31)))
    for (int H : {1, 2, 3, 5, 8, 21, 64, 131})
      for (int B : {1, 2, 3, 7, 61, 1500}) {
        if ((ll)B * H * W > 300000) continue;
        if (!check_all(B, H, W)) return 1;
        stacked += grid3_of(B, H, W).per > 1;
      }
  const ll small = checked;
  for (int W = 1; W <= 300; ++W) {
    const int H = int(std::min<ll>((1ll << 30) / W, 715827882ll));
    const Grid3 g = grid3_of(1, H, W);
    const ll n = g.tps;
    if (n != ((ll)H * g.PW + 127) / 128 || (ll)g.tiles != n * g.strips) {
      printf("H %d W %d: %d tiles per strip\n", H, W, g.tps);
      return 1;
    }
    // the numbers where floor(2^32 / PW) + 1 stops being exact, and the tiles about them
    const ll e = (ll)g.rPW * g.PW - (1ll << 32), first = (1ll << 32) / e / 128;
    std::vector<ll> at;
    for (ll c : {(ll)0, n / 2, n - 1, first, 2 * first, 4 * first, 8 * first})
      for (ll d = -12; d <= 12; ++d) at.push_back(c + d);
    for (int i = 0; i < 300; ++i) at.push_back(ll(next_u64() % uint64_t(n)));
    for (ll i : at)
      if (i >= 0 && i < n)
        for (int s = 0; s < g.strips; ++s)
          if (!check_tile(g, s * n + i, nullptr)) return 1;
  }
  const ll tall = checked - small;
  for (int H : {1, 2, 3, 5, 8, 13})
    for (int W : {1, 2, 3, 5, 8, 14, 64, 126, 127, 260}) {
      const Grid3 g = grid3_of(int((1ll << 30) / ((ll)H * W)), H, W);
      for (ll c : {(ll)0, (ll)g.tps, (ll)g.tiles / 2, (ll)g.tiles - 1})
        for (ll d = -40; d <= 40; ++d)
          if (c + d >= 0 && c + d < g.tiles && !check_tile(g, c + d, nullptr)) return 1;
      for (int i = 0; i < 300; ++i)
        if (!check_tile(g, ll(next_u64() % uint64_t(g.tiles)), nullptr)) return 1;
    }
  for (int H = 1; H <= 40; ++H)
    for (int W = 1; W <= 140; ++W) {
      const Grid3 g = grid3_of(4096, H, W);
      const ll full = (4096ll * (H + 1) * g.PW + 127) / 128 * g.strips;
      if (7LL * g.tiles > 8 * (full + 4LL * g.strips * (full / 1024 + 1))) {  // an eighth, and a partly empty tile per stack
        printf("H %d W %d: %d tiles for %lld tiles' positions\n", H, W, g.tiles, full);
        return 1;
      }
    }
  printf("ok small %lld (%lld grids stacked) tall %lld many %lld\n", small, stacked, tall, checked - small - tall);
  return 0;
}
