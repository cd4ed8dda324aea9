// Host check of the batch launch rules (gmmsp_batch_rules.h).  Prints "ok" and exits 0, or the first mismatch.
#include <stdio.h>

#include "gmmsp_batch_rules.h"

int main() {
  // finalizes at most one level ahead of the caller's stream, and at a level that the device has
  for (int most = -5; most <= 0; ++most)
    for (int caller = most; caller <= 0; ++caller) {
      const int p = gmmsp::finalize_priority(caller, most);
      if (p < most || p > caller || caller - p > 1 || (caller > most && p != caller - 1)) {
        printf("priority %d for a stream at %d (most urgent %d)\n", p, caller, most);
        return 1;
      }
    }
  struct {
    int n;
    long long cells;
    int bps, first;
    bool two;
  } cases[] = {{1, 100000, 6, 6, false}, {2, 16 * 152, 6, 6, true}, {2, 16 * 152 - 1, 6, 6, false},
               {256, 185856, 7, 6, true}, {256, 185856, 5, 6, false}, {256, 185856, 6, 5, false}};
  for (const auto& c : cases)
    if (gmmsp::two_parts(c.n, c.cells, 152, c.bps, c.first) != c.two) {
      printf("parts of %d images, %lld cells, %d and %d blocks per SM\n", c.n, c.cells, c.bps, c.first);
      return 1;
    }
  struct {
    int n;
    long long cells;
    bool gray;
    int blocks;
  } untuned[] = {{4, 400, false, 5},          {4, 400, true, 6},  {1, 20 * 152, false, 5}, {1, 20 * 152 + 1, false, 6},
                 {2, 16 * 152 - 1, false, 5}, {2, 16 * 152, false, 6}, {256, 185856, false, 6}};
  for (const auto& u : untuned)
    if (gmmsp::default_blocks(u.n, u.cells, 152, u.gray) != u.blocks) {
      printf("untuned blocks per SM of %d images, %lld cells\n", u.n, u.cells);
      return 1;
    }
  printf("ok\n");
  return 0;
}
