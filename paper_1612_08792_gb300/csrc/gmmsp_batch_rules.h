// Launch rules of a batch context that are plain integer arithmetic (checked
// by the host test suite).
#pragma once

namespace gmmsp {

// Launch priority of the finalizes of a batch that runs as two parts
// (numerically lower is more urgent; `caller` is the caller's stream's, `most`
// the device's most urgent): one level above the caller's stream, so that they
// go before the other part's E + M blocks and before nothing else that the
// caller put further ahead.  The device's most urgent level is no faster (256
// uneven images 41.19 ms at either); the caller's own is (44.47 ms).
inline int finalize_priority(int caller, int most) { return caller - 1 > most ? caller - 1 : most; }

// Whether a batch of n images and `cells` cells runs as two parts: from 16 cells
// per SM on, with the one-cell-per-warp E + M kernels (6 blocks per SM or more
// in the first pass and the others).
inline bool two_parts(int n, long long cells, int sms, int bps, int first_bps) {
  return n > 1 && cells >= 16LL * sms && bps >= 6 && first_bps >= 6;
}

// Blocks per SM of the E + M pass before any tuning.  6 (one cell per warp) is
// the fastest on every larger batch measured: 256 images of 481x321 0.895 ms a
// pass against 1.007 at 4 persistent blocks, 64 grey 640x480 0.328 against
// 0.366.  A launch that does not fill 5 blocks per SM gains nothing from room
// for a sixth and pays its register bound (56 bytes of spill a thread; none in
// the grayscale model), unless it runs as two parts, which take 6: 10 iterations
// on 4 images of 1000x1000 at v = 100 2.95 ms at 5, 3.46 at 6, 20 of 320x240 at
// v = 30 0.644 and 0.673, one of 1000x700 at v = 20 0.419 and 0.429; 4 of
// 481x321 0.402 as one part at 5, 0.397 as two at 6.
inline int default_blocks(int n, long long cells, int sms, bool gray) {
  if (gray || two_parts(n, cells, sms, 6, 6)) return 6;
  return cells <= 4LL * 5 * sms ? 5 : 6;
}

}  // namespace gmmsp
