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

}  // namespace gmmsp
