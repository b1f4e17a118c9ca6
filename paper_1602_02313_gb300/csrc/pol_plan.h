// Split of the tensor-core polarization's K chunks into segments (plain C++ as well, so that the test suite
// can run it over all sizes on the host).
#pragma once
#include "cvt.cuh"

namespace gwi {

// Chunks of a segment: segment s of nseg covers the chunks [s L, min(total, (s + 1) L)).
GW_HD int pol_seg_len(int total, int nseg) { return (total + nseg - 1) / nseg; }

// Number of K segments for `total` chunks of 32 pairs: segments of at most seg_chunks (the FP32 accumulation
// error grows with the MMAs chained into one accumulator), more of them while the base_units units of one
// segment do not fill two waves of the GPU and the segments stay at 4 chunks or more; then only as many as
// segments of that length reach (16 chunks in 10 segments would be 8 of 2 and two empty ones).
inline int pol_segments(int total, int base_units, int seg_chunks, int sms) {
  int nseg = (total + seg_chunks - 1) / seg_chunks;
  if (nseg < 1) nseg = 1;
  while (base_units * nseg < 2 * sms && (total + nseg) / (nseg + 1) >= 4) ++nseg;
  const int len = pol_seg_len(total, nseg);
  return (total + len - 1) / len;
}

}  // namespace gwi
