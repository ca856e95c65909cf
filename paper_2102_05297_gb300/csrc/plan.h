// How steps are split over the GPU's SMs: host arithmetic alone, so that it can be
// compiled and checked without a GPU.
#pragma once

#include <stdint.h>

#include <algorithm>

namespace ktune {

// CTAs of the persistent step of a search over N configurations, by default and below
// 2^18 of them (larger spaces fill the GPU in any case).  The kernel holds an SM per
// CTA for as long as its chain of latencies lasts, so with a CTA on every SM the steps
// of several searches run one after the other.
//
// waits: the caller waits for every step (ktune_step), so a step's own time counts
// first.  As few CTAs as cost it nothing: 1,024 configurations each (two per thread)
// or, where that takes more than the SMs, 1,536 (a walk of 3 per thread costs what 4
// do); at most 7/8 of the SMs then, so that a step starts beside another's draws.
// Otherwise (ktune_step_device) the caller enqueues and may have many searches in
// flight: a quarter of the SMs, or full chunks of 4,096.
//
// us per step, depth-12 trees for 32 counters, 152 SMs: one search waited for / one
// enqueued / 8 threads waiting, a search each / 8 searches enqueued on 8 streams
//   configurations   four kernels           a CTA on every SM       this rule
//        40,960      56.1 47.8 17.5  7.3    43.3 33.3 30.9 28.4     42.7 33.5 16.6  7.4
//       131,072      55.2 45.9 17.9  7.5    42.2 32.1 32.1 30.0     43.0 37.9 22.9  8.3
//       163,840      56.5 47.9 18.0  8.1    42.9 33.6 31.8 29.8     43.4 37.9 23.0  8.2
//       245,760      56.8 48.1 18.2  9.8    44.4 34.3 33.3 31.2     45.1 37.8 26.0 12.3
// (about 7 of the last column are the host's enqueueing, 17 of the third the interpreter's)
inline int shared_grid(int64_t N, int sms, bool waits) {
  const int64_t by_1024 = std::max<int64_t>(16, (N + 1023) / 1024);
  const int64_t g = waits ? (by_1024 <= sms ? by_1024 : std::min<int64_t>((N + 1535) / 1536, sms - sms / 8))
                          : std::max(std::min<int64_t>(by_1024, std::max(1, sms / 4)), (N + 4095) / 4096);
  return (int)std::min<int64_t>(g, sms);
}

}  // namespace ktune
