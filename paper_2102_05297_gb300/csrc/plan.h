// How steps are split over the GPU's SMs: host arithmetic alone, so that it can be
// compiled and checked without a GPU.
#pragma once

#include <stdint.h>

#include <algorithm>
#include <vector>

namespace ktune {

// Weighted-draw steps over materialised one-word spaces that one CTA does by default: up
// to kSmallMax configurations, four per thread, while the staged trees come in few
// groups (147 KB: four of depth 12, two of depth 13, one of depth 14; a group is a round
// trip and three barriers, and every tree's summands are made by this CTA alone).  us
// per step, 32 counters (one CTA / the persistent kernel / four kernels), 1,024, 2,048,
// 3,072 and 4,096 configurations:
//   depth  8   23.8 / 35.3 / 41.2   25.0 / 34.8 / 41.2   28.4 / 34.2 / 40.6   30.3 / 38.1 / 43.7
//   depth 12   33.5 / 41.8 / 48.4   34.9 / 40.1 / 49.5   39.4 / 40.8 / 51.3   40.0 / 38.6 / 48.9
//   depth 13   40.7 / 41.8 / 48.0   46.2 / 46.9 / 54.4   51.1 / 46.9 / 55.3   54.2 / 47.6 / 56.1
//   depth 14   64.5 / 61.1 / 66.1   67.5 / 60.3 / 68.6   74.5 / 62.0 / 69.4   75.0 / 58.5 / 66.1
constexpr int64_t kSmallMax = 4096;
inline bool small_step(int64_t N, int D) { return N <= kSmallMax && D <= (N <= 2048 ? 13 : 12); }

// CTAs of the persistent step of a search over N configurations, by default and below
// 2^18 of them (larger spaces fill the GPU in any case).  The kernel holds an SM per
// CTA for as long as its chain of latencies lasts, so with a CTA on every SM the steps
// of several searches run one after the other.
//
// waits: the caller waits for every step (ktune_step), so a step's own time counts
// first: 1,024 configurations per CTA (two per thread), where more CTAs gain nothing,
// and all but four SMs at most, which costs a step nothing either and lets it start
// while the last CTAs of up to four others draw.  Otherwise (ktune_step_device) the
// caller enqueues and may have many searches in flight: a quarter of the SMs, or full
// chunks of 4,096.
//
// us per step, depth-12 trees for 32 counters, 152 SMs: one search waited for / one
// enqueued / 8 threads waiting, a search each / 8 searches enqueued on 8 streams
//   configurations   four kernels           a CTA on every SM       this rule
//        40,960      56.1 47.8 17.5  7.3    43.3 33.3 30.9 28.4     42.7 33.5 16.6  7.4
//       131,072      55.2 45.9 17.9  7.5    42.2 32.1 32.1 30.0     43.0 37.9 22.9  8.3
//       163,840      56.5 47.9 18.0  8.1    43.8 33.6 31.2 29.8     44.0 37.9 24.7  8.2
//       245,760      56.8 48.1 18.2  9.8    43.6 34.3 32.7 31.2     42.8 37.8 26.3 12.3
// (about 7 of the last column are the host's enqueueing, 16 of the third the
// interpreter's.  Half of the SMs for those that wait: 20.5 at 163,840 and 8 threads,
// but 46.7 alone.)
inline int shared_grid(int64_t N, int sms, bool waits) {
  const int64_t by_1024 = std::max<int64_t>(16, (N + 1023) / 1024);
  const int64_t g = waits ? std::min<int64_t>(by_1024, std::max(1, sms - 4))
                          : std::max(std::min<int64_t>(by_1024, std::max(1, sms / 4)), (N + 4095) / 4096);
  return (int)std::min<int64_t>(g, sms);
}

// A batch's searches, of units[i] configurations (raw tiles on the fly), cut into work
// items, item after item dealt into at most `bins` bins (a CTA's share): bin b holds
// items first[b] .. first[b + 1).  A CTA takes a whole chunk of configurations in the
// time of one, so items are whole chunks but for a search's last, and an item costs
// its chunks and `piece` more, as it stages its search's trees.  The bins' common size
// is the smallest with which they suffice: searches that need no cutting have a bin
// each while there are bins.  us per batched step, depth-12 trees for 32 counters, 152
// SMs (pieces of total / SMs configurations of each search, dealt out in turn / even
// bins with room to spare / here): 64 searches of 500 configurations 281 / 286 / 268,
// 32 each of 40,960 and 500 332 / 354 / 299, 8 each of 196,608, 3,600, 500 and 16,384
// 245 / 284 / 199.
struct Cut {
  int search;
  int64_t lo, hi;
};
inline void cut_bins(const std::vector<int64_t> &units, int bins, int64_t chunk, int64_t piece,
                     std::vector<Cut> *items, std::vector<int> *first) {
  int64_t total = 0;
  for (int64_t u : units)
    if (u > 0) total += (u + chunk - 1) / chunk * chunk + piece;
  auto fill = [&](int64_t size) {
    int64_t room = 0;
    items->clear();
    first->clear();
    for (size_t i = 0; i < units.size(); ++i)
      for (int64_t lo = 0; lo < units[i];) {
        if (room < piece + chunk) {
          first->push_back((int)items->size());
          room = size;
        }
        const int64_t n = std::min((room - piece) / chunk, (units[i] - lo + chunk - 1) / chunk);
        const int64_t hi = std::min(units[i], lo + n * chunk);
        items->push_back({(int)i, lo, hi});
        room -= piece + n * chunk;
        lo = hi;
      }
    return (int)first->size();
  };
  int64_t size = std::max(piece + chunk, (total + bins - 1) / bins);
  while (fill(size) > bins) size += piece;
  first->push_back((int)items->size());
}

}  // namespace ktune
