// Algorithm 1's k draws without replacement over a step's integer weights, by
// one CTA.
//
// Draw j takes the configuration holding r_j = floor(u_j W_j / 2^64) in the
// prefix sums of the weights that the earlier picks have left, W_j their total.
// Nothing is ever taken off the sums here: removing the picks' intervals maps
// the remaining range onto the original one by x = r + (the weights of the picks
// whose interval begins at or before r, their own beginnings counted without the
// picks before them).  So every level -- sub-tiles, groups of 32, weights -- is a
// search of prefix sums that stay as they were made, and all a draw waits for is
// its predecessors' intervals, which lanes hold in registers.
//
// Before the draws, each warp locates one draw as if it were the first, fetches
// that sub-tile's weights and scans the draw's group of 32; the true position is
// then a few weights away, most often in the same group, nearly always in the same
// sub-tile.  What bounds it: two dependent L2 round trips and the chain of the k
// draws (with the picks taken off the sums, every draw searched the three levels
// again: about 2,500 cycles each).
#pragma once

#include "step_common.cuh"

namespace ktune {
namespace {

constexpr int kDrawBufs = 16;     // sub-tiles fetched ahead, per round of as many draws
constexpr int kDrawTop = 4096;    // sub-tile (or, where there are more, super-tile) sums kept
// what the draws share beside the sums and buffers (dynamic too: the fused step's
// kernel uses nearly all of an SM's shared memory that way)
struct DrawShared {
  uint64_t scan[32];
  uint64_t base[kDrawBufs];      // the weight before the sub-tile in a buffer
  uint64_t sum[kDrawBufs];       // and its own
  uint64_t gbase[kDrawBufs];     // the same of the group looked ahead to
  uint64_t gsum[kDrawBufs];
  uint64_t incl[kDrawBufs][32];  // that group's inclusive prefix sums
  uint64_t rb[KTUNE_MAX_K];      // the picks for the next round's look ahead
  uint64_t W;
  uint32_t w[KTUNE_MAX_K];
  int g[kDrawBufs];              // the sub-tile in a buffer (-1: none)
  int og[kDrawBufs];             // the group in it
  int n;
};
constexpr int kDrawSmem =
    kDrawTop * 8 + (kDrawBufs + 1) * (32 * 8 + kSubTile * 4) + (int)((sizeof(DrawShared) + 15) / 16 * 16);

// Called by the whole CTA; pick[] (shared) receives the ordinals in draw order,
// the return value is their number.  The picks' weights are zeroed and their
// evaluated bits set.  smem: kDrawSmem bytes, 16-byte aligned.
__device__ __noinline__ int draw_k(const SearchDev &sd, const StepDev &st, uint8_t *smem, int64_t *pick) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int THREADS = blockDim.x;
  const int64_t N = sd.N;
  const int k = st.k;
  uint64_t *top = reinterpret_cast<uint64_t *>(smem);            // inclusive prefix sums
  uint64_t *gp = top + kDrawTop;                                 // [bufs + 1][32] per sub-tile: its groups'
  uint32_t *buf = reinterpret_cast<uint32_t *>(gp + (kDrawBufs + 1) * 32);   // [bufs + 1][kSubTile] weights
  DrawShared &sh = *reinterpret_cast<DrawShared *>(buf + (kDrawBufs + 1) * kSubTile);
  const int n_sub = (int)((N + kSubTile - 1) / kSubTile), n_super = (n_sub + kSuper - 1) / kSuper;
  const bool cached = n_sub <= kDrawTop;
  const int n_top = cached ? n_sub : n_super;
  const uint64_t *src = cached ? sd.sub_sum : sd.super_sum;
  for (int i = threadIdx.x; 2 * i < n_top; i += THREADS) {      // every copy in flight before one wait
    if (2 * i + 1 < n_top) cp_async16(top + 2 * i, src + 2 * i);
    else top[2 * i] = __ldcg(src + 2 * i);
  }
  // the draws' variates meanwhile (draw `lane`, `lane + 32`)
  const uint64_t u_lo = philox_u64(sd.seed, sd.search_id, st.step, (uint32_t)lane, 0u);
  const uint64_t u_hi =
      lane + 32 < k ? philox_u64(sd.seed, sd.search_id, st.step, (uint32_t)(lane + 32), 0u) : 0ull;
  auto variate = [&](int j) {
    return j < 32 ? __shfl_sync(kFullMask, u_lo, j) : __shfl_sync(kFullMask, u_hi, j - 32);
  };
  cp_async_wait_all();
  __syncthreads();
  {   // prefix sums in place, a run of entries per thread
    const int per = (n_top + THREADS - 1) / THREADS;
    const int lo = min(n_top, per * (int)threadIdx.x), hi = min(n_top, lo + per);
    uint64_t s = 0, tot;
    for (int i = lo; i < hi; ++i) s += top[i];
    uint64_t acc = block_incl<uint64_t>(s, sh.scan, &tot) - s;
    for (int i = lo; i < hi; ++i) {
      acc += top[i];
      top[i] = acc;
    }
  }
  __syncthreads();

  // the sub-tile holding x: its index, the weight before it and its own (a warp;
  // false if x is not below the total or the sums are inconsistent)
  auto locate = [&](uint64_t x, int &g, uint64_t &base, uint64_t &sum) -> bool {
    const int S = (n_top + 31) / 32;
    const uint64_t pv = lane * S < n_top ? top[min((lane + 1) * S, n_top) - 1] : ~0ull;
    unsigned over = __ballot_sync(kFullMask, lane * S < n_top && pv > x);
    if (!over) return false;
    const int c = (__ffs(over) - 1) * S, end = min(c + S, n_top);
    int t = -1;
    for (int b = c; b < end && t < 0; b += 32) {
      over = __ballot_sync(kFullMask, b + lane < end && top[min(b + lane, end - 1)] > x);
      if (over) t = b + __ffs(over) - 1;
    }
    if (t < 0) return false;
    base = t ? top[t - 1] : 0ull;
    sum = top[t] - base;
    g = t;
    if (!cached) {
      const int gi = t * kSuper + lane;
      const uint64_t v = gi < n_sub ? __ldcg(sd.sub_sum + gi) : 0ull;
      const uint64_t inc = warp_incl(v), y = x - base;
      const int at = __ffs(__ballot_sync(kFullMask, inc - v <= y && y < inc)) - 1;
      if (at < 0) return false;
      g = t * kSuper + at;
      base += __shfl_sync(kFullMask, inc - v, at);
      sum = __shfl_sync(kFullMask, v, at);
    }
    return g < n_sub;
  };
  // sub-tile g's weights into buffer b, every copy in flight at once, and the
  // inclusive prefix over its groups of 32 (a warp)
  auto fetch = [&](int b, int g) {
    const int64_t i0 = (int64_t)g * kSubTile;
    uint32_t *d = buf + b * kSubTile;
    for (int q = lane; q < kSubTile / 4; q += 32) {
      const int64_t i = i0 + 4 * q;
      if (i + 3 < N) {
        cp_async16(d + 4 * q, sd.w + i);
      } else {
        uint4 x;
        x.x = i < N ? __ldcg(sd.w + i) : 0u;
        x.y = i + 1 < N ? __ldcg(sd.w + i + 1) : 0u;
        x.z = i + 2 < N ? __ldcg(sd.w + i + 2) : 0u;
        x.w = 0u;
        reinterpret_cast<uint4 *>(d)[q] = x;
      }
    }
    cp_async_wait_all();
    __syncwarp();
    // lane l sums weights 32 l .. 32 l + 31 (the lanes start at different
    // quarters of their 128 bytes, so that a load spreads over all banks)
    const uint4 *s4 = reinterpret_cast<const uint4 *>(d + lane * 32);
    uint64_t ls = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const uint4 x = s4[(q + lane) & 7];
      ls += (uint64_t)x.x + x.y + (uint64_t)x.z + x.w;
    }
    gp[b * 32 + lane] = warp_incl(ls);
    __syncwarp();
  };

  // warp 0: lane q holds pick q and q + 32 -- where its interval begins, without
  // any pick removed (pb) and without the picks before it (rb), and its weight
  uint64_t pb0 = ~0ull, pb1 = ~0ull, rb0 = ~0ull, rb1 = ~0ull;
  uint32_t pw0 = 0, pw1 = 0;
  int count = 0;
  uint64_t W = top[n_top - 1];
  for (int j0 = 0; j0 < k; j0 += kDrawBufs) {
    const int n = min(kDrawBufs, k - j0);
    for (int b = warp; b < n; b += nw) {
      const uint64_t u = variate(j0 + b);
      int g = -1;
      uint64_t base = 0, sum = 0;
      if (W > 0) {
        uint64_t x = scaled_draw(u, W);
        if (j0) {
          const uint32_t a = lane < count && sh.rb[lane] <= x ? sh.w[lane] : 0u;
          const uint32_t c = lane + 32 < count && sh.rb[lane + 32] <= x ? sh.w[lane + 32] : 0u;
          x += warp_sum30(a, c);
        }
        if (locate(x, g, base, sum)) {
          fetch(b, g);
          const uint64_t gl = gp[b * 32 + lane];
          const unsigned over = __ballot_sync(kFullMask, gl > x - base);
          const int og = over ? __ffs(over) - 1 : 31;
          const uint64_t end = __shfl_sync(kFullMask, gl, og), before = __shfl_sync(kFullMask, gl, og > 0 ? og - 1 : 0);
          const uint64_t gb = og > 0 ? before : 0ull;
          sh.incl[b][lane] = warp_incl((uint64_t)buf[b * kSubTile + og * 32 + lane]);
          if (lane == 0) {
            sh.og[b] = og;
            sh.gbase[b] = base + gb;
            sh.gsum[b] = end - gb;
          }
        } else {
          g = -1;
        }
      }
      if (lane == 0) {
        sh.g[b] = g;
        sh.base[b] = base;
        sh.sum[b] = sum;
      }
    }
    __syncthreads();
    if (warp == 0) {
      const int my_spec = lane < n ? sh.g[lane] : -1;
      for (int b = 0; b < n; ++b) {
        if (W == 0) break;
        const uint64_t r = scaled_draw(variate(j0 + b), W);
        const uint64_t add = warp_sum30(rb0 <= r ? pw0 : 0u, rb1 <= r ? pw1 : 0u);
        const uint64_t x = r + add;
        int g = sh.g[b];
        uint32_t w;
        uint64_t at;
        int qs, og = sh.og[b];
        const uint64_t y0 = x - sh.gbase[b];
        if (g >= 0 && x >= sh.gbase[b] && y0 < sh.gsum[b]) {      // in the group looked ahead to
          const uint32_t wq = buf[b * kSubTile + og * 32 + lane];
          const uint64_t iq = sh.incl[b][lane];
          qs = __ffs(__ballot_sync(kFullMask, iq > y0)) - 1;
          w = __shfl_sync(kFullMask, wq, qs);
          at = sh.gbase[b] + __shfl_sync(kFullMask, iq, qs) - w;
        } else {
          int bsel = b;
          uint64_t base = sh.base[b], sum = sh.sum[b];
          if (!(g >= 0 && x >= base && x - base < sum)) {
            if (!locate(x, g, base, sum)) break;           // cannot happen with consistent sums
            const unsigned has = __ballot_sync(kFullMask, my_spec == g);
            bsel = has ? __ffs(has) - 1 : kDrawBufs;
            if (!has) fetch(kDrawBufs, g);
          }
          const uint64_t y = x - base;
          const uint64_t gl = gp[bsel * 32 + lane];
          const unsigned over = __ballot_sync(kFullMask, gl > y);
          if (!over) break;                                // cannot happen with consistent sums
          og = __ffs(over) - 1;
          const uint32_t wq = buf[bsel * kSubTile + og * 32 + lane];
          const uint64_t before = __shfl_sync(kFullMask, gl, og > 0 ? og - 1 : 0);
          const uint64_t gbase = og > 0 ? before : 0ull;
          const uint64_t iq = warp_incl((uint64_t)wq);
          const unsigned hit = __ballot_sync(kFullMask, iq > y - gbase);
          if (!hit) break;                                 // cannot happen with consistent sums
          qs = __ffs(hit) - 1;
          w = __shfl_sync(kFullMask, wq, qs);
          at = base + gbase + __shfl_sync(kFullMask, iq, qs) - w;
        }
        if (lane == 0) pick[count] = (int64_t)g * kSubTile + og * 32 + qs;
        // the pick's interval: later intervals begin earlier without it
        if (pb0 > at && pw0) rb0 -= w;
        if (pb1 > at && pw1) rb1 -= w;
        if (lane == (count & 31)) {
          if (count < 32) {
            pb0 = at;
            rb0 = at - add;
            pw0 = w;
          } else {
            pb1 = at;
            rb1 = at - add;
            pw1 = w;
          }
        }
        W -= w;
        ++count;
      }
      sh.rb[lane] = rb0;
      sh.rb[lane + 32] = rb1;
      sh.w[lane] = pw0;
      sh.w[lane + 32] = pw1;
      if (lane == 0) {
        sh.n = count;
        sh.W = W;
      }
    }
    __syncthreads();
    count = sh.n;
    W = sh.W;
    if (count < j0 + n) break;
  }
  // the picks' weights read 0 from now on
  if ((int)threadIdx.x < count) {
    const int64_t i = pick[threadIdx.x];
    sd.w[i] = 0u;
    atomicOr(sd.eval + (i >> 5), 1u << (i & 31));
  }
  return count;
}

}  // namespace
}  // namespace ktune
