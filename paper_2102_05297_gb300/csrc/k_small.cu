// The whole step of a tree search over a small space (materialised one-word
// digits, at most kSmallMax configurations, weighted draws) as one CTA.
//
// What bounds it: latency alone -- a step of 1,824 configurations is 130,000 node
// visits.  So everything between the trees' node words and the outputs stays in
// shared memory and registers: the trees with a Delta are staged with their leaf
// values in one asynchronous round trip, c_profile walks them there, the leaf
// values become the step's summands in place, each thread scores up to four
// neighbouring configurations, the extremes and the weights' prefix sums are block
// reductions, and warp 0 draws from them (by interval mapping, see draws.cuh).
// Scores and weights are stored for read-back only.  As four kernels the same
// step is 38 us of kernels and their hand-overs (prepare 6, score 15, weights 7,
// select 10), as the persistent kernel 26 us (two grid barriers and every phase's
// results through L2); host call to host result, 1,920 configurations, depth 8:
// 44, 36 and here 27 us (depth 12 for 32 counters: 54, 41 and 40).  A second CTA
// would need both of those hand-overs again;
// with more than four configurations a thread the walk itself passes them.
#include <float.h>
#include <limits.h>

#include <algorithm>
#include <atomic>

#include "step_common.cuh"

namespace ktune {

namespace {

constexpr int kSmallThreads = 1024;
constexpr int kSmallSmem = 200 * 1024;
// per configuration: weight, score, digits; per thread: prefix sum
constexpr int kSmallFixed = kSmallMax * 12 + kSmallThreads * 8;
static_assert(kSmallFixed + 2 * (8 << 13) <= kSmallSmem, "two trees of depth 13");

template <int CPT>
__global__ void __launch_bounds__(kSmallThreads, 1) k_step_small(const __grid_constant__ FusedArgs fa) {
  extern __shared__ __align__(16) uint8_t smem[];
  __shared__ float sh_dl[KTUNE_MAX_COUNTERS], sh_A[KTUNE_MAX_COUNTERS];
  __shared__ int sh_p[KTUNE_MAX_COUNTERS];
  __shared__ int sh_n, sh_act;
  __shared__ float red_mn[32], red_mx[32];
  __shared__ uint64_t sh_scan[32];
  const SearchDev &sd = fa.sd;
  const StepDev &st = fa.st;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int D = sd.D, L = 1 << D, N = (int)sd.N, k = st.k;
  uint32_t *sh_w = reinterpret_cast<uint32_t *>(smem);                 // [kSmallMax] weights
  float *sh_s = reinterpret_cast<float *>(sh_w + kSmallMax);           // scores
  uint32_t *sh_W = reinterpret_cast<uint32_t *>(sh_s + kSmallMax);     // digits
  uint64_t *sh_pre = reinterpret_cast<uint64_t *>(sh_W + kSmallMax);   // [threads] inclusive prefix sums
  uint32_t *trees = reinterpret_cast<uint32_t *>(sh_pre + kSmallThreads);
  const int per_group = (kSmallSmem - kSmallFixed) / (8 * L);

  // this thread's configurations
  const int i0 = (int)threadIdx.x * CPT;
  uint32_t W[CPT];
  float s[CPT];
#pragma unroll
  for (int c = 0; c < CPT; ++c) {
    W[c] = i0 + c < N ? __ldg(sd.narrow + i0 + c) : 0u;
    s[c] = 0.0f;
  }
  const uint32_t ev = i0 < N ? sd.eval[i0 >> 5] >> (i0 & 31) : ~0u;   // CPT divides 32: one word
  // the counters with a Delta, ascending
  if (warp == 0) {
    int base = 0;
    for (int c0 = 0; c0 < sd.K; c0 += 32) {
      const int p = c0 + lane;
      const float dl = p < sd.K ? st.delta[p] : 0.0f;
      const unsigned m = __ballot_sync(kFullMask, dl != 0.0f);
      if (dl != 0.0f) {
        const int a = base + __popc(m & ((1u << lane) - 1u));
        sh_p[a] = p;
        sh_dl[a] = dl;
      }
      base += __popc(m);
    }
    if (lane == 0) {
      sh_n = base;
      sh_act = 0;
    }
  }
  __syncthreads();
  const int n = sh_n;
  uint32_t cw = 0;   // c_profile's digits in the one-word form
  for (int j = 0; j < sd.sa.P; ++j) cw |= nib64(st.cprof_packed, j) << sd.pos[j];
  // the draws' variates
  const uint64_t u_lo = warp == 0 ? philox_u64(sd.seed, sd.search_id, st.step, (uint32_t)lane, 0u) : 0ull;
  const uint64_t u_hi =
      warp == 0 && lane + 32 < k ? philox_u64(sd.seed, sd.search_id, st.step, (uint32_t)(lane + 32), 0u) : 0ull;

  for (int t0 = 0; t0 < n; t0 += per_group) {
    const int nt = min(per_group, n - t0);
    // node words at 1 .. L - 1, leaf values (then summands) at L .. 2 L - 1
    for (int a = 0; a < nt; ++a) {
      const int p = sh_p[t0 + a];
      uint32_t *dst = trees + (size_t)a * 2 * L;
      const uint32_t *ws = fa.words + (size_t)p * L;
      const float *ls = sd.leaves + (size_t)p * L;
      if (L >= 4) {
        for (int i = threadIdx.x; i < L / 2; i += kSmallThreads) {
          if (i < L / 4) cp_async16(dst + 4 * i, ws + 4 * i);
          else cp_async16(dst + 4 * i, ls + 4 * i - L);
        }
      } else if ((int)threadIdx.x < 2 * L) {
        const int i = threadIdx.x;
        dst[i] = i < L ? __ldg(ws + i) : __float_as_uint(__ldg(ls + i - L));
      }
    }
    cp_async_wait_all();
    __syncthreads();
    if ((int)threadIdx.x < nt) {   // c_profile, a tree per thread
      const uint32_t *tr = trees + (size_t)threadIdx.x * 2 * L;
      uint32_t j = 1;
      for (int l = 0; l < D; ++l) j = narrow_visit(j, tr[j], cw);
      const float A = __uint_as_float(tr[j]);
      sh_A[threadIdx.x] = A;
      if (A != 0.0f) atomicAdd(&sh_act, 1);
    }
    __syncthreads();
    // summand of a leaf: Delta (x - A) / (x + A), 0 where x or x + A is 0
    for (int e = threadIdx.x; e < nt * L; e += kSmallThreads) {
      const int a = e >> D;
      float *x = reinterpret_cast<float *>(trees + (size_t)a * 2 * L + L + (e & (L - 1)));
      const float A = sh_A[a], v = *x, den = __fadd_rn(v, A);
      float t = 0.0f;
      if (v != 0.0f && den != 0.0f) t = __fmul_rn(sh_dl[t0 + a], __fdiv_rn(__fsub_rn(v, A), den));
      *x = t;
    }
    __syncthreads();
    if (i0 < N)
      for (int a = 0; a < nt; ++a) {
        if (sh_A[a] == 0.0f) continue;      // not in PC_used
        const uint32_t *tr = trees + (size_t)a * 2 * L;
        uint32_t j[CPT];
#pragma unroll
        for (int c = 0; c < CPT; ++c) j[c] = 1;
        for (int l = 0; l < D; ++l)
#pragma unroll
          for (int c = 0; c < CPT; ++c) j[c] = narrow_visit(j[c], tr[j[c]], W[c]);
#pragma unroll
        for (int c = 0; c < CPT; ++c) s[c] = __fadd_rn(s[c], __uint_as_float(tr[j[c]]));
      }
    __syncthreads();
  }
  // extremes over the unevaluated configurations
  float mn = INFINITY, mx = -INFINITY;
#pragma unroll
  for (int c = 0; c < CPT; ++c) {
    const bool open = i0 + c < N && !((ev >> c) & 1u);
    if (open) {
      mn = fminf(mn, s[c]);
      mx = fmaxf(mx, s[c]);
    } else {
      s[c] = 0.0f;
    }
    if (i0 + c < N) {
      sd.s[i0 + c] = s[c];
      sh_s[i0 + c] = s[c];
      sh_W[i0 + c] = W[c];
    }
  }
  for (int o = 16; o; o >>= 1) {
    mn = fminf(mn, __shfl_xor_sync(kFullMask, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, o));
  }
  if (lane == 0) {
    red_mn[warp] = mn;
    red_mx[warp] = mx;
  }
  __syncthreads();
  mn = red_mn[lane];
  mx = red_mx[lane];
  for (int o = 16; o; o >>= 1) {
    mn = fminf(mn, __shfl_xor_sync(kFullMask, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(kFullMask, mx, o));
  }
  if (threadIdx.x == 0) {
    sd.mm[0] = mn <= mx ? okey(mn) : INT_MAX;
    sd.mm[1] = mn <= mx ? okey(mx) : INT_MIN;
    *sd.n_active = sh_act;
  }
  // weights and their prefix sums, thread by thread
  uint64_t sum = 0;
#pragma unroll
  for (int c = 0; c < CPT; ++c) {
    const bool open = i0 + c < N && !((ev >> c) & 1u);
    const uint32_t w = open ? (uint32_t)weight_of(s[c], mn, mx, sd.gamma) : 0u;
    if (i0 + c < N) sd.w[i0 + c] = w;
    sh_w[i0 + c] = w;
    sum += w;
  }
  {
    uint64_t tot;
    const uint64_t incl = block_incl<uint64_t>(sum, sh_scan, &tot);
    sh_pre[threadIdx.x] = incl;
  }
  __syncthreads();
  if (warp) return;

  // ---- the draws (warp 0) ----------------------------------------------------------
  const uint64_t ends = sh_pre[lane * 32 + 31];
  uint64_t Wt = __shfl_sync(kFullMask, ends, 31);
  uint64_t pb0 = ~0ull, pb1 = ~0ull, rb0 = ~0ull, rb1 = ~0ull;   // lane q: picks q and q + 32
  uint32_t pw0 = 0, pw1 = 0;
  int my0 = 0, my1 = 0, count = 0;
  for (int j = 0; j < k && Wt; ++j) {
    const uint64_t u = j < 32 ? __shfl_sync(kFullMask, u_lo, j) : __shfl_sync(kFullMask, u_hi, j - 32);
    const uint64_t r = scaled_draw(u, Wt);
    const uint64_t add = warp_sum30(rb0 <= r ? pw0 : 0u, rb1 <= r ? pw1 : 0u);
    const uint64_t x = r + add;
    unsigned over = __ballot_sync(kFullMask, ends > x);
    if (!over) break;                        // cannot happen with consistent sums
    const int wsel = __ffs(over) - 1;
    const uint64_t pv = sh_pre[wsel * 32 + lane];
    over = __ballot_sync(kFullMask, pv > x);
    if (!over) break;
    const int t = wsel * 32 + __ffs(over) - 1;
    uint64_t at = t ? sh_pre[t - 1] : 0ull;
    int pick = t * CPT;
    uint32_t w = sh_w[pick];
#pragma unroll
    for (int c = 1; c < CPT; ++c)
      if (x >= at + w) {
        at += w;
        w = sh_w[++pick];
      }
    // the pick's interval: later intervals begin earlier without it
    if (pw0 && pb0 > at) rb0 -= w;
    if (pw1 && pb1 > at) rb1 -= w;
    if (lane == (count & 31)) {
      if (count < 32) {
        pb0 = at;
        rb0 = at - add;
        pw0 = w;
        my0 = pick;
      } else {
        pb1 = at;
        rb1 = at - add;
        pw1 = w;
        my1 = pick;
      }
    }
    Wt -= w;
    ++count;
  }
  for (int q = lane; q < count; q += 32) {
    const int i = q < 32 ? my0 : my1;
    const uint32_t word = sh_W[i];
    uint64_t p = 0;
    int64_t raw = 0;
    for (int d = 0; d < sd.sa.P; ++d) {
      const uint32_t dg = (word >> sd.pos[d]) & ((1u << sd.width[d]) - 1u);
      p |= (uint64_t)dg << (4 * d);
      raw += (int64_t)dg * sd.sa.stride[d];
    }
    st.out_raw[q] = raw;
    st.out_score[q] = sh_s[i];
    if (st.out_packed) st.out_packed[q] = p;
    sd.w[i] = 0u;
    atomicOr(sd.eval + (i >> 5), 1u << (i & 31));
  }
  if (lane == 0 && st.n_out) *st.n_out = count;
}

template <int CPT>
cudaError_t launch_small_t(const FusedArgs &fa, cudaStream_t st) {
  static std::atomic<uint64_t> done{0};   // bit d: the shared-memory opt-in made on device d
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < 64 ? 1ull << dev : 0ull;
  if (!bit || !(done.load() & bit)) {
    e = cudaFuncSetAttribute(k_step_small<CPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmem);
    if (e != cudaSuccess) return e;
    done.fetch_or(bit);
  }
  // what the trees of this depth fill, at most all of it
  const size_t smem = std::min<size_t>(kSmallSmem, kSmallFixed + ((size_t)8 << fa.sd.D) * fa.sd.K);
  k_step_small<CPT><<<1, kSmallThreads, smem, st>>>(fa);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_step_small(const FusedArgs &fa, cudaStream_t st) {
  if (fa.sd.N <= kSmallThreads) return launch_small_t<1>(fa, st);
  if (fa.sd.N <= 2 * kSmallThreads) return launch_small_t<2>(fa, st);
  return launch_small_t<4>(fa, st);
}

}  // namespace ktune
