// Neighbourhood-restricted steps (the footnote of Section 3.5: score only a
// neighbourhood of c_profile when the space is too large to score whole; the
// local search of Section 3.8.1).  The candidates are the configurations
// whose digits differ from c_profile's in 1 .. R parameters (R = 1 or 2), in
// a canonical order: distance 1 first (parameter j ascending, new digit
// ascending), then distance 2 (pairs i < j lexicographic, new digit of i
// ascending, then of j).  Only valid, unevaluated candidates are scored; the
// step normalises over them and draws k with the full step's integer weights
// and Philox draws, prefix sums in the canonical order, or takes the top k.
//
//   k_nbr_score   one warp per candidate: decode, constraint check, TS
//                 ordinal (a 32-way search over the ascending raw order),
//                 evaluated bit, one or two trees per lane, Eq. score;
//                 the last block does the step's set-up (c_profile's prediction,
//                 Delta, resets)
//   k_nbr_draws   one CTA, up to 4,096 candidates: min / max, weights and k draws
//                 without replacement from registers, outputs and marks
//   k_nbr_select  one CTA, larger neighbourhoods and the top k: compaction in
//                 canonical order first
#include <float.h>
#include <limits.h>

#include <algorithm>

#include "device_common.cuh"
#include "internal.h"
#include "step_common.cuh"

namespace ktune {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kScoreBlock = 256;

__device__ __forceinline__ int okey_n(float f) {
  const int b = __float_as_int(f);
  return b >= 0 ? b : b ^ 0x7FFFFFFF;
}

__device__ __forceinline__ float term_n(float a, float A, float dl) {
  const float den = __fadd_rn(a, A);
  return (a != 0.0f && den != 0.0f) ? __fmul_rn(dl, __fdiv_rn(__fsub_rn(a, A), den)) : 0.0f;
}

__device__ __forceinline__ bool valid_nbr(uint64_t p, const GroupDev *__restrict__ g, int n_groups,
                                          const uint32_t *__restrict__ table) {
  for (int k = 0; k < n_groups; ++k) {
    uint32_t sub = 0;
    for (int i = 0; i < g[k].n; ++i) sub += nib64(p, g[k].param[i]) * g[k].sub_stride[i];
    if (!((__ldg(table + g[k].off_words + (sub >> 5)) >> (sub & 31)) & 1u)) return false;
  }
  return true;
}

__device__ __forceinline__ int64_t raw_of(const SpaceArgs &sa, uint64_t p) {
  int64_t r = 0;
  for (int j = 0; j < sa.P; ++j) r += (int64_t)nib64(p, j) * sa.stride[j];
  return r;
}

// Index of the last of off[0 .. n) (ascending, off[0] = 0) that is <= e; the
// whole warp, e the same in every lane.
__device__ __forceinline__ int last_le(const int *off, int n, int e) {
  const int lane = threadIdx.x & 31;
  int q = 0;
  for (int q0 = 0; q0 < n; q0 += 32)
    q += __popc(__ballot_sync(FULL, q0 + lane < n && __ldg(off + q0 + lane) <= e));
  return q - 1;
}

// Digits of candidate e of the canonical order around cp (the whole warp).
__device__ __forceinline__ uint64_t candidate(const NbrDev &nb, uint64_t cp, int P, int e) {
  auto put = [](uint64_t p, int j, uint32_t t) {
    const uint32_t c = nib64(p, j);
    const uint32_t d = t < c ? t : t + 1;          // the t-th digit other than c
    return (p & ~(15ull << (4 * j))) | ((uint64_t)d << (4 * j));
  };
  if (e < nb.C1) {
    const int j = last_le(nb.off1, P, e);
    return put(cp, j, (uint32_t)(e - nb.off1[j]));
  }
  const int e2 = e - nb.C1;
  const int q = last_le(nb.off2, nb.n_pairs, e2);
  const int t = e2 - nb.off2[q];
  const int i = nb.pi[q], j = nb.pj[q];
  const int rj = nb.radix_m1[j];
  return put(put(cp, i, (uint32_t)(t / rj)), j, (uint32_t)(t % rj));
}

// What bounds it: one chain of dependent loads per candidate.  A warp's lanes
// hold one counter each (and one 32 above it) and walk its tree for c_profile and
// for the candidate together, between the rounds of the candidate's search in TS;
// no warp waits for another.
__global__ void __launch_bounds__(kScoreBlock) k_nbr_score(const SearchDev *__restrict__ srch,
                                                           StepDev *__restrict__ steps_dev,
                                                           const __grid_constant__ StepBatch<1> sb) {
  pdl_launch_dependents();
  const SearchDev &sd = srch[0];
  const StepDev &st = sb.st[0];
  const NbrDev &nb = *sd.nbr;
  const int K = sd.K, D = sd.D, L = 1 << D, P = sd.sa.P;
  const uint64_t cp = st.cprof_packed;
  const int lane = threadIdx.x & 31;
  const int warps = kScoreBlock / 32;
  const uint32_t cp_lo = (uint32_t)cp, cp_hi = (uint32_t)(cp >> 32);
  if (blockIdx.x == gridDim.x - 1) {
    // the last block publishes the step: its parameters, Delta, the prediction
    // of every counter for c_profile, the resets
    __shared__ int s_na;
    if (threadIdx.x == 0) s_na = 0;
    __syncthreads();
    if (threadIdx.x < K) {
      const uint32_t leaf = tree_leaf(sd.nodes + (size_t)threadIdx.x * L, D, cp);
      const float A = __ldg(sd.leaves + (size_t)threadIdx.x * L + leaf), dl = st.delta[threadIdx.x];
      sd.pcprof[threadIdx.x] = A;
      sd.delta[threadIdx.x] = dl;
      if (dl != 0.0f && A != 0.0f) atomicAdd(&s_na, 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      steps_dev[0] = st;
      sd.mm[0] = INT_MAX;
      sd.mm[1] = INT_MIN;
      if (st.n_out) *st.n_out = 0;
      *sd.n_active = s_na;
    }
    return;
  }
  // one warp per candidate: every lane holds the same candidate; the TS
  // search probes 32 positions per round
  const float dl0 = lane < K ? st.delta[lane] : 0.0f;
  const float dl1 = lane + 32 < K ? st.delta[lane + 32] : 0.0f;
  const uint8_t *n0 = sd.nodes + (size_t)lane * L, *n1 = n0 + (size_t)32 * L;
  const float *v0 = sd.leaves + (size_t)lane * L, *v1 = v0 + (size_t)32 * L;
  for (int e = blockIdx.x * warps + (threadIdx.x >> 5); e < nb.C; e += (gridDim.x - 1) * warps) {
    const uint64_t p = candidate(nb, cp, P, e);
    const uint32_t p_lo = (uint32_t)p, p_hi = (uint32_t)(p >> 32);
    uint32_t ord = 0xFFFFFFFFu;
    float s = 0.0f;
    if (valid_nbr(p, sd.groups, sd.sa.n_groups, sd.table)) {
      uint32_t a0 = 0, a1 = 0, b0 = 0, b1 = 0;   // nodes: c_profile's and the candidate's, of both counters
      int lev = 0;
      auto walk = [&](int n) {
        for (; n > 0 && lev < D; --n, ++lev) {
          if (dl0 != 0.0f) {
            const uint32_t x = __ldg(n0 + a0), y = __ldg(n0 + b0);
            a0 = tree_step(a0, x, cp_lo, cp_hi);
            b0 = tree_step(b0, y, p_lo, p_hi);
          }
          if (dl1 != 0.0f) {
            const uint32_t x = __ldg(n1 + a1), y = __ldg(n1 + b1);
            a1 = tree_step(a1, x, cp_lo, cp_hi);
            b1 = tree_step(b1, y, p_lo, p_hi);
          }
        }
      };
      // first ordinal a in [lo, hi] whose raw index is >= raw (TS ascending)
      const int64_t raw = raw_of(sd.sa, p);
      int64_t lo = 0, hi = sd.N;
      while (hi - lo > 32) {
        const int64_t m = lo + ((hi - lo) * (lane + 1)) / 33;
        const uint64_t probe = __ldg(sd.packed + m);
        walk(3);
        const bool below = raw_of(sd.sa, probe) < raw;
        const int c = __popc(__ballot_sync(FULL, below));
        const int64_t m_lo = __shfl_sync(FULL, m, c > 0 ? c - 1 : 0);
        const int64_t m_hi = __shfl_sync(FULL, m, c < 32 ? c : 31);
        if (c > 0) lo = m_lo + 1;
        if (c < 32) hi = m_hi;
      }
      const bool below = lo + lane < hi && raw_of(sd.sa, __ldg(sd.packed + lo + lane)) < raw;
      const int64_t a = lo + __popc(__ballot_sync(FULL, below));
      if (a < sd.N && raw_of(sd.sa, __ldg(sd.packed + a)) == raw &&
          !((__ldg(sd.eval + (a >> 5)) >> (a & 31)) & 1u)) {
        ord = (uint32_t)a;
        walk(D);
        const uint32_t first = (uint32_t)(L - 1);
        float t0 = 0.0f, t1 = 0.0f, A0 = 0.0f, A1 = 0.0f;
        if (dl0 != 0.0f) {
          A0 = __ldg(v0 + (a0 - first));
          t0 = term_n(__ldg(v0 + (b0 - first)), A0, dl0);
        }
        if (dl1 != 0.0f) {
          A1 = __ldg(v1 + (a1 - first));
          t1 = term_n(__ldg(v1 + (b1 - first)), A1, dl1);
        }
        // the terms of the active counters in ascending order, as every other
        // path sums them
        for (unsigned m = __ballot_sync(FULL, dl0 != 0.0f && A0 != 0.0f); m; m &= m - 1)
          s = __fadd_rn(s, __shfl_sync(FULL, t0, __ffs(m) - 1));
        for (unsigned m = __ballot_sync(FULL, dl1 != 0.0f && A1 != 0.0f); m; m &= m - 1)
          s = __fadd_rn(s, __shfl_sync(FULL, t1, __ffs(m) - 1));
      }
    }
    if (lane == 0) {
      nb.ord_e[e] = ord;
      nb.s_e[e] = s;
      nb.p_e[e] = p;
    }
  }
}

// Block-wide exclusive scan of one value per thread (1024 threads); returns
// the thread's exclusive prefix and writes the total to *total.
template <typename T>
__device__ __forceinline__ T block_scan(T v, T *warp_buf, T *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T inc = v;
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(FULL, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_buf[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    T w = lane < (int)(blockDim.x >> 5) ? warp_buf[lane] : (T)0;
    T winc = w;
    for (int o = 1; o < 32; o <<= 1) {
      const T y = __shfl_up_sync(FULL, winc, o);
      if (lane >= o) winc += y;
    }
    warp_buf[lane] = winc - w;
    if (lane == 31) *total = winc;
  }
  __syncthreads();
  const T ex = warp_buf[warp] + inc - v;
  __syncthreads();
  return ex;
}

__global__ void __launch_bounds__(1024) k_nbr_select(const SearchDev *__restrict__ srch,
                                                     const StepDev *__restrict__ steps_dev) {
  __shared__ uint64_t wbuf[32];
  __shared__ int ibuf[32];
  __shared__ uint64_t s_tot;
  __shared__ int s_itot;
  __shared__ float red_a[32], red_b[32];
  __shared__ int red_i[32];
  __shared__ int64_t red_r[32];
  __shared__ int s_pick;
  const SearchDev &sd = srch[0];
  const StepDev &st = steps_dev[0];
  const NbrDev &nb = *sd.nbr;
  const int C = nb.C, T = blockDim.x, t = threadIdx.x;
  const int lane = t & 31, warp = t >> 5;
  // compaction of the kept candidates, canonical order kept: thread t owns a
  // contiguous chunk of the candidates
  const int q = (C + T - 1) / T;
  const int lo = min(C, t * q), hi = min(C, lo + q);
  int cnt = 0;
  for (int e = lo; e < hi; ++e) cnt += nb.ord_e[e] != 0xFFFFFFFFu;
  const int at0 = block_scan<int>(cnt, ibuf, &s_itot);
  const int n = s_itot;
  {
    int at = at0;
    for (int e = lo; e < hi; ++e) {
      const uint32_t o = nb.ord_e[e];
      if (o == 0xFFFFFFFFu) continue;
      nb.ord[at] = o;
      nb.s[at] = nb.s_e[e];
      nb.p[at] = nb.p_e[e];
      ++at;
    }
  }
  if (t == 0) *nb.count = n;
  __syncthreads();
  if (n == 0) return;
  const int kk = min(st.k, n);
  // chunks of the compacted list
  const int q2 = (n + T - 1) / T;
  const int lo2 = min(n, t * q2), hi2 = min(n, lo2 + q2);
  // min / max
  float mn = FLT_MAX, mx = -FLT_MAX;
  for (int i = lo2; i < hi2; ++i) {
    mn = fminf(mn, nb.s[i]);
    mx = fmaxf(mx, nb.s[i]);
  }
  for (int o = 16; o; o >>= 1) {
    mn = fminf(mn, __shfl_xor_sync(FULL, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
  }
  if (lane == 0) {
    red_a[warp] = mn;
    red_b[warp] = mx;
  }
  __syncthreads();
  if (t == 0) {
    float a = FLT_MAX, b = -FLT_MAX;
    for (int w = 0; w < (T >> 5); ++w) {
      a = fminf(a, red_a[w]);
      b = fmaxf(b, red_b[w]);
    }
    red_a[0] = a;
    red_b[0] = b;
    sd.mm[0] = okey_n(a);
    sd.mm[1] = okey_n(b);
  }
  __syncthreads();
  const float smin = red_a[0], smax = red_b[0];
  const bool topk = sd.select == KTUNE_SELECT_TOPK;
  for (int i = lo2; i < hi2; ++i) nb.w[i] = topk ? 0 : weight_of(nb.s[i], smin, smax, sd.gamma);
  __syncthreads();
  for (int j = 0; j < kk; ++j) {
    if (topk) {
      // highest score, ties to the lower raw index, among those not taken
      float bs = -INFINITY;
      int64_t br = INT64_MAX;
      int bi = -1;
      for (int i = lo2; i < hi2; ++i) {
        if (nb.w[i]) continue;
        const float v = nb.s[i];
        const int64_t r = raw_of(sd.sa, nb.p[i]);
        if (bi < 0 || v > bs || (v == bs && r < br)) {
          bs = v;
          br = r;
          bi = i;
        }
      }
      for (int o = 16; o; o >>= 1) {
        const float v = __shfl_xor_sync(FULL, bs, o);
        const int64_t r = __shfl_xor_sync(FULL, br, o);
        const int i = __shfl_xor_sync(FULL, bi, o);
        if (i >= 0 && (bi < 0 || v > bs || (v == bs && r < br))) {
          bs = v;
          br = r;
          bi = i;
        }
      }
      if (lane == 0) {
        red_a[warp] = bs;
        red_r[warp] = br;
        red_i[warp] = bi;
      }
      __syncthreads();
      if (t == 0) {
        float v0 = -INFINITY;
        int64_t r0 = INT64_MAX;
        int i0 = -1;
        for (int w = 0; w < (T >> 5); ++w) {
          const int i = red_i[w];
          if (i >= 0 && (i0 < 0 || red_a[w] > v0 || (red_a[w] == v0 && red_r[w] < r0))) {
            v0 = red_a[w];
            r0 = red_r[w];
            i0 = i;
          }
        }
        s_pick = i0;
        nb.w[i0] = 1;   // taken
      }
      __syncthreads();
    } else {
      uint64_t sum = 0;
      for (int i = lo2; i < hi2; ++i) sum += nb.w[i];
      const uint64_t ex = block_scan<uint64_t>(sum, wbuf, &s_tot);
      const uint64_t W = s_tot;
      const uint64_t r = scaled_draw(philox_u64(sd.seed, sd.search_id, st.step, (uint32_t)j, 0), W);
      // the first index whose inclusive prefix exceeds r lies in the chunk
      // whose [ex, ex + sum) holds r
      if (sum && r >= ex && r < ex + sum) {
        uint64_t run = ex;
        for (int i = lo2; i < hi2; ++i) {
          run += nb.w[i];
          if (run > r) {
            s_pick = i;
            nb.w[i] = 0;
            break;
          }
        }
      }
      __syncthreads();
    }
    if (t == 0) {
      const int i = s_pick;
      const uint32_t o = nb.ord[i];
      st.out_raw[j] = raw_of(sd.sa, nb.p[i]);
      st.out_score[j] = nb.s[i];
      if (st.out_packed) st.out_packed[j] = nb.p[i];
      atomicOr(sd.eval + (o >> 5), 1u << (o & 31));
    }
    __syncthreads();
  }
  if (t == 0 && st.n_out) *st.n_out = kk;
}

// The weighted draws among at most kNbrThreads * kNbrEach candidates: a thread
// keeps its run of candidates and their weights in registers, candidates that
// are not scored with weight 0 (no draw can land on them, and the prefix sums
// are the compacted list's).  One scan serves every draw: taking a pick out
// lowers the prefixes behind it by its weight.  With the compacted list in
// memory and a scan per draw, as k_nbr_select does, a step of 2,257,920
// configurations at distance <= 2 took 48 us, now 33 (both kernels changed).
constexpr int kNbrThreads = 512, kNbrEach = 8;

__global__ void __launch_bounds__(kNbrThreads) k_nbr_draws(const SearchDev *__restrict__ srch,
                                                           const StepDev *steps_dev) {
  __shared__ uint64_t wbuf[32];
  __shared__ uint64_t s_tot;
  __shared__ uint64_t s_u[KTUNE_MAX_K];
  __shared__ uint64_t s_w[KTUNE_MAX_K];
  __shared__ int s_at[KTUNE_MAX_K];       // pick j's candidate
  __shared__ float red_a[kNbrThreads / 32], red_b[kNbrThreads / 32];
  __shared__ int red_n[kNbrThreads / 32];
  const SearchDev &sd = srch[0];
  const StepDev &st = steps_dev[0];
  const NbrDev &nb = *sd.nbr;
  const int C = nb.C, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const float gamma = sd.gamma;
  const int each = (C + kNbrThreads - 1) / kNbrThreads, lo = t * each;
  pdl_wait();                 // the candidates' scores, this step's parameters
  float s[kNbrEach];
  bool ok[kNbrEach];
  float mn = FLT_MAX, mx = -FLT_MAX;
  int n = 0;
#pragma unroll
  for (int u = 0; u < kNbrEach; ++u) {
    ok[u] = u < each && lo + u < C && __ldcg(nb.ord_e + lo + u) != 0xFFFFFFFFu;
    s[u] = ok[u] ? __ldcg(nb.s_e + lo + u) : 0.0f;
  }
#pragma unroll
  for (int u = 0; u < kNbrEach; ++u)
    if (ok[u]) {
      ++n;
      mn = fminf(mn, s[u]);
      mx = fmaxf(mx, s[u]);
    }
  const int k = st.k;
  if (t < k) s_u[t] = philox_u64(sd.seed, sd.search_id, st.step, (uint32_t)t, 0);
  for (int o = 16; o; o >>= 1) {
    mn = fminf(mn, __shfl_xor_sync(FULL, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
    n += __shfl_xor_sync(FULL, n, o);
  }
  if (lane == 0) {
    red_a[warp] = mn;
    red_b[warp] = mx;
    red_n[warp] = n;
  }
  __syncthreads();
  n = 0;
#pragma unroll
  for (int w = 0; w < kNbrThreads / 32; ++w) {
    mn = fminf(mn, red_a[w]);
    mx = fmaxf(mx, red_b[w]);
    n += red_n[w];
  }
  if (t == 0) *nb.count = n;
  if (n == 0) return;
  if (t == 0) {
    sd.mm[0] = okey_n(mn);
    sd.mm[1] = okey_n(mx);
  }
  const int kk = min(k, n);
  uint64_t w[kNbrEach], sum = 0;
#pragma unroll
  for (int u = 0; u < kNbrEach; ++u) {
    w[u] = ok[u] ? weight_of(s[u], mn, mx, gamma) : 0ull;
    sum += w[u];
  }
  uint64_t ex = block_scan<uint64_t>(sum, wbuf, &s_tot);
  uint64_t W = s_tot;
  for (int j = 0; j < kk; ++j) {
    const uint64_t r = scaled_draw(s_u[j], W);
    if (sum && r >= ex && r < ex + sum) {
      uint64_t run = ex, taken = 0;
      int at = -1;
#pragma unroll
      for (int u = 0; u < kNbrEach; ++u) {
        run += w[u];
        if (at < 0 && run > r) {
          at = u;
          taken = w[u];
          w[u] = 0;
        }
      }
      sum -= taken;
      s_at[j] = lo + at;
      s_w[j] = taken;
    }
    __syncthreads();
    W -= s_w[j];
    if (lo > s_at[j]) ex -= s_w[j];
  }
  if (t < kk) {
    const int e = s_at[t];
    const uint32_t o = __ldcg(nb.ord_e + e);
    const uint64_t p = __ldcg(nb.p_e + e);
    st.out_raw[t] = raw_of(sd.sa, p);
    st.out_score[t] = __ldcg(nb.s_e + e);
    if (st.out_packed) st.out_packed[t] = p;
    atomicOr(sd.eval + (o >> 5), 1u << (o & 31));
  }
  if (t == 0 && st.n_out) *st.n_out = kk;
}

template <typename... KArgs>
void launch_after(void (*kern)(KArgs...), int block, cudaStream_t st, KArgs... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1);
  cfg.blockDim = dim3((unsigned)block);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = st != nullptr ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace

void launch_nbr_step(const SearchDev *srch, StepDev *steps_dev, const StepBatch<1> &sb, int C, bool topk,
                     int num_sms, cudaStream_t st) {
  const int warps = kScoreBlock / 32;
  const int blocks = std::max(1, std::min((C + warps - 1) / warps, num_sms * 8));
  k_nbr_score<<<blocks + 1, kScoreBlock, 0, st>>>(srch, steps_dev, sb);   // (the last one publishes)
  // the draws in registers where the candidates fit one thread's eight; the
  // top k and larger neighbourhoods through the compacted list
  if (!topk && C <= kNbrThreads * kNbrEach) launch_after(k_nbr_draws, kNbrThreads, st, srch, (const StepDev *)steps_dev);
  else k_nbr_select<<<1, C <= 4096 ? 128 : 1024, 0, st>>>(srch, steps_dev);
}

const void *nbr_score_func() { return (const void *)k_nbr_score; }

}  // namespace ktune
