// Pipelined fused forward of the MLP counter model on Blackwell tensor cores,
// one CTA pair (a cluster of two, cta_group::2 MMAs) on two 256-row tiles in
// ping-pong.  Each CTA holds 128 rows of both tiles and half of every layer's
// output rows of the weights:
//   warp 0       streams its weight halves, layer by layer in chunks of 64
//                K-columns already laid out as the shared-memory operand,
//                through a ring with asynchronous bulk copies; a chunk serves
//                both tiles before its slot is free again;
//   warp 1       even CTA: issues the MMAs of tile x (x = 0, 1) into that
//                tile's 256 tensor-memory columns, one layer at a time; odd
//                CTA: tells the even one which of its chunks have landed;
//   warps 2..17  drain tile 0's accumulator, then tile 1's, all 16 warps on
//                one tile (64 columns of 32 rows each, the next 16 columns in
//                flight): bias + GELU + bfloat16 into the tile's activation
//                buffer (the next layer's A operand), or, after the output
//                layer, the predicted counters or the Eq. score of every
//                configuration with the minimum and maximum over the
//                unevaluated ones, and the next tile's features;
//   warp 18      shows the activations that all 16 have stored to the tensor
//                cores (a proxy fence) and tells the even CTA.
// The MMAs of one tile run during the epilogue of the other.
//
// What bounds it: the FMA pipe in the epilogue (12 paired and 4 single
// instructions for two activations, 28 cycles of the pipe; 3.6k cycles per tile
// and layer, 4.4k measured) and, tile by tile, the chain from a tile's last
// stored activation to its next accumulator (5.2k cycles: both CTAs' hand-over
// 1.8k, 16 MMAs 2.5k, completion 0.5k), which the other tile's epilogue covers
// but for 0.5k.  Tensor pipe 0.29, FMA pipe 0.59 of peak.  2.0M predictions of
// 40 counters: 0.98 ms, 0.61 PFLOP/s (1.44 ms with one CTA per tile, see below).
// The weights come from L2 at 0.65 KB per configuration: a chunk feeds 512
// rows of the pair, each CTA copying half of it.
// Measured and left (2.0M predictions):
//  - one CTA per tile, every 128 rows streaming the whole network (2.5 KB per
//    configuration, 1.0 ms of L2 traffic on its own): 1.44 ms;
//  - all weights resident, the activations in a small ring, one tile at a time:
//    2.05 ms (a proxy fence and an arrival per 8 columns, and nothing to do
//    while a layer's last columns are multiplied);
//  - eight epilogue warps per tile: 1.19 ms (both tiles fall into step and wait
//    for their chains together; all 16 on one tile keep them half a period apart);
//  - proxy fences in the epilogue warps: 1.12 ms.
// Roundings: the products accumulate in FP32 in tensor memory in steps of 16
// columns of K; bias, GELU (its erf from a published rational approximation,
// gelu2_bf) and the output scale in FP32; activations rounded to bfloat16; the
// score sums its counters in ascending order, each term one float32 operation
// sequence.  Every wait is bounded: on time-out the kernel records
// KTUNE_ETIMEOUT, drains its own copies and MMAs (bounded) and returns after a
// cluster barrier.
#include <float.h>
#include <limits.h>
#include <stddef.h>

#include <algorithm>

#include "device_common.cuh"
#include "internal.h"
#include "mlp_epi.cuh"
#include "tc.cuh"

namespace ktune {

namespace {

constexpr uint64_t kPairWait = 1000000000ull;             // 1 s: the drain waits after a time-out
constexpr int kPairEpiWarps = 16;                         // 4 per tensor-memory lane quarter
constexpr int kPairThreads = 96 + 32 * kPairEpiWarps;
constexpr int kActBytes = 128 * kMlpHidden * 2;           // one CTA's rows of one tile (64 KB)
constexpr int kSlotBytes = kMlpHidden / 2 * kMlpChunkK * 2;   // half the rows of a weight chunk (16 KB)
constexpr int kSlots = 4;                                 // a hidden layer's chunks
constexpr int kMaxGroups8 = kMlpMaxF / 8;                 // 8-column feature groups
// (parameter, group) pairs: a parameter's one-hot columns reach into a new
// group at most once per group, its u column lies in one; a group has at most
// eight of them (each covers at least one of its columns)
constexpr int kMaxParts = 2 * KTUNE_MAX_PARAMS + kMaxGroups8;
constexpr unsigned FULL = 0xffffffffu;

// What follows the activations and the ring in shared memory.
struct alignas(16) PairShared {
  uint64_t full[kSlots], empty[kSlots], act[2], act_ready[2], acc_full[2], drain, never;
  uint32_t tmem_base;
  alignas(16) float bias[3 * kMlpHidden + 64];
  alignas(16) float rng[KTUNE_MAX_COUNTERS];
  float2 react[kMlpMaxShare][KTUNE_MAX_COUNTERS];           // (pc(c_profile), Delta) of the active counters
  uint8_t react_c[kMlpMaxShare][KTUNE_MAX_COUNTERS];        // their counter slots, ascending
  int n_react[kMlpMaxShare];
  // a feature group's pairs, in one or two fours: offset in part << 8 | 4 x parameter
  alignas(16) uint32_t quad[kMaxGroups8][8];
  uint8_t quads[kMaxGroups8];
  uint8_t part_j[kMaxParts], part_g[kMaxParts];           // a pair's parameter and group
  int parts;
  alignas(16) uint4 part[kMaxParts + 1][16];              // 8 columns of bfloat16 by digit; the last 0
};
static_assert(offsetof(PairShared, bias) % 16 == 0, "bias is read as float4");
constexpr int kPairSmem = 2 * kActBytes + kSlots * kSlotBytes + (int)sizeof(PairShared);
static_assert(kPairSmem <= 227 * 1024, "shared memory of one CTA");
// the MMAs of a layer wait for all of its chunks, and only they free the ring's slots
static_assert((kMlpMaxF + kMlpChunkK - 1) / kMlpChunkK <= kSlots && kMlpHidden / kMlpChunkK <= kSlots,
              "a layer's chunks fit the ring");
static_assert(mlp_n4(KTUNE_MAX_COUNTERS) / 2 * kMlpHidden * 2 <= kSlotBytes, "the output layer's half is one slot");
static_assert(kMaxGroups8 <= 32, "a lane per feature group");

__device__ __forceinline__ void ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15])
      : "r"(taddr));
}
// The registers pass through the wait so that nothing reads them before it.
__device__ __forceinline__ void ld16_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                 "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]),
                 "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :: "memory");
}
__device__ __forceinline__ void ld1(uint32_t taddr, uint32_t &r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr));
}
__device__ __forceinline__ void ld8_wait(uint32_t (&r)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                 "+r"(r[7]) :: "memory");
}

// Eight feature columns [8 G, 8 G + 8) of a configuration: the group's
// parameters each contribute 16 bytes, by digit (a one at its place, or its
// u); four independent look-ups at a time.
__device__ __forceinline__ uint4 feature8(const PairShared &sh, int G, uint64_t pk) {
  uint4 v = make_uint4(0, 0, 0, 0);
  const uint8_t *tab = reinterpret_cast<const uint8_t *>(sh.part);
  auto four = [&](const uint4 &m) {
    auto get = [&](uint32_t e) {
      return *reinterpret_cast<const uint4 *>(tab + (e >> 8) + (((uint32_t)(pk >> (e & 63u)) & 15u) << 4));
    };
    const uint4 a = get(m.x), b = get(m.y), c = get(m.z), d = get(m.w);
    v.x |= a.x | b.x | c.x | d.x;
    v.y |= a.y | b.y | c.y | d.y;
    v.z |= a.z | b.z | c.z | d.z;
    v.w |= a.w | b.w | c.w | d.w;
  };
  four(*reinterpret_cast<const uint4 *>(&sh.quad[G][0]));
  if (sh.quads[G] > 1) four(*reinterpret_cast<const uint4 *>(&sh.quad[G][4]));
  return v;
}

template <int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
    k_mlp_pair(const MlpDev md, const uint64_t *__restrict__ packed, int64_t n,
               float *__restrict__ out, const __grid_constant__ MlpTargets tg, int *status) {
  extern __shared__ __align__(1024) uint8_t sm[];
  uint8_t *ring = sm + 2 * kActBytes;
  PairShared &sh = *reinterpret_cast<PairShared *>(ring + kSlots * kSlotBytes);
  const int F = md.F, N4 = mlp_n4(md.K);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = tc::cluster_rank();
  const int64_t n_tiles = (n + 255) / 256;
  const int64_t cluster = blockIdx.x >> 1, n_clusters = gridDim.x >> 1;
  // this pair's tiles: cluster, cluster + n_clusters, ...; two at a time
  const int64_t my_tiles = (n_tiles - 1 - cluster) / n_clusters + 1;   // the grid has no idle pair

  if (warp == 1) tc::tmem_alloc2(&sh.tmem_base, 512);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kSlots; ++s) {
      tc::mbar_init(&sh.full[s], rank == 0 ? 2 : 1);   // even CTA: its own copy and its peer's
      tc::mbar_init(&sh.empty[s], 1);
    }
    for (int x = 0; x < 2; ++x) {
      tc::mbar_init(&sh.act[x], kPairEpiWarps);
      tc::mbar_init(&sh.act_ready[x], 2);              // both CTAs' activations (the even CTA's is used)
      tc::mbar_init(&sh.acc_full[x], 1);
    }
    tc::mbar_init(&sh.drain, 1);
    tc::mbar_init(&sh.never, 1);   // no thread ever arrives here (md.stall)
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < 3 * kMlpHidden; i += blockDim.x) sh.bias[i] = md.b[i >> 8][i & 255];
  for (int i = threadIdx.x; i < md.Kp; i += blockDim.x) sh.bias[3 * kMlpHidden + i] = md.b[3][i];
  for (int i = threadIdx.x; i < md.K; i += blockDim.x) sh.rng[i] = md.range[i];
  const int my_off = warp == 0 && lane <= md.P ? md.off[lane] : 0;
  if (warp == 0) {   // the (parameter, group) pairs, by group: lane G lists group G's
    uint32_t in = 0;
    const int u0 = __shfl_sync(FULL, my_off, md.P);
    for (int j = 0; j < md.P; ++j) {
      const int o0 = __shfl_sync(FULL, my_off, j), o1 = __shfl_sync(FULL, my_off, j + 1);
      const int u = u0 + j - 8 * lane;
      if ((o0 < 8 * lane + 8 && o1 > 8 * lane) || (u >= 0 && u < 8)) in |= 1u << j;
    }
    if (lane >= F / 8) in = 0;
    int incl = __popc(in);
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) sh.parts = incl;
    sh.quads[lane] = (uint8_t)((__popc(in) + 3) / 4);
    for (int e = 0; e < 8; ++e) sh.quad[lane][e] = kMaxParts * 256u << 8;   // zeros
    int e = 0;
    for (int p = incl - __popc(in); in; in &= in - 1, ++p, ++e) {
      const int j = __ffs(in) - 1;
      sh.part_j[p] = (uint8_t)j;
      sh.part_g[p] = (uint8_t)lane;
      sh.quad[lane][e] = ((uint32_t)p * 256u << 8) | (uint32_t)(4 * j);
    }
  }
  if (threadIdx.x < 16) sh.part[kMaxParts][threadIdx.x] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  for (int i = threadIdx.x; i < sh.parts * 16; i += blockDim.x) {
    const int p = i >> 4, dg = i & 15, j = sh.part_j[p], G = sh.part_g[p];
    uint16_t v[8];
    for (int e = 0; e < 8; ++e) {
      const int c = 8 * G + e;
      v[e] = c == md.off[md.P] + j ? md.utab[j * 16 + dg]
             : c == md.off[j] + dg && dg < md.off[j + 1] - md.off[j] ? (uint16_t)0x3F80 : (uint16_t)0;
    }
    sh.part[p][dg] = make_uint4(v[0] | ((uint32_t)v[1] << 16), v[2] | ((uint32_t)v[3] << 16),
                                v[4] | ((uint32_t)v[5] << 16), v[6] | ((uint32_t)v[7] << 16));
  }
  if (MODE == 1 && warp >= 2)
    // the counters each search reacts to, in ascending order
    for (int q = warp - 2; q < tg.S; q += kPairEpiWarps) {
      int cnt = 0;
      for (int c0 = 0; c0 < md.K; c0 += 32) {
        const int c = c0 + lane;
        const float A = c < md.K ? tg.pcprof[q][c] : 0.0f, dl = c < md.K ? tg.delta[q][c] : 0.0f;
        const bool on = dl != 0.0f && A != 0.0f;
        const unsigned b = __ballot_sync(FULL, on);
        if (on) {
          const int a = cnt + __popc(b & ((1u << lane) - 1u));
          sh.react[q][a] = make_float2(A, dl);
          sh.react_c[q][a] = (uint8_t)c;
        }
        cnt += __popc(b);
      }
      if (lane == 0) sh.n_react[q] = cnt;
    }
  tc::fence_before();
  __syncthreads();
  tc::cluster_sync();
  tc::fence_after();
  const uint32_t tmem = sh.tmem_base;

  if (warp == 0) {
    // ---- producer: this CTA's half of every chunk, in the order of use ---------------
    if (lane == 0) {
      // md.stall: a wait that runs out before any copy is issued
      bool ok = !md.stall || tc::mbar_wait(&sh.never, 0u, md.wait_ns);
      uint32_t use = 0, st = 0, ph = 1u;
      const uint32_t ring_a = tc::smem_u32(ring);
      for (int64_t j = 0; j < my_tiles && ok; j += 2)
        for (int l = 0; l < 4 && ok; ++l) {
          const int Kl = l == 0 ? F : kMlpHidden, Nl = l == 3 ? N4 : kMlpHidden;
          const uint8_t *src = md.wc + md.wc_off[l];
          const int step = mlp_chunk_k(l);
          for (int k0 = 0; k0 < Kl; k0 += step) {
            const int kc = min(step, Kl - k0);
            if (!tc::mbar_wait_idle(&sh.empty[st], ph, md.wait_ns)) {
              ok = false;
              break;
            }
            const uint32_t bytes = (uint32_t)(Nl * kc);       // Nl / 2 rows of kc bfloat16
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                             tc::smem_u32(&sh.full[st])), "r"(bytes) : "memory");
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    ring_a + st * (uint32_t)kSlotBytes),
                "l"(src + (size_t)k0 * Nl * 2 + rank * bytes), "r"(bytes),
                "r"(tc::smem_u32(&sh.full[st])) : "memory");
            ++use;
            if (++st == (uint32_t)kSlots) {
              st = 0;
              ph ^= 1u;
            }
          }
        }
      if (!ok) atomicExch(status, KTUNE_ETIMEOUT);
      // copies still in flight land before the CTA leaves
      for (uint32_t u = use > (uint32_t)kSlots ? use - kSlots : 0u; u < use; ++u)
        tc::mbar_wait(&sh.full[u % kSlots], (u / kSlots) & 1u, kPairWait);
    }
  } else if (warp == 1 && rank == 1) {
    if (lane == 0) {
      // ---- the odd CTA's chunks that have landed, told to the even one ---------------
      bool ok = true;
      uint32_t st = 0, ph = 0;
      const int chunks = (F + kMlpChunkK - 1) / kMlpChunkK + 2 * (kMlpHidden / kMlpChunkK) + 1;
      const uint32_t peer0 = tc::map_rank(tc::smem_u32(&sh.full[0]), 0);
      for (int64_t j = 0; j < my_tiles && ok; j += 2)
        for (int c = 0; c < chunks; ++c) {
          if (!tc::mbar_wait_idle(&sh.full[st], ph, md.wait_ns)) {
            ok = false;
            break;
          }
          tc::mbar_arrive_cluster(peer0 + st * 8u);
          if (++st == (uint32_t)kSlots) {
            st = 0;
            ph ^= 1u;
          }
        }
      if (!ok) atomicExch(status, KTUNE_ETIMEOUT);
    }
  } else if (warp == 1) {
    // ---- MMA issuer: the whole warp runs the loop, so that descriptors and
    // counters live in uniform registers, and one lane issues -------------------------
    const bool lead = tc::elect_one();
    // md.stall: a wait that runs out before any MMA is issued
    bool ok = !md.stall || __all_sync(FULL, tc::mbar_wait(&sh.never, 0u, md.wait_ns));
    uint32_t st0 = 0, ph0 = 0, aph = 0;              // slot and phase of the layer's first chunk
    const uint32_t act_a = tc::smem_u32(sm), ring_a = tc::smem_u32(ring);
    for (int64_t j = 0; j < my_tiles && ok; j += 2) {
      const int nx = j + 1 < my_tiles ? 2 : 1;
      for (int l = 0; l < 4 && ok; ++l) {
        const int Kl = l == 0 ? F : kMlpHidden;
        const uint32_t idesc = tc::idesc_bf16(256, l == 3 ? N4 : kMlpHidden);
        const uint32_t a_hi = tc::sdesc_hi((uint32_t)Kl * 16u);
        const int step = mlp_chunk_k(l), chunks = (Kl + step - 1) / step;
        // the layer's weights first: both halves have usually landed by now, and
        // nothing is left to wait for between its MMAs
        uint32_t st = st0, ph = ph0;
        for (int c = 0; c < chunks && ok; ++c) {
          ok = __all_sync(FULL, tc::mbar_wait(&sh.full[st], ph, md.wait_ns));
          if (++st == (uint32_t)kSlots) {
            st = 0;
            ph ^= 1u;
          }
        }
        const uint32_t st_next = st, ph_next = ph;
        for (int x = 0; x < nx && ok; ++x) {
          ok = __all_sync(FULL, tc::mbar_wait(&sh.act_ready[x], (aph >> x) & 1u, md.wait_ns));
          if (!ok) break;
          aph ^= 1u << x;
          tc::fence_after();
          const uint32_t d = tmem + (uint32_t)x * 256u;
          uint32_t a_lo = tc::sdesc_lo(act_a + (uint32_t)x * kActBytes, 128);
          uint32_t acc = 0;
          st = st0;
          for (int left = Kl; left > 0; left -= step) {
            const int kc = min(step, left);
            uint32_t b_lo = tc::sdesc_lo(ring_a + st * (uint32_t)kSlotBytes, 128);
            const uint32_t b_hi = tc::sdesc_hi((uint32_t)kc * 16u);
            for (int k = 0; k < kc; k += kMlpChunkK) {
              if (lead)
#pragma unroll
                for (int q = 0; q < kMlpChunkK; q += 16)   // 128 bytes per 8 columns: 16 units of 16 bytes
                  if (k + q < kc)
                    tc::mma_bf16_pair(d, tc::sdesc_of(a_lo + q, a_hi), tc::sdesc_of(b_lo + q, b_hi), idesc,
                                      q ? 1u : acc);
              acc = 1u;
              a_lo += kMlpChunkK;
              b_lo += kMlpChunkK;
            }
            if (lead && x == nx - 1) tc::mma_commit_pair(&sh.empty[st], 3);
            if (++st == (uint32_t)kSlots) st = 0;
          }
          if (ok && lead) tc::mma_commit_pair(&sh.acc_full[x], 3);
        }
        st0 = st_next;
        ph0 = ph_next;
      }
    }
    // every MMA issued has completed before tensor memory is released
    if (lead) {
      if (!ok) atomicExch(status, KTUNE_ETIMEOUT);
      tc::mma_commit_pair(&sh.drain, 1);
      tc::mbar_wait(&sh.drain, 0u, kPairWait);
    }
  } else if (warp == 2 + kPairEpiWarps) {
    // ---- this CTA's activations, shown to the tensor cores and told to the even CTA ----
    if (lane == 0) {
      bool ok = true;
      uint32_t aph = 0;
      const uint32_t ready0 = tc::map_rank(tc::smem_u32(&sh.act_ready[0]), 0);
      for (int64_t j = 0; j < my_tiles && ok; j += 2)
        for (int l = 0; l < 4 && ok; ++l)
          for (int x = 0; x < 2 && j + x < my_tiles; ++x) {
            ok = tc::mbar_wait(&sh.act[x], (aph >> x) & 1u, md.wait_ns);
            if (!ok) break;
            aph ^= 1u << x;
            tc::fence_async_smem();
            tc::mbar_arrive_cluster(ready0 + (uint32_t)x * 8u);
          }
      if (!ok) atomicExch(status, KTUNE_ETIMEOUT);
    }
  } else {
    // ---- epilogue ----------------------------------------------------------------------
    const int quarter = warp & 3;             // tensor-memory lanes this warp may read
    const int g = (warp - 2) >> 2;            // hidden columns [64 g, 64 g + 64)
    const int row = quarter * 32 + lane;      // row of this CTA's half tile
    const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
    bool ok = true;
    uint32_t aph = 0u;                        // bit x: phase of acc_full[x]
    float s_mn[2] = {INFINITY, INFINITY}, s_mx[2] = {-INFINITY, -INFINITY};
    auto wait_acc = [&](int x) {
      ok = __all_sync(FULL, tc::mbar_wait(&sh.acc_full[x], (aph >> x) & 1u, md.wait_ns));
      aph ^= 1u << x;
      tc::fence_after();
    };
    // this warp's part of tile x's next input is in place, its accumulator read.
    // The proxy fence that shows the stores to the tensor cores follows once, in
    // the thread that has waited for all 16 warps: it takes about 1,000 cycles
    // and would hold up every warp here.
    auto arrive = [&](int x) {
      tc::fence_before();
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(&sh.act[x])) : "memory");
    };
    auto row_of = [&](int64_t j) -> int64_t {
      return (cluster + j * n_clusters) * 256 + (int64_t)rank * 128 + row;
    };
    auto features = [&](int x, uint64_t pk, bool live) {
      for (int G = g; G < F / 8; G += 8) {      // two groups' look-ups in flight
        const bool two = G + 4 < F / 8;
        const uint4 zero = make_uint4(0, 0, 0, 0);
        const uint4 v0 = live ? feature8(sh, G, pk) : zero;
        const uint4 v1 = live && two ? feature8(sh, G + 4, pk) : zero;
        *reinterpret_cast<uint4 *>(sm + x * kActBytes + tc::core_off(row, 8 * G, F)) = v0;
        if (two) *reinterpret_cast<uint4 *>(sm + x * kActBytes + tc::core_off(row, 8 * (G + 4), F)) = v1;
      }
      arrive(x);
    };
    for (int x = 0; x < 2 && x < my_tiles; ++x) {
      const int64_t i = row_of(x);
      features(x, i < n ? packed[i] : 0ull, i < n);
    }
    for (int64_t j = 0; j < my_tiles && ok; j += 2) {
      const int nx = j + 1 < my_tiles ? 2 : 1;
      // what the end of this pair of tiles needs from memory, in flight meanwhile
      uint64_t pk_next[2] = {0ull, 0ull};
      uint32_t ev[2][2] = {{0u, 0u}, {0u, 0u}};
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int64_t i = row_of(j + x), i_next = row_of(j + 2 + x);
        if (j + 2 + x < my_tiles && i_next < n) pk_next[x] = packed[i_next];
        if (MODE == 1 && x < nx && i < n) {
          if (g < tg.S) ev[x][0] = tg.eval[g][i >> 5];
          if (g + 4 < tg.S) ev[x][1] = tg.eval[g + 4][i >> 5];
        }
      }
      for (int l = 0; l < 3 && ok; ++l)
        for (int x = 0; x < nx; ++x) {
          wait_acc(x);
          if (!ok) break;
          const uint32_t d = tmem + (uint32_t)x * 256u + lanes + 64u * g;
          const float *bias = sh.bias + l * kMlpHidden + 64 * g;
          uint8_t *H = sm + x * kActBytes + tc::core_off(row, 64 * g, kMlpHidden);
          uint32_t ra[16], rb[16];
          auto drain16 = [&](const uint32_t (&r)[16], int c) {
#pragma unroll
            for (int e = 0; e < 16; e += 8) {
              const float4 b0 = *reinterpret_cast<const float4 *>(bias + 16 * c + e);
              const float4 b1 = *reinterpret_cast<const float4 *>(bias + 16 * c + e + 4);
              uint4 q;
              q.x = gelu2_bf(__uint_as_float(r[e]), b0.x, __uint_as_float(r[e + 1]), b0.y);
              q.y = gelu2_bf(__uint_as_float(r[e + 2]), b0.z, __uint_as_float(r[e + 3]), b0.w);
              q.z = gelu2_bf(__uint_as_float(r[e + 4]), b1.x, __uint_as_float(r[e + 5]), b1.y);
              q.w = gelu2_bf(__uint_as_float(r[e + 6]), b1.z, __uint_as_float(r[e + 7]), b1.w);
              *reinterpret_cast<uint4 *>(H + (16 * c + e) * 16) = q;   // 128 bytes per 8 columns
            }
          };
          ld16(d, ra);
          ld16_wait(ra);
          ld16(d + 16u, rb);
          drain16(ra, 0);
          ld16_wait(rb);
          ld16(d + 32u, ra);
          drain16(rb, 1);
          ld16_wait(ra);
          ld16(d + 48u, rb);
          drain16(ra, 2);
          ld16_wait(rb);
          drain16(rb, 3);
          arrive(x);
        }
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (x >= nx || !ok) break;
        const int64_t i = row_of(j + x), i_next = row_of(j + 2 + x);
        const bool more = j + 2 + x < my_tiles;
        wait_acc(x);
        if (!ok) break;
        const uint32_t d = tmem + (uint32_t)x * 256u + lanes;
        const float *b4 = sh.bias + 3 * kMlpHidden;
        if (MODE == 0) {
          // predicted counters, 16 per column group
          if (16 * g < md.K) {
            float v[16];
            tc::tmem_ld16(d + 16 * g, v);
            const int left = min(16, md.K - 16 * g);
#pragma unroll
            for (int e = 0; e < 16; e += 4) {
              const float4 b = *reinterpret_cast<const float4 *>(b4 + 16 * g + e);
              const float4 r = *reinterpret_cast<const float4 *>(sh.rng + 16 * g + e);
              v[e] = __fmul_rn(__fadd_rn(v[e], b.x), r.x);
              v[e + 1] = __fmul_rn(__fadd_rn(v[e + 1], b.y), r.y);
              v[e + 2] = __fmul_rn(__fadd_rn(v[e + 2], b.z), r.z);
              v[e + 3] = __fmul_rn(__fadd_rn(v[e + 3], b.w), r.w);
            }
            if (i < n) {
              float *o = out + (size_t)i * md.K + 16 * g;
              if ((md.K & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
#pragma unroll
                for (int e = 0; e < 16; e += 4)
                  if (e < left)
                    *reinterpret_cast<float4 *>(o + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
              } else {
#pragma unroll
                for (int e = 0; e < 16; ++e)
                  if (e < left) o[e] = v[e];
              }
            }
          }
        } else {
          // Eq. score for the searches q = g and g + 4, over their active counters in
          // ascending order (a counter without a reaction adds +0: left out)
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int q = g + 4 * u;
            if (q >= tg.S) break;
            const int na = sh.n_react[q];
            float s = 0.0f;
            for (int a0 = 0; a0 < na; a0 += 8) {      // eight independent terms at a time
              uint32_t v[8];
              float term[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) ld1(d + sh.react_c[q][min(a0 + e, na - 1)], v[e]);
              ld8_wait(v);
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                const int at = min(a0 + e, na - 1), c = sh.react_c[q][at];
                const float2 ad = sh.react[q][at];
                const float a = __fmul_rn(__fadd_rn(__uint_as_float(v[e]), b4[c]), sh.rng[c]);
                const float den = __fadd_rn(a, ad.x);
                const float t = __fmul_rn(ad.y, __fdiv_rn(__fsub_rn(a, ad.x), den));
                term[e] = a != 0.0f && den != 0.0f ? t : 0.0f;
              }
#pragma unroll
              for (int e = 0; e < 8; ++e)
                if (a0 + e < na) s = __fadd_rn(s, term[e]);
            }
            if (i < n) {
              tg.s[q][i] = s;
              if (!((ev[x][u] >> (i & 31)) & 1u)) {
                s_mn[u] = fminf(s_mn[u], s);
                s_mx[u] = fmaxf(s_mx[u], s);
              }
            }
          }
        }
        if (more) features(x, pk_next[x], i_next < n);
      }
    }
    if (!ok) {
      if (lane == 0) atomicExch(status, KTUNE_ETIMEOUT);
    } else if (MODE == 1) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int q = g + 4 * u;
        if (q >= tg.S) break;
        float mn = s_mn[u], mx = s_mx[u];
        for (int o = 16; o; o >>= 1) {
          mn = fminf(mn, __shfl_xor_sync(FULL, mn, o));
          mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
        }
        if (lane == 0 && mn <= mx) {
          atomicMin(tg.mm[q], okey_p(mn));
          atomicMax(tg.mm[q] + 1, okey_p(mx));
        }
      }
    }
  }
  // neither CTA leaves while the other may still reach its shared or tensor memory
  tc::fence_before();
  __syncthreads();
  tc::cluster_sync();
  if (warp == 1) tc::tmem_dealloc2(tmem, 512);
}

// The four layers' bf16 weights (whole-layer operand layout) into the chunked one:
// chunk c of a layer holds columns [64 c, 64 c + kc) (the output layer: all 256)
// of every output row as core matrices with KC = kc, so each CTA's half of the rows is contiguous.
// One thread moves 8 consecutive columns; the output layer's rows are padded
// with zeros to a multiple of 32.
struct PackArgs {
  const uint16_t *w[4];
  int rows[4], padded[4], cols[4];
  uint32_t dst[4];
};
__global__ void k_pack_wc(const __grid_constant__ PackArgs pa, uint8_t *__restrict__ dst) {
  const int l = blockIdx.y;
  const int Kl = pa.cols[l], Nl = pa.padded[l], per_row = Kl >> 3;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= Nl * per_row) return;
  const int r = p / per_row, k = (p - r * per_row) * 8;
  const int step = mlp_chunk_k(l), c = k / step, kk = k - c * step;
  const int kc = min(step, Kl - c * step);
  const uint4 v = r < pa.rows[l] ? *reinterpret_cast<const uint4 *>(pa.w[l] + (tc::core_off(r, k, Kl) >> 1))
                                 : make_uint4(0, 0, 0, 0);
  *reinterpret_cast<uint4 *>(dst + pa.dst[l] + (size_t)c * Nl * step * 2 + tc::core_off(r, kk, kc)) = v;
}

}  // namespace

void mlp_pair_set_attrs() {
  cudaFuncSetAttribute(k_mlp_pair<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem);
  cudaFuncSetAttribute(k_mlp_pair<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem);
}

void launch_pack_wc(const uint16_t *const w[4], int F, int K, int Kp, const uint32_t off[4], uint8_t *dst,
                    cudaStream_t st) {
  PackArgs pa{};
  for (int l = 0; l < 4; ++l) {
    pa.w[l] = w[l];
    pa.rows[l] = l == 3 ? Kp : kMlpHidden;
    pa.padded[l] = l == 3 ? mlp_n4(K) : kMlpHidden;
    pa.cols[l] = l == 0 ? F : kMlpHidden;
    pa.dst[l] = off[l];
  }
  k_pack_wc<<<dim3((kMlpHidden * kMlpHidden / 8 + 255) / 256, 4), 256, 0, st>>>(pa, dst);
}

// mode 0: predicted counters of n configurations into out; mode 1: scores for
// the searches of tg.  At most max_ctas CTAs (always whole pairs).
void launch_mlp_pair(int mode, const MlpDev &md, const uint64_t *packed, int64_t n, float *out,
                     const MlpTargets &tg, int *status, int max_ctas, cudaStream_t st) {
  const int64_t tiles = (n + 255) / 256;
  if (tiles == 0) return;
  const int64_t cap = max_ctas > 1 ? max_ctas / 2 : 1;
  const unsigned grid = 2u * (unsigned)std::min<int64_t>(tiles, cap);
  if (mode == 0) k_mlp_pair<0><<<grid, kPairThreads, kPairSmem, st>>>(md, packed, n, out, tg, status);
  else k_mlp_pair<1><<<grid, kPairThreads, kPairSmem, st>>>(md, packed, n, out, tg, status);
}

}  // namespace ktune
