// One training step of the MLP counter model in three launches.
//
//   k_train_rows   everything that is independent per row -- features, the
//                  three hidden layers, the output layer with the loss and its
//                  gradient, and the three backward layers -- for 128 rows per
//                  cluster of four CTAs.  CTA r computes columns [64 r, 64 r + 64)
//                  of every hidden layer (tcgen05, M = 128, N = 64), stores its
//                  bfloat16 activations into its block of the operand buffer and
//                  sends the block to the other three by bulk copies between
//                  their shared memories, each counted in by an mbarrier of its
//                  reader (no cluster barrier between layers); pre-activations
//                  stay in tensor memory as accumulators (z = accumulator + bias
//                  again in the backward pass), so no layer reads or writes
//                  memory but for the transposes that the weight gradients need;
//   k_train_wgrad  the four weight gradients, whose reduction runs over the
//                  batch, split over up to 64 slices of rows, each slice's tile
//                  into a workspace, and the bias gradients' row-block sums;
//   k_train_update the slices summed in a fixed order, and Adam.
// What bounds it: latency.  The step's arithmetic is 0.4 GFLOP x 9 (about 2 us of
// tensor work at 4,096 rows); k_train_rows is a chain of seven layers, each an
// MMA, an epilogue of erff / expf and an exchange of blocks.  4,096 rows (128
// CTAs): k_train_rows 36 us, k_train_wgrad 18, k_train_update 6; the update of
// one step and the rows of the next do not overlap (the weights), the other two
// launches are scheduled while their predecessor drains (82 -> 77 us per step,
// 16 steps of 4,096 rows; as 38 launches, one GEMM per layer and direction,
// transposes, sums and one Adam per tensor, a step took 299 us).
// Every wait is bounded: on time-out the kernels record KTUNE_ETIMEOUT, wait once
// more (bounded) for the copies and MMAs in flight and go on to their end with
// whatever was computed.
#include <float.h>
#include <limits.h>

#include <algorithm>

#include "device_common.cuh"
#include "internal.h"
#include "mlp_epi.cuh"
#include "tc.cuh"

namespace ktune {

namespace {

constexpr uint64_t kTrainWait = 1000000000ull;   // 1 s per tensor-core wait
constexpr int kRows = 128;                       // rows per cluster
constexpr int kSplitN = 4;                       // CTAs per cluster
constexpr int kCols = kMlpHidden / kSplitN;      // hidden columns per CTA
constexpr int kRowThreads = 512;
constexpr int kActBuf = kRows * kMlpHidden * 2;  // 64 KB
constexpr int kWBuf = kCols * kMlpHidden * 2;    // 32 KB: 64 x 256 (or K x 256 of the output layer)
constexpr int kRowSmem = 2 * kActBuf + 2 * kWBuf;
// tensor-memory columns: the hidden layers' accumulators, the output layer's,
// a backward layer's, erf(z / sqrt 2) of the hidden layers
constexpr uint32_t kOutCol = 3 * kCols, kGradCol = 4 * kCols, kErfCol = 5 * kCols;

// GELU and its derivative from z and erf(z / sqrt 2), which both need.
__device__ __forceinline__ float gelu_f(float z, float erf) { return 0.5f * z * (1.0f + erf); }
__device__ __forceinline__ float gelu_grad_f(float z, float erf) {
  return 0.5f * (1.0f + erf) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

// 32 lanes x 16 columns into tensor memory; complete after the wait.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]),
      "f"(v[9]), "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld1(uint32_t taddr, float &v) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=f"(v) : "r"(taddr));
}

// Bulk copies with completion on an mbarrier: global to this CTA, and this CTA's
// shared memory to another CTA of the cluster (dst and bar mapped there).
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint64_t *bar) {
  const uint32_t b = tc::smem_u32(bar);
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(b) : "memory");
}
__device__ __forceinline__ void bulk_s2c(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "r"(src), "r"(bytes), "r"(bar) : "memory");
}

__global__ void __cluster_dims__(kSplitN, 1, 1) __launch_bounds__(kRowThreads, 1)
    k_train_rows(const __grid_constant__ TrainDev td) {
  extern __shared__ __align__(1024) uint8_t sm[];
  // completion of MMAs; weights in buffer s; the other CTAs' activations (exchanges in
  // turn); the other CTAs are done with the output layer's input
  __shared__ uint64_t mma, w_full[2], a_full[2], freed;
  __shared__ uint32_t tmem_base;
  __shared__ float sh_b[3][kCols], sh_b4[KTUNE_MAX_COUNTERS];
  // a feature column: 4 x parameter (its shift), | 64 for u, 128 for padding; its digit
  __shared__ uint8_t sh_col[kMlpMaxF], sh_dig[kMlpMaxF];
  __shared__ uint16_t sh_utab[KTUNE_MAX_PARAMS * 16];
  __shared__ int sh_off[KTUNE_MAX_PARAMS + 1];
  const uint32_t act0 = tc::smem_u32(sm), wb0 = act0 + 2u * kActBuf;
  const int F = td.F, K = td.K, Kp = td.Kp, B = td.B, H = kMlpHidden;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)tc::cluster_rank(), n0 = rank * kCols;
  const int row = (warp & 3) * 32 + lane, part = warp >> 2, chunk = 16 * part;   // this thread's row and columns
  const int b = (int)(blockIdx.x / kSplitN) * kRows + row;                       // its batch row
  const bool live = b < B;
  bool ok = true;
  pdl_launch_dependents();

  if (threadIdx.x == 0) {
    tc::mbar_init(&mma, 1);
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(&w_full[s], 1);
      tc::mbar_init(&a_full[s], 1);
    }
    tc::mbar_init(&freed, kSplitN - 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    // weights of the first two layers on their way (operand layout: 64 rows are contiguous)
    bulk_g2s(wb0, td.w[0] + (size_t)n0 * F, (uint32_t)(kCols * F * 2), &w_full[0]);
    bulk_g2s(wb0 + kWBuf, td.w[1] + (size_t)n0 * H, (uint32_t)(kCols * H * 2), &w_full[1]);
  }
  if (warp == 1) tc::tmem_alloc(&tmem_base, 512);
  const int src = live ? td.idx[b] : 0;
  const uint64_t pk = live ? td.data[src] : 0ull;
  for (int i = threadIdx.x; i < 3 * kCols; i += blockDim.x) sh_b[i / kCols][i % kCols] = td.b[i / kCols][n0 + i % kCols];
  for (int i = threadIdx.x; i < Kp; i += blockDim.x) sh_b4[i] = td.b[3][i];
  for (int i = threadIdx.x; i <= td.P; i += blockDim.x) sh_off[i] = td.off[i];
  for (int i = threadIdx.x; i < td.P * 16; i += blockDim.x) sh_utab[i] = td.utab[i];
  __syncthreads();
  for (int c = threadIdx.x; c < F; c += blockDim.x) {
    int j = 0;
    while (j + 1 < td.P && sh_off[j + 1] <= c) ++j;
    const int u = c - sh_off[td.P];
    sh_col[c] = (uint8_t)(u >= td.P ? 128 : u >= 0 ? 64 | 4 * u : 4 * j);
    sh_dig[c] = (uint8_t)(c - sh_off[j]);
  }
  __syncthreads();
  // features: one-hot digits, u per parameter, zeros; four threads per row, each CTA
  // of the cluster storing a quarter of the transpose
  for (int G = part; G < F / 8; G += 4) {
    uint32_t v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int c = 8 * G + e;
      const uint32_t m = sh_col[c], dg = (uint32_t)(pk >> (m & 63u)) & 15u;   // 4 x parameter | kind, digit
      v[e] = !live || (m & 128u) ? 0u : (m & 64u) ? sh_utab[(m & 60u) * 4u + dg] : dg == sh_dig[c] ? 0x3F80u : 0u;
    }
    if (live && (G & 3) == rank)
#pragma unroll
      for (int e = 0; e < 8; ++e) td.xt[(size_t)(8 * G + e) * B + b] = (uint16_t)v[e];
    *reinterpret_cast<uint4 *>(sm + tc::core_off(row, 8 * G, F)) =
        make_uint4(v[0] | v[1] << 16, v[2] | v[3] << 16, v[4] | v[5] << 16, v[6] | v[7] << 16);
  }
  tc::fence_async_smem();
  tc::fence_before();
  __syncthreads();
  tc::cluster_sync();      // every CTA of the cluster runs: its shared memory may be written
  tc::fence_after();
  const uint32_t tmem = tmem_base, lanes = (uint32_t)((warp & 3) * 32) << 16;
  const bool lead = warp == 0 && tc::elect_one();
  // A wait that has run out waits once more: what it waited for (a copy into this CTA, MMAs
  // of its own) is not to arrive after the CTA has left.
  auto wait = [&](uint64_t *bar, uint32_t phase) {
    if (tc::mbar_wait(bar, phase, kTrainWait)) return true;
    tc::mbar_wait(bar, phase, kTrainWait);
    return false;
  };
  uint32_t n_mma = 0, n_w[2] = {0u, 0u}, n_x = 0;     // phases passed; exchanges begun

  // Layer i of seven (forward 0..3, backward 4..6): D[dcol ..) = a * w^T over Kd columns,
  // a whole (one KC = Kd buffer) or as the four CTAs' blocks of 64 columns (wait for
  // exchange x >= 0); then the weights of layer i + 2 go into the buffer that is free.
  auto layer = [&](int i, uint32_t a, int x, int Kd, int N, uint32_t dcol, const uint16_t *next, int next_bytes) {
    const int s = i & 1;
    if (warp == 0) {                 // the whole warp, so that descriptors live in uniform registers
      ok = wait(&w_full[s], n_w[s] & 1u) && ok;
      if (x >= 0) ok = wait(&a_full[x & 1], (uint32_t)(x >> 1) & 1u) && ok;
      tc::fence_async_smem();
      tc::fence_after();
      const uint32_t idesc = tc::idesc_bf16(128, N);
      const uint32_t w_hi = tc::sdesc_hi((uint32_t)Kd * 16u), a_hi = x >= 0 ? tc::sdesc_hi(kCols * 16u) : w_hi;
      uint32_t wl = tc::sdesc_lo(wb0 + (uint32_t)s * kWBuf, 128);
      const uint32_t al = tc::sdesc_lo(a, 128);
      for (int k = 0; k < Kd; k += 16, wl += 16) {           // 256 bytes per step, 16 KB per block of 64 columns
        const uint32_t ak = x >= 0 ? (uint32_t)((k >> 6) * 1024 + (k & 63)) : (uint32_t)k;
        if (lead) tc::mma_bf16(tmem + dcol, tc::sdesc_of(al + ak, a_hi), tc::sdesc_of(wl, w_hi), idesc, k ? 1u : 0u);
      }
      if (lead) tc::mma_commit(&mma);
      __syncwarp();
    }
    ++n_w[s];
    ok = wait(&mma, n_mma & 1u) && ok;
    ++n_mma;
    tc::fence_after();
    if (next && threadIdx.x == 0) bulk_g2s(wb0 + (uint32_t)s * kWBuf, next, (uint32_t)next_bytes, &w_full[s]);
  };
  // This thread's 16 bf16 into this CTA's block of buffer `a`, and the block to the others.
  auto share = [&](uint32_t a, const uint32_t (&h)[8]) {
    uint8_t *blk = sm + (a - act0) + rank * (kActBuf / kSplitN);
    *reinterpret_cast<uint4 *>(blk + tc::core_off(row, chunk, kCols)) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4 *>(blk + tc::core_off(row, chunk + 8, kCols)) = make_uint4(h[4], h[5], h[6], h[7]);
    tc::fence_async_smem();
    tc::fence_before();
    __syncthreads();
    if (threadIdx.x == 0) {
      const uint32_t at = a + (uint32_t)rank * (kActBuf / kSplitN), bar = tc::smem_u32(&a_full[n_x & 1]);
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                   "r"((kSplitN - 1) * (kActBuf / kSplitN)) : "memory");
      for (int r = 1; r < kSplitN; ++r) {
        const uint32_t to = (uint32_t)((rank + r) & (kSplitN - 1));
        bulk_s2c(tc::map_rank(at, to), at, kActBuf / kSplitN, tc::map_rank(bar, to));
      }
    }
    ++n_x;
  };
  // the same into the transpose [256][B] of a layer
  auto store_t = [&](uint16_t *t, const uint32_t (&h)[8]) {
    if (live)
#pragma unroll
      for (int i = 0; i < 16; ++i)
        t[(size_t)(n0 + chunk + i) * B + b] = (uint16_t)(i & 1 ? h[i >> 1] >> 16 : h[i >> 1]);
  };

  // ---- forward: hidden layers 0..2 (accumulators in columns 64 l) ----------------------
#pragma unroll 1
  for (int l = 0; l < 3; ++l) {
    layer(l, act0 + (uint32_t)(l & 1) * kActBuf, l - 1, l == 0 ? F : H, kCols, (uint32_t)(l * kCols),
          l == 0 ? td.w[2] + (size_t)n0 * H : l == 1 ? td.w[3] : td.wt[3] + (size_t)n0 * Kp,
          l == 0 ? kCols * H * 2 : l == 1 ? Kp * H * 2 : kCols * Kp * 2);
    float v[16], erf[16];
    uint32_t h[8];
    tc::tmem_ld16(tmem + lanes + (uint32_t)(l * kCols + chunk), v);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float z = __fadd_rn(v[i], sh_b[l][chunk + i]);
      erf[i] = erff(z * 0.70710678118654752f);
      v[i] = gelu_f(z, erf[i]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] = bf2(v[2 * i], v[2 * i + 1]);
    share(act0 + (uint32_t)((l + 1) & 1) * kActBuf, h);
    store_t(td.at[l], h);
    tmem_st16(tmem + lanes + kErfCol + (uint32_t)(l * kCols + chunk), erf);
  }
  // ---- output layer, loss and its gradient: every CTA all of it, a quarter of the columns
  // per thread; one CTA per quarter adds the errors and stores ---------------------------
  double e = 0.0;
  {
    const int nc = Kp >> 2, c0 = part * nc;           // 4, 8, 12 or 16 columns
    const bool mine = part == rank;
    float t[16], v[16];
    const float *trow = td.target + (size_t)src * K + c0;
    const bool vec = (K & 3) == 0;
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
      float4 q = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (i < nc && live && c0 + i < K) {
        if (vec) {
          q = *reinterpret_cast<const float4 *>(trow + i);
        } else {
          q.x = trow[i];
          if (c0 + i + 1 < K) q.y = trow[i + 1];
          if (c0 + i + 2 < K) q.z = trow[i + 2];
          if (c0 + i + 3 < K) q.w = trow[i + 3];
        }
      }
      t[i] = q.x;
      t[i + 1] = q.y;
      t[i + 2] = q.z;
      t[i + 3] = q.w;
    }
    layer(3, act0 + kActBuf, 2, H, Kp, kOutCol, td.wt[2] + (size_t)n0 * H, kCols * H * 2);
    if (threadIdx.x == 0)      // the others may write this buffer again
      for (int r = 1; r < kSplitN; ++r)
        tc::mbar_arrive_cluster(tc::map_rank(tc::smem_u32(&freed), (uint32_t)((rank + r) & (kSplitN - 1))));
#pragma unroll
    for (int i = 0; i < 16; ++i) tmem_ld1(tmem + lanes + kOutCol + (uint32_t)min(c0 + i, Kp - 1), v[i]);
#pragma unroll
    for (int i = 0; i < 16; i += 4)
      asm volatile("tcgen05.wait::ld.sync.aligned;"
                   : "+f"(v[i]), "+f"(v[i + 1]), "+f"(v[i + 2]), "+f"(v[i + 3])::"memory");
    const float bk = (float)B * (float)K;      // below 2^24: exact
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (i >= nc) break;
      float g = 0.0f;
      if (live && c0 + i < K) {
        const float d = __fsub_rn(__fadd_rn(v[i], sh_b4[c0 + i]), t[i]);
        if (mine) e += (double)d * (double)d;
        // 2 d / (B K), one rounding (a float64 quotient rounded to float32 is the same number)
        g = __fdiv_rn(2.0f * d, bk);
      }
      v[i] = g;
    }
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
      if (i >= nc) break;
      const uint32_t lo = bf2(v[i], v[i + 1]), hi = bf2(v[i + 2], v[i + 3]);
      *reinterpret_cast<uint2 *>(sm + tc::core_off(row, c0 + i, Kp)) = make_uint2(lo, hi);
      if (mine && live) {
        uint16_t *gt = td.gbt + (size_t)(c0 + i) * B + b;
        gt[0] = (uint16_t)lo;
        gt[B] = (uint16_t)(lo >> 16);
        gt[2 * (size_t)B] = (uint16_t)hi;
        gt[3 * (size_t)B] = (uint16_t)(hi >> 16);
#pragma unroll
        for (int q = 0; q < 4; ++q) td.g[(size_t)(c0 + i + q) * B + b] = v[i + q];
      }
    }
    tc::fence_async_smem();
    tc::fence_before();
    __syncthreads();
  }
  // ---- backward: g_z(l) = (g(l + 1) W(l + 1)) GELU'(z(l)), l = 2, 1, 0 -------------------
#pragma unroll 1
  for (int l = 2; l >= 0; --l) {
    layer(6 - l, act0 + (uint32_t)(l & 1) * kActBuf, l == 2 ? -1 : 4 - l, l == 2 ? Kp : H, kCols, kGradCol,
          l == 2 ? td.wt[1] + (size_t)n0 * H : nullptr, kCols * H * 2);
    float v[16];
    uint32_t h[8];
    {
      float z[16], erf[16];
      tc::tmem_ld16(tmem + lanes + (uint32_t)(l * kCols + chunk), z);
      tc::tmem_ld16(tmem + lanes + kErfCol + (uint32_t)(l * kCols + chunk), erf);
#pragma unroll
      for (int i = 0; i < 16; ++i) z[i] = gelu_grad_f(__fadd_rn(z[i], sh_b[l][chunk + i]), erf[i]);
      tc::tmem_ld16(tmem + lanes + kGradCol + (uint32_t)chunk, v);
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = __fmul_rn(v[i], z[i]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) h[i] = bf2(v[2 * i], v[2 * i + 1]);
    if (l == 2) ok = wait(&freed, 0u) && ok;
    if (l > 0) share(act0 + (uint32_t)((l & 1) ^ 1) * kActBuf, h);
    else tc::fence_before();
    store_t(td.gzt[l], h);
    if (live)
#pragma unroll
      for (int i = 0; i < 16; ++i) td.gz[l][(size_t)(n0 + chunk + i) * B + b] = v[i];
  }
  for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if (lane == 0 && e != 0.0) atomicAdd(td.loss, e);
  if (!ok && lane == 0) atomicExch(td.status, KTUNE_ETIMEOUT);
  tc::fence_before();
  __syncthreads();
  tc::cluster_sync();        // the blocks sent from here have arrived
  if (warp == 1) tc::tmem_dealloc(tmem, 512);
}

// ---- weight gradients ---------------------------------------------------------------
constexpr int kWgThreads = 256;
constexpr int kWgTile = 128;                     // output rows and columns per CTA
constexpr int kWgStage = 2 * kWgTile * 64 * 2;   // both operands' 64 columns of K
constexpr int kWgSmem = 2 * kWgStage;            // three CTAs per SM
constexpr int kColRows = 256;                    // rows per block of the bias gradients' sums

// Blocks below wg_blocks: slice z of one 128 x 128 tile of a weight gradient
// (G^T X over the slice's rows) into the workspace.  The blocks behind them: one
// (32 columns, 256 rows) block of a bias gradient, in the order of a 32-row
// stride: rows y, y + 32, ... per y in float32, then the 32 partials in y order.
__global__ void __launch_bounds__(kWgThreads) k_train_wgrad(const __grid_constant__ WgradDev wd) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ uint64_t mbar;
  __shared__ uint32_t tmem_base;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int B = wd.B;
  pdl_wait();                 // the rows' activations and gradients
  pdl_launch_dependents();
  if ((int)blockIdx.x >= wd.wg_blocks) {
    int q = (int)blockIdx.x - wd.wg_blocks;
    const int nb = (B + kColRows - 1) / kColRows;
    const int rb = q % nb;
    q /= nb;
    int t = 0;
    while (q >= (wd.c_cols[t] + 31) / 32) q -= (wd.c_cols[t++] + 31) / 32;
    const int C = wd.c_cols[t];
    const int r0 = rb * kColRows, r1 = min(B, r0 + kColRows);
    for (int cc = q * 32 + warp; cc < min(C, q * 32 + 32); cc += kWgThreads / 32) {
      const float *g = wd.c_src[t] + (size_t)cc * B;
      float s = 0.0f;                          // lane y: rows y, y + 32, ... of the block
      for (int r = r0 + lane; r < r1; r += 32) s = __fadd_rn(s, g[r]);
      float sum = 0.0f;
      for (int y = 0; y < 32; ++y) sum = __fadd_rn(sum, __shfl_sync(0xffffffffu, s, y));
      if (lane == 0) wd.c_part[t][(size_t)rb * C + cc] = sum;
    }
    return;
  }
  int tile = (int)blockIdx.x / wd.splits, p = 0;
  const int z = (int)blockIdx.x - tile * wd.splits;
  while (tile >= wd.tiles[p]) tile -= wd.tiles[p++];
  // the accumulator's rows are the weight's columns (the layer's inputs) and its
  // columns the weight's rows: lanes then store neighbouring addresses
  const int M = wd.N[p], N = wd.M[p], nt = (N + kWgTile - 1) / kWgTile;
  const int m0 = tile / nt * kWgTile, c0 = tile % nt * kWgTile;
  const int Nt = min(kWgTile, N - c0);
  const uint16_t *A = wd.X[p] + (size_t)m0 * B, *X = wd.A[p] + (size_t)c0 * B;
  // this slice's rows, in whole chunks of 64
  const int n_chunks = (B + 63) / 64;
  const int lo = (int)((int64_t)n_chunks * z / wd.splits), hi = (int)((int64_t)n_chunks * (z + 1) / wd.splits);
  if (warp == 0) tc::tmem_alloc(&tmem_base, 128);
  if (threadIdx.x == 0) tc::mbar_init(&mbar, 1);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_base;
  uint32_t phase = 0;
  bool ok = true;
  auto issue = [&](int c) {
    const int k0 = c * 64, kc = min(64, B - k0);
    uint8_t *s = sm + (c & 1) * kWgStage;
    tc::load_tile(s, A, B, kWgTile, M - m0, k0, kc);
    tc::load_tile(s + kWgStage / 2, X, B, Nt, Nt, k0, kc);
    cp_async_commit();
  };
  auto done = [&]() {
    bool w = tc::mbar_wait(&mbar, phase, kTrainWait);
    if (!w) w = tc::mbar_wait(&mbar, phase, kTrainWait) && false;
    phase ^= 1u;
    ok = ok && w;
    tc::fence_after();
  };
  issue(lo);                  // (never more slices than chunks: none is empty)
  for (int c = lo; c < hi; ++c) {
    // the MMAs of chunk c - 1 read the stage that chunk c + 1 is copied into
    if (c > lo) {
      done();
      __syncthreads();
    }
    if (c + 1 < hi) {
      issue(c + 1);
      cp_async_wait_group<1>();
    } else {
      cp_async_wait_group<0>();
    }
    tc::fence_async_smem();
    __syncthreads();
    if (threadIdx.x == 0) {
      tc::fence_after();
      const int kc = min(64, B - c * 64);
      const uint32_t idesc = tc::idesc_bf16(128, Nt), dh = tc::sdesc_hi((uint32_t)kc * 16u);
      const uint32_t s = tc::smem_u32(sm + (c & 1) * kWgStage);
      uint32_t al = tc::sdesc_lo(s, 128), xl = tc::sdesc_lo(s + kWgStage / 2, 128);
      for (int k = 0; k < kc; k += 16, al += 16, xl += 16)
        tc::mma_bf16(tmem, tc::sdesc_of(al, dh), tc::sdesc_of(xl, dh), idesc, c > lo || k ? 1u : 0u);
      tc::mma_commit(&mbar);
    }
  }
  done();
  const int row = m0 + (warp & 3) * 32 + lane;
  float *out = wd.ws[p] + (size_t)z * M * N + (size_t)c0 * M + row;
  for (int c = 16 * (warp >> 2); c < Nt; c += 32) {
    float v[16];
    tc::tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + c, v);
    if (row < M)
#pragma unroll
      for (int i = 0; i < 16; ++i) out[(size_t)(c + i) * M] = v[i];
  }
  if (!ok && threadIdx.x == 0) atomicExch(wd.status, KTUNE_ETIMEOUT);
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 128);
}

// ---- sums over the slices and Adam ----------------------------------------------------
// One thread per parameter: a weight's slices in order (float32), a bias's row
// blocks in order (float64), then, if adam, the update (every operation one
// float32 rounding) with the refreshed bf16 copy and its transpose; otherwise
// the gradient itself.
__global__ void __launch_bounds__(256) k_train_update(const __grid_constant__ UpdateDev ud) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_wait();                 // the slices and row blocks
  if (i >= ud.total) return;
  int t = 0;
  while (i >= (int64_t)ud.rows[t] * ud.cols[t]) i -= (int64_t)ud.rows[t] * ud.cols[t], ++t;
  float gi;
  if (t & 1) {
    double s = 0.0;
    for (int q = 0; q < ud.n_part; ++q) s += (double)ud.part[t >> 1][(size_t)q * ud.cols[t] + i];
    gi = (float)s;
  } else {
    const float *w = ud.ws[t >> 1] + i;
    const size_t stride = (size_t)ud.rows[t] * ud.cols[t];
    gi = 0.0f;
    int z = 0;
    for (; z + 16 <= ud.splits; z += 16) {     // sixteen loads in flight, added in order
      float v[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) v[e] = w[(size_t)(z + e) * stride];
#pragma unroll
      for (int e = 0; e < 16; ++e) gi = __fadd_rn(gi, v[e]);
    }
    for (; z < ud.splits; ++z) gi = __fadd_rn(gi, w[(size_t)z * stride]);
  }
  if (!ud.adam) {
    ud.g[t][i] = gi;
    return;
  }
  const AdamArgs &a = ud.a;
  const float mi = __fadd_rn(__fmul_rn(a.b1, ud.m[t][i]), __fmul_rn(a.om1, gi));
  const float vi = __fadd_rn(__fmul_rn(a.b2, ud.v[t][i]), __fmul_rn(__fmul_rn(a.om2, gi), gi));
  ud.m[t][i] = mi;
  ud.v[t][i] = vi;
  const float mh = __fdiv_rn(mi, a.c1), vh = __fdiv_rn(vi, a.c2);
  const float pi =
      __fsub_rn(ud.p[t][i], __fdiv_rn(__fmul_rn(a.lr, mh), __fadd_rn(__fsqrt_rn(vh), a.eps)));
  ud.p[t][i] = pi;
  if (t & 1) return;
  const uint16_t h = tc::f2bf(pi);
  const int rows = ud.rows[t], cols = ud.cols[t], r = (int)(i / cols), c = (int)(i - (int64_t)r * cols);
  ud.wb[t >> 1][tc::core_off(r, c, cols) >> 1] = h;
  if (ud.wt[t >> 1]) ud.wt[t >> 1][tc::core_off(c, r, rows) >> 1] = h;
}

// A launch that may be scheduled while its predecessor finishes; the kernel
// waits for it in pdl_wait() before touching its results.
template <typename A>
void launch_early(void (*kern)(A), int grid, int block, size_t smem, cudaStream_t st, const A &arg) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = st != nullptr ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kern, arg);
}

}  // namespace

void mlp_train_set_attrs() {
  cudaFuncSetAttribute(k_train_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmem);
  cudaFuncSetAttribute(k_train_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgSmem);
}

void launch_train_rows(const TrainDev &td, cudaStream_t st) {
  k_train_rows<<<kSplitN * ((td.B + kRows - 1) / kRows), kRowThreads, kRowSmem, st>>>(td);
}

int train_part_rows(int B) { return (B + kColRows - 1) / kColRows; }

void launch_train_wgrad(WgradDev wd, cudaStream_t st) {
  int blocks = 0;
  for (int p = 0; p < 4; ++p) {
    wd.tiles[p] = ((wd.M[p] + kWgTile - 1) / kWgTile) * ((wd.N[p] + kWgTile - 1) / kWgTile);
    blocks += wd.tiles[p] * wd.splits;
  }
  wd.wg_blocks = blocks;
  for (int t = 0; t < 4; ++t) blocks += (wd.c_cols[t] + 31) / 32 * train_part_rows(wd.B);
  launch_early(k_train_wgrad, blocks, kWgThreads, kWgSmem, st, wd);
}

void launch_train_update(const UpdateDev &ud, cudaStream_t st) {
  launch_early(k_train_update, (int)((ud.total + 255) / 256), 256, 0, st, ud);
}

}  // namespace ktune
