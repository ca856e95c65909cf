// The MLP counter model on Blackwell tensor cores (BF16 operands, FP32
// accumulators in tensor memory).
//
//   k_gemm_tc     C = A * B^T (A: M x K, B: N x K, both bf16 row-major), exposed
//                 for validation of the operand layouts; 128-row x 256-column
//                 tiles, K in chunks of 64
//   helpers       bf16 copies of the parameters, the per-step set-up of a search
//   (the fused forward of predictions and scores: k_mlp_pair.cu; training:
//   k_mlp_train.cu)
//
// Every wait on the tensor cores is bounded: on time-out the kernel records
// KTUNE_ETIMEOUT, waits once more (bounded) for its MMAs in flight, frees its
// tensor memory and returns.
#include <float.h>
#include <limits.h>

#include "device_common.cuh"
#include "internal.h"
#include "tc.cuh"

namespace ktune {

namespace {

constexpr uint64_t kWaitLimit = 1000000000ull;   // 1 s per tensor-core wait

// MMAs over one K chunk: D (+)= A[:, a_k0 : a_k0 + kc] * B^T, A stored with
// KC = kcA (128 rows), the B chunk with KC = kc (N rows).
__device__ __forceinline__ void issue_chunk(uint32_t tmem, const uint8_t *sA, int kcA, int a_k0,
                                            const uint8_t *sB, int kc, int N, bool first) {
  const uint32_t idesc = tc::idesc_bf16(128, N);
  const uint32_t a0 = tc::smem_u32(sA), b0 = tc::smem_u32(sB);
  for (int q = 0; q < kc / 16; ++q) {
    const uint64_t ad = tc::sdesc(a0 + (uint32_t)((a_k0 + q * 16) >> 3) * 128u, 128, kcA * 16);
    const uint64_t bd = tc::sdesc(b0 + (uint32_t)q * 256u, 128, kc * 16);
    tc::mma_bf16(tmem, ad, bd, idesc, (first && q == 0) ? 0u : 1u);
  }
}

constexpr int kGemmStage = 16384 + 32768;         // A 128 x 64 and B 256 x 64 bf16
constexpr int kGemmSmem = 2 * kGemmStage;          // two stages: two CTAs per SM (2 x 256 TMEM columns)

// 16 floats (v) of one row into dst (16-byte aligned): four vector stores.
__device__ __forceinline__ void store16f(float *dst, const float (&v)[16]) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
    reinterpret_cast<float4 *>(dst)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}
// C = A * B^T, 128 x 256 tiles: the K chunks of 64 run through two shared-memory
// stages, the copies of chunk c + 1 in flight while the tensor cores work on
// chunk c.
__global__ void __launch_bounds__(128, 1)
    k_gemm_tc(const uint16_t *__restrict__ A, int lda, const uint16_t *__restrict__ B, int ldb,
              int M, int N, int K, float *__restrict__ C, int ldc, int *status) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ uint64_t mbar;
  __shared__ uint32_t tmem_base;
  const int warp = threadIdx.x >> 5;
  const int m0 = blockIdx.x * 128;
  const int n0 = blockIdx.y * 256;
  const int Nt = N - n0 < 256 ? N - n0 : 256;
  const int c_lo = 0, c_hi = (K + 63) / 64;
  if (warp == 0) tc::tmem_alloc(&tmem_base, 256);
  if (threadIdx.x == 0) tc::mbar_init(&mbar, 1);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_base;
  uint32_t phase = 0;
  bool ok = true;
  auto stage_a = [&](int c) { return sm + (c & 1) * kGemmStage; };
  auto stage_b = [&](int c) { return sm + (c & 1) * kGemmStage + 16384; };
  auto issue = [&](int c) {
    const int k0 = c * 64, kc = K - k0 < 64 ? K - k0 : 64;
    tc::load_tile(stage_a(c), A + (size_t)m0 * lda, lda, 128, M - m0, k0, kc);
    tc::load_tile(stage_b(c), B + (size_t)n0 * ldb, ldb, Nt, Nt, k0, kc);
    cp_async_commit();
  };
  if (c_lo < c_hi) issue(c_lo);
  for (int c = c_lo; c < c_hi; ++c) {
    // the MMAs of chunk c - 1 read the stage chunk c + 1 is copied into
    if (c > c_lo) {
      const bool w = tc::mbar_wait(&mbar, phase, kWaitLimit);
      if (w) phase ^= 1;
      tc::fence_after();
      if (!__syncthreads_and(w)) {
        ok = false;
        break;
      }
    }
    if (c + 1 < c_hi) {
      issue(c + 1);
      cp_async_wait_group<1>();
    } else {
      cp_async_wait_group<0>();
    }
    tc::fence_async_smem();
    __syncthreads();
    if (threadIdx.x == 0) {
      tc::fence_after();
      const int kc = K - c * 64 < 64 ? K - c * 64 : 64;
      issue_chunk(tmem, stage_a(c), kc, 0, stage_b(c), kc, Nt, c == c_lo);
      tc::mma_commit(&mbar);
    }
  }
  if (ok && c_lo < c_hi) {
    const bool w = tc::mbar_wait(&mbar, phase, kWaitLimit);
    if (w) phase ^= 1;
    tc::fence_after();
    ok = __syncthreads_and(w);
  }
  cp_async_wait_all();
  if (!ok) {
    tc::mbar_wait(&mbar, phase, kWaitLimit);   // the MMAs still in flight, if any
    if (threadIdx.x == 0) atomicExch(status, KTUNE_ETIMEOUT);
  } else {
    const int row = m0 + threadIdx.x;
    for (int c0 = 0; c0 < Nt; c0 += 16) {
      float v[16];
      tc::tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + c0, v);
      if (row < M) store16f(C + (size_t)row * ldc + n0 + c0, v);
    }
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

// bf16 copy (and optional transpose) of float32 parameters in the tensor cores'
// operand layout (core matrices over the whole matrix, KC = its row length).
__global__ void k_to_bf16(const float *__restrict__ p, int rows, int cols,
                          uint16_t *__restrict__ wb, uint16_t *__restrict__ wt) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= (int64_t)rows * cols) return;
  const uint16_t h = tc::f2bf(p[i]);
  const int r = (int)(i / cols), c = (int)(i - (int64_t)r * cols);
  wb[tc::core_off(r, c, cols) >> 1] = h;
  if (wt) wt[tc::core_off(c, r, rows) >> 1] = h;
}

// Per-step set-up of a search scored by the MLP (one CTA): publish the step's
// by-value parameters, Delta, reset the min / max keys, the output count and
// the super-tile sums, and count the counters with a non-zero Delta.  Same
// parameter list as the tree path's prepare kernel.
__global__ void __launch_bounds__(256) k_mlp_prep(const SearchDev *__restrict__ srch,
                                                  StepDev *__restrict__ steps_dev,
                                                  const __grid_constant__ StepBatch<1> sb) {
  const SearchDev &sd = srch[0];
  const StepDev &st = sb.st[0];
  if (threadIdx.x == 0) {
    steps_dev[0] = st;
    sd.mm[0] = INT_MAX;
    sd.mm[1] = INT_MIN;
    if (st.n_out) *st.n_out = 0;
    int na = 0;
    for (int c = 0; c < sd.K; ++c) na += st.delta[c] != 0.0f;
    *sd.n_active = na;
  }
  for (int c = threadIdx.x; c < sd.K; c += blockDim.x) sd.delta[c] = st.delta[c];
  if (sd.select == KTUNE_SELECT_SAMPLE) {
    const int64_t n_super = ((sd.N + kSubTile - 1) / kSubTile + kSuper - 1) / kSuper;
    for (int64_t i = threadIdx.x; i < n_super; i += blockDim.x) sd.super_sum[i] = 0;
  }
}

}  // namespace

// ---- host launchers -------------------------------------------------------------------------
void mlp_set_attrs(int) {
  cudaFuncSetAttribute(k_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kGemmSmem);
  mlp_train_set_attrs();
  mlp_pair_set_attrs();
}

void launch_gemm_tc(const uint16_t *A, int lda, const uint16_t *B, int ldb, int M, int N, int Kd, float *c,
                    int ldc, int *status, cudaStream_t st) {
  const dim3 grid((M + 127) / 128, (N + 255) / 256);
  k_gemm_tc<<<grid, 128, kGemmSmem, st>>>(A, lda, B, ldb, M, N, Kd, c, ldc, status);
}

void launch_to_bf16(const float *p, int rows, int cols, uint16_t *wb, uint16_t *wt,
                    cudaStream_t st) {
  const int64_t n = (int64_t)rows * cols;
  k_to_bf16<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(p, rows, cols, wb, wt);
}

// The fused forward (k_mlp_pair): mode 0 predicted counters, mode 1 Eq. score.
void launch_mlp_fwd(int mode, const MlpDev &md, const uint64_t *packed, int64_t n, float *out,
                    const float *pcprof, const float *delta, const uint32_t *evaluated,
                    int *minmax, int *status, int grid, cudaStream_t st) {
  int sms = grid;
  if (sms <= 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  }
  MlpTargets tg{};
  if (mode == 1) {
    tg.S = 1;
    tg.pcprof[0] = pcprof;
    tg.delta[0] = delta;
    tg.s[0] = out;
    tg.eval[0] = evaluated;
    tg.mm[0] = minmax;
  }
  launch_mlp_pair(mode, md, packed, n, out, tg, status, sms, st);
}

void launch_mlp_score_shared(const MlpDev &md, const uint64_t *packed, int64_t n,
                             const MlpTargets &tg, int *status, int max_ctas, cudaStream_t st) {
  if (tg.S >= 1) launch_mlp_pair(1, md, packed, n, nullptr, tg, status, max_ctas, st);
}

void launch_mlp_prep(const SearchDev *srch, StepDev *steps_dev, const StepBatch<1> &sb,
                     cudaStream_t st) {
  k_mlp_prep<<<1, 256, 0, st>>>(srch, steps_dev, sb);
}

const void *mlp_prep_func() { return (const void *)k_mlp_prep; }

}  // namespace ktune
