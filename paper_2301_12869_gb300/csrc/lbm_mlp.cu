// Learned warm start for the liquid-column runs: a 6 -> 128 -> 128 -> 128 -> 1 SiLU
// network that predicts the steady density profile rho(z)/rho_c of a column from
// (T/T_c, log10|g|, gravity form, <rho>/rho_c, z/H, log2 H). It has no counterpart in the paper;
// it only initialises lattice Boltzmann runs (Sec. IV set-up), which decide the result.
//
// Arithmetic: bfloat16 inputs, weights and activations as matrix operands, FP32
// accumulation, FP32 biases, output layer, loss and Adam (FP32 master weights).
//
// Every matrix product runs on the tcgen05 tensor cores. The bare product (lbm_mlp_gemm) is one
// GEMM kernel, C[M x N] = A[M x K] B[N x K]^T with A and B bfloat16, K contiguous:
//  * a CTA (4 warps) owns a 128 x 128 output tile whose FP32 accumulator lives in 128
//    TMEM columns; K is consumed in chunks of 64 through kStages shared-memory stages;
//  * one thread (the producer) fills a stage with two TMA tile copies: a 2-D tensor map
//    over each row-major operand with a 64-element (128 B) x 128-row box and the 128-byte
//    swizzle lands the chunk as 128 rows of 128 B, the 16-byte pieces of row r permuted by
//    r mod 8 - the K-major SWIZZLE_128B layout that the MMA's matrix descriptor names
//    (8-row groups 1024 B apart; the K = 16 steps start 32 B apart); the copies complete
//    on the stage's `full` mbarrier;
//  * a second thread waits for a full stage, issues four 128 x 128 x 16 MMAs on it and
//    commits them to the stage's `empty` mbarrier, which the producer waits for before
//    refilling the stage, and after the last chunk to the `done` mbarrier;
//  * the epilogue reads the accumulator with tcgen05.ld (warp w: rows 32w..32w+31, one row
//    per lane), turns each 32 x 32 piece around in shared memory so that the lanes run
//    along a row of C, and stores or adds (split K) it with coalesced accesses.
// The network itself takes two fused kernels: mlp_forward_kernel (inference) and
// mlp_train_kernel (a training step's forward and backward pass).
// Waits are bounded (clock64); a timeout sets the status word and the CTA still waits
// (bounded) for its MMAs and frees its TMEM before returning.
#include "lbm.h"
#include "lbm_internal.h"
#include "lbm_ptx.cuh"
#include "lbm_vec.cuh"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

namespace {

using bf16 = __nv_bfloat16;
using lbm::kWaitCycles;

constexpr int W = LBM_MLP_WIDTH;      // 128
constexpr int KIN = LBM_MLP_IN_PAD;   // 16: inputs padded to one MMA K step
constexpr int OFF_W1 = 0;
constexpr int OFF_B1 = OFF_W1 + W * KIN;
constexpr int OFF_W2 = OFF_B1 + W;
constexpr int OFF_B2 = OFF_W2 + W * W;
constexpr int OFF_W3 = OFF_B2 + W;
constexpr int OFF_B3 = OFF_W3 + W * W;
constexpr int OFF_W4 = OFF_B3 + W;
constexpr int OFF_B4 = OFF_W4 + W;
constexpr int NPARAM = OFF_B4 + 1;
static_assert(NPARAM == LBM_MLP_NPARAMS, "parameter layout");

// feature normalisation x_norm = (x - c) / s
__constant__ float kCenter[LBM_MLP_INPUTS] = {0.825f, -5.0f, 1.5f, 1.4f, 0.5f, 8.0f};
__constant__ float kScale[LBM_MLP_INPUTS] = {0.125f, 1.0f, 0.5f, 1.1f, 0.5f, 2.0f};

// ------------------------------------------------------------------ GEMM
constexpr int BM = 128, BN = 128, BK = 64, GT = 128;
constexpr int kStages = 3;
constexpr int TILE_BYTES = BM * BK * 2;   // one operand, one stage: 16 KB
constexpr int GEMM_SMEM = 2 * kStages * TILE_BYTES + 1024 + 128;  // stages, alignment, barriers
// instruction descriptor, kind::f16: D FP32 (bits 4-5 = 1), A and B bfloat16 (bits 7-9,
// 10-12 = 1), both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at bits 24-28
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(BN >> 3) << 17) | (uint32_t(BM >> 4) << 24);

enum Epi : int { EPI_STORE = 0, EPI_ATOMIC = 1 };

struct GemmArgs {
  const bf16* A;
  int lda;
  const bf16* B;
  int ldb;
  int M, N, K, k_split;  // k_split: K range per blockIdx.z (multiple of BK)
  float* C;              // EPI_STORE / EPI_ATOMIC: C[m * ldc + n]
  int ldc;
  int* status;
};

// shared-memory matrix descriptor, K-major with the 128-byte swizzle (layout type 2 in bits
// 61-63): SBO = 1024 B between 8-row groups, LBO unused inside one swizzle atom (16 B by
// convention), descriptor version 1 (bits 46-47); p lies in a 1024-byte aligned tile,
// offset by 32 B per K = 16 step
__device__ __forceinline__ uint64_t smem_desc(const void* p) {
  const uint32_t a = lbm::smem_u32(p);
  return uint64_t((a >> 4) & 0x3FFF) | (uint64_t(1) << 16) | (uint64_t(1024 >> 4) << 32) | (uint64_t(1) << 46) |
         (uint64_t(2) << 61);
}

// TMA: one box of a 2-D tensor map (x = element along K, y = row) into shared memory,
// completing on an mbarrier
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          lbm::smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(lbm::smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(lbm::smem_u32(bar)), "r"(bytes)
               : "memory");
}

template <int EPI>
__global__ void __launch_bounds__(GT, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, const GemmArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;                          // stage s at sA + s * TILE_BYTES
  uint8_t* sB = smem + kStages * TILE_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + 2 * kStages * TILE_BYTES);
  uint64_t* empty = full + kStages;
  uint64_t* done = empty + kStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  int* err_s = reinterpret_cast<int*>(tmem_slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int kbeg = blockIdx.z * g.k_split;
  const int kend = min(g.K, kbeg + g.k_split);
  const int nchunks = kend > kbeg ? (kend - kbeg + BK - 1) / BK : 0;
  if (nchunks == 0) return;  // uniform over the CTA, before any allocation

  if (tid == 0) {
    for (int i = 0; i < kStages; ++i) {
      lbm::mbar_init(&full[i], 1);
      lbm::mbar_init(&empty[i], 1);
    }
    lbm::mbar_init(done, 1);
    *err_s = 0;
    lbm::fence_mbar_init();
  }
  if (warp == 0) {
    lbm::tmem_alloc(tmem_slot, BN);
    lbm::tmem_relinquish();
  }
  lbm::tc_fence_before();
  __syncthreads();
  lbm::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // K = 16 steps of chunk c (the last chunk may be short: K is a multiple of 16; the box
  // reads zeros beyond K, and a split boundary is a multiple of BK)
  auto ksteps = [&](int c) { return min(BK, kend - (kbeg + c * BK)) / 16; };

  int c = 0;  // producer: chunks whose copies were issued
  if (tid == 0) {
    // producer: TMA copies of A and B for every chunk, each into a free stage
    for (; c < nchunks; ++c) {
      const int st = c % kStages;
      if (c >= kStages && !lbm::mbar_wait_bounded(&empty[st], uint32_t(((c / kStages) - 1) & 1))) {
        atomicOr(err_s, 1);
        break;
      }
      mbar_expect_tx(&full[st], uint32_t(2 * TILE_BYTES));  // whole boxes, zero fill included
      const int k = kbeg + c * BK;
      tma_load_2d(sA + st * TILE_BYTES, &mapA, k, m0, &full[st]);
      tma_load_2d(sB + st * TILE_BYTES, &mapB, k, n0, &full[st]);
    }
  } else if (tid == 32) {
    // MMA issuer: four K = 16 steps per chunk, the stage freed by the commit
    for (int c = 0; c < nchunks; ++c) {
      const int st = c % kStages;
      if (!lbm::mbar_wait_bounded(&full[st], uint32_t((c / kStages) & 1))) {
        atomicOr(err_s, 1);
        break;
      }
      lbm::tc_fence_after();
      const int steps = ksteps(c);
      for (int j = 0; j < steps; ++j)
        lbm::tc_mma_f16(tmem, smem_desc(sA + st * TILE_BYTES + 32 * j), smem_desc(sB + st * TILE_BYTES + 32 * j),
                        kIdesc, (c > 0 || j > 0) ? 1u : 0u);
      lbm::tc_commit(&empty[st]);
    }
    lbm::tc_commit(done);  // every MMA issued so far, also after an error
  }
  // the accumulator is final once `done` completes
  const bool fin = lbm::mbar_wait_bounded(done, 0u);
  bool ok = __syncthreads_and(fin && *err_s == 0);
  lbm::tc_fence_after();
  if (!ok) {
    if (tid == 0) {
      atomicOr(g.status, lbm::STATUS_TIMEOUT);
      // copies in flight must land before the CTA's shared memory goes away: only the last
      // kStages issued chunks can be outstanding (a stage is refilled after its previous
      // chunk was consumed); bounded waits
      for (int q = max(0, c - kStages); q < c; ++q)
        (void)lbm::mbar_wait_bounded(&full[q % kStages], uint32_t((q / kStages) & 1), kWaitCycles / 8);
    }
  } else {
    // each warp stages its 32 x 32 pieces of the accumulator through a padded shared tile
    // (the drained stage buffers) so that global rows are written by 32 lanes at once:
    // t[r][c] holds row 32 warp + r, column nb + c
    float* t = reinterpret_cast<float*>(smem) + warp * (32 * 33);
    const int mw = m0 + 32 * warp;
#pragma unroll 1
    for (int cc = 0; cc < BN / 32; ++cc) {
      float v[32];
      lbm::tmem_ld32(tmem + (uint32_t(32 * warp) << 16) + uint32_t(32 * cc), v);
      const int nb = n0 + 32 * cc;
      const int n = nb + lane;
#pragma unroll
      for (int i = 0; i < 32; ++i) t[lane * 33 + i] = v[i];
      __syncwarp();
#pragma unroll 4
      for (int r = 0; r < 32; ++r) {
        const int m = mw + r;
        const bool in = m < g.M && n < g.N;
        const float x = t[r * 33 + lane];
        if constexpr (EPI == EPI_STORE) {
          if (in) g.C[size_t(m) * g.ldc + n] = x;
        } else {
          if (in) atomicAdd(g.C + size_t(m) * g.ldc + n, x);
        }
      }
      __syncwarp();
    }
  }
  lbm::tc_fence_before();
  __syncthreads();
  if (warp == 0) lbm::tmem_dealloc(tmem, BN);
}

// ------------------------------------------------------------------ fused forward pass
// The whole network for 128-row tiles in one persistent kernel (inference: lbm_mlp_predict
// and the warm start). The weights stay in shared memory for the CTA's lifetime (TMA, the
// GEMM's 128-byte-swizzled K-major layout), the biases and w4 beside them. The CTA runs
// four independent tile pipelines (groups of 4 warps), each with its own activation
// buffer, TMEM accumulator (128 of the SM's 512 columns), mbarrier and named barrier, so
// the groups' MMAs overlap each other's epilogues. Per tile
// the group's 128 threads (one row each) write their normalised bfloat16 inputs into the
// A-operand buffer, one thread issues the layer's MMAs, and every thread reads its row
// back (tcgen05.ld), adds the bias, applies SiLU and writes the bfloat16 activations
// straight into the same A-operand buffer in the swizzled layout the next layer's
// descriptor names (16-byte piece j of row r at piece position j ^ (r mod 8)). After the
// third layer the output layer is a dot product with w4 in registers. Rounding points as
// in the GEMM path: bfloat16 inputs, weights and H1, H2; FP32 accumulation, biases, H3
// and output.
constexpr int FF_GROUPS = 4;                         // most tile pipelines per CTA
constexpr int FF_THREADS = 512;                      // 16 warps
constexpr int FF_BOX = BK * 128 * 2;                 // one 64-element x 128-row swizzled box: 16 KB
constexpr int FF_W1 = 0;                             // W1 (K = 16, zero-filled to the box)
constexpr int FF_W2 = FF_W1 + FF_BOX;                // W2: two K boxes
constexpr int FF_W3 = FF_W2 + 2 * FF_BOX;            // W3: two K boxes
constexpr int FF_H = FF_W3 + 2 * FF_BOX;             // per group: activations / inputs, two K boxes
constexpr int FF_VEC = FF_H + 2 * FF_BOX * FF_GROUPS; // b1, b2, b3, w4 (FP32), b4
constexpr int FF_BAR = FF_VEC + (4 * 128 + 4) * 4;   // mbarriers, TMEM slot
constexpr int FF_SMEM = FF_BAR + 64 + 1024;          // + alignment slack: 211 KB

// 16-byte piece (8 bfloat16 values, k = 8 j .. 8 j + 7) of row r of a K-major operand held in
// 128-byte-swizzled boxes of 64 K values
__device__ __forceinline__ void ff_store8(uint8_t* base, int r, int j, const float (&v)[8]) {
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    w[i] = *reinterpret_cast<const uint32_t*>(&b);
  }
  uint8_t* dst = base + (j >> 3) * FF_BOX + r * 128 + (((j & 7) ^ (r & 7)) << 4);
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(lbm::smem_u32(dst)), "r"(w[0]), "r"(w[1]),
               "r"(w[2]), "r"(w[3])
               : "memory");
}

// z / (1 + exp(-z)) of a pair: the hardware's exponential and reciprocal (a few ulp)
__device__ __forceinline__ lbm::f2 silu_fast(lbm::f2 z) {
  const lbm::f2 t = z * lbm::cst<lbm::f2>(-1.4426950408889634);
  float e0, e1;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(lbm::lo(t)));
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(lbm::hi(t)));
  const lbm::f2 d = lbm::cst<lbm::f2>(1.0) + lbm::make_f2(e0, e1);
  return z * lbm::make_f2(lbm::rcp_approx(lbm::lo(d)), lbm::rcp_approx(lbm::hi(d)));
}
// the pair as bfloat16, the first value in the low half
__device__ __forceinline__ uint32_t bf16_pair(lbm::f2 v) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(lbm::lo(v), lbm::hi(v));
  return *reinterpret_cast<const uint32_t*>(&b);
}

// barrier among the `count` threads of group g (named barrier 1 + g) returning the AND of v
__device__ __forceinline__ bool group_and(bool v, int g, int count) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %1, 0;\n\t"
      "bar.red.and.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(uint32_t(v)), "r"(1 + g), "r"(count)
      : "memory");
  return r != 0;
}

// G: tile pipelines of the CTA's 16 warps - four of 4 warps (a thread does a row), or one of 16 (a
// thread does 32 columns of a row), which takes a quarter of the time for a single tile
template <int G>
__global__ void __launch_bounds__(FF_THREADS, 1)
    mlp_forward_kernel(const __grid_constant__ CUtensorMap mapW1, const __grid_constant__ CUtensorMap mapW2,
                       const __grid_constant__ CUtensorMap mapW3, const float* __restrict__ P,
                       const float* __restrict__ feat, long long n, float* __restrict__ y, int* status) {
  using lbm::f2;
  constexpr int COLS = 32 * G;          // columns a thread does of its row
  constexpr int GT_ = FF_THREADS / G;   // threads of a group
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* wbar = reinterpret_cast<uint64_t*>(smem + FF_BAR);
  uint64_t* mbars = wbar + 1;  // one per group
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mbars + FF_GROUPS);
  float* vec = reinterpret_cast<float*>(smem + FF_VEC);  // b1 [0, 128), b2, b3, w4, b4 [512]
  float* ypart = reinterpret_cast<float*>(smem + FF_H + 2 * FF_BOX);  // G = 1: partial outputs [4][128]
  const int tid = threadIdx.x, warp = tid >> 5;
  const int g = tid / GT_, cg = (tid % GT_) >> 7;        // group, column group
  const int r = 32 * (warp & 3) + (tid & 31);            // this thread's row within the tile
  const long long ntiles = (n + 127) / 128;

  if (tid == 0) {
    lbm::mbar_init(wbar, 1);
    for (int i = 0; i < FF_GROUPS; ++i) lbm::mbar_init(&mbars[i], 1);
    lbm::fence_mbar_init();
  }
  for (int i = tid; i < 4 * 128 + 1; i += FF_THREADS)
    vec[i] = P[i < 128 ? OFF_B1 + i : (i < 256 ? OFF_B2 + i - 128 : (i < 384 ? OFF_B3 + i - 256 : (i < 512 ? OFF_W4 + i - 384 : OFF_B4)))];
  if (warp == 0) {
    lbm::tmem_alloc(tmem_slot, 128 * G);
    lbm::tmem_relinquish();
  }
  lbm::tc_fence_before();
  __syncthreads();
  lbm::tc_fence_after();
  const uint32_t tmem_acc = *tmem_slot + uint32_t(128 * g);
  const uint32_t tmem = tmem_acc + (uint32_t(32 * (warp & 3)) << 16) + uint32_t(COLS * cg);  // warp lanes, columns
  uint8_t* sH = smem + FF_H + g * 2 * FF_BOX;
  uint64_t* mbar = &mbars[g];
  if (tid == 0) {  // the three weight matrices, once per CTA
    mbar_expect_tx(wbar, uint32_t(5 * FF_BOX));
    tma_load_2d(smem + FF_W1, &mapW1, 0, 0, wbar);
    tma_load_2d(smem + FF_W2, &mapW2, 0, 0, wbar);
    tma_load_2d(smem + FF_W2 + FF_BOX, &mapW2, BK, 0, wbar);
    tma_load_2d(smem + FF_W3, &mapW3, 0, 0, wbar);
    tma_load_2d(smem + FF_W3 + FF_BOX, &mapW3, BK, 0, wbar);
  }
  bool ok = true, weights = false;  // the weights are waited for before the first product
  uint32_t uses = 0;                // completed phases of this group's mbarrier
  // one layer: the group's A buffer is complete; one thread issues k_steps K = 16 MMAs of
  // A (sH) and B (weights) into the group's accumulator and commits them to its mbarrier
  auto mma_layer = [&](const uint8_t* sB, int k_steps) {
    lbm::fence_proxy_async_smem();  // this group's st.shared of A -> visible to the tensor cores
    lbm::tc_fence_before();
    if (!weights) weights = lbm::mbar_wait_bounded(wbar, 0u);
    if (!group_and(weights, g, GT_)) return false;
    lbm::tc_fence_after();
    if (tid % GT_ == 0) {
      for (int j = 0; j < k_steps; ++j) {
        const int off = (j >> 2) * FF_BOX + 32 * (j & 3);
        lbm::tc_mma_f16(tmem_acc, smem_desc(sH + off), smem_desc(sB + off), kIdesc, j > 0 ? 1u : 0u);
      }
      lbm::tc_commit(mbar);
    }
    const bool done = lbm::mbar_wait_bounded(mbar, uses & 1u);
    ++uses;
    lbm::tc_fence_after();
    return group_and(done, g, GT_);
  };
  // tile t of the CTA's sequence goes to its group t % G: CTAs have the same number of tiles but one
  for (long long t = blockIdx.x + (long long)gridDim.x * g; t < ntiles; t += (long long)gridDim.x * G) {
    const long long m = t * 128 + r;  // this thread's row
    if (cg == 0) {  // normalised inputs, bfloat16, K = 16 (6 used)
      float a[8], b[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) a[j] = b[j] = 0.0f;
      if (m < n) {
#pragma unroll
        for (int j = 0; j < LBM_MLP_INPUTS; ++j) a[j] = (feat[m * LBM_MLP_INPUTS + j] - kCenter[j]) / kScale[j];
      }
      ff_store8(sH, r, 0, a);
      ff_store8(sH, r, 1, b);
    }
    float out = cg == 0 ? vec[512] : 0.0f;
#pragma unroll 1
    for (int layer = 0; layer < 3; ++layer) {
      const uint8_t* sB = smem + (layer == 0 ? FF_W1 : (layer == 1 ? FF_W2 : FF_W3));
      if (!mma_layer(sB, layer == 0 ? 1 : 8)) {
        ok = false;
        break;
      }
      const float* bias = vec + 128 * layer + COLS * cg;
#pragma unroll 1
      for (int cc = 0; cc < G; ++cc) {  // 32 of the thread's columns
        float v[32];
        lbm::tmem_ld32(tmem + uint32_t(32 * cc), v);
        f2 h[16];
#pragma unroll
        for (int i = 0; i < 16; ++i)
          h[i] = silu_fast(lbm::make_f2(v[2 * i], v[2 * i + 1]) + *reinterpret_cast<const f2*>(bias + 32 * cc + 2 * i));
        if (layer < 2) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {  // 16-byte piece j of row r at piece position j ^ (r mod 8)
            const int j = (COLS * cg) / 8 + 4 * cc + q;
            uint8_t* dst = sH + (j >> 3) * FF_BOX + r * 128 + (((j & 7) ^ (r & 7)) << 4);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(lbm::smem_u32(dst)),
                         "r"(bf16_pair(h[4 * q])), "r"(bf16_pair(h[4 * q + 1])), "r"(bf16_pair(h[4 * q + 2])),
                         "r"(bf16_pair(h[4 * q + 3]))
                         : "memory");
          }
        } else {
          const float* w4 = vec + 384 + COLS * cg + 32 * cc;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            out = fmaf(lbm::lo(h[i]), w4[2 * i], out);
            out = fmaf(lbm::hi(h[i]), w4[2 * i + 1], out);
          }
        }
      }
      // every read of the accumulator is complete before the group's next MMAs overwrite it
      lbm::tc_fence_before();
    }
    if (!ok) break;
    if constexpr (G == 1) {  // the four column groups' parts of a row's output
      ypart[128 * cg + r] = out;
      __syncthreads();
      if (cg == 0 && m < n) y[m] = (out + ypart[128 + r]) + (ypart[256 + r] + ypart[384 + r]);
    } else if (m < n) {
      y[m] = out;
    }
  }
  if (!ok && tid % GT_ == 0) {
    atomicOr(status, lbm::STATUS_TIMEOUT);
    // this group's issued MMAs finish before the CTA goes (bounded)
    lbm::tc_commit(mbar);
    (void)lbm::mbar_wait_bounded(mbar, uses & 1u, kWaitCycles / 8);
  }
  // the weight copies land before the CTA goes (bounded), also where no tile waited for them
  if (!weights) (void)lbm::mbar_wait_bounded(wbar, 0u, kWaitCycles / 8);
  lbm::tc_fence_before();
  __syncthreads();
  if (warp == 0) lbm::tmem_dealloc(*tmem_slot, 128 * G);
}

// ------------------------------------------------------------------ other kernels
__device__ __forceinline__ uint64_t splitmix64(uint64_t counter, uint64_t seed) {
  uint64_t z = seed + (counter + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// ------------------------------------------------------------------ fused training pass
// One training step's forward and backward pass over 128-row tiles, with the gradients of every
// parameter: what took eleven launches (gather, six GEMMs with their operands and transposes in
// global memory, a head of one row a thread) is one. A CTA of 16 warps holds the three weight
// matrices (TMA) and a tile's operands in shared memory, and all accumulators in TMEM: the
// layer's 128 columns, and dW3, dW2, dW1 summed over the CTA's tiles.
//
// Every product reads the same 128-byte-swizzled boxes (row r at 128 r bytes, 64 elements a box):
// K-major where K runs along the rows (activations x weights of the forward pass), and
// MN-major - the descriptor's other reading - where K is the row index: the weight gradients
// dZ^T H sum over the tile's rows, and the backward products dZ W read W [out][in] by its rows,
// so no transposed copy is made anywhere.
//
// Epilogues: warp w owns rows 32 (w % 4) .. + 31 (one a lane) and columns 32 (w / 4) .. + 31 of
// each layer, and keeps silu'(z) of its 32 values in registers for the backward pass. The
// gradients of b1, b2, b3 and w4 are column sums over a warp's rows (a transposing butterfly: lane
// j ends with column j). The FP32 gradients leave the CTA once, as four-wide reductions.
// Rounding points: bfloat16 x, W, H1, H2, dZ1..dZ3 as matrix operands; FP32 accumulation,
// biases, output layer, loss and column sums.
//
// Bound by its chain of six products and epilogues, one tile a CTA (8192 rows: 64 tiles): 27.6 us a
// step with the update, 26.5 with what does not depend on the kernel before (the samples here, the
// parameters and Adam's moments there) read while that one ends.
constexpr int TR_THREADS = 512;
constexpr int TR_W1 = 0;                       // W1 (K = 16, zero-filled to the box)
constexpr int TR_W2 = TR_W1 + FF_BOX;
constexpr int TR_W3 = TR_W2 + 2 * FF_BOX;
constexpr int TR_X = TR_W3 + 2 * FF_BOX;       // inputs (K = 16 of a box)
constexpr int TR_H1 = TR_X + FF_BOX;
constexpr int TR_H2 = TR_H1 + 2 * FF_BOX;
constexpr int TR_DZ = TR_H2 + 2 * FF_BOX;
constexpr int TR_VEC = TR_DZ + 2 * FF_BOX;     // b1, b2, b3, w4, b4 (FP32)
constexpr int TR_Y = TR_VEC + (4 * 128 + 4) * 4;  // [4][128] partial outputs, then [128] targets
constexpr int TR_BAR = TR_Y + 5 * 128 * 4;
constexpr int TR_SMEM = TR_BAR + 32 + 1024;    // + alignment slack: 203 KB
// TMEM columns: the layer, dW3, dW2, dW1
constexpr int TC_Z = 0, TC_W3 = 128, TC_W2 = 256, TC_W1 = 384, TC_ALL = 512;

// instruction descriptor with A and / or B read MN-major (bits 15, 16), N columns
__host__ __device__ constexpr uint32_t idesc_of(bool a_mn, bool b_mn, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(a_mn) << 15) | (uint32_t(b_mn) << 16) |
         (uint32_t(n >> 3) << 17) | (uint32_t(BM >> 4) << 24);
}
// MN-major matrix descriptor of a box pair: 64 elements along M or N a box, FF_BOX to the next
// (leading offset), 8 rows of K in 1024 B (stride offset)
__device__ __forceinline__ uint64_t smem_desc_mn(const void* p) {
  const uint32_t a = lbm::smem_u32(p);
  return uint64_t((a >> 4) & 0x3FFF) | (uint64_t(FF_BOX >> 4) << 16) | (uint64_t(1024 >> 4) << 32) |
         (uint64_t(1) << 46) | (uint64_t(2) << 61);
}

// 1/x of x >= 1 to within an FP32 rounding: the hardware's reciprocal and one Newton step
__device__ __forceinline__ float rcp_newton(float x) {
  const float r = lbm::rcp_approx(x);
  return fmaf(r, fmaf(-x, r, 1.0f), r);
}
// silu(z) and silu'(z); d: silu' = s (1 + z (1 - s))
__device__ __forceinline__ float silu_both(float z, float& d) {
  const float den = 1.0f + expf(-z);
  const float s = den < 1e30f ? rcp_newton(den) : 0.0f;  // exp overflow: sigmoid 0
  d = s * (1.0f + z * (1.0f - s));
  return z * s;
}

// sums over the warp's lanes of 32 values each: lane j gets the sum of v[j]. Overwrites v.
__device__ __forceinline__ float column_sums(float (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int m = 16; m; m >>= 1) {
    const bool up = lane & m;
#pragma unroll
    for (int i = 0; i < m; ++i) {
      const float give = up ? v[i] : v[i + m], keep = up ? v[i + m] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, m);
    }
  }
  return v[0];
}

__device__ __forceinline__ void red_add4(float* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

struct TrainArgs {
  const float* P;
  const float* feat;
  const float* tgt;
  long long n;        // samples
  int count;          // rows of this pass: samples 0 .. count - 1, or with random SplitMix64 draws
  int random;
  unsigned long long seed;
  long long step;
  float* grad;        // += the gradients of every parameter
  double* loss;       // += the sum of squared errors
  int* status;
};

__global__ void __launch_bounds__(TR_THREADS, 1)
    mlp_train_kernel(const __grid_constant__ CUtensorMap mapW1, const __grid_constant__ CUtensorMap mapW2,
                     const __grid_constant__ CUtensorMap mapW3, const TrainArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* wbar = reinterpret_cast<uint64_t*>(smem + TR_BAR);
  uint64_t* mbar = wbar + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mbar + 1);
  float* vec = reinterpret_cast<float*>(smem + TR_VEC);
  float* ypart = reinterpret_cast<float*>(smem + TR_Y);
  float* tgt_s = ypart + 4 * 128;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cg = warp >> 2;                    // column group
  const int r = 32 * (warp & 3) + lane;        // row of the tile
  const int ntiles = (a.count + 127) / 128;

  if (tid == 0) {
    lbm::mbar_init(wbar, 1);
    lbm::mbar_init(mbar, 1);
    lbm::fence_mbar_init();
  }
  if (warp == 0) {
    lbm::tmem_alloc(tmem_slot, TC_ALL);
    lbm::tmem_relinquish();
  }
  // inputs of tile t: normalised, bfloat16, K = 16 (6 used); rows beyond count are zero. The samples are
  // the caller's, which no kernel of a run writes, so the first tile's are read while the update of
  // the step before still runs
  auto gather = [&](int t) {
    if (tid < 128) {
      const int i = t * 128 + tid;
      float x[8], z8[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = z8[j] = 0.0f;
      float tv = 0.0f;
      if (i < a.count) {
        const long long idx =
            a.random ? (long long)(splitmix64((unsigned long long)a.step * (unsigned long long)a.count + i, a.seed) %
                                   (unsigned long long)a.n)
                     : i;
#pragma unroll
        for (int j = 0; j < LBM_MLP_INPUTS; ++j) x[j] = (a.feat[idx * LBM_MLP_INPUTS + j] - kCenter[j]) / kScale[j];
        tv = a.tgt[idx];
      }
      ff_store8(smem + TR_X, tid, 0, x);
      ff_store8(smem + TR_X, tid, 1, z8);
      tgt_s[tid] = tv;
    }
  };
  gather(blockIdx.x);
  lbm::griddep_wait();  // launched as a dependent of the parameter update
  lbm::griddep_launch_dependents();
  for (int i = tid; i < 4 * 128 + 1; i += TR_THREADS)
    vec[i] = a.P[i < 128 ? OFF_B1 + i : (i < 256 ? OFF_B2 + i - 128 : (i < 384 ? OFF_B3 + i - 256 : (i < 512 ? OFF_W4 + i - 384 : OFF_B4)))];
  lbm::tc_fence_before();
  __syncthreads();
  lbm::tc_fence_after();
  const uint32_t tbase = *tmem_slot;
  const uint32_t trow = tbase + (uint32_t(32 * (warp & 3)) << 16) + uint32_t(32 * cg);  // this warp's lanes, columns
  if (tid == 0) {
    mbar_expect_tx(wbar, uint32_t(5 * FF_BOX));
    tma_load_2d(smem + TR_W1, &mapW1, 0, 0, wbar);
    tma_load_2d(smem + TR_W2, &mapW2, 0, 0, wbar);
    tma_load_2d(smem + TR_W2 + FF_BOX, &mapW2, BK, 0, wbar);
    tma_load_2d(smem + TR_W3, &mapW3, 0, 0, wbar);
    tma_load_2d(smem + TR_W3 + FF_BOX, &mapW3, BK, 0, wbar);
  }
  uint32_t uses = 0;  // completed phases of mbar
  // the CTA's writes of the operands are complete: one thread issues the products, all wait for
  // them; false on a timeout (uniform)
  auto products = [&](auto issue) {
    lbm::fence_proxy_async_smem();
    lbm::tc_fence_before();
    __syncthreads();
    lbm::tc_fence_after();
    if (tid == 0) {
      issue();
      lbm::tc_commit(mbar);
    }
    const bool done = lbm::mbar_wait_bounded(mbar, uses & 1u);
    ++uses;
    lbm::tc_fence_after();
    return __syncthreads_and(done) != 0;
  };
  auto k_off = [](int j) { return (j >> 2) * FF_BOX + 32 * (j & 3); };  // K-major step of 16
  auto forward = [&](int src, int w, int steps) {
    return products([&] {
      for (int j = 0; j < steps; ++j)
        lbm::tc_mma_f16(tbase + TC_Z, smem_desc(smem + src + k_off(j)), smem_desc(smem + w + k_off(j)),
                        idesc_of(false, false, 128), j > 0 ? 1u : 0u);
    });
  };
  bool first = true;  // the CTA's first tile: the gradients' accumulators start at zero
  // dW (+)= dZ^T H over the tile's rows, and with wsrc the layer below: dH = dZ W
  auto backward = [&](int h, int dw, int n, int wsrc) {
    return products([&] {
      for (int j = 0; j < 8; ++j)
        lbm::tc_mma_f16(tbase + dw, smem_desc_mn(smem + TR_DZ + 2048 * j), smem_desc_mn(smem + h + 2048 * j),
                        idesc_of(true, true, n), first && j == 0 ? 0u : 1u);
      if (wsrc >= 0)
        for (int j = 0; j < 8; ++j)
          lbm::tc_mma_f16(tbase + TC_Z, smem_desc(smem + TR_DZ + k_off(j)), smem_desc_mn(smem + wsrc + 2048 * j),
                          idesc_of(false, true, 128), j > 0 ? 1u : 0u);
    });
  };
  // this warp's 32 values of a row into an operand buffer
  auto store_row = [&](int dst, const float (&v)[32]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float piece[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) piece[i] = v[8 * q + i];
      ff_store8(smem + dst, r, 4 * cg + q, piece);
    }
  };

  bool ok = __syncthreads_and(lbm::mbar_wait_bounded(wbar, 0u));
  float gb1 = 0.f, gb2 = 0.f, gb3 = 0.f, gw4 = 0.f, gb4 = 0.f;  // column 32 cg + lane over this warp's rows
  double e2 = 0.0;
  for (int t = blockIdx.x; ok && t < ntiles; t += gridDim.x) {
    if (!first) gather(t);
    float v[32], d1[32], d2[32];
    // ---- forward
    if (!(ok = forward(TR_X, TR_W1, 1))) break;
    lbm::tmem_ld32(trow + TC_Z, v);
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = silu_both(v[i] + vec[32 * cg + i], d1[i]);
    store_row(TR_H1, v);
    if (!(ok = forward(TR_H1, TR_W2, 8))) break;
    lbm::tmem_ld32(trow + TC_Z, v);
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = silu_both(v[i] + vec[128 + 32 * cg + i], d2[i]);
    store_row(TR_H2, v);
    if (!(ok = forward(TR_H2, TR_W3, 8))) break;
    lbm::tmem_ld32(trow + TC_Z, v);
    // ---- head: y = h3 . w4 + b4, the error, and dZ3 = dy w4 silu'(z3)
    {
      float d3[32], yp = 0.0f;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        v[i] = silu_both(v[i] + vec[256 + 32 * cg + i], d3[i]);
        yp = fmaf(v[i], vec[384 + 32 * cg + i], yp);
      }
      ypart[128 * cg + r] = yp;
      __syncthreads();
      const float y = vec[512] + ((ypart[r] + ypart[128 + r]) + (ypart[256 + r] + ypart[384 + r]));
      const float e = t * 128 + r < a.count ? y - tgt_s[r] : 0.0f;
      const float dy = 2.0f * e / float(a.count);
      if (cg == 0) {
        e2 += double(e) * double(e);
        gb4 += dy;
      }
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] *= dy;
      gw4 += column_sums(v);
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = dy * vec[384 + 32 * cg + i] * d3[i];
    }
    store_row(TR_DZ, v);
    gb3 += column_sums(v);
    // ---- backward
    if (!(ok = backward(TR_H2, TC_W3, 128, TR_W3))) break;
    lbm::tmem_ld32(trow + TC_Z, v);
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] *= d2[i];
    store_row(TR_DZ, v);
    gb2 += column_sums(v);
    if (!(ok = backward(TR_H1, TC_W2, 128, TR_W2))) break;
    lbm::tmem_ld32(trow + TC_Z, v);
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] *= d1[i];
    store_row(TR_DZ, v);
    gb1 += column_sums(v);
    if (!(ok = backward(TR_X, TC_W1, 16, -1))) break;
    first = false;
  }
  if (ok && !first) {
    // ---- the CTA's gradients: this warp's rows are outputs r of dW, its columns inputs; CTAs start
    // at different pieces so that they do not queue on the same addresses
#pragma unroll 1
    for (int m = 0; m < 2; ++m) {
      float v[32];
      lbm::tmem_ld32(trow + (m == 0 ? TC_W3 : TC_W2), v);
      float* dst = a.grad + (m == 0 ? OFF_W3 : OFF_W2) + r * W + 32 * cg;
#pragma unroll
      for (int i = 0; i < 8; ++i) red_add4(dst + 4 * i, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
    if (cg == 0) {  // dW1: 16 columns
      float v[32];
      lbm::tmem_ld32(tbase + (uint32_t(32 * (warp & 3)) << 16) + TC_W1, v);
      float* dst = a.grad + OFF_W1 + r * KIN;
#pragma unroll
      for (int i = 0; i < KIN / 4; ++i) red_add4(dst + 4 * i, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
    }
    const int j = 32 * cg + lane;
    atomicAdd(a.grad + OFF_B1 + j, gb1);
    atomicAdd(a.grad + OFF_B2 + j, gb2);
    atomicAdd(a.grad + OFF_B3 + j, gb3);
    atomicAdd(a.grad + OFF_W4 + j, gw4);
    if (cg == 0) {
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        e2 += __shfl_xor_sync(0xffffffffu, e2, o);
        gb4 += __shfl_xor_sync(0xffffffffu, gb4, o);
      }
      if (lane == 0) {
        atomicAdd(a.loss, e2);
        atomicAdd(a.grad + OFF_B4, gb4);
      }
    }
  }
  if (!ok && tid == 0) {
    atomicOr(a.status, lbm::STATUS_TIMEOUT);
    // the weight copies and the issued MMAs finish before the CTA goes (bounded)
    (void)lbm::mbar_wait_bounded(wbar, 0u, kWaitCycles / 8);
    lbm::tc_commit(mbar);
    (void)lbm::mbar_wait_bounded(mbar, uses & 1u, kWaitCycles / 8);
  }
  lbm::tc_fence_before();
  __syncthreads();
  if (warp == 0) lbm::tmem_dealloc(tbase, TC_ALL);
}

// Adam on the FP32 master weights (lr > 0), the gradients zeroed for the next step, and the
// bfloat16 operand copies W1 [128][16], W2, W3 [out][in]; lr = 0: the copies alone
__global__ void adam_kernel(float* __restrict__ P, float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                            float lr, float b1, float b2, float eps, float bc1, float bc2, bf16* __restrict__ W1,
                            bf16* __restrict__ W2, bf16* __restrict__ W3) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = i < NPARAM;
  // launched as a dependent of the training pass, which waited for whatever wrote these three
  float p = in ? __ldcg(P + i) : 0.0f, mi = in ? __ldcg(m + i) : 0.0f, vi = in ? __ldcg(v + i) : 0.0f;
  lbm::griddep_wait();
  lbm::griddep_launch_dependents();
  if (!in) return;
  if (lr > 0.0f) {
    const float gi = g[i];
    mi = b1 * mi + (1.0f - b1) * gi;
    vi = b2 * vi + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    P[i] = p;
    g[i] = 0.0f;
  }
  const bf16 b = __float2bfloat16_rn(p);
  if (i < OFF_B1)
    W1[i - OFF_W1] = b;
  else if (i >= OFF_W2 && i < OFF_B2)
    W2[i - OFF_W2] = b;
  else if (i >= OFF_W3 && i < OFF_B3)
    W3[i - OFF_W3] = b;
}

struct ColFeat {
  int ny;
  long long row_off;   // first row of this column in the concatenated row list
  long long node_off;  // first node of this column in the concatenated [col][y][x] fields
  float t, lg, form, mean;  // T/T_c, log10|g|, form, <rho>/rho_c (NaN: from rho)
  float lh;                 // log2 H
};

// raw features (T/T_c, log10|g|, form, <rho>/rho_c, z/H, log2 H) of every row of every column;
// with rho != NULL also the targets rho(y, x = 0)/rho_c and <rho> from rho itself
__global__ void features_kernel(const ColFeat* __restrict__ cols, int ncols, int nx, const double* __restrict__ rho,
                                double rho_c, float* __restrict__ feat, float* __restrict__ tgt) {
  const int c = blockIdx.x;
  if (c >= ncols) return;
  const ColFeat cf = cols[c];
  __shared__ double part[32];
  float mean = cf.mean;
  if (rho) {  // column mean of rho (every node)
    double s = 0.0;
    for (long long q = threadIdx.x; q < (long long)cf.ny * nx; q += blockDim.x) s += rho[cf.node_off + q];
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    double tot = 0.0;
    for (int w = 0; w < int(blockDim.x >> 5); ++w) tot += part[w];
    mean = float(tot / (double(cf.ny) * nx) / rho_c);
  }
  for (int y = threadIdx.x; y < cf.ny; y += blockDim.x) {
    float* f = feat + (cf.row_off + y) * LBM_MLP_INPUTS;
    f[0] = cf.t;
    f[1] = cf.lg;
    f[2] = cf.form;
    f[3] = mean;
    f[4] = (float(y) + 0.5f) / float(cf.ny);
    f[5] = cf.lh;
    if (rho && tgt) tgt[cf.row_off + y] = float(rho[cf.node_off + (long long)y * nx] / rho_c);
  }
}

// FP64 sum over the block (every thread gets it); red: 32 doubles of shared memory
__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();  // red may still be read from the previous call
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double tot = 0.0;
  for (int w = 0; w < int(blockDim.x >> 5); ++w) tot += red[w];
  return tot;
}

// warm start: rho0 of column c = the predicted profile p(y) (times rho_c, floored at rho_min)
// moved along y by the shift s that gives the column's mass, the same on every x. The moved
// profile at row y is p at y - s, linear between rows and constant beyond the ends, so its
// mass M(s) runs from ny p(ny - 1) (s = -ny: the top value everywhere) to ny p(0) (s = ny);
// s follows by bisection on [-ny, ny] (60 halvings). Matching the mass by moving the
// profile keeps the predicted bulk densities: scaling it instead would change them by the
// relative mass error, a pressure error in the nearly incompressible liquid that excites
// the column's slowest mode. A mass outside that range (no bracket) keeps s = 0. A last
// factor M_target / M(s), within rounding of 1, makes the mass exact.
__global__ void warm_profile_kernel(const ColFeat* __restrict__ cols, int ncols, int nx, const float* __restrict__ yhat,
                                    const double* __restrict__ mean_rho, double rho_c, double rho_min,
                                    double* __restrict__ rho0) {
  const int c = blockIdx.x;
  if (c >= ncols) return;
  const ColFeat cf = cols[c];
  __shared__ double red[32];
  const int ny = cf.ny;
  auto prof = [&](int y) { return fmax(double(yhat[cf.row_off + y]) * rho_c, rho_min); };
  auto moved = [&](int y, double sh) {
    const double z = double(y) - sh;
    if (!(z > 0.0)) return prof(0);
    if (z >= double(ny - 1)) return prof(ny - 1);
    const int k = int(z);
    const double t = z - double(k);
    const double p0 = prof(k);
    return p0 + t * (prof(k + 1) - p0);
  };
  auto mass = [&](double sh) {
    double v = 0.0;
    for (int y = threadIdx.x; y < ny; y += blockDim.x) v += moved(y, sh);
    return block_sum(v, red);
  };
  const double target = mean_rho[c] * double(ny);
  double lo = -double(ny), hi = double(ny), sh = 0.0;
  if (mass(lo) <= target && target <= mass(hi)) {
    for (int it = 0; it < 60; ++it) {
      const double mid = 0.5 * (lo + hi);
      if (mass(mid) < target) lo = mid; else hi = mid;
    }
    sh = 0.5 * (lo + hi);
  }
  const double scale = target / mass(sh);
  for (long long q = threadIdx.x; q < (long long)ny * nx; q += blockDim.x) {
    const int y = int(q / nx);
    rho0[cf.node_off + q] = moved(y, sh) * scale;
  }
}

thread_local char g_err[512] = "";
int fail(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  lbm::set_last_error(g_err);
  return code;
}

}  // namespace

// ------------------------------------------------------------------ handle
constexpr int kLossSlots = 1024;  // training steps between two reads of their losses

struct lbm_mlp {
  cudaStream_t stream = nullptr;
  int Bc = 0;  // batch capacity (multiple of 128)
  void* mem = nullptr;
  float *P = nullptr, *G = nullptr, *Mo = nullptr, *Vo = nullptr;
  bf16 *W1 = nullptr, *W2 = nullptr, *W3 = nullptr;
  CUtensorMap mW1, mW2, mW3;  // of the bfloat16 weights
  double* loss = nullptr;     // kLossSlots sums of squared errors
  int* status = nullptr;
  int nsm = 0;
  long long adam_t = 0;
};

namespace {

#define MLP_CUDA(call)                                                                  \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess) return fail(LBM_ECUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

cudaError_t gemm_prepare() {
  cudaError_t e = cudaSuccess;
  for (const void* fn : {(const void*)gemm_kernel<EPI_STORE>, (const void*)gemm_kernel<EPI_ATOMIC>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, GEMM_SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute((const void*)mlp_forward_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, FF_SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute((const void*)mlp_forward_kernel<FF_GROUPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, FF_SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute((const void*)mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TR_SMEM);
  return e;
}

// cuTensorMapEncodeTiled, looked up once through the runtime (no libcuda link)
using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled encoder() {
  static EncodeTiled fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeTiled>(p);
  }();
  return fn;
}

// 2-D map of a row-major bfloat16 matrix (rows x cols, ld elements per row) with a
// BK-element x 128-row box written with the 128-byte swizzle; reads outside the matrix
// fill zeros
bool make_map(CUtensorMap* m, const bf16* base, int rows, int cols, int ld) {
  EncodeTiled enc = encoder();
  if (!enc) return false;
  const cuuint64_t dims[2] = {cuuint64_t(cols), cuuint64_t(rows)};
  const cuuint64_t strides[1] = {cuuint64_t(ld) * 2};
  const cuuint32_t box[2] = {BK, 128};
  const cuuint32_t estr[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int EPI>
cudaError_t gemm(const GemmArgs& a, int splits, cudaStream_t s) {
  const dim3 grid((a.M + BM - 1) / BM, (a.N + BN - 1) / BN, splits);
  CUtensorMap mA, mB;
  if (!make_map(&mA, a.A, a.M, a.K, a.lda) || !make_map(&mB, a.B, a.N, a.K, a.ldb)) return cudaErrorInvalidValue;
  gemm_kernel<EPI><<<grid, GT, GEMM_SMEM, s>>>(mA, mB, a);
  return cudaGetLastError();
}

GemmArgs gargs(const bf16* A, int lda, const bf16* B, int ldb, int M, int N, int K, int* status) {
  GemmArgs a{};
  a.A = A;
  a.lda = lda;
  a.B = B;
  a.ldb = ldb;
  a.M = M;
  a.N = N;
  a.K = K;
  a.k_split = (K + BK - 1) / BK * BK;
  a.status = status;
  return a;
}

int status_of(lbm_mlp* h) {
  int st = 0;
  MLP_CUDA(cudaMemcpyAsync(&st, h->status, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  MLP_CUDA(cudaStreamSynchronize(h->stream));
  if (st & lbm::STATUS_TIMEOUT) return fail(LBM_ETIMEOUT, "a tensor-core wait timed out");
  return LBM_OK;
}

// gradients (added to G) and loss (added to *loss) of rows 0 .. count - 1, or of a random minibatch
cudaError_t train_pass(lbm_mlp* h, const float* x, const float* t, long long n, int count, bool random,
                       unsigned long long seed, long long step, double* loss) {
  const TrainArgs a{h->P, x, t, n, count, random ? 1 : 0, seed, step, h->G, loss, h->status};
  const int grid = std::min(h->nsm, (count + 127) / 128);
  return lbm::launch_dependent(mlp_train_kernel, dim3(grid), dim3(TR_THREADS), TR_SMEM, h->stream, h->mW1, h->mW2,
                               h->mW3, a);
}

cudaError_t update(lbm_mlp* h, float lr) {
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float bc1 = 1.0f - std::pow(b1, float(h->adam_t)), bc2 = 1.0f - std::pow(b2, float(h->adam_t));
  return lbm::launch_dependent(adam_kernel, dim3((NPARAM + 255) / 256), dim3(256), 0, h->stream, h->P, h->G, h->Mo,
                               h->Vo, lr, b1, b2, eps, bc1, bc2, h->W1, h->W2, h->W3);
}

bool device_pointer(const void* p) {
  cudaPointerAttributes at{};
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

int column_table(const lbm_column* cols, int ncols, int nx, double a, double b, double R, const double* mean_rho,
                 std::vector<ColFeat>& out, double* rho_c, long long* rows) {
  double rc, Tc, pc;
  if (lbm_critical_point(a, b, R, &rc, &Tc, &pc) != LBM_OK) return fail(LBM_EINVAL, "need a, b, R > 0");
  out.resize(ncols);
  long long r = 0, q = 0;
  for (int c = 0; c < ncols; ++c) {
    const lbm_column& in = cols[c];
    if (in.ny <= 0) return fail(LBM_EINVAL, "column %d has ny <= 0", c);
    const double gmag = std::sqrt(in.gx * in.gx + in.gy * in.gy);
    ColFeat& f = out[c];
    f.ny = in.ny;
    f.row_off = r;
    f.node_off = q;
    f.t = float(in.T / Tc);
    f.lg = float(gmag > 0 ? std::log10(gmag) : -12.0);
    f.form = float(in.gravity_form);
    f.mean = mean_rho ? float(mean_rho[c] / rc) : NAN;
    f.lh = float(std::log2(double(in.ny)));
    r += in.ny;
    q += (long long)in.ny * nx;
  }
  *rho_c = rc;
  *rows = r;
  return LBM_OK;
}

}  // namespace

// ================================================================== public ABI
extern "C" {

int lbm_mlp_create(const float* params, int batch_capacity, void* stream, lbm_mlp** out) {
  if (!params || !out) return fail(LBM_EINVAL, "params and out must not be NULL");
  if (batch_capacity < 128 || batch_capacity % 128 || batch_capacity > (1 << 22))
    return fail(LBM_EINVAL, "batch_capacity must be a multiple of 128 in [128, 4194304]");
  *out = nullptr;
  cudaError_t e = gemm_prepare();
  if (e != cudaSuccess) return fail(LBM_ECUDA, "kernel attributes: %s", cudaGetErrorString(e));
  lbm_mlp* h = new (std::nothrow) lbm_mlp();
  if (!h) return fail(LBM_ENOMEM, "out of host memory");
  h->stream = static_cast<cudaStream_t>(stream);
  h->Bc = batch_capacity;
  size_t off = 0;
  auto take = [&](size_t bytes) { const size_t at = off; off = (off + bytes + 255) / 256 * 256; return at; };
  const size_t oP = take(4 * NPARAM), oG = take(4 * NPARAM), oM = take(4 * NPARAM), oV = take(4 * NPARAM);
  const size_t oW1 = take(2 * W * KIN), oW2 = take(2 * W * W), oW3 = take(2 * W * W);
  const size_t oL = take(8 * kLossSlots), oS = take(4);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&h->nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    delete h;
    return fail(LBM_ECUDA, "no CUDA device");
  }
  e = cudaMalloc(&h->mem, off);
  if (e != cudaSuccess) {
    delete h;
    return fail(LBM_ENOMEM, "cudaMalloc %zu bytes: %s", off, cudaGetErrorString(e));
  }
  char* base = static_cast<char*>(h->mem);
  h->P = reinterpret_cast<float*>(base + oP);
  h->G = reinterpret_cast<float*>(base + oG);
  h->Mo = reinterpret_cast<float*>(base + oM);
  h->Vo = reinterpret_cast<float*>(base + oV);
  h->W1 = reinterpret_cast<bf16*>(base + oW1);
  h->W2 = reinterpret_cast<bf16*>(base + oW2);
  h->W3 = reinterpret_cast<bf16*>(base + oW3);
  h->loss = reinterpret_cast<double*>(base + oL);
  h->status = reinterpret_cast<int*>(base + oS);
  int rc = LBM_OK;
  if (!make_map(&h->mW1, h->W1, W, KIN, KIN) || !make_map(&h->mW2, h->W2, W, W, W) ||
      !make_map(&h->mW3, h->W3, W, W, W))
    rc = fail(LBM_ECUDA, "tensor maps of the weights");
  if (!rc) rc = lbm_mlp_set_params(h, params);
  if (rc) {
    lbm_mlp_destroy(h);
    return rc;
  }
  *out = h;
  return LBM_OK;
}

int lbm_mlp_set_params(lbm_mlp* h, const float* params) {
  if (!h || !params) return fail(LBM_EINVAL, "handle and params must not be NULL");
  MLP_CUDA(cudaMemcpyAsync(h->P, params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, h->stream));
  MLP_CUDA(cudaMemsetAsync(h->Mo, 0, sizeof(float) * NPARAM, h->stream));
  MLP_CUDA(cudaMemsetAsync(h->Vo, 0, sizeof(float) * NPARAM, h->stream));
  MLP_CUDA(cudaMemsetAsync(h->status, 0, sizeof(int), h->stream));
  h->adam_t = 0;
  MLP_CUDA(update(h, 0.0f));  // the bfloat16 copies
  MLP_CUDA(cudaStreamSynchronize(h->stream));
  return LBM_OK;
}

int lbm_mlp_get_params(lbm_mlp* h, float* params) {
  if (!h || !params) return fail(LBM_EINVAL, "handle and params must not be NULL");
  MLP_CUDA(cudaMemcpyAsync(params, h->P, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, h->stream));
  MLP_CUDA(cudaStreamSynchronize(h->stream));
  return LBM_OK;
}

int lbm_mlp_gradients(lbm_mlp* h, const float* x, const float* t, int n, float* grads, double* loss) {
  if (!h || !x || !t || !grads) return fail(LBM_EINVAL, "handle, x, t and grads must not be NULL");
  if (n < 1 || n > h->Bc) return fail(LBM_EINVAL, "n must be in [1, batch_capacity]");
  if (!device_pointer(x) || !device_pointer(t)) return fail(LBM_EINVAL, "x and t must be device pointers");
  MLP_CUDA(cudaMemsetAsync(h->G, 0, sizeof(float) * NPARAM, h->stream));
  MLP_CUDA(cudaMemsetAsync(h->loss, 0, sizeof(double), h->stream));
  MLP_CUDA(train_pass(h, x, t, n, n, false, 0, 0, h->loss));
  MLP_CUDA(cudaMemcpyAsync(grads, h->G, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, h->stream));
  double l = 0.0;
  MLP_CUDA(cudaMemcpyAsync(&l, h->loss, sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  const int rc = status_of(h);
  if (loss) *loss = l / n;
  return rc;
}

int lbm_mlp_train(lbm_mlp* h, const float* x, const float* t, long long n, int batch, int iters, float lr,
                  unsigned long long seed, float* losses) {
  if (!h || !x || !t) return fail(LBM_EINVAL, "handle, x and t must not be NULL");
  if (n < 1 || batch < 1 || batch > h->Bc || iters < 0 || !(lr > 0))
    return fail(LBM_EINVAL, "need n >= 1, 1 <= batch <= batch_capacity, iters >= 0, lr > 0");
  if (!device_pointer(x) || !device_pointer(t)) return fail(LBM_EINVAL, "x and t must be device pointers");
  MLP_CUDA(cudaMemsetAsync(h->G, 0, sizeof(float) * NPARAM, h->stream));
  std::vector<double> sums(losses ? std::min(iters, kLossSlots) : 0);
  for (int first = 0; first < iters; first += kLossSlots) {
    const int block = std::min(kLossSlots, iters - first);
    MLP_CUDA(cudaMemsetAsync(h->loss, 0, sizeof(double) * kLossSlots, h->stream));
    for (int it = 0; it < block; ++it) {
      MLP_CUDA(train_pass(h, x, t, n, batch, true, seed, h->adam_t, h->loss + it));
      ++h->adam_t;
      MLP_CUDA(update(h, lr));
    }
    if (losses) {
      MLP_CUDA(cudaMemcpyAsync(sums.data(), h->loss, sizeof(double) * block, cudaMemcpyDeviceToHost, h->stream));
      MLP_CUDA(cudaStreamSynchronize(h->stream));
      for (int it = 0; it < block; ++it) losses[first + it] = float(sums[it] / batch);
    }
  }
  return status_of(h);
}

int lbm_mlp_predict(lbm_mlp* h, const float* x, long long n, float* y) {
  if (!h || !x || !y) return fail(LBM_EINVAL, "handle, x and y must not be NULL");
  if (n < 0) return fail(LBM_EINVAL, "n must be >= 0");
  if (!device_pointer(x) || !device_pointer(y)) return fail(LBM_EINVAL, "x and y must be device pointers");
  if (n == 0) return LBM_OK;
  // the fused forward kernel, one persistent CTA per SM at most: all its warps on a tile while there
  // are no more tiles than SMs, four tiles in flight beyond
  const long long ntiles = (n + 127) / 128;
  const int grid = int(std::min<long long>(h->nsm, ntiles));
  auto fn = ntiles <= h->nsm ? mlp_forward_kernel<1> : mlp_forward_kernel<FF_GROUPS>;
  fn<<<grid, FF_THREADS, FF_SMEM, h->stream>>>(h->mW1, h->mW2, h->mW3, h->P, x, n, y, h->status);
  MLP_CUDA(cudaGetLastError());
  return status_of(h);
}

int lbm_mlp_features(const lbm_column* cols, int ncols, int nx, double a, double b, double R, const double* rho,
                     const double* mean_rho, float* x, float* t, void* stream) {
  if (!cols || ncols < 1 || nx < 1 || !x) return fail(LBM_EINVAL, "cols, ncols >= 1, nx >= 1 and x are required");
  if (!rho && !mean_rho) return fail(LBM_EINVAL, "one of rho (device) and mean_rho (host) is required");
  if (!device_pointer(x) || (t && !device_pointer(t)) || (rho && !device_pointer(rho)))
    return fail(LBM_EINVAL, "x, t and rho must be device pointers");
  std::vector<ColFeat> tab;
  double rho_c;
  long long rows;
  int rc = column_table(cols, ncols, nx, a, b, R, rho ? nullptr : mean_rho, tab, &rho_c, &rows);
  if (rc) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  ColFeat* dtab = nullptr;
  MLP_CUDA(cudaMallocAsync(reinterpret_cast<void**>(&dtab), sizeof(ColFeat) * ncols, s));
  cudaError_t e = cudaMemcpyAsync(dtab, tab.data(), sizeof(ColFeat) * ncols, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    features_kernel<<<ncols, 256, 0, s>>>(dtab, ncols, nx, rho, rho_c, x, t);
    e = cudaGetLastError();
  }
  cudaFreeAsync(dtab, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return fail(LBM_ECUDA, "features: %s", cudaGetErrorString(e));
  return LBM_OK;
}

int lbm_mlp_warm_start(lbm_mlp* h, const lbm_column* cols, int ncols, int nx, double a, double b, double R,
                       const double* mean_rho, double* rho0) {
  if (!h || !cols || ncols < 1 || nx < 1 || !mean_rho || !rho0)
    return fail(LBM_EINVAL, "handle, cols, ncols >= 1, nx >= 1, mean_rho and rho0 are required");
  if (!device_pointer(rho0)) return fail(LBM_EINVAL, "rho0 must be a device pointer");
  std::vector<ColFeat> tab;
  double rho_c;
  long long rows;
  int rc = column_table(cols, ncols, nx, a, b, R, mean_rho, tab, &rho_c, &rows);
  if (rc) return rc;
  cudaStream_t s = h->stream;
  char* mem = nullptr;
  const size_t b_tab = (sizeof(ColFeat) * ncols + 255) / 256 * 256, b_mean = (8 * size_t(ncols) + 255) / 256 * 256;
  const size_t b_feat = (4 * LBM_MLP_INPUTS * size_t(rows) + 255) / 256 * 256;
  MLP_CUDA(cudaMallocAsync(reinterpret_cast<void**>(&mem), b_tab + b_mean + b_feat + 4 * size_t(rows), s));
  ColFeat* dtab = reinterpret_cast<ColFeat*>(mem);
  double* dmean = reinterpret_cast<double*>(mem + b_tab);
  float* feat = reinterpret_cast<float*>(mem + b_tab + b_mean);
  float* yhat = reinterpret_cast<float*>(mem + b_tab + b_mean + b_feat);
  cudaError_t e = cudaMemcpyAsync(dtab, tab.data(), sizeof(ColFeat) * ncols, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(dmean, mean_rho, 8 * size_t(ncols), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    features_kernel<<<ncols, 256, 0, s>>>(dtab, ncols, nx, nullptr, rho_c, feat, nullptr);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) rc = lbm_mlp_predict(h, feat, rows, yhat);
  if (e == cudaSuccess && rc == LBM_OK) {
    // floor: a tenth of the smallest coexistence vapour density the inputs cover
    warm_profile_kernel<<<ncols, 256, 0, s>>>(dtab, ncols, nx, yhat, dmean, rho_c, 1e-3, rho0);
    e = cudaGetLastError();
  }
  cudaFreeAsync(mem, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return fail(LBM_ECUDA, "warm start: %s", cudaGetErrorString(e));
  return rc;
}

namespace {
// checks of lbm_mlp_gemm / lbm_mlp_gemm_enqueue, then the launch on stream s
int gemm_launch(const uint16_t* A, int lda, const uint16_t* B, int ldb, float* C, int ldc, int M, int N, int K,
                int k_split, int accumulate, int* status, cudaStream_t s) {
  if (!A || !B || !C || M < 1 || N < 1 || K < 16 || K % 16) return fail(LBM_EINVAL, "need M, N >= 1 and K a multiple of 16");
  if (lda % 8 || ldb % 8 || lda < K || ldb < K || ldc < N) return fail(LBM_EINVAL, "lda, ldb multiples of 8 and >= K; ldc >= N");
  if ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) return fail(LBM_EINVAL, "A and B 16-byte aligned");
  if (k_split <= 0) k_split = K;
  if (k_split % BK && k_split < K) return fail(LBM_EINVAL, "k_split must be a multiple of 64");
  if (!accumulate && k_split < K) return fail(LBM_EINVAL, "split K needs accumulate");
  cudaError_t e = gemm_prepare();
  if (e != cudaSuccess) return fail(LBM_ECUDA, "kernel attributes: %s", cudaGetErrorString(e));
  GemmArgs a = gargs(reinterpret_cast<const bf16*>(A), lda, reinterpret_cast<const bf16*>(B), ldb, M, N, K, status);
  a.k_split = std::min(K, (k_split + BK - 1) / BK * BK);
  a.C = C;
  a.ldc = ldc;
  const int splits = (K + a.k_split - 1) / a.k_split;
  e = accumulate ? gemm<EPI_ATOMIC>(a, splits, s) : gemm<EPI_STORE>(a, 1, s);
  if (e != cudaSuccess) return fail(LBM_ECUDA, "gemm: %s", cudaGetErrorString(e));
  return LBM_OK;
}
}  // namespace

int lbm_mlp_gemm(const uint16_t* A, int lda, const uint16_t* B, int ldb, float* C, int ldc, int M, int N, int K,
                 int k_split, int accumulate, void* stream) {
  int* status = nullptr;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  MLP_CUDA(cudaMallocAsync(reinterpret_cast<void**>(&status), sizeof(int), s));
  cudaError_t e = cudaMemsetAsync(status, 0, sizeof(int), s);
  int rc = e == cudaSuccess ? gemm_launch(A, lda, B, ldb, C, ldc, M, N, K, k_split, accumulate, status, s)
                            : fail(LBM_ECUDA, "gemm: %s", cudaGetErrorString(e));
  int st = 0;
  if (rc == LBM_OK) e = cudaMemcpyAsync(&st, status, sizeof(int), cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(status, s);
  const cudaError_t es = cudaStreamSynchronize(s);
  if (rc != LBM_OK) return rc;
  if (e == cudaSuccess) e = es;
  if (e != cudaSuccess) return fail(LBM_ECUDA, "gemm: %s", cudaGetErrorString(e));
  if (st & lbm::STATUS_TIMEOUT) return fail(LBM_ETIMEOUT, "a tensor-core wait timed out");
  return LBM_OK;
}

int lbm_mlp_gemm_enqueue(const uint16_t* A, int lda, const uint16_t* B, int ldb, float* C, int ldc, int M, int N,
                         int K, int k_split, int accumulate, int* status, void* stream) {
  if (!status || reinterpret_cast<uintptr_t>(status) % alignof(int)) return fail(LBM_EINVAL, "status: an aligned device int");
  return gemm_launch(A, lda, B, ldb, C, ldc, M, N, K, k_split, accumulate, status, static_cast<cudaStream_t>(stream));
}

int lbm_mlp_destroy(lbm_mlp* h) {
  if (!h) return LBM_OK;
  int rc = LBM_OK;
  if (h->mem) {
    cudaStreamSynchronize(h->stream);
    if (cudaFree(h->mem) != cudaSuccess) rc = LBM_ECUDA;
  }
  delete h;
  return rc;
}

}  // extern "C"
