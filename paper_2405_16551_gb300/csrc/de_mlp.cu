// de_mlp.cu -- the surrogate network: MLP 20 -> 256 -> 256 -> 1 (ReLU) with
// BF16 operands on tcgen05 tensor cores, FP32 accumulation in TMEM, FP32
// master weights and Adam.
//
// The paper has no surrogate; this network serves the surrogate-assisted
// workload: it ranks several candidate trials per target so that only one
// reaches a costly objective (the paper's Abstract motivates costly
// objectives).  Input x in [-100, 100]^20 enters as x / 100, with a constant 1
// in column 20 so that the first bias is column 20 of W1.
//
//   k_mlp_pass<false>  rows -> y; one CTA per 128 rows: layer 1 (K = 32) and
//                   layer 2 (K = 256) as tcgen05 products, ReLU / bias /
//                   output dot product in the TMEM epilogues
//   k_mlp_pass<true>   one training step's forward and backward pass for one
//                   128-row half of a 256-row minibatch: dZ2 = dy w3 relu',
//                   dH1 = dZ2 W2 on the tensor cores, dZ1 = dH1 relu'; stores
//                   H1, dZ2, dZ1 and the inputs as they are
//   k_mlp_update    weight gradients as products over the batch
//                   (dW2 = dZ2^T H1 with a ones row for db2, dW1 = dZ1^T A1),
//                   each tile's Adam step on the FP32 masters, and the BF16
//                   operand copies of W1 | b1 and W2
//
// A training step is a chain of latencies, not of work (3 GFLOP a step).  What
// it cost before (48.5 + 11.4 + 3.7 us in three kernels): transposed 2-byte
// stores of three activations, a 5-step shuffle sum per column of dw3, a second
// copy of W2, FP64 conversions; now the weight gradients read the stored tiles
// MN-major, and a step is two kernels chained by programmatic launches.
//
// Operand layout in shared and global memory: the canonical K-major, no
// swizzle layout of de_tcgen05.cuh (core matrices of 8 rows x 16 bytes).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <cmath>
#include <stdint.h>
#include <string.h>

#include <string>
#include <vector>

#include "de.h"
#include "de_common.cuh"
#include "de_mlp.h"
#include "de_tcgen05.cuh"

namespace de {

constexpr uint32_t kPurposeSurr = 5u;  // minibatch draws of surrogate training

// ------------------------------------------------------------------ layout helpers
// Byte offset of bf16 element (row, k) in a K-major tile with RG row groups.
__device__ __forceinline__ uint32_t toff(int row, int k, int RG) {
  return (uint32_t)(((((k >> 3) * RG) + (row >> 3)) << 7) + ((row & 7) << 4) + ((k & 7) << 1));
}

__device__ __forceinline__ uint32_t idesc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
}

// A tile of RG row groups read the other way round: its columns as the rows of
// the operand (M or N) and its rows as K ("MN-major": a core matrix holds 8
// columns of 8 rows, the columns contiguous).  So the transposed products need
// no transposed copy.  Byte strides: between 8-column groups RG * 128, between
// 8-row groups 128.
__device__ __forceinline__ uint64_t desc_mn(uint32_t addr, int rg) { return smem_desc(addr, 128u, (uint32_t)rg * 128u); }
constexpr uint32_t kAMn = 1u << 15, kBMn = 1u << 16;  // instruction descriptor: A / B is MN-major

// D (TMEM) = or += A (M = 128, K = 16 ksteps) B^T (N rows); A and B K-major
// with RGa / RGb row groups.
__device__ __forceinline__ void mma_bf16(uint32_t d, uint32_t a, int rga, uint32_t b, int rgb, int ksteps, int n,
                                         bool accumulate) {
  const uint32_t la = (uint32_t)rga * 128u, lb = (uint32_t)rgb * 128u, id = idesc_bf16(n);
  for (int ks = 0; ks < ksteps; ++ks)
    mma_split<2>(d, smem_desc(a + (uint32_t)ks * 2u * la, la, 128u), smem_desc(b + (uint32_t)ks * 2u * lb, lb, 128u),
                 id, (accumulate || ks > 0) ? 1u : 0u);
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  // one conversion for two values: conversions bound the epilogues (16 lanes a
  // clock and SM)
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}

__device__ __forceinline__ void st_bf16(uint8_t* base, uint32_t off, float v) {
  *reinterpret_cast<__nv_bfloat16*>(base + off) = __float2bfloat16_rn(v);
}

// 8 consecutive columns (k0 multiple of 8) of row `row` as one 16-byte store.
__device__ __forceinline__ void st_bf16x8(uint8_t* base, int row, int k0, int RG, const float* v) {
  uint4 u;
  u.x = pack_bf16x2(v[0], v[1]);
  u.y = pack_bf16x2(v[2], v[3]);
  u.z = pack_bf16x2(v[4], v[5]);
  u.w = pack_bf16x2(v[6], v[7]);
  *reinterpret_cast<uint4*>(base + toff(row, k0, RG)) = u;
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ncols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}
__device__ __forceinline__ void tc_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Row index of minibatch row m at training step `step` (Philox, purpose SURR).
__device__ __forceinline__ int batch_row(const MlpStepArgs& a, int m) {
  if (a.sample_n <= 0) return m;  // the first rows, in order
  const U32x4 w = draw_block(a.seed, kPurposeSurr, 0u, 0u, (uint32_t)a.step, (uint32_t)(m >> 2), 0u);
  const uint32_t u = word_of(w, m & 3);
  return (int)((a.sample_base + map_to_range(u, (uint32_t)a.sample_n)) % (uint32_t)a.sample_cap);
}

// ------------------------------------------------------------------ forward / backward
// Shared memory of k_mlp_pass (dynamic, 1024-aligned).
constexpr uint32_t kSBig = 0;                 // 128 KB: W2k (layer 2, and read MN-major for dH1)
constexpr uint32_t kSH1 = 131072;             // 64 KB: H1 (A operand of layer 2); later dZ2 (A operand of dH1)
constexpr uint32_t kSW1 = 196608;             // 16 KB: W1k
constexpr uint32_t kSA1 = 212992;             // 8 KB: A1 (inputs)
constexpr uint32_t kMlpSmem = 221184;

// TRAIN = false: forward of n rows of x (row stride ld) to y.
// TRAIN = true : forward + backward of minibatch half blockIdx.x.
// 16 warps: warp w has tile rows 32 (w mod 4) .. + 31 and columns 64 (w / 4) ..
// + 63.  The epilogues are a thread's walk along its columns, so they take half
// the time that 8 warps of 128 columns took (12.2 us a pass).
constexpr int kPassThreads = 512;
template <bool TRAIN>
__global__ void __launch_bounds__(kPassThreads, 1) k_mlp_pass(MlpDev P, MlpStepArgs a, const double* __restrict__ x,
                                                     int64_t ld, int n, const float* __restrict__ t,
                                                     float* __restrict__ yout) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t bars[2];  // weights, mma
  __shared__ uint32_t s_tmem;
  __shared__ float s_y[2][kTileM];
  __shared__ float s_t[kTileM];
  __shared__ __align__(16) float s_b2[kMlpH], s_w3[kMlpH];
  __shared__ float s_dw3[4][kMlpH];
  __shared__ float s_red[kPassThreads / 32][2];
  __shared__ int s_err;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q = warp & 3, h = warp >> 2;
  const int m = 32 * q + lane;                 // tile row of this thread in the epilogues
  const int row0 = blockIdx.x * kTileM;
  const uint32_t sb = smem_u32(smem);
  const uint32_t b_w = smem_u32(&bars[0]), b_mma = smem_u32(&bars[1]);

  if (tid == 0) {
    for (int k = 0; k < 2; ++k) mbar_init(smem_u32(&bars[k]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_err = 0;
  }
  if (warp == 0) tmem_alloc(&s_tmem, 512);

  // ---- inputs: A1 row = (x / 100, 1, 0 ...) in bf16; four threads per row.
  // They do not depend on the weights: a training step reads them before it
  // waits for the step before.
  {
    const int r = tid >> 2, part = tid & 3;
    const int grow = row0 + r;
    int src = -1;
    if (TRAIN) src = batch_row(a, grow);
    else if (grow < n) src = grow;
    float v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int col = 8 * part + c;
      float val = 0.f;
      if (src >= 0) {
        if (col < kMlpIn) val = to_f32_rn(x[(size_t)src * ld + col] * 0.01);
        else if (col == kMlpIn) val = 1.f;
      }
      v[c] = val;
    }
    st_bf16x8(smem + kSA1, r, 8 * part, 16, v);
    if (TRAIN && part == 0) s_t[r] = src >= 0 ? t[src] : 0.f;
    if (TRAIN) {
      pdl_wait();
      // (after the wait: the update before this step no longer reads it)
      st_bf16x8(P.a1 + (size_t)blockIdx.x * kMlpA1Bytes, r, 8 * part, 16, v);
      pdl_launch_dependents();
    }
  }
  if (tid == 0) {
    // the operands were written by ordinary stores of the kernel before
    asm volatile("fence.proxy.async.global;" ::: "memory");
    mbar_expect_tx(b_w, kMlpW1Bytes + kMlpW2Bytes);
    bulk_g2s(sb + kSW1, P.w1k, kMlpW1Bytes, b_w);
    bulk_g2s(sb + kSBig, P.w2k, kMlpW2Bytes, b_w);
  }
  if (tid < kMlpH) {
    s_b2[tid] = P.b2[tid];
    s_w3[tid] = P.w3[tid];
  }
  fence_async_smem();
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  const uint32_t tmem = s_tmem;
  const uint32_t lane_base = (uint32_t)(32 * q) << 16;

  // ---- layer 1: Z1 = A1 W1k^T -> TMEM columns [0, 256)
  if (tid == 0) {
    if (!mbar_wait(b_w, 0)) s_err = 1;
    else {
      tc_after_sync();
      mma_bf16(tmem, sb + kSA1, 16, sb + kSW1, 32, 2, kMlpH, false);
    }
    mma_commit(b_mma);
  }
  if (!mbar_wait(b_mma, 0)) s_err = 1;
  tc_after_sync();

  // ---- epilogue 1: H1 = relu(Z1) to shared memory (A operand of layer 2);
  // training: also to global memory
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int c0 = 64 * h + 32 * j;
    float v[32];
    tmem_ld_cols32(tmem + lane_base + (uint32_t)c0, v);
#pragma unroll
    for (int e = 0; e < 32; ++e) v[e] = fmaxf(v[e], 0.f);
#pragma unroll
    for (int e = 0; e < 32; e += 8) {
      st_bf16x8(smem + kSH1, m, c0 + e, 16, v + e);
      if (TRAIN) st_bf16x8(P.h1 + (size_t)blockIdx.x * kMlpActBytes, m, c0 + e, 16, v + e);
    }
  }
  fence_async_smem();
  tc_before_sync();
  __syncthreads();
  tc_after_sync();

  // ---- layer 2: Z2 = H1 W2k^T -> TMEM columns [256, 512)
  if (tid == 0) {
    if (!s_err) mma_bf16(tmem + 256, sb + kSH1, 16, sb + kSBig, 32, 16, kMlpH, false);
    mma_commit(b_mma);
  }
  if (!mbar_wait(b_mma, 1)) s_err = 1;
  tc_after_sync();
  // ---- epilogue 2: y = w3 . relu(Z2 + b2) + b3, H2 = relu(Z2 + b2) in registers.
  // A chain of additions covers 128 columns, i.e. two threads' in turn.
  float h2[2][32];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int c0 = 64 * h + 32 * j;
    tmem_ld_cols32(tmem + lane_base + 256u + (uint32_t)c0, h2[j]);
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
      const float4 b = *reinterpret_cast<const float4*>(s_b2 + c0 + e);
      h2[j][e] = fmaxf(h2[j][e] + b.x, 0.f);
      h2[j][e + 1] = fmaxf(h2[j][e + 1] + b.y, 0.f);
      h2[j][e + 2] = fmaxf(h2[j][e + 2] + b.z, 0.f);
      h2[j][e + 3] = fmaxf(h2[j][e + 3] + b.w, 0.f);
    }
  }
  auto dot = [&](float yp) {
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int e = 0; e < 32; e += 4) {
        const float4 w = *reinterpret_cast<const float4*>(s_w3 + 64 * h + 32 * j + e);
        yp = fmaf(h2[j][e], w.x, yp);
        yp = fmaf(h2[j][e + 1], w.y, yp);
        yp = fmaf(h2[j][e + 2], w.z, yp);
        yp = fmaf(h2[j][e + 3], w.w, yp);
      }
    return yp;
  };
  if (!(h & 1)) s_y[h >> 1][m] = dot(0.f);
  __syncthreads();
  if (h & 1) s_y[h >> 1][m] = dot(s_y[h >> 1][m]);
  __syncthreads();
  const float y = s_y[0][m] + s_y[1][m] + P.b3[0];
  if (!TRAIN) {
    if (h == 0 && row0 + m < n) yout[row0 + m] = y;
  } else {
    // mean squared error over the 256-row minibatch
    const float r = y - s_t[m];
    const float dy = 2.f * r / (float)kMlpBatch;
    // dZ2 = dy w3 relu'(Z2 + b2): A operand of dH1 (in H1's place, which
    // layer 2 has consumed) and of dW2 (global); dw3 = sum over rows of H2 dy
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c0 = 64 * h + 32 * j;
      float(&v)[32] = h2[j];
#pragma unroll
      for (int e = 0; e < 32; e += 8) {
        float dz[8], w[8];
        *reinterpret_cast<float4*>(w) = *reinterpret_cast<const float4*>(s_w3 + c0 + e);
        *reinterpret_cast<float4*>(w + 4) = *reinterpret_cast<const float4*>(s_w3 + c0 + e + 4);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          dz[u] = v[e + u] > 0.f ? dy * w[u] : 0.f;
          v[e + u] *= dy;  // row contribution to dw3[c0 + e + u]
        }
        st_bf16x8(smem + kSH1, m, c0 + e, 16, dz);
        st_bf16x8(P.dz2 + (size_t)blockIdx.x * kMlpActBytes, m, c0 + e, 16, dz);
      }
      // sums over the 32 rows of all 32 columns: at each step a lane keeps the
      // columns whose index agrees with it in one bit, so 31 additions do
      // (the pairs added are those of the xor tree)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int e = 0; e < o; ++e) {
          const float keep = up ? v[e + o] : v[e], give = up ? v[e] : v[e + o];
          v[e] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
      }
      s_dw3[q][c0 + lane] = v[0];
    }
    // loss and db3 partials of this half
    float rs = r * r, ds = dy;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      rs += __shfl_xor_sync(0xffffffffu, rs, o);
      ds += __shfl_xor_sync(0xffffffffu, ds, o);
    }
    if (lane == 0) {
      s_red[warp][0] = rs;
      s_red[warp][1] = ds;
    }
    fence_async_smem();
    tc_before_sync();
    __syncthreads();
    tc_after_sync();
    if (tid < kMlpH) {
      // fixed order over the four row quarters
      P.part[blockIdx.x * kMlpPart + tid] = ((s_dw3[0][tid] + s_dw3[1][tid]) + s_dw3[2][tid]) + s_dw3[3][tid];
    }
    if (tid == 0) {
      // db3 and the squared error from the h = 0 warps (each row once)
      P.part[blockIdx.x * kMlpPart + kMlpH] = ((s_red[0][1] + s_red[1][1]) + s_red[2][1]) + s_red[3][1];
      P.part[blockIdx.x * kMlpPart + kMlpH + 1] = ((s_red[0][0] + s_red[1][0]) + s_red[2][0]) + s_red[3][0];
    }

    // ---- dH1 = dZ2 W2: A = dZ2 (shared), B = W2 read MN-major -> TMEM [256, 512)
    // (H2 is in registers; Z1 stays for the last epilogue)
    if (tid == 0) {
      const uint32_t id = idesc_bf16(kMlpH) | kBMn;
      for (int ks = 0; ks < 16; ++ks)
        mma_split<2>(tmem + 256, smem_desc(sb + kSH1 + (uint32_t)ks * 4096u, 2048u, 128u),
                     desc_mn(sb + kSBig + (uint32_t)ks * 256u, 32), id, ks > 0 ? 1u : 0u);
      mma_commit(b_mma);
    }
    if (!mbar_wait(b_mma, 0)) s_err = 1;
    tc_after_sync();

    // ---- epilogue 3: dZ1 = dH1 relu'(Z1) to global memory
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c0 = 64 * h + 32 * j;
      float v[32], z[32];
      tmem_ld_cols32(tmem + lane_base + (uint32_t)c0, z);
      tmem_ld_cols32(tmem + lane_base + 256u + (uint32_t)c0, v);
#pragma unroll
      for (int e = 0; e < 32; ++e) v[e] = z[e] > 0.f ? v[e] : 0.f;
#pragma unroll
      for (int e = 0; e < 32; e += 8) st_bf16x8(P.dz1 + (size_t)blockIdx.x * kMlpActBytes, m, c0 + e, 16, v + e);
    }
  }
  tc_before_sync();
  __syncthreads();
  if (s_err && tid == 0) atomicOr(P.err, 1);
  if (warp == 0) tmem_free(tmem, 512);
}

// ------------------------------------------------------------------ weight gradients + Adam
struct AdamArgs {
  float lr, c1, c2, eps, beta1, beta2;  // c1 = 1 - beta1^t, c2 = 1 - beta2^t
  float omb1, omb2;                     // 1 - beta1, 1 - beta2 (rounded once from FP64)
};

__device__ __forceinline__ float adam_step(float w, float g, float& m, float& v, const AdamArgs& A) {
  const float mn = fmaf(A.beta1, m, A.omb1 * g);
  const float vn = fmaf(A.beta2, v, A.omb2 * g * g);
  m = mn;
  v = vn;
  return w - A.lr * (mn / A.c1) / (sqrtf(vn / A.c2) + A.eps);
}

// Weight gradients of one step and their Adam update (apply = 0: into P.grad
// only).  Blocks 0 .. 31: rows 128 (b / 16) .. + 127 of W2, columns 16 (b mod 16)
// .. + 15 (the first column block also b2); blocks 32 .. 39: a quarter of the
// parameters of 128 rows of W1 and b1 (block 32 also w3, b3 and the loss).  The products leave a tile of gradients
// in shared memory, from which each thread updates 8 consecutive parameters:
// coalesced masters and moments, 16-byte operand stores.
//
// Masters and moments are read before the wait for the step's pass: only the
// update before wrote them, and that one had finished when the pass released
// this launch.  (Read where they are used, a few at a time, they took 10.4 k
// cycles in the blocks of W2, then 32 columns wide, and 17 k in those of W1.)
constexpr int kUpW2 = 32, kUpW1 = 8;  // blocks of W2, of W1
constexpr uint32_t kUpA = 0, kUpB = 65536, kUpOnes = kUpB + 16384, kUpG = kUpOnes + 8192;
constexpr int kUpStride = 36;  // floats per row of the gradient tile (16-byte rows, spread over the banks)
constexpr uint32_t kUpSmem = kUpG + 128u * kUpStride * 4u;

__global__ void __launch_bounds__(256, 1) k_mlp_update(MlpDev P, AdamArgs A, int apply) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ uint32_t s_tmem;
  __shared__ int s_err;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q = warp & 3, h = warp >> 2;
  const uint32_t sb = smem_u32(smem);
  const uint32_t b_ld = smem_u32(&bars[0]), b_mma = smem_u32(&bars[1]);
  const bool w2 = blockIdx.x < kUpW2;
  const int ob = w2 ? blockIdx.x >> 4 : (blockIdx.x - kUpW2) >> 2, ig = w2 ? blockIdx.x & 15 : 0;
  const int part1 = (blockIdx.x - kUpW2) & 3;  // quarter of W1's rows' parameters
  const bool bias = w2 && ig == 0;
  float* gt = reinterpret_cast<float*>(smem + kUpG);
  if (tid == 0) {
    mbar_init(b_ld, 1);
    mbar_init(b_mma, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_err = 0;
  }
  if (warp == 0) tmem_alloc(&s_tmem, 64);
  if (bias) {
    // a ones row (row 0 of a 16-row operand): the sum over the batch, i.e. the
    // gradient of b2
    for (int e = tid; e < 16 * kMlpBatch / 8; e += blockDim.x) {
      const int r = e & 15, k8 = e >> 4;
      const uint32_t one = r == 0 ? 0x3F803F80u : 0u;
      *reinterpret_cast<uint4*>(smem + kUpOnes + toff(r, 8 * k8, 2)) = make_uint4(one, one, one, one);
    }
  }
  // the next step's kernel may start (its inputs do not depend on this one)
  pdl_launch_dependents();
  // ---- this thread's parameters
  struct Par {
    float w, m, v;
  };
  auto fetch = [&](int k) { return Par{__ldcg(P.W1 + k), __ldcg(P.mW1 + k), __ldcg(P.vW1 + k)}; };
  // W2: row r2, 8 columns from c2 on
  const int r2 = tid >> 1, c2 = 8 * (tid & 1), k2 = kMlpOffW2 + (128 * ob + r2) * kMlpH + 16 * ig + c2;
  const int kb = kMlpOffB2 + 128 * ob + 32 * q + lane;  // b2 (bias, h = 0)
  // W1 (256 x 20) and, in column 20, b1: elements of 128 x 21, this quarter's
  // from e1 on
  constexpr int kN1 = 128 * (kMlpIn + 1) / 4, kU1 = (kN1 + 255) / 256;
  const int e1 = part1 * kN1;
  auto k1 = [&](int e) {
    const int r = e / (kMlpIn + 1), c = e - r * (kMlpIn + 1), o = 128 * ob + r;
    return c < kMlpIn ? kMlpOffW1 + o * kMlpIn + c : kMlpOffB1 + o;
  };
  float w8[8], m8[8], v8[8];
  Par p1[kU1], px{};
  if (apply && w2) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      *reinterpret_cast<float4*>(w8 + 4 * e) = __ldcg(reinterpret_cast<const float4*>(P.W1 + k2) + e);
      *reinterpret_cast<float4*>(m8 + 4 * e) = __ldcg(reinterpret_cast<const float4*>(P.mW1 + k2) + e);
      *reinterpret_cast<float4*>(v8 + 4 * e) = __ldcg(reinterpret_cast<const float4*>(P.vW1 + k2) + e);
    }
    if (bias && h == 0) px = fetch(kb);
  } else if (apply) {
#pragma unroll
    for (int u = 0; u < kU1; ++u)
      if (tid + 256 * u < kN1) p1[u] = fetch(k1(e1 + tid + 256 * u));
    if (blockIdx.x == kUpW2) px = fetch(kMlpOffW3 + tid);
  }
  pdl_wait();
  if (tid == 0) {
    const uint8_t *sa = w2 ? P.dz2 : P.dz1, *sbm = w2 ? P.h1 : P.a1;
    const size_t bh = w2 ? kMlpActBytes : kMlpA1Bytes;  // bytes of one half of the batch
    asm volatile("fence.proxy.async.global;" ::: "memory");
    const uint32_t bb = w2 ? 4096u : 8192u;  // 16 or 32 columns of one half
    mbar_expect_tx(b_ld, 65536u + 2u * bb);
    for (int f = 0; f < 2; ++f) {
      bulk_g2s(sb + kUpA + 32768u * f, sa + (size_t)f * kMlpActBytes + (size_t)ob * 32768u, 32768u, b_ld);
      bulk_g2s(sb + kUpB + 8192u * f, sbm + f * bh + (size_t)ig * 4096u, bb, b_ld);
    }
  }
  fence_async_smem();
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  const uint32_t tmem = s_tmem;
  if (tid == 0) {
    if (!mbar_wait(b_ld, 0)) s_err = 1;
    else {
      tc_after_sync();
      const uint32_t id = idesc_bf16(w2 ? 16 : 32) | kAMn | kBMn;
      for (int ks = 0; ks < 16; ++ks) {
        const uint32_t f = ks >> 3, kk = (uint32_t)(ks & 7) * 256u;
        const uint64_t da = desc_mn(sb + kUpA + 32768u * f + kk, 16);
        mma_split<2>(tmem, da, desc_mn(sb + kUpB + 8192u * f + kk, 16), id, ks > 0 ? 1u : 0u);
        if (bias)
          mma_split<2>(tmem + 32, da, smem_desc(sb + kUpOnes + (uint32_t)ks * 512u, 256u, 128u), idesc_bf16(16) | kAMn,
                       ks > 0 ? 1u : 0u);
      }
    }
    mma_commit(b_mma);
  }
  if (!mbar_wait(b_mma, 0)) s_err = 1;
  tc_after_sync();
  const uint32_t lane_base = (uint32_t)(32 * q) << 16;
  // gradient tile: row 32 q + lane, half of the columns per half of the warps
  if (w2) {
    float g[8];
    tmem_ld8(tmem + lane_base + 8u * (uint32_t)h, g);
    float4* dst = reinterpret_cast<float4*>(gt + (32 * q + lane) * kUpStride + 8 * h);
    dst[0] = make_float4(g[0], g[1], g[2], g[3]);
    dst[1] = make_float4(g[4], g[5], g[6], g[7]);
  } else {
    float g[16];
    tmem_ld_cols16(tmem + lane_base + 16u * (uint32_t)h, g);
    float4* dst = reinterpret_cast<float4*>(gt + (32 * q + lane) * kUpStride + 16 * h);
#pragma unroll
    for (int e = 0; e < 4; ++e) dst[e] = make_float4(g[4 * e], g[4 * e + 1], g[4 * e + 2], g[4 * e + 3]);
  }
  const float gb = bias && h == 0 ? tmem_ld1(tmem + lane_base + 32u) : 0.f;
  tc_before_sync();
  __syncthreads();
  // one parameter of the vector: its gradient, or its update
  auto one = [&](int k, float g, Par p) -> float {
    if (!apply) {
      P.grad[k] = g;
      return 0.f;
    }
    const float w = adam_step(p.w, g, p.m, p.v, A);
    P.W1[k] = w;
    P.mW1[k] = p.m;
    P.vW1[k] = p.v;
    return w;
  };
  if (bias && h == 0) one(kb, gb, px);
  if (w2) {
    float g[8];
    const float4* gs = reinterpret_cast<const float4*>(gt + r2 * kUpStride + c2);
    *reinterpret_cast<float4*>(g) = gs[0];
    *reinterpret_cast<float4*>(g + 4) = gs[1];
    if (!apply) {
#pragma unroll
      for (int e = 0; e < 8; ++e) P.grad[k2 + e] = g[e];
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) w8[e] = adam_step(w8[e], g[e], m8[e], v8[e], A);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        reinterpret_cast<float4*>(P.W1 + k2)[e] = *reinterpret_cast<const float4*>(w8 + 4 * e);
        reinterpret_cast<float4*>(P.mW1 + k2)[e] = *reinterpret_cast<const float4*>(m8 + 4 * e);
        reinterpret_cast<float4*>(P.vW1 + k2)[e] = *reinterpret_cast<const float4*>(v8 + 4 * e);
      }
      st_bf16x8(P.w2k, 128 * ob + r2, 16 * ig + c2, 32, w8);
    }
  } else {
#pragma unroll
    for (int u = 0; u < kU1; ++u) {
      if (tid + 256 * u >= kN1) continue;
      const int e = e1 + tid + 256 * u;
      const int r = e / (kMlpIn + 1), c = e - r * (kMlpIn + 1);
      const float w = one(k1(e), gt[r * kUpStride + c], p1[u]);
      if (apply) st_bf16(P.w1k, toff(128 * ob + r, c, 32), w);
    }
    if (blockIdx.x == kUpW2) {
      // w3 and b3 from the two halves' partial sums, in a fixed order
      one(kMlpOffW3 + tid, P.part[tid] + P.part[kMlpPart + tid], px);
      if (tid == 0) {
        one(kMlpOffB3, P.part[kMlpH] + P.part[kMlpPart + kMlpH], apply ? fetch(kMlpOffB3) : Par{});
        P.loss[0] = (P.part[kMlpH + 1] + P.part[kMlpPart + kMlpH + 1]) / (float)kMlpBatch;
      }
    }
  }
  tc_before_sync();
  __syncthreads();
  if (s_err && tid == 0) atomicOr(P.err, 1);
  if (warp == 0) tmem_free(tmem, 64);
}

// BF16 operand copies from the FP32 masters (after set-up or a parameter load).
__global__ void k_mlp_pack(MlpDev P) {
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  for (int e = tid; e < kMlpH * 32; e += stride) {
    const int o = e / 32, c = e % 32;
    const float v = c < kMlpIn ? P.W1[o * kMlpIn + c] : (c == kMlpIn ? P.b1[o] : 0.f);
    st_bf16(P.w1k, toff(o, c, 32), v);
  }
  for (int e = tid; e < kMlpH * kMlpH; e += stride) {
    const int o = e / kMlpH, i = e % kMlpH;
    st_bf16(P.w2k, toff(o, i, 32), P.W2[e]);
  }
}

// ------------------------------------------------------------------ host side
void mlp_configure() {
  cudaFuncSetAttribute(k_mlp_pass<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMlpSmem);
  cudaFuncSetAttribute(k_mlp_pass<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMlpSmem);
  cudaFuncSetAttribute(k_mlp_update, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kUpSmem);
}

void mlp_pack_launch(const MlpDev& P, cudaStream_t s) { k_mlp_pack<<<64, 256, 0, s>>>(P); }

void mlp_forward_launch(const MlpDev& P, const double* x, int64_t ld, int n, float* y, cudaStream_t s) {
  if (n <= 0) return;
  MlpStepArgs a{};
  k_mlp_pass<false><<<(n + kTileM - 1) / kTileM, kPassThreads, kMlpSmem, s>>>(P, a, x, ld, n, nullptr, y);
}

// chained: the launch before this one on the stream is a step's k_mlp_update,
// whose tail this step's first kernel may overlap.
void mlp_step_launch(const MlpDev& P, const MlpStepArgs& a, const double* x, int64_t ld, const float* t, float lr,
                     bool apply, bool chained, cudaStream_t s) {
  AdamArgs A;
  const double b1 = 0.9, b2 = 0.999;
  A.lr = lr;
  A.beta1 = (float)b1;
  A.beta2 = (float)b2;
  A.c1 = (float)(1.0 - pow(b1, (double)(a.step + 1)));
  A.c2 = (float)(1.0 - pow(b2, (double)(a.step + 1)));
  A.eps = 1e-8f;
  A.omb1 = (float)(1.0 - b1);
  A.omb2 = (float)(1.0 - b2);
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kPassThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.gridDim = dim3(kMlpBatch / kTileM);
  cfg.dynamicSmemBytes = kMlpSmem;
  cfg.numAttrs = chained ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k_mlp_pass<true>, P, a, x, ld, 0, t, (float*)nullptr);
  cfg.gridDim = dim3(kUpW2 + kUpW1);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = kUpSmem;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_mlp_update, P, A, apply ? 1 : 0);
}

}  // namespace de

// ------------------------------------------------------------------ C ABI
struct de_mlp {
  cudaStream_t stream = nullptr;
  uint64_t seed = 0;
  long long step = 0;
  void* arena = nullptr;
  de::MlpDev P{};
  std::string err;
};

namespace de {

static de_status mlp_fail(de_mlp* m, de_status s, const std::string& msg) {
  if (s == DE_ERR_CUDA || s == DE_ERR_OOM) cudaGetLastError();  // reported here, not by the next call
  if (m) m->err = msg;
  set_last_error(msg);
  return s;
}

static bool mlp_dev_ptr(const void* p) {
  cudaPointerAttributes a{};
  if (!p || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice;
}

static uint64_t mlp_splitmix(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// He-uniform weights (bound sqrt(6 / fan_in)), zero biases, from the seed.
void mlp_init_params(uint64_t seed, float* p) {
  uint64_t s = seed ^ 0x5EED5EEDull;
  auto fill = [&](int off, int count, int fan_in) {
    const double b = sqrt(6.0 / fan_in);
    for (int e = 0; e < count; ++e) p[off + e] = (float)(-b + 2.0 * b * ((mlp_splitmix(s) >> 11) * 0x1.0p-53));
  };
  memset(p, 0, sizeof(float) * kMlpParams);
  fill(kMlpOffW1, kMlpH * kMlpIn, kMlpIn);
  fill(kMlpOffW2, kMlpH * kMlpH, kMlpH);
  fill(kMlpOffW3, kMlpH, kMlpH);
}

static de_status mlp_upload(de_mlp* m, const float* p) {
  cudaError_t e = cudaMemcpyAsync(m->P.W1, p, sizeof(float) * kMlpParams, cudaMemcpyHostToDevice, m->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->P.mW1, 0, sizeof(float) * kMlpParams, m->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->P.vW1, 0, sizeof(float) * kMlpParams, m->stream);
  if (e == cudaSuccess) {
    mlp_pack_launch(m->P, m->stream);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return mlp_fail(m, DE_ERR_CUDA, std::string("surrogate parameters: ") + cudaGetErrorString(e));
  m->step = 0;
  return DE_OK;
}

static de_status mlp_check(de_mlp* m) {
  int err = 0;
  cudaError_t e = cudaMemcpyAsync(&err, m->P.err, sizeof(int), cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return mlp_fail(m, DE_ERR_CUDA, std::string("surrogate: ") + cudaGetErrorString(e));
  if (err) return mlp_fail(m, DE_ERR_TIMEOUT, "surrogate: a device-side wait timed out");
  return DE_OK;
}

de_status mlp_create(uint64_t seed, cudaStream_t stream, de_mlp** out) {
  de_mlp* m = new de_mlp();
  m->stream = stream;
  m->seed = seed;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    off = (off + 1023) / 1024 * 1024;
    const size_t o = off;
    off += bytes;
    return o;
  };
  const size_t pw = take(sizeof(float) * kMlpParams), pm = take(sizeof(float) * kMlpParams),
               pv = take(sizeof(float) * kMlpParams);
  const size_t o_w1k = take(kMlpW1Bytes), o_w2k = take(kMlpW2Bytes);
  const size_t o_h1 = take(2 * kMlpActBytes), o_dz2 = take(2 * kMlpActBytes), o_dz1 = take(2 * kMlpActBytes);
  const size_t o_a1 = take(2 * kMlpA1Bytes), o_part = take(sizeof(float) * 2 * kMlpPart);
  const size_t o_grad = take(sizeof(float) * kMlpParams), o_loss = take(sizeof(float)), o_err = take(sizeof(int));
  cudaError_t e = cudaMalloc(&m->arena, off);
  if (e != cudaSuccess) {
    delete m;
    return mlp_fail(nullptr, e == cudaErrorMemoryAllocation ? DE_ERR_OOM : DE_ERR_CUDA,
                    std::string("surrogate arena: ") + cudaGetErrorString(e));
  }
  uint8_t* A = (uint8_t*)m->arena;
  auto views = [&](float* base, float*& W1, float*& b1, float*& W2, float*& b2, float*& w3, float*& b3) {
    W1 = base + kMlpOffW1;
    b1 = base + kMlpOffB1;
    W2 = base + kMlpOffW2;
    b2 = base + kMlpOffB2;
    w3 = base + kMlpOffW3;
    b3 = base + kMlpOffB3;
  };
  MlpDev& P = m->P;
  views((float*)(A + pw), P.W1, P.b1, P.W2, P.b2, P.w3, P.b3);
  views((float*)(A + pm), P.mW1, P.mb1, P.mW2, P.mb2, P.mw3, P.mb3);
  views((float*)(A + pv), P.vW1, P.vb1, P.vW2, P.vb2, P.vw3, P.vb3);
  P.w1k = A + o_w1k;
  P.w2k = A + o_w2k;
  P.h1 = A + o_h1;
  P.dz2 = A + o_dz2;
  P.dz1 = A + o_dz1;
  P.a1 = A + o_a1;
  P.part = (float*)(A + o_part);
  P.grad = (float*)(A + o_grad);
  P.loss = (float*)(A + o_loss);
  P.err = (int*)(A + o_err);
  mlp_configure();
  e = cudaMemsetAsync(m->arena, 0, off, stream);
  if (e != cudaSuccess) {
    cudaFree(m->arena);
    delete m;
    return mlp_fail(nullptr, DE_ERR_CUDA, std::string("surrogate arena: ") + cudaGetErrorString(e));
  }
  std::vector<float> p(kMlpParams);
  mlp_init_params(seed, p.data());
  const de_status s = mlp_upload(m, p.data());
  if (s != DE_OK) {
    const std::string msg = m->err;
    cudaFree(m->arena);
    delete m;
    return mlp_fail(nullptr, s, msg);
  }
  *out = m;
  return DE_OK;
}

de_status mlp_reset(de_mlp* m) {
  std::vector<float> p(kMlpParams);
  mlp_init_params(m->seed, p.data());
  return mlp_upload(m, p.data());
}

void mlp_destroy(de_mlp* m) {
  if (!m) return;
  if (m->stream) cudaStreamSynchronize(m->stream);
  if (m->arena) cudaFree(m->arena);
  delete m;
}

const MlpDev& mlp_dev(const de_mlp* m) { return m->P; }

// `steps` Adam steps on minibatches drawn from rows [base, base + n) of a ring
// of `cap` rows (x: FP64 rows of stride ld, t: FP32 targets, same indexing).
de_status mlp_train_rows(de_mlp* m, const double* x, int64_t ld, const float* t, int n, int base, int cap, int steps,
                         float lr) {
  for (int k = 0; k < steps; ++k) {
    MlpStepArgs a{m->seed, m->step, n, base, cap};
    mlp_step_launch(m->P, a, x, ld, t, lr, true, k > 0, m->stream);
    ++m->step;
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return mlp_fail(m, DE_ERR_CUDA, std::string("surrogate training: ") + cudaGetErrorString(e));
  return DE_OK;
}

}  // namespace de

using namespace de;

extern "C" {

de_status de_mlp_create(uint64_t seed, void* cuda_stream, de_mlp** out) {
  if (!out) return mlp_fail(nullptr, DE_ERR_INVALID_ARG, "out is NULL");
  return mlp_create(seed, (cudaStream_t)cuda_stream, out);
}

de_status de_mlp_destroy(de_mlp* m) {
  mlp_destroy(m);
  return DE_OK;
}

de_status de_mlp_set_params(de_mlp* m, const float* params) {
  if (!m || !params) return mlp_fail(m, DE_ERR_INVALID_ARG, "handle or params is NULL");
  for (int e = 0; e < kMlpParams; ++e)
    if (!std::isfinite(params[e])) return mlp_fail(m, DE_ERR_NONFINITE, "params has a non-finite entry");
  return mlp_upload(m, params);
}

de_status de_mlp_get_params(de_mlp* m, float* params) {
  if (!m || !params) return mlp_fail(m, DE_ERR_INVALID_ARG, "handle or params is NULL");
  cudaError_t e = cudaMemcpyAsync(params, m->P.W1, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return mlp_fail(m, DE_ERR_CUDA, std::string("surrogate parameters: ") + cudaGetErrorString(e));
  return DE_OK;
}

de_status de_mlp_forward(de_mlp* m, const double* x_dev, int64_t ld, int32_t n, float* y_dev) {
  if (!m) return mlp_fail(nullptr, DE_ERR_INVALID_ARG, "handle is NULL");
  if (n < 0 || ld < kMlpIn) return mlp_fail(m, DE_ERR_INVALID_ARG, "need n >= 0 and ld >= 20");
  if (n == 0) return DE_OK;
  if (!mlp_dev_ptr(x_dev) || !mlp_dev_ptr(y_dev))
    return mlp_fail(m, DE_ERR_INVALID_ARG, "x_dev and y_dev must be device memory");
  mlp_forward_launch(m->P, x_dev, ld, n, y_dev, m->stream);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return mlp_fail(m, DE_ERR_CUDA, std::string("surrogate forward: ") + cudaGetErrorString(e));
  return DE_OK;
}

de_status de_mlp_grad(de_mlp* m, const double* x_dev, int64_t ld, const float* t_dev, float* grad, float* loss) {
  if (!m) return mlp_fail(nullptr, DE_ERR_INVALID_ARG, "handle is NULL");
  if (ld < kMlpIn) return mlp_fail(m, DE_ERR_INVALID_ARG, "ld must be >= 20");
  if (!mlp_dev_ptr(x_dev) || !mlp_dev_ptr(t_dev))
    return mlp_fail(m, DE_ERR_INVALID_ARG, "x_dev and t_dev must be device memory");
  MlpStepArgs a{m->seed, m->step, 0, 0, 1};
  mlp_step_launch(m->P, a, x_dev, ld, t_dev, 0.f, false, false, m->stream);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return mlp_fail(m, DE_ERR_CUDA, std::string("surrogate gradient: ") + cudaGetErrorString(e));
  de_status s = mlp_check(m);
  if (s != DE_OK) return s;
  if (grad) e = cudaMemcpyAsync(grad, m->P.grad, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess && loss) e = cudaMemcpyAsync(loss, m->P.loss, sizeof(float), cudaMemcpyDeviceToHost, m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) return mlp_fail(m, DE_ERR_CUDA, std::string("surrogate gradient: ") + cudaGetErrorString(e));
  return DE_OK;
}

de_status de_mlp_train(de_mlp* m, const double* x_dev, int64_t ld, const float* t_dev, int32_t n, int32_t steps,
                       float lr, float* loss) {
  if (!m) return mlp_fail(nullptr, DE_ERR_INVALID_ARG, "handle is NULL");
  if (n < 1 || steps < 0 || ld < kMlpIn || !(lr > 0.f) || !std::isfinite(lr))
    return mlp_fail(m, DE_ERR_INVALID_ARG, "need n >= 1, steps >= 0, ld >= 20 and a finite lr > 0");
  if (!mlp_dev_ptr(x_dev) || !mlp_dev_ptr(t_dev))
    return mlp_fail(m, DE_ERR_INVALID_ARG, "x_dev and t_dev must be device memory");
  de_status s = mlp_train_rows(m, x_dev, ld, t_dev, n, 0, n, steps, lr);
  if (s != DE_OK) return s;
  s = mlp_check(m);
  if (s != DE_OK) return s;
  if (loss) {
    cudaError_t e = cudaMemcpyAsync(loss, m->P.loss, sizeof(float), cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return mlp_fail(m, DE_ERR_CUDA, std::string("surrogate loss: ") + cudaGetErrorString(e));
  }
  return DE_OK;
}

}  // extern "C"
