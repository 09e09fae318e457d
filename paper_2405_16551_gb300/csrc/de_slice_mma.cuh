// de_slice_mma.cuh -- the digit products of de_slice.cuh on mma.sync, for
// rotations of at most 64 coordinates.
//
// The sums are the same integers as in tensor memory (exact in FP32 whatever
// the order), so z is the same bit for bit.  What differs is what a CTA holds:
// tensor memory belongs to one CTA per SM (its columns, and all of the SM's shared
// memory where CTAs wait for one another: fp64_exclusive_smem), and a tile is a
// chain of latencies (trials, digits, products, read-back, terms, sums) that one
// CTA of eight warps cannot hide.  Here the operands take 32 KB (d <= 32) or 94 KB
// (d <= 64) of shared memory and nothing else, so two or more CTAs share an SM,
// and at these widths the products themselves cost no more than the issue and
// commit of tcgen05.
#pragma once
#include <cuda_runtime.h>
#include <math_constants.h>

#include "de_device.cuh"
#include "de_internal.cuh"
#include "de_slice.cuh"

namespace de {

constexpr int kMmaDMax = 64;

// Width of the operand layout (32 or 64 coordinates), and its parts: y's digits
// as slice_digits writes them, M's digits [digit][8-coordinate group][output] of
// 16 bytes, the group sums [group][row][output] (4 floats between rows, so that
// the accumulators' stores meet no bank twice).
__host__ __device__ constexpr int mma_width(int kpad) { return kpad <= 32 ? 32 : 64; }
__host__ __device__ constexpr uint32_t mma_b_bytes(int kpad) { return (uint32_t)(mma_width(kpad) / 8) * kSliceKg; }
__host__ __device__ constexpr uint32_t mma_a_bytes(int kpad) {
  return (uint32_t)(kSlices * (mma_width(kpad) / 8) * mma_width(kpad)) * 16u;
}
__host__ __device__ constexpr int mma_pst(int kpad) { return mma_width(kpad) + 4; }
__host__ __device__ constexpr uint32_t mma_p_bytes(int kpad) { return 9u * kSliceRows * (uint32_t)mma_pst(kpad) * 4u; }
__host__ __device__ constexpr uint32_t mma_smem(int kpad) {
  return (mma_b_bytes(kpad) + mma_a_bytes(kpad) + mma_p_bytes(kpad) + 127u) / 128u * 128u;
}

__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, "
      "%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The sums of outputs 16 mt .. + 15 in one group, from the accumulators.
__device__ __forceinline__ void mma_put(float* P, int pst, int group, int mt, int lane, const float (&c)[4]) {
  float* p = P + (size_t)(group * kSliceRows + 2 * (lane & 3)) * pst + 16 * mt + (lane >> 2);
  p[0] = c[0];
  p[pst] = c[1];
  p[8] = c[2];
  p[pst + 8] = c[3];
}

// Width 32: the digit products of outputs 16 mt .. + 15 in groups G0 >= G1 >= G2
// (the pairs of digits s of y and t of M with s + t = g; -1: none).  Integers
// below 2^23 in FP32: exact.
template <int G0, int G1, int G2>
__device__ __forceinline__ void mma_products32(uint32_t sB, uint32_t sA, float* P, int mt, int lane) {
  const int i = lane >> 3, r = lane & 7;
  uint32_t b[kSlices][4];  // per digit of y: the 8-coordinate groups 0 .. 3
#pragma unroll
  for (int s = 0; s < kSlices; ++s)
    if (s <= G0) ldmatrix4(b[s], sB + (uint32_t)i * kSliceKg + (uint32_t)s * 128u + (uint32_t)r * 16u);
  float c[3][4] = {};
  const uint32_t a0 = sA + ((uint32_t)(i >> 1) * 32u + (uint32_t)(16 * mt + 8 * (i & 1) + r)) * 16u;
#pragma unroll
  for (int t = 0; t < kSlices; ++t) {
    if (t > G0) continue;
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      uint32_t a[4];
      ldmatrix4(a, a0 + (uint32_t)(t * 4 + 2 * ks) * 512u);
      if (G0 - t >= 0 && G0 - t < kSlices) mma_16816(c[0], a, b[(G0 - t) & 7][2 * ks], b[(G0 - t) & 7][2 * ks + 1]);
      if (G1 - t >= 0 && G1 - t < kSlices) mma_16816(c[1], a, b[(G1 - t) & 7][2 * ks], b[(G1 - t) & 7][2 * ks + 1]);
      if (G2 - t >= 0 && G2 - t < kSlices) mma_16816(c[2], a, b[(G2 - t) & 7][2 * ks], b[(G2 - t) & 7][2 * ks + 1]);
    }
  }
  constexpr int G[3] = {G0, G1, G2};
#pragma unroll
  for (int q = 0; q < 3; ++q)
    if (G[q] >= 0) mma_put(P, mma_pst(32), G[q], mt, lane, c[q]);
}

// Width 64: the groups of the set (21 of the 43 pairs of digits in 8, 7, 5,
// the other 22 in the others), K step by K step.
template <bool HIGH>
__device__ __forceinline__ void mma_products64(uint32_t sB, uint32_t sA, float* P, int mt, int ksteps, int lane) {
  constexpr int NG = HIGH ? 3 : 6;
  constexpr int G[6] = {HIGH ? 8 : 6, HIGH ? 7 : 4, HIGH ? 5 : 3, 2, 1, 0};
  const int i = lane >> 3, r = lane & 7;
  float c[NG][4] = {};
  const uint32_t b0 = sB + (uint32_t)(i & 1) * kSliceKg + (uint32_t)(i >> 1) * 128u + (uint32_t)r * 16u;
  const uint32_t a0 = sA + ((uint32_t)(i >> 1) * 64u + (uint32_t)(16 * mt + 8 * (i & 1) + r)) * 16u;
#pragma unroll 1
  for (int ks = 0; ks < ksteps; ++ks) {
    uint32_t b[kSlices / 2][4];  // digits 2 q, 2 q + 1 of y: the K step's two 8-coordinate groups
#pragma unroll
    for (int q = 0; q < kSlices / 2; ++q)
      if (2 * q <= G[0]) ldmatrix4(b[q], b0 + (uint32_t)(2 * ks) * kSliceKg + (uint32_t)q * 256u);
#pragma unroll
    for (int t = 0; t < kSlices; ++t) {
      if (t > G[0]) continue;
      uint32_t a[4];
      ldmatrix4(a, a0 + (uint32_t)(t * 8 + 2 * ks) * 1024u);
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        const int s = G[q] - t;
        if (s >= 0 && s < kSlices) mma_16816(c[q], a, b[(s & 7) >> 1][2 * (s & 1)], b[(s & 7) >> 1][2 * (s & 1) + 1]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < NG; ++q) mma_put(P, mma_pst(64), G[q], mt, lane, c[q]);
}

// The parts of a CTA's operands (mma_smem(kpad) bytes at smem, kpad the largest
// of the matrices it will load), the operand of y's digits zero; by all threads,
// which synchronise before the first digits (mma_load_m does).
__device__ __forceinline__ void mma_begin(SliceCtx& c, uint8_t* smem, int kpad, SliceShared& sh) {
  c.sh = &sh;
  c.sB = smem;
  c.sA = smem + mma_b_bytes(kpad);
  c.sP = reinterpret_cast<float*>(c.sA + mma_a_bytes(kpad));
  c.s_exp = sh.exp;
  c.s_bad = &sh.bad;
  c.cur = nullptr;
  if (threadIdx.x == 0) sh.bad = 0u;
  for (uint32_t q = threadIdx.x * 16u; q < mma_b_bytes(kpad); q += blockDim.x * 16u)
    *reinterpret_cast<uint4*>(smem + q) = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
}

// One matrix's digits into the layout of its own width; by all threads (256),
// without a barrier.
__device__ __forceinline__ void mma_copy_m(uint8_t* sA, const uint8_t* __restrict__ sl, int kpad) {
  const int nkg = kpad / 8;
  if (kpad <= 32) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = (int)threadIdx.x + 256 * u, t = e >> 7, kg = (e >> 5) & 3, r = e & 31;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (kg < nkg) v = __ldg(reinterpret_cast<const uint4*>(sl + (size_t)t * slice_bytes(kpad) + (size_t)kg * 2048u + r * 16));
      *reinterpret_cast<uint4*>(sA + (size_t)e * 16u) = v;
    }
  } else {
#pragma unroll 8
    for (int u = 0; u < 16; ++u) {
      const int e = (int)threadIdx.x + 256 * u, t = e >> 9, kg = (e >> 6) & 7, r = e & 63;
      if (kg < nkg)
        *reinterpret_cast<uint4*>(sA + (size_t)e * 16u) =
            __ldg(reinterpret_cast<const uint4*>(sl + (size_t)t * slice_bytes(kpad) + (size_t)kg * 2048u + r * 16));
    }
  }
}

__device__ __forceinline__ void mma_load_m(SliceCtx& c, const uint8_t* __restrict__ sl, int kpad) {
  __syncthreads();  // no product of the previous matrix is running
  mma_copy_m(c.sA, sl, kpad);
  __syncthreads();
  c.cur = sl;
}

// The products of the tile's digits with the loaded matrix, into the sums; by
// all threads (8 warps), after a CTA barrier that follows the digits.
__device__ __forceinline__ void mma_products(SliceCtx& c, int kpad, int d) {
  const int lane = threadIdx.x & 31;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
  const uint32_t sB = smem_u32(c.sB), sA = smem_u32(c.sA);
  if (kpad <= 32) {
    // a warp takes 16 outputs and 10 to 12 of the 43 pairs of digits
    if (16 * (warp & 1) < d) {
      switch (warp >> 1) {
        case 0: mma_products32<8, 3, -1>(sB, sA, c.sP, warp & 1, lane); break;
        case 1: mma_products32<7, 2, -1>(sB, sA, c.sP, warp & 1, lane); break;
        case 2: mma_products32<6, 1, 0>(sB, sA, c.sP, warp & 1, lane); break;
        default: mma_products32<5, 4, -1>(sB, sA, c.sP, warp & 1, lane); break;
      }
    }
  } else if (16 * (warp & 3) < d) {
    if (warp < 4) mma_products64<true>(sB, sA, c.sP, warp & 3, kpad / 16, lane);
    else mma_products64<false>(sB, sA, c.sP, warp & 3, kpad / 16, lane);
  }
  __syncthreads();
}

// z_j of the row whose digits this warp wrote, lane j holding z_j and
// z_{32 + j} (0 past d), after the products.  Yr: the row of y, for the DFMA
// chain where the row takes it (every term and their order as in slice_z).
__device__ __forceinline__ void mma_z(SliceCtx& c, const int32_t* __restrict__ fexp, const double* __restrict__ MT,
                                      const double* __restrict__ Yr, int kpad, int d, int warp, int lane,
                                      double (&z)[2]) {
  const int pst = mma_pst(kpad);
  const int e0 = c.s_exp[warp];
  const bool chain = (*(volatile uint32_t*)c.s_bad >> warp) & 1u;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int j = 32 * e + lane;
    z[e] = 0.0;
    if (32 * e >= d) continue;
    float p[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) p[q] = c.sP[(q * kSliceRows + warp) * pst + j];
    const double zj = slice_combine(p, e0 + (j < d ? __ldg(fexp + j) : 0) - 76);
    z[e] = j < d ? zj : 0.0;
  }
  if (chain) {
    __syncwarp();  // every lane has read the flag
    if (lane == 0) atomicAnd(c.s_bad, ~(1u << warp));
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int j = 32 * e + lane;
      double s = 0.0;
      if (j < d)
        for (int k = 0; k < d; ++k) s = fma(__ldg(MT + (size_t)k * d + j), Yr[k], s);
      z[e] = s;
    }
    __syncwarp();
  }
}

// Objective (0 .. 3) of a row, lane j holding z_j and z_{32 + j} (0 past d);
// every lane returns it.  The sums are those of slice_fitness: over the lanes of each
// 32 outputs, then over the 32s.
__device__ __forceinline__ double mma_objective(int obj, const double (&z)[2], int d, int lane) {
  double t[2] = {}, u[2] = {};
  const double first = obj == kObjRosenbrock ? __shfl_sync(0xffffffffu, z[1], 0) : 0.0;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int j = 32 * e + lane;
    if (32 * e >= d) continue;
    if (obj == kObjRosenbrock) {
      double zn = __shfl_down_sync(0xffffffffu, z[e], 1);
      if (e == 0 && lane == 31) zn = first;
      const double t0 = z[e] + 1.0, tn = zn + 1.0;
      const double a = tn - t0 * t0, b = t0 - 1.0;
      t[e] = j + 1 < d ? 100.0 * a * a + b * b : 0.0;
    } else if (obj == kObjRastrigin) {
      t[e] = fma(z[e], z[e], rastrigin_w(z[e]));
    } else {
      t[e] = z[e] * z[e];
      if (obj == kObjAckley) {
        const double w = cos2pi_fix(z[e]);
        u[e] = j < d ? w : 0.0;
      }
    }
  }
  double s1 = warp_sum(t[0]);
  if (d > 32) s1 += warp_sum(t[1]);
  if (obj != kObjAckley) return s1;
  double s2 = warp_sum(u[0]);
  if (d > 32) s2 += warp_sum(u[1]);
  return ackley_value((lane & 1 ? s2 : s1) / d, lane);
}

// slice_fitness of the tile's rows: warp r < nrows returns the fitness of row r
// (every lane).  Y: the tile's rows of y.
__device__ __forceinline__ double mma_fitness(SliceCtx& c, const RunDesc& R, const double* __restrict__ Y, int nrows) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  mma_products(c, R.sl_kpad, R.d);
  if (warp >= nrows) return 0.0;
  double z[2];
  mma_z(c, R.slx, R.MT, Y + warp * R.dp, R.sl_kpad, R.d, warp, lane, z);
  return mma_objective(R.obj, z, R.d, lane);
}

// slice_rotate: z into Z[r][j] (row stride dp) for the tile's rows.  The
// caller's CTA barrier makes Z visible.
__device__ __forceinline__ void mma_rotate(SliceCtx& c, int kpad, const int32_t* __restrict__ fexp,
                                           const double* __restrict__ MT, const double* __restrict__ Y,
                                           double* __restrict__ Z, int nrows, int d, int dp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  mma_products(c, kpad, d);
  if (warp >= nrows) return;
  double z[2];
  mma_z(c, fexp, MT, Y + warp * dp, kpad, d, warp, lane, z);
#pragma unroll
  for (int e = 0; e < 2; ++e)
    if (32 * e + lane < d) Z[warp * dp + 32 * e + lane] = z[e];
}

// How a kernel instance runs the sliced rotations of its runs: it has none; on
// tcgen05; on mma.sync (all of at most 64 coordinates).
enum SliceForm { kNoSlices = 0, kSliceTc = 1, kSliceMma = 2 };

template <int FORM>
__device__ __forceinline__ void form_begin(SliceCtx& c, uint8_t* smem, int kpad, uint32_t cols, SliceShared& sh) {
  if constexpr (FORM == kSliceMma) mma_begin(c, smem, kpad, sh);
  else slice_begin(c, smem, kpad, cols, sh);
}
template <int FORM>
__device__ __forceinline__ void form_end(SliceCtx& c) {
  if constexpr (FORM == kSliceTc) slice_end(c);
}
template <int FORM>
__device__ __forceinline__ void form_load_m(SliceCtx& c, const uint8_t* __restrict__ sl, int kpad) {
  if constexpr (FORM == kSliceMma) mma_load_m(c, sl, kpad);
  else slice_load_m(c, sl, kpad);
}
template <int FORM>
__device__ __forceinline__ double form_fitness(SliceCtx& c, const RunDesc& R, const double* __restrict__ Y,
                                               double* __restrict__ Zf, int nrows) {
  if constexpr (FORM == kSliceMma) return mma_fitness(c, R, Y, nrows);
  else return slice_fitness(c, R, Y, Zf, nrows);
}
template <int FORM>
__device__ __forceinline__ void form_rotate(SliceCtx& c, int kpad, const int32_t* __restrict__ fexp,
                                            const double* __restrict__ MT, const double* __restrict__ Y,
                                            double* __restrict__ Z, int nrows, int d, int dp) {
  if constexpr (FORM == kSliceMma) mma_rotate(c, kpad, fexp, MT, Y, Z, nrows, d, dp);
  else slice_rotate(c, kpad, fexp, MT, Y, Z, nrows, d, dp);
}
// shared memory of the operands
template <int FORM>
__host__ __device__ constexpr uint32_t form_smem(int kpad) {
  return FORM == kSliceMma ? mma_smem(kpad) : FORM == kSliceTc ? slice_smem(kpad) : 0u;
}

}  // namespace de
