// de_fp64_tc.cu -- FP64 kernels whose rotation runs as exact digit products on
// the tensor cores (de_slice.cuh on tcgen05, de_slice_mma.cuh on mma.sync):
//
//   k_slice_m       digit slices and row exponents of a run's matrices (once, at de_init)
//   k_gen_fp64_tc   one generation of the runs of one form: each CTA works
//                   through a contiguous share of the (run, tile) items and
//                   loads a run's matrix once
//   k_eval_rows_tc  f of caller rows: one matrix per CTA for all its tiles
//
// The persistent kernel's sliced instances are in de_fp64.cu.  All of them use
// the same tile routines, and the products are exact in either form, so a run's
// numbers do not depend on which one ran.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "de_common.cuh"
#include "de_device.cuh"
#include "de_gen_tile.cuh"
#include "de_internal.cuh"
#include "de_kernels.h"

namespace de {

// One CTA (128 threads) per row of the 128-row operand: thread k holds M_jk.
__global__ void __launch_bounds__(128) k_slice_m(const double* __restrict__ MT, int d, int kpad, uint8_t* __restrict__ sl,
                                                 int32_t* __restrict__ fexp) {
  const int c = blockIdx.y, j = blockIdx.x, k = threadIdx.x;
  __shared__ uint32_t s_mx[4];
  const double m = j < d && k < d ? MT[(size_t)c * d * d + (size_t)k * d + j] : 0.0;
  const uint32_t hw = (uint32_t)__double2hiint(m) & 0x7FFFFFFFu;
  const uint32_t w = __reduce_max_sync(0xffffffffu, hw);
  if ((k & 31) == 0) s_mx[k >> 5] = w;
  __syncthreads();
  const int ex = (int)(max(max(s_mx[0], s_mx[1]), max(s_mx[2], s_mx[3])) >> 20);
  if (k == 0) fexp[c * kSliceDMax + j] = ex - 1022;
  if (k >= kpad) return;
  const long long b = __double_as_longlong(m);
  const int ek = (int)(hw >> 20), sh = ex - ek;
  unsigned long long u = (((unsigned long long)b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL) << 9;
  if (ek == 0 || sh > 62) u = 0ULL;
  else if (sh > 0) u = (u + (1ULL << (sh - 1))) >> sh;
  const unsigned long long v = (unsigned long long)(b < 0 ? -(long long)u : (long long)u) + 0x8080808080808080ULL;
  uint8_t* dst = sl + (size_t)c * kSlices * slice_bytes(kpad) + (size_t)(k >> 3) * 2048u + (size_t)j * 16u + (size_t)(k & 7) * 2u;
  for (int t = 0; t < kSlices; ++t) {
    const int digit = (int)((v >> (56 - 8 * t)) & 0xFFu) - 128;
    *reinterpret_cast<__nv_bfloat16*>(dst + (size_t)t * slice_bytes(kpad)) = __float2bfloat16_rn((float)digit);
  }
}

// Shared memory: operands of the sliced rotation (op bytes), then the tile
// buffers.  shares: per CTA the items [x, y).
constexpr int kCompGroup = 64;  // rows of a composition function per matrix load

template <bool VAR, bool SUITE, int FORM>
__global__ void __launch_bounds__(256, FORM == kSliceMma ? 2 : 1)
    k_gen_fp64_tc(const RunDesc* __restrict__ runs, const int4* __restrict__ items, const int2* __restrict__ shares,
                  int kpad, uint32_t cols) {
  extern __shared__ __align__(1024) uint8_t smem_tc[];
  __shared__ SliceShared s_sl;
  __shared__ RunDesc sR;
  __shared__ int s_stop, s_last, s_best;
  __shared__ long long s_gen;
  __shared__ double s_bf[8];
  __shared__ long long s_bk[8];
  __shared__ int s_bi[8];
  __shared__ double s_fsuite[SUITE ? kCompGroup : 1];
  __shared__ double s_comp[SUITE ? kCompGroup : 1][10];
  double* sm = reinterpret_cast<double*>(smem_tc + form_smem<FORM>(kpad));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nwarps = blockDim.x >> 5;
  const int2 share = shares[blockIdx.x];
  SliceCtx sc;
  form_begin<FORM>(sc, smem_tc, kpad, cols, s_sl);
  // only now: the next generation's CTAs must not take tensor memory that a
  // CTA of this one still waits for
  pdl_launch_dependents();
  pdl_wait();
  for (int i = share.x; i < share.y;) {
    const int4 it = items[i];
    // the items of this run in this CTA's share
    int e = i + 1;
    while (e < share.y && items[e].x == it.x) ++e;
    __syncthreads();
    load_desc(sR, runs + it.x);
    __syncthreads();
    const RunDesc& R = sR;
    RunState* st = R.st;
    if (tid == 0) {
      s_stop = *(volatile int32_t*)&st->stop;
      s_gen = *(volatile int64_t*)&st->gen;
      s_best = max(*(volatile int32_t*)&st->best_idx, 0);
    }
    __syncthreads();
    if (s_stop) {
      i = e;
      continue;
    }
    const int64_t g = s_gen + 1;
    Best bb;
    bb.init();
    if (SUITE && R.sl && R.obj >= kObjComposition1) {
      // a matrix is loaded once for a group of rows, not per tile
      const int cur = (int)((g - 1) & 1), dp = R.dp;
      const bool var = VAR && (R.strategy != 0 || R.jde);
      const double* jFc = VAR && R.jde ? R.jF[cur] : nullptr;
      const double* jCRc = VAR && R.jde ? R.jCR[cur] : nullptr;
      const int row_end = items[e - 1].z + items[e - 1].w;
      double* Y = sm;                       // 8 x dp; also takes the trials' shifted rows, which are not used
      double* Z = Y + kSliceRows * dp;      // 8 x dp
      double* T = Z + kSliceRows * dp;      // kCompGroup x dp
      for (int row0 = it.z; row0 < row_end; row0 += kCompGroup) {
        const int nr = min(kCompGroup, row_end - row0);
        for (int r = warp; r < nr; r += nwarps) {
          if (var)
            build_trial_row<true>(R, R.X[cur], (uint32_t)(row0 + r), g, lane, T + r * dp, Y + warp * dp, s_best, jFc, jCRc);
          else
            build_trial_row<false, true>(R, R.X[cur], (uint32_t)(row0 + r), g, lane, T + r * dp, Y + warp * dp);
        }
        __syncthreads();
        suite_comp_sliced<FORM>(R, T, dp, nr, Y, Z, s_fsuite, s_comp, sc);
        for (int r = warp; r < nr; r += nwarps)
          bb.offer(gen_select<VAR>(R, g, row0 + r, s_fsuite[r], T + r * dp, lane), row0 + r);
        __syncthreads();
      }
    } else {
      for (int k = i; k < e; ++k) {
        const int4 t = items[k];
        const Best b = gen_tile<VAR, SUITE, FORM>(R, g, t.z, t.w, R.rows, s_best, sm, s_fsuite, s_comp, &sc);
        bb.take(b.f, b.k, b.i);
        __syncthreads();
      }
    }
    if (lane == 0) { s_bf[warp] = bb.f; s_bk[warp] = bb.k; s_bi[warp] = bb.i; }
    __syncthreads();
    if (tid == 0) {
      bb.init();
      for (int w = 0; w < nwarps; ++w) bb.take(s_bf[w], s_bk[w], s_bi[w]);
      // one partial for the share's tiles of this run; the other slots hold none
      for (int k = i; k < e; ++k) {
        R.part[items[k].y].f = k == i ? bb.f : CUDART_INF;
        R.part[items[k].y].idx = k == i ? bb.i : -1;
      }
      if (FORM == kSliceTc && *sc.s_fail) atomicOr(&st->err, kErrTimeout);
      __threadfence();
      const uint32_t n = (uint32_t)(e - i);
      s_last = atomicAdd(&st->ticket, n) + n == (uint32_t)R.ntiles;
    }
    __syncthreads();
    if (s_last) {
      __threadfence();
      finish_generation(R, g, R.ntiles, R.part, R.X[g & 1]);
    }
    i = e;
  }
  form_end<FORM>(sc);
}

// f of rows r0 .. r1 - 1 of x (row stride ld) with a sliced run; a warp per row
// of the 8-row tiles.  Y, Z: 8 x dp doubles, ncomp times that (a composition
// function's, when the rows are at most 8).
template <int FORM>
__device__ __forceinline__ void eval_sliced(const RunDesc& R, SliceCtx& sc, const double* __restrict__ x, int64_t ld,
                                            int r0, int r1, double* __restrict__ fout, uint8_t* __restrict__ fx_out,
                                            double* Y, double* s_f, double (*s_comp)[10], int ncomp) {
  const int d = R.d, dp = R.dp, obj = R.obj, kpad = R.sl_kpad;
  double* Z = Y + ncomp * kSliceRows * dp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool suite = suite_objective(obj);
  const int step = suite && obj >= kObjComposition1 ? kCompGroup : kSliceRows;
  for (int row0 = r0; row0 < r1; row0 += step) {
    const int nr = min(step, r1 - row0);
    if (suite) {
      suite_tile<FORM>(R, x + (size_t)row0 * ld, ld, nr, Y, Z, s_f, s_comp, &sc, ncomp == 1);
      for (int r = threadIdx.x; r < nr; r += blockDim.x) {
        fout[row0 + r] = s_f[r];
        if (fx_out) fx_out[row0 + r] = 1;
      }
      __syncthreads();
      continue;
    }
    if (warp < nr) {
      const double* xr = x + (size_t)(row0 + warp) * ld;
      double y[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
      for (int m = 0; m < 4; ++m)
        if (4 * lane + m < d) y[m] = shifted(xr[4 * lane + m], R.o[4 * lane + m], R);
      if (4 * lane < dp) {
        *reinterpret_cast<double2*>(Y + warp * dp + 4 * lane) = make_double2(y[0], y[1]);
        *reinterpret_cast<double2*>(Y + warp * dp + 4 * lane + 2) = make_double2(y[2], y[3]);
      }
      slice_digits(sc, warp, lane, kpad, R.sl_qmin[0], y);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    if (sc.cur != R.sl) form_load_m<FORM>(sc, R.sl, kpad);
    const double f = form_fitness<FORM>(sc, R, Y, Z, nr);
    if (warp < nr) {
      if (lane == 0) {
        fout[row0 + warp] = f;
        if (fx_out) fx_out[row0 + warp] = 1;
      }
    }
  }
  // a wait that gave up (it should not on a healthy device) cannot be
  // returned by this launch: the rows come back as NaN, the run is marked
  __syncthreads();
  if (FORM == kSliceTc && *sc.s_fail) {
    for (int r = r0 + (int)threadIdx.x; r < r1; r += blockDim.x) fout[r] = CUDART_NAN;
    if (threadIdx.x == 0) atomicOr(&R.st->err, kErrTimeout);
  }
}

// n rows of x with run `run`'s objective, in contiguous shares of whole tiles.
template <int FORM>
__global__ void __launch_bounds__(256, FORM == kSliceMma ? 2 : 1)
    k_eval_rows_tc(const RunDesc* __restrict__ runs, int run, const double* __restrict__ x, int64_t ld, int n,
                   double* __restrict__ fout, uint8_t* __restrict__ fx_out, int kpad, uint32_t cols, int ncomp) {
  extern __shared__ __align__(1024) uint8_t smem_tc[];
  __shared__ SliceShared s_sl;
  __shared__ RunDesc sR;
  __shared__ double s_f[kCompGroup];
  __shared__ double s_comp[kCompGroup][10];
  load_desc(sR, runs + run);
  SliceCtx sc;
  form_begin<FORM>(sc, smem_tc, kpad, cols, s_sl);
  double* Y = reinterpret_cast<double*>(smem_tc + form_smem<FORM>(kpad));
  const int tiles = (n + kSliceRows - 1) / kSliceRows;
  const int r0 = (int)((long long)tiles * blockIdx.x / gridDim.x) * kSliceRows;
  const int r1 = min(n, (int)((long long)tiles * (blockIdx.x + 1) / gridDim.x) * kSliceRows);
  eval_sliced<FORM>(sR, sc, x, ld, r0, r1, fout, fx_out, Y, s_f, s_comp, ncomp);
  form_end<FORM>(sc);
}

// The populations X[0] of the sliced runs, in the shares of k_gen_fp64_tc.
template <int FORM>
__global__ void __launch_bounds__(256, FORM == kSliceMma ? 2 : 1)
    k_eval_pops_tc(const RunDesc* __restrict__ runs, const int4* __restrict__ items, const int2* __restrict__ shares,
                   int kpad, uint32_t cols) {
  extern __shared__ __align__(1024) uint8_t smem_tc[];
  __shared__ SliceShared s_sl;
  __shared__ RunDesc sR;
  __shared__ double s_f[kCompGroup];
  __shared__ double s_comp[kCompGroup][10];
  SliceCtx sc;
  form_begin<FORM>(sc, smem_tc, kpad, cols, s_sl);
  double* Y = reinterpret_cast<double*>(smem_tc + form_smem<FORM>(kpad));
  const int2 share = shares[blockIdx.x];
  for (int i = share.x; i < share.y;) {
    int e = i + 1;
    while (e < share.y && items[e].x == items[i].x) ++e;
    __syncthreads();
    load_desc(sR, runs + items[i].x);
    __syncthreads();
    if (sR.sl)
      eval_sliced<FORM>(sR, sc, sR.X[0], sR.dp, items[i].z, items[e - 1].z + items[e - 1].w, sR.f[0], sR.fx[0], Y, s_f, s_comp, 1);
    i = e;
  }
  form_end<FORM>(sc);
}

// ------------------------------------------------------------------ host side
// Whether the rotations of a run can be sliced, and the least count of large
// coordinates a row needs per matrix (de_slice.cuh).  M: nc row-major d x d
// matrices.
bool slice_plan(const double* M, int nc, int d, int32_t qmin[5]) {
  // below 16 coordinates the chain of d DFMAs is shorter than the products' latency
  if (d < kSliceDMin || d > kSliceDMax) return false;
  for (int c = 0; c < nc; ++c) {
    int cm = 0;
    for (int j = 0; j < d; ++j) {
      const double* row = M + ((size_t)c * d + j) * d;
      double mx = 0.0, sum = 0.0;
      for (int k = 0; k < d; ++k) {
        mx = std::max(mx, std::fabs(row[k]));
        sum += std::fabs(row[k]);
      }
      if (!(mx > 0x1p-100 && mx < 0x1p100)) return false;
      int small = 0;
      for (int k = 0; k < d; ++k) small += std::fabs(row[k]) < 0.125 * mx;
      cm = std::max(cm, small);
      // the leading digits' products sum below 2^19 (H below 2^51): |v_0,jk| <=
      // 64 |M_jk| / 2^f_j + 1 and |u_0| <= 64
      int f;
      std::frexp(mx, &f);
      if (64.0 * std::ldexp(sum, -f) + d > 8000.0) return false;
    }
    qmin[c] = cm + (d + 7) / 8;
    if (4 * qmin[c] > 3 * d) return false;
  }
  return true;
}

size_t slice_matrix_bytes(int d) { return (size_t)kSlices * slice_bytes(slice_kpad(d)); }

void k_slice_m_launch(const double* MT, int nc, int d, uint8_t* sl, int32_t* fexp, cudaStream_t s) {
  k_slice_m<<<dim3(kSliceDMax, (unsigned)nc), 128, 0, s>>>(MT, d, slice_kpad(d), sl, fexp);
}

int slice_kpad_of(int d) { return slice_kpad(d); }
uint32_t slice_kernel_cols(int kpad) { return slice_tmem_cols(kpad); }
// mma.sync up to 64 coordinates, the widest whose operands leave room for two
// CTAs on an SM.  On tcgen05 there is one, and a tile of short rows is a chain of
// latencies: a generation (us, tcgen05 -> mma.sync) of NP = 1500 at D = 16 / 40 /
// 64 took 25.7 / 24.0 / 24.7 -> 10.1 / 12.3 / 12.9 (that many tiles do not fit
// k_gen_sliced), of 60 uneven runs 713 -> 306, of 48 runs of NP = 500, D = 30
// 181 -> 82; 16384 rows of Zakharov's function at D = 30 113 -> 64.
int slice_form(int kpad) { return kpad <= kMmaDMax ? kSliceMma : kSliceTc; }
size_t slice_form_smem(int form, int kpad) { return form == kSliceMma ? mma_smem(kpad) : slice_smem(kpad); }
size_t slice_group_smem(int dp) { return (size_t)(2 * kSliceRows + kCompGroup) * dp * sizeof(double); }
static_assert(kSliceExp == kSliceDMax, "row exponents per matrix");

template <int FORM>
static const void* gen_kernel_of(bool var, bool suite) {
  return var && suite ? (const void*)k_gen_fp64_tc<true, true, FORM>
         : var        ? (const void*)k_gen_fp64_tc<true, false, FORM>
         : suite      ? (const void*)k_gen_fp64_tc<false, true, FORM>
                      : (const void*)k_gen_fp64_tc<false, false, FORM>;
}
static const void* gen_kernel(int form, bool var, bool suite) {
  return form == kSliceMma ? gen_kernel_of<kSliceMma>(var, suite) : gen_kernel_of<kSliceTc>(var, suite);
}

int k_gen_fp64_tc_per_sm(const SlicePlan& p, bool var, bool suite) {
  int n = 0;
  const void* k = gen_kernel(p.form, var, suite);
  if (allow_dynamic_smem(k) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, 256, p.smem) != cudaSuccess)
    cudaGetLastError();
  // (at least one: a launch that does not fit reports it)
  return std::max(1, p.form == kSliceTc ? std::min(n, (int)(512u / p.cols)) : n);
}

void k_gen_fp64_tc_launch(const RunDesc* runs, const int4* items, const int2* shares, int nct, const SlicePlan& p,
                          bool var, bool suite, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)nct);
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int kpad = p.kpad;
  uint32_t cols = p.cols;
  void* args[] = {(void*)&runs, (void*)&items, (void*)&shares, (void*)&kpad, (void*)&cols};
  cudaLaunchKernelExC(&cfg, gen_kernel(p.form, var, suite), args);
}

void k_tc_configure() {
  for (int q = 0; q < 8; ++q) allow_dynamic_smem(gen_kernel(q & 4 ? kSliceMma : kSliceTc, q & 1, (q & 2) != 0));
  for (const void* k : {(const void*)k_eval_rows_tc<kSliceTc>, (const void*)k_eval_rows_tc<kSliceMma>,
                        (const void*)k_eval_pops_tc<kSliceTc>, (const void*)k_eval_pops_tc<kSliceMma>})
    allow_dynamic_smem(k);
}

void k_eval_pops_tc_launch(const RunDesc* runs, const int4* items, const int2* shares, int nct, const SlicePlan& p,
                           cudaStream_t s) {
  const size_t smem = p.smem_op + (size_t)2 * kSliceRows * p.dp_max * sizeof(double);
  if (p.form == kSliceMma) k_eval_pops_tc<kSliceMma><<<nct, 256, smem, s>>>(runs, items, shares, p.kpad, p.cols);
  else k_eval_pops_tc<kSliceTc><<<nct, 256, smem, s>>>(runs, items, shares, p.kpad, p.cols);
}

void k_eval_rows_tc_launch(const RunDesc* runs, int run, const RunDesc& Rh, const double* x, int64_t ld, int n,
                           double* f, uint8_t* fx, cudaStream_t s) {
  int dev = 0, nsm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int kpad = Rh.sl_kpad, form = slice_form(kpad);
  const uint32_t cols = slice_tmem_cols(kpad);
  const int per_sm = form == kSliceMma ? 2 : 1;
  const int tiles = (n + kSliceRows - 1) / kSliceRows, grid = std::min(tiles, nsm * per_sm);
  // a composition function's components side by side where no CTA has a second
  // tile (on tcgen05 the loads of the matrices are the longer part: no gain)
  const int ncomp = form == kSliceMma && tiles <= grid ? suite_comps(Rh) : 1;
  const size_t smem = slice_form_smem(form, kpad) + (size_t)2 * ncomp * kSliceRows * Rh.dp * sizeof(double);
  if (form == kSliceMma) k_eval_rows_tc<kSliceMma><<<grid, 256, smem, s>>>(runs, run, x, ld, n, f, fx, kpad, cols, ncomp);
  else k_eval_rows_tc<kSliceTc><<<grid, 256, smem, s>>>(runs, run, x, ld, n, f, fx, kpad, cols, ncomp);
}

}  // namespace de
