// de_gen_tile.cuh -- one tile (at most 8 targets) of an FP64 generation: trials,
// rotation, objective, greedy selection.  Shared by the per-generation
// kernels and the persistent one.
#pragma once
#include <cuda_runtime.h>
#include <math_constants.h>

#include "de_common.cuh"
#include "de_device.cuh"
#include "de_internal.cuh"
#include "de_slice_mma.cuh"
#include "de_suite.cuh"

namespace de {

// Q groups of 32 flattened outputs (row r, coordinate j) of the tile's
// rotation, one per accumulator chain: z[r][j] = sum_k M^T[k][j] y[r][k].
template <int Q>
__device__ __forceinline__ void rotate_groups(const RunDesc& R, const double* __restrict__ Y, double* __restrict__ Z,
                                              int w0, int stride, int lane, int nout, int dp) {
  const int d = R.d;
  int rr[Q], jj[Q];
  bool ok[Q];
  double acc[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int e = (w0 + q * stride) * 32 + lane;
    ok[q] = e < nout;
    const int ec = ok[q] ? e : nout - 1;
    rr[q] = ec / d;
    jj[q] = ec - rr[q] * d;
    acc[q] = 0.0;
  }
  for (int k = 0; k < d; ++k) {
    const double* mk = R.MT + (size_t)k * d;
#pragma unroll
    for (int q = 0; q < Q; ++q) acc[q] = fma(__ldg(mk + jj[q]), Y[rr[q] * dp + k], acc[q]);
  }
#pragma unroll
  for (int q = 0; q < Q; ++q)
    if (ok[q]) Z[rr[q] * dp + jj[q]] = acc[q];
}

// Greedy selection of target i against its trial (row Trow, fitness ft), into
// the other population buffer; one warp.  Returns the fitness kept.
template <bool VAR>
__device__ __forceinline__ double gen_select(const RunDesc& R, int64_t g, int i, double ft, const double* Trow,
                                             int lane) {
  const int cur = (int)((g - 1) & 1), nxt = cur ^ 1;
  const double* X = R.X[cur];
  double* __restrict__ Xn = R.X[nxt];
  const double* fX = R.f[cur];
  double* __restrict__ fn = R.f[nxt];
  const int dp = R.dp;
  const double* jFc = VAR && R.jde ? R.jF[cur] : nullptr;
  const double* jCRc = VAR && R.jde ? R.jCR[cur] : nullptr;
  const double fi = __ldcg(fX + i);
  const bool acc = fit_key(ft) <= fit_key(fi) && fit_key(ft) != 0x7FFFFFFFFFFFFFFFLL;  // ft <= fi, NaN never
  double2* dst = reinterpret_cast<double2*>(Xn + (size_t)i * dp);
  if (acc) {
    const double2* src = reinterpret_cast<const double2*>(Trow);
    for (int j = lane; j < dp / 2; j += 32) dst[j] = src[j];
  } else {
    const double2* src = reinterpret_cast<const double2*>(X + (size_t)i * dp);
    for (int j = lane; j < dp / 2; j += 32) dst[j] = __ldcg(src + j);
  }
  const double fnew = acc ? ft : fi;
  if (VAR && R.jde && lane == 0) {
    // jDE: an accepted trial passes its F_i and CR_i on
    double Fi = __ldcg(jFc + i), CRi = __ldcg(jCRc + i);
    if (acc) jde_params(R, (uint32_t)i, g, jFc, jCRc, Fi, CRi);
    R.jF[nxt][i] = Fi;
    R.jCR[nxt][i] = CRi;
  }
  if (lane == 0) {
    fn[i] = fnew;
    if (R.dbg_ftrial) {
      R.dbg_ftrial[i] = ft;
      R.dbg_accept[i] = acc ? 1 : 0;
      R.dbg_fp64[i] = 1;
    }
  }
  return fnew;
}

// The trials of targets row0 .. row0 + nrows - 1 (a warp per target) into T, their
// shifted rows into Y.
template <bool VAR>
__device__ __forceinline__ void gen_trials(const RunDesc& R, int64_t g, int row0, int nrows, int best, double* T,
                                           double* Y) {
  const int cur = (int)((g - 1) & 1), dp = R.dp;
  const double* X = R.X[cur];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  const bool var = VAR && (R.strategy != 0 || R.jde);
  const double* jFc = VAR && R.jde ? R.jF[cur] : nullptr;
  const double* jCRc = VAR && R.jde ? R.jCR[cur] : nullptr;
  if (var) {
    for (int rl = warp; rl < nrows; rl += nwarps)
      build_trial_row<true>(R, X, (uint32_t)(row0 + rl), g, lane, T + rl * dp, Y + rl * dp, best, jFc, jCRc);
  } else if (R.unit_scale) {
    // a unit domain scale: no multiplication on the FP64 pipe (the compiler
    // would otherwise run it speculatively)
    for (int rl = warp; rl < nrows; rl += nwarps)
      build_trial_row<false, true>(R, X, (uint32_t)(row0 + rl), g, lane, T + rl * dp, Y + rl * dp);
  } else {
    for (int rl = warp; rl < nrows; rl += nwarps)
      build_trial_row<false>(R, X, (uint32_t)(row0 + rl), g, lane, T + rl * dp, Y + rl * dp);
  }
}

// One tile of generation g: the trials of targets row0 .. row0 + nrows - 1
// (a warp per target), their fitness, and greedy selection into the other
// population buffer.  Shared memory sm: T (trials), Y (shifted trials), Z
// (rotated), W (second term sum of Ackley), each rows_max x dp doubles.
// best: the current population's best row (DE/best/1).  Returns the calling
// warp's best (f, index) over the tile's new population rows (the same in
// every lane).  Population rows, fitness and jDE parameters of generation
// g - 1 are read at L2.
// VAR / SUITE: strategy variants and jDE / the benchmark suite's objectives.
// FORM: whether and how a run's rotation may be sliced (R.sl != NULL then).
template <bool VAR, bool SUITE, int FORM = kNoSlices>
__device__ __forceinline__ Best gen_tile(const RunDesc& R, int64_t g, int row0, int nrows, int rows_max, int best,
                                         double* sm, double* s_fsuite, double (*s_comp)[10], SliceCtx* sc = nullptr) {
  const int d = R.d, dp = R.dp;
  double* T = sm;
  double* Y = T + rows_max * dp;
  double* Z = Y + rows_max * dp;
  double* W = Z + rows_max * dp;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nwarps = blockDim.x >> 5;

  gen_trials<VAR>(R, g, row0, nrows, best, T, Y);
  const bool suite = SUITE && suite_objective(R.obj);
  const bool sliced = FORM != kNoSlices && R.sl != nullptr && !suite;
  if (sliced && warp < nrows) {
    // the digits of the row this warp built, as few coordinates a lane as the
    // width allows
    const double* yr = Y + warp * dp;
    if (FORM == kSliceMma && R.sl_kpad <= 32) {
      __syncwarp();
      const double y[1] = {lane < d ? yr[lane] : 0.0};
      slice_digits(*sc, warp, lane, R.sl_kpad, R.sl_qmin[0], y);
    } else if (FORM == kSliceMma) {
      __syncwarp();
      const double y[2] = {2 * lane < d ? yr[2 * lane] : 0.0, 2 * lane + 1 < d ? yr[2 * lane + 1] : 0.0};
      slice_digits(*sc, warp, lane, R.sl_kpad, R.sl_qmin[0], y);
    } else {
      // (its lanes wrote these coordinates)
      double y[4] = {0.0, 0.0, 0.0, 0.0};
      if (4 * lane < d) {
#pragma unroll
        for (int m = 0; m < 4; ++m) y[m] = yr[4 * lane + m];
      }
      slice_digits(*sc, warp, lane, R.sl_kpad, R.sl_qmin[0], y);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();

  const int nout = nrows * d;
  double fsl = 0.0;
  if (sliced) {
    if (sc->cur != R.sl) form_load_m<FORM>(*sc, R.sl, R.sl_kpad);
    fsl = form_fitness<FORM>(*sc, R, Y, Z, nrows);
  } else if (suite) {
    // ---- the proposed benchmark's functions (Sec. 7.3, Table 2)
    const int ncomp = R.obj >= kObjComposition1 ? R.nc : 1;  // Y and Z hold every component of the tile
    suite_tile<FORM>(R, T, dp, nrows, Y, Y + (size_t)ncomp * rows_max * dp, s_fsuite, s_comp, sc);
  } else if (R.obj == kObjOde) {
    // ---- ODE objective: a warp integrates one trial's chain; f to W[row][0]
    for (int rl = warp; rl < nrows; rl += nwarps) {
      const double s = warp_sum(ode_chain(T + rl * dp, lane, R.ode_ref, nullptr));
      if (lane == 0) W[rl * dp] = s / (double)(kOdeSteps * kOdeN);
    }
    __syncthreads();
  } else {
    // ---- rotation, flattened over (row, output): output e = 32 w + lane of
    // warp-group w; a warp takes groups warp, warp + 8, ... and runs up to four
    // of them at once (independent accumulator chains)
    if (R.rotate) {
      const int ngroups = (nout + 31) / 32;
      for (int w0 = warp; w0 < ngroups; w0 += 4 * nwarps) {
        const int qn = min(4, (ngroups - w0 + nwarps - 1) / nwarps);  // uniform in the warp
        if (qn == 4) rotate_groups<4>(R, Y, Z, w0, nwarps, lane, nout, dp);
        else if (qn == 3) rotate_groups<3>(R, Y, Z, w0, nwarps, lane, nout, dp);
        else if (qn == 2) rotate_groups<2>(R, Y, Z, w0, nwarps, lane, nout, dp);
        else rotate_groups<1>(R, Y, Z, w0, nwarps, lane, nout, dp);
      }
    } else {
      for (int e = tid; e < nout; e += blockDim.x) {
        const int r = e / d, j = e - r * d;
        Z[r * dp + j] = Y[r * dp + j];
      }
    }
    __syncthreads();

    // ---- objective terms, flattened; Y and W receive the per-coordinate terms
    for (int e = tid; e < nout; e += blockDim.x) {
      const int r = e / d, j = e - r * d;
      const double z = Z[r * dp + j];
      double t1 = 0.0, t2 = 0.0;
      if (R.obj == kObjSphere) {
        t1 = z * z;
      } else if (R.obj == kObjRastrigin) {
        t1 = fma(z, z, rastrigin_w(z));
      } else if (R.obj == kObjAckley) {
        t1 = z * z;
        t2 = cos2pi_fix(z);
      } else if (R.obj == kObjRosenbrock) {
        if (j + 1 < d) {
          const double t0 = z + 1.0, tn = Z[r * dp + j + 1] + 1.0;
          const double a = tn - t0 * t0, b = t0 - 1.0;
          t1 = 100.0 * a * a + b * b;
        }
      } else {
        t1 = CUDART_NAN;
      }
      Y[r * dp + j] = t1;
      W[r * dp + j] = t2;
    }
    __syncthreads();
  }

  // ---- row sums, greedy selection, best partial (a warp per row)
  Best bb;
  bb.init();
  for (int rl = warp; rl < nrows; rl += nwarps) {
    const int i = row0 + rl;
    double ft;
    if (sliced) {
      ft = fsl;
    } else if (suite) {
      ft = s_fsuite[rl];
    } else if (R.obj == kObjOde) {
      ft = W[rl * dp];
    } else {
      double s1 = 0.0, s2 = 0.0;
      for (int j = lane; j < d; j += 32) {
        s1 += Y[rl * dp + j];
        s2 += W[rl * dp + j];
      }
      s1 = warp_sum(s1);
      s2 = warp_sum(s2);
      ft = R.obj == kObjAckley ? 20.0 + 2.718281828459045 - 20.0 * exp(-0.2 * sqrt(s1 / d)) - exp(s2 / d) : s1;
    }
    const double fnew = gen_select<VAR>(R, g, i, ft, T + rl * dp, lane);
    bb.offer(fnew, i);
  }
  return bb;
}

// The tile of a composition function whose components run on CTAs of their own,
// in two steps with a barrier of all of them between: component c's part, and
// (one of the CTAs) the mix and the selection from all parts.  sm: T, Y, Z.
template <bool VAR, int FORM>
__device__ __forceinline__ void gen_comp_part(const RunDesc& R, int64_t g, int row0, int nrows, int rows_max, int best,
                                              double* sm, int c, SliceCtx& sc) {
  double* Y = sm + rows_max * R.dp;
  gen_trials<VAR>(R, g, row0, nrows, best, sm, Y);
  __syncthreads();
  suite_comp_part<FORM>(R, sm, R.dp, row0, nrows, Y, Y + rows_max * R.dp, c, sc);
}
template <bool VAR>
__device__ __forceinline__ Best gen_comp_finish(const RunDesc& R, int64_t g, int row0, int nrows, const double* T,
                                                double* s_f, double (*s_comp)[10]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  for (int e = threadIdx.x; e < nrows * R.nc; e += blockDim.x) {
    const int r = e / R.nc, c = e - r * R.nc;
    const double2 v = __ldcg(R.cpart + (size_t)(row0 + r) * 5 + c);
    s_comp[r][c] = v.x;
    s_comp[r][5 + c] = v.y;
  }
  __syncthreads();
  comp_mix(R, s_comp, s_f, nrows);
  Best bb;
  bb.init();
  for (int r = warp; r < nrows; r += nwarps)
    bb.offer(gen_select<VAR>(R, g, row0 + r, s_f[r], T + r * R.dp, lane), row0 + r);
  return bb;
}

// Copy of a run descriptor into shared memory (its fields are read in every
// phase, after barriers that would force global reloads).
__device__ __forceinline__ void load_desc(RunDesc& sR, const RunDesc* src) {
  for (int q = threadIdx.x; q < (int)(sizeof(RunDesc) / 8); q += blockDim.x)
    reinterpret_cast<uint64_t*>(&sR)[q] = reinterpret_cast<const uint64_t*>(src)[q];
}

}  // namespace de
