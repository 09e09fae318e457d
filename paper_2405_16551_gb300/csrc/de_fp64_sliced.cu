// de_fp64_sliced.cu -- the FP64 generation loop of plain DE/rand/1/bin runs
// whose rotations are sliced (de_slice.cuh), as one cooperative launch.
//
// CTA t owns item t's targets (at most 8, a warp each) for every generation.
// With the rotation and the cosines off the FP64 pipe a generation is a chain of
// latencies (NP = 1024, D = 100, cycles before this kernel, which ran the
// general tile routine: trials 4.2 k, digits 1.8 k, products 5.9 k, terms 3.5 k,
// sums and selection 6.0 k, barrier 3.0 k, best record 3.7 k), so it is arranged
// to shorten that chain:
//   - a target's row and fitness stay in its warp's registers: selection reads
//     nothing back, and trials load only the three donors;
//   - the draws of the next generation (indices, j_rand, crossover block: they
//     depend on (seed, generation, target) only) are made while the products
//     run;
//   - the digits are cut from the registers that hold y, and the terms are
//     computed by the thread that holds z (slice_fitness);
//   - the best record and the stop rule of the previous generation are
//     reduced beside the trials (by the warp without a target, if there is one),
//     with three warp-wide integer minima in place of a shuffle tree; nothing of
//     a generation is written before its stop decision.
// The generation's numbers are those of the general kernels (gen_tile): the
// same trial and fitness routines, the same selection.
//
// Barriers and the runs' stop counting are those of k_gen_fp64_persist; ISL:
// the runs are islands (migration after a grid barrier, common stop).
#include <cuda_runtime.h>
#include <math_constants.h>

#include <algorithm>

#include "de_common.cuh"
#include "de_device.cuh"
#include "de_gen_tile.cuh"
#include "de_internal.cuh"
#include "de_island_dev.cuh"
#include "de_kernels.h"
#include "de_slice.cuh"

namespace de {

constexpr long long kSlicedSpin = 1LL << 22;  // polls of the grid barrier (each a round trip to L2: seconds in all)

// CPL: coordinates per lane (1, 2 or 4: d <= 32, 64, 128).  An FP64 instruction
// costs its unit the same however few lanes are active, so short rows take one
// coordinate a lane, not four on a quarter of the lanes.
template <bool ISL, bool UNIT, int CPL>
__global__ void __launch_bounds__(256, 1)
    k_gen_sliced(const RunDesc* __restrict__ runs, const int4* __restrict__ items, int nruns, PersistCtl* ctl,
                 long long gens, IslandCtl* isl, IslandStage stage, int kpad, uint32_t cols) {
  extern __shared__ __align__(1024) uint8_t smem_s[];
  __shared__ SliceShared s_sl;
  __shared__ RunDesc sR;
  __shared__ int s_stop, s_abort, s_done, s_best;
  __shared__ unsigned s_below;
  __shared__ long long s_evals;
  __shared__ double s_bestf, s_f[kSliceRows];
  const int4 it = items[blockIdx.x];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  load_desc(sR, runs + it.x);
  __syncthreads();
  const RunDesc& R = sR;
  RunState* st = R.st;
  const unsigned nct = gridDim.x;
  const int ntiles = R.ntiles, d = R.d, dp = R.dp, nrows = it.w;
  if (tid == 0) {
    s_stop = st->stop;
    s_evals = st->evals;
    s_bestf = st->best_f;
    s_best = st->best_idx;
    s_abort = 0;
    s_done = 0;
    s_below = 0u;
    if (blockIdx.x == 0) ctl->gen0 = st->gen;
    if (s_stop && it.y == 0 && nruns > 1) atomicAdd(&ctl->stopped[2], 1u);
  }
  __syncthreads();
  if (nruns == 1 && s_stop) return;
  // (read before the first barrier: no island has advanced)
  const int interval = ISL && islands_together(runs, nruns, true) ? isl->interval : 0;
  SliceCtx sc;
  slice_begin(sc, smem_s, kpad, cols, s_sl);
  slice_load_m(sc, R.sl, R.sl_kpad);
  double* Y = reinterpret_cast<double*>(smem_s + slice_smem(kpad));
  double* Zf = Y + kSliceRows * dp;

  // ---- this warp's target: its row, fitness and the lane's part of the shift
  const bool mine = warp < nrows;
  const uint32_t i = (uint32_t)(it.z + warp);
  const int j0 = CPL * lane;
  const bool in = mine && j0 < d;
  double tx[CPL] = {}, tr[CPL] = {}, ov[CPL] = {}, fi = 0.0;
  long long gen = *(volatile int64_t*)&st->gen;
  auto load_row = [&](int cur) {
    if (in) ld_coords(R.X[cur] + (size_t)i * dp + j0, tx);
    if (mine) fi = __ldcg(R.f[cur] + i);
  };
#pragma unroll
  for (int m = 0; m < CPL; ++m)
    if (in && j0 + m < d) ov[m] = R.o[j0 + m];
  load_row((int)(gen & 1));
  TrialSetup ts{};
  U32x4 ub{};
  auto draw = [&](long long g) {
    if (mine) {
      ts = trial_setup(R, i, g, lane, 0u, false);
      if (in) ub = draw_block(R.seed, kPurposeStep, R.run_id, 0u, (uint32_t)g, i, 1u + (uint32_t)(j0 >> 2));
    }
  };
  if (!s_stop) draw(gen + 1);

  unsigned nstopped = 0;  // runs known stopped (thread 0)
  const bool test_skip = ctl->test_skip == (int)blockIdx.x + 1;
  const long long spin_limit = ctl->test_spin > 0 ? ctl->test_spin : kSlicedSpin;
  unsigned nbar = 0;
  // warp 0: arrive (unless the CTA leaves) and poll until every CTA did
  auto grid_sync = [&]() -> bool {
    if (lane == 0 && !(test_skip && nbar == 0))
      asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(&ctl->bar), "r"(1u) : "memory");
    __syncwarp();
    const unsigned target = (nbar + 1u) * nct;
    bool ok = false;
    for (long long k = 0; k < spin_limit; ++k) {
      unsigned v = 0u;
      if (lane == 0) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&ctl->bar) : "memory");
      if (__shfl_sync(0xffffffffu, v, 0) >= target) {
        ok = true;
        break;
      }
      // the abort flag every 16th poll (a read after every poll doubles
      // the round trips per poll)
      if ((k & 15) == 15 && *(volatile int*)&ctl->abort) break;
    }
    __syncwarp();
    ++nbar;
    return ok;
  };
  auto give_up = [&]() {
    atomicExch(&ctl->abort, 1);
    atomicOr(&st->err, kErrTimeout);
    s_abort = 1;
  };
  auto full_sync = [&]() {
    __syncthreads();
    if (warp == 0) {
      const bool ok = grid_sync();
      if (!ok && lane == 0) give_up();
    }
    __syncthreads();
  };
  // the warp that reduces the best record beside the trials
  const int rw = nrows < kSliceRows ? kSliceRows - 1 : 0;
  // best record and stop rule of generation gb (partials complete), the same
  // in every CTA of the run; warp rw.  slot: where a stop is counted.
  auto reduce_best = [&](long long gb, int slot) {
    long long bk = 0x7FFFFFFFFFFFFFFFLL;
    int bi = -1;
    const BestPartial* q = R.part + (size_t)(gb & 1) * ntiles;
    for (int t = lane; t < ntiles; t += 32) {
      const long long k = fit_key(__ldcg(&q[t].f));
      const int x = __ldcg(&q[t].idx);
      if (x >= 0 && (bi < 0 || k < bk || (k == bk && x < bi))) {
        bk = k;
        bi = x;
      }
    }
    warp_best(bk, bi);
    if (lane == 0) {
      const bool have = bi >= 0;
      if (have) {
        // the key is the value's integer image
        s_bestf = __longlong_as_double(bk >= 0 ? bk : (long long)(0x8000000000000000ULL | (unsigned long long)(-bk)));
        s_best = bi;
      }
      const int64_t evals = s_evals + R.np;
      int stop = 0;
      if (ISL && s_below > 0u) stop = 1;  // some island is below the target
      else if (R.target > 0.0 && s_best >= 0 && s_bestf < R.target) stop = 1;
      else if (R.max_evals > 0 && evals >= R.max_evals) stop = 2;
      else if (gb >= R.max_gens) stop = 3;
      s_evals = evals;
      s_stop = stop;
      if (it.y == 0) {
        if (have) {
          st->best_f = s_bestf;
          st->best_idx = bi;
        } else {
          atomicOr(&st->err, kErrNonFinite);
        }
        st->gen = gb;
        st->evals = evals;
        st->stop = stop;
        if (stop && nruns > 1) atomicAdd(&ctl->stopped[slot], 1u);
      }
    }
  };
  bool live = s_stop == 0;  // the run had not stopped at the last decision taken
  bool pending = false;     // generation gen's partials are complete, its stop decision not taken

  for (long long itg = 0;; ++itg) {
    const long long g = gen + 1;
    const bool more = itg < gens;
    // ---- the donors' loads, then (one warp) the last generation's decision
    double x1[CPL], x2[CPL], x3[CPL];
    if (live && more && in) {
      const double* X = R.X[gen & 1] + j0;
      ld_coords(X + (size_t)ts.r1 * dp, x1);
      ld_coords(X + (size_t)ts.r2 * dp, x2);
      ld_coords(X + (size_t)ts.r3 * dp, x3);
    }
    // (counted in the slot of the iteration that ran generation gen)
    if (pending && warp == rw) reduce_best(gen, (int)((itg + 2) % 3));
    // ---- trials: Eq. 2, Eq. 3, bound repair; y = (t - o) s as digits
    if (live && more && mine) {
      double y[CPL] = {};
      if (in) {
        uint32_t u[CPL];
#pragma unroll
        for (int m = 0; m < CPL; ++m) u[m] = word_of(ub, (j0 + m) & 3);
        trial_coords<CPL>(R, ts.jr, j0, tx, x1, x2, x3, u, tr, R.F, R.cr_thr, 0);
#pragma unroll
        for (int m = 0; m < CPL; ++m) y[m] = j0 + m < d ? shifted_as<UNIT>(tr[m], ov[m], R.scale) : 0.0;
        st_coords(Y + warp * dp + j0, y);
      }
      slice_digits(sc, warp, lane, R.sl_kpad, R.sl_qmin[0], y);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    pending = false;
    live = live && s_stop == 0;
    if (!more || s_done || (nruns == 1 && !live)) break;
    if (live) {
      // ---- fitness; the warps that do not issue the products draw the next
      // generation's numbers meanwhile
      if (warp != kSliceIssuer) draw(g + 1);
      const double ft = slice_fitness(sc, R, Y, Zf, nrows);
      // ---- selection: ft <= fi accepts, a NaN never
      if (mine) {
        const long long kt = fit_key(ft);
        const bool acc = kt <= fit_key(fi) && kt != 0x7FFFFFFFFFFFFFFFLL;
        if (acc) {
          fi = ft;
#pragma unroll
          for (int m = 0; m < CPL; ++m) tx[m] = tr[m];
        }
        if constexpr (CPL == 4) {
          if (in) st_row4(R.X[g & 1] + (size_t)i * dp + j0, tx);
        } else {
          if (in) st_coords(R.X[g & 1] + (size_t)i * dp + j0, tx);
        }
        if (lane == 0) {
          R.f[g & 1][i] = fi;
          s_f[warp] = fi;
        }
      }
      if (tid == 0 && s_sl.fail) give_up();
      __syncthreads();  // every row is written
    }
    if (warp == 0) {
      if (live) {
        long long bk = 0x7FFFFFFFFFFFFFFFLL;
        int bi = -1;
        if (lane < nrows) {
          bk = fit_key(s_f[lane]);
          bi = it.z + lane;
        }
        warp_best(bk, bi);
        if (lane == 0) {
          BestPartial* pp = R.part + (size_t)(g & 1) * ntiles + it.y;
          const double bf = bi >= 0 ? s_f[bi - it.z] : CUDART_INF;
          pp->f = bf;
          pp->idx = bi;
          // island model: the model stops as a whole once any island's best is
          // below the target (counted before the barrier, read after it)
          if (ISL && R.target > 0.0 && bi >= 0 && bf < R.target) atomicAdd(&ctl->below[itg % 3], 1u);
        }
      }
      const bool ok = *(volatile int*)&s_abort == 0 && grid_sync();
      if (lane == 0) {
        if (!ok) {
          give_up();
        } else if (nruns > 1) {
          // runs stopped by the decisions before this barrier
          nstopped += __ldcg(&ctl->stopped[(itg + 2) % 3]);
          // every CTA read slot (itg + 1) % 3 after the previous barrier; it
          // is next counted after the next one
          if (blockIdx.x == 0) ctl->stopped[(itg + 1) % 3] = 0u;
          if (nstopped >= (unsigned)nruns) s_done = 1;
        }
        if (ISL && ok) {
          s_below = __ldcg(&ctl->below[itg % 3]);
          // every CTA read slot (itg + 2) % 3 before arriving at this barrier;
          // it is next counted at iteration itg + 2
          if (blockIdx.x == 0) ctl->below[(itg + 2) % 3] = 0u;
        }
      }
    } else if (live && warp == kSliceIssuer) {
      draw(g + 1);
    }
    __syncthreads();
    if (s_abort) break;
    if (!live) continue;
    gen = g;
    pending = true;
    if constexpr (ISL) {
      if (!(interval > 0 && g % interval == 0)) continue;
      // island model: the stop decision, then migration after generation g
      // (islands that are together advance together, so every CTA takes this branch).  The CTA
      // of each island's tile 0 exchanges; a grid barrier then keeps every
      // tile from building generation g + 1 before the migrants are in place.
      if (warp == rw) reduce_best(g, (int)(itg % 3));
      pending = false;
      __syncthreads();
      live = s_stop == 0;
      const int cur = (int)(g & 1);
      const bool owner = it.y == 0;
      if (isl->async) {
        // one interval late, through the mailbox (k_island_async's rule)
        const int64_t ep = g / isl->interval;
        // post_gen is written by CTA 0 after an earlier migration's barrier: read at L2
        const long long pg = *(volatile long long*)&isl->post_gen;
        const bool take = pg >= 0 && pg == g - isl->interval;
        if (owner)
          island_exchange(R, it.x, isl->m, isl->nmig, cur, stage, true, (size_t)(ep & 1) * stage.slot, take,
                          (size_t)((ep & 1) ^ 1) * stage.slot);
      } else {
        // every island posts before any island takes
        if (owner) island_exchange(R, it.x, isl->m, isl->nmig, cur, stage, true, 0, false, 0);
        full_sync();
        if (s_abort) break;
        if (owner) island_exchange(R, it.x, isl->m, isl->nmig, cur, stage, false, 0, true, 0);
      }
      full_sync();
      if (s_abort) break;
      // the rows and fitness this CTA holds, after the exchange
      load_row(cur);
      if (blockIdx.x == 0 && tid == 0) {
        isl->mig_gen = g;
        if (isl->async) isl->post_gen = g;
      }
    }
  }
  slice_end(sc);
}

// ------------------------------------------------------------------ host side
static const void* sliced_kernel(bool isl, bool unit, int kpad) {
#define DE_SLICED(c)                                                                                       \
  (isl ? (unit ? (const void*)k_gen_sliced<true, true, c> : (const void*)k_gen_sliced<true, false, c>)     \
       : (unit ? (const void*)k_gen_sliced<false, true, c> : (const void*)k_gen_sliced<false, false, c>))
  return kpad <= 32 ? DE_SLICED(1) : kpad <= 64 ? DE_SLICED(2) : DE_SLICED(4);
#undef DE_SLICED
}

// All of an SM's shared memory, as the sliced instances of the general
// cooperative kernel take (fp64_exclusive_smem).
int k_gen_sliced_capacity(bool isl, bool unit, const SlicePlan& p, size_t smem) {
  const void* k = sliced_kernel(isl, unit, p.kpad);
  const size_t dyn = fp64_exclusive_smem(k, smem);
  int per_sm = 0, dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (allow_dynamic_smem(k) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 256, dyn) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return per_sm * nsm;
}

size_t sliced_loop_smem(const SlicePlan& p, int dp_max) {
  return slice_smem(p.kpad) + (size_t)2 * kSliceRows * dp_max * sizeof(double);
}

cudaError_t k_gen_sliced_launch(const RunDesc* runs, const int4* items, int nitems, int nruns, PersistCtl* ctl,
                                long long gens, const SlicePlan& p, bool unit, size_t smem, cudaStream_t s,
                                int test_skip, IslandCtl* isl, const IslandStage* stage) {
  cudaError_t e = persist_ctl_reset(ctl, test_skip, s);
  if (e != cudaSuccess) return e;
  IslandStage st{};
  if (stage) st = *stage;
  int kpad = p.kpad;
  uint32_t cols = p.cols;
  void* args[] = {(void*)&runs, (void*)&items, (void*)&nruns, (void*)&ctl, (void*)&gens,
                  (void*)&isl,  (void*)&st,    (void*)&kpad,  (void*)&cols};
  const void* k = sliced_kernel(isl != nullptr, unit, p.kpad);
  return cudaLaunchCooperativeKernel(k, dim3((unsigned)nitems), dim3(256), args, fp64_exclusive_smem(k, smem), s);
}

}  // namespace de
