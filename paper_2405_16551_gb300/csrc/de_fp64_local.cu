// de_fp64_local.cu -- the FP64 generation loop of small runs, a thread-block
// cluster per run with the population in shared memory.
//
// A run of at most 64 targets of at most 64 coordinates is a chain of latencies:
// NP = 64, D = 10 (sphere) took 6.35 us a generation in the general loop, for
// 0.1 us of FP64 work, in trips to L2 (donors, partials, fitness), barriers, and
// FP64 instructions on 3 of 32 lanes; here it takes 2.55 us.
//   - every CTA of the run's cluster (at most 8, a warp per target) keeps a copy
//     of the whole population in shared memory, double buffered: donors are
//     local loads; a target's next row goes to every CTA's copy through
//     distributed shared memory, with its fitness key;
//   - the one synchronisation of a generation is the cluster barrier (the next
//     generation's draws are made between arriving and waiting); after it every
//     warp takes the best record and the stop decision from the keys itself;
//   - a lane holds one coordinate (two for d > 32): an FP64 instruction costs
//     the same however few lanes are active;
//   - for d <= 32 the digit products of a rotation run on mma.sync: at 32 x 32
//     the issue, commit and read-back of tcgen05 cost more than the products,
//     and its tensor memory would need a whole SM per CTA (fp64_exclusive_smem),
//     which 16 islands of 8 CTAs do not get (15 such clusters fit at once).
// Populations, fitness and state go to global memory at the end of the launch.
// The numbers are those of the general kernels: the same
// trial, rotation (sliced, or the DFMA chain for the others) and term routines,
// and the same order of every sum.
//
// ISL: the runs are islands.  The model stops as a whole at the first
// generation in which some island's best is below the target; an island learns
// of that one generation late (the counter it would have to wait for has had
// a generation's time to fill), and then takes back its last one, whose
// predecessor is still in the other buffer.  At migration points the islands
// meet (bounded waits on global counters); a warp picks the migrants from the
// keys and passes them through the mailbox, in island_exchange's order (that
// routine, a CTA on the populations in global memory, took 35 us a point).
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math_constants.h>

#include <algorithm>
#include <vector>

#include "de_common.cuh"
#include "de_device.cuh"
#include "de_gen_tile.cuh"
#include "de_internal.cuh"
#include "de_kernels.h"
#include "de_slice_mma.cuh"

namespace cg = cooperative_groups;

namespace de {

constexpr int kLocalNp = 64;                // targets of a run (8 CTAs of 8 warps)
constexpr long long kLocalSpin = 1LL << 22;  // polls of an island counter (each a round trip to L2)

// How the rotation runs: not at all or as the DFMA chain; as digit products
// on tcgen05; as digit products on mma.sync (d <= 32).
enum LocalRot { kRotChain = 0, kRotTc = 1, kRotMma = 2 };

// Bytes of the mma.sync form's operands (de_slice_mma.cuh, width 32).
constexpr uint32_t kMmaB = mma_b_bytes(32), kMmaA = mma_a_bytes(32), kMmaP = mma_p_bytes(32);
constexpr int kMmaPst = mma_pst(32);

// Byte offsets of a CTA's dynamic shared memory: operands of the digit
// products, FP64 rows of y and of the rows that take the chain, the two
// population buffers, M^T (chain).
struct LocalLayout {
  uint32_t y, z, pop, mt, total;
};
__host__ __device__ inline LocalLayout local_layout(int rot, int kpad, int dp, int d, bool rotate) {
  LocalLayout L;
  L.y = rot == kRotTc ? slice_smem(kpad) : rot == kRotMma ? kMmaB + kMmaA + kMmaP : 0u;
  L.z = L.y + (uint32_t)(kSliceRows * dp) * 8u;
  L.pop = L.z + (rot == kRotTc ? (uint32_t)(kSliceRows * dp) * 8u : 0u);
  L.mt = L.pop + 2u * (uint32_t)(kLocalNp * dp) * 8u;
  L.total = L.mt + (rot == kRotChain && rotate ? (uint32_t)(d * d) * 8u : 0u);
  return L;
}

// M's digits and the zeroed operand of y's, by the whole CTA (which
// synchronises before the first product).
__device__ __forceinline__ void local_load_m(const RunDesc& R, uint8_t* smem) {
  for (uint32_t q = threadIdx.x * 16u; q < kMmaB; q += blockDim.x * 16u)
    *reinterpret_cast<uint4*>(smem + q) = make_uint4(0u, 0u, 0u, 0u);
  mma_copy_m(smem + kMmaB, R.sl, R.sl_kpad);
}

// z_j (lane j) of the row of y (lane k: y_k) whose digits this warp has
// written; the whole CTA calls it (a warp without a row: mine = false).  fj: the
// exponent of M's row j; Yr: room for the row where it takes the DFMA chain.
__device__ __forceinline__ double local_rotate(const RunDesc& R, uint8_t* smem, SliceShared& sh, int fj, double* Yr,
                                               double y, bool mine, int warp, int lane) {
  const int d = R.d;
  __syncthreads();
  float* sP = reinterpret_cast<float*>(smem + kMmaB + kMmaA);
  const uint32_t sB = smem_u32(smem), sA = sB + kMmaB;
  // a warp takes 16 outputs and 10 to 12 of the 43 pairs of digits
  if (16 * (warp & 1) < d) {
    switch (warp >> 1) {
      case 0: mma_products32<8, 3, -1>(sB, sA, sP, warp & 1, lane); break;
      case 1: mma_products32<7, 2, -1>(sB, sA, sP, warp & 1, lane); break;
      case 2: mma_products32<6, 1, 0>(sB, sA, sP, warp & 1, lane); break;
      default: mma_products32<5, 4, -1>(sB, sA, sP, warp & 1, lane); break;
    }
  }
  __syncthreads();
  if (!mine) return 0.0;
  float p[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) p[q] = sP[(q * kSliceRows + warp) * kMmaPst + lane];
  const double zj = slice_combine(p, sh.exp[warp] + fj - 76);
  double z = lane < d ? zj : 0.0;
  if ((*(volatile uint32_t*)&sh.bad >> warp) & 1u) {
    // outside the splitting's comparison: the DFMA chain
    if (lane < d) Yr[lane] = y;
    __syncwarp();
    if (lane == 0) atomicAnd(&sh.bad, ~(1u << warp));
    z = 0.0;
    if (lane < d)
      for (int k = 0; k < d; ++k) z = fma(__ldg(R.MT + (size_t)k * d + lane), Yr[k], z);
    __syncwarp();
  }
  return z;
}

// Objective of a row, lane j holding z_j (d <= 32); every lane returns it.
__device__ __forceinline__ double local_objective(int obj, double z, int d, int lane) {
  double t1 = 0.0, t2 = 0.0;
  if (obj == kObjRosenbrock) {
    const double zn = __shfl_down_sync(0xffffffffu, z, 1);
    if (lane + 1 < d) {
      const double t0 = z + 1.0, tn = zn + 1.0;
      const double a = tn - t0 * t0, b = t0 - 1.0;
      t1 = 100.0 * a * a + b * b;
    }
  } else if (lane < d) {
    if (obj == kObjRastrigin) {
      t1 = fma(z, z, rastrigin_w(z));
    } else {
      t1 = z * z;
      if (obj == kObjAckley) t2 = cos2pi_fix(z);
    }
  }
  if (obj != kObjAckley) return warp_sum(t1);
  const double s1 = warp_sum(t1), s2 = warp_sum(t2);
  return ackley_value((lane & 1 ? s2 : s1) / d, lane);
}

// The fitness of a key (NaN for the largest).
__device__ __forceinline__ double key_value(long long k) {
  if (k == 0x7FFFFFFFFFFFFFFFLL) return CUDART_NAN;
  return __longlong_as_double(k >= 0 ? k : (long long)(0x8000000000000000ULL | (unsigned long long)(-k)));
}

// island_pick over at most 64 keys in shared memory, n <= 32 times without
// repetition, by one warp: lane q returns the index of the q-th smallest
// (key, index), or largest.
__device__ __forceinline__ int local_pick(const long long* keys, int np, int n, bool worst, int lane) {
  // the largest as the smallest of the complements; idle entries come last
  long long k[2];
  int x[2], sel = 0;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int i = lane + 32 * e;
    const bool in = i < np;
    k[e] = in ? (worst ? ~keys[i] : keys[i]) : 0x7FFFFFFFFFFFFFFFLL;
    x[e] = in ? (worst ? kLocalNp - 1 - i : i) : 2 * kLocalNp;
  }
  for (int q = 0; q < n; ++q) {
    const int a = k[1] < k[0] || (k[1] == k[0] && x[1] < x[0]) ? 1 : 0;
    const long long v = a ? k[1] : k[0];
    const int hi = __reduce_min_sync(0xffffffffu, (int)(v >> 32));
    const unsigned lo = __reduce_min_sync(0xffffffffu, (int)(v >> 32) == hi ? (unsigned)v : 0xffffffffu);
    const bool cand = (int)(v >> 32) == hi && (unsigned)v == lo;
    const int w = __reduce_min_sync(0xffffffffu, cand ? (a ? x[1] : x[0]) : 4 * kLocalNp);
    if (lane == q) sel = worst ? kLocalNp - 1 - w : w;
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (x[e] == w) {
        k[e] = 0x7FFFFFFFFFFFFFFFLL;
        x[e] = 2 * kLocalNp;
      }
  }
  return sel;
}

template <int CPL, int ROT, bool ISL>
__global__ void __launch_bounds__(256, ROT == kRotTc ? 1 : 2)
    k_gen_local(const RunDesc* __restrict__ runs, PersistCtl* ctl, long long gens, int csize, IslandCtl* isl,
                IslandStage stage, int kpad, uint32_t cols, int dp_max) {
  extern __shared__ __align__(1024) uint8_t smem_l[];
  __shared__ SliceShared s_sl;
  __shared__ RunDesc sR;
  __shared__ long long s_key[2][kLocalNp];
  // by generation parity: 1 the model had stopped before it, 2 a wait gave up;
  // nonzero when a CTA's products did
  __shared__ int s_flag[2], s_fail[2];
  __shared__ int s_over;
  cg::cluster_group cluster = cg::this_cluster();
  const int run = (int)blockIdx.x / csize, rank = (int)blockIdx.x % csize;
  // a launch without its cluster dimension (a tool that launches the kernel
  // again by itself) has no peers to write to: an error, not a fault
  if ((int)cluster.num_blocks() != csize) {
    if (threadIdx.x == 0) atomicOr(&runs[run].st->err, kErrTimeout);
    return;
  }
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  load_desc(sR, runs + run);
  if (tid < 2) s_flag[tid] = s_fail[tid] = 0;
  if (tid < 2 * kLocalNp) s_key[tid / kLocalNp][tid % kLocalNp] = 0x7FFFFFFFFFFFFFFFLL;
  __syncthreads();
  const RunDesc& R = sR;
  RunState* st = R.st;
  const int np = R.np, d = R.d, dp = R.dp, obj = R.obj;
  const bool stopped0 = *(volatile int32_t*)&st->stop != 0;
  if (!ISL && stopped0) return;  // the whole cluster
  constexpr bool SL = ROT == kRotTc, MM = ROT == kRotMma;
  const LocalLayout L = local_layout(ROT, kpad, dp_max, 0, false);
  double* Y = reinterpret_cast<double*>(smem_l + L.y);
  double* Zf = reinterpret_cast<double*>(smem_l + L.z);
  double* pop = reinterpret_cast<double*>(smem_l + L.pop);
  double* mts = reinterpret_cast<double*>(smem_l + L.mt);
  const int psz = kLocalNp * dp_max;  // doubles per population buffer
  SliceCtx sc;
  if constexpr (SL) {
    slice_begin(sc, smem_l, kpad, cols, s_sl);
    slice_load_m(sc, R.sl, R.sl_kpad);
  } else if constexpr (MM) {
    sc.sB = smem_l;
    sc.s_exp = s_sl.exp;
    sc.s_bad = &s_sl.bad;
    if (tid == 0) s_sl.bad = 0u;
    local_load_m(R, smem_l);
  } else if (R.rotate) {
    for (int e = tid; e < d * d; e += blockDim.x) mts[e] = __ldg(R.MT + e);
  }
  const int fj = MM && lane < d ? __ldg(R.slx + lane) : 0;
  long long gen = *(volatile int64_t*)&st->gen;
  int64_t evals = *(volatile int64_t*)&st->evals;
  double bestf = *(volatile double*)&st->best_f;
  int best = *(volatile int32_t*)&st->best_idx;
  int stop = stopped0 ? *(volatile int32_t*)&st->stop : 0;
  int err = 0;

  const int i = 8 * rank + warp;  // this warp's target
  const bool mine = i < np;
  const int nrows = max(0, min(8, np - 8 * rank));  // targets of this CTA
  const int j0 = CPL * lane;
  const bool in = mine && j0 < d;
  double tx[CPL] = {}, tr[CPL] = {}, ov[CPL] = {}, fi = 0.0, fp = 0.0;
#pragma unroll
  for (int m = 0; m < CPL; ++m)
    if (in && j0 + m < d) ov[m] = R.o[j0 + m];
  // the population of generation g from global memory into the CTA's copy,
  // this warp's row and fitness into registers
  auto load_pop = [&](long long g) {
    const double* X = R.X[g & 1];
    double* p = pop + (size_t)(g & 1) * psz;
    for (int e = tid; e < np * dp; e += blockDim.x) p[e] = __ldcg(X + e);
    if (in) ld_coords(X + (size_t)i * dp + j0, tx);
    if (mine) fi = __ldcg(R.f[g & 1] + i);
  };
  auto store_rows = [&](long long g) {
    if (in) st_coords(R.X[g & 1] + (size_t)i * dp + j0, tx);
    if (mine && lane == 0) R.f[g & 1][i] = fi;
  };
  load_pop(gen);
  TrialSetup ts{};
  U32x4 ub{};
  auto draw = [&](long long g) {
    if (mine) {
      ts = trial_setup(R, (uint32_t)i, g, lane, 0u, false);
      if (in) ub = draw_block(R.seed, kPurposeStep, R.run_id, 0u, (uint32_t)g, (uint32_t)i, 1u + (uint32_t)(j0 >> 2));
    }
  };
  draw(gen + 1);
  const bool common = ISL && R.target > 0.0;  // the islands' common stop applies
  const unsigned m_isl = ISL ? (unsigned)isl->m : 1u;
  const bool test_skip = ISL && ctl->test_skip == run + 1;
  const long long spin = ISL && ctl->test_spin > 0 ? ctl->test_spin : kLocalSpin;
  // One island's arrival at iteration k is one relaxed addition to the counter
  // of k's parity: 1, plus 2^32 when its best is below the target.  No other
  // memory hangs on it, so nothing waits for a fence (an island is at most one
  // iteration ahead of another that it waits for, and none passes a point where
  // they meet, so a counter that reads complete holds no later arrival).
  auto count_of = [&](long long k) -> unsigned long long* { return &ctl->isl_cnt[k & 1]; };
  auto count_want = [&](long long k) { return m_isl * (unsigned)(k / 2 + 1); };
  auto read_count = [&](long long k) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(count_of(k)) : "memory");
    return v;
  };
  auto arrive = [&](long long k, bool below) {
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(count_of(k)), "l"(1ULL + (below ? 1ULL << 32 : 0ULL))
                 : "memory");
  };
  // until every island has arrived at iteration k (v: the counter as read
  // before; one lane polls): 0, 1 when some island is below the target, 2 gave up
  auto wait_islands = [&](long long k, unsigned long long v) -> int {
    for (long long q = 0; q < spin; ++q) {
      if ((unsigned)v >= count_want(k)) return v >> 32 ? 1 : 0;
      if ((q & 15) == 15 && *(volatile int*)&ctl->abort) break;
      v = read_count(k);
    }
    atomicExch(&ctl->abort, 1);
    return 2;
  };
  // the migrations' own counter: orders the mailbox's writes before its reads
  auto wait_posted = [&](unsigned want) -> bool {
    for (long long q = 0; q < spin; ++q) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&ctl->sbar[0]) : "memory");
      if (v >= want) return true;
      if ((q & 15) == 15 && *(volatile int*)&ctl->abort) break;
    }
    atomicExch(&ctl->abort, 1);
    return false;
  };
  // every CTA is running and has loaded before any peer writes its memory
  cluster.sync();

  bool changed = true;  // the row in the other buffer is not the one before this
  // the best of the keys of generation gen (every warp)
  auto reduce_best = [&]() {
    long long bk = lane < np ? s_key[gen & 1][lane] : 0x7FFFFFFFFFFFFFFFLL;
    int bi = lane < np ? lane : -1;
    const long long k2 = lane + 32 < np ? s_key[gen & 1][lane + 32] : 0x7FFFFFFFFFFFFFFFLL;
    if (k2 < bk) {
      bk = k2;
      bi = lane + 32;
    }
    warp_best(bk, bi);
    if (bi >= 0) {
      bestf = key_value(bk);
      best = bi;
    }
    return bi >= 0;
  };
  long long it = 0;
  for (; it < gens && !stop && !err; ++it) {
    const long long g = gen + 1;
    const double* P = pop + (size_t)(gen & 1) * psz;
    double ft = 0.0;
    unsigned long long early = 0ULL;  // rank 0, thread 0: the islands' last counter, read ahead of its use
    double y[CPL] = {};
    // ---- trial: Eq. 2, Eq. 3, bound repair; y = (t - o) s
    if (in) {
      double x1[CPL], x2[CPL], x3[CPL];
      uint32_t u[CPL];
#pragma unroll
      for (int m = 0; m < CPL; ++m) {
        x1[m] = P[ts.r1 * dp + j0 + m];
        x2[m] = P[ts.r2 * dp + j0 + m];
        x3[m] = P[ts.r3 * dp + j0 + m];
        u[m] = word_of(ub, (j0 + m) & 3);
      }
      trial_coords<CPL>(R, ts.jr, j0, tx, x1, x2, x3, u, tr, R.F, R.cr_thr, 0);
#pragma unroll
      for (int m = 0; m < CPL; ++m) y[m] = j0 + m < d ? shifted(tr[m], ov[m], R) : 0.0;
    }
    // ---- fitness
    if constexpr (SL) {
      if (mine) {
        if (in) st_coords(Y + warp * dp + j0, y);
        slice_digits(sc, warp, lane, R.sl_kpad, R.sl_qmin[0], y);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      }
      __syncthreads();
      ft = slice_fitness(sc, R, Y, Zf, nrows);
    } else {
      // one coordinate a lane (d <= 32): the sums of the general kernels, whose
      // lane j holds coordinate j
      double z = y[0];
      if constexpr (MM) {
        if (mine) slice_digits(sc, warp, lane, R.sl_kpad, R.sl_qmin[0], y);
        const double zj = local_rotate(R, smem_l, s_sl, fj, Y + warp * dp, y[0], mine, warp, lane);
        if (mine) z = zj;
      } else if (mine && R.rotate) {
        double* yr = Y + warp * dp;
        if (lane < d) yr[lane] = y[0];
        __syncwarp();
        z = 0.0;
        if (lane < d)
          for (int k = 0; k < d; ++k) z = fma(mts[k * d + lane], yr[k], z);
        __syncwarp();
      }
      if (common && rank == 0 && tid == 0 && it > 0) early = read_count(it - 1);
      if (mine) ft = local_objective(obj, z, d, lane);
    }
    // ---- selection; the row and its key to every CTA of the cluster
    if (mine) {
      fp = fi;
      const long long kt = fit_key(ft);
      const bool acc = kt <= fit_key(fi) && kt != 0x7FFFFFFFFFFFFFFFLL;  // ft <= fi, NaN never
      if (acc) {
        fi = ft;
#pragma unroll
        for (int m = 0; m < CPL; ++m) tx[m] = tr[m];
      }
      // the buffer holds the row of two generations ago: nothing to write for a
      // row that neither this generation nor the last one changed
      const bool write = acc || changed;
      changed = acc;
      if (in && write) {
        double* q = pop + (size_t)(g & 1) * psz + (size_t)i * dp + j0;
        for (int c = 0; c < csize; ++c) st_coords(cluster.map_shared_rank(q, c), tx);
      }
      if (lane < csize) *cluster.map_shared_rank(&s_key[g & 1][i], lane) = fit_key(fi);
    }
    if (SL && tid == 0 && s_sl.fail)
      for (int c = 0; c < csize; ++c) *cluster.map_shared_rank(&s_fail[g & 1], c) = 1;
    if (common && rank == 0 && tid == 0 && it > 0) {
      // whether the model stopped at the generation before this
      const int f = wait_islands(it - 1, early);
      if (f)
        for (int c = 0; c < csize; ++c) *cluster.map_shared_rank(&s_flag[g & 1], c) = f;
    }
    cg::cluster_group::arrival_token tok = cluster.barrier_arrive();
    draw(g + 1);
    cluster.barrier_wait(std::move(tok));
    const int flag = *(volatile int*)&s_flag[g & 1];
    if (flag == 2 || *(volatile int*)&s_fail[g & 1]) {
      err = kErrTimeout;
      break;
    }
    if (ISL && flag == 1) {
      // the model stopped at generation gen: back to it
      if (in) {
#pragma unroll
        for (int m = 0; m < CPL; ++m) tx[m] = P[(size_t)i * dp + j0 + m];
      }
      fi = fp;
      stop = 1;
      break;
    }
    // ---- best record and stop rule, by every warp
    gen = g;
    evals += np;
    if (!reduce_best() && rank == 0 && tid == 0) atomicOr(&st->err, kErrNonFinite);
    const bool below = R.target > 0.0 && best >= 0 && bestf < R.target;
    if (!ISL && below) stop = 1;
    else if (R.max_evals > 0 && evals >= R.max_evals) stop = 2;
    else if (gen >= R.max_gens) stop = 3;
    if constexpr (ISL) {
      if (rank == 0 && tid == 0 && (common || isl->interval > 0)) {
        if (!(test_skip && it == 0)) arrive(it, common && below);
      }
      const bool mig = isl->interval > 0 && gen % isl->interval == 0;
      if (mig || stop || it + 1 >= gens) {
        // the islands meet: the common stop at this generation, and migration,
        // by the first warp of rank 0, which holds the whole population
        if (mig) cluster.sync();  // every warp has taken the best of the keys that migration changes
        if (rank == 0 && warp == 0) {
          int f = 0;
          if (lane == 0 && (common || mig)) f = wait_islands(it, read_count(it));
          f = __shfl_sync(0xffffffffu, f, 0);
          if (mig && f != 2) {
            // with the fence after the last exchange: what it read is read, and
            // its mailbox may be written again
            __threadfence();
            double* p = pop + (size_t)(gen & 1) * psz;
            long long* keys = s_key[gen & 1];
            const int m = isl->m, nmig = isl->nmig;
            const int64_t ep = gen / isl->interval;
            // asynchronous: one interval late, from the slot of the last point
            // (k_island_async's rule)
            const bool late = isl->async != 0;
            const long long pg = *(volatile long long*)&isl->post_gen;
            const bool take = !late || (pg >= 0 && pg == gen - isl->interval);
            const size_t wslot = late ? (size_t)(ep & 1) * stage.slot : 0;
            const size_t rslot = late ? (size_t)((ep & 1) ^ 1) * stage.slot : 0;
            const int good = local_pick(keys, np, nmig, false, lane);
            const int poor = take ? local_pick(keys, np, nmig, true, lane) : 0;
            for (int q = 0; q < nmig; ++q) {
              const int i1 = __shfl_sync(0xffffffffu, good, q);
              const size_t e = wslot + (size_t)run * nmig + q;
              for (int j = lane; j < dp; j += 32) stage.x[e * stage.dp + j] = p[(size_t)i1 * dp + j];
              if (lane == 0) {
                stage.f[e] = key_value(keys[i1]);
                stage.fx[e] = 1;
              }
            }
            __syncwarp();
            // every island has posted (asynchronous: and read post_gen)
            auto posted = [&]() {
              int ok = 1;
              if (lane == 0) {
                asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(&ctl->sbar[0]), "r"(1u) : "memory");
                ok = wait_posted(m_isl * (unsigned)(ep - (gen - it - 1) / isl->interval)) ? 1 : 0;
              }
              ok = __shfl_sync(0xffffffffu, ok, 0);
              __syncwarp();
              if (!ok) f = 2;
            };
            if (!late) posted();
            const int from = (run + m - 1) % m;
            for (int q = 0; take && f != 2 && q < nmig; ++q) {
              const int i1 = __shfl_sync(0xffffffffu, poor, q);
              const size_t e = rslot + (size_t)from * nmig + q;
              for (int j = lane; j < dp; j += 32) {
                const double v = __ldcg(stage.x + e * stage.dp + j);
                for (int c = 0; c < csize; ++c) *cluster.map_shared_rank(p + (size_t)i1 * dp + j, c) = v;
              }
              const long long k = fit_key(__ldcg(stage.f + e));
              if (lane < csize) *cluster.map_shared_rank(keys + i1, lane) = k;
            }
            __syncwarp();
            if (late) posted();
            if (run == 0 && lane == 0 && f != 2) {
              isl->mig_gen = gen;
              if (late) isl->post_gen = gen;
            }
            __threadfence();
          }
          if (lane < csize) *cluster.map_shared_rank(&s_over, lane) = f;
        }
        cluster.sync();
        const int over = *(volatile int*)&s_over;
        if (over == 2) {
          err = kErrTimeout;
          break;
        }
        if (over == 1) stop = 1;
        if (mig) {
          if (in) {
#pragma unroll
            for (int e = 0; e < CPL; ++e) tx[e] = pop[(size_t)(gen & 1) * psz + (size_t)i * dp + j0 + e];
          }
          if (mine) fi = key_value(s_key[gen & 1][i]);
          changed = true;
          reduce_best();
        }
      }
    }
  }
  // ---- what the caller reads
  if (!err) {
    store_rows(gen);
    if (rank == 0 && tid == 0) {
      st->best_f = bestf;
      st->best_idx = best;
      st->gen = gen;
      st->evals = evals;
      st->stop = stop;
    }
  } else if (rank == 0 && tid == 0) {
    atomicOr(&st->err, err);
  }
  cluster.sync();  // no peer writes this CTA's memory any more
  if constexpr (SL) slice_end(sc);
}

// ------------------------------------------------------------------ evaluation
// f of n rows of x (row stride ld) of a sliced run with d <= 32, a warp per
// row, `rows` <= 8 rows a tile, CTA b taking tiles b, b + gridDim.x, ...  Bound
// by its latencies: the descriptor is a parameter, M's digits are loaded while
// the rows are, and few rows are spread over every SM (a row's FP64
// instructions do not wait for another's).
__global__ void __launch_bounds__(256, 2)
    k_eval_few(const __grid_constant__ RunDesc R, const double* __restrict__ x, int64_t ld, int n, int rows,
               double* __restrict__ fout, uint8_t* __restrict__ fx_out) {
  __shared__ __align__(16) uint8_t smem[kMmaB + kMmaA + kMmaP];
  __shared__ SliceShared sh;
  __shared__ double sY[kSliceRows][32];
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
  const int d = R.d;
  SliceCtx sc;
  sc.sB = smem;
  sc.s_exp = sh.exp;
  sc.s_bad = &sh.bad;
  const double o = lane < d ? __ldg(R.o + lane) : 0.0;
  const int fj = lane < d ? __ldg(R.slx + lane) : 0;
  int row = blockIdx.x * rows + warp;
  double xv = warp < rows && row < n && lane < d ? __ldg(x + (size_t)row * ld + lane) : 0.0;
  if (threadIdx.x == 0) sh.bad = 0u;
  local_load_m(R, smem);
  __syncthreads();
  for (int t0 = blockIdx.x * rows; t0 < n; t0 += gridDim.x * rows) {
    row = t0 + warp;
    const bool mine = warp < rows && row < n;
    const double y[1] = {mine && lane < d ? shifted(xv, o, R) : 0.0};
    const int nx = row + (int)gridDim.x * rows;
    xv = warp < rows && nx < n && lane < d ? __ldg(x + (size_t)nx * ld + lane) : 0.0;
    if (mine) slice_digits(sc, warp, lane, R.sl_kpad, R.sl_qmin[0], y);
    const double z = local_rotate(R, smem, sh, fj, sY[warp], y[0], mine, warp, lane);
    if (!mine) continue;
    const double f = local_objective(R.obj, z, d, lane);
    if (lane == 0) {
      fout[row] = f;
      if (fx_out) fx_out[row] = 1;
    }
  }
}

// ------------------------------------------------------------------ host side
bool k_eval_few_launch(const RunDesc& Rh, const double* x, int64_t ld, int n, double* f, uint8_t* fx, cudaStream_t s) {
  if (!Rh.sl || Rh.d > 32 || Rh.obj > kObjAckley) return false;
  int dev = 0, nsm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int rows = std::max(1, std::min(kSliceRows, (n + nsm - 1) / nsm));
  const int tiles = (n + rows - 1) / rows;
  k_eval_few<<<std::min(tiles, 2 * nsm), 256, 0, s>>>(Rh, x, ld, n, rows, f, fx);
  return true;
}

static int local_rot(const LocalPlan& p) { return !p.sl ? kRotChain : p.kpad <= 32 ? kRotMma : kRotTc; }

static const void* local_kernel(const LocalPlan& p, bool isl) {
  switch (local_rot(p)) {
    case kRotChain: return isl ? (const void*)k_gen_local<1, kRotChain, true> : (const void*)k_gen_local<1, kRotChain, false>;
    case kRotMma: return isl ? (const void*)k_gen_local<1, kRotMma, true> : (const void*)k_gen_local<1, kRotMma, false>;
    default: return isl ? (const void*)k_gen_local<2, kRotTc, true> : (const void*)k_gen_local<2, kRotTc, false>;
  }
}

static size_t local_smem(const LocalPlan& p, const void* k) {
  const size_t need = local_layout(local_rot(p), p.kpad, p.dp_max, p.d_max, p.rotate).total;
  // with tensor memory: a whole SM (fp64_exclusive_smem: the cluster's CTAs
  // wait for one another while they hold it)
  return local_rot(p) == kRotTc ? fp64_exclusive_smem(k, need) : need;
}

static cudaLaunchConfig_t local_config(const LocalPlan& p, const void* k, int nruns, bool isl, cudaStream_t s,
                                       cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nruns * p.csize));
  cfg.blockDim = dim3(256);
  cfg.dynamicSmemBytes = local_smem(p, k);
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)p.csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  // the islands wait for one another: every cluster resident, or no launch
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = isl ? 2 : 1;
  return cfg;
}

// Whether the runs fit the form (np <= 64; sliced runs of d <= 64, or none
// sliced and d <= 32), and its launch.
bool local_plan(LocalPlan& p, const std::vector<RunDesc>& runs, const SlicePlan& sp) {
  p = LocalPlan{};
  int np_max = 0;
  p.sl = sp.on;
  for (const RunDesc& R : runs) {
    p.csize = 0;  // does not fit, unless it gets to the end
    if (R.np > kLocalNp || R.obj > kObjAckley || R.strategy != 0 || R.jde || R.dbg_trial) return false;
    if (sp.on != (R.sl != nullptr)) return false;
    if (R.d > (sp.on ? 64 : 32)) return false;
    np_max = std::max(np_max, R.np);
    p.d_max = std::max(p.d_max, R.d);
    p.dp_max = std::max(p.dp_max, R.dp);
    p.rotate = p.rotate || R.rotate;
  }
  p.csize = (np_max + 7) / 8;
  p.kpad = sp.kpad;
  p.cols = sp.cols;
  return true;
}

bool local_fits(const LocalPlan& p, int nruns, bool isl) {
  const void* k = local_kernel(p, isl);
  cudaLaunchAttribute attr[2];
  int n = 0;
  const cudaLaunchConfig_t cfg = local_config(p, k, nruns, isl, 0, attr);
  if (allow_dynamic_smem(k) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return n >= (isl ? nruns : 1);
}

cudaError_t k_gen_local_launch(const RunDesc* runs, int nruns, const LocalPlan& p, PersistCtl* ctl, long long gens,
                               cudaStream_t s, int test_skip, IslandCtl* isl, const IslandStage* stage) {
  cudaError_t e = persist_ctl_reset(ctl, test_skip, s);
  if (e != cudaSuccess) return e;
  IslandStage st{};
  if (stage) st = *stage;
  const void* k = local_kernel(p, isl != nullptr);
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = local_config(p, k, nruns, isl != nullptr, s, attr);
  int csize = p.csize, kpad = p.kpad, dp_max = p.dp_max;
  uint32_t cols = p.cols;
  void* args[] = {(void*)&runs, (void*)&ctl, (void*)&gens, (void*)&csize, (void*)&isl,
                  (void*)&st,   (void*)&kpad, (void*)&cols, (void*)&dp_max};
  return cudaLaunchKernelExC(&cfg, k, args);
}

}  // namespace de
