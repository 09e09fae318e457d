// de_slice.cuh -- the FP64 rotation z = M y as exact integer products on the
// tensor cores (an Ozaki-type splitting; Ozaki, Ogita, Oishi, Rump, Numerical
// Algorithms 59 (2012), with signed 8-bit digits in BF16 operands).
//
// Why: a DFMA warp instruction occupies a sub-partition's FP64 unit for 64
// cycles on this part (1.06 TFLOP/s in all), and the rotation is 2 d of the
// about 2 d + 55 FP64 operations of a coordinate.  BF16 tensor products run
// about 1800 times faster, so 43 digit products per FP64 product cost 2% of it.
//
// Arithmetic.  With 2^e > max_k |y_k| and 2^f_j > max_k |M_jk|,
//   U_k = round(y_k 2^(62 - e)),  V_jk = round(M_jk 2^(62 - f_j)),  |U|, |V| <= 2^62,
// each written in 8 signed digits of 8 bits (base 256, the digits in
// [-128, 127], the leading one in [-65, 65]).  A digit is exact in BF16, a
// product of two is exact, and for d <= 128 the sum over k of all digit
// products of one weight group g = s + t <= 8 stays below 2^24 in size, so
// its FP32 accumulation in tensor memory is exact:
//   P_g = sum_k sum_{s + t = g} u_s,k v_t,jk,   z_j = 2^(e + f_j - 76) sum_{g <= 8} 256^(8 - g) P_g
// with one rounding at the end (in integers; the sum is below 2^83).  What is
// lost: bits of y_k (M_jk) below 2^-63 of the row's largest, and the groups g >= 9.
// Of 2^(e + f_j) that is about 2^-64 as a rule, and at most about d 2^-67 (six
// pairs of digits of 128 in group 9 for every k; 2^-60 at d = 128).  A chain of d
// DFMAs rounds each of its sums to 2^-53 of it.
//
// A row is computed this way only when that comparison holds: with at least
// qmin = cM + ceil(d / 8) coordinates of size >= 2^-6 max|y| (cM: the most
// entries below 1/8 of a row of M's largest), every z_j sums at least d / 8
// products of size >= 2^-9 of the largest possible one (2^(e + f_j - 2) or more),
// whose sizes add up to d 2^-14 or more: the chain may lose d 2^-67 in a single
// rounding of such a sum, as much as is lost here at most.  Other rows (and rows
// with non-finite, subnormal or extreme values) take the DFMA chain,
// and matrices whose cM leaves no room (sparse ones) are not
// sliced at all, so no row is computed less precisely than by the chain.
//
// Operands: A = M (128 rows, rows past d zero), one slice per digit t,
// resident for as long as the CTA works on that matrix: the first nsm
// slices in shared memory (their products are the widest, which hides the
// 4 KB of A each reads), the others in tensor memory.  B = the digits of up to
// 8 rows of y: row 8 s + r holds digit s of tile row r, so that one product
// of slice t with digits 0 .. 8 - t adds its sums to the groups t .. 8, which
// lie side by side in tensor memory (10 groups x 8 columns).  8 products
// per 16 coordinates; 20 to 33 cycles each when issued from warp-uniform code
// under elect.sync (60 to 80 from a divergent branch).
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "de_device.cuh"
#include "de_tcgen05.cuh"

namespace de {

constexpr int kSliceIssuer = 7;     // the warp that issues the products
constexpr int kSlices = 8;          // digits per number
constexpr int kSliceRows = 8;       // rows of y per product
constexpr int kSliceDMin = 16;
constexpr int kSliceDMax = 128;     // largest d (the exactness bound and the 128 rows of A)
constexpr uint32_t kSliceKg = 1296; // bytes between 8-coordinate groups of B: 80 rows x 16, + 16 against bank conflicts
constexpr uint32_t kSliceAcc = 80;  // accumulator columns: 10 groups x 8 rows

__host__ __device__ inline int slice_kpad(int d) { return (d + 15) / 16 * 16; }
// bytes of one slice of M: kpad / 8 groups of 128 rows x 16 bytes
__host__ __device__ constexpr uint32_t slice_bytes(int kpad) { return (uint32_t)(kpad / 8) * 2048u; }
// slices kept in shared memory (the others fit tensor memory's 512 columns)
__host__ __device__ constexpr int slice_nsm(int kpad) {
  const int fit = (int)(512u - kSliceAcc) / (kpad / 2);
  return fit >= kSlices ? 0 : kSlices - fit;
}
__host__ __device__ inline uint32_t slice_tmem_cols(int kpad) {
  const uint32_t need = kSliceAcc + (uint32_t)(kSlices - slice_nsm(kpad)) * (uint32_t)(kpad / 2);
  return need <= 128u ? 128u : need <= 256u ? 256u : 512u;
}
// shared memory of the operands: B, then the resident slices
__host__ __device__ constexpr uint32_t slice_b_bytes(int kpad) { return ((uint32_t)(kpad / 8) * kSliceKg + 1023u) / 1024u * 1024u; }
__host__ __device__ constexpr uint32_t slice_smem(int kpad) { return slice_b_bytes(kpad) + (uint32_t)slice_nsm(kpad) * slice_bytes(kpad); }

// Its part in static shared memory.
struct SliceShared {
  double sum[2][4][kSliceRows];  // per quarter of the outputs and tile row: term sums
  double edge[4][kSliceRows];    // ... the quarter's first output (Rosenbrock)
  uint64_t bar;
  uint32_t tmem, bad;
  int fail;
  int exp[kSliceRows];
};

// One CTA's state of the sliced rotation (the same in every thread).
struct SliceCtx {
  SliceShared* sh;
  uint8_t* sB;       // B operand (1024-byte aligned)
  uint8_t* sA;       // slices resident in shared memory
  float* sP;         // mma.sync form: the group sums (de_slice_mma.cuh)
  uint32_t tmem;     // accumulators at column 0, slices from column kSliceAcc on
  uint32_t bar;      // mbarrier of the products
  uint32_t phase;
  int* s_exp;        // per tile row: e
  uint32_t* s_bad;   // bit r: tile row r takes the DFMA chain
  int* s_fail;       // set when a wait for the products gave up
  const uint8_t* cur;  // the matrix loaded (its slices in global memory)
  uint32_t cols;       // tensor-memory columns allocated
};

// The slices of one matrix (global layout = operand layout) into shared and
// tensor memory, by all threads of the CTA (256).
__device__ __forceinline__ void slice_load_m(SliceCtx& c, const uint8_t* __restrict__ sl, int kpad) {
  const int nsm = slice_nsm(kpad), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sbytes = slice_bytes(kpad);
  __syncthreads();  // no product of the previous matrix is in flight and none of its slices is being read
  for (uint32_t q = (uint32_t)tid * 16u; q < (uint32_t)nsm * sbytes; q += blockDim.x * 16u)
    *reinterpret_cast<uint4*>(c.sA + q) = __ldg(reinterpret_cast<const uint4*>(sl + q));
  // row r of a slice in lane r, 4 columns per 8-coordinate group; warps w and
  // w + 4 share the lanes 32 (w mod 4) .. + 31 and take alternate groups
  const int q4 = warp & 3, r = 32 * q4 + lane, nkg = kpad / 8;
  const uint32_t ta0 = c.tmem + ((uint32_t)(32 * q4) << 16) + kSliceAcc;
  const uint8_t* src = sl + (size_t)nsm * sbytes + (size_t)r * 16u;
  const int n = (kSlices - nsm) * nkg;  // slices are contiguous, so the groups are too
#pragma unroll 8
  for (int g = warp >> 2; g < n; g += 2) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(src + (size_t)g * 2048u));
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(ta0 + 4u * (uint32_t)g), "r"(v.x),
                 "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
  }
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  c.cur = sl;
}

// Allocates tensor memory, sets up the barrier and the zero rows of B; by
// all threads, before any other use.  kpad: the largest of the matrices this
// CTA will load (smem holds slice_smem(kpad) bytes), cols: their columns.
__device__ __forceinline__ void slice_begin(SliceCtx& c, uint8_t* smem, int kpad, uint32_t cols, SliceShared& sh) {
  c.sh = &sh;
  c.cols = cols;
  c.sB = smem;
  c.sA = smem + slice_b_bytes(kpad);
  c.bar = smem_u32(&sh.bar);
  c.phase = 0;
  c.s_exp = sh.exp;
  c.s_bad = &sh.bad;
  c.s_fail = &sh.fail;
  c.cur = nullptr;
  if (threadIdx.x == 0) {
    mbar_init(c.bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sh.bad = 0u;
    sh.fail = 0;
  }
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh.tmem)),
                 "r"(cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  for (uint32_t q = threadIdx.x * 16u; q < slice_b_bytes(kpad); q += blockDim.x * 16u)
    *reinterpret_cast<uint4*>(smem + q) = make_uint4(0u, 0u, 0u, 0u);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  c.tmem = sh.tmem;
}

// Waits (bounded) for products still in flight after a failed wait, then
// frees tensor memory; by all threads.
__device__ __forceinline__ void slice_end(SliceCtx& c) {
  if (threadIdx.x == 0 && *c.s_fail) mbar_wait(c.bar, c.phase ^ 1u);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(c.tmem), "r"(c.cols));
}

// Digits of one row of y into row r of the tile (one warp; lane L holds
// coordinates N L .. N L + N - 1, zero past d; N = 1, 2 or 4, 32 N >= kpad).
template <int N>
__device__ __forceinline__ void slice_digits(const SliceCtx& c, int r, int lane, int kpad, int qmin,
                                             const double (&y)[N]) {
  uint32_t hw[N], mx = 0u, any = 0u;
#pragma unroll
  for (int m = 0; m < N; ++m) {
    hw[m] = (uint32_t)__double2hiint(y[m]) & 0x7FFFFFFFu;
    mx = max(mx, hw[m]);
    any |= (uint32_t)__double2loint(y[m]);
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  const int ex = (int)(mx >> 20);  // 2^(ex - 1022) exceeds every |y_k|
  // coordinates of at least 2^-6 of the largest (by the high words)
  const uint32_t thr = mx > (6u << 20) ? mx - (6u << 20) : 1u;
  int q = 0;
#pragma unroll
  for (int m = 0; m < N; ++m) q += __popc(__ballot_sync(0xffffffffu, hw[m] >= thr));
  // a row of zeros is exact; z stays in the normal range for e in [-800, 800]
  const bool zero = mx == 0u && __all_sync(0xffffffffu, any == 0u);
  const bool bad = !zero && (q < qmin || ex < 1022 - 800 || ex > 1022 + 800);
  if (lane == 0) {
    c.s_exp[r] = ex - 1022;
    if (bad) atomicOr(c.s_bad, 1u << r);
  }
  if (N * lane >= kpad) return;
  uint32_t lo[N], hi[N];
#pragma unroll
  for (int m = 0; m < N; ++m) {
    const long long b = __double_as_longlong(y[m]);
    const int ek = (int)(hw[m] >> 20);
    // significand at bits 9 .. 61, shifted down to the row's exponent with
    // rounding (an exact shift by up to 9 bits)
    unsigned long long u = (((unsigned long long)b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL) << 9;
    const int sh = ex - ek;
    if (ek == 0 || sh > 62) u = 0ULL;
    else if (sh > 0) u = (u + (1ULL << (sh - 1))) >> sh;
    const long long v = (b < 0 ? -(long long)u : (long long)u) + (long long)0x8080808080808080ULL;
    lo[m] = (uint32_t)v;
    hi[m] = (uint32_t)((unsigned long long)v >> 32);
  }
  // byte s of v (from the top) is digit s plus 128; in the low byte of
  // 2^23 + byte, minus 2^23 + 128, it is the digit in FP32, whose upper half
  // is its exact BF16 form
  const uint32_t k0 = (uint32_t)(N * lane);
  uint8_t* dst = c.sB + (k0 >> 3) * kSliceKg + (uint32_t)r * 16u + (k0 & 7u) * 2u;
#pragma unroll
  for (int s = 0; s < kSlices; ++s) {
    float f[N];
#pragma unroll
    for (int m = 0; m < N; ++m) {
      const uint32_t w = s < 4 ? hi[m] : lo[m];
      f[m] = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7550u | (uint32_t)(3 - (s & 3)))) - 8388736.0f;
    }
    if constexpr (N == 1) {
      *reinterpret_cast<uint16_t*>(dst + s * 128) = (uint16_t)(__float_as_uint(f[0]) >> 16);
    } else if constexpr (N == 2) {
      *reinterpret_cast<uint32_t*>(dst + s * 128) = __byte_perm(__float_as_uint(f[0]), __float_as_uint(f[1]), 0x7632u);
    } else {
      uint2 p;
      p.x = __byte_perm(__float_as_uint(f[0]), __float_as_uint(f[1]), 0x7632u);
      p.y = __byte_perm(__float_as_uint(f[2]), __float_as_uint(f[3]), 0x7632u);
      *reinterpret_cast<uint2*>(dst + s * 128) = p;
    }
  }
}

// Issues the products of the tile's digits with the loaded matrix and waits
// for them; by all threads, after a CTA barrier that follows the digits.
__device__ __forceinline__ void slice_products(SliceCtx& c, int kpad) {
  const int lane = threadIdx.x & 31;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);
  if (warp == kSliceIssuer) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int nsm = slice_nsm(kpad), ksteps = kpad / 16;
    const uint32_t sbytes = slice_bytes(kpad);
    const uint64_t db0 = smem_desc(smem_u32(c.sB), kSliceKg, 128u);
    const uint64_t da0 = smem_desc(smem_u32(c.sA), 2048u, 128u);
    constexpr uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTileM >> 4) << 24);
    constexpr uint32_t bstep = (2u * kSliceKg) >> 4, astep = 4096u >> 4;
    if (elect_one()) {
#pragma unroll
      for (int t = 0; t < kSlices; ++t) {
        // digits 0 .. 8 - t (at most 8 of them, an even number: N is a multiple of 16)
        const uint32_t ns = t <= 2 ? 8u : (uint32_t)((10 - t) / 2 * 2);
        const uint32_t idesc = idesc0 | (ns << 17);
        const uint32_t dcol = c.tmem + (uint32_t)t * 8u;
        for (int ks = 0; ks < ksteps; ++ks) {
          const uint64_t db = db0 + (uint64_t)(bstep * (uint32_t)ks);
          // the first product also covers groups 8 and 9 (B's zero rows), so
          // that every group starts at zero
          const uint32_t id = t == 0 && ks == 0 ? (idesc0 | (10u << 17)) : idesc;
          const uint32_t acc = t == 0 && ks == 0 ? 0u : 1u;
          if (t < nsm)
            mma_split<2>(dcol, da0 + (uint64_t)((uint32_t)t * (sbytes >> 4) + astep * (uint32_t)ks), db, id, acc);
          else
            mma_split_ta<2>(dcol, c.tmem + kSliceAcc + (uint32_t)(t - nsm) * (uint32_t)(kpad / 2) + 8u * (uint32_t)ks, db,
                            id, acc);
        }
      }
      mma_commit(c.bar);
    }
    __syncwarp();
    const bool ok = mbar_wait(c.bar, c.phase);
    if (!__all_sync(0xffffffffu, ok) && lane == 0) *c.s_fail = 1;
  }
  c.phase ^= 1u;
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// The tile rows of warp w's threads: rows slice_row0 .. + slice_nrow - 1 (the
// two halves of the warps share the tile's rows evenly), outputs
// 32 (w mod 4) + lane.
__device__ __forceinline__ int slice_row0(int warp, int nrows) { return (warp >> 2) * ((nrows + 1) >> 1); }
__device__ __forceinline__ int slice_nrow(int warp, int nrows) {
  return warp < 4 ? (nrows + 1) >> 1 : nrows >> 1;
}

// sum_g 256^(8 - g) P_g 2^sc rounded once to FP64, in integers (three FP64
// operations would take 192 cycles of the FP64 pipe a warp and row).
__device__ __forceinline__ double slice_combine(const float (&p)[9], int sc) {
  int P[9];
#pragma unroll
  for (int g = 0; g < 9; ++g) P[g] = __float2int_rn(p[g]);
  const int a = P[0] * 256 + P[1], b = P[2] * 256 + P[3];
  const long long H = (long long)a * 16777216LL + ((long long)b * 256LL + P[4]);
  const long long L = ((long long)P[5] * 256LL + P[6]) * 65536LL + ((long long)P[7] * 256LL + P[8]);
  // T = H 2^32 + L, |T| < 2^83, as sign and magnitude (hi, lo); no branches,
  // so that a thread's rows run interleaved
  unsigned long long lo = ((unsigned long long)H << 32) + (unsigned long long)L;
  unsigned long long hi = (unsigned long long)((H >> 32) + (L >> 63) + (lo < (unsigned long long)L ? 1LL : 0LL));
  const bool neg = (long long)hi < 0;
  const unsigned long long m = neg ? ~0ULL : 0ULL;
  lo = (lo ^ m) + (neg ? 1ULL : 0ULL);
  hi = (hi ^ m) + (neg && lo == 0ULL ? 1ULL : 0ULL);
  // the leading 64 bits, with everything below as one sticky bit
  const bool wide = hi != 0ULL;
  const unsigned long long h2 = wide ? hi : lo, l2 = wide ? lo : 0ULL;
  const int lz = __clzll((long long)h2);  // 64 for T = 0
  const unsigned long long n = (h2 << (lz & 63)) | ((l2 >> 1) >> (63 - (lz & 63)));
  const unsigned long long rest = l2 << (lz & 63);
  unsigned long long k = n >> 11;
  const unsigned int rem = ((unsigned int)n & 0x7FFu) | (rest ? 1u : 0u);
  k += (rem > 0x400u || (rem == 0x400u && (k & 1ULL))) ? 1ULL : 0ULL;
  const long long e = 1023 + 126 - 64 - lz + (wide ? 64 : 0) + sc;
  const double z = __longlong_as_double((long long)(((unsigned long long)e << 52) + k) | (neg ? (long long)0x8000000000000000ULL : 0LL));
  return h2 == 0ULL ? 0.0 : z;
}

// z of this thread's output and rows from the accumulators (after
// slice_products); rows past the tile and outputs past d give 0.  A row that
// takes the DFMA chain is computed over MT from Y (FP64 rows of stride dp)
// into Zf (as Y).
__device__ __forceinline__ void slice_z(SliceCtx& c, const int32_t* __restrict__ fexp, const double* __restrict__ MT,
                                        const double* __restrict__ Y, double* __restrict__ Zf, int nrows, int d, int dp,
                                        double (&z)[4]) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int q4 = warp & 3, r0 = slice_row0(warp, nrows), nr = slice_nrow(warp, nrows), j = 32 * q4 + lane;
#pragma unroll
  for (int e = 0; e < 4; ++e) z[e] = 0.0;
  if (nr > 0 && 32 * q4 < d) {
    uint32_t v[9][4];
    const uint32_t ta = c.tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)r0;
#pragma unroll
    for (int g = 0; g < 9; ++g)
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                   : "=r"(v[g][0]), "=r"(v[g][1]), "=r"(v[g][2]), "=r"(v[g][3])
                   : "r"(ta + 8u * (uint32_t)g));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    // the values are used only after the wait
#pragma unroll
    for (int g = 0; g < 9; ++g)
      asm volatile("" : "+r"(v[g][0]), "+r"(v[g][1]), "+r"(v[g][2]), "+r"(v[g][3]));
    const int fj = j < d ? __ldg(fexp + j) : 0;
    // rows past the tile (at most one here) are computed and dropped
    auto rows = [&](auto count) {
#pragma unroll
      for (int e = 0; e < decltype(count)::value; ++e) {
        float p[9];
#pragma unroll
        for (int g = 0; g < 9; ++g) p[g] = __uint_as_float(v[g][e]);
        const double ze = slice_combine(p, c.s_exp[min(r0 + e, kSliceRows - 1)] + fj - 76);
        z[e] = j < d && e < nr ? ze : 0.0;
      }
    };
    if (nr > 2) rows(std::integral_constant<int, 4>{});
    else rows(std::integral_constant<int, 2>{});
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  const uint32_t bad = *c.s_bad;
  if (bad) {
    // rows outside the splitting's comparison: one DFMA chain per output
    __syncthreads();
    if (tid == 0) *c.s_bad = 0u;
    for (int e = tid; e < nrows * d; e += (int)blockDim.x) {
      const int r = e / d, jj = e - r * d;
      if (!((bad >> r) & 1u)) continue;
      double s = 0.0;
      for (int k = 0; k < d; ++k) s = fma(__ldg(MT + (size_t)k * d + jj), Y[r * dp + k], s);
      Zf[r * dp + jj] = s;
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (e < nr && j < d && ((bad >> (r0 + e)) & 1u)) z[e] = Zf[(r0 + e) * dp + j];
  }
}

// z into Z[r][j] (row stride dp) for the tile's rows.  The caller's CTA
// barrier makes Z visible.
__device__ __forceinline__ void slice_rotate(SliceCtx& c, int kpad, const int32_t* __restrict__ fexp,
                                             const double* __restrict__ MT, const double* __restrict__ Y,
                                             double* __restrict__ Z, int nrows, int d, int dp) {
  const int warp = threadIdx.x >> 5, j = 32 * (warp & 3) + (threadIdx.x & 31);
  slice_products(c, kpad);
  double z[4];
  slice_z(c, fexp, MT, Y, Z, nrows, d, dp, z);
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (e < slice_nrow(warp, nrows) && j < d) Z[(slice_row0(warp, nrows) + e) * dp + j] = z[e];
}

// Sums of 4 rows' values over the lanes of a warp: 6 FP64 additions (the lanes
// of bit 16, then of bit 8, keep half of the rows each) instead of 20.  The lanes of
// (bit 16, bit 8) return the sum of row 2 (bit 16) + (bit 8); a row's order of
// additions does not depend on its place.
__device__ __forceinline__ double slice_sum4(const double (&v)[4], int lane) {
  const bool h = lane & 16, g = lane & 8;
  const double b0 = h ? v[0] : v[2], b1 = h ? v[1] : v[3];
  const double a0 = (h ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, b0, 16);
  const double a1 = (h ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, b1, 16);
  double s = (g ? a1 : a0) + __shfl_xor_sync(0xffffffffu, g ? a0 : a1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// Fitness of the tile's rows (objectives 0 .. 3), after a CTA barrier that
// follows the digits: products, z in registers, the objective's terms in the
// thread that holds z, sums over lanes and then over the four quarters of
// the outputs.  Warp r < nrows returns the fitness of row r (every lane).
__device__ __forceinline__ double slice_fitness(SliceCtx& c, const RunDesc& R, const double* __restrict__ Y,
                                                double* __restrict__ Zf, int nrows) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q4 = warp & 3;
  const int d = R.d, dp = R.dp, obj = R.obj, j = 32 * q4 + lane;
  const int r0 = slice_row0(warp, nrows), nr = slice_nrow(warp, nrows);
  slice_products(c, R.sl_kpad);
  double z[4], t[4], u[4];
  slice_z(c, R.slx, R.MT, Y, Zf, nrows, d, dp, z);
  if (obj == kObjRosenbrock) {
    // the next quarter's first output
    if (lane == 0) {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (e < nr) c.sh->edge[q4][r0 + e] = z[e];
    }
    __syncthreads();
  }
  if (nr > 0 && 32 * q4 < d) {
    const int srow = ((lane >> 4) & 1) * 2 + ((lane >> 3) & 1);
#pragma unroll
    for (int e = 0; e < 4; ++e) t[e] = u[e] = 0.0;
    // z is 0 past the tile's rows and past d, where every term but
    // Rosenbrock's is 0 (Ackley's cosine is masked)
    auto terms = [&](auto count) {
      constexpr int N = decltype(count)::value;
      if (obj == kObjRosenbrock) {
#pragma unroll
        for (int e = 0; e < N; ++e) {
          double zn = __shfl_down_sync(0xffffffffu, z[e], 1);
          if (lane == 31 && q4 < 3 && e < nr) zn = c.sh->edge[q4 + 1][r0 + e];
          const double t0 = z[e] + 1.0, tn = zn + 1.0;
          const double a = tn - t0 * t0, b = t0 - 1.0;
          t[e] = e < nr && j + 1 < d ? 100.0 * a * a + b * b : 0.0;
        }
      } else if (obj == kObjRastrigin) {
#pragma unroll
        for (int e = 0; e < N; ++e) t[e] = fma(z[e], z[e], rastrigin_w(z[e]));
      } else {
#pragma unroll
        for (int e = 0; e < N; ++e) t[e] = z[e] * z[e];
        if (obj == kObjAckley) {
#pragma unroll
          for (int e = 0; e < N; ++e) {
            const double w = cos2pi_fix(z[e]);
            u[e] = e < nr && j < d ? w : 0.0;
          }
        }
      }
    };
    if (nr > 2) terms(std::integral_constant<int, 4>{});
    else terms(std::integral_constant<int, 2>{});
    const double s = slice_sum4(t, lane);
    if ((lane & 7) == 0 && srow < nr) c.sh->sum[0][q4][r0 + srow] = s;
    if (obj == kObjAckley) {
      const double s2 = slice_sum4(u, lane);
      if ((lane & 7) == 0 && srow < nr) c.sh->sum[1][q4][r0 + srow] = s2;
    }
  }
  __syncthreads();
  if (warp >= nrows) return 0.0;
  double s1 = c.sh->sum[0][0][warp];
  for (int q = 1; 32 * q < d; ++q) s1 += c.sh->sum[0][q][warp];
  if (obj != kObjAckley) return s1;
  double s2 = c.sh->sum[1][0][warp];
  for (int q = 1; 32 * q < d; ++q) s2 += c.sh->sum[1][q][warp];
  return ackley_value((lane & 1 ? s2 : s1) / d, lane);
}

}  // namespace de
