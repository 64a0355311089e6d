// FP64 grade product on the tensor cores: gamma_i = max_p |(b_i A^-1)_p| (Section II.D) with FP64
// rows, from exact integer products.
//
// GB300 does 2 FP64 FMAs per clock and SM, so the SIMT product of 16,384 rows with m = 651 takes
// 11 ms at that rate.  Here both factors are cut into slices of 7 bits (the error-free splitting of
// Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012): with X = A^-1,
//   row k of X scaled by 2^-g_k and column k of B by 2^g_k (so that no row of X outweighs another),
//   row i of B scaled by 2^-E_i, column p of X by 2^-f_p, entries below 1 in magnitude,
//   t = sum_{s < 9} d_s 2^(-6 - 7 s), digits |d_s| <= 64 as bf16 integers (63 bits of the row's
//   largest entry, 10 more than the factors have),
//   C_ip = 2^(E_i + f_p) sum_{s + t < 9} 2^(-12 - 7 (s + t)) sum_k d_s,ik d'_t,kp.
// The inner sums run as tcgen05.mma kind::f16 with FP32 accumulation in tensor memory: products of
// digits are at most 2^12, so a sum of K of them over up to 4096 / K slice pairs is an integer of at most
// 2^24, exact in FP32; such groups of pairs with equal s + t share an accumulator (12 of them at
// m = 651, in two sweeps over K).  The epilogue adds the accumulators as 64-bit integers and rounds to
// FP64 once per sweep.
//
// Precision.  The sums are exact; what is lost is the fixed point of the operands (an entry more than
// 2^10 below the largest of its scaled row or column keeps fewer than its 53 bits) and the slice pairs
// with s + t >= 9: at most 1.3 2^-60 2^(E_i + f_p) per term.  FP64 accumulation loses up to
// 2^-53 sum_k |b_k X_kp| in each of its m steps, which is more as long as that sum is at least
// 2^(E_i + f_p - 6), the largest product or a 64th of it.  k_check_fp64 bounds it from below for the column
// that wins, by the leading digits; a row where it is not shown (large terms that cancel exactly beside
// a column of small ones) is redone by plain FP64 sums, like the rows that hold an infinity or NaN and
// all rows where X holds one.  (Host emulation, 21 sets of cond 1 to 1e18, levels 8 to 20: 2 of 17,544
// rows redone; the sums are 3 to 500 times the limit.)
//
// One persistent CTA per SM as in grade_tc.cu: warp 0 TMA producer (all 18 slices of a 64-wide K
// chunk, one stage of 216 KB, 128B swizzle), warp 1 tcgen05.mma issuer (M 128, N 64, K 16), warps 2-9
// epilogue, a row and 32 columns per thread.  Every wait is bounded, with the same drain.
// 16,384 rows, m = 651: 14.8 -> 1.21 ms (slicing 0.16, product 1.01: 66 clocks per MMA, bound by reading the
// 128-row operand from shared memory; an N of 32 took as long per MMA).
#include <algorithm>
#include <type_traits>

#include "profiler.h"
#include "tc.h"

namespace mtp {

void run_grade_simt(mtp_model* md, int64_t N, bool fp64, const double* rows, const float* rows_f, int64_t ld,
                    double* gamma, int32_t* argmax, cudaStream_t s);

namespace {

constexpr int NS = 9;              // slices
constexpr int FM = 128;            // rows per tile
constexpr int FN = 64;             // columns per tile (32: the same time per MMA, half the work)
constexpr int EN = 32;             // columns per epilogue thread
constexpr int FK = 64;             // digits per 128-byte swizzle row
constexpr int FSTEP = 16;          // K per tcgen05.mma kind::f16
constexpr int FA = FM * FK * 2;    // one slice of a row tile's chunk: 16 KB
constexpr int FB = FN * FK * 2;    // 8 KB
constexpr int SEG = 768;           // K per accumulation (digits' sums below 2^24 with 5 pairs)
constexpr int S1 = 5;              // slice sums s < S1 in a first sweep over K, the others in a second: at most
                                   // 8 accumulators of FN columns each, the 512 of tensor memory
constexpr int FTHREADS = 64 + 256;
constexpr size_t FSMEM = NS * (FA + FB) + 256 + 1024;
// rows sliced at a time: 0.8 GB of slices at m = 651, at most 1 GB, down to kLeastRows where memory is
// short (16 row tiles: still more tiles than SMs from m = 577 on)
constexpr int64_t kChunkRows = 65536, kLeastRows = 2048;
constexpr size_t kSliceBytes = size_t(1) << 30;

// exponent e with |v| < 2^e (v finite), a very low one for zero
__device__ __forceinline__ int exponent_of(double v) {
  const int e = static_cast<int>((__double_as_longlong(v) >> 52) & 0x7ff);
  return e ? e - 1022 : (v == 0.0 ? -4000 : -1021);
}

// v 2^shift rounded to an integer, as NS digits of 7 bits, most significant first
__device__ __forceinline__ void digits_of(double v, int shift, uint16_t (&d)[NS]) {
  long long f = __double2ll_rn(scalbn(v, shift));
#pragma unroll
  for (int s = NS - 1; s > 0; --s) {
    const int low = static_cast<int>(f & 127);
    const int dig = low >= 64 ? low - 128 : low;
    f = (f - dig) >> 7;
    d[s] = static_cast<uint16_t>(__float_as_uint(static_cast<float>(dig)) >> 16);
  }
  d[0] = static_cast<uint16_t>(__float_as_uint(static_cast<float>(f)) >> 16);
}

// a warp per row k; *xbad (starts 0) = 1 where X has an infinity or NaN (an inverse can overflow: its
// pivots are judged against max |A|)
__global__ void k_x_row_scale(const double* X, int64_t m, int* g, int* f, int* xbad) {
  const int64_t k = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
  if (k >= m) return;
  int e = -4000;
  for (int64_t p = threadIdx.x & 31; p < m; p += 32) e = max(e, exponent_of(X[k * m + p]));
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) {
    g[k] = e < -3000 ? 0 : e;
    f[k] = -4000;
    if (e > 1024) *xbad = 1;   // exponent field 0x7ff
  }
}

__global__ void k_x_col_scale(const double* X, int64_t m, const int* g, int* f) {   // f starts very low
  const int64_t p = blockIdx.x * 32LL + (threadIdx.x & 31);
  if (p >= m) return;
  int e = -4000;
  for (int64_t k = blockIdx.y * 8LL + (threadIdx.x >> 5); k < m; k += 8LL * gridDim.y) {
    const int x = exponent_of(X[k * m + p]);
    if (x > -3000) e = max(e, x - g[k]);
  }
  if (e > -4000) atomicMax(f + p, e);
}

// slices of X transposed: out[s][p][k], zero past m (kp = K rounded up to FK, pp = rows of a slice)
__global__ void k_slice_x(const double* X, int64_t m, const int* g, const int* f, int kp, int pp, uint16_t* out) {
  const int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (e >= static_cast<int64_t>(kp) * pp) return;
  const int p = static_cast<int>(e / kp), k = static_cast<int>(e - static_cast<int64_t>(p) * kp);
  uint16_t d[NS];
  digits_of((p < m && k < m) ? X[k * m + p] : 0.0, (p < m && k < m) ? 62 - g[k] - f[p] : 0, d);
#pragma unroll
  for (int s = 0; s < NS; ++s) out[static_cast<int64_t>(s) * pp * kp + e] = d[s];
}

// slices of the rows r0 .. r0 + n - 1 of B: out[s][r][k] (np rows per slice), their exponents, and
// bad[r] where a row is not finite (every row where X is not).  A warp per row.
__global__ void __launch_bounds__(256) k_slice_rows(const double* __restrict__ B, int64_t ldb, int64_t m, int64_t n, const int* g, const int* xbad,
                                                    int kp, int64_t np, uint16_t* out, int* E, unsigned char* bad) {
  const int64_t r = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
  if (r >= n) return;
  const int lane = threadIdx.x & 31;
  const double* b = B + r * ldb;
  int e = -4000;
  bool nonfinite = *xbad != 0;
  for (int64_t k = lane; k < m; k += 32) {
    const double v = b[k];
    nonfinite |= ((__double_as_longlong(v) >> 52) & 0x7ff) == 0x7ff;
    const int x = exponent_of(v);
    if (x > -3000) e = max(e, x + g[k]);
  }
  e = __reduce_max_sync(0xffffffffu, e);
  nonfinite = __any_sync(0xffffffffu, nonfinite);
  if (e < -3000 || nonfinite) e = 0;
  if (lane == 0) {
    E[r] = e;
    if (nonfinite) bad[r] = 1;
  }
  for (int k = 2 * lane; k < kp; k += 64) {   // two digits of a slice per store
    uint16_t d0[NS], d1[NS];
    digits_of((k < m && !nonfinite) ? b[k] : 0.0, k < m ? 62 + g[k] - e : 0, d0);
    digits_of((k + 1 < m && !nonfinite) ? b[k + 1] : 0.0, k + 1 < m ? 62 + g[k + 1] - e : 0, d1);
#pragma unroll
    for (int s = 0; s < NS; ++s)
      *reinterpret_cast<uint32_t*>(out + (static_cast<int64_t>(s) * np + r) * kp + k) =
          d0[s] | (static_cast<uint32_t>(d1[s]) << 16);
  }
}

struct F64Args {
  int64_t N;           // rows of this chunk
  int64_t np;          // rows of a slice
  int m, pp;           // valid columns, rows of a slice of X
  int n_col;           // column tiles
  int k_chunks;        // K chunks of FK
  int64_t n_work;      // row tiles * n_col
  int maxp;            // slice pairs per accumulator
  const int* f;        // column exponents
  double* pbest;       // [n_best x N], n_best groups of EN columns
  int32_t* parg;
  unsigned* err;
  uint32_t wait_limit;
};

__global__ void __launch_bounds__(FTHREADS, 1) k_grade_fp64(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB,
                                                            F64Args a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + NS * (FA + FB));
  uint64_t* full = bars;
  uint64_t* empty = bars + 1;
  uint64_t* accf = bars + 2;
  uint64_t* acce = bars + 3;
  uint64_t* drain = bars + 4;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars + 6);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(full, 1);
    mbar_init(empty, 1);
    mbar_init(accf, 1);
    mbar_init(acce, 8);
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  constexpr int SEGC = SEG / FK;   // chunks per accumulation

  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;
      for (int64_t w = blockIdx.x; w < a.n_work && !*abort_flag; w += gridDim.x) {
        const int64_t tile = w / a.n_col;
        const int col = static_cast<int>(w - tile * a.n_col);
        for (int k0 = 0; k0 < a.k_chunks && !*abort_flag; k0 += SEGC)
          for (int sweep = 0; sweep < 2 && !*abort_flag; ++sweep)
            for (int kc = k0; kc < min(k0 + SEGC, a.k_chunks); ++kc, ++it) {
              if (it > 0 && !mbar_wait(empty, (it - 1) & 1, abort_flag, a.wait_limit)) { *abort_flag = 1; break; }
              const int ns = sweep ? NS : S1;   // the first sweep needs slices 0 .. S1 - 1 only
              mbar_expect_tx(full, ns * (FA + FB));
              for (int s = 0; s < ns; ++s) {
                tma_load_2d(smem + s * FA, &mA, kc * FK, static_cast<int>(s * a.np + tile * FM), full);
                tma_load_2d(smem + NS * FA + s * FB, &mB, kc * FK, s * a.pp + col * FN, full);
              }
            }
      }
      if (*abort_flag && it > 0) {   // the copies already issued land before shared memory goes away
        volatile int no_abort = 0;
        mbar_wait(full, (it - 1) & 1, &no_abort);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // D FP32, A and B bf16, both K-major
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(FN >> 3) << 17) |
                             (static_cast<uint32_t>(FM >> 4) << 24);
      const uint64_t da0 = smem_desc(smem), db0 = smem_desc(smem + NS * FA);
      uint32_t it = 0, acc_it = 0;
      bool issued = false;
      // the pairs (q, s - q) of the sums [lo, hi); descriptors by addition (addresses in units of 16
      // bytes: building each took longer than its MMA)
      auto chunk = [&](auto Lo, auto Hi, bool fresh) {
        uint32_t dt = tmem;
#pragma unroll
        for (int s = decltype(Lo)::value; s < decltype(Hi)::value; ++s) {
          int left = a.maxp;   // pairs the accumulator still takes
#pragma unroll
          for (int q = 0; q <= s; ++q) {
            if (left == 0) { dt += FN; left = a.maxp; }
            const uint64_t da = da0 + q * (FA >> 4), db = db0 + (s - q) * (FB >> 4);
            const uint32_t add = (fresh && left == a.maxp) ? 0u : 1u;
            mma_f16(dt, da, db, idesc, add);
#pragma unroll
            for (int ks = 1; ks < FK / FSTEP; ++ks)
              mma_f16(dt, da + ks * (FSTEP * 2 >> 4), db + ks * (FSTEP * 2 >> 4), idesc, 1u);
            --left;
          }
          dt += FN;
        }
      };
      for (int64_t w = blockIdx.x; w < a.n_work && !*abort_flag; w += gridDim.x)
        for (int k0 = 0; k0 < a.k_chunks && !*abort_flag; k0 += SEGC)
          for (int sweep = 0; sweep < 2 && !*abort_flag; ++sweep) {
            // the epilogue has read the last accumulation
            if (acc_it > 0 && !mbar_wait(acce, (acc_it - 1) & 1, abort_flag, a.wait_limit)) { *abort_flag = 1; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int kc = k0; kc < min(k0 + SEGC, a.k_chunks); ++kc, ++it) {
              if (!mbar_wait(full, it & 1, abort_flag, a.wait_limit)) { *abort_flag = 1; break; }
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              if (sweep == 0) chunk(std::integral_constant<int, 0>{}, std::integral_constant<int, S1>{}, kc == k0);
              else chunk(std::integral_constant<int, S1>{}, std::integral_constant<int, NS>{}, kc == k0);
              issued = true;
              mma_commit(empty);
            }
            if (*abort_flag) break;
            mma_commit(accf);
            ++acc_it;
          }
      if (issued) {   // all MMAs of this thread complete before tensor memory is released
        mma_commit(drain);
        volatile int no_abort = 0;
        mbar_wait(drain, 0, &no_abort);
      }
    }
    __syncwarp();
  } else {
    const int quarter = warp & 3;            // tensor-memory lane quarter of this warp
    const int half = (warp - 2) >> 2;        // columns 32 half .. of the tile
    uint32_t acc_it = 0;
    // (an abort ends the walk at the next wait, by lane 0 for the whole warp: lanes that read the flag
    // themselves could leave a warp whose others wait for them)
    for (int64_t w = blockIdx.x; w < a.n_work; w += gridDim.x) {
      const int64_t tile = w / a.n_col;
      const int col0 = static_cast<int>(w - tile * a.n_col) * FN + half * EN;
      double c[EN];
#pragma unroll
      for (int j = 0; j < EN; ++j) c[j] = 0.0;
      bool ok = true;
      for (int k0 = 0; k0 < a.k_chunks && ok; k0 += SEGC)
        for (int sweep = 0; sweep < 2; ++sweep, ++acc_it) {
          if (lane == 0) ok = mbar_wait(accf, acc_it & 1, abort_flag, a.wait_limit);
          ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          uint32_t ta = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + half * EN;
          // sums of equal s + t as integers: sum_s T_s 128^(last s of the sweep - s)
          long long h[EN];
#pragma unroll
          for (int j = 0; j < EN; ++j) h[j] = 0;
          const int s0 = sweep ? S1 : 0, s1 = sweep ? NS : S1;
          for (int s = s0; s < s1; ++s)
            for (int q = 0; q <= s; q += a.maxp, ta += FN) {
              float v[32];
              tmem_ld32(ta, v);
#pragma unroll
              for (int j = 0; j < EN; ++j) h[j] = (q == 0 ? h[j] * 128 : h[j]) + __float2int_rn(v[j]);
            }
          const double scale = sweep ? 0x1p-68 : 0x1p-40;   // 2^(-12 - 7 * 8), 2^(-12 - 7 * 4)
#pragma unroll
          for (int j = 0; j < EN; ++j) c[j] = fma(static_cast<double>(h[j]), scale, c[j]);
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(acce);
        }
      if (!ok) { if (lane == 0) *abort_flag = 1; break; }
      double best = -1.0;
      int barg = 0;
#pragma unroll
      for (int j = 0; j < EN; ++j) {
        const int p = col0 + j;
        if (p < a.m) {
          const double v = scalbn(fabs(c[j]), a.f[p]);
          if (abs_key(v) > (best < 0.0 ? -1 : abs_key(best))) { best = v; barg = p; }
        }
      }
      const int64_t row = tile * FM + quarter * 32 + lane;
      if (row < a.N) {
        a.pbest[static_cast<int64_t>(col0 / EN) * a.N + row] = best;
        a.parg[static_cast<int64_t>(col0 / EN) * a.N + row] = barg;
      }
    }
  }
  if (threadIdx.x == 0 && *abort_flag) atomicOr(a.err, 1u);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
}

// gamma and argmax of the chunk's rows from the column tiles' maxima (in column order, strict '>');
// the argmax also over parg's first plane
__global__ void k_combine_fp64(int64_t N, int n_best, const double* pbest, int32_t* parg, const int* E, double* gamma,
                               int32_t* argmax) {
  const int64_t r = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (r >= N) return;
  double best = -1.0;
  int arg = 0;
  bool nan = false;
  for (int p = 0; p < n_best; ++p) {
    const double v = pbest[p * N + r];
    nan = nan || v != v;
    if (v > best) { best = v; arg = parg[p * N + r]; }
  }
  gamma[r] = nan ? __longlong_as_double(0x7ff8000000000000LL) : scalbn(best, E[r]);
  parg[r] = arg;
  if (argmax) argmax[r] = arg;
}

// bad[r] where sum_k |b_k X_kp| of the winning column is not shown to be at least 2^(E + f - 6): with the
// leading digits d, d' of the scaled entries (|entry| >= (|d| - 1/2) / 64 where d is not 0) it is at least
// 2^(E + f) sum (2 |d| - 1)(2 |d'| - 1) / 2^14.  A warp per row; rows of slice 0 only, so 2 x 2 kp bytes.
// (Unfinished rows, gamma NaN, stay.)
__global__ void __launch_bounds__(256) k_check_fp64(int64_t N, int kp, const uint16_t* __restrict__ sl, const uint16_t* __restrict__ xs,
                                                    const int32_t* arg, const double* gamma, unsigned char* bad) {
  const int64_t r = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
  if (r >= N) return;
  const int lane = threadIdx.x & 31;
  const uint32_t* a = reinterpret_cast<const uint32_t*>(sl + r * kp);
  const uint32_t* x = reinterpret_cast<const uint32_t*>(xs + static_cast<int64_t>(arg[r]) * kp);
  auto weight = [](uint32_t bf16_bits) {
    const float d = fabsf(__uint_as_float(bf16_bits << 16));
    return d > 0.f ? d + d - 1.f : 0.f;
  };
  float sum = 0.f;
  for (int k = lane; k < kp / 2; k += 32) {
    const uint32_t u = a[k], v = x[k];
    sum = fmaf(weight(u & 0xffffu), weight(v & 0xffffu), sum);
    sum = fmaf(weight(u >> 16), weight(v >> 16), sum);
  }
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0 && !(sum >= 256.f) && gamma[r] == gamma[r]) bad[r] = 1;
}

// Marked rows by plain FP64 sums over k (the arithmetic, order and comparisons of the SIMT kernel): a
// block per 32 rows, a thread per column of a row at a time.  Bound by FP64 (2 FMAs per clock and SM),
// so a row costs a block 0.1 ms at m = 651 where the SIMT kernel's tile of 64 rows takes 7.
constexpr int kRedoRows = 32;
__global__ void __launch_bounds__(256) k_redo_rows(const double* __restrict__ B, int64_t ldb, const double* __restrict__ X, int64_t m,
                                                   int64_t N, const unsigned char* bad, double* gamma, int32_t* argmax) {
  __shared__ double s_v[8];
  __shared__ int s_p[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t r0 = blockIdx.x * static_cast<int64_t>(kRedoRows);
  unsigned marked = __ballot_sync(0xffffffffu, r0 + lane < N && bad[r0 + lane] != 0);   // the same in every warp
  while (marked) {
    const int64_t r = r0 + __ffs(marked) - 1;
    marked &= marked - 1;
    const double* b = B + r * ldb;
    double best = -1.0;
    int arg = 0;
    for (int64_t p = threadIdx.x; p < m; p += 256) {
      double acc = 0.0;
#pragma unroll 8
      for (int64_t k = 0; k < m; ++k) acc = fma(b[k], X[k * m + p], acc);
      const double v = fabs(acc);
      if (v > best) { best = v; arg = static_cast<int>(p); }
    }
    auto take = [&](double v, int p) {
      if (v > best || (v == best && p < arg)) { best = v; arg = p; }
    };
    for (int o = 16; o; o >>= 1) {
      const double v = __shfl_xor_sync(0xffffffffu, best, o);
      const int p = __shfl_xor_sync(0xffffffffu, arg, o);
      take(v, p);
    }
    if (lane == 0) { s_v[w] = best; s_p[w] = arg; }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int u = 1; u < 8; ++u) take(s_v[u], s_p[u]);
      gamma[r] = best;
      if (argmax) argmax[r] = arg;
    }
    __syncthreads();
  }
}

CUtensorMap slice_map(const uint16_t* base, int64_t rows, int64_t kp, int box_rows) {
  CUtensorMap t;
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(kp), static_cast<cuuint64_t>(rows)};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(kp) * 2};
  const cuuint32_t box[2] = {FK, static_cast<cuuint32_t>(box_rows)};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = encode_fn()(&t, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(base), dims, strides, box, estr,
                                 CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                                 CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw Fail{MTP_ERR_CUDA, "cuTensorMapEncodeTiled failed"};
  return t;
}

unsigned nblk(int64_t n, int t) { return static_cast<unsigned>((n + t - 1) / t); }

struct XPlan {
  int kp, pp;
  size_t bytes;
  int *g, *f, *xbad;
  uint16_t* slices;
};

XPlan x_plan(int64_t m, void* base) {
  XPlan x;
  x.kp = static_cast<int>((m + FK - 1) / FK * FK);
  x.pp = static_cast<int>((m + FN - 1) / FN * FN);
  const size_t head = ((2 * static_cast<size_t>(m) + 1) * sizeof(int) + 255) & ~size_t(255);
  x.bytes = head + static_cast<size_t>(NS) * x.pp * x.kp * sizeof(uint16_t);
  x.g = static_cast<int*>(base);
  x.f = x.g + m;
  x.xbad = x.f + m;
  x.slices = reinterpret_cast<uint16_t*>(static_cast<char*>(base) + head);
  return x;
}

}  // namespace

// from m = 64 on the slices pay: the SIMT kernel's time goes by column tiles of 64 (m = 54 79 us for 108
// atoms and 144 for 16,384; m = 75 186 and 348, where the slices take 68 and 135)
bool grade_fp64_sliced(int64_t m) { return m >= 64 && m <= 16384; }

// slices of A^-1; without the memory for them (18 m^2 bytes) the SIMT kernel grades
void slice_active_inverse(mtp_model* md, int64_t m, cudaStream_t s) {
  md->have_slices = grade_fp64_sliced(m) && md->ainv_s.try_ensure(x_plan(m, nullptr).bytes, s);
  if (!md->have_slices) return;
  const XPlan x = x_plan(m, md->ainv_s.p);
  const double* X = md->ainv_d.as<double>();
  MTP_CUDA(cudaMemsetAsync(x.xbad, 0, sizeof(int), s));
  k_x_row_scale<<<nblk(m * 32, 256), 256, 0, s>>>(X, m, x.g, x.f, x.xbad);
  ProfRegion::launched();
  k_x_col_scale<<<dim3(nblk(m, 32), 16), 256, 0, s>>>(X, m, x.g, x.f);
  ProfRegion::launched();
  k_slice_x<<<nblk(static_cast<int64_t>(x.kp) * x.pp, 256), 256, 0, s>>>(X, m, x.g, x.f, x.kp, x.pp, x.slices);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
}

namespace {

// ws_grade for chunks of cn of N rows
struct RowPlan {
  int64_t np;
  int n_best;
  size_t sl, e, best, arg, bad;
  RowPlan(const XPlan& x, int64_t cn, int64_t N)
      : np((cn + FM - 1) / FM * FM),
        n_best(x.pp / EN),
        sl(static_cast<size_t>(NS) * np * x.kp * sizeof(uint16_t)),
        e((np * sizeof(int) + 255) & ~size_t(255)),
        best(static_cast<size_t>(n_best) * cn * sizeof(double)),
        arg(static_cast<size_t>(n_best) * cn * sizeof(int32_t)),
        bad(static_cast<size_t>(N)) {}
  size_t bytes() const { return sl + e + best + arg + bad + 256; }
};

// Takes the workspace of an FP64 grade of N rows; returns the rows it grades at a time, 0 where the SIMT
// kernel has to (no slices of A^-1, or no memory even for chunks of kLeastRows).  Asked for once the site
// pass is enqueued: the host's allocation of up to a GB (0.2 ms) then lies beside it.
int64_t reserve(mtp_model* md, int64_t N, cudaStream_t s) {
  if (!md->have_slices || N == 0) return 0;
  const XPlan x = x_plan(md->m_active, md->ainv_s.p);
  const int64_t fit = static_cast<int64_t>(kSliceBytes / (static_cast<size_t>(NS) * x.kp * sizeof(uint16_t))) / FM * FM;
  int64_t cn = std::min<int64_t>(N, std::max(kLeastRows, std::min(kChunkRows, fit)));
  while (!md->ws_grade.try_ensure(RowPlan(x, cn, N).bytes(), s)) {
    if (cn <= kLeastRows) return 0;
    cn = std::max(kLeastRows, cn / 2 / FM * FM);
  }
  return cn;
}

}  // namespace

void run_grade_fp64(mtp_model* md, int64_t N, const double* rows, int64_t ld, double* gamma, int32_t* argmax, cudaStream_t s) {
  const int64_t m = md->m_active;
  if (N == 0) return;
  const int64_t cn = reserve(md, N, s);
  if (cn == 0) {
    run_grade_simt(md, N, true, rows, nullptr, ld, gamma, argmax, s);
    return;
  }
  const XPlan x = x_plan(m, md->ainv_s.p);
  const RowPlan rp(x, cn, N);
  const int64_t np = rp.np;
  const int n_col = x.pp / FN, n_best = rp.n_best;
  char* base = md->ws_grade.as<char>();
  uint16_t* sl = reinterpret_cast<uint16_t*>(base);
  int* E = reinterpret_cast<int*>(base + rp.sl);
  double* pbest = reinterpret_cast<double*>(base + rp.sl + rp.e);
  int32_t* parg = reinterpret_cast<int32_t*>(base + rp.sl + rp.e + rp.best);
  unsigned char* bad = reinterpret_cast<unsigned char*>(base + rp.sl + rp.e + rp.best + rp.arg);
  MTP_CUDA(cudaMemsetAsync(bad, 0, rp.bad, s));
  int nsm = 0;
  MTP_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, md->device));
  MTP_CUDA(cudaFuncSetAttribute(k_grade_fp64, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(FSMEM)));
  const CUtensorMap mB = slice_map(x.slices, static_cast<int64_t>(NS) * x.pp, x.kp, FN);
  const CUtensorMap mA = slice_map(sl, static_cast<int64_t>(NS) * np, x.kp, FM);
  ProfRegion pr("grade_fp64", s);
  for (int64_t r0 = 0; r0 < N; r0 += cn) {
    const int64_t n = std::min<int64_t>(cn, N - r0);
    k_slice_rows<<<nblk(n * 32, 256), 256, 0, s>>>(rows + r0 * ld, ld, m, n, x.g, x.xbad, x.kp, np, sl, E, bad + r0);
    ProfRegion::launched();
    // partials start as NaN: a tile that does not run (a bounded wait expired) leaves gamma NaN
    MTP_CUDA(cudaMemsetAsync(pbest, 0xFF, static_cast<size_t>(n_best) * n * sizeof(double), s));
    F64Args a{};
    a.N = n;
    a.np = np;
    a.m = static_cast<int>(m);
    a.pp = x.pp;
    a.n_col = n_col;
    a.k_chunks = x.kp / FK;
    a.n_work = (n + FM - 1) / FM * n_col;
    a.maxp = std::min<int>(NS, 4096 / static_cast<int>(std::min<int64_t>(SEG, m)));   // >= 5: at most 8 accumulators per sweep
    a.f = x.f;
    a.pbest = pbest;
    a.parg = parg;
    a.err = md->async_err.as<unsigned>();
    // host-side fault injection: a single try per wait makes the first unsatisfied wait expire
    a.wait_limit = take_injected(g_inject_grade_wait) ? 1u : WAIT_LIMIT;
    const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(a.n_work, nsm)));
    k_grade_fp64<<<grid, FTHREADS, FSMEM, s>>>(mA, mB, a);
    ProfRegion::launched();
    k_combine_fp64<<<nblk(n, 256), 256, 0, s>>>(n, n_best, pbest, parg, E, gamma + r0, argmax ? argmax + r0 : nullptr);
    ProfRegion::launched();
    k_check_fp64<<<nblk(n * 32, 256), 256, 0, s>>>(n, x.kp, sl, x.slices, parg, gamma + r0, bad + r0);
    ProfRegion::launched();
    MTP_CUDA(cudaGetLastError());
  }
  k_redo_rows<<<nblk(N, kRedoRows), 256, 0, s>>>(rows, ld, md->ainv_d.as<double>(), m, N, bad, gamma, argmax);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
}

}  // namespace mtp
