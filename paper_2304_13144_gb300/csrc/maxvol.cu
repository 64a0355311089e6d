// MaxVol update of the active set (Section II.D, D-optimality), FP64 on the GPU.
//
// The active set is the m x m matrix A of maximal |det A|.  For candidate rows B (n x m),
// C = B A^-1; replacing active row j by candidate row i multiplies |det A| by |C_ij|.  While the
// largest |C_ij| exceeds 1 + eps the swap is made and C and A^-1 follow by rank-one corrections
// (Sherman-Morrison):
//   u = (C_i. - e_j) / C_ij,   C <- C - C_.j u,   A^-1 <- A^-1 - (A^-1)_.j u,   A_j. <- B_i.
// (row i of C becomes e_j, so a candidate enters at most once; the row swapped out is dropped).
// The swaps run inside one persistent kernel (a block per SM at most, two grid barriers per swap):
// the rank-one update of C finds the next largest entry in the same pass over C.  Five launches and
// a read-back per swap took 46 us; now 10.7 us (level 16, 2,000 candidates, m = 222), bound by the
// barriers.
// At the end A^-1 is formed afresh from the final A by LU, which also refreshes the split copies
// used by the mixed-precision grade.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "mtp_internal.h"
#include "profiler.h"

namespace mtp {

void run_lu_inverse(mtp_model* md, const double* A, int64_t m, cudaStream_t s);

namespace {

constexpr int GT = 32;   // GEMM tile (rows, columns and k)
constexpr int GR = 8;    // thread rows per tile (each thread computes GT / GR outputs)

// C[n x m] = B[n x m] X[m x m] (row-major, FP64)
__global__ void __launch_bounds__(GT * GR) k_gemm(const double* __restrict__ B, const double* __restrict__ X,
                                                  double* __restrict__ C, int64_t n, int m) {
  __shared__ double sB[GT][GT + 1];
  __shared__ double sX[GT][GT + 1];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int col = blockIdx.x * GT + tx;
  const int64_t row_tiles = (n + GT - 1) / GT;
  for (int64_t rt = blockIdx.y; rt < row_tiles; rt += gridDim.y) {
    const int64_t row0 = rt * GT;
    double acc[GT / GR];
#pragma unroll
    for (int q = 0; q < GT / GR; ++q) acc[q] = 0.0;
    for (int k0 = 0; k0 < m; k0 += GT) {
      for (int r = ty; r < GT; r += GR) {
        const int64_t gr = row0 + r;
        const int gk = k0 + tx;
        sB[r][tx] = (gr < n && gk < m) ? B[gr * m + gk] : 0.0;
        const int xr = k0 + r;
        sX[r][tx] = (xr < m && col < m) ? X[static_cast<int64_t>(xr) * m + col] : 0.0;
      }
      __syncthreads();
#pragma unroll 8
      for (int k = 0; k < GT; ++k) {
        const double x = sX[k][tx];
#pragma unroll
        for (int q = 0; q < GT / GR; ++q) acc[q] = fma(sB[ty + GR * q][k], x, acc[q]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < GT / GR; ++q) {
      const int64_t gr = row0 + ty + GR * q;
      if (gr < n && col < m) C[gr * m + col] = acc[q];
    }
  }
}

struct Best {
  long long key;   // abs_key of the value
  long long idx;   // flat row-major index
};

__device__ __forceinline__ Best better(Best a, Best b) {
  return (b.key > a.key || (b.key == a.key && b.idx < a.idx)) ? b : a;
}

constexpr Best kNone{-2, 0x7fffffffffffffffLL};

__device__ Best block_best(Best b) {
  __shared__ Best sh[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  warp_best(b.key, b.idx);
  if (lane == 0) sh[w] = b;
  __syncthreads();
  b = lane < static_cast<int>(blockDim.x >> 5) ? sh[lane] : kNone;
  warp_best(b.key, b.idx);   // every warp: all threads get the block's
  __syncthreads();
  return b;
}

struct SwapState {
  long long swaps;          // made so far
  int stop;                 // no entry above 1 + eps
  unsigned arrived;         // grid barrier: arrivals of this launch
  unsigned timeout;         // a barrier gave up
};

struct SwapArgs {
  double* C;
  double* Ainv;
  const double* B;
  double* A;
  int64_t n;
  int m;
  double limit;         // 1 + eps
  long long max_swaps;  // in all
  long long last;       // this launch returns at the latest after this many swaps in all
  double *u, *v, *w;
  Best* part;           // [gridDim.x]
  long long* source;    // [m]
  SwapState* st;
};

// all blocks of a cooperative launch (arrivals count up from the launch's zero; release and acquire
// at the counter order the blocks' writes); bounded: after about a second it gives up.  ABSENT (fault
// injection): it waits, for a millisecond, for one block more than there are.  (A template: limits in
// the arguments cost each barrier 0.04 us.)
template <bool ABSENT>
__device__ bool grid_barrier(SwapState* st, unsigned& round) {
  constexpr int kTries = ABSENT ? 1000 : 4000000;
  __shared__ int s_ok;
  __syncthreads();
  ++round;
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned target = round * gridDim.x + (ABSENT ? 1u : 0u);
    unsigned seen;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&st->arrived) : "memory");
    for (int tries = 0;; ++tries) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&st->arrived) : "memory");
      if (seen >= target) break;
      if (tries > kTries) {
        atomicExch(&st->timeout, 1u);
        ok = 0;
        break;
      }
      if (tries > 1000) __nanosleep(100);
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Values written by other blocks are read through L2 (__ldcg); each entry of C and A^-1 is updated
// by one thread throughout.
template <bool ABSENT>
__global__ void __launch_bounds__(1024, 1) k_swaps(SwapArgs P) {
  const int64_t tid = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  const int64_t nt = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int m = P.m;
  const long long total = P.n * static_cast<long long>(m), total_a = static_cast<long long>(m) * m;
  const int64_t r0 = tid / m, dr = nt / m;   // this thread's first row and column, and its steps
  const int c0 = static_cast<int>(tid - r0 * m), dc = static_cast<int>(nt - dr * m);
  unsigned round = 0;
  long long swaps = *reinterpret_cast<volatile long long*>(&P.st->swaps);
  auto publish = [&](Best b) {
    b = block_best(b);
    if (threadIdx.x == 0) { __stcg(&P.part[blockIdx.x].key, b.key); __stcg(&P.part[blockIdx.x].idx, b.idx); }
  };
  {
    Best b = kNone;
    for (long long t = tid; t < total; t += nt) {
      const long long k = abs_key(__ldcg(P.C + t));
      if (k > b.key) b = Best{k, t};   // ascending per thread: keeps the lowest index
    }
    publish(b);
  }
  if (!grid_barrier<ABSENT>(P.st, round)) return;
  while (true) {
    Best b = kNone;
    for (int k = threadIdx.x; k < static_cast<int>(gridDim.x); k += blockDim.x)
      b = better(b, Best{__ldcg(&P.part[k].key), __ldcg(&P.part[k].idx)});
    b = block_best(b);
    const bool stop = b.key < 0 || !(__longlong_as_double(b.key) > P.limit);
    if (stop || swaps >= P.max_swaps || swaps >= P.last) {
      if (tid == 0) { P.st->swaps = swaps; P.st->stop = stop ? 1 : 0; }
      return;
    }
    const int64_t i = b.idx / m;
    const int j = static_cast<int>(b.idx - i * m);
    // u = (C_i. - e_j) / C_ij, v = C_.j, w = (A^-1)_.j, A_j. = B_i., spread thinly over the blocks
    // (an FP64 division per entry)
    const int64_t s_tid = threadIdx.x * static_cast<int64_t>(gridDim.x) + blockIdx.x;
    for (int64_t t = s_tid; t < max(P.n, static_cast<int64_t>(m)); t += nt) {
      if (t < m) {
        const double cij = __ldcg(P.C + i * m + j);
        __stcg(P.u + t, (__ldcg(P.C + i * m + t) - (t == j ? 1.0 : 0.0)) / cij);
        __stcg(P.w + t, __ldcg(P.Ainv + t * m + j));
        P.A[static_cast<int64_t>(j) * m + t] = P.B[i * m + t];
      }
      if (t < P.n) __stcg(P.v + t, __ldcg(P.C + t * m + j));
    }
    if (tid == 0) P.source[j] = i;
    if (!grid_barrier<ABSENT>(P.st, round)) return;
    // C -= v u (and the largest entry of the result), A^-1 -= w u
    Best nb = kNone;
    int64_t r = r0;
    int c = c0;
    for (long long t = tid; t < total; t += nt) {
      const double u = __ldcg(P.u + c);
      const double x = fma(-__ldcg(P.v + r), u, __ldcg(P.C + t));
      __stcg(P.C + t, x);
      const long long k = abs_key(x);
      if (k > nb.key) nb = Best{k, t};
      if (t < total_a) __stcg(P.Ainv + t, fma(-__ldcg(P.w + r), u, __ldcg(P.Ainv + t)));
      r += dr;
      c += dc;
      if (c >= m) { c -= m; ++r; }
    }
    for (long long t = tid + (total > tid ? (total - tid + nt - 1) / nt * nt : 0); t < total_a; t += nt) {
      const long long ra = t / m;   // (fewer candidates than parameters)
      const int ca = static_cast<int>(t - ra * m);
      __stcg(P.Ainv + t, fma(-__ldcg(P.w + ra), __ldcg(P.u + ca), __ldcg(P.Ainv + t)));
    }
    publish(nb);
    ++swaps;
    if (!grid_barrier<ABSENT>(P.st, round)) return;
  }
}

}  // namespace

int64_t run_maxvol(mtp_model* md, const double* B, int64_t n, double eps, int64_t max_swaps, int64_t* source,
                   cudaStream_t s) {
  const int64_t m = md->m_active;
  int64_t swaps = 0;
  ScopedBuf work(s);
  const size_t cbytes = static_cast<size_t>(n) * m * sizeof(double);
  int dev = 0, nsm = 0;
  MTP_CUDA(cudaGetDevice(&dev));
  MTP_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  with_memory(md, s, [&] {
    work.ensure(cbytes + (n + 3 * m) * sizeof(double) + nsm * sizeof(Best) + sizeof(SwapState) + 256, s);
  });
  long long* src = work.as<long long>();
  double* C = reinterpret_cast<double*>(src + m);
  double* v = C + n * m;
  double* u = v + n;
  double* w = u + m;
  Best* part = reinterpret_cast<Best*>(w + m);
  SwapState* st = reinterpret_cast<SwapState*>(part + nsm);
  MTP_CUDA(cudaMemsetAsync(src, 0xff, m * sizeof(long long), s));   // -1: kept
  if (n > 0) {
    ProfRegion pr("active_set_maxvol", s);
    {
      const dim3 blk(GT, GR);
      const dim3 grd(static_cast<unsigned>((m + GT - 1) / GT),
                     static_cast<unsigned>(std::min<int64_t>((n + GT - 1) / GT, 65535)));
      k_gemm<<<grd, blk, 0, s>>>(B, md->ainv_d.as<double>(), C, n, static_cast<int>(m));
      ProfRegion::launched();
      MTP_CUDA(cudaGetLastError());
    }
    MTP_CUDA(cudaMemsetAsync(st, 0, sizeof(SwapState), s));
    SwapArgs P{C, md->ainv_d.as<double>(), B, md->a_d.as<double>(), n, static_cast<int>(m), 1.0 + eps, max_swaps, 0,
               u, v, w, part, src, st};
    auto kern = take_injected(g_inject_maxvol_wait) ? k_swaps<true> : k_swaps<false>;
    // the swaps change A and A^-1 in place: until the inverse of the final A is there the model has
    // no active set, whichever way this call ends
    md->have_ainv = false;
    const int64_t want = (std::max<int64_t>(n * m, m * m) + 1023) / 1024;
    const unsigned grid = static_cast<unsigned>(std::max<int64_t>(1, std::min<int64_t>(want, nsm)));
    while (swaps < max_swaps) {
      MTP_CUDA(cudaMemsetAsync(&st->arrived, 0, sizeof(unsigned), s));
      P.last = swaps + 4096;   // swaps of one launch: about 45 ms at 2,000 x 222 entries
      void* args[] = {&P};
      MTP_CUDA(cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kern), dim3(grid), dim3(1024), args, 0, s));
      ProfRegion::launched();
      SwapState h{};
      MTP_CUDA(cudaMemcpyAsync(&h, st, sizeof(h), cudaMemcpyDeviceToHost, s));
      MTP_CUDA(cudaStreamSynchronize(s));
      if (h.timeout) throw Fail{MTP_ERR_TIMEOUT, "a bounded wait of the MaxVol update expired; the model has no active set now"};
      swaps = h.swaps;
      if (h.stop) break;
    }
  }
  if (source) MTP_CUDA(cudaMemcpyAsync(source, src, m * sizeof(int64_t), cudaMemcpyDeviceToDevice, s));
  if (swaps > 0) {
    with_memory(md, s, [&] { run_lu_inverse(md, md->a_d.as<double>(), m, s); });
  } else {
    MTP_CUDA(cudaStreamSynchronize(s));
    md->have_ainv = true;   // nothing was changed
  }
  return swaps;
}

}  // namespace mtp
