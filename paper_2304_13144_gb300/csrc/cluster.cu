// Spherical cut of neighborhoods into non-periodic clusters (Section II.E, option (ii)).
//
// For a center atom c of configuration k: every atom j of k and periodic image n (periodic
// axes only) with |x_j + n H - x_c| < radius, the center itself first at the origin, then in
// ascending (j, n0, n1, n2).  Each center's atoms are split into `parts` contiguous ranges, one
// block per (center, range), so that few centers fill the GPU too; a block takes 256 consecutive
// atoms at a time, each thread walks its atom's images in order, and a block prefix sum places the
// hits in j order, so the output order is fixed.  Two passes (count, then fill at the scanned
// offsets of the ranges).
//
// What bounded it: FP64 (2 FMAs per clock and SM) spent on 125 images of every atom, by one warp
// per center.  An image can lie in the sphere only if its fractional coordinate relative to the
// center is within radius / face distance on every axis, so each axis gets its interval of images
// from an FP32 fractional coordinate with a margin, and only the images in all three intervals
// (of most atoms none) are tested in FP64.  (Where the margin would reach a quarter of a cell, an
// atom some 10^5 cells away, the FP64 coordinate's nearest image gives the interval.)  32 centers among 16,000 atoms, radius 8 A
// (one call for the sizes, one for the clusters: three passes): 677 -> 0.21 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include <cub/cub.cuh>

#include "mtp_internal.h"
#include "profiler.h"

namespace mtp {
namespace {

constexpr unsigned ERR_CENTER = 1u;
constexpr unsigned ERR_FILL = 2u;
constexpr int kMaxImages = 64;   // per axis and direction

struct CutArgs {
  const int64_t* atom_offset;
  int n_cfg;
  const double* pos;
  const int32_t* type;
  const double* cell;     // n_cfg x 9, rows = lattice vectors
  const uint8_t* pbc;     // n_cfg x 3
  const int64_t* centers;
  int64_t n;
  double radius;
  int parts;              // ranges per center
  long long* count;       // [n parts + 1]
  const long long* off;   // [n parts + 1] (fill pass)
  double* out_pos;
  int32_t* out_type;
  int64_t* out_src;
  unsigned* err;
};

__device__ int config_of(const CutArgs& A, int64_t atom) {
  int lo = 0, hi = A.n_cfg - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (A.atom_offset[mid] <= atom) lo = mid; else hi = mid - 1;
  }
  return lo;
}

constexpr int kCutThreads = 256;

template <bool FILL>
__global__ void __launch_bounds__(kCutThreads) k_cut(CutArgs A) {
  __shared__ int s_warp[kCutThreads / 32];
  __shared__ double s_G[9];
  __shared__ float s_reach[3];
  __shared__ int s_K[3], s_per[3];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t slot = blockIdx.x;   // (center, range)
  const int64_t q = slot / A.parts;
  const int part = static_cast<int>(slot - q * A.parts);
  const int64_t c = A.centers[q];
  const int64_t n_atoms = A.atom_offset[A.n_cfg];
  if (c < 0 || c >= n_atoms) {
    if (threadIdx.x == 0) { atomicOr(A.err, ERR_CENTER); if (!FILL) A.count[slot] = 0; }
    return;
  }
  const int k = config_of(A, c);
  const int64_t c0a = A.atom_offset[k], c1a = A.atom_offset[k + 1];
  const int64_t len = (c1a - c0a + A.parts - 1) / A.parts;
  const int64_t a0 = min(c1a, c0a + part * len), a1 = min(c1a, a0 + len);
  const double* H = A.cell + 9 * static_cast<int64_t>(k);
  // reciprocal vectors (fractional coordinate a = x . G_a) and the sphere's fractional half widths,
  // a lane of the first warp per entry (FP64 divisions by every thread took most of the pass)
  if (threadIdx.x < 9) {
    const int a = threadIdx.x / 3, d = threadIdx.x - 3 * a;
    auto cross = [&](int u, int v, int w) {   // component w of row u x row v
      const int y = w == 2 ? 0 : w + 1, z = w == 0 ? 2 : w - 1;
      return H[3 * u + y] * H[3 * v + z] - H[3 * u + z] * H[3 * v + y];
    };
    const double vol = H[0] * cross(1, 2, 0) + H[1] * cross(1, 2, 1) + H[2] * cross(1, 2, 2);
    const int u = a == 2 ? 0 : a + 1, v = a == 0 ? 2 : a - 1;
    s_G[threadIdx.x] = cross(u, v, d) / vol;
    if (d == 0) {
      const double cx = cross(u, v, 0), cy = cross(u, v, 1), cz = cross(u, v, 2);
      const double t = A.radius * sqrt(cx * cx + cy * cy + cz * cz) / fabs(vol);   // radius / face distance
      const bool per = A.pbc[3 * k + a] != 0;
      const double want = ceil(t) + 1.0;
      s_reach[a] = static_cast<float>(t);
      s_K[a] = per ? (want < kMaxImages ? static_cast<int>(want) : kMaxImages) : 0;
      s_per[a] = per ? (want < kMaxImages ? 1 : 2) : 0;   // 2: more images than kMaxImages
    }
  }
  __syncthreads();
  bool per[3];
  float reach[3], Gf[9];
  for (int a = 0; a < 3; ++a) { per[a] = s_per[a] != 0; reach[a] = s_reach[a]; }
  const bool capped = s_per[0] == 2 || s_per[1] == 2 || s_per[2] == 2;
  for (int d = 0; d < 9; ++d) Gf[d] = static_cast<float>(s_G[d]);
  const double xc[3] = {A.pos[3 * c], A.pos[3 * c + 1], A.pos[3 * c + 2]};
  const double rad = A.radius;
  long long base = FILL ? A.off[slot] : 0;
  const long long end = FILL ? A.off[slot + 1] : 0;
  if (part == 0) {   // the center first
    if (FILL && threadIdx.x == 0) {
      if (base < end) {
        A.out_pos[3 * base] = 0.0; A.out_pos[3 * base + 1] = 0.0; A.out_pos[3 * base + 2] = 0.0;
        A.out_type[base] = A.type[c];
        A.out_src[base] = c;
      } else {
        atomicOr(A.err, ERR_FILL);
      }
    }
    base += 1;
  }
  for (int64_t j0 = a0; j0 < a1; j0 += kCutThreads) {
    const int64_t j = j0 + threadIdx.x;
    const bool act = j < a1;
    double xj[3] = {0.0, 0.0, 0.0};
    int lo[3] = {0, 0, 0}, hi[3] = {-1, -1, -1};
    if (act) {
      float df[3];
      for (int d = 0; d < 3; ++d) {
        xj[d] = A.pos[3 * j + d];
        df[d] = static_cast<float>(xj[d] - xc[d]);
      }
      for (int a = 0; a < 3; ++a) {
        lo[a] = hi[a] = 0;
        if (!per[a]) continue;
        const float t0 = df[0] * Gf[3 * a], t1 = df[1] * Gf[3 * a + 1], t2 = df[2] * Gf[3 * a + 2];
        float f = t0 + t1 + t2;
        // its error: three rounded products and inputs, two sums (a few 2^-24 of the terms)
        const float eps = 1e-6f * (fabsf(t0) + fabsf(t1) + fabsf(t2) + reach[a] + 1.f);
        // -- images n with |f + n| <= reach
        const float l = ceilf(-f - reach[a] - eps), u = floorf(-f + reach[a] + eps);
        int n_lo, n_hi;
        if (capped || !(eps < 0.25f)) {
          // thin cells, whose images are cut off at kMaxImages around the nearest one; atoms so far
          // from their center that the margin would let in whole layers of images
          const double fd = (xj[0] - xc[0]) * s_G[3 * a] + (xj[1] - xc[1]) * s_G[3 * a + 1] + (xj[2] - xc[2]) * s_G[3 * a + 2];
          const int sn = static_cast<int>(rint(fd));
          n_lo = -s_K[a] - sn;
          n_hi = s_K[a] - sn;
        } else {
          n_lo = static_cast<int>(l);
          n_hi = static_cast<int>(u);
        }
        lo[a] = n_lo;
        hi[a] = n_hi;
      }
    }
    // pass over this thread's images in ascending (n0, n1, n2): count, or count and write
    auto visit = [&](auto emit) {
      int hits = 0;
      for (int n0 = lo[0]; n0 <= hi[0]; ++n0)
        for (int n1 = lo[1]; n1 <= hi[1]; ++n1)
          for (int n2 = lo[2]; n2 <= hi[2]; ++n2) {
            if (j == c && n0 == 0 && n1 == 0 && n2 == 0) continue;
            double r[3];
            for (int d = 0; d < 3; ++d) {
              const double sh = __dadd_rn(__dadd_rn(__dmul_rn(static_cast<double>(n0), H[d]),
                                                    __dmul_rn(static_cast<double>(n1), H[3 + d])),
                                          __dmul_rn(static_cast<double>(n2), H[6 + d]));
              r[d] = __dsub_rn(__dadd_rn(xj[d], sh), xc[d]);
            }
            const double rr = __dadd_rn(__dadd_rn(__dmul_rn(r[0], r[0]), __dmul_rn(r[1], r[1])), __dmul_rn(r[2], r[2]));
            if (__dsqrt_rn(rr) < rad) { emit(hits, r); ++hits; }
          }
      return hits;
    };
    const int mine = visit([](int, const double*) {});
    // block exclusive prefix of the threads' hits (threads hold ascending j)
    int incl = mine;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    __syncthreads();   // s_warp of the previous atoms has been read
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    int before = 0, round_total = 0;
    for (int w = 0; w < kCutThreads / 32; ++w) {
      const int t = s_warp[w];
      if (w < warp) before += t;
      round_total += t;
    }
    if (FILL && mine) {
      const long long at = base + before + incl - mine;
      visit([&](int h, const double* r) {
        const long long o = at + h;
        if (o < end) {
          A.out_pos[3 * o] = r[0]; A.out_pos[3 * o + 1] = r[1]; A.out_pos[3 * o + 2] = r[2];
          A.out_type[o] = A.type[j];
          A.out_src[o] = j;
        } else {
          atomicOr(A.err, ERR_FILL);
        }
      });
    }
    base += round_total;
  }
  if (threadIdx.x == 0) {
    if (!FILL) A.count[slot] = base;
    else if (base != end) atomicOr(A.err, ERR_FILL);
  }
}

// off[q] = offset of center q's first range (off[n] = the total)
__global__ void k_cut_offsets(const long long* part_off, int parts, int64_t n, long long* off) {
  const int64_t q = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (q <= n) off[q] = part_off[q * parts];
}

}  // namespace

int64_t run_cut_clusters(const mtp_batch* b, const int64_t* centers, int64_t n, double radius, int64_t* off,
                         double* pos, int32_t* type, int64_t* src, int64_t capacity, cudaStream_t s) {
  // ranges per center: about 2,048 blocks in all (13 per SM), at most 128 per center
  int parts = 1;
  while (parts < 128 && n * parts * 2 <= 2048) parts *= 2;
  const int64_t slots = n * parts;
  if (slots >= (int64_t(1) << 31)) throw Fail{MTP_ERR_UNSUPPORTED, "more than 2^31 centers"};
  size_t bytes = 0;
  long long* offl = reinterpret_cast<long long*>(off);
  MTP_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, bytes, offl, offl, static_cast<int>(slots + 1), s));
  ScopedBuf work(s);   // counts and offsets of the ranges, the error flag, the scan's scratch
  work.ensure(2 * (slots + 1) * sizeof(long long) + 512 + bytes, s);
  long long* cnt = work.as<long long>();
  long long* part_off = cnt + slots + 1;
  unsigned* err = reinterpret_cast<unsigned*>(part_off + slots + 1);
  void* scan_tmp = reinterpret_cast<char*>(work.p) + ((2 * (slots + 1) * sizeof(long long) + 16 + 255) & ~size_t(255));
  MTP_CUDA(cudaMemsetAsync(err, 0, sizeof(unsigned), s));
  MTP_CUDA(cudaMemsetAsync(cnt + slots, 0, sizeof(long long), s));
  CutArgs A{};
  A.atom_offset = b->atom_offset;
  A.n_cfg = b->n_cfg;
  A.pos = b->pos;
  A.type = b->type;
  A.cell = b->cell;
  A.pbc = b->pbc;
  A.centers = centers;
  A.n = n;
  A.parts = parts;
  A.radius = radius;
  A.count = cnt;
  A.err = err;
  ProfRegion pr("cut_clusters", s);
  if (n > 0) {
    k_cut<false><<<static_cast<unsigned>(slots), kCutThreads, 0, s>>>(A);
    ProfRegion::launched();
    MTP_CUDA(cudaGetLastError());
  }
  // offsets of the ranges: exclusive scan of the counts; the centers' are every parts-th
  MTP_CUDA(cub::DeviceScan::ExclusiveSum(scan_tmp, bytes, cnt, part_off, static_cast<int>(slots + 1), s));
  k_cut_offsets<<<static_cast<unsigned>(n / 256 + 1), 256, 0, s>>>(part_off, parts, n, offl);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
  long long total = 0;
  unsigned flag = 0;
  MTP_CUDA(cudaMemcpyAsync(&total, offl + n, sizeof(long long), cudaMemcpyDeviceToHost, s));
  MTP_CUDA(cudaMemcpyAsync(&flag, err, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  MTP_CUDA(cudaStreamSynchronize(s));
  if (flag & ERR_CENTER) throw Fail{MTP_ERR_ARG, "center atom index out of range"};
  if (!pos || !type || !src || total > capacity) return total;
  if (n == 0) return total;
  A.off = part_off;
  A.out_pos = pos;
  A.out_type = type;
  A.out_src = src;
  k_cut<true><<<static_cast<unsigned>(slots), kCutThreads, 0, s>>>(A);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
  MTP_CUDA(cudaMemcpyAsync(&flag, err, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  MTP_CUDA(cudaStreamSynchronize(s));
  if (flag) throw Fail{MTP_ERR_NUMERIC, "cluster cut: count and fill passes disagree"};
  return total;
}

}  // namespace mtp
