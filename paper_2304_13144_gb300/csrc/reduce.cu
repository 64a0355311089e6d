// Forces, per-configuration sums, flag compaction, neighborhood extraction and the loss
// reductions of the training step.
//
// Forces (F = -dE/dx, used by eq. 7): with G_p = dV_i/dr_ij for pair p = (i -> j, n) and
// rev(p) = (j -> i, -n),  F_i = sum_{p in nbh(i)} (G_p - G_rev(p)); a deterministic gather in
// FP64 (no atomics).  Energies (eq. 1) and virials are summed per configuration over fixed
// atom segments, then per configuration over its segments, in a fixed order.
#include <cub/cub.cuh>
#include <thrust/iterator/counting_iterator.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "mtp_internal.h"
#include "profiler.h"

namespace mtp {
namespace {

int nblk(int64_t n, int t) { return static_cast<int>(std::max<int64_t>(1, (n + t - 1) / t)); }

// FP64 gradients: one thread per atom, pairs in list order
__global__ void k_forces(DevNbr nb, const double* G, double* F) {
  int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= nb.n_atoms) return;
  double f0 = 0, f1 = 0, f2 = 0;
  for (int64_t p = nb.off[i]; p < nb.off[i + 1]; ++p) {
    const int64_t q = nb.prev[p];
    f0 += G[3 * p + 0] - G[3 * q + 0];
    f1 += G[3 * p + 1] - G[3 * q + 1];
    f2 += G[3 * p + 2] - G[3 * q + 2];
  }
  F[3 * i + 0] = f0;
  F[3 * i + 1] = f1;
  F[3 * i + 2] = f2;
}

// FP32 gradients, LPA lanes per atom: each component summed as an unevaluated pair hi + lo of
// floats with error-free additions (TwoSum), as accurate as an FP64 accumulation on the FP32
// pipes (FP64 throughput is a small fraction of FP32 on this GPU); lane k of an atom's group
// takes pairs k, k + LPA, ..., and the group combines its partial pairs in a fixed tree
template <int LPA>
__global__ void k_forces_grp(DevNbr nb, const float* G, double* F) {
  const int64_t gid = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) / LPA;
  const int k = threadIdx.x & (LPA - 1);
  const bool act = gid < nb.n_atoms;
  const int64_t i = act ? gid : 0;
  float h[3] = {0.f, 0.f, 0.f}, l[3] = {0.f, 0.f, 0.f};
  auto two = [](float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  };
  if (act) {
    const int64_t p1 = nb.off[i + 1];
    for (int64_t p = nb.off[i] + k; p < p1; p += LPA) {
      const int64_t q = nb.prev[p];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float s, e;
        two(h[c], G[3 * p + c], s, e);
        h[c] = s; l[c] = __fadd_rn(l[c], e);
        two(h[c], -G[3 * q + c], s, e);
        h[c] = s; l[c] = __fadd_rn(l[c], e);
      }
    }
  }
#pragma unroll
  for (int m = LPA / 2; m; m >>= 1)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float oh = __shfl_xor_sync(0xffffffffu, h[c], m), ol = __shfl_xor_sync(0xffffffffu, l[c], m);
      // the lower lane of each pair adds the upper one's, so both get the same sum
      float s, e;
      if (k & m) two(oh, h[c], s, e); else two(h[c], oh, s, e);
      h[c] = s;
      l[c] = __fadd_rn(__fadd_rn((k & m) ? ol : l[c], (k & m) ? l[c] : ol), e);
    }
  if (act && k < 3) {
    const float hv = k == 0 ? h[0] : (k == 1 ? h[1] : h[2]);
    const float lv = k == 0 ? l[0] : (k == 1 ? l[1] : l[2]);
    F[3 * i + k] = static_cast<double>(hv) + static_cast<double>(lv);
  }
}

// one block per segment (cfg, a0, a1): partial[seg][0] = sum V, [1..9] = sum W.  With PER = 1 a block
// takes one of the ten sums (blockIdx.y): few segments would leave 10 x 4096 FP64 additions to one SM
// each (its FP64 pipe does 2 per clock; 16,384 atoms 25.7 -> 7.4 us); many segments share the loads
// instead (PER = 10).  The order of every sum is the same.  Both sums' kernels, PER 1 against 10, us: 4
// full segments 14.3, 32.7; 32 18.4, 42.1; 123 36.4, 45.0; 256 59.4, 54.8; small configurations, 16
// segments 13.4, 16.6; 64 16.4, 17.5; 128 20.4, 19.5; 512 35.2, 20.8.
template <int PER>
__global__ void k_seg_sums(const int64_t* seg, const double* V, const double* Wat, double* part) {
  const int64_t s = blockIdx.x;
  const int k0 = PER == 1 ? blockIdx.y : 0;
  const int64_t a0 = seg[3 * s + 1], a1 = seg[3 * s + 2];
  __shared__ double red[PER][256];
  double acc[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) acc[k] = 0.0;
  for (int64_t a = a0 + threadIdx.x; a < a1; a += blockDim.x) {
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      if (k0 + k == 0) {
        if (V) acc[k] += V[a];
      } else if (Wat) {
        acc[k] += Wat[9 * a + (k0 + k - 1)];
      }
    }
  }
#pragma unroll
  for (int k = 0; k < PER; ++k) red[k][threadIdx.x] = acc[k];
  __syncthreads();
  for (int w = blockDim.x / 2; w; w >>= 1) {
    if (threadIdx.x < w)
#pragma unroll
      for (int k = 0; k < PER; ++k) red[k][threadIdx.x] += red[k][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x < PER) part[10 * s + k0 + threadIdx.x] = red[threadIdx.x][0];
}

void launch_seg_sums(const mtp_nbr* nb, const double* V, const double* Wat, double* part, cudaStream_t s) {
  const unsigned n = static_cast<unsigned>(nb->n_seg);
  if (n <= 64) k_seg_sums<1><<<dim3(n, 10), 256, 0, s>>>(nb->seg.as<int64_t>(), V, Wat, part);
  else k_seg_sums<10><<<n, 256, 0, s>>>(nb->seg.as<int64_t>(), V, Wat, part);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
}

__global__ void k_cfg_sums(const int64_t* seg, int64_t n_seg, const double* part, int n_cfg, double* E, double* W) {
  // warp per config; the config's segments (contiguous in seg) are taken by lane s mod 32 in
  // order, then summed over the lanes in a fixed shuffle tree
  const int lane = threadIdx.x & 31;
  const int k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (k >= n_cfg) return;   // whole warps
  int64_t lo = 0, hi = n_seg;   // first segment of config k
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (seg[3 * mid] < k) lo = mid + 1; else hi = mid;
  }
  double acc[10];
  for (int q = 0; q < 10; ++q) acc[q] = 0.0;
  for (int64_t s = lo + lane; s < n_seg && seg[3 * s] == k; s += 32)
    for (int q = 0; q < 10; ++q) acc[q] += part[10 * s + q];
  for (int m = 16; m; m >>= 1)
    for (int q = 0; q < 10; ++q) {
      const double o = __shfl_xor_sync(0xffffffffu, acc[q], m);
      acc[q] = (lane & m) ? o + acc[q] : acc[q] + o;   // both lanes of a pair form the same sum
    }
  if (lane == 0) {
    if (E) E[k] = acc[0];
    if (W)
      for (int q = 0; q < 9; ++q) W[9 * k + q] = acc[1 + q];
  }
}

struct AboveThreshold {
  const double* gamma;
  double thr;
  __device__ bool operator()(int i) const { return gamma[i] > thr; }
};

__global__ void k_extract_counts(DevNbr nb, const int32_t* idx, int64_t n, long long* cnt, unsigned* bad) {
  int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (k > n) return;
  if (k == n) { cnt[k] = 0; return; }
  const int i = idx[k];
  if (i < 0 || i >= nb.n_atoms) { atomicOr(bad, 1u); cnt[k] = 0; return; }
  cnt[k] = nb.off[i + 1] - nb.off[i];
}

// a warp per atom, a lane per pair: 2,000 atoms' pairs by one thread per atom were a serial chain
// of dependent loads
__global__ void k_extract_fill(DevNbr nb, const double* pos, const int* type, const double* cell,
                               const int32_t* idx, int64_t n, const long long* off, double* r, int32_t* ty,
                               int32_t* jout) {
  const int64_t k = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
  if (k >= n) return;
  const int i = idx[k];
  if (i < 0 || i >= nb.n_atoms) return;
  const double* H = cell + 9 * nb.atom_cfg[i];
  const int64_t p0 = nb.off[i], np = nb.off[i + 1] - p0;
  for (int64_t t = threadIdx.x & 31; t < np; t += 32) {
    const int64_t o = off[k] + t;
    const int j = nb.pj[p0 + t];
    const int img = nb.pimg[p0 + t];
    const int n0 = unpack_img(img, 0), n1 = unpack_img(img, 1), n2 = unpack_img(img, 2);
    if (r)
      for (int c = 0; c < 3; ++c) {
        const double sh = n0 * H[c] + n1 * H[3 + c] + n2 * H[6 + c];
        r[3 * o + c] = (pos[3 * j + c] + sh) - pos[3 * i + c];
      }
    if (ty) ty[o] = type[j];
    if (jout) jout[o] = j;
  }
}

// U_i = 2 w_f (F_i - F*_i); per-block partial of sum |F - F*|^2
__global__ void k_train_forces(int64_t n, const double* F, const double* Fref, double w_f, double* U, double* part) {
  __shared__ double red[256];
  double acc = 0.0;
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    for (int c = 0; c < 3; ++c) {
      const double d = F[3 * i + c] - Fref[3 * i + c];
      U[3 * i + c] = 2.0 * w_f * d;
      acc += d * d;
    }
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int w = blockDim.x / 2; w; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

__global__ void k_train_cfg(int n_cfg, const double* E, const double* Eref, const double* W, const double* Wref,
                            double w_e, double w_f, double w_s, const double* fpart, int n_fpart, double* coef,
                            double* S, double* loss) {
  __shared__ double red[256];
  double acc = 0.0;
  for (int k = threadIdx.x; k < n_cfg; k += blockDim.x) {
    const double dE = E[k] - Eref[k];
    coef[k] = 2.0 * w_e * dE;
    acc += w_e * dE * dE;
    for (int q = 0; q < 9; ++q) {
      const double dW = (w_s != 0.0 && Wref) ? W[9 * k + q] - Wref[9 * k + q] : 0.0;
      S[9 * k + q] = 2.0 * w_s * dW;
      acc += w_s * dW * dW;
    }
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int w = blockDim.x / 2; w; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    double f = 0.0;
    for (int b = 0; b < n_fpart; ++b) f += fpart[b];
    loss[0] = red[0] + w_f * f;
  }
}

// column sums of part[nrows x m] in a fixed order: a block takes 32 columns, its 32 warps every
// 32nd row each (several loads in flight), then the warps' sums are added in order.  One thread per
// column walked the rows one load after the other (2,432 rows of 383: 0.27 ms).
__global__ void __launch_bounds__(1024) k_sum_rows(const double* __restrict__ part, int nrows, int64_t m, double* out) {
  __shared__ double red[32][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t c = blockIdx.x * 32LL + lane;
  double acc = 0.0;
  if (c < m) {
    const double* p = part + c;
    int r = w;
    for (; r + 7 * 32 < nrows; r += 8 * 32) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = p[static_cast<int64_t>(r + 32 * u) * m];
#pragma unroll
      for (int u = 0; u < 8; ++u) acc += v[u];
    }
    for (; r < nrows; r += 32) acc += p[static_cast<int64_t>(r) * m];
  }
  red[w][lane] = acc;
  __syncthreads();
  if (w == 0 && c < m) {
    for (int k = 1; k < 32; ++k) acc += red[k][lane];
    out[c] = acc;
  }
}

}  // namespace

void run_forces(const mtp_nbr* nb, bool fp64, const void* G, double* F, cudaStream_t s) {
  ProfRegion pr("force_gather", s);
  if (fp64) {
    k_forces<<<nblk(nb->n_atoms, 256), 256, 0, s>>>(nb->dn, static_cast<const double*>(G), F);
    ProfRegion::launched();
  } else {
    k_forces_grp<8><<<nblk(nb->n_atoms * 8, 256), 256, 0, s>>>(nb->dn, static_cast<const float*>(G), F);
    ProfRegion::launched();
  }
  MTP_CUDA(cudaGetLastError());
}

void load_efs_sums() {
  cudaFuncAttributes a;
  MTP_CUDA(cudaFuncGetAttributes(&a, k_forces));
  MTP_CUDA(cudaFuncGetAttributes(&a, k_forces_grp<8>));
  MTP_CUDA(cudaFuncGetAttributes(&a, k_seg_sums<1>));
  MTP_CUDA(cudaFuncGetAttributes(&a, k_seg_sums<10>));
  MTP_CUDA(cudaFuncGetAttributes(&a, k_cfg_sums));
}

size_t config_sums_scratch(const mtp_nbr* nb) { return nb->n_seg * 10 * sizeof(double); }

void run_config_sums(const mtp_nbr* nb, const double* V, const double* Wat, double* E, double* W, DevBuf& tmp,
                     cudaStream_t s) {
  tmp.ensure(config_sums_scratch(nb), s);
  ProfRegion pr("config_sums", s);
  launch_seg_sums(nb, V, Wat, tmp.as<double>(), s);
  k_cfg_sums<<<nblk(nb->n_cfg * 32, 128), 128, 0, s>>>(nb->seg.as<int64_t>(), nb->n_seg, tmp.as<double>(),
                                                 static_cast<int>(nb->n_cfg), E, W);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
}

void run_config_sums_into(const mtp_nbr* nb, const double* V, const double* Wat, double* E, double* W, double* part,
                          cudaStream_t s) {
  ProfRegion pr("config_sums", s);
  launch_seg_sums(nb, V, Wat, part, s);
  k_cfg_sums<<<nblk(nb->n_cfg * 32, 128), 128, 0, s>>>(nb->seg.as<int64_t>(), nb->n_seg, part, static_cast<int>(nb->n_cfg),
                                                 E, W);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
}

namespace {
constexpr int kSortAtoms = 2048, kSortThreads = 256, kMaxTypes = 64;   // atoms per block, species (mtp_load's limit)

__device__ __forceinline__ int clamp_type(int z, int T) { return min(max(z, 0), T - 1); }

// hist[z n_blk + block] = atoms of species z among the block's
__global__ void __launch_bounds__(kSortThreads) k_type_hist(const int32_t* type, int64_t N, int T, int n_blk, int* hist) {
  __shared__ int h[kMaxTypes];
  for (int z = threadIdx.x; z < T; z += kSortThreads) h[z] = 0;
  __syncthreads();
  const int64_t a0 = blockIdx.x * static_cast<int64_t>(kSortAtoms), a1 = min(N, a0 + kSortAtoms);
  for (int64_t a = a0 + threadIdx.x; a < a1; a += kSortThreads) atomicAdd(&h[clamp_type(type[a], T)], 1);
  __syncthreads();
  for (int z = threadIdx.x; z < T; z += kSortThreads) hist[z * n_blk + blockIdx.x] = h[z];
}

// exclusive sums in place, by one block
__global__ void __launch_bounds__(1024, 1) k_type_scan(int* hist, int n) {
  __shared__ int warp_sum[32];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int per = (n + 1023) / 1024, b0 = min(n, tid * per), b1 = min(n, b0 + per);
  int mine = 0;
  for (int k = b0; k < b1; ++k) mine += hist[k];
  int incl = mine;
  for (int m = 1; m < 32; m <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, m);
    if (lane >= m) incl += v;
  }
  if (lane == 31) warp_sum[w] = incl;
  __syncthreads();
  int at = incl - mine;
  for (int k = 0; k < w; ++k) at += warp_sum[k];
  for (int k = b0; k < b1; ++k) {
    const int v = hist[k];
    hist[k] = at;
    at += v;
  }
}

__global__ void __launch_bounds__(kSortThreads) k_type_place(const int32_t* type, int64_t N, int T, int n_blk, const int* first,
                                                             int32_t* zrow, int64_t* order, int64_t* rank) {
  constexpr int NW = kSortThreads / 32;
  __shared__ int base[kMaxTypes], cnt[NW][kMaxTypes];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int z = threadIdx.x; z < T; z += kSortThreads) base[z] = first[z * n_blk + blockIdx.x];
  const int64_t a0 = blockIdx.x * static_cast<int64_t>(kSortAtoms), a1 = min(N, a0 + kSortAtoms);
  for (int64_t r = a0; r < a1; r += kSortThreads) {
    const int64_t a = r + threadIdx.x;
    const int t = a < a1 ? type[a] : 0, z = a < a1 ? clamp_type(t, T) : kMaxTypes;
    for (int e = threadIdx.x; e < NW * kMaxTypes; e += kSortThreads) cnt[e / kMaxTypes][e % kMaxTypes] = 0;
    __syncthreads();
    const unsigned same = __match_any_sync(0xffffffffu, z);
    const int before = __popc(same & ((1u << lane) - 1u));
    if (z < kMaxTypes && before == 0) cnt[w][z] = __popc(same);
    __syncthreads();
    if (z < kMaxTypes) {
      int at = base[z] + before;
      for (int u = 0; u < w; ++u) at += cnt[u][z];
      order[at] = a;
      zrow[at] = t;
      rank[a] = at;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < T; e += kSortThreads)
      for (int u = 0; u < NW; ++u) base[e] += cnt[u][e];
    __syncthreads();
  }
}
}  // namespace

void run_species_order(const int32_t* type, int64_t N, int n_types, int32_t* zrow, int64_t* order, DevBuf& tmp,
                       cudaStream_t s) {
  // a stable counting sort of the atom indices by species (ties keep index order); the library radix
  // sort took 34 us for 4,000 atoms and more on the host, this 19 (1,048,576 atoms: 50, 24)
  ProfRegion pr("grade_row_order", s);
  const int n_blk = nblk(N, kSortAtoms);
  tmp.ensure(static_cast<size_t>(n_types) * n_blk * sizeof(int), s);
  int* hist = tmp.as<int>();
  k_type_hist<<<n_blk, kSortThreads, 0, s>>>(type, N, n_types, n_blk, hist);
  ProfRegion::launched();
  k_type_scan<<<1, 1024, 0, s>>>(hist, n_types * n_blk);
  ProfRegion::launched();
  k_type_place<<<n_blk, kSortThreads, 0, s>>>(type, N, n_types, n_blk, hist, zrow, order, order + N);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
}

size_t flag_scratch(int64_t N) {
  size_t bytes = 0;
  thrust::counting_iterator<int> it(0);
  MTP_CUDA(cub::DeviceSelect::If(nullptr, bytes, it, static_cast<int32_t*>(nullptr), static_cast<int64_t*>(nullptr),
                                 static_cast<int>(N), AboveThreshold{nullptr, 0.0}));
  return bytes;
}

void run_flag(int64_t N, const double* gamma, double threshold, int32_t* flagged, int64_t* n_flagged, DevBuf& tmp,
              cudaStream_t s) {
  AboveThreshold pred{gamma, threshold};
  ProfRegion pr("flag_compact", s);
  thrust::counting_iterator<int> it(0);
  size_t bytes = 0;
  MTP_CUDA(cub::DeviceSelect::If(nullptr, bytes, it, flagged, n_flagged, static_cast<int>(N), pred, s));
  tmp.ensure(bytes, s);
  MTP_CUDA(cub::DeviceSelect::If(tmp.p, bytes, it, flagged, n_flagged, static_cast<int>(N), pred, s));
}

int64_t run_extract(const mtp_nbr* nb, const mtp_batch* b, const int32_t* idx, int64_t n, int64_t* off, double* r,
                    int32_t* type, int32_t* j, int64_t capacity, cudaStream_t s) {
  size_t bytes = 0;
  long long* offl = reinterpret_cast<long long*>(off);
  MTP_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, bytes, offl, offl, n + 1, s));
  ScopedBuf work(s);   // counts, the error flag, the scan's scratch
  const size_t at = ((n + 1) * sizeof(long long) + 16 + 255) & ~size_t(255);
  work.ensure(at + bytes, s);
  long long* cnt = work.as<long long>();
  unsigned* bad = reinterpret_cast<unsigned*>(cnt + n + 1);
  MTP_CUDA(cudaMemsetAsync(bad, 0, sizeof(unsigned), s));
  k_extract_counts<<<nblk(n + 1, 256), 256, 0, s>>>(nb->dn, idx, n, cnt, bad);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
  MTP_CUDA(cub::DeviceScan::ExclusiveSum(reinterpret_cast<char*>(work.p) + at, bytes, cnt, offl, n + 1, s));
  long long total = 0;
  unsigned badh = 0;
  MTP_CUDA(cudaMemcpyAsync(&total, offl + n, sizeof(long long), cudaMemcpyDeviceToHost, s));
  MTP_CUDA(cudaMemcpyAsync(&badh, bad, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  MTP_CUDA(cudaStreamSynchronize(s));
  if (badh) throw Fail{MTP_ERR_ARG, "atom index out of range"};
  if (total > capacity) return total;
  if (n > 0) {
    k_extract_fill<<<nblk(n * 32, 128), 128, 0, s>>>(nb->dn, b->pos, b->type, b->cell, idx, n, offl, r, type, j);
    ProfRegion::launched();
    MTP_CUDA(cudaGetLastError());
  }
  return total;
}

namespace {
constexpr int kResidualBlocks = 256;
}
size_t train_prep_scratch() { return kResidualBlocks * sizeof(double); }

void run_train_prep(const mtp_nbr* nb, int n_cfg, const double* E, const double* F, const double* W,
                    const double* E_ref, const double* F_ref, const double* W_ref, double w_e, double w_f,
                    double w_s, double* coef, double* U, double* Scfg, double* loss, DevBuf& tmp, cudaStream_t s) {
  const int nb_f = kResidualBlocks;
  tmp.ensure(train_prep_scratch(), s);
  ProfRegion pr("train_residuals", s);
  k_train_forces<<<nb_f, 256, 0, s>>>(nb->n_atoms, F, F_ref, w_f, U, tmp.as<double>());
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
  k_train_cfg<<<1, 256, 0, s>>>(n_cfg, E, E_ref, W, W_ref, w_e, w_f, w_s, tmp.as<double>(), nb_f, coef, Scfg, loss);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
}

void run_sum_rows(const double* part, int nrows, int64_t m, double* out, cudaStream_t s) {
  ProfRegion pr("train_grad_sum", s);
  k_sum_rows<<<nblk(m, 32), 1024, 0, s>>>(part, nrows, m, out);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
}

}  // namespace mtp
