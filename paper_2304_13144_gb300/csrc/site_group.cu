// Contraction and its adjoint (eqs. 2, 5-6) for four neighborhoods at a time.
//
// A term of the schedule reads two values and adds their product to a sum, for every
// neighborhood alike, so the contraction is bound by shared-memory reads and by issuing and
// decoding the terms' words.  Here the values of four neighborhoods lie side by side (one float4
// per value), so a decoded word serves four terms, each operand is one 128-bit load and the
// arithmetic is two packed FP32 multiplies and two packed FMAs (fma.rn.f32x2: the rounding of
// the scalar instructions).  What bounds it is the shared-memory bandwidth: 6,012 load and 540
// store wavefronts per group at level 20, of which 4,392 are the operands without bank
// conflicts (the words are ordered for conflict-free quarter warps), in 8,850 cycles.
//
// W warps share a group: they split each dependency wave's rounds (the host balances them) and
// meet at a named barrier per wave.  At level 20 a group's values and adjoints take 36 KB, six
// groups per SM, so that one warp per group leaves 1.5 warps per scheduler (35 % issue); at
// level 24 one group takes 123 KB.  The schedule's words are read from tensor memory at level 20
// (70 KB), shared memory below, and at level 24 (0.35 MB) from L2 a step ahead.
//
// Per pass, before (k_contract, its default shape, words ordered for its 32-bit loads) and now: level
// 20, 1,048,576 atoms 15.3 -> 7.37 ms (tensor-memory shape of k_contract: 13.1); level 16, 128,000
// atoms 0.491 -> 0.215; level 24, 131,072 atoms 21.2 -> 5.72 ms.  With the words in this kernel's
// order k_contract's shapes take 1 to 8 % more (0.498 at level 16, 23.0 at level 24).
//
// The terms of a destination, their order and the two accumulator chains (row parity) are those
// of k_contract (site_split.cu), whose packed rounds this kernel walks: the results are bitwise
// the same.
#include "site_group.h"

#include <algorithm>
#include <type_traits>

#include "f32x2.h"
#include "profiler.h"

namespace mtp {
namespace {

constexpr int kNB = 4;            // neighborhoods per group (one float4 lane word)
constexpr int kTmemCols = 512;

struct GroupArgs {
  DevSchedule d;
  SiteOutputs o;
  const int* type;
  int64_t n_work, n_groups;
  float* mom;
  int ldm;
  const int* slot_comp;
  int NV;                 // value slots per group (the values and the always-zero slot)
  int ovf_row;            // tensor memory: first row kept in shared memory instead
  int n_rows;             // rows of the word stream (all warps' lists with their padding)
  size_t o_coef, o_round, o_ent, o_rows, o_vals;   // shared-memory layout (bytes)
  size_t group_bytes;
};

// where a warp reads the schedule's words
enum : int { SRC_GLOBAL = 0, SRC_SHARED = 1, SRC_TMEM = 2 };

template <int SRC>
struct Words {
  const uint32_t* rows;   // global / shared: row r at rows[32 r] (this lane's word)
  const uint32_t* ovf;    // tensor memory: row r >= ovf_row at ovf[32 (r - ovf_row)]
  uint32_t tq;            // tensor memory: address of column 0 in this warp's lane quarter
  int ovf_row;

  template <int U>
  __device__ __forceinline__ void load(int row, uint32_t (&w)[U]) const {
    if constexpr (SRC == SRC_TMEM) {
      if (row + U <= kTmemCols) {
#pragma unroll
        for (int u = 0; u < U; ++u)
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(w[u]) : "r"(tq + row + u) : "memory");
      } else {
        const uint32_t* p = ovf + 32 * (row - ovf_row);
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = p[32 * u];
      }
    } else {
      const uint32_t* p = rows + 32 * row;
#pragma unroll
      for (int u = 0; u < U; ++u) w[u] = SRC == SRC_GLOBAL ? __ldg(p + 32 * u) : p[32 * u];
    }
  }
  // before the words of the last load are used (names them, so that no use moves above it)
  template <int U>
  __device__ __forceinline__ void wait(uint32_t (&w)[U]) const {
    if constexpr (SRC == SRC_TMEM) {
      if constexpr (U == 4)
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3])::"memory");
      else if constexpr (U == 8)
        asm volatile("tcgen05.wait::ld.sync.aligned;"
                     : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3]), "+r"(w[4]), "+r"(w[5]), "+r"(w[6]), "+r"(w[7])::"memory");
      else static_assert(U == 4 || U == 8, "steps of 4 or 8 words");
    }
  }
};

// one word: a += c v[x] w[y] for the four neighborhoods
template <bool INL>
__device__ __forceinline__ void term(uint32_t wd, const float* coef, const char* v, const char* w, u64 (&a)[2]) {
  float c;
  uint32_t x, y;
  if constexpr (INL) {
    c = __uint_as_float(((wd >> 22) << 17) + 0x3F800000u);
    x = (wd & 2047u) << 4;
    y = ((wd >> 11) & 2047u) << 4;
  } else {
    c = coef[wd >> 24];
    x = (wd & 4095u) << 4;
    y = ((wd >> 12) & 4095u) << 4;
  }
  const ulonglong2 p = *reinterpret_cast<const ulonglong2*>(v + x);
  const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(w + y);
  const u64 cc = pack2(c, c);
  a[0] = fma2(cc, mul2(p.x, q.x), a[0]);
  a[1] = fma2(cc, mul2(p.y, q.y), a[1]);
}

template <bool INL, int PRE, int SRC, int W, int U, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) k_contract_group(GroupArgs P) {
  extern __shared__ __align__(16) unsigned char smem[];
  const DevSchedule& d = P.d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* coef = reinterpret_cast<float*>(smem + P.o_coef);
  if constexpr (!INL)
    for (int k = threadIdx.x; k < d.n_coef; k += blockDim.x) coef[k] = d.coef_f[k];
  int2* s_round = reinterpret_cast<int2*>(smem + P.o_round);
  uint16_t* s_ent = reinterpret_cast<uint16_t*>(smem + P.o_ent);
  for (int k = threadIdx.x; k < d.n_ground; k += blockDim.x) s_round[k] = d.ground[k];
  for (int k = threadIdx.x; k < 16 * d.n_ground; k += blockDim.x)   // 32 entries of 16 bits per round
    reinterpret_cast<uint32_t*>(s_ent)[k] = reinterpret_cast<const uint32_t*>(d.gent)[k];
  Words<SRC> words{};
  __shared__ uint32_t tmem_slot;
  uint32_t* s_rows = reinterpret_cast<uint32_t*>(smem + P.o_rows);
  if constexpr (SRC == SRC_GLOBAL) {
    words.rows = d.gslab + lane;
  } else if constexpr (SRC == SRC_SHARED) {
    for (int k = threadIdx.x; k < 32 * P.n_rows; k += blockDim.x) s_rows[k] = d.gslab[k];
    words.rows = s_rows + lane;
  } else {
    // rows [0, 512) in the block's tensor-memory columns, a copy in every lane quarter (a warp
    // reads the quarter of its index mod 4); the last of them and the rows past them also in
    // shared memory, so that a step's words come from one place
    const int nw = blockDim.x >> 5;
    if (warp == 0) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                       static_cast<unsigned>(__cvta_generic_to_shared(&tmem_slot))),
                   "r"(kTmemCols));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int q = warp & 3, TT = min(P.n_rows, kTmemCols);
    words.tq = tmem_slot + (static_cast<uint32_t>(32 * q) << 16);
    const int nq = (nw - q + 3) / 4;   // warps of this quarter
    for (int r = warp >> 2; r < TT; r += nq) {
      const uint32_t word = d.gslab[32 * r + lane];
      asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(words.tq + r), "r"(word) : "memory");
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    for (int k = threadIdx.x; k < 32 * (P.n_rows - P.ovf_row); k += blockDim.x) s_rows[k] = d.gslab[32 * P.ovf_row + k];
    words.ovf = s_rows + lane;
    words.ovf_row = P.ovf_row;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
  const int NV = P.NV;
  const int grp = warp / W, wig = warp - grp * W;   // the warp's group in the block, its place in the group
  float4* const v4 = reinterpret_cast<float4*>(smem + P.o_vals + grp * P.group_bytes);
  float4* const g4 = v4 + NV;
  const char* const vb = reinterpret_cast<const char*>(v4);
  const char* const gb = reinterpret_cast<const char*>(g4);
  const int tl = 32 * wig + lane;   // thread of the group
  for (int k = tl; k < 2 * NV; k += 32 * W) v4[k] = make_float4(0.f, 0.f, 0.f, 0.f);   // the zero slot stays 0
  auto group_sync = [&] {
    if constexpr (W == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "n"(32 * W) : "memory");
  };
  const int4 meta = d.gmeta[wig];   // first round, forward rounds, reverse rounds, first row
  const int T = d.n_types, n_mom = d.n_mom;
  int sc[PRE];
#pragma unroll
  for (int r = 0; r < PRE; ++r) {
    const int k = tl + 32 * W * r;
    sc[r] = k < n_mom ? P.slot_comp[k] : -1;
  }
  // the next group's moments, loaded a group ahead
  float pre[kNB][PRE];
  auto fetch = [&](int64_t w0) {
#pragma unroll
    for (int j = 0; j < kNB; ++j) {
      const bool live = w0 + j < P.n_work;
      const float* src = P.mom + (w0 + j) * P.ldm + tl;
#pragma unroll
      for (int r = 0; r < PRE; ++r) pre[j][r] = (live && sc[r] >= 0) ? __ldcs(src + 32 * W * r) : 0.f;
    }
  };
  const int gpb = static_cast<int>(blockDim.x) / (32 * W);   // groups per block
  int64_t gi = static_cast<int64_t>(blockIdx.x) * gpb + grp;
  const int64_t gstride = static_cast<int64_t>(gridDim.x) * gpb;
  if (gi < P.n_groups) fetch(gi * kNB);
  __syncthreads();
  // the word stream: the rows of this warp's rounds follow one another; `nxt` holds rows pos ..
  int pos = meta.w;
  uint32_t nxt[U];
  words.template load<U>(pos, nxt);
  words.template wait<U>(nxt);
  // one round: L rows into the lane's sums (chain = row parity), starting from `init`
  auto run_round = [&](int L, float init, const char* yb, float (&acc)[kNB]) {
    u64 a0[2] = {0ull, 0ull}, a1[2] = {0ull, 0ull};
    for (int it = 0; it < L; it += U) {
      uint32_t wd[U];
#pragma unroll
      for (int u = 0; u < U; ++u) wd[u] = nxt[u];
      const int used = min(U, L - it);
      pos += used;
      words.template load<U>(pos, nxt);
      if (used == U) {
#pragma unroll
        for (int u = 0; u < U; ++u) term<INL>(wd[u], coef, vb, yb, (u & 1) ? a1 : a0);
      } else {
#pragma unroll
        for (int u = 0; u < U - 1; ++u)
          if (u < used) term<INL>(wd[u], coef, vb, yb, (u & 1) ? a1 : a0);
      }
      words.template wait<U>(nxt);
    }
    const u64 i2 = pack2(init, init);
    unpack2(add2(i2, add2(a0[0], a1[0])), acc[0], acc[1]);
    unpack2(add2(i2, add2(a0[1], a1[1])), acc[2], acc[3]);
  };
  // lists split over aligned lane groups: `stages` butterfly steps, each lane by its group's size
  auto combine = [&](int stages, int lg, float (&acc)[kNB]) {
    for (int st = 0; st < stages; ++st) {
#pragma unroll
      for (int j = 0; j < kNB; ++j) {
        const float t = __shfl_xor_sync(0xffffffffu, acc[j], 1 << st);
        if (lg > st) acc[j] += t;
      }
    }
  };
  for (; gi < P.n_groups; gi += gstride) {
    const int64_t w0 = gi * kNB;
#pragma unroll
    for (int r = 0; r < PRE; ++r)
      if (sc[r] >= 0) v4[sc[r]] = make_float4(pre[0][r], pre[1][r], pre[2][r], pre[3][r]);
    if (gi + gstride < P.n_groups) fetch((gi + gstride) * kNB);
    group_sync();
    // ---------------- forward contraction (eqs. 5-6) ----------------
    const int2* rd_p = s_round + meta.x;
    const uint16_t* en_p = s_ent + 32 * meta.x + lane;
    int2 rd_n = rd_p[0];
    int en_n = en_p[0];
    for (int r = 0; r < meta.y; ++r) {
      const int2 rd = rd_n;
      const int ent = en_n;
      rd_n = rd_p[r + 1];   // (the reverse rounds follow)
      en_n = en_p[32 * (r + 1)];
      float acc[kNB];
      run_round(rd.x, 0.f, vb, acc);
      if (rd.y >> 1) combine(rd.y >> 1, (ent >> 12) & 7, acc);
      if (ent & 0x8000) v4[ent & 4095] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      if (rd.y & 1) group_sync();
    }
    // ---------------- site energy (eq. 2), FP32 sum, FP64 result ----------------
    if (P.o.V && wig == 0) {
      float e[kNB] = {0.f, 0.f, 0.f, 0.f};
      for (int a = lane; a < d.n_lin; a += 32) {
        const float xi = d.theta_f[T + a];
        const float4 b = v4[d.basis_idx[a]];
        e[0] = fmaf(xi, b.x, e[0]);
        e[1] = fmaf(xi, b.y, e[1]);
        e[2] = fmaf(xi, b.z, e[2]);
        e[3] = fmaf(xi, b.w, e[3]);
      }
#pragma unroll
      for (int j = 0; j < kNB; ++j)
        for (int m = 16; m; m >>= 1) e[j] += __shfl_xor_sync(0xffffffffu, e[j], m);
      const float ej = lane == 0 ? e[0] : (lane == 1 ? e[1] : (lane == 2 ? e[2] : e[3]));
      if (lane < kNB && w0 + lane < P.n_work)
        P.o.V[w0 + lane] = static_cast<double>(ej) + d.theta_d[P.type[w0 + lane]];
    }
    // ---------------- adjoint of the contraction (gather form), seeded with xi ----------------
    rd_p += meta.y;
    en_p += 32 * meta.y;
    const int nr = meta.z;
    int en_nn = nr > 1 ? en_p[32] : 0;
    float sd_n = (en_n & 0x8000) ? d.seed_f[en_n & 4095] : 0.f;
    for (int r = 0; r < nr; ++r) {
      const int2 rd = rd_n;
      const int ent = en_n;
      const float sd = sd_n;
      if (r + 1 < nr) rd_n = rd_p[r + 1];
      en_n = en_nn;
      sd_n = (r + 1 < nr && (en_n & 0x8000)) ? d.seed_f[en_n & 4095] : 0.f;
      if (r + 2 < nr) en_nn = en_p[32 * (r + 2)];
      float acc[kNB];
      run_round(rd.x, sd, gb, acc);
      if (rd.y >> 1) combine(rd.y >> 1, (ent >> 12) & 7, acc);
      if (ent & 0x8000) g4[ent & 4095] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      if (rd.y & 1) group_sync();
    }
    pos = meta.w;   // the stream repeats for the next group
    words.template load<U>(pos, nxt);
    words.template wait<U>(nxt);
    group_sync();
    // ---------------- outputs: dV/dM over the moments, the basis part of b_i ----------------
#pragma unroll
    for (int r = 0; r < PRE; ++r)
      if (sc[r] >= 0) {
        const float4 g = g4[sc[r]];
        const float gj[kNB] = {g.x, g.y, g.z, g.w};
#pragma unroll
        for (int j = 0; j < kNB; ++j)
          if (w0 + j < P.n_work) __stcs(P.mom + (w0 + j) * P.ldm + tl + 32 * W * r, gj[j]);
      }
    if (P.o.rows_hi) {
      int64_t ro[kNB];
      int zj[kNB];
#pragma unroll
      for (int j = 0; j < kNB; ++j) {
        const bool live = w0 + j < P.n_work;
        ro[j] = live ? (P.o.row_pos ? P.o.row_pos[w0 + j] : w0 + j) * P.o.rows_ld : -1;
        zj[j] = live ? P.type[w0 + j] : 0;
      }
      float* const hi = P.o.rows_hi;
      float* const lo = P.o.rows_lo;
      for (int k = tl; k < T + d.n_lin; k += 32 * W) {
        const float4 b = k < T ? make_float4(k == zj[0], k == zj[1], k == zj[2], k == zj[3]) : v4[d.basis_idx[k - T]];
        const float bj[kNB] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int j = 0; j < kNB; ++j) {
          if (ro[j] < 0) continue;
          if (lo) {
            const float h = tf32_rn(bj[j]);
            __stcs(hi + ro[j] + k, h);
            __stcs(lo + ro[j] + k, tf32_rn(bj[j] - h));
          } else {
            __stcs(hi + ro[j] + k, bj[j]);
          }
        }
      }
    }
    group_sync();
  }
  if constexpr (SRC == SRC_TMEM) {   // every warp is past its last tensor-memory read
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_slot), "r"(kTmemCols));
    }
  }
}

constexpr size_t kSmem = kMaxSmem - 16;
constexpr int kU = 4;   // words per step (the word stream has kGroupPad >= kU rows past its last round)
static_assert(kU <= kGroupPad, "a step reads up to kU rows past the last round");

size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

// groups per block by warps per group (threads and registers)
constexpr int group_max(int W) {
  return W == kGroupWarpsSmall ? 16 / kGroupWarpsSmall : (W == kGroupWarpsMid ? 6 : 1);
}

struct Plan {
  GroupArgs P;
  int src, groups;   // groups per block
  size_t smem;
};

// shared-memory layout for `src` with at most `max_groups` groups per block
bool make_plan(const DevSchedule& d, int src, int max_groups, Plan& pl) {
  GroupArgs& P = pl.P;
  P.d = d;
  P.NV = padded_nv(d.n_vals);
  P.n_rows = d.n_grows;
  P.group_bytes = static_cast<size_t>(2 * P.NV) * sizeof(float4);
  size_t at = 0;
  auto take = [&](size_t n) { const size_t o = at; at = align16(at + n); return o; };
  P.o_coef = take(d.coef_inline ? 0 : d.n_coef * sizeof(float));
  P.o_round = take(d.n_ground * sizeof(int2));
  P.o_ent = take(static_cast<size_t>(d.n_ground) * 32 * sizeof(uint16_t));
  P.ovf_row = std::max(0, std::min(P.n_rows, kTmemCols - kU + 1));
  P.o_rows = take(src == SRC_SHARED ? static_cast<size_t>(P.n_rows) * 128
                                    : (src == SRC_TMEM ? static_cast<size_t>(P.n_rows - P.ovf_row) * 128 : 0));
  P.o_vals = at;
  if (at + P.group_bytes > kSmem) return false;
  const int fit = static_cast<int>((kSmem - at) / P.group_bytes);
  pl.src = src;
  pl.groups = std::min(max_groups, fit);
  pl.smem = at + pl.groups * P.group_bytes;
  return true;
}

template <class K>
void launch(K kern, Plan& pl, int grid, cudaStream_t s) {
  // a block that holds the tensor-memory columns takes more than half the shared memory, so that
  // no second block shares its SM (it would wait for the columns)
  if (pl.src == SRC_TMEM) pl.smem = std::max<size_t>(pl.smem, 120 * 1024);
  allow_smem(kern, 16);   // (its tensor-memory address)
  ProfRegion pr("site_contract", s);
  kern<<<grid, pl.groups * pl.P.d.group_warps * 32, pl.smem, s>>>(pl.P);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
}

}  // namespace

bool contract_group_available(const DevSchedule& d) {
  Plan pl;
  const int comps = d.group_warps == kGroupWarpsSmall ? 160 : (d.group_warps == kGroupWarpsMid ? 320 : 608);
  if (d.n_mom > comps) return false;
  return d.gslab && d.n_vals < 4096 && make_plan(d, SRC_GLOBAL, 1, pl);
}

int run_contract_group(const DevSchedule& d, const SiteOutputs& o, const int* type, int64_t n_work, float* mom,
                       int ldm, const int* slot_comp, cudaStream_t s) {
  int dev = 0, nsm = 0;
  MTP_CUDA(cudaGetDevice(&dev));
  MTP_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  Plan pl{};
  const int64_t groups = (n_work + kNB - 1) / kNB;
  // groups per block: as many as shared memory holds (at most 16, 6 or 1 by the group's size)
  const int max_groups = group_max(d.group_warps);
  int src = SRC_GLOBAL;
  if (d.coef_inline) {
    // the words: read from global memory (L1, L2) where a group of warps carries its only
    // neighborhoods (staging them costs more than reading them once), else from shared memory
    // where they take at most 32 KB, else tensor memory
    make_plan(d, SRC_GLOBAL, max_groups, pl);
    if (groups > static_cast<int64_t>(nsm) * pl.groups) {
      if (static_cast<size_t>(d.n_grows) * 128 <= 32 * 1024) src = SRC_SHARED;
      else if (d.n_grows <= kTmemCols + 128) src = SRC_TMEM;
    }
  }
  if (!make_plan(d, src, max_groups, pl)) throw Fail{MTP_ERR_UNSUPPORTED, "contraction group does not fit shared memory"};
  // few groups: spread them over the SMs before filling a block
  const int64_t per_sm = std::max<int64_t>(1, (groups + nsm - 1) / nsm);
  if (per_sm < pl.groups) {
    pl.smem -= (pl.groups - per_sm) * pl.P.group_bytes;
    pl.groups = static_cast<int>(per_sm);
  }
  GroupArgs& P = pl.P;
  P.o = o;
  P.type = type;
  P.n_work = n_work;
  P.n_groups = groups;
  P.mom = mom;
  P.ldm = ldm;
  P.slot_comp = slot_comp;
  const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((groups + pl.groups - 1) / pl.groups, nsm)));
  auto pick = [&](auto w) {
    constexpr int W = decltype(w)::value;
    constexpr int PRE = (W == kGroupWarpsSmall ? 160 : (W == kGroupWarpsMid ? 320 : 608)) / (32 * W) +
                        ((W == kGroupWarpsSmall ? 160 : (W == kGroupWarpsMid ? 320 : 608)) % (32 * W) != 0);
    constexpr int MAXT = 32 * W * group_max(W);
    if (!d.coef_inline) launch(k_contract_group<false, PRE, SRC_GLOBAL, W, kU, MAXT>, pl, grid, s);
    else if (src == SRC_TMEM) launch(k_contract_group<true, PRE, SRC_TMEM, W, kU, MAXT>, pl, grid, s);
    else if (src == SRC_SHARED) launch(k_contract_group<true, PRE, SRC_SHARED, W, kU, MAXT>, pl, grid, s);
    else launch(k_contract_group<true, PRE, SRC_GLOBAL, W, kU, MAXT>, pl, grid, s);
  };
  if (d.group_warps == kGroupWarpsSmall) pick(std::integral_constant<int, kGroupWarpsSmall>{});
  else if (d.group_warps == kGroupWarpsMid) pick(std::integral_constant<int, kGroupWarpsMid>{});
  else pick(std::integral_constant<int, kGroupWarpsLarge>{});
  return src == SRC_TMEM ? 3 : (src == SRC_SHARED ? 1 : 2);
}

}  // namespace mtp
