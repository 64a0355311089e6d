// Active-set inverse (FP64 LU with partial pivoting) and the SIMT grade product.
//
// Sections II.C-D: the grade of neighborhood i is gamma_i = max_p |(b_i A^-1)_p| for the
// active-set matrix A (rows = parameter rows of the active neighborhoods).  A^-1 is formed
// once per active set: LU with partial pivoting, P A = L U, then A^-1 = U^-1 L^-1 P.
//   The factorisation goes by panels of kPanel columns, three launches each: the panel itself by
// one block with its rows in registers (pivot search, scaling, rank-one updates of the panel);
// the row exchanges and the triangular solve with the panel's unit lower block, a thread per
// column; and the rank-kPanel update of the rows below.  L is not kept: the same exchanges,
// solves and updates applied to the columns left of the panel carry L^-1 there (below the
// diagonal, in the place of L), so that the forward substitution of A^-1 costs no launch of its
// own.  Back substitution goes by kBack rows, two launches each, with the diagonal blocks of U inverted
// beforehand (all at once).
//   What bounded it: three launches per column (1,955 at m = 651) and a thread per column of the
// inverse walking m^2 dependent steps.  Now the panels (1.3 of 3.2 ms: a pivot chain of about 2 us
// per column, and FP64 at 2 FMAs per clock in the one SM; pivots are compared as integers, FP64
// comparisons alone took twice that) and 174 dependent launches.  A^-1 at m = 651: 44.2 -> 3.14 ms,
// m = 222: 6.3 -> 0.86, m = 1,636: 271 -> 18.3.
// The grade product C = B A^-1 is fused with its row epilogue (max |C_ip| and the lowest p
// attaining it), so C is never written.  This SIMT kernel serves small active sets; the mixed path
// uses the tensor-core kernel in grade_tc.cu, the FP64 path the one in grade_fp64.cu.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "mtp_internal.h"
#include "profiler.h"

namespace mtp {
namespace {

// max |A| as the bits of a non-negative double (their order is that of the integers)
__global__ void k_maxabs(const double* A, int64_t n, unsigned long long* out) {
  double v = 0.0;
  for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < n;
       k += static_cast<int64_t>(gridDim.x) * blockDim.x)
    v = fmax(v, fabs(A[k]));
  for (int o = 16; o; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, static_cast<unsigned long long>(__double_as_longlong(v)));
}

constexpr int kPanel = 16;   // columns per panel (m = 651: 8 columns 3.31 ms, 16 3.24)
constexpr int kBack = 32;    // rows per step of the back substitution
constexpr int kPanelRows = 2048;   // rows a panel's block holds in registers

// what one panel's exchanges do to the other columns: row to[e] takes the old row from[e]; the
// first kPanel entries are the panel's own rows
struct PanelMoves {
  int to[2 * kPanel], from[2 * kPanel];
  int n;
};

__global__ void k_lu_init(int* perm, int64_t m) {
  const int64_t r = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (r < m) perm[r] = static_cast<int>(r);
}

// Factorises columns k0 .. k0 + nb - 1 of the rows k0 .. m - 1: each thread holds R rows of the
// panel in registers and their current positions (exchanges move positions, not data).  Writes the
// panel's U and unit L blocks to M, the multipliers of the rows below to Lp[position][kPanel], the
// exchanges to *mv and to perm (position -> row of A); a pivot below 1e-13 max|A| sets *flag.
template <int R, int NT>
__global__ void __launch_bounds__(NT, 1) k_panel(double* M, int64_t m, int k0, int nb, double* Lp, PanelMoves* mv,
                                                            int* perm, const unsigned long long* maxabs, unsigned* flag) {
  constexpr int NW = NT / 32;
  __shared__ long long s_v[2][NW];
  __shared__ int s_p[2][NW];
  __shared__ double s_row[2][kPanel];
  __shared__ double s_inv[2];
  __shared__ int s_src[kPanel];   // row (position before the panel) of the panel's j-th pivot
  __shared__ int s_from[kPanel];  // the position it was taken from
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  double a[R][kPanel];
  int pos[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int64_t r = k0 + tid + static_cast<int64_t>(q) * NT;
    pos[q] = r < m ? static_cast<int>(r) : -1;
#pragma unroll
    for (int c = 0; c < kPanel; ++c) a[q][c] = (r < m && c < nb) ? M[r * m + k0 + c] : 0.0;
  }
  const double tiny = 1e-13 * __longlong_as_double(static_cast<long long>(*maxabs));
#pragma unroll
  for (int j = 0; j < kPanel; ++j) {
    if (j >= nb) break;
    const int k = k0 + j, ph = j & 1;
    // largest |a_j| of the rows not taken yet, the lowest position on ties
    long long best = -2, at = 0x7fffffff;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const long long v = abs_key(a[q][j]);
      if (pos[q] >= k && (v > best || (v == best && pos[q] < at))) { best = v; at = pos[q]; }
    }
    warp_best(best, at);
    if (lane == 0) { s_v[ph][w] = best; s_p[ph][w] = static_cast<int>(at); }
    __syncthreads();
    best = lane < NW ? s_v[ph][lane] : -2;
    at = lane < NW ? s_p[ph][lane] : 0x7fffffff;
    warp_best(best, at);
    const int bp = best < 0 ? k : static_cast<int>(at);   // no comparable entry (NaN): the diagonal
#pragma unroll
    for (int q = 0; q < R; ++q)
      if (pos[q] == bp) {
        const double d = a[q][j];
        s_inv[ph] = d != 0.0 ? 1.0 / d : 0.0;
#pragma unroll
        for (int c = 0; c < kPanel; ++c) s_row[ph][c] = a[q][c];
        s_src[j] = k0 + tid + q * NT;
        s_from[j] = bp;
        if (!(fabs(d) > tiny)) atomicOr(flag, 1u);
      }
    __syncthreads();
    const double inv = s_inv[ph];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      // the pivot's row goes to position k, the row there to the pivot's old position
      if (pos[q] == bp) pos[q] = k;
      else if (pos[q] == k) pos[q] = bp;
      if (pos[q] > k) {
        const double l = a[q][j] * inv;
        a[q][j] = l;
#pragma unroll
        for (int c = j + 1; c < kPanel; ++c) a[q][c] = fma(-l, s_row[ph][c], a[q][c]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < R; ++q) {
    if (pos[q] < 0) continue;
    const int64_t p = pos[q];
    if (p < k0 + nb) {
#pragma unroll
      for (int c = 0; c < kPanel; ++c)
        if (c < nb) M[p * m + k0 + c] = a[q][c];
    } else {
#pragma unroll
      for (int c = 0; c < kPanel; ++c) Lp[p * kPanel + c] = c < nb ? a[q][c] : 0.0;
    }
  }
  // rows that moved: the panel's positions first, then displaced rows that ended below the panel
  if (tid < nb) { mv->to[tid] = k0 + tid; mv->from[tid] = s_src[tid]; }
  __shared__ int s_n;
  if (tid == 0) s_n = nb;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const int r = k0 + tid + q * NT;
    if (pos[q] >= k0 + nb && pos[q] != r) {   // a row displaced from the panel's positions (or twice)
      const int e = atomicAdd(&s_n, 1);
      mv->to[e] = pos[q];
      mv->from[e] = r;
    }
  }
  if (tid == 0)
    for (int j = 0; j < nb; ++j) {   // perm follows the exchanges in order
      const int t = perm[k0 + j];
      perm[k0 + j] = perm[s_from[j]];
      perm[s_from[j]] = t;
    }
  __syncthreads();
  if (tid == 0) mv->n = s_n;
}

// The panel's exchanges in the other columns and the solve with its unit lower block, a thread per
// column: M[panel rows][c] = L11^-1 (P M)[panel rows][c]; for the panel's own columns L11^-1 itself
// goes to Tp (the other blocks still read the panel's block of M).
__global__ void __launch_bounds__(128) k_swap_solve(double* M, int64_t m, int k0, int nb, const PanelMoves* mv, double* Tp) {
  __shared__ double L[kPanel][kPanel + 1];
  __shared__ PanelMoves s;
  for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
    const int r = e / nb, c = e - r * nb;
    L[r][c] = M[static_cast<int64_t>(k0 + r) * m + k0 + c];
  }
  for (int e = threadIdx.x; e < mv->n; e += blockDim.x) { s.to[e] = mv->to[e]; s.from[e] = mv->from[e]; }
  if (threadIdx.x == 0) s.n = mv->n;
  __syncthreads();
  const int64_t c = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  const int64_t n_out = m - nb;   // columns outside the panel, then the panel's nb
  if (c >= n_out + nb) return;
  const bool own = c >= n_out;
  const int64_t col = own ? k0 + (c - n_out) : (c < k0 ? c : c + nb);
  double x[2 * kPanel];
#pragma unroll
  for (int e = 0; e < 2 * kPanel; ++e) x[e] = 0.0;
  if (own) {
#pragma unroll
    for (int j = 0; j < kPanel; ++j) x[j] = j == static_cast<int>(c - n_out) ? 1.0 : 0.0;
  } else {
#pragma unroll
    for (int e = 0; e < 2 * kPanel; ++e)
      if (e < s.n) x[e] = M[static_cast<int64_t>(s.from[e]) * m + col];
#pragma unroll
    for (int e = 0; e < 2 * kPanel; ++e)
      if (e >= nb && e < s.n) M[static_cast<int64_t>(s.to[e]) * m + col] = x[e];
  }
#pragma unroll
  for (int j = 0; j < kPanel; ++j) {
    if (j >= nb) break;
#pragma unroll
    for (int i = j + 1; i < kPanel; ++i)
      if (i < nb) x[i] = fma(-L[i][j], x[j], x[i]);
  }
#pragma unroll
  for (int j = 0; j < kPanel; ++j) {
    if (j >= nb) break;
    if (own) {
      Tp[j * kPanel + (c - n_out)] = x[j];
    } else {
      M[static_cast<int64_t>(k0 + j) * m + col] = x[j];
    }
  }
}

// M[r][c] -= sum_k Lp[r][k] T[k][c] for the rows below the panel, T = M[panel rows][c] or, for the
// panel's own columns (which start from zero), Tp; and L11^-1 into M's panel block, strictly below
// the diagonal.  32 x 32 tiles, 2 x 2 outputs per thread.
__global__ void __launch_bounds__(256) k_panel_update(double* M, int64_t m, int k0, int nb, const double* Lp, const double* Tp) {
  __shared__ double sL[32][kPanel + 1];
  __shared__ double sT[kPanel][32];
  const int64_t r0 = k0 + nb + blockIdx.y * 32LL, c0 = blockIdx.x * 32LL;
  if (blockIdx.x == 0 && blockIdx.y == 0)
    for (int e = threadIdx.x; e < nb * nb; e += 256) {
      const int j = e / nb, i = e - j * nb;
      if (j > i) M[static_cast<int64_t>(k0 + j) * m + k0 + i] = Tp[j * kPanel + i];
    }
  for (int e = threadIdx.x; e < 32 * kPanel; e += 256) {
    const int r = e / kPanel, k = e % kPanel;
    sL[r][k] = r0 + r < m ? Lp[(r0 + r) * kPanel + k] : 0.0;
    const int kk = e / 32, c = e % 32;
    const int64_t gc = c0 + c;
    const bool own = gc >= k0 && gc < k0 + nb;
    sT[kk][c] = (kk < nb && gc < m) ? (own ? Tp[kk * kPanel + (gc - k0)] : M[static_cast<int64_t>(k0 + kk) * m + gc]) : 0.0;
  }
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
  for (int k = 0; k < kPanel; ++k) {
    const double l0 = sL[ty][k], l1 = sL[ty + 16][k], t0 = sT[k][tx], t1 = sT[k][tx + 16];
    acc[0][0] = fma(l0, t0, acc[0][0]);
    acc[0][1] = fma(l0, t1, acc[0][1]);
    acc[1][0] = fma(l1, t0, acc[1][0]);
    acc[1][1] = fma(l1, t1, acc[1][1]);
  }
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int64_t r = r0 + ty + 16 * a, c = c0 + tx + 16 * b;
      if (r >= m || c >= m) continue;
      const bool own = c >= k0 && c < k0 + nb;
      M[r * m + c] = (own ? 0.0 : M[r * m + c]) - acc[a][b];
    }
}

// Inverses of U's diagonal blocks of kBack rows (zero-padded), a block each, a thread per column
__global__ void __launch_bounds__(kBack) k_diag_inverse(const double* M, int64_t m, double* D) {
  __shared__ double U[kBack][kBack + 1], inv[kBack];
  const int i0 = blockIdx.x * kBack, nb = static_cast<int>(min(static_cast<int64_t>(kBack), m - i0));
  const int c = threadIdx.x;
  for (int r = 0; r < kBack; ++r)
    U[r][c] = (r < nb && c < nb) ? M[static_cast<int64_t>(i0 + r) * m + i0 + c] : (r == c ? 1.0 : 0.0);
  __syncwarp();
  inv[c] = 1.0 / U[c][c];
  __syncwarp();
  double x[kBack];
#pragma unroll
  for (int r = 0; r < kBack; ++r) x[r] = r == c ? 1.0 : 0.0;
#pragma unroll
  for (int k = kBack - 1; k >= 0; --k) {
    x[k] *= inv[k];
#pragma unroll
    for (int r = 0; r < k; ++r) x[r] = fma(-U[r][k], x[k], x[r]);
  }
  double* out = D + static_cast<int64_t>(blockIdx.x) * kBack * kBack;
#pragma unroll
  for (int r = 0; r < kBack; ++r) out[r * kBack + c] = x[r];
}

// One step of the back substitution U X = L^-1: rows i0 .. i0 + nb - 1 of W (the right-hand sides)
// become X = (diagonal block)^-1 W.  32 columns per block, 4 outputs per thread.
__global__ void __launch_bounds__(256) k_back_solve(const double* D, int64_t m, int i0, int nb, double* W) {
  __shared__ double sD[kBack][kBack + 1], sW[kBack][32];
  const int64_t c0 = blockIdx.x * 32LL;
  const double* d = D + static_cast<int64_t>(i0 / kBack) * kBack * kBack;
  for (int e = threadIdx.x; e < kBack * kBack; e += 256) {
    const int r = e / kBack, c = e % kBack;
    sD[r][c] = d[e];
    sW[r][c] = (r < nb && c0 + c < m) ? W[static_cast<int64_t>(i0 + r) * m + c0 + c] : 0.0;
  }
  __syncthreads();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // rows ty, ty + 8, ..
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int k = 0; k < kBack; ++k) {
    const double x = sW[k][tx];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (k >= 8 * q) acc[q] = fma(sD[ty + 8 * q][k], x, acc[q]);   // (zero below the diagonal)
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int r = ty + 8 * q;
    if (r < nb && c0 + tx < m) W[static_cast<int64_t>(i0 + r) * m + c0 + tx] = acc[q];
  }
}
static_assert(kBack == 32, "k_back_solve: 32 x 32 blocks, 8 rows of threads");

// W[r][c] -= sum_k M[r][i0 + k] W[i0 + k][c] for r < i0
__global__ void __launch_bounds__(256) k_back_update(const double* M, int64_t m, int i0, int nb, double* W) {
  __shared__ double sU[32][kBack + 1];
  __shared__ double sX[kBack][32];
  const int64_t r0 = blockIdx.y * 32LL, c0 = blockIdx.x * 32LL;
  for (int e = threadIdx.x; e < 32 * kBack; e += 256) {
    const int r = e / kBack, k = e % kBack;
    sU[r][k] = (r0 + r < i0 && k < nb) ? M[(r0 + r) * m + i0 + k] : 0.0;
    sX[r][k] = (r < nb && c0 + k < m) ? W[static_cast<int64_t>(i0 + r) * m + c0 + k] : 0.0;
  }
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
  for (int k = 0; k < kBack; ++k) {
    const double l0 = sU[ty][k], l1 = sU[ty + 16][k], t0 = sX[k][tx], t1 = sX[k][tx + 16];
    acc[0][0] = fma(l0, t0, acc[0][0]);
    acc[0][1] = fma(l0, t1, acc[0][1]);
    acc[1][0] = fma(l1, t0, acc[1][0]);
    acc[1][1] = fma(l1, t1, acc[1][1]);
  }
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int64_t r = r0 + ty + 16 * a, c = c0 + tx + 16 * b;
      if (r < i0 && c < m) W[r * m + c] -= acc[a][b];
    }
}

// W = L^-1 (unit lower triangular, from below M's diagonal)
__global__ void k_lower(const double* M, int64_t m, double* W) {
  const int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (e >= m * m) return;
  const int64_t r = e / m, c = e - r * m;
  W[e] = c < r ? M[e] : (c == r ? 1.0 : 0.0);
}

// A^-1[:, perm[p]] = X[:, p]
__global__ void k_unpermute(const double* X, const int* perm, int64_t m, double* out) {
  const int64_t e = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (e >= m * m) return;
  const int64_t r = e / m, p = e - r * m;
  out[r * m + perm[p]] = X[e];
}

// --- column by column, for matrices whose panel does not fit one block's registers ---

// pivot search in column k, row swap, singularity flag
__global__ void k_pivot(double* LU, int64_t m, int64_t k, int* piv, const unsigned long long* maxabs, unsigned* flag) {
  __shared__ double bv[1024];
  __shared__ int64_t bi[1024];
  double best = -1.0;
  int64_t bidx = k;
  for (int64_t r = k + threadIdx.x; r < m; r += blockDim.x) {
    const double v = fabs(LU[r * m + k]);
    if (v > best) { best = v; bidx = r; }
  }
  bv[threadIdx.x] = best;
  bi[threadIdx.x] = bidx;
  __syncthreads();
  for (int w = blockDim.x / 2; w; w >>= 1) {
    if (threadIdx.x < w) {
      const double o = bv[threadIdx.x + w];
      const int64_t oi = bi[threadIdx.x + w];
      if (o > bv[threadIdx.x] || (o == bv[threadIdx.x] && oi < bi[threadIdx.x])) { bv[threadIdx.x] = o; bi[threadIdx.x] = oi; }
    }
    __syncthreads();
  }
  const int64_t p = bi[0];
  if (threadIdx.x == 0) {
    piv[k] = static_cast<int>(p);
    if (!(bv[0] > 1e-13 * __longlong_as_double(static_cast<long long>(maxabs[0])))) atomicOr(flag, 1u);
  }
  if (p != k)
    for (int64_t c = threadIdx.x; c < m; c += blockDim.x) {
      const double t = LU[k * m + c];
      LU[k * m + c] = LU[p * m + c];
      LU[p * m + c] = t;
    }
}

__global__ void k_lcol(double* LU, int64_t m, int64_t k) {
  const int64_t r = k + 1 + blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (r >= m) return;
  const double d = LU[k * m + k];
  LU[r * m + k] = d != 0.0 ? LU[r * m + k] / d : 0.0;
}

__global__ void k_trail(double* LU, int64_t m, int64_t k) {
  const int64_t c = k + 1 + blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  const int64_t r = k + 1 + blockIdx.y;
  if (c >= m || r >= m) return;
  LU[r * m + c] -= LU[r * m + k] * LU[k * m + c];
}

// column c of A^-1: solve L U x = P e_c
__global__ void k_inverse_cols(const double* LU, const int* piv, int64_t m, double* X) {
  const int64_t c = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (c >= m) return;
  // y = P e_c : apply the row swaps in order to the unit vector
  int64_t pos = c;  // position of the 1 after the swaps
  for (int64_t k = 0; k < m; ++k) {
    const int64_t p = piv[k];
    if (pos == k) pos = p;
    else if (pos == p) pos = k;
  }
  for (int64_t r = 0; r < m; ++r) {
    double v = (r == pos) ? 1.0 : 0.0;
    for (int64_t k = 0; k < r; ++k) v -= LU[r * m + k] * X[k * m + c];
    X[r * m + c] = v;
  }
  for (int64_t r = m - 1; r >= 0; --r) {
    double v = X[r * m + c];
    for (int64_t k = r + 1; k < m; ++k) v -= LU[r * m + k] * X[k * m + c];
    X[r * m + c] = v / LU[r * m + r];
  }
}

// Split A^-1 into TF32 pieces hi + lo (each rounded to nearest TF32), transposed to K-major
// [n][k] and zero-padded to ld x ld: the B operand of the tensor-core grade.
__global__ void k_split_ainv(const double* X, int64_t m, int64_t ld, float* hi, float* lo) {
  const int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (idx >= ld * ld) return;
  const int64_t n = idx / ld, k = idx % ld;   // output row n (= column of A^-1), col k
  const double v = (n < m && k < m) ? X[k * m + n] : 0.0;
  const float h = tf32_rn(static_cast<float>(v));
  hi[idx] = h;
  lo[idx] = tf32_rn(static_cast<float>(v - static_cast<double>(h)));
}

// Grade product with fused row epilogue.  Block: 256 threads, 64 rows; column tiles of 64;
// K steps of 16; each thread owns a 4 x 4 micro-tile.
template <class T>
__global__ void __launch_bounds__(256) k_grade_simt(const T* B, int64_t ldb, const T* X, int64_t m, int64_t N,
                                                     double* gamma, int32_t* argmax) {
  __shared__ T sB[16][64 + 1];
  __shared__ T sX[16][64 + 1];
  __shared__ double rowmax[64];
  __shared__ int rowarg[64];
  __shared__ double tmax[16][64];
  __shared__ int targ[16][64];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int64_t row0 = static_cast<int64_t>(blockIdx.x) * 64;
  if (threadIdx.x < 64) { rowmax[threadIdx.x] = -1.0; rowarg[threadIdx.x] = 0; }
  for (int64_t col0 = 0; col0 < m; col0 += 64) {
    T acc[4][4];
    for (int a = 0; a < 4; ++a)
      for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
    for (int64_t k0 = 0; k0 < m; k0 += 16) {
      for (int e = threadIdx.x; e < 16 * 64; e += 256) {
        const int kk = e / 64, rr = e % 64;
        const int64_t gr = row0 + rr, gk = k0 + kk;
        sB[kk][rr] = (gr < N && gk < m) ? B[gr * ldb + gk] : T(0);
        const int64_t gc = col0 + rr;
        sX[kk][rr] = (gk < m && gc < m) ? X[gk * m + gc] : T(0);
      }
      __syncthreads();
      for (int kk = 0; kk < 16; ++kk) {
        T bv[4], xv[4];
        for (int a = 0; a < 4; ++a) bv[a] = sB[kk][ty * 4 + a];
        for (int b = 0; b < 4; ++b) xv[b] = sX[kk][tx * 4 + b];
        for (int a = 0; a < 4; ++a)
          for (int b = 0; b < 4; ++b) acc[a][b] += bv[a] * xv[b];
      }
      __syncthreads();
    }
    for (int a = 0; a < 4; ++a) {
      double best = -1.0;
      int barg = 0;
      for (int b = 0; b < 4; ++b) {
        const int64_t gc = col0 + tx * 4 + b;
        const double v = fabs(static_cast<double>(acc[a][b]));
        if (gc < m && v > best) { best = v; barg = static_cast<int>(gc); }
      }
      tmax[tx][ty * 4 + a] = best;
      targ[tx][ty * 4 + a] = barg;
    }
    __syncthreads();
    if (threadIdx.x < 64) {
      double best = rowmax[threadIdx.x];
      int barg = rowarg[threadIdx.x];
      for (int t = 0; t < 16; ++t) {
        const double v = tmax[t][threadIdx.x];
        const int g = targ[t][threadIdx.x];
        if (v > best || (v == best && g < barg)) { best = v; barg = g; }
      }
      rowmax[threadIdx.x] = best;
      rowarg[threadIdx.x] = barg;
    }
    __syncthreads();
  }
  if (threadIdx.x < 64) {
    const int64_t gr = row0 + threadIdx.x;
    if (gr < N) {
      gamma[gr] = rowmax[threadIdx.x];
      if (argmax) argmax[gr] = rowarg[threadIdx.x];
    }
  }
}

__global__ void k_to_float(const double* X, int64_t n, float* Y) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i < n) Y[i] = static_cast<float>(X[i]);
}

}  // namespace

namespace {
unsigned blocks(int64_t n, int t) { return static_cast<unsigned>((n + t - 1) / t); }

void invert_by_panels(double* M, double* W, double* D, double* Lp, double* Tp, PanelMoves* mv, int* perm, int64_t m,
                      const unsigned long long* maxabs, unsigned* flag, double* out, cudaStream_t s) {
  for (int k0 = 0; k0 < m; k0 += kPanel) {
    const int nb = static_cast<int>(std::min<int64_t>(kPanel, m - k0));
    const int64_t rows = m - k0;
    // a row per thread up to 1,024 rows (two rows in 512 threads: 51 us per panel at 651 rows), then four
    auto panel = rows <= 512 ? k_panel<1, 512> : (rows <= 1024 ? k_panel<1, 1024> : k_panel<4, 512>);
    panel<<<1, rows <= 512 || rows > 1024 ? 512 : 1024, 0, s>>>(M, m, k0, nb, Lp, mv, perm, maxabs, flag);
    ProfRegion::launched();
    k_swap_solve<<<blocks(m, 128), 128, 0, s>>>(M, m, k0, nb, mv, Tp);
    ProfRegion::launched();
    const dim3 g(blocks(m, 32), std::max(1u, blocks(rows - nb, 32)));
    k_panel_update<<<g, 256, 0, s>>>(M, m, k0, nb, Lp, Tp);
    ProfRegion::launched();
  }
  MTP_CUDA(cudaGetLastError());
  k_lower<<<blocks(m * m, 256), 256, 0, s>>>(M, m, W);
  ProfRegion::launched();
  k_diag_inverse<<<blocks(m, kBack), kBack, 0, s>>>(M, m, D);
  ProfRegion::launched();
  for (int i0 = static_cast<int>((m - 1) / kBack) * kBack; i0 >= 0; i0 -= kBack) {
    const int nb = static_cast<int>(std::min<int64_t>(kBack, m - i0));
    k_back_solve<<<blocks(m, 32), 256, 0, s>>>(D, m, i0, nb, W);
    ProfRegion::launched();
    if (i0 > 0) {
      k_back_update<<<dim3(blocks(m, 32), blocks(i0, 32)), 256, 0, s>>>(M, m, i0, nb, W);
      ProfRegion::launched();
    }
  }
  k_unpermute<<<blocks(m * m, 256), 256, 0, s>>>(W, perm, m, out);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
}

void invert_by_columns(double* LU, int* piv, int64_t m, const unsigned long long* maxabs, unsigned* flag, double* out,
                       cudaStream_t s) {
  for (int64_t k = 0; k < m; ++k) {
    k_pivot<<<1, 1024, 0, s>>>(LU, m, k, piv, maxabs, flag);
    ProfRegion::launched();
    const int64_t rem = m - k - 1;
    if (rem > 0) {
      k_lcol<<<static_cast<unsigned>((rem + 255) / 256), 256, 0, s>>>(LU, m, k);
      ProfRegion::launched();
      dim3 g(static_cast<unsigned>((rem + 127) / 128), static_cast<unsigned>(rem));
      k_trail<<<g, 128, 0, s>>>(LU, m, k);
      ProfRegion::launched();
    }
  }
  k_inverse_cols<<<static_cast<unsigned>((m + 63) / 64), 64, 0, s>>>(LU, piv, m, out);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
}
}  // namespace

void slice_active_inverse(mtp_model* md, int64_t m, cudaStream_t s);

void run_lu_inverse(mtp_model* md, const double* A, int64_t m, cudaStream_t s) {
  ScopedBuf work(s);
  const size_t mm = static_cast<size_t>(m * m);
  const bool panels = m <= kPanelRows;
  const size_t panel_doubles = panels ? mm + (m + kBack) * kBack + m * kPanel + kPanel * kPanel : 0;   // W, D, Lp, Tp
  work.ensure((mm + panel_doubles + 1) * sizeof(double) + sizeof(PanelMoves) + m * sizeof(int) + 64, s);
  double* M = work.as<double>();
  unsigned long long* maxabs = reinterpret_cast<unsigned long long*>(M + mm + panel_doubles);
  PanelMoves* mv = reinterpret_cast<PanelMoves*>(maxabs + 1);
  int* perm = reinterpret_cast<int*>(mv + 1);
  md->err_flag.ensure(sizeof(unsigned), s);
  MTP_CUDA(cudaMemsetAsync(md->err_flag.p, 0, sizeof(unsigned), s));
  MTP_CUDA(cudaMemsetAsync(maxabs, 0, sizeof(unsigned long long), s));
  MTP_CUDA(cudaMemcpyAsync(M, A, mm * sizeof(double), cudaMemcpyDeviceToDevice, s));
  ProfRegion pr("active_set_lu_inverse", s);
  k_maxabs<<<std::min(blocks(m * m, 1024), 128u), 256, 0, s>>>(A, m * m, maxabs);
  ProfRegion::launched();
  k_lu_init<<<blocks(m, 256), 256, 0, s>>>(perm, m);
  ProfRegion::launched();
  md->ainv_d.ensure(mm * sizeof(double), s);
  double* inv = md->ainv_d.as<double>();
  unsigned* flag_d = md->err_flag.as<unsigned>();
  if (panels) {
    double* W = M + mm;
    double* D = W + mm;
    double* Lp = D + (m + kBack) * kBack;
    double* Tp = Lp + m * kPanel;
    invert_by_panels(M, W, D, Lp, Tp, mv, perm, m, maxabs, flag_d, inv, s);
  } else {
    invert_by_columns(M, perm, m, maxabs, flag_d, inv, s);
  }
  // mixed-path copies: K-major padded split (tensor cores) and plain FP32 (SIMT)
  const int64_t ld = grade_tc_ld(m);
  md->ainv_ld = ld;
  md->ainv_f.ensure((2 * ld * ld + m * m) * sizeof(float), s);
  float* hi = md->ainv_f.as<float>();
  k_split_ainv<<<static_cast<unsigned>((ld * ld + 255) / 256), 256, 0, s>>>(md->ainv_d.as<double>(), m, ld, hi, hi + ld * ld);
  ProfRegion::launched();
  k_to_float<<<static_cast<unsigned>((m * m + 255) / 256), 256, 0, s>>>(md->ainv_d.as<double>(), m * m, hi + 2 * ld * ld);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
  slice_active_inverse(md, m, s);
  unsigned flag = 0;
  MTP_CUDA(cudaMemcpyAsync(&flag, md->err_flag.p, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  MTP_CUDA(cudaStreamSynchronize(s));
  if (flag) throw Fail{MTP_ERR_SINGULAR, "active-set matrix is singular (LU pivot below 1e-13 max|A|)"};
  md->m_active = m;
  md->have_ainv = true;
}

void run_grade_simt(mtp_model* md, int64_t N, bool fp64, const double* rows, const float* rows_f, int64_t ld,
                    double* gamma, int32_t* argmax, cudaStream_t s) {
  const int64_t m = md->m_active;
  const unsigned g = static_cast<unsigned>((N + 63) / 64);
  if (N == 0) return;
  ProfRegion pr(fp64 ? "grade_simt_fp64" : "grade_simt_fp32", s);
  if (fp64) {
    k_grade_simt<double><<<g, 256, 0, s>>>(rows, ld, md->ainv_d.as<double>(), m, N, gamma, argmax);
    ProfRegion::launched();
  } else {
    k_grade_simt<float><<<g, 256, 0, s>>>(rows_f, ld, md->ainv_f.as<float>() + 2 * md->ainv_ld * md->ainv_ld, m, N,
                                               gamma, argmax);
    ProfRegion::launched();
  }
  MTP_CUDA(cudaGetLastError());
}

}  // namespace mtp
