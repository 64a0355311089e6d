// Per-neighborhood pass in FP64, and in dual numbers (the tangent of the parameter rows, FP64 or
// FP32), as three kernels arranged around the FP64 pipe.
//
// GB300 does 2 FP64 FMAs per clock and SM (a sixty-fourth of its FP32 rate): one warp-wide FP64
// instruction keeps the pipe busy for 16 cycles of the SM, and loads, index arithmetic, shuffles
// and shared-memory traffic in between cost next to nothing.  So these kernels spend instructions
// of every other kind to save FP64 ones and to keep all 32 lanes busy in those that remain:
//   k_wide_moments  (eqs. 3-4)  a warp takes several neighborhoods and walks their pairs as one
//       list, 32 at a time (radial functions with a lane per pair, no idle lanes at the ends of
//       neighborhoods); the pairs' monomials are formed once in shared memory (one multiply each),
//       then each lane owns every 32nd moment component: one FMA per pair and component.
//   k_wide_contract (eqs. 2, 5-6 and the adjoint)  the packed rounds of the three-kernel mixed
//       pass, their words ordered so that the terms with coefficient 1 (63 % at level 20) come
//       last: a row of 32 such words costs one FMA, another row a multiply more.
//   k_wide_adjoint  (forces, virial, radial block of eq. 9)  a lane per pair of the joint list; the
//       polynomials P_mu(r) = sum_k (dV/dM_mu,k) x^a y^b z^c and their gradients by nested Horner
//       schemes (2 FMAs per component and about 3 per (a, b), no monomials and no products of
//       powers; the generic kernel takes 13 operations per component).
//
// Per pass, before (the generic kernel, site.cu) and now:
//   FP64 energies, forces, rows, level 20, 16,384 atoms      14.1 -> 4.44 ms (1.21 + 1.60 + 1.63)
//   FP64 energies and forces, level 8, 256,000 atoms         17.3 -> 6.60
//   the same, level 24, 16,384 atoms of the liquid           83.9 -> 14.7
//   FP64 training step, level 16, 512 cells (both passes)    32.5 -> 11.3
//   mixed training step of the same cells (FP32 tangent)     3.58 -> 1.66
// At level 20 the FP64 pipe would take 2.8 ms for the operations that remain.
//
// The order of every sum over pairs and terms is fixed by the neighbor list, whatever the launch shape.
// The tangent's sums over atoms go to a row per warp or group first, so their order follows the grid
// (the SMs of the device and the number of atoms): the same from call to call.
#include <algorithm>
#include <string>
#include <type_traits>
#include <vector>

#include "dual.h"
#include "profiler.h"
#include "site_wide.h"

namespace mtp {
namespace {

constexpr int NQ = 8;       // radial polynomials of this pass
constexpr int MAXMU = 8;    // radial functions (6 at level 24)
constexpr int MAXNBW = 8;   // neighborhoods a warp takes at a time
constexpr int WPB = 8;      // warps per block of the per-pair kernels

struct WideArgs {
  DevSchedule d;
  DevNbr nb;
  const double* pos;
  const int* type;
  const double* cell;
  int64_t n_work;
  SiteOutputs o;
  void* mom;               // S[n_work x n_mom], slot order (mu, then descending a, b, c)
  const int* slot_comp;    // slot -> value index
  const int* slot_mk;      // slot -> mu | monomial << 8
  const int* mono;         // monomial -> ab pair | c << 16
  const int* ab;           // ab pair -> a | b << 8
  int n_mono, n_ab;
  int numax[MAXMU];
  const uint32_t* words_f;   // packed rounds (pfround, prround), words a | b << 12 | coefficient << 24
  const uint32_t* words_r;
  const double* coef;        // [n_coef]
  int unit;                  // the coefficient index of 1
  int nbw;                   // neighborhoods per warp (per-pair kernels)
  int pb;                    // pairs per monomial batch (moments)
  // contraction: warps per neighborhood and neighborhoods per block
  int cw, cg;
  size_t warp_bytes, c_bytes;
};

template <class R> __device__ __forceinline__ const R* theta_of(const DevSchedule& d) {
  if constexpr (std::is_same<R, float>::value) return d.theta_f;
  else return d.theta_d;
}

// the neighborhoods w0 .. w0 + nbw - 1 of a warp, their pairs as one list: lane b holds
// neighborhood b's first pair, the pairs before it in the list, its species and atom
struct Segs {
  int64_t p0;
  int64_t i;
  int pre, zi;
  int total;
  __device__ __forceinline__ void load(const WideArgs& P, int64_t w0, int lane) {
    int np = 0;
    p0 = 0; i = 0; zi = 0;
    if (lane < P.nbw && w0 + lane < P.n_work) {
      i = P.o.atom_list ? P.o.atom_list[w0 + lane] : w0 + lane;
      zi = P.type[i];
      p0 = P.nb.off[i];
      np = static_cast<int>(P.nb.off[i + 1] - p0);
    }
    int incl = np;
    for (int m = 1; m < 32; m <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, m);
      if (lane >= m) incl += v;
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
    pre = incl - np;   // lanes past the last neighborhood: total
  }
  // neighborhood of pair t of the list (the last one that starts at or before t and is not empty)
  __device__ __forceinline__ int of(const WideArgs& P, int t) const {
    int b = 0;
    for (int k = 1; k < P.nbw; ++k)
      if (__shfl_sync(0xffffffffu, pre, k) <= t) b = k;
    return b;
  }
};

// r_ij = (x_j + n.H) - x_i (and its tangent U_j - U_i + S r) for pair p of center i
template <class S, class R>
__device__ __forceinline__ void pair_vector(const WideArgs& P, int64_t i, int64_t p, int j, S& rx, S& ry, S& rz) {
  R x, y, z;
  if constexpr (std::is_same<R, float>::value) {
    const float4 v = P.nb.pr32[p];
    x = v.x; y = v.y; z = v.z;
  } else {
    const int img = P.nb.pimg[p];
    double sh0 = 0.0, sh1 = 0.0, sh2 = 0.0;
    if (img) {
      const int n0 = unpack_img(img, 0), n1 = unpack_img(img, 1), n2 = unpack_img(img, 2);
      const double* H = P.cell + 9 * static_cast<int64_t>(P.nb.atom_cfg[i]);
      sh0 = n0 * H[0] + n1 * H[3] + n2 * H[6];
      sh1 = n0 * H[1] + n1 * H[4] + n2 * H[7];
      sh2 = n0 * H[2] + n1 * H[5] + n2 * H[8];
    }
    x = (P.pos[3 * static_cast<int64_t>(j) + 0] + sh0) - P.pos[3 * i + 0];
    y = (P.pos[3 * static_cast<int64_t>(j) + 1] + sh1) - P.pos[3 * i + 1];
    z = (P.pos[3 * static_cast<int64_t>(j) + 2] + sh2) - P.pos[3 * i + 2];
  }
  if constexpr (std::is_same<S, R>::value) {
    rx = x; ry = y; rz = z;
  } else {
    const double* U = P.o.U;
    const double* Sm = P.o.Scfg + 9 * static_cast<int64_t>(P.nb.atom_cfg[i]);
    const int64_t jj = j;
    const R dx = R(U[3 * jj + 0] - U[3 * i + 0]) + (R(Sm[0]) * x + R(Sm[1]) * y + R(Sm[2]) * z);
    const R dy = R(U[3 * jj + 1] - U[3 * i + 1]) + (R(Sm[3]) * x + R(Sm[4]) * y + R(Sm[5]) * z);
    const R dz = R(U[3 * jj + 2] - U[3 * i + 2]) + (R(Sm[6]) * x + R(Sm[7]) * y + R(Sm[8]) * z);
    rx = {x, dx}; ry = {y, dy}; rz = {z, dz};
  }
}

// Chebyshev polynomials of one distance: T_b, U_b (T_b' = b U_(b-1)), the cut-off factor, 1 / |r|
template <class R>
struct Radial {
  R T[NQ], U[NQ];
  R w, w2, dxw2, inv, rdot;   // R_cut - r, its square, (dx/dr) w^2, 1 / r, dr/dt
  template <class S>
  __device__ __forceinline__ void set(S rx, S ry, S rz, R rmin, R rcut) {
    const R x = vpart(rx), y = vpart(ry), z = vpart(rz);
    const R rr = ssqrt(madd(x, x, madd(y, y, z * z)));
    inv = R(1) / rr;
    rdot = (x * dpart(rx) + y * dpart(ry) + z * dpart(rz)) * inv;
    const R sc = R(1) / (rcut - rmin);
    const R t = (R(2) * rr - (rmin + rcut)) * sc;
    const R t2 = t + t;
    w = rcut - rr;
    w2 = w * w;
    dxw2 = (sc + sc) * w2;
    T[0] = R(1); T[1] = t;
    U[0] = R(1); U[1] = t2;
#pragma unroll
    for (int b = 2; b < NQ; ++b) {
      T[b] = madd(t2, T[b - 1], -T[b - 2]);
      U[b] = madd(t2, U[b - 1], -U[b - 2]);
    }
  }
  // f_mu (and f'_mu) from the coefficients c and b c
  template <bool DER>
  __device__ __forceinline__ void f(const R* c, const R* bc, R& fv, R& fd) const {
    R F = c[0];   // T_0 = 1
#pragma unroll
    for (int b = 1; b < NQ; ++b) F = madd(c[b], T[b], F);
    fv = F * w2;
    if constexpr (DER) {
      R D = bc[1];   // U_0 = 1
#pragma unroll
      for (int b = 2; b < NQ; ++b) D = madd(bc[b], U[b - 1], D);
      fd = madd(dxw2, D, R(-2) * w * F);
    }
  }
  // Q_b, and as a dual its derivative along the tangent
  template <class S>
  __device__ __forceinline__ S q(int b, R Tb, R Ub1) const {
    if constexpr (std::is_same<S, R>::value) return Tb * w2;
    else return S{Tb * w2, (dxw2 * (R(b) * Ub1) - R(2) * (w * Tb)) * rdot};
  }
};

// radial coefficients c and b c (the derivative's) in shared memory
template <class R>
__device__ __forceinline__ void stage_coefficients(const DevSchedule& d, R* c, R* bc, int nc) {
  const R* th = theta_of<R>(d) + d.n_types + d.n_lin;
  for (int k = threadIdx.x; k < nc; k += blockDim.x) {
    c[k] = th[k];
    bc[k] = R(k % NQ) * th[k];
  }
}

// ------------------------------------------------------------------------------------
// moments (eqs. 3-4): lane l owns slots l, l + 32, ...; RND rounds of 32 slots
// ------------------------------------------------------------------------------------
template <class S, class R, int RND>
__global__ void __launch_bounds__(WPB * 32, 1) k_wide_moments(WideArgs P) {
  extern __shared__ __align__(16) unsigned char smem[];
  const DevSchedule& d = P.d;
  const int T = d.n_types, NR = d.n_rad, nc = T * T * NR * NQ;
  R* ctab = reinterpret_cast<R*>(smem);
  R* btab = ctab + nc;
  stage_coefficients<R>(d, ctab, btab, nc);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int D1 = d.nu_max + 1, PB = P.pb, NM = P.n_mono, NAB = P.n_ab;
  S* F = reinterpret_cast<S*>(smem + P.c_bytes + warp * P.warp_bytes);   // [32][NR]
  S* X = F + 32 * NR;             // [3][32]: the pairs' vectors
  S* PW = X + 96;                 // [PB][3][D1]: powers
  S* XY = PW + PB * 3 * D1;       // [PB][NAB]
  S* MO = XY + PB * NAB;          // [PB][NM]
  __syncthreads();
  const R rmin = R(d.r_min), rcut = R(d.r_cut);
  const int n_mom = d.n_mom;
  int slot[RND];
#pragma unroll
  for (int r = 0; r < RND; ++r) {
    const int s = lane + 32 * r;
    slot[r] = s < n_mom ? P.slot_mk[s] : 0;
  }
  S* const mom = static_cast<S*>(P.mom);
  const int64_t n_tasks = (P.n_work + P.nbw - 1) / P.nbw;
  for (int64_t task = static_cast<int64_t>(blockIdx.x) * nw + warp; task < n_tasks;
       task += static_cast<int64_t>(gridDim.x) * nw) {
    const int64_t w0 = task * P.nbw;
    const int n_nb = static_cast<int>(min(static_cast<int64_t>(P.nbw), P.n_work - w0));
    Segs sg;
    sg.load(P, w0, lane);
    S acc[RND];
#pragma unroll
    for (int r = 0; r < RND; ++r) acc[r] = mk<S>(R(0));
    int cur = 0;   // neighborhood being summed
    auto flush_to = [&](int nb) {
      for (; cur < nb; ++cur) {
        S* out = mom + (w0 + cur) * n_mom;
#pragma unroll
        for (int r = 0; r < RND; ++r) {
          if (lane + 32 * r < n_mom) out[lane + 32 * r] = acc[r];
          acc[r] = mk<S>(R(0));
        }
      }
    };
    for (int base = 0; base < sg.total; base += 32) {
      const int t = base + lane;
      const bool act = t < sg.total;
      const int nb = sg.of(P, act ? t : sg.total - 1);
      const int64_t p0 = __shfl_sync(0xffffffffu, sg.p0, nb), i = __shfl_sync(0xffffffffu, sg.i, nb);
      const int pre = __shfl_sync(0xffffffffu, sg.pre, nb), zi = __shfl_sync(0xffffffffu, sg.zi, nb);
      __syncwarp();
      if (act) {
        const int64_t p = p0 + (t - pre);
        const int j = P.nb.pj[p];
        S rx, ry, rz;
        pair_vector<S, R>(P, i, p, j, rx, ry, rz);
        Radial<R> ra;
        ra.set(rx, ry, rz, rmin, rcut);
        const R* cz = ctab + (zi * T + P.type[j]) * NR * NQ;
        const R* bz = btab + (zi * T + P.type[j]) * NR * NQ;
        for (int mu = 0; mu < NR; ++mu) {
          R fv, fd = R(0);
          ra.template f<!std::is_same<S, R>::value>(cz + mu * NQ, bz + mu * NQ, fv, fd);
          F[lane * NR + mu] = mk2<S>(fv, fd * ra.rdot);
        }
        X[lane] = rx; X[32 + lane] = ry; X[64 + lane] = rz;
      }
      __syncwarp();
      const int n_here = min(32, sg.total - base);
      for (int q0 = 0; q0 < n_here; q0 += PB) {
        const int nq = min(PB, n_here - q0);
        for (int e = lane; e < 3 * nq; e += 32) {
          const int q = e / 3, ax = e - 3 * q;
          S* pw = PW + e * D1;
          const S x = X[32 * ax + q0 + q];
          S v = x;
          pw[0] = mk<S>(R(1));
          if (D1 > 1) pw[1] = v;
          for (int k = 2; k < D1; ++k) { v = v * x; pw[k] = v; }
        }
        __syncwarp();
        for (int e = lane; e < nq * NAB; e += 32) {
          const int q = e / NAB, ab = P.ab[e - q * NAB];
          const S* pw = PW + q * 3 * D1;
          XY[e] = pw[ab & 255] * pw[D1 + (ab >> 8)];
        }
        __syncwarp();
        for (int e = lane; e < nq * NM; e += 32) {
          const int q = e / NM, m = P.mono[e - q * NM];
          MO[e] = XY[q * NAB + (m & 0xffff)] * PW[(q * 3 + 2) * D1 + (m >> 16)];
        }
        __syncwarp();
        for (int q = 0; q < nq; ++q) {
          flush_to(__shfl_sync(0xffffffffu, nb, q0 + q));
          const S* f = F + (q0 + q) * NR;
          const S* mo = MO + q * NM;
#pragma unroll
          for (int r = 0; r < RND; ++r)
            if (32 * r < n_mom) acc[r] = madd(f[slot[r] & 255], mo[slot[r] >> 8], acc[r]);
        }
        __syncwarp();
      }
    }
    flush_to(n_nb);
    __syncwarp();
  }
}

// ------------------------------------------------------------------------------------
// contraction and its adjoint (eqs. 2, 5-6): P.cw warps per neighborhood, P.cg neighborhoods per block
// ------------------------------------------------------------------------------------
enum : int { W_EFS = 1, W_ROWS = 2, W_TAN = 4 };

template <class S, class R, int MODE>
__global__ void __launch_bounds__(512, 1) k_wide_contract(WideArgs P) {
  extern __shared__ __align__(16) unsigned char smem[];
  const DevSchedule& d = P.d;
  R* coef = reinterpret_cast<R*>(smem);
  for (int k = threadIdx.x; k < d.n_coef; k += blockDim.x) coef[k] = static_cast<R>(P.coef[k]);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int W = P.cw, grp = warp / W, wig = warp - grp * W, tl = 32 * wig + lane, nt = 32 * W;
  const int NV = d.n_vals + 1;   // values and the always-zero slot of the padding words
  S* vals = reinterpret_cast<S*>(smem + P.c_bytes + grp * P.warp_bytes);
  S* grads = vals + NV;
  if (tl == 0) { vals[d.n_vals] = mk<S>(R(0)); grads[d.n_vals] = mk<S>(R(0)); }
  const R* theta = theta_of<R>(d);
  const R* seed;
  if constexpr (std::is_same<R, float>::value) seed = d.seed_f;
  else seed = d.seed_d;
  __syncthreads();
  auto group_sync = [&] {
    if (W == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(nt) : "memory");
  };
  const int T = d.n_types, n_mom = d.n_mom;
  S* const mom = static_cast<S*>(P.mom);
  // the rounds of one direction: every warp of the group walks the headers and takes its own
  auto walk = [&](const int4* rounds, const int* entries, const uint32_t* words, int n, const S* yv, S* dst, bool seeded) {
    int k = 0;   // round within the wave
    for (int r = 0; r < n; ++r) {
      const int4 rd = rounds[r];
      if (W == 1 || k % W == wig) {
        const int ent = entries[32 * r + lane];
        const bool lead = ent >= 0 && ((ent >> 20) & 1);
        S a0 = mk<S>((seeded && lead) ? seed[ent & 0xffff] : R(0)), a1 = mk<S>(R(0));
        const uint32_t* wp = words + rd.y + lane;
        const int L = rd.x;
        uint32_t nxt[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) nxt[u] = u < L ? wp[32 * u] : 0u;
        for (int it = 0; it < L; it += 4) {
          uint32_t wd[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) wd[u] = nxt[u];
#pragma unroll
          for (int u = 0; u < 4; ++u) nxt[u] = it + 4 + u < L ? wp[32 * (it + 4 + u)] : 0u;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (it + u >= L) break;
            const int ci = static_cast<int>(wd[u] >> 24);
            S a = vals[wd[u] & 4095u];
            const S b = yv[(wd[u] >> 12) & 4095u];
            if (__any_sync(0xffffffffu, ci != P.unit)) a = coef[ci] * a;
            if (u & 1) a1 = madd(a, b, a1);
            else a0 = madd(a, b, a0);
          }
        }
        if (L > 1) a0 = a0 + a1;
        if (rd.w) {
          const int g = 1 << ((ent >> 16) & 15);
          for (int s = 1; s < 32; s <<= 1) {
            if (!__any_sync(0xffffffffu, ent >= 0 && g > s)) break;
            const S o = shfl_xor(a0, s);
            if (g > s) a0 = a0 + o;
          }
        }
        if (lead) dst[ent & 0xffff] = a0;
      }
      ++k;
      if (rd.z) { group_sync(); k = 0; }
    }
  };
  for (int64_t wk = static_cast<int64_t>(blockIdx.x) * P.cg + grp; wk < P.n_work;
       wk += static_cast<int64_t>(gridDim.x) * P.cg) {
    const int64_t i = P.o.atom_list ? P.o.atom_list[wk] : wk;
    S* const mg = mom + wk * n_mom;
    for (int s = tl; s < n_mom; s += nt) vals[P.slot_comp[s]] = mg[s];
    group_sync();
    walk(d.pfround, d.pfr_dst, P.words_f, d.n_pfround, vals, vals, false);
    const int zi = P.type[i];
    if constexpr ((MODE & W_EFS) != 0) {
      if (wig == 0) {
        S acc = mk<S>(R(0));
        for (int a = lane; a < d.n_lin; a += 32) acc = madd(theta[T + a], vals[d.basis_idx[a]], acc);
        acc = warp_sum(acc);
        if (lane == 0) P.o.V[i] = static_cast<double>(vpart(acc)) + d.theta_d[zi];
      }
    }
    walk(d.prround, d.prr_val, P.words_r, d.n_prround, grads, grads, true);
    for (int s = tl; s < n_mom; s += nt) mg[s] = grads[P.slot_comp[s]];
    if constexpr ((MODE & W_ROWS) != 0) {
      double* out = P.o.rows + (P.o.row_pos ? P.o.row_pos[i] : wk) * P.o.rows_ld;
      for (int k = tl; k < T + d.n_lin; k += nt)
        out[k] = k < T ? (k == zi ? 1.0 : 0.0) : static_cast<double>(vpart(vals[d.basis_idx[k - T]]));
    }
    if constexpr ((MODE & W_TAN) != 0) {
      // coef b_i - d/dt b_i, into this group's row of partial sums
      double* acc = P.o.grad_part + (static_cast<int64_t>(blockIdx.x) * P.cg + grp) * d.n_params;
      const double cf = P.o.coef[P.nb.atom_cfg[i]];
      for (int k = tl; k < T + d.n_lin; k += nt) {
        if (k < T) {
          if (k == zi) acc[k] += cf;
        } else {
          const S B = vals[d.basis_idx[k - T]];
          acc[k] += fma(cf, static_cast<double>(vpart(B)), -static_cast<double>(dpart(B)));
        }
      }
    }
    group_sync();
  }
}

// ------------------------------------------------------------------------------------
// pair adjoint: a lane per pair of the warp's joint list
// ------------------------------------------------------------------------------------
template <class S, class R, int MODE>
__global__ void __launch_bounds__(WPB * 32, 1) k_wide_adjoint(WideArgs P) {
  constexpr bool EFS = (MODE & W_EFS) != 0;
  constexpr bool BLK = (MODE & (W_ROWS | W_TAN)) != 0;   // radial block of the rows
  extern __shared__ __align__(16) unsigned char smem[];
  const DevSchedule& d = P.d;
  const int T = d.n_types, NR = d.n_rad, nc = T * T * NR * NQ;
  R* ctab = reinterpret_cast<R*>(smem);
  R* btab = ctab + nc;
  stage_coefficients<R>(d, ctab, btab, nc);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int n_mom = d.n_mom, nblk = BLK ? NR * NQ : 0, CBN = T * nblk;
  // per pair of a round: g_mu, Q_b (radial block), -dV/dr, r (virial); an odd stride
  const int rec = ((BLK ? NR + NQ : 0) + (EFS ? 6 : 0)) | 1;
  S* G = reinterpret_cast<S*>(smem + P.c_bytes + warp * P.warp_bytes);   // [nbw][n_mom]
  S* ST = G + P.nbw * n_mom;    // [32][rec]
  S* CB = ST + 32 * rec;        // [T][NR][NQ] then the virial [9]
  __syncthreads();
  const R rmin = R(d.r_min), rcut = R(d.r_cut);
  const int64_t off_c = T + d.n_lin;
  // this lane's entries of (radial block | virial): offsets of the two factors in the record
  const int n_ent = nblk + (EFS ? 9 : 0);
  const S* const mom = static_cast<const S*>(P.mom);
  const int64_t n_tasks = (P.n_work + P.nbw - 1) / P.nbw;
  for (int64_t task = static_cast<int64_t>(blockIdx.x) * nw + warp; task < n_tasks;
       task += static_cast<int64_t>(gridDim.x) * nw) {
    const int64_t w0 = task * P.nbw;
    const int n_nb = static_cast<int>(min(static_cast<int64_t>(P.nbw), P.n_work - w0));
    Segs sg;
    sg.load(P, w0, lane);
    for (int k = lane; k < n_nb * n_mom; k += 32) G[k] = mom[w0 * n_mom + k];
    for (int k = lane; k < CBN + 9; k += 32) CB[k] = mk<S>(R(0));
    __syncwarp();
    int cur = 0;
    auto flush_to = [&](int nb) {
      for (; cur < nb; ++cur) {
        __syncwarp();
        const int64_t wk = w0 + cur;
        const int64_t i = __shfl_sync(0xffffffffu, sg.i, cur);
        const int zi = __shfl_sync(0xffffffffu, sg.zi, cur);
        if constexpr (EFS) {
          if (lane < 9) P.o.Wat[9 * i + lane] = static_cast<double>(vpart(CB[CBN + lane]));
        }
        if constexpr ((MODE & W_ROWS) != 0) {
          double* out = P.o.rows + (P.o.row_pos ? P.o.row_pos[i] : wk) * P.o.rows_ld;
          for (int z = 0; z < T; ++z)
            for (int e = lane; e < CBN; e += 32)
              out[off_c + static_cast<int64_t>(z) * CBN + e] = z == zi ? static_cast<double>(vpart(CB[e])) : 0.0;
          for (int64_t k = d.n_params + lane; k < P.o.rows_ld; k += 32) out[k] = 0.0;
        }
        if constexpr ((MODE & W_TAN) != 0) {
          double* acc = P.o.grad_part + (static_cast<int64_t>(blockIdx.x) * nw + warp) * d.n_params + off_c +
                        static_cast<int64_t>(zi) * CBN;
          const double cf = P.o.coef[P.nb.atom_cfg[i]];
          for (int e = lane; e < CBN; e += 32)
            acc[e] += fma(cf, static_cast<double>(vpart(CB[e])), -static_cast<double>(dpart(CB[e])));
        }
        __syncwarp();
        for (int k = lane; k < CBN + 9; k += 32) CB[k] = mk<S>(R(0));
        __syncwarp();
      }
    };
    for (int base = 0; base < sg.total; base += 32) {
      const int t = base + lane;
      const bool act = t < sg.total;
      const int nb = sg.of(P, act ? t : sg.total - 1);
      const int64_t p0 = __shfl_sync(0xffffffffu, sg.p0, nb), i = __shfl_sync(0xffffffffu, sg.i, nb);
      const int pre = __shfl_sync(0xffffffffu, sg.pre, nb), zi = __shfl_sync(0xffffffffu, sg.zi, nb);
      const int64_t p = p0 + ((act ? t : sg.total - 1) - pre);   // an idle lane repeats the last pair
      const int j = P.nb.pj[p];
      const int zj = P.type[j];
      S rx, ry, rz;
      pair_vector<S, R>(P, i, p, j, rx, ry, rz);
      Radial<R> ra;
      ra.set(rx, ry, rz, rmin, rcut);
      const R* cz = ctab + (zi * T + zj) * NR * NQ;
      const R* bz = btab + (zi * T + zj) * NR * NQ;
      const S* g = G + nb * n_mom;
      S* st = ST + lane * rec;
      __syncwarp();
      if constexpr (BLK) {
#pragma unroll
        for (int b = 0; b < NQ; ++b) st[NR + b] = ra.template q<S>(b, ra.T[b], b > 0 ? ra.U[b > 0 ? b - 1 : 0] : R(0));
      }
      S gx = mk<S>(R(0)), gy = mk<S>(R(0)), gz = mk<S>(R(0));
      R rad = R(0);
      for (int mu = 0; mu < NR; ++mu) {
        const int n = P.numax[mu];
        // Horner in x of Horner in y of Horner in z, with the derivatives
        S p_v = mk<S>(R(0)), p_x = mk<S>(R(0)), p_y = mk<S>(R(0)), p_z = mk<S>(R(0));
        for (int a = n; a >= 0; --a) {
          S a_v = mk<S>(R(0)), a_y = mk<S>(R(0)), a_z = mk<S>(R(0));
          const int nb1 = n - a;
          for (int b = nb1; b >= 0; --b) {
            S tv = *g++, uv = mk<S>(R(0));
            int c = nb1 - b;
            if (c > 0) {
              if (EFS) uv = tv;
              tv = madd(tv, rz, *g++);
              for (--c; c > 0; --c) {
                if (EFS) uv = madd(uv, rz, tv);
                tv = madd(tv, rz, *g++);
              }
            }
            if (b == nb1) {
              a_v = tv;
              if (EFS) a_z = uv;
            } else {
              if (EFS) {
                a_y = b == nb1 - 1 ? a_v : madd(a_y, ry, a_v);
                a_z = madd(a_z, ry, uv);
              }
              a_v = madd(a_v, ry, tv);
            }
          }
          if (a == n) {
            p_v = a_v;
            if (EFS) { p_y = a_y; p_z = a_z; }
          } else {
            if (EFS) {
              p_x = a == n - 1 ? p_v : madd(p_x, rx, p_v);
              p_y = madd(p_y, rx, a_y);
              p_z = madd(p_z, rx, a_z);
            }
            p_v = madd(p_v, rx, a_v);
          }
        }
        if constexpr (EFS) {
          R fv, fd;
          ra.template f<true>(cz + mu * NQ, bz + mu * NQ, fv, fd);
          gx = madd(mk<S>(fv), p_x, gx);
          gy = madd(mk<S>(fv), p_y, gy);
          gz = madd(mk<S>(fv), p_z, gz);
          rad = madd(fd, vpart(p_v), rad);
        }
        if constexpr (BLK) st[mu] = p_v;
      }
      if constexpr (EFS) {
        const S s = mk<S>(rad * ra.inv);
        gx = madd(s, rx, gx);
        gy = madd(s, ry, gy);
        gz = madd(s, rz, gz);
        if (act) {
          R* out = static_cast<R*>(P.o.G) + 3 * p;
          out[0] = vpart(gx); out[1] = vpart(gy); out[2] = vpart(gz);
        }
        S* e = st + (BLK ? NR + NQ : 0);
        e[0] = mk<S>(-vpart(gx)); e[1] = mk<S>(-vpart(gy)); e[2] = mk<S>(-vpart(gz));
        e[3] = rx; e[4] = ry; e[5] = rz;
      }
      __syncwarp();
      // sums over the pairs of a neighborhood, in list order: entry e of the radial block of the
      // neighbor's species, or of the virial, is one product of two record fields per pair
      const int n_here = min(32, sg.total - base);
      for (int q = 0; q < n_here; ++q) {
        flush_to(__shfl_sync(0xffffffffu, nb, q));
        const int z = __shfl_sync(0xffffffffu, zj, q);
        const S* r = ST + q * rec;
        for (int e = lane; e < n_ent; e += 32) {
          const bool blk = e < nblk;
          const int w = e - nblk;
          const int ia = blk ? e / NQ : (BLK ? NR + NQ : 0) + w / 3;
          const int ib = blk ? NR + e % NQ : (BLK ? NR + NQ : 0) + 3 + w % 3;
          S* at = CB + (blk ? z * nblk + e : CBN + w);
          *at = madd(r[ia], r[ib], *at);
        }
      }
      __syncwarp();
    }
    flush_to(n_nb);
    __syncwarp();
  }
}

int num_sms() {
  int dev = 0, nsm = 0;
  MTP_CUDA(cudaGetDevice(&dev));
  MTP_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  return nsm;
}

constexpr size_t kSmem = 227 * 1024;
size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

// launches `kern` with `warps` warps of `warp_bytes` each (halved until they fit) over `tasks` warp
// tasks; returns the warps launched
template <class K>
int64_t launch_warps(K kern, WideArgs P, size_t warp_bytes, int64_t tasks, int64_t max_warps, const char* name,
                     cudaStream_t s) {
  int warps = WPB;
  while (warps > 1 && P.c_bytes + warps * warp_bytes > kSmem) --warps;
  const size_t smem = P.c_bytes + warps * warp_bytes;
  P.warp_bytes = warp_bytes;
  allow_smem(kern);
  int per = 0;
  MTP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, warps * 32, smem));
  int64_t grid = std::min<int64_t>((tasks + warps - 1) / warps, static_cast<int64_t>(num_sms()) * std::max(per, 1));
  if (max_warps > 0) grid = std::min<int64_t>(grid, std::max<int64_t>(1, max_warps / warps));
  grid = std::max<int64_t>(grid, 1);
  ProfRegion pr(name, s);
  kern<<<static_cast<unsigned>(grid), warps * 32, smem, s>>>(P);
  ProfRegion::launched();
  MTP_CUDA(cudaGetLastError());
  return grid * warps;
}

// bytes per warp of the per-pair kernels
template <class S>
size_t moments_bytes(const DevSchedule& d, int n_mono, int n_ab, int pb) {
  return align16((32 * d.n_rad + 96 + static_cast<size_t>(pb) * (3 * (d.nu_max + 1) + n_ab + n_mono)) * sizeof(S));
}
template <class S>
size_t adjoint_bytes(const DevSchedule& d, int nbw) {
  return align16((static_cast<size_t>(nbw) * d.n_mom + 32 * ((d.n_rad + NQ + 6) | 1) + d.n_types * d.n_rad * NQ + 9) * sizeof(S));
}
template <class S>
size_t group_bytes(const DevSchedule& d) {
  return align16(2 * static_cast<size_t>(d.n_vals + 1) * sizeof(S));
}
template <class R>
size_t coef_bytes(const DevSchedule& d) {
  return align16(std::max<size_t>(2 * static_cast<size_t>(d.n_types) * d.n_types * d.n_rad * NQ, 256) * sizeof(R));
}

template <class S, class R>
bool fits(const mtp_model* m) {
  const DevSchedule& d = m->ds;
  const size_t c = coef_bytes<R>(d);
  return c + moments_bytes<S>(d, m->wide.n_mono, m->wide.n_ab, 1) <= kSmem && c + adjoint_bytes<S>(d, 1) <= kSmem &&
         align16(256 * sizeof(R)) + group_bytes<S>(d) <= kSmem;
}

template <class S, class R, int MODE>
void launch_wide(const mtp_model* m, WideArgs P, int64_t max_part, int64_t* n_part, cudaStream_t s) {
  const DevSchedule& d = P.d;
  const int nsm = num_sms();
  // neighborhoods per warp: up to 8, fewer where there would not be two tasks per warp of the GPU
  P.nbw = MAXNBW;
  while (P.nbw > 1 && P.n_work < static_cast<int64_t>(nsm) * WPB * 2 * P.nbw) P.nbw /= 2;
  P.c_bytes = coef_bytes<R>(d);
  // ---- moments ----
  {
    // pairs per monomial batch: 16 where eight warps' tables fit shared memory; in FP32, which is
    // bound by latency and not by its pipe, where two such blocks fit (level 16 tangent of 34,968
    // atoms: 1.16 -> 0.72 ms; FP64 gains nothing at that size)
    const size_t room = sizeof(R) == 4 ? kSmem / 2 : kSmem;
    P.pb = 16;
    while (P.pb > 1 && P.c_bytes + WPB * moments_bytes<S>(d, P.n_mono, P.n_ab, P.pb) > room) P.pb /= 2;
    const size_t wb = moments_bytes<S>(d, P.n_mono, P.n_ab, P.pb);
    const int64_t tasks = (P.n_work + P.nbw - 1) / P.nbw;
    auto go = [&](auto kern) { launch_warps(kern, P, wb, tasks, 0, "wide_moments", s); };
    if (d.n_mom <= 64) go(k_wide_moments<S, R, 2>);
    else if (d.n_mom <= 160) go(k_wide_moments<S, R, 5>);
    else if (d.n_mom <= 320) go(k_wide_moments<S, R, 10>);
    else go(k_wide_moments<S, R, 19>);
  }
  int64_t rows_used = 0;
  // ---- contraction ----
  {
    WideArgs C = P;
    C.c_bytes = align16(256 * sizeof(R));
    C.warp_bytes = group_bytes<S>(d);
    // neighborhoods per block: at most 8 (a warp each); larger arrays leave several warps for each
    C.cg = static_cast<int>(std::min<size_t>(8, (kSmem - C.c_bytes) / C.warp_bytes));
    C.cw = C.cg >= 6 ? 1 : (C.cg >= 4 ? 2 : (C.cg >= 2 ? 4 : 12));
    const size_t smem = C.c_bytes + C.cg * C.warp_bytes;
    auto kern = k_wide_contract<S, R, MODE>;
    allow_smem(kern);
    int per = 0;
    MTP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, C.cg * C.cw * 32, smem));
    int64_t grid = std::min<int64_t>((P.n_work + C.cg - 1) / C.cg, static_cast<int64_t>(nsm) * std::max(per, 1));
    if (MODE & W_TAN) grid = std::min<int64_t>(grid, max_part / C.cg);
    grid = std::max<int64_t>(grid, 1);
    ProfRegion pr("wide_contract", s);
    kern<<<static_cast<unsigned>(grid), C.cg * C.cw * 32, smem, s>>>(C);
    ProfRegion::launched();
    MTP_CUDA(cudaGetLastError());
    rows_used = grid * C.cg;
  }
  // ---- pair adjoint ----
  {
    while (P.nbw > 1 && P.c_bytes + WPB * adjoint_bytes<S>(d, P.nbw) > kSmem) P.nbw /= 2;
    const int64_t tasks = (P.n_work + P.nbw - 1) / P.nbw;
    const int64_t used = launch_warps(k_wide_adjoint<S, R, MODE>, P, adjoint_bytes<S>(d, P.nbw), tasks,
                                      (MODE & W_TAN) ? max_part : 0, "wide_adjoint", s);
    rows_used = std::max(rows_used, used);
  }
  if (n_part) *n_part = rows_used;
}

}  // namespace

// Tables of the pass (at load time): slots in Horner order, monomials, the words with the unit
// coefficients last.  Left empty for shapes without the pass.
void wide_prepare(mtp_model* m) {
  const DevSchedule& d = m->ds;
  const Schedule& S = m->sched;
  m->wide = {};
  if (!m->wide_words.n_coef || d.n_q != NQ || d.n_rad > MAXMU || d.n_mom > 608 || d.n_vals + 1 > 4096) return;
  std::vector<int> numax(d.n_rad, -1);
  for (int c = 0; c < d.n_mom; ++c) {
    const int deg = S.comp_exp[c][0] + S.comp_exp[c][1] + S.comp_exp[c][2];
    numax[S.comp_mu[c]] = std::max(numax[S.comp_mu[c]], deg);
  }
  // monomials x^a y^b z^c of degree <= nu_max, by (a, b), then c
  const int nu = d.nu_max;
  std::vector<int> ab, mono;
  std::vector<int> first((nu + 1) * (nu + 1), -1);
  for (int a = 0; a <= nu; ++a)
    for (int b = 0; a + b <= nu; ++b) {
      first[a * (nu + 1) + b] = static_cast<int>(mono.size());
      for (int c = 0; a + b + c <= nu; ++c) mono.push_back(static_cast<int>(ab.size()) | (c << 16));
      ab.push_back(a | (b << 8));
    }
  // slots: mu, then descending a, b, c; every (mu, a, b, c) of degree <= numax(mu) must be present
  std::vector<int> slot_comp, slot_mk;
  for (int mu = 0; mu < d.n_rad; ++mu) {
    if (numax[mu] < 0 || numax[mu] > nu) return;
    for (int a = numax[mu]; a >= 0; --a)
      for (int b = numax[mu] - a; b >= 0; --b)
        for (int c = numax[mu] - a - b; c >= 0; --c) {
          int at = -1;
          for (int k = 0; k < d.n_mom; ++k)
            if (S.comp_mu[k] == mu && S.comp_exp[k][0] == a && S.comp_exp[k][1] == b && S.comp_exp[k][2] == c) at = k;
          if (at < 0) return;
          slot_comp.push_back(at);
          slot_mk.push_back(mu | ((first[a * (nu + 1) + b] + c) << 8));
        }
  }
  if (static_cast<int>(slot_comp.size()) != d.n_mom) return;
  std::vector<int> blob;
  auto put = [&](const std::vector<int>& v) {
    const size_t at = blob.size();
    blob.insert(blob.end(), v.begin(), v.end());
    return at;
  };
  const size_t o_sc = put(slot_comp), o_mk = put(slot_mk), o_mo = put(mono), o_ab = put(ab);
  m->wide_tab.ensure(blob.size() * sizeof(int), 0);
  MTP_CUDA(cudaMemcpy(m->wide_tab.p, blob.data(), blob.size() * sizeof(int), cudaMemcpyHostToDevice));
  const int* base = m->wide_tab.as<int>();
  m->wide.slot_comp = base + o_sc;
  m->wide.slot_mk = base + o_mk;
  m->wide.mono = base + o_mo;
  m->wide.ab = base + o_ab;
  m->wide.n_mono = static_cast<int>(mono.size());
  m->wide.n_ab = static_cast<int>(ab.size());
  m->wide.numax = numax;
}

size_t wide_workspace(const mtp_model* m, int64_t n_work, bool fp64, bool tangent) {
  if (!m->wide.slot_comp) return 0;
  const bool ok = tangent ? (fp64 ? fits<Dual<double>, double>(m) : fits<Dual<float>, float>(m))
                          : (fp64 ? fits<double, double>(m) : fits<float, float>(m));
  if (!ok) return 0;
  return static_cast<size_t>(std::max<int64_t>(n_work, 1)) * m->ds.n_mom * (fp64 ? 8 : 4) * (tangent ? 2 : 1);
}

bool run_sites_wide(mtp_model* m, const mtp_batch* b, const mtp_nbr* nb, bool fp64, const SiteOutputs& o, bool tangent,
                    int64_t max_part, int64_t* n_part, cudaStream_t s) {
  const int64_t n_work = o.atom_list ? o.n_list : nb->n_atoms;
  if (!o.wide || !wide_workspace(m, n_work, fp64, tangent)) return false;
  const bool efs = o.V != nullptr, rows = o.rows != nullptr;
  if (o.rows_hi || (!tangent && !efs && !rows) || (efs && (!o.G || !o.Wat || !fp64))) return false;
  WideArgs P{};
  P.d = m->ds;
  P.nb = nb->dn;
  P.pos = b->pos;
  P.type = b->type;
  P.cell = b->cell;
  P.n_work = n_work;
  P.o = o;
  P.mom = o.wide;
  P.slot_comp = m->wide.slot_comp;
  P.slot_mk = m->wide.slot_mk;
  P.mono = m->wide.mono;
  P.ab = m->wide.ab;
  P.n_mono = m->wide.n_mono;
  P.n_ab = m->wide.n_ab;
  for (int k = 0; k < m->ds.n_rad; ++k) P.numax[k] = m->wide.numax[k];
  P.words_f = m->wide_words.f;
  P.words_r = m->wide_words.r;
  P.coef = m->wide_words.coef;
  P.unit = m->wide_words.unit;
  m->last_fast = m->last_split = false;
  m->last_wide = true;
  m->last_warps = WPB;
  if (n_part) *n_part = 0;
  if (n_work == 0) return true;
  if (tangent) {
    if (fp64) launch_wide<Dual<double>, double, W_TAN>(m, P, max_part, n_part, s);
    else launch_wide<Dual<float>, float, W_TAN>(m, P, max_part, n_part, s);
  } else if (!fp64) {
    launch_wide<float, float, W_ROWS>(m, P, 0, nullptr, s);
  } else if (efs && rows) {
    launch_wide<double, double, W_EFS | W_ROWS>(m, P, 0, nullptr, s);
  } else if (efs) {
    launch_wide<double, double, W_EFS>(m, P, 0, nullptr, s);
  } else {
    launch_wide<double, double, W_ROWS>(m, P, 0, nullptr, s);
  }
  return true;
}

}  // namespace mtp
