// K6 (FP64 path) and K7: the dense reduced Hessian
//   K_hat = sum_i (Z_i^T Y_i + Y_u,i) + Sigma_u + (first-stage cost curvature)
// (Prop. 2.3, K_hat = Z^T K Z, summed over scenarios as the global reduction of
// §3.2 does with MPI_Allreduce), and its dense Cholesky factorization
// (§4: the Schur complement is factorized with dense LAPACK on the GPU).
//
// The scenario sum is part of the contraction: K runs over (scenario, row)
// pairs.  CTAs split that range into fixed groups of scenarios and write
// partial tiles; one pass then adds the groups in index order (deterministic).
// Only upper tiles (i <= j) are computed; the symmetric result is mirrored.
#include <atomic>

#include <cooperative_groups.h>

#include "dev.cuh"
#include "kernels.h"
#include "trsv.cuh"


namespace {

constexpr int TB = 64;   // output tile
constexpr int TK = 16;   // k chunk

// One 64 x 64 tile of A^T B over the rows [r0, r1) of the (rows x nu)
// matrices A, B (scenario-major storage makes the scenario sum one
// contraction over the concatenated rows); the tile goes to P (row-major).
// FP64-bound (98 % of the pipe's cycles), so no multiply-add is issued for
// nothing: a warp holds 32 x 16 of the tile, 4 x 4 per thread, and skips the
// products when that block lies below the diagonal or past n_u (its part of P
// is not written; nobody reads it).  With eight 8 x 64 strips, which can skip
// nothing: n_u = 299 12.1 -> 10.6 ms (64 scenarios), n_u = 129 660 -> 451 us
// (19), the assembly included.  `rot` varies which warps skip, so that the
// CTAs of an SM level out.
__device__ __forceinline__ void tile_tn64(long long r0, long long r1, int nu, int i0, int j0,
                                          const double *__restrict__ A, const double *__restrict__ B,
                                          double *P, double (*As)[TB], double (*Bs)[TB], int rot) {
  const int tid = threadIdx.x, lane = tid & 31, w = ((tid >> 5) & 4) | (((tid >> 5) + rot) & 3);
  const int m0 = 32 * (w >> 2) + 4 * (lane >> 2), n0 = 16 * (w & 3) + 4 * (lane & 3);  // the thread's 4 x 4
  const int wm = 32 * (w >> 2), wn = 16 * (w & 3);
  const bool skip = i0 + wm >= nu || j0 + wn >= nu || j0 + wn + 15 < i0 + wm;
  double acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
  for (long long k0 = r0; k0 < r1; k0 += TK) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int e = tid + q * 256, kk = e >> 6, cc = e & 63;
      const long long k = k0 + kk;
      As[kk][cc] = (k < r1 && i0 + cc < nu) ? A[k * nu + i0 + cc] : 0.0;
      Bs[kk][cc] = (k < r1 && j0 + cc < nu) ? B[k * nu + j0 + cc] : 0.0;
    }
    __syncthreads();
    if (!skip)
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      double av[4], bv[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) av[a] = As[kk][m0 + a];
#pragma unroll
      for (int b = 0; b < 4; ++b) bv[b] = Bs[kk][n0 + b];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = fma(av[a], bv[b], acc[a][b]);
    }
    __syncthreads();
  }
  if (skip) return;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) P[(m0 + a) * TB + n0 + b] = acc[a][b];
}

// partial[g][tile t][64*64] = A^T B on tile t over the rows [g*kc, (g+1)*kc)
__global__ void __launch_bounds__(256) k_gemm_tn64(long long krows, long long kc, int nu,
                                                   const double *__restrict__ A,
                                                   const double *__restrict__ B,
                                                   const int2 *__restrict__ tiles, double *partial) {
  __shared__ double As[TK][TB];
  __shared__ double Bs[TK][TB];
  const int t = blockIdx.x, g = blockIdx.y;
  const long long r0 = (long long)g * kc, r1 = min(krows, r0 + kc);
  tile_tn64(r0, r1, nu, tiles[t].x * TB, tiles[t].y * TB, A, B,
            partial + ((size_t)g * gridDim.x + t) * TB * TB, As, Bs, g);
}

// The same contraction for many independent instances in one persistent
// launch: every (instance, tile, scenario group) is a work item; CTAs take
// items from an atomic counter (items are sorted by decreasing length, so
// the long ones start first).  Each item writes the partial tile that the
// instance's own launch would write, so the result does not depend on which
// CTA ran it.
__global__ void __launch_bounds__(256) k_gemm_grouped(const GemmItem *__restrict__ items, int nitems,
                                                      int *counter) {
  __shared__ double As[TK][TB];
  __shared__ double Bs[TK][TB];
  __shared__ int w;
  for (;;) {
    if (threadIdx.x == 0) w = atomicAdd(counter, 1);
    __syncthreads();
    const int it = w;
    __syncthreads();
    if (it >= nitems) break;
    const GemmItem g = items[it];
    tile_tn64(g.r0, g.r1, g.nu, g.i0, g.j0, g.A, g.B, g.P, As, Bs, it);
  }
}

// K_hat[i][j] = K_hat[j][i] = sum_g partial + sum_s Yu[s][i][j] + diag  (i <= j)
__global__ void k_khat_assemble(int nu, int N, int ngroups, int ntiles, int nt1,
                                const double *__restrict__ partial, const int *__restrict__ tile_of,
                                const double *__restrict__ Yu, const double *__restrict__ diag,
                                double *Khat) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)nu * nu) return;
  const int i = (int)(t / nu), j = (int)(t % nu);
  if (i > j) return;
  const int ti = i / TB, tj = j / TB;
  const int tt = tile_of[ti * nt1 + tj];
  const double *p = partial + (size_t)tt * TB * TB + (i - ti * TB) * TB + (j - tj * TB);
  const size_t st = (size_t)ntiles * TB * TB;
  double v = 0.0;
  for (int g0 = 0; g0 < ngroups; g0 += 16) {  // added in order, the loads of 16 chunks in flight
    double a[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) a[q] = g0 + q < ngroups ? p[(g0 + q) * st] : 0.0;
#pragma unroll
    for (int q = 0; q < 16; ++q) v += a[q];
  }
  if (Yu)
    for (int s = 0; s < N; ++s) v += Yu[(size_t)s * nu * nu + (size_t)i * nu + j];
  if (diag && i == j) v += diag[i];
  Khat[(size_t)i * nu + j] = v;
  Khat[(size_t)j * nu + i] = v;
}

// F = Khat + delta (M + I) + tau I   (tau: shift of a preconditioner only)
__global__ void k_shift(int nu, const double *Khat, const double *M, double delta, double tau, double *F) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)nu * nu) return;
  const int i = (int)(t / nu), j = (int)(t % nu);
  double v = Khat[t];
  if (delta != 0.0) v += delta * (M[t] + (i == j ? 1.0 : 0.0));
  if (i == j) v += tau;
  F[t] = v;
}

// out[0] = max_i |A_ii|
__global__ void k_maxdiag(int n, const double *A, double *out) {
  double m = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) m = fmax(m, fabs(A[(size_t)i * n + i]));
  m = warp_max(m);
  __shared__ double sh[32];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r = fmax(r, sh[w]);
    out[0] = r;
  }
}

constexpr int CB = 32;  // Cholesky block
constexpr int CHOL_SMALL = 64;  // rows of K_hat of the small problems (ipm_internal.h) with 15 % generators

// factor the CB x CB diagonal block at (k0, k0) in place (lower), unblocked

// Right-looking Cholesky of the nb x nb block a (lower part, in shared
// memory) by the calling CTA: thread 0 takes each pivot's reciprocal square
// root, then warps 0-3 scale the column and update the trailing columns
// (warp w: columns j = w mod 4; lane = row; column entries by shuffles).  A
// non-positive or non-finite pivot raises FLAG_NOT_PD and is replaced by 1.
// For K_hat of at most CHOL_SMALL rows, the small problems, whose whole solves
// keep these operations (ipm_internal.h).
__device__ void potrf_plain(int nb, int *flags, double (*a)[CB + 1], double *rs_sh) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int k = 0; k < nb; ++k) {
    if (tid == 0) {
      double d = a[k][k];
      if (!(d > 0.0) || !isfinite(d)) {
        flags[FLAG_NOT_PD] = 1;
        d = 1.0;
      }
      const double rs = rsqrt_newton(d);
      *rs_sh = rs;
      a[k][k] = d * rs;
    }
    __syncthreads();
    double lik = 0.0;
    if (warp < 4) {
      lik = (lane > k && lane < nb) ? a[lane][k] * *rs_sh : 0.0;
      for (int j = k + 1 + ((warp - (k + 1)) & 3); j < nb; j += 4) {
        const double ljk = __shfl_sync(0xffffffffu, lik, j);
        if (lane >= j && lane < nb) a[lane][j] -= lik * ljk;
      }
    }
    __syncthreads();
    // column k is read by no later step: written after the barrier
    if (warp == 0 && lane > k && lane < nb) a[lane][k] = lik;
  }
  __syncthreads();
}

// The same as L D L^T with the square roots taken for all columns at the end:
// only a reciprocal is on the chain from pivot to pivot, formed for the next
// column, which is updated first, under the others' updates; one barrier per
// column.  Latency-bound; the whole factorization at n_u = 299 412 -> 391 us,
// 899 1,275 -> 1,215.
__device__ void potrf_ldl(int nb, int *flags, double (*a)[CB + 1], double *rs_sh) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const auto pivot = [&](int k) {
    double d = a[k][k];
    if (!(d > 0.0) || !isfinite(d)) {
      flags[FLAG_NOT_PD] = 1;
      a[k][k] = d = 1.0;
    }
    rs_sh[k & 1] = rcp_newton(d);
  };
  if (tid == 0) pivot(0);
  __syncthreads();
  for (int k = 0; k < nb; ++k) {
    if (warp < 4) {
      const double v = lane > k && lane < nb ? a[lane][k] : 0.0;  // column k: written by no later step
      const double l = v * rs_sh[k & 1];
      for (int j = k + 1 + ((warp - (k + 1)) & 3); j < nb; j += 4) {
        const double vj = __shfl_sync(0xffffffffu, v, j);
        if (lane >= j && lane < nb) a[lane][j] -= l * vj;
        if (j == k + 1 && lane == j) pivot(j);
        __syncwarp();
      }
    }
    __syncthreads();
  }
  double *rs = rs_sh + 2;  // 1 / sqrt(d_k)
  if (tid < nb) rs[tid] = rsqrt_newton(a[tid][tid]);
  __syncthreads();
  for (int e = tid; e < nb * nb; e += blockDim.x) {
    const int i = e / nb, j = e % nb;
    if (j <= i) a[i][j] *= rs[j];
  }
  __syncthreads();
}

// (rs_sh: 2 + CB doubles)
template <bool LDL>
__device__ __forceinline__ void potrf_block(int nb, int *flags, double (*a)[CB + 1], double *rs_sh) {
  if (LDL) potrf_ldl(nb, flags, a, rs_sh);
  else potrf_plain(nb, flags, a, rs_sh);
}

// Load, factor and store the diagonal block at (k0, k0) (upper part of the
// block set to zero).
template <bool LDL>
__device__ void potrf_tile(int n, int k0, double *A, int *flags, double (*a)[CB + 1], double *rs_sh) {
  const int nb = min(CB, n - k0), tid = threadIdx.x;
  for (int e = tid; e < nb * nb; e += blockDim.x) a[e / nb][e % nb] = A[(size_t)(k0 + e / nb) * n + k0 + e % nb];
  __syncthreads();
  potrf_block<LDL>(nb, flags, a, rs_sh);
  for (int e = tid; e < nb * nb; e += blockDim.x) {
    const int i = e / nb, j = e % nb;
    A[(size_t)(k0 + i) * n + k0 + j] = (j <= i) ? a[i][j] : 0.0;
  }
  __syncthreads();
}

template <bool LDL>
__global__ void k_potrf_diag(int n, int k0, double *A, int *flags) {
  __shared__ double a[CB][CB + 1];
  __shared__ double rs_sh[2 + CB];
  potrf_tile<LDL>(n, k0, A, flags, a, rs_sh);
}

// rows below the diagonal block: L_ik = A_ik L_kk^{-T}
__global__ void k_trsm_panel(int n, int k0, double *A) {
  __shared__ double Lk[CB][CB + 1];
  const int nb = min(CB, n - k0), tid = threadIdx.x;
  for (int e = tid; e < nb * nb; e += blockDim.x) Lk[e / nb][e % nb] = A[(size_t)(k0 + e / nb) * n + k0 + e % nb];
  __syncthreads();
  const int i = k0 + nb + blockIdx.x * blockDim.x + tid;
  if (i >= n) return;
  double x[CB];
  for (int j = 0; j < nb; ++j) {
    double v = A[(size_t)i * n + k0 + j];
    for (int t = 0; t < j; ++t) v -= x[t] * Lk[j][t];
    x[j] = v / Lk[j][j];
  }
  for (int j = 0; j < nb; ++j) A[(size_t)i * n + k0 + j] = x[j];
}

// trailing update of the lower part: A_ij -= sum_t L_it L_jt (tiles CB x CB)
__global__ void k_syrk_trail(int n, int k0, double *A) {
  const int nb = min(CB, n - k0);
  const int r0 = k0 + nb;
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj > bi) return;
  __shared__ double Li[CB][CB + 1], Lj[CB][CB + 1];
  const int tid = threadIdx.x;
  const int i0 = r0 + bi * CB, j0 = r0 + bj * CB;
  for (int e = tid; e < CB * nb; e += blockDim.x) {
    const int rr = e / nb, t = e % nb;
    Li[rr][t] = (i0 + rr < n) ? A[(size_t)(i0 + rr) * n + k0 + t] : 0.0;
    Lj[rr][t] = (j0 + rr < n) ? A[(size_t)(j0 + rr) * n + k0 + t] : 0.0;
  }
  __syncthreads();
  for (int e = tid; e < CB * CB; e += blockDim.x) {
    const int ii = e / CB, jj = e % CB, i = i0 + ii, j = j0 + jj;
    if (i >= n || j >= n || j > i) continue;
    double v = 0.0;
    for (int t = 0; t < nb; ++t) v += Li[ii][t] * Lj[jj][t];
    A[(size_t)i * n + j] -= v;
  }
}

// The same blocked factorization as one cooperative launch (grid-wide
// barriers between the steps instead of three launches per block column).
// Per block column k0 (32 wide): (a) every CTA with panel rows loads L_kk and
// solves its rows x L_kk^T = a (a warp per row, lane = column, shuffles; the
// multipliers L_jt / L_tt are formed once per CTA so each step is one
// shuffle and one multiply-add); (b) the trailing matrix is updated: CTA 0
// forms the next diagonal block in one pass straight into shared memory and
// factors it right away, the other lower 16 x 16 tiles go round-robin to
// the remaining CTAs.
constexpr int CT = 16;  // trailing-update tile

__device__ void syrk_tile16(int n, int k0, int nb, int i0, int j0, double *A, double (*Li)[CB + 1],
                            double (*Lj)[CB + 1]) {
  const int tid = threadIdx.x;
  __syncthreads();
  for (int e = tid; e < CT * nb; e += blockDim.x) {
    const int rr = e / nb, t = e % nb;
    Li[rr][t] = (i0 + rr < n) ? A[(size_t)(i0 + rr) * n + k0 + t] : 0.0;
    Lj[rr][t] = (j0 + rr < n) ? A[(size_t)(j0 + rr) * n + k0 + t] : 0.0;
  }
  __syncthreads();
  if (tid < CT * CT) {
    const int ii = tid / CT, jj = tid % CT, i = i0 + ii, j = j0 + jj;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
    int t = 0;
    for (; t + 4 <= nb; t += 4) {
      s0 = fma(Li[ii][t], Lj[jj][t], s0);
      s1 = fma(Li[ii][t + 1], Lj[jj][t + 1], s1);
      s2 = fma(Li[ii][t + 2], Lj[jj][t + 2], s2);
      s3 = fma(Li[ii][t + 3], Lj[jj][t + 3], s3);
    }
    for (; t < nb; ++t) s0 = fma(Li[ii][t], Lj[jj][t], s0);
    if (i < n && j < n && j <= i) A[(size_t)i * n + j] -= (s0 + s1) + (s2 + s3);
  }
}

template <bool LDL>
__global__ void __launch_bounds__(256) k_chol_coop(int n, double *A, int *flags) {
  cooperative_groups::grid_group grid = cooperative_groups::this_grid();
  __shared__ double a[CB][CB + 1], b2[CB][CB + 1];
  __shared__ double rinv[CB], rs_sh[2 + CB];
  const int G = gridDim.x, bk = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (bk == 0) potrf_tile<LDL>(n, 0, A, flags, a, rs_sh);
  grid.sync();
  for (int k0 = 0; k0 < n; k0 += CB) {
    const int nb = min(CB, n - k0), r0 = k0 + nb, rest = n - r0;
    if (rest <= 0) break;
    // (a) panel rows
    if (r0 + bk * 8 < n) {
      for (int e = tid; e < CB * CB; e += blockDim.x) {
        const int rr = e / CB, cc = e % CB;
        a[rr][cc] = (rr < nb && cc <= rr) ? A[(size_t)(k0 + rr) * n + k0 + cc] : 0.0;
      }
      __syncthreads();
      if (tid < CB) rinv[tid] = tid < nb ? 1.0 / a[tid][tid] : 0.0;
      __syncthreads();
      for (int e = tid; e < CB * CB; e += blockDim.x) {
        const int rr = e / CB, cc = e % CB;
        b2[rr][cc] = cc < rr ? a[rr][cc] * rinv[cc] : 0.0;  // L_jt / L_tt (j = rr, t = cc)
      }
      __syncthreads();
      for (int i = r0 + bk * 8 + warp; i < n; i += G * 8) {
        double v = lane < nb ? A[(size_t)i * n + k0 + lane] : 0.0;
        for (int t = 0; t < nb; ++t) {
          const double vt = __shfl_sync(0xffffffffu, v, t);
          if (lane > t) v = fma(-b2[lane][t], vt, v);
        }
        if (lane < nb) A[(size_t)i * n + k0 + lane] = v * rinv[lane];
      }
    }
    grid.sync();
    // (b) trailing update; tiles with bi, bj < 2 form the next diagonal block
    const int nt = (rest + CT - 1) / CT;
    const int ndt = nt >= 2 ? 3 : 1;
    const int ntl = nt * (nt + 1) / 2 - ndt;
    if (bk == 0) {
      if (G == 1)
        for (int t = 0; t < ntl; ++t) {
          int bi = 2, rem = t;
          while (rem > bi) { rem -= bi + 1; ++bi; }
          syrk_tile16(n, k0, nb, r0 + bi * CT, r0 + rem * CT, A, a, b2);
        }
      // the next diagonal block, A_dd - L_d L_d^T, straight into shared
      // memory (one pass over its lower part), then factored and stored
      const int nb2 = min(CB, rest);
      __syncthreads();
      for (int e = tid; e < CB * nb; e += blockDim.x) {
        const int rr = e / nb, t = e % nb;
        b2[rr][t] = rr < nb2 ? A[(size_t)(r0 + rr) * n + k0 + t] : 0.0;
      }
      __syncthreads();
      for (int e = tid; e < nb2 * nb2; e += blockDim.x) {
        const int i = e / nb2, j = e % nb2;
        if (j > i) continue;
        double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
        int t = 0;
        for (; t + 4 <= nb; t += 4) {
          s0 = fma(b2[i][t], b2[j][t], s0);
          s1 = fma(b2[i][t + 1], b2[j][t + 1], s1);
          s2 = fma(b2[i][t + 2], b2[j][t + 2], s2);
          s3 = fma(b2[i][t + 3], b2[j][t + 3], s3);
        }
        for (; t < nb; ++t) s0 = fma(b2[i][t], b2[j][t], s0);
        a[i][j] = A[(size_t)(r0 + i) * n + r0 + j] - ((s0 + s1) + (s2 + s3));
      }
      __syncthreads();
      potrf_block<LDL>(nb2, flags, a, rs_sh);
      for (int e = tid; e < nb2 * nb2; e += blockDim.x) {
        const int i = e / nb2, j = e % nb2;
        A[(size_t)(r0 + i) * n + r0 + j] = (j <= i) ? a[i][j] : 0.0;
      }
      __syncthreads();
    } else {
      for (int t = bk - 1; t < ntl; t += G - 1) {
        // t-th lower tile in rows bi >= 2: row bi holds bi + 1 tiles
        int bi = 2, rem = t;
        while (rem > bi) { rem -= bi + 1; ++bi; }
        syrk_tile16(n, k0, nb, r0 + bi * CT, r0 + rem * CT, A, a, b2);
      }
    }
    grid.sync();
  }
}

// Inverses of the NB x NB diagonal blocks of L (row-major, lower, ld n), one
// CTA per block, for the triangular sweeps of k_chol_solve: block b at
// b NB^2, (i, k) at i NB + k, identity past n.  L = L' diag(l_kk) with L'
// unit lower, so L^{-1} = diag(1 / l_kk) L'^{-1}.
template <int NB>
__global__ void __launch_bounds__(128) k_chol_inverse(int n, const double *__restrict__ L, double *inv) {
  extern __shared__ double smi[];
  double(*D)[NB + 1] = reinterpret_cast<double(*)[NB + 1]>(smi), (*X)[NB + 1] = D + NB;
  __shared__ double rk[NB];
  const int tid = threadIdx.x, b0 = blockIdx.x * NB;
  if (tid < NB) rk[tid] = b0 + tid < n ? 1.0 / L[(size_t)(b0 + tid) * n + b0 + tid] : 1.0;
  __syncthreads();
  for (int e = tid; e < NB * NB; e += 128) {
    const int i = e / NB, k = e % NB;
    D[i][k] = k < i && b0 + i < n ? L[(size_t)(b0 + i) * n + b0 + k] * rk[k] : 0.0;
    X[i][k] = i == k ? 1.0 : 0.0;
  }
  __syncthreads();
  trsv::unit_inverse(D, X, min(NB, n - b0), false, tid, 128);
  for (int e = tid; e < NB * NB; e += 128) {
    const int i = e / NB, k = e % NB;
    inv[(size_t)blockIdx.x * NB * NB + e] = X[i][k] * rk[i];
  }
}

// Solve L L^T x = b in place: one CTA, or (MULTI) a cluster of C CTAs.  The
// chain of the blocks bounds it, and the factor's bytes through the cluster's
// SMs on the larger ones.  Against one CTA with 32 x 32 diagonal blocks
// solved step by step: n_u = 299 118 -> 45 us, 1,999 1,820 -> 290 us.
template <int TH, int NB, bool MULTI>
__global__ void __launch_bounds__(TH) k_chol_solve(int n, const double *__restrict__ L, const double *__restrict__ inv,
                                                   double *b, int C) {
  extern __shared__ double smc[];
  const int rank = MULTI ? (int)blockIdx.x : 0;
  const auto ldx = [&](int i) { return MULTI ? __ldcg(b + i) : b[i]; };
  const auto stx = [&](int i, double y) {
    if (MULTI) __stcg(b + i, y);
    else b[i] = y;
  };
  if (MULTI) {  // every CTA has started before its shared memory is written
    trsv::cluster_arrive();
    trsv::cluster_wait();
  }
  trsv::sweep<TH, NB, MULTI>(L, (size_t)n, n, true, false, inv, NB * NB, C, rank, smc, ldx, stx);
  trsv::sweep<TH, NB, MULTI>(L, (size_t)n, n, false, true, inv, NB * NB, C, rank, smc, ldx, stx);
}

// The same for few rows, one CTA with the vector in shared memory: the
// diagonal blocks step by step by one warp (lane = row, reciprocal pivots
// formed by all lanes at once), the rows past a block by a thread each with
// four partial sums: the order of operations of the small problems' whole
// solves (ipm_internal.h).  n_u = 35 14 us and 63 22, against 7 and 7 by the
// inverses, which take 12 to form once per factorization.
__global__ void __launch_bounds__(128) k_chol_solve_small(int n, const double *__restrict__ L, double *b) {
  __shared__ double x[CHOL_SMALL], blk[32][33];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < n) x[tid] = b[tid];
  __syncthreads();
  const auto sweep = [&](bool up) {
    for (int s = 0; s < n; s += 32) {
      const int kb = up ? (n - 1) / 32 * 32 - s : s, w = min(32, n - kb);
      for (int e = tid; e < 32 * w; e += 128) {
        const int r = e >> 5, c = e & 31;
        blk[r][c] = c <= r ? L[(size_t)(kb + r) * n + kb + c] : 0.0;
      }
      __syncthreads();
      if (warp == 0) {
        const double ri = lane < w ? 1.0 / blk[lane][lane] : 0.0;
        double v = lane < w ? x[kb + lane] : 0.0;
        for (int q = 0; q < w; ++q) {
          const int k = up ? w - 1 - q : q;
          if (lane == k) v *= ri;
          const double xk = __shfl_sync(0xffffffffu, v, k);
          if (up ? lane < k : lane > k && lane < w) v -= (up ? blk[k][lane] : blk[lane][k]) * xk;
        }
        if (lane < w) x[kb + lane] = v;
      }
      __syncthreads();
      if (up ? tid < kb : tid >= kb + w && tid < n) {
        const double *p = up ? L + (size_t)kb * n + tid : L + (size_t)tid * n + kb;
        const size_t st = up ? n : 1;
        double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
        int j = 0;
        for (; j + 4 <= w; j += 4) {
          s0 = fma(p[j * st], x[kb + j], s0);
          s1 = fma(p[(j + 1) * st], x[kb + j + 1], s1);
          s2 = fma(p[(j + 2) * st], x[kb + j + 2], s2);
          s3 = fma(p[(j + 3) * st], x[kb + j + 3], s3);
        }
        for (; j < w; ++j) s0 = fma(p[j * st], x[kb + j], s0);
        x[tid] -= (s0 + s1) + (s2 + s3);
      }
      __syncthreads();
    }
  };
  sweep(false);
  sweep(true);
  if (tid < n) b[tid] = x[tid];
}

// diagonal blocks of 64 rows from here on
constexpr int CHOL_NB64 = 512;

template <int NB>
void chol_inverse(int n, const double *L, double *inv, cudaStream_t st) {
  static const bool cap = raise_smem_cap(k_chol_inverse<NB>);
  (void)cap;
  k_chol_inverse<NB><<<(n + NB - 1) / NB, 128, 2 * NB * (NB + 1) * sizeof(double), st>>>(n, L, inv);
  ipm_count_launch();
}

template <int TH, int NB, int C>
void chol_solve_cluster(int n, const double *L, const double *inv, double *b, cudaStream_t st) {
  static const bool cap = raise_smem_cap(k_chol_solve<TH, NB, true>);
  (void)cap;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C);
  cfg.blockDim = dim3(TH);
  cfg.dynamicSmemBytes = trsv::smem_doubles<TH, NB>(((n + NB - 1) / NB + C - 1) / C) * sizeof(double);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_chol_solve<TH, NB, true>, n, L, inv, b, C); ipm_count_launch();
}

template <int TH>
void chol_solve_single(int n, const double *L, const double *inv, double *b, cudaStream_t st) {
  static const bool cap = raise_smem_cap(k_chol_solve<TH, 32, false>);
  (void)cap;
  k_chol_solve<TH, 32, false><<<1, TH, trsv::smem_doubles<TH, 32>((n + 31) / 32) * sizeof(double), st>>>(n, L, inv, b,
                                                                                                     1);
  ipm_count_launch();
}

}  // namespace

void launch_gemm_tn64(long long krows, long long kc, int nu, int ngroups, const double *A, const double *B,
                      const int2 *tiles, int ntiles, double *partial, cudaStream_t st) {
  dim3 grid(ntiles, ngroups);
  k_gemm_tn64<<<grid, 256, 0, st>>>(krows, kc, nu, A, B, tiles, partial); ipm_count_launch();
}
void launch_gemm_grouped(const GemmItem *items, int nitems, int *counter, cudaStream_t st) {
  static const int ctas = [] {
    int per_sm = 0, dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_gemm_grouped, 256, 0) != cudaSuccess || per_sm < 1)
      per_sm = 1;
    return sms * per_sm;
  }();
  cudaMemsetAsync(counter, 0, sizeof(int), st);
  const int grid = nitems < ctas ? nitems : ctas;
  if (grid > 0) {
    k_gemm_grouped<<<grid, 256, 0, st>>>(items, nitems, counter);
    ipm_count_launch();
  }
}

void launch_khat_assemble(int nu, int N, int ngroups, int ntiles, int nt1, const double *partial,
                          const int *tile_of, const double *Yu, const double *diag, double *Khat,
                          cudaStream_t st) {
  long long tot = (long long)nu * nu;
  k_khat_assemble<<<(int)((tot + 255) / 256), 256, 0, st>>>(nu, N, ngroups, ntiles, nt1, partial,
                                                             tile_of, Yu, diag, Khat); ipm_count_launch();
}
void launch_shift(int nu, const double *Khat, const double *M, double delta, double tau, double *F,
                  cudaStream_t st) {
  long long tot = (long long)nu * nu;
  k_shift<<<(int)((tot + 255) / 256), 256, 0, st>>>(nu, Khat, M, delta, tau, F); ipm_count_launch();
}
void launch_maxdiag(int n, const double *A, double *out, cudaStream_t st) {
  k_maxdiag<<<1, 256, 0, st>>>(n, A, out); ipm_count_launch();
}
template <bool LDL>
static void cholesky(int n, double *A, int *flags, cudaStream_t st) {
  // one cooperative launch when the device allows it (all CTAs resident)
  static const int coop_ctas = [] {
    int dev = 0, ok = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&ok, cudaDevAttrCooperativeLaunch, dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (!ok || cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_chol_coop<LDL>, 256, 0) != cudaSuccess || per < 1)
      return 0;
    return sms;  // one CTA per SM
  }();
  if (coop_ctas > 0) {
    const int nt = (n + CT - 1) / CT;
    int G = 1 + nt * (nt + 1) / 2;  // CTA 0 plus one per lower tile of the first trailing update
    G = G < coop_ctas ? G : coop_ctas;
    if (G < 1) G = 1;
    void *args[] = {(void *)&n, (void *)&A, (void *)&flags};
    if (cudaLaunchCooperativeKernel((const void *)k_chol_coop<LDL>, dim3(G), dim3(256), args, 0, st) == cudaSuccess) {
      ipm_count_launch();
      return;
    }
    cudaGetLastError();
  }
  for (int k0 = 0; k0 < n; k0 += CB) {
    k_potrf_diag<LDL><<<1, 256, 0, st>>>(n, k0, A, flags); ipm_count_launch();
    const int nb = n - k0 < CB ? n - k0 : CB;
    const int rest = n - k0 - nb;
    if (rest > 0) {
      k_trsm_panel<<<(rest + 127) / 128, 128, 0, st>>>(n, k0, A); ipm_count_launch();
      const int nt = (rest + CB - 1) / CB;
      k_syrk_trail<<<dim3(nt, nt), 256, 0, st>>>(n, k0, A); ipm_count_launch();
    }
  }
}
void launch_cholesky(int n, double *A, int *flags, cudaStream_t st) {
  if (n <= CHOL_SMALL) cholesky<false>(n, A, flags, st);
  else cholesky<true>(n, A, flags, st);
}
size_t chol_inverse_doubles(int n) { return (size_t)((n + 63) / 64) * 64 * 64; }
void launch_chol_inverse(int n, const double *L, double *inv, cudaStream_t st) {
  if (n <= CHOL_SMALL) return;
  if (n < CHOL_NB64) chol_inverse<32>(n, L, inv, st);
  else chol_inverse<64>(n, L, inv, st);
}
// One SM applies a 32 x 32 tile in ~0.3 us (its FP64 units), so from a few
// blocks on the tiles are dealt to a cluster, although its barrier costs ten
// of a CTA's.
void launch_chol_solve(int n, const double *L, const double *inv, double *b, cudaStream_t st) {
  if (n <= CHOL_SMALL) {
    k_chol_solve_small<<<1, 128, 0, st>>>(n, L, b);
    ipm_count_launch();
  } else if (n <= 128) chol_solve_single<128>(n, L, inv, b, st);
  else if (n < CHOL_NB64) chol_solve_cluster<256, 32, 4>(n, L, inv, b, st);
  else if (n <= 16384) chol_solve_cluster<512, 64, 8>(n, L, inv, b, st);
  else chol_solve_cluster<256, 64, 8>(n, L, inv, b, st);  // 256 accumulators per block and CTA
}
