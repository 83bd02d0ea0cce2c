// Single-vector solves G_x v = b and G_x^T v = b with the static-pivot LU of
// every scenario (in place, position order).
//
// Paper: §3.2, G_x^{-1} b = Q U^{-1} L^{-1} P b and its transpose: the reduced
// right-hand side, the recovery of p_x and p_y, and every product with the
// exact reduced operator of the mixed path's conjugate gradients.
//
// A solve is a chain: the sparse rows level by level (about 20 levels each
// way), the dense trailing block between them.  Bound by the latency of that
// chain on the small networks, by the factor's bytes (the trailing block,
// 25 MB per scenario at 10,000 buses) and the FP64 units on the large ones.
//  * Sparse rows: the work of a level comes in units, one warp and four
//    products per lane each, 1 to 32 lanes to a row by its length
//    (symbolic.cpp; a warp-wide FP64 operation takes ~19 cycles of an SM
//    whatever its lanes hold, so a row's products go to few lanes).  The
//    schedule does not depend on the data, so a warp fetches its next unit's
//    products two units ahead and their factor values one ahead, across the
//    level barriers; a level then costs the operands' loads, a few FP64
//    operations and the barrier instead of four dependent loads.
//  * Trailing block, by 64 x 64 blocks (32 x 32 up to 400 states): the
//    inverses of the diagonal blocks are formed once per factorization, so a
//    block of the solution is two small products instead of as many dependent
//    steps as it has rows, and the rest of the block column is applied behind
//    the chain.
//  * Large networks: a cluster of 4 or 8 CTAs per scenario shares both
//    (hardware cluster barriers), the blocks dealt in turn to the CTAs; the
//    CTA holding the next block updates and solves it first, and everybody
//    updates the other blocks between arriving at the barrier and waiting.
//  * Small problems (S.ordered): the same units with 4 or 8 lanes per row, the
//    trailing block by substitution, so that their sums keep one order.
//
// Measured, one solve (before: one CTA per scenario, or 54 launches through
// the large blocks, a row's loads issued in turn and 64 steps per diagonal
// block): 1,000 buses x 64 scenarios 280-355 -> 91-106 us, 3,000 x 10 1,090 ->
// 235 us, 10,000 x 32 4,660 -> 700 us.
#include "dev.cuh"
#include "kernels.h"
#include "trsv.cuh"

namespace {

// Rows of a diagonal block: 64 in the large trailing blocks (half the steps
// of the chain), 32 in the others (a quarter of the inverses' FP64 work,
// which is what counts when a factorization serves only a few solves).
constexpr int NB_BIG = 64, NB_SMALL = 32;

// Inverses of the diagonal blocks of the trailing block's L (unit lower) and
// U, [N][blocks][2][NB * NB], (i, k) at k NB + i; rows and columns past nd
// are those of the identity.  One CTA per block, half of its threads for
// either.  U = U' diag(u_kk) with U' unit upper, so U^{-1} = diag(1 / u_kk)
// U'^{-1}.  Bound by the FP64 units: 17 us at 1,000 buses x 64 scenarios (86
// with blocks of 64 rows), 226 us at 10,000 x 32.
template <int NB>
__global__ void __launch_bounds__(256) k_diag_inverse(DevSym S, const double *__restrict__ LU,
                                                      const double *__restrict__ rd) {
  extern __shared__ double smd[];
  double(*D)[NB + 1] = reinterpret_cast<double(*)[NB + 1]>(smd);
  double(*X)[NB + 1] = D + NB, (*Y)[NB + 1] = X + NB;
  __shared__ double rk[NB];
  const int sc = blockIdx.y, b = blockIdx.x, tid = threadIdx.x, nd = S.nd, b0 = b * NB;
  const double *A = LU + (size_t)sc * S.nnzLU + S.dense_base;
  if (tid < NB) rk[tid] = b0 + tid < nd ? rd[(size_t)sc * S.nx + S.t0 + b0 + tid] : 1.0;
  __syncthreads();
  for (int e = tid; e < NB * NB; e += blockDim.x) {
    const int i = e % NB, k = e / NB;
    const double a = b0 + i < nd && b0 + k < nd ? A[(size_t)(b0 + k) * nd + b0 + i] : 0.0;
    D[i][k] = i < k ? a * rk[k] : a;
    X[i][k] = Y[i][k] = i == k ? 1.0 : 0.0;
  }
  __syncthreads();
  const int half = tid >> 7;
  trsv::unit_inverse(D, half ? Y : X, min(NB, nd - b0), half != 0, tid & 127, 128);
  double *out = S.dinv + ((size_t)sc * gridDim.x + b) * 2 * NB * NB;
  for (int e = tid; e < NB * NB; e += blockDim.x) {
    const int i = e % NB, k = e / NB;
    out[e] = X[i][k];
    out[NB * NB + e] = Y[i][k] * rk[i];
  }
}

// The trailing block of a small network (S.ordered), T = L or U^T going
// down, U or L^T going up, on x (the block's entries): 32 x 32 diagonal
// blocks step by step by one warp (lane = row; where T's diagonal is the
// pivots, their reciprocals are in the block's columns), the rows past a
// block by a thread each with four partial sums.  Bound by the chain; a solve
// at 120 buses x 17 takes 31 us, by the diagonal blocks' inverses 24 and 7 to
// form them once per factorization.
template <int TH>
__device__ void dense_small(const double *__restrict__ D, const double *__restrict__ r, int nd, bool trans, bool up,
                            double *x, double (*blk)[33]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool scale = trans != up;  // U^T going down, U going up
  const size_t si = trans ? nd : 1, sk = trans ? 1 : nd;  // T(i, k) = D[i si + k sk]
  for (int s = 0; s < nd; s += 32) {
    const int kb = up ? (nd - 1) / 32 * 32 - s : s, w = min(32, nd - kb);
    for (int e = tid; e < 32 * w; e += TH) {
      const int i = e >> 5, k = e & 31;
      double t = 0.0;
      if (up ? k > i && k < w : k < i) t = D[(kb + i) * si + (kb + k) * sk] * (scale ? r[kb + k] : 1.0);
      blk[i][k] = t;
    }
    __syncthreads();
    if (warp == 0) {
      double v = lane < w ? x[kb + lane] : 0.0;
      for (int q = 0; q < w; ++q) {
        const int k = up ? w - 1 - q : q;
        const double xk = __shfl_sync(0xffffffffu, v, k);
        if (up ? lane < k : lane > k && lane < w) v = fma(-blk[lane][k], xk, v);
      }
      if (lane < w) x[kb + lane] = scale ? v * r[kb + lane] : v;
    }
    __syncthreads();
    for (int i = up ? tid : kb + w + tid; i < (up ? kb : nd); i += TH) {
      const double *p = D + i * si + kb * sk;
      double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
      int j = 0;
      for (; j + 4 <= w; j += 4) {
        s0 = fma(p[j * sk], x[kb + j], s0);
        s1 = fma(p[(j + 1) * sk], x[kb + j + 1], s1);
        s2 = fma(p[(j + 2) * sk], x[kb + j + 2], s2);
        s3 = fma(p[(j + 3) * sk], x[kb + j + 3], s3);
      }
      for (; j < w; ++j) s0 = fma(p[j * sk], x[kb + j], s0);
      x[i] -= (s0 + s1) + (s2 + s3);
    }
    __syncthreads();
  }
}

// Vector b of v ([N * vps][n_x]) belongs to scenario b / vps.  MULTI: a
// cluster of C CTAs per vector, the vector in global memory (read and
// written past L1); else one CTA per vector, the vector in shared memory
// when it fits (in_smem).  ORDERED (small networks, the vector in shared
// memory): the products of a lane one after the other, the lanes joined from
// the widest distance down, the trailing block by dense_small.
template <int TH, int NB, bool MULTI, bool ORDERED = false>
__global__ void __launch_bounds__(TH, MULTI && TH == 512 ? 2 : 1) k_solve1(DevSym S, const double *__restrict__ LU, const double *__restrict__ rd,
                                               double *v, int trans, int vps, int C, int in_smem) {
  extern __shared__ double sm1[];
  constexpr int NW = TH / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int vec = MULTI ? blockIdx.x / C : blockIdx.x, rank = MULTI ? blockIdx.x % C : 0;
  const int sc = vec / vps, nx = S.nx, t0 = S.t0, nd = S.nd, nblk = (nd + NB - 1) / NB;
  const double *A = LU + (size_t)sc * S.nnzLU, *r = rd + (size_t)sc * nx;
  __shared__ double blk[ORDERED ? 32 : 1][33];
  double *xsm = sm1 + (ORDERED ? 0 : trsv::smem_doubles<TH, NB>((nblk + C - 1) / C));
  double *vs = v + (size_t)vec * nx, *x = !MULTI && in_smem ? xsm : vs;
  const auto ldx = [&](int i) { return MULTI ? __ldcg(x + i) : x[i]; };
  const auto stx = [&](int i, double y) {
    if (MULTI) __stcg(x + i, y);
    else x[i] = y;
  };
  const auto sync_all = [] {
    if (MULTI) {
      __syncwarp();
      trsv::cluster_arrive();
      trsv::cluster_wait();
    } else {
      __syncthreads();
    }
  };
  if (!MULTI && in_smem) {
    for (int i = tid; i < nx; i += TH) x[i] = vs[i];
    __syncthreads();
  }

  // sparse rows of levels [0, L), units lp[l] .. lp[l + 1): x[row] -= sum of
  // the row's products, then the reciprocal pivot (scale)
  const auto sweep = [&](const int *__restrict__ lp, int L, bool scale) {
    const auto advance = [&](int &l, int &u, bool first) {
      if (!first) u += C * NW;
      while (first || u >= lp[l + 1]) {
        first = false;
        if (++l >= L) return;
        u = lp[l] + rank * NW + warp;
      }
    };
    struct Unit {
      int2 p[SWP];  // {column, slot}, slot -1: none
      int rc;       // row | code << 26, -1: none
    };
    const int2 *__restrict__ items = S.sw_item + (trans ? S.sw_items : 0);
    const auto fetch = [&](int l, int u) {
      Unit q;
#pragma unroll
      for (int h = 0; h < SWP; ++h) q.p[h] = l < L ? items[((size_t)u * SWP + h) * 32 + lane] : make_int2(0, -1);
      q.rc = l < L ? S.sw_row[(size_t)u * 32 + lane] : -1;
      return q;
    };
    const auto value = [&](int2 p) { return p.y >= 0 ? A[p.y] : 0.0; };
    const auto operand = [&](int2 p) { return p.y >= 0 ? ldx(p.x) : 0.0; };
    const auto pivot = [&](int rc) { return scale && rc >= 0 ? r[rc & 0x3ffffff] : 1.0; };
    int l0 = -1, u0 = 0;
    advance(l0, u0, true);
    int l1 = l0, u1 = u0;
    if (l0 < L) advance(l1, u1, false);
    Unit q1;  // the next unit's products
    int2 p0[SWP];
    double a0[SWP];
    int rc;
    double rr;
    {
      const Unit q0 = fetch(l0, u0);
      q1 = fetch(l1, u1);
      rc = q0.rc;
      rr = pivot(rc);
#pragma unroll
      for (int h = 0; h < SWP; ++h) {
        p0[h] = q0.p[h];
        a0[h] = value(p0[h]);
      }
    }
    for (int k = 0; k < l0; ++k) sync_all();
    while (l0 < L) {
      int l2 = l1, u2 = u1;
      if (l1 < L) advance(l2, u2, false);
      const Unit q2 = fetch(l2, u2);
      double b0[SWP];
#pragma unroll
      for (int h = 0; h < SWP; ++h) b0[h] = value(q1.p[h]);
      const double rn = pivot(q1.rc);
      // lane 0 holds a row in every unit, so its code is the unit's
      const int code = __shfl_sync(0xffffffffu, rc, 0) >> 26, g = 1 << (code & 7);
      const bool lead = (lane & (g - 1)) == 0 && rc >= 0;
      double x0[SWP];
#pragma unroll
      for (int h = 0; h < SWP; ++h) x0[h] = operand(p0[h]);
      const double xr = lead ? ldx(rc & 0x3ffffff) : 0.0;
      double part = 0.0;
      if (ORDERED) {
#pragma unroll
        for (int h = 0; h < SWP; ++h) part = fma(a0[h], x0[h], part);
      } else {
        part = fma(a0[0], x0[0], a0[1] * x0[1]) + fma(a0[2], x0[2], a0[3] * x0[3]);
      }
      if (code & 8) {  // the products left over
        const int2 ex = S.sw_extra[u0];
        for (int k = 0; k < ex.y; ++k) {
#pragma unroll
          for (int h = 0; h < SWP; ++h) {
            const int2 p = items[((size_t)(ex.x + k) * SWP + h) * 32 + lane];
            part = fma(value(p), operand(p), part);
          }
        }
      }
      if (ORDERED)
        for (int o = g >> 1; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      else
        for (int o = 1; o < g; o <<= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      if (lead) stx(rc & 0x3ffffff, (xr - part) * rr);
      for (; l0 < l1; ++l0) sync_all();
      u0 = u1;
      l1 = l2;
      u1 = u2;
#pragma unroll
      for (int h = 0; h < SWP; ++h) {
        p0[h] = q1.p[h];
        a0[h] = b0[h];
      }
      rc = q1.rc;
      rr = rn;
      q1 = q2;
    }
  };

  // the trailing block: T = L or U^T going down, U or L^T going up, at
  // LU[k nd + i], or LU[i nd + k] with trans
  const auto dense = [&](bool up) {
    if (ORDERED) {
      dense_small<TH>(A + S.dense_base, r + t0, nd, trans != 0, up, x + t0, blk);
      return;
    }
    const double *inv = S.dinv + (size_t)sc * nblk * 2 * NB * NB + ((trans != 0) != up ? NB * NB : 0);
    trsv::sweep<TH, NB, MULTI>(
        A + S.dense_base, (size_t)nd, nd, trans != 0, up, inv, 2 * NB * NB, C, rank, sm1,
        [&](int i) { return ldx(t0 + i); }, [&](int i, double y) { stx(t0 + i, y); });
  };

  sweep(S.swf_lev, S.swf_n - (nd > 0 ? 1 : 0), trans != 0);
  if (nd > 0) {
    sweep(S.swf_lev + S.swf_n - 1, 1, false);  // the sparse part of the trailing rows
    dense(false);
    dense(true);
  }
  sweep(S.swb_lev, S.swb_n, trans == 0);
  if (!MULTI && in_smem)
    for (int i = tid; i < nx; i += TH) vs[i] = x[i];
}

template <class K>
size_t dyn_smem_cap(K kernel) {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess || !raise_smem_cap(kernel)) return 48 * 1024;
  return (size_t)optin - fa.sharedSizeBytes;
}

// one CTA per vector; the vector in shared memory when it fits there
template <int TH, int NB>
void solve1_single(const DevSym &S, const double *LU, const double *rd, double *v, int trans, int vps, cudaStream_t st) {
  static const size_t cap = dyn_smem_cap(k_solve1<TH, NB, false>);
  const size_t base = trsv::smem_doubles<TH, NB>((S.nd + NB - 1) / NB) * sizeof(double);
  const size_t vec = (size_t)S.nx * sizeof(double);
  const int in = base + vec <= cap ? 1 : 0;
  k_solve1<TH, NB, false><<<(unsigned)(S.N * (long long)vps), TH, base + (in ? vec : 0), st>>>(S, LU, rd, v, trans, vps,
                                                                                         1, in);
  ipm_count_launch();
}

// the small networks: one CTA per vector
template <int TH>
void solve1_ordered(const DevSym &S, const double *LU, const double *rd, double *v, int trans, int vps, cudaStream_t st) {
  k_solve1<TH, NB_SMALL, false, true><<<(unsigned)(S.N * (long long)vps), TH, (size_t)S.nx * sizeof(double), st>>>(
      S, LU, rd, v, trans, vps, 1, 1);
  ipm_count_launch();
}

// a cluster of 8 CTAs per vector while the SMs hold them all at once (two
// per SM), else 4
template <int TH>
void solve1_cluster_launch(const DevSym &S, const double *LU, const double *rd, double *v, int trans, int vps, int C,
                           cudaStream_t st) {
  static const size_t cap = dyn_smem_cap(k_solve1<TH, NB_BIG, true>);
  (void)cap;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((long long)S.N * vps * C));
  cfg.blockDim = dim3(TH);
  cfg.dynamicSmemBytes =
      trsv::smem_doubles<TH, NB_BIG>(((S.nd + NB_BIG - 1) / NB_BIG + C - 1) / C) * sizeof(double);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_solve1<TH, NB_BIG, true>, S, LU, rd, v, trans, vps, C, 0); ipm_count_launch();
}
void solve1_cluster(const DevSym &S, const double *LU, const double *rd, double *v, int trans, int vps,
                    cudaStream_t st) {
  const int C = (long long)S.N * vps <= 38 || S.nd > 8192 ? 8 : 4;
  // the accumulators take TH doubles per block and CTA: fewer threads for the
  // larger blocks, up to the largest that a scenario's factor can index
  constexpr auto fits = [](size_t doubles) { return doubles * sizeof(double) <= 227 * 1024; };
  static_assert(fits(trsv::smem_doubles<512, NB_BIG>(8192 / NB_BIG / 4)), "512 threads, clusters of 4");
  static_assert(fits(trsv::smem_doubles<256, NB_BIG>(40448 / NB_BIG / 8)), "256 threads");
  static_assert(fits(trsv::smem_doubles<128, NB_BIG>((46340 / NB_BIG + 8) / 8)), "nd^2 < 2^31");
  if (S.nd <= 8192) solve1_cluster_launch<512>(S, LU, rd, v, trans, vps, C, st);
  else if (S.nd <= 40448) solve1_cluster_launch<256>(S, LU, rd, v, trans, vps, C, st);
  else solve1_cluster_launch<128>(S, LU, rd, v, trans, vps, C, st);
}

template <int NB>
void diag_inverse(const DevSym &S, const double *LU, const double *rd, cudaStream_t st) {
  constexpr size_t bytes = 3 * NB * (NB + 1) * sizeof(double);
  static const bool cap = raise_smem_cap(k_diag_inverse<NB>);
  (void)cap;
  k_diag_inverse<NB><<<dim3((S.nd + NB - 1) / NB, S.N), 256, bytes, st>>>(S, LU, rd); ipm_count_launch();
}

}  // namespace

size_t diag_inverse_doubles(const DevSym &S) {
  const int NB = S.big ? NB_BIG : NB_SMALL;
  if (S.ordered) return 0;  // k_solve1 does without
  return (size_t)S.N * ((S.nd + NB - 1) / NB) * 2 * NB * NB;
}

void launch_diag_inverse(const DevSym &S, const double *LU, const double *rd, cudaStream_t st) {
  if (S.nd == 0 || S.ordered) return;
  if (S.big) diag_inverse<NB_BIG>(S, LU, rd, st);
  else diag_inverse<NB_SMALL>(S, LU, rd, st);
}

void launch_solve1(const DevSym &S, const double *LU, const double *rd, double *v, int trans, cudaStream_t st) {
  if (S.big) {
    solve1_cluster(S, LU, rd, v, trans, 1, st);
    return;
  }
  // one warp per scheduled unit is enough on the small networks, and a
  // barrier over four warps is cheaper than over eight
  if (S.ordered) solve1_ordered<128>(S, LU, rd, v, trans, 1, st);
  else if (S.nx <= 400) solve1_single<128, NB_SMALL>(S, LU, rd, v, trans, 1, st);
  else solve1_single<256, NB_SMALL>(S, LU, rd, v, trans, 1, st);
}

void launch_solve1_batched(const DevSym &S, const double *LU, const double *rd, double *v, int trans, int vps,
                           cudaStream_t st) {
  if (S.ordered) solve1_ordered<128>(S, LU, rd, v, trans, vps, st);
  else if (!S.big) solve1_single<128, NB_SMALL>(S, LU, rd, v, trans, vps, st);
  else if (S.nd <= 4096) solve1_single<256, NB_BIG>(S, LU, rd, v, trans, vps, st);  // 128 KB of accumulators
  else solve1_cluster(S, LU, rd, v, trans, vps, st);
}
