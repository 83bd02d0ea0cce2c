// Triangular sweeps of one vector through a dense matrix, by blocks of NB
// rows whose diagonal blocks' inverses are at hand: the building block of
// the single-vector solves with G_x (the dense trailing block) and with the
// Cholesky factor of K_hat.
//
// A block of the solution takes one product with the next tile of the factor
// and one with the inverse, a chain of a few FP64 operations, barriers and
// (MULTI) one cluster barrier; the tiles of the blocks after it are applied
// behind that chain.  With the inverses, a block is two small products
// instead of NB dependent steps of ~100 cycles each.
#pragma once
#include "dev.cuh"

namespace trsv {

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void copy8_async(double *dst, const double *src) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void store_rank(double *local, unsigned rank, double v) {
  const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(local));
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
}

// Inverse of a unit triangular m x m block (m <= NB) held in shared memory
// (T: the strict triangle, the diagonal taken as 1), into X (identity on
// entry), by elimination steps in which every entry of X is independent:
// lower from the first row down, upper from the last row up.  Threads t of
// nt; every step ends with a CTA barrier, so all threads of the CTA call it
// with the same m.  FP64-bound: m^3 / 6 multiply-adds.
template <class Mat>
__device__ void unit_inverse(Mat T, Mat X, int m, bool upper, int t, int nt) {
  for (int s = 0; s < m - 1; ++s) {
    const int k = upper ? m - 1 - s : s, w = s + 1, n = (m - 1 - s) * w;
    for (int e = t; e < n; e += nt) {
      const int i = upper ? e / w : k + 1 + e / w, j = upper ? k + e % w : e % w;
      X[i][j] -= T[i][k] * X[k][j];
    }
    __syncthreads();
  }
}

// doubles of dynamic shared memory of a sweep with `own` blocks per CTA
template <int TH, int NB>
__host__ __device__ constexpr size_t smem_doubles(int own) {
  return (size_t)TH + 3 * NB + 2 * (NB / (TH / NB)) * TH + (size_t)own * TH;
}

// One sweep, down (up = false) or up, of the n x n triangular matrix
// T(i, k) = M[k ld + i], or M[i ld + k] with swap; inv: the inverses of the
// diagonal blocks, block b at inv + b inv_st, (i, k) at k NB + i, or i NB + k
// with swap.  Element i of the vector is read and written by ldx(i),
// stx(i, value).  Block b belongs to CTA b mod C of the cluster (C = 1
// without MULTI).  G threads share a row of a block, each with CPG of its
// columns, so that a warp reads whole segments of the factor: 32 rows of one
// column, or with swap G neighbouring columns of 32 / G rows (rows of 64
// contiguous bytes per thread were read at half the rate).  A thread sums its
// share of the updates of each of the CTA's blocks in accs; the next tile and
// inverse of the chain come by asynchronous copies, every thread its own,
// while the CTA waits or updates its other blocks.  A solved block is stored
// into the shared memory of every CTA of the cluster.  Called by all threads
// with the vector's rows visible (and every CTA of the cluster started);
// ends so.
template <int TH, int NB, bool MULTI, class Ldx, class Stx>
__device__ __forceinline__ void sweep(const double *__restrict__ M, size_t ld, int n, bool swap, bool up,
                                      const double *__restrict__ inv, size_t inv_st, int C, int rank,
                                      double *sm, Ldx ldx, Stx stx) {
  constexpr int G = TH / NB, CPG = NB / G;
  const int tid = threadIdx.x, nblk = (n + NB - 1) / NB;
  const int rr = swap ? tid / G : tid % NB, g = swap ? tid % G : tid / NB;  // row and share of a block
  const int k0 = swap ? g : CPG * g, ks = swap ? G : 1;                     // columns k0 + j ks
  double *red = sm, *xs = red + TH, *xb = xs + NB, *pre = xb + 2 * NB, *accs = pre + 2 * CPG * TH;
  for (int o = 0; o * C + rank < nblk; ++o) accs[o * TH + tid] = 0.0;
  const auto sync_all = [] {
    if (MULTI) {
      __syncwarp();
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
  };
  const auto tile_ptr = [&](int jb, int kb) {
    const size_t i = (size_t)jb * NB + rr, k = (size_t)kb * NB + k0;
    return swap ? M + i * ld + k : M + k * ld + i;
  };
  const size_t st = swap ? (size_t)G : ld;
  const auto products = [&](const double(&a)[CPG], const double(&x)[CPG]) {
    double s0 = 0.0, s1 = 0.0;
#pragma unroll
    for (int j = 0; j < CPG; j += 2) {
      s0 = fma(a[j], x[j], s0);
      s1 = fma(a[j + 1], x[j + 1], s1);
    }
    return s0 + s1;
  };
  // accs of block jb += tile (jb, kb) x
  const auto tile = [&](int jb, int kb, const double(&xk)[CPG]) {
    if (jb * NB + rr >= n) return;
    const double *p = tile_ptr(jb, kb);
    double a[CPG];
#pragma unroll
    for (int j = 0; j < CPG; ++j) a[j] = kb * NB + k0 + j * ks < n ? __ldg(p + j * st) : 0.0;
    accs[(jb / C) * TH + tid] += products(a, xk);
  };
  // the thread's shares of the tile (b, kb) and of block b's inverse
  double own = 0.0;  // of threads tid < NB: their row of the block fetched
  const auto fetch = [&](int b, int kb) {
    if (tid < NB && b * NB + tid < n) own = ldx(b * NB + tid);
    const double *p = tile_ptr(b, kb), *I = inv + (size_t)b * inv_st;
#pragma unroll
    for (int j = 0; j < CPG; ++j) {
      const int k = k0 + j * ks;
      if (kb >= 0) {
        if (b * NB + rr < n && kb * NB + k < n) copy8_async(&pre[j * TH + tid], p + j * st);
        else pre[j * TH + tid] = 0.0;
      }
      copy8_async(&pre[(CPG + j) * TH + tid], swap ? I + rr * NB + k : I + k * NB + rr);
    }
  };
  const auto sum_groups = [&](int i) {
    double s[G];
#pragma unroll
    for (int q = 0; q < G; ++q) s[q] = red[q * NB + i];
#pragma unroll
    for (int o = G / 2; o > 0; o /= 2)
#pragma unroll
      for (int q = 0; q < G; ++q)
        if (q < o) s[q] += s[q + o];
    return s[0];
  };
  // solve block b (its owner, fetch(b, .) done before); part: the thread's
  // share of the last update; the block goes to slot `slot` of xb everywhere
  const auto chain = [&](int b, double part, int slot) {
    const int row = b * NB + tid;
    red[g * NB + rr] = accs[(b / C) * TH + tid] + part;
    __syncthreads();
    if (tid < NB) xs[tid] = row < n ? own - sum_groups(tid) : 0.0;
    __syncthreads();
    double m[CPG], x[CPG];
#pragma unroll
    for (int j = 0; j < CPG; ++j) {
      m[j] = pre[(CPG + j) * TH + tid];
      x[j] = xs[k0 + j * ks];
    }
    red[g * NB + rr] = products(m, x);
    __syncthreads();
    if (tid < NB) {
      const double y = row < n ? sum_groups(tid) : 0.0;
      if (MULTI)
        for (int q = 0; q < C; ++q) store_rank(&xb[slot * NB + tid], (unsigned)q, y);
      else xb[slot * NB + tid] = y;
      if (row < n) stx(row, y);
    }
  };
  const int first = up ? nblk - 1 : 0, dir = up ? -1 : 1;
  if (first % C == rank) {
    fetch(first, -1);
    copy_wait();
    chain(first, 0.0, first & 1);
  }
  if (nblk > 1 && (first + dir) % C == rank) fetch(first + dir, first);
  sync_all();
  for (int b = first; b + dir >= 0 && b + dir < nblk; b += dir) {
    const int nb = b + dir, nn = nb + dir;
    double xk[CPG];
#pragma unroll
    for (int j = 0; j < CPG; ++j) xk[j] = xb[(b & 1) * NB + k0 + j * ks];
    if (nb % C == rank) {
      copy_wait();
      double a[CPG];
#pragma unroll
      for (int j = 0; j < CPG; ++j) a[j] = pre[j * TH + tid];
      chain(nb, products(a, xk), nb & 1);
    }
    if (MULTI) {
      __syncwarp();
      cluster_arrive();
    }
    if (nn >= 0 && nn < nblk && nn % C == rank) fetch(nn, nb);
    // the CTA's other blocks, away from nb
    if (up) {
      for (int j = rank; j < nb; j += C) tile(j, b, xk);
    } else {
      for (int j = (nb / C) * C + rank; j < nblk; j += C)
        if (j > nb) tile(j, b, xk);
    }
    if (MULTI) cluster_wait();
    else __syncthreads();
  }
}

}  // namespace trsv
