// K3-K5: batched static-pivot sparse LU of G_x (one pattern for all
// scenarios) and the multi-RHS reduction solves Z = -G_x^{-1} G_u fused with
// the products Y = K [Z; I].
//
// Paper: §3.2 "Assembling the sparse matrices" (batched LU sharing one
// pattern, G_x^{-1} b = Q U^{-1} L^{-1} P b) and "Local reduction" (steps
// 1-2: T_x = -G_x^{-1} G_u V, [L_x; L_u] = K [T_x; V]).  Here V runs over
// all Cartesian vectors at once, split into RHS panels of 32 columns.
//
// Scheduling: the LU runs on a cluster of two CTAs per scenario (cluster
// barriers between its steps; a one-CTA kernel when the trailing block does
// not fit the pair's shared memory; with a large trailing block up to eight
// CTAs for the sparse part, the block by the kernels of kernels_big.cu), the
// multi-RHS solves on CTAs that work through (scenario, RHS panel) items, b
// in the last panel's free column; each walks a level schedule of the shared
// pattern with a barrier between levels.  No grid-wide synchronisation and no
// waits between CTAs other than the cluster barriers.  The single-vector
// solves are in kernels_solve1.cu.
#include <algorithm>
#include <atomic>

#include "dev.cuh"
#include "kernels.h"


namespace {

__device__ __forceinline__ double block_max(double v, double *sh) {
  v = warp_max(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    v = (lane < (blockDim.x >> 5)) ? sh[lane] : 0.0;
    v = warp_max(v);
    if (lane == 0) sh[0] = v;
  }
  __syncthreads();
  const double r = sh[0];
  __syncthreads();
  return r;
}

// Batched LU: the sparse pivots follow the level schedule (gather-form
// updates), then the dense trailing block [t0, nx) is factorized right-looking
// in shared memory when it fits (dynamic shared memory of nd*nd doubles),
// else in place through the slot map.
// Cluster helpers: rank in the cluster, a barrier over both CTAs with
// release/acquire ordering (shared and global memory), and a load from the
// peer CTA's shared memory.
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive_all() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_all() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ double ld_peer(const double *local, unsigned peer) {
  const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(local));
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(peer));
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(ra) : "memory");
  return v;
}

// Sparse part of the factorization of one scenario: values of G_x into the
// LU pattern, the level-scheduled sparse pivots (gather form), the scaling
// of L, and the products of the sparse pivots into the dense trailing
// block.  One CTA, or (CL) the C CTAs of a cluster sharing every step by
// index with cluster barriers between the steps.  Returns max |G_x| (the
// reference of the pivot test).  Bound by the latency of its gathers: a
// product's three places come in one load, and the lists of the trailing
// block fetch the next eight products' places under this eight's values.
template <bool CL>
__device__ double lu_sparse_part(const DevSym &S, int nL, const double *__restrict__ J, double *A, double *r,
                                 int *flags, double piv_tol, int sc, double *sh, unsigned rank, int C) {
  const int tid = threadIdx.x, bd = blockDim.x;
  const int t0i = CL ? tid + (int)rank * bd : tid, step = CL ? C * bd : bd;
  auto sync = [] {
    if (CL) cluster_sync_all();
    else __syncthreads();
  };
  double amax = 0.0;
  for (int p0 = t0i; p0 < S.nnzLU; p0 += 4 * step) {  // four entries' loads in flight
    double v[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int p = p0 + b * step, src = p < S.nnzLU ? S.lu_init[p] : -1;
      v[b] = src >= 0 ? J[(size_t)src * S.N + sc] : 0.0;
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      if (p0 + b * step < S.nnzLU) A[p0 + b * step] = v[b];
      amax = fmax(amax, fabs(v[b]));
    }
  }
  amax = block_max(amax, sh);
  if (CL) {
    if (tid == 0) sh[16] = amax;
    cluster_sync_all();
    for (int q = 0; q < C; ++q) amax = fmax(amax, ld_peer(&sh[16], (unsigned)q));
  }
  for (int l = 0; l < S.nlev_f; ++l) {
    for (int e = S.f_piv_ptr[l] + t0i; e < S.f_piv_ptr[l + 1]; e += step) {
      const int k = S.f_piv[e];
      const double d = A[S.lu_diag[k]];
      if (!(fabs(d) > piv_tol * amax)) flags[FLAG_SINGULAR] = 1;
      r[k] = 1.0 / d;
    }
    sync();
    for (int t = S.f_lev_ptr[l] + t0i; t < S.f_lev_ptr[l + 1]; t += step) {
      const int slot = S.f_tgt[t], o1 = S.f_op_ptr[t + 1];
      double acc = A[slot];
      for (int o = S.f_op_ptr[t]; o < o1; ++o) {
        const int4 op = S.f_op[o];
        acc -= A[op.x] * (A[op.y] * r[op.z]);
      }
      A[slot] = acc;
    }
    sync();
  }
  for (int e = t0i; e < nL; e += step) A[S.lsc_slot[e]] *= r[S.lsc_k[e]];
  sync();
  if (S.nd == 0) return amax;
  // Products of the sparse pivots into the trailing block (L already
  // scaled): each entry owned by one of the lists, its products summed and
  // subtracted once; lists interleaved (coalesced), list q taken by thread q
  // of the cluster (or the threads in turn).  The products read sparse L and
  // U slots only, never a trailing-block slot, so batches of eight have all
  // their loads issued before the multiply-adds and stores.
  const double *__restrict__ Ar = A;
  const int lists = S.lu_lists;
  for (int q = t0i; q < lists; q += step) {
    const int len = S.tw_len[q];
    double acc = 0.0;
    int ln[8], un[8], en[8];
    const auto places = [&](int q0) {
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        ln[b] = un[b] = en[b] = -1;
        if (q0 + b < len) {
          const size_t at = (size_t)(q0 + b) * lists + q;
          ln[b] = S.tw_l[at];
          un[b] = S.tw_u[at];
          en[b] = S.tw_e[at];
        }
      }
    };
    places(0);
    for (int q0 = 0; q0 < len; q0 += 8) {
      double lv[8], uv[8];
      int ev[8];
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        lv[b] = ln[b] >= 0 ? Ar[ln[b]] : 0.0;
        uv[b] = un[b] >= 0 ? Ar[un[b]] : 0.0;
        ev[b] = en[b];
      }
      places(q0 + 8);
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        if (q0 + b < len) {
          acc = fma(lv[b], uv[b], acc);
          if (ev[b] >= 0) {
            A[ev[b]] -= acc;
            acc = 0.0;
          }
        }
      }
    }
  }
  sync();
  return amax;
}

// The sparse part alone, by a cluster of C CTAs per scenario: networks with a
// large trailing block, which the batched kernels factor next.
__global__ void __launch_bounds__(512) k_lu_sparse(DevSym S, int nL, const double *__restrict__ J, double *LU,
                                                   double *rd, int *flags, double piv_tol, int C) {
  __shared__ double sh[32];
  const unsigned rank = cluster_rank();
  const int sc = blockIdx.x / C;
  const double amax = lu_sparse_part<true>(S, nL, J, LU + (size_t)sc * S.nnzLU, rd + (size_t)sc * S.nx, flags,
                                           piv_tol, sc, sh, rank, C);
  if (rank == 0 && threadIdx.x == 0) S.lu_amax[sc] = amax;
  cluster_sync_all();  // no CTA leaves while another may still read its maximum
}

__global__ void k_lu_factor(DevSym S, int nL, const double *__restrict__ J, double *LU, double *rd,
                            int *flags, double piv_tol, int ns) {
  __shared__ double sh[32];
  extern __shared__ double T[];
  const int sc = blockIdx.x, tid = threadIdx.x, bd = blockDim.x;
  double *A = LU + (size_t)sc * S.nnzLU;
  double *r = rd + (size_t)sc * S.nx;
  const double amax = lu_sparse_part<false>(S, nL, J, A, r, flags, piv_tol, sc, sh, 0u, 1);
  const int nd = S.nd, t0 = S.t0;
  if (nd == 0) return;
  const int *ts = S.tail_slot;
  // dense trailing block: columns [0, k0) in place through the slot map,
  // then the remaining (nd-k0)^2 block in shared memory (k0 = nd - ns)
  const int k0 = nd - ns;
  // columns [0, k0 - 1) through the slot map; the last of them is fused
  // into the load of the shared-memory block
  for (int k = 0; k < k0; ++k) {
    if (tid == 0) {
      const double d = A[ts[k * nd + k]];
      if (!(fabs(d) > piv_tol * amax)) flags[FLAG_SINGULAR] = 1;
      r[t0 + k] = 1.0 / d;
      sh[0] = r[t0 + k];
    }
    __syncthreads();
    const double rk = sh[0];
    const int m = nd - k - 1;
    if (k + 1 == k0) {
      // T = A22 - (A21 / d) A12, and L21 = A21 / d written back
      for (int e = tid; e < ns * ns; e += bd) {
        const int a = k0 + e / ns, b = k0 + e % ns;
        T[e] = A[ts[a * nd + b]] - (A[ts[a * nd + k]] * rk) * A[ts[k * nd + b]];
      }
      __syncthreads();
      for (int e = tid; e < m; e += bd) A[ts[(k + 1 + e) * nd + k]] *= rk;
      break;
    }
    for (int e = tid; e < m; e += bd) A[ts[(k + 1 + e) * nd + k]] *= rk;
    __syncthreads();
    for (int e = tid; e < m * m; e += bd) {
      const int a = k + 1 + e / m, b = k + 1 + e % m;
      A[ts[a * nd + b]] -= A[ts[a * nd + k]] * A[ts[k * nd + b]];
    }
    __syncthreads();
  }
  if (ns == 0) return;
  if (k0 == 0)
    for (int e = tid; e < ns * ns; e += bd) T[e] = A[ts[(k0 + e / ns) * nd + k0 + e % ns]];
  __syncthreads();
  // Blocked right-looking LU of the ns x ns block in shared memory (static
  // diagonal pivots): per panel of PB columns, (a) the panel column by
  // column, (b) U12 = L11^{-1} A12 (thread per column), (c) the trailing
  // update A22 -= L21 U12 with 4 x 4 register tiles (one shared-memory read
  // per 4 multiply-adds instead of three per multiply-add).
  constexpr int PB = 16;
  for (int kb = 0; kb < ns; kb += PB) {
    const int pb = min(PB, ns - kb), ke = kb + pb;
    for (int k = kb; k < ke; ++k) {
      // one thread forms the pivot's reciprocal (a dependent FP64 division
      // is ~9 multiply-adds of FP64 work: not once per thread)
      if (tid == 0) {
        const double d = T[k * ns + k];
        if (!(fabs(d) > piv_tol * amax)) flags[FLAG_SINGULAR] = 1;
        r[t0 + k0 + k] = 1.0 / d;
        sh[0] = r[t0 + k0 + k];
      }
      __syncthreads();
      const double rk = sh[0];
      // thread per row: scale L(i, k), update the rest of the panel row
      for (int i = k + 1 + tid; i < ns; i += bd) {
        const double l = T[i * ns + k] * rk;
        T[i * ns + k] = l;
        for (int j = k + 1; j < ke; ++j) T[i * ns + j] -= l * T[k * ns + j];
      }
      __syncthreads();
    }
    if (ke >= ns) break;
    for (int j = ke + tid; j < ns; j += bd)
      for (int k = kb; k < ke; ++k) {
        const double x = T[k * ns + j];
        for (int i = k + 1; i < ke; ++i) T[i * ns + j] -= T[i * ns + k] * x;
      }
    __syncthreads();
    const int m = ns - ke, nt4 = (m + 3) / 4;
    for (int e = tid; e < nt4 * nt4; e += bd) {
      const int i0 = ke + (e / nt4) * 4, j0 = ke + (e % nt4) * 4;
      double c[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) c[a][b] = 0.0;
      for (int k = kb; k < ke; ++k) {
        double lv[4], uv[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) lv[a] = i0 + a < ns ? T[(i0 + a) * ns + k] : 0.0;
#pragma unroll
        for (int b = 0; b < 4; ++b) uv[b] = j0 + b < ns ? T[k * ns + j0 + b] : 0.0;
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) c[a][b] = fma(lv[a], uv[b], c[a][b]);
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
          if (i0 + a < ns && j0 + b < ns) T[(i0 + a) * ns + j0 + b] -= c[a][b];
    }
    __syncthreads();
  }
  for (int e = tid; e < ns * ns; e += bd) A[ts[(k0 + e / ns) * nd + k0 + e % ns]] = T[e];
}

// C consecutive elements in one 16-byte (or 8-byte) access
template <typename T, int C>
struct alignas(sizeof(T) * C) Pack {
  T v[C];
};

// One scheduled row: its place, its products [f0, f0 + len).
struct RowDesc {
  int row, f0, len;
};

// Walks the rows of levels [0, nlev) (rows lev(l) .. lev(l + 1) of a
// schedule; a CTA barrier after every level), W lanes to a row and C columns
// of the right-hand sides to a lane: acc = init(row), then the row's
// products in their order, acc -= (or +=) value * operand(place), then
// finish(row, acc).  The lanes of a row fetch the places and values of W
// products side by side (each once per row instead of once per lane) and
// hand them round by shuffles; U products' operands are in flight.
// meta(f, place, slot), value(slot); operand(place, mine) may clear mine
// (no product for this lane, whatever the value).  Called by all threads.
// Fetching the next chunk's places and values ahead of this one's operands
// was measured too: its registers cost more warps than it hid latency
// (3.58 -> 4.20 ms FP64, 1.27 -> 1.85 ms FP32 at 1,000 buses x 64).
template <typename T, int W, int C, int U, bool SUB, class Lev, class Desc, class Meta, class Value, class Operand,
          class Init, class Finish>
__device__ __forceinline__ void sweep_rows(int nlev, Lev lev, Desc desc, Meta meta, Value value, Operand operand,
                                           Init init, Finish finish) {
  constexpr int R = 32 / W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, cl = lane % W;
  for (int l = 0; l < nlev; ++l) {
    const int e1 = lev(l + 1);
    for (int eb = lev(l) + warp * R; eb < e1; eb += (blockDim.x >> 5) * R) {
      const int e = eb + lane / W;
      RowDesc d = {-1, 0, 0};
      if (e < e1) d = desc(e);
      const int mlen = W == 32 ? d.len : (int)__reduce_max_sync(0xffffffffu, (unsigned)d.len);
      Pack<T, C> acc = {};
      if (d.row >= 0) acc = init(d.row);
      for (int base = 0; base < mlen; base += W) {
        int at = 0, slot;
        T val = 0;
        if (base + cl < d.len) {
          meta(d.f0 + base + cl, at, slot);
          val = value(slot);
        }
        const int n = min(W, mlen - base);
        for (int j = 0; j < n; j += U) {
          T v[U];
          Pack<T, C> z[U];
#pragma unroll
          for (int k = 0; k < U; ++k) {
            const int p = __shfl_sync(0xffffffffu, at, j + k, W);
            v[k] = __shfl_sync(0xffffffffu, val, j + k, W);
            z[k] = Pack<T, C>{};
            bool mine = base + j + k < d.len;
            if (mine) z[k] = operand(p, mine);
            if (!mine) v[k] = 0;
          }
#pragma unroll
          for (int k = 0; k < U; ++k)
#pragma unroll
            for (int q = 0; q < C; ++q) acc.v[q] = SUB ? acc.v[q] - v[k] * z[k].v[q] : acc.v[q] + v[k] * z[k].v[q];
        }
      }
      if (d.row >= 0) finish(d.row, acc);
    }
    __syncthreads();
  }
}

// Multi-RHS reduction solve for one scenario and one panel of PW = W C RHS
// columns: Z = -U^{-1} L^{-1} (P G_u) (rows in LU position order), then
// Y = K_x [Z; I] and Y_u = K_u [Z; I].  The sparse rows follow the level
// schedule (W lanes per row, C columns per lane); the dense trailing block
// [t0, nx) is solved by the whole CTA in shared memory.  T is the
// storage/arithmetic type of Z, Y (double on the FP64 path, float on the
// mixed path); Y_u accumulates in FP64.  A, r (factor values, reciprocal
// pivots) and, on the mixed path, Kp (K in the order of the product lists)
// are of type T: GB300 converts between FP64 and FP32 at the rate of its
// FP64 units (a warp-wide conversion every ~19 cycles per SM), so a
// conversion per product and lane made the FP32 solve as slow as the FP64
// one; the mixed path converts each value once (k_round_factors, k_round_k).
//
// The panel is worked on in Zp, a contiguous buffer of the CTA's own
// ([nx][PW], lane cl's C columns side by side: element cl C + q of a row is
// column c0 + q W + cl), and written to Z as Y is formed: an operand is one
// 16-byte load per lane at a shifted index, and a warp works on 32 / W rows
// at once.  Bound by the FP64 units (75 % of their cycles) on the FP64 path
// and by the latency of the operand loads on the mixed one.  Measured (the
// whole solve, against a warp per row of 32 columns with one column and
// every product's column, slot and value loaded by every lane): 1,000 buses
// x 64 4.03 -> 3.54 ms FP64 and 3.08 -> 1.13 ms FP32, 433 buses x 19 685 ->
// 413 us FP64, 10,000 buses x 32 67.3 -> 39.1 ms FP32 (17 ms of it the dense
// block's own kernels).  W x C = 8 x 4 on the mixed path: 22.1 ms at 10,000 x
// 32 and 4.3 at 3,000 x 40, 16 x 2 24.4 and 4.6, 32 x 1 40.1 and 6.9.  CTAs of
// 512 threads take 19.8 and 3.6 there, of 1,024 21.7 and 4.2, of 128 26.1
// (10,000 x 32); 256 were taken when the backward sweep had many more levels
// (817 instead of 25 at 10,000 buses), which the larger CTAs paid for.
//
// phase (large trailing block, S.big): 1 = the forward sparse rows and the
// trailing rows' right-hand sides only (left in Z for the batched block
// solves), 2 = the rest, the trailing rows taken from Z (the forward sparse
// rows, a few percent of the products, are formed again); 0 = all.
template <typename T, int W, int C>
__device__ void zsolve_panel(const DevSym &S, int sc, int panel, const T *__restrict__ A, const T *__restrict__ r,
                             const double *__restrict__ J, const double *__restrict__ K, const T *__restrict__ Kp,
                             T *__restrict__ Zp, T *Zs, T *Ys, double *Yus, T *sh, const double *__restrict__ gvec,
                             T *bs, int *ezy, int phase) {
  using P = Pack<T, C>;
  constexpr int R = 32 / W, PW = W * C, U = 4;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int cl = lane % W, grp = warp * R + lane / W, ngrp = nw * R;
  const int nu = S.nu, nx = S.nx, N = S.N;
  const int c0 = panel * PW, c = c0 + cl;  // the lane's columns c, c + W, ...
  const int t0 = S.t0, nd = S.nd;
  // Optional extra column n_u (bs given): b = G_x^{-1} g of the reduced
  // right-hand side, in the first free place of the last panel (there is
  // one: n_u = 2 n_g - 1 is odd).  Its forward sweep is dense, so that panel
  // takes the schedule of all rows (+11 % of one panel's products at 1,000
  // buses, against +85 % for a panel of its own).
  const auto zrow = [&](int row) { return reinterpret_cast<P *>(Zp + (size_t)row * PW) + cl; };
  const auto zread = [&](int row, bool &) { return *zrow(row); };
  const auto lu_meta = [](const int2 *pr) {
    return [pr](int f, int &col, int &slot) {
      const int2 p = pr[f];
      col = p.x;
      slot = p.y;
    };
  };
  const auto lu_value = [&](int slot) { return A[slot]; };
  // right-hand side of a row: -G_u (or g, for b)
  const auto rhs_of = [&](int row) {
    P acc = {};
    for (int g = S.gu_ptr[row]; g < S.gu_ptr[row + 1]; ++g) {
      const int d = S.gu_col[g] - c;
      if (d >= 0 && d < PW && d % W == 0) {
        const int src = S.gu_src[g];
        const T v = src >= 0 ? (T)J[(size_t)src * N + sc] : (T)-1.0;
#pragma unroll
        for (int q = 0; q < C; ++q)
          if (d == q * W) acc.v[q] -= v;
      }
    }
    if (bs)
#pragma unroll
      for (int q = 0; q < C; ++q)
        if (c + q * W == nu) acc.v[q] = (T)gvec[(size_t)sc * nx + S.iperm[row]];
    return acc;
  };
  // forward, sparse rows: the schedule of the 32-column panel that holds
  // this one (rows its columns of G_u reach, products against such rows
  // only; the other rows are zero), or of all rows beside b
  const int pan = bs != nullptr && c0 + PW > nu ? S.zp_npan - 1 : c0 / 32;
  for (int e = S.zp_zptr[pan] + grp; e < S.zp_zptr[pan + 1]; e += ngrp) *zrow(S.zp_zrows[e]) = P{};
  {
    const int *lp = S.zp_lev_ptr + S.zp_lev_off[pan];
    sweep_rows<T, W, C, U, true>(
        S.zp_lev_off[pan + 1] - S.zp_lev_off[pan], [&](int l) { return lp[l]; },
        [&](int e) { return RowDesc{S.zp_rows[e], S.zp_eptr[e], S.zp_eptr[e + 1] - S.zp_eptr[e]}; },
        lu_meta(S.zp2), lu_value, zread, rhs_of, [&](int row, const P &acc) { *zrow(row) = acc; });
  }
  if (phase == 2) {  // the solved trailing rows
    for (int i = grp; i < nd; i += ngrp) {
      P z = {};
#pragma unroll
      for (int q = 0; q < C; ++q)
        if (c + q * W < nu) z.v[q] = Zs[(size_t)(unsigned)(t0 + i) * (unsigned)nu + c + q * W];
      *zrow(t0 + i) = z;
    }
    __syncthreads();
  } else {
    // trailing block: right-hand side and the sparse part of each row
    P *shp = reinterpret_cast<P *>(sh) + cl;  // row i at shp[i * W]
    const int *tp = S.zp_tptr + pan * nd;
    sweep_rows<T, W, C, U, true>(
        1, [&](int l) { return l * nd; }, [&](int i) { return RowDesc{i, tp[i], tp[i + 1] - tp[i]}; },
        lu_meta(S.zpt2), lu_value, zread, [&](int i) { return rhs_of(t0 + i); },
        [&](int i, const P &acc) {
          if (phase == 0) {
            shp[i * W] = acc;
          } else {
#pragma unroll
            for (int q = 0; q < C; ++q)
              if (c + q * W < nu) Zs[(size_t)(unsigned)(t0 + i) * (unsigned)nu + c + q * W] = acc.v[q];
          }
        });
    if (phase == 1) return;  // the block is solved by the batched kernels
    // Blocked by 32 in shared memory: one warp solves each diagonal block (R
    // rows at a time), then every warp applies the block's columns to the
    // remaining rows.  The block is column-major with leading dimension nd
    // in LU storage (the same address for all lanes of a row).  Backward
    // values are scaled as they are found.
    const T *D = A + S.dense_base;
    const auto sub = [&](int i, const P &x, T a) {
      P y = shp[i * W];
#pragma unroll
      for (int q = 0; q < C; ++q) y.v[q] -= a * x.v[q];
      shp[i * W] = y;
    };
    const auto apply = [&](int i, int kb, int w) {
      P acc = shp[i * W];
      const T *di = D + (size_t)kb * nd + i;
#pragma unroll 4
      for (int j = 0; j < w; ++j) {
        const T a = di[(size_t)j * nd];
        const P x = shp[(kb + j) * W];
#pragma unroll
        for (int q = 0; q < C; ++q) acc.v[q] -= a * x.v[q];
      }
      shp[i * W] = acc;
    };
    for (int kb = 0; kb < nd; kb += 32) {
      const int w = min(32, nd - kb);
      if (warp == 0) {
        for (int jj = 0; jj < w; ++jj) {
          const P xj = shp[(kb + jj) * W];
          const T *col = D + (size_t)(kb + jj) * nd + kb;  // L(kb + i2, kb + jj) = col[i2]
          for (int i2 = jj + 1 + lane / W; i2 < w; i2 += R) sub(kb + i2, xj, col[i2]);
          __syncwarp();
        }
      }
      __syncthreads();
      for (int i = kb + w + grp; i < nd; i += ngrp) apply(i, kb, w);
      __syncthreads();
    }
    for (int kb = ((nd - 1) / 32) * 32; kb >= 0 && nd > 0; kb -= 32) {
      const int w = min(32, nd - kb);
      if (warp == 0) {
        for (int jj = w - 1; jj >= 0; --jj) {
          P xj = shp[(kb + jj) * W];
          const T rk = r[t0 + kb + jj];
#pragma unroll
          for (int q = 0; q < C; ++q) xj.v[q] *= rk;
          __syncwarp();
          if (lane < W) shp[(kb + jj) * W] = xj;
          const T *col = D + (size_t)(kb + jj) * nd + kb;  // U(kb + i2, kb + jj) = col[i2]
          for (int i2 = lane / W; i2 < jj; i2 += R) sub(kb + i2, xj, col[i2]);
          __syncwarp();
        }
      }
      __syncthreads();
      for (int i = grp; i < kb; i += ngrp) apply(i, kb, w);
      __syncthreads();
    }
    for (int i = grp; i < nd; i += ngrp) *zrow(t0 + i) = shp[i * W];
    __syncthreads();
  }
  // backward, sparse rows
  sweep_rows<T, W, C, U, true>(
      S.nlev_bs, [&](int l) { return S.bs_lev_ptr[l]; },
      [&](int e) {
        const int4 q = S.bs4[e];
        return RowDesc{q.x, q.y, q.z - q.y};
      },
      lu_meta(S.br2), lu_value, zread, [&](int row) { return *zrow(row); },
      [&](int row, P acc) {
        const T rr = r[row];
#pragma unroll
        for (int q = 0; q < C; ++q) acc.v[q] *= rr;
        *zrow(row) = acc;
      });
  if (bs)
#pragma unroll
    for (int q = 0; q < C; ++q)
      if (c + q * W == nu)
        for (int row = grp; row < nx; row += ngrp) bs[row] = Zp[(size_t)row * PW + cl * C + q];
  // an operand of K's products: a row of Z, or of I (places from nx on: no
  // product in the other columns, whatever the entry)
  const auto zi_read = [&](int p, bool &mine) {
    if (p < nx) return *zrow(p);
    P z = {};
    mine = false;
#pragma unroll
    for (int q = 0; q < C; ++q) {
      z.v[q] = (T)(p - nx == c + q * W);
      mine |= p - nx == c + q * W;
    }
    return z;
  };
  const T *Ks = Kp ? Kp + (size_t)sc * S.kx_ptr[nx] : nullptr;
  sweep_rows<T, W, C, U, false>(
      1, [&](int l) { return l * nx; },
      [&](int row) { return RowDesc{row, S.kx_ptr[row], S.kx_ptr[row + 1] - S.kx_ptr[row]}; },
      [&](int f, int &col, int &slot) {
        if (Ks) {
          col = S.kx_col[f];
          slot = f;
        } else {
          const int2 p = S.kx2[f];
          col = p.x;
          slot = p.y;
        }
      },
      [&](int slot) { return Ks ? Ks[slot] : (T)K[(size_t)slot * N + sc]; }, zi_read, [](int) { return P{}; },
      [&](int row, const P &acc) {
        const P own = *zrow(row);
        const size_t at = (size_t)(unsigned)row * (unsigned)nu + c;
        // largest biased exponents of the row of Z and of Y (the row balancing
        // of the emulated contraction), over the panels by atomic maximum;
        // ezy[k] for Z and ezy[N nx + k] for Y, k = sc nx + row
        const auto expo = [](T v) {
          return (unsigned)(((unsigned long long)__double_as_longlong((double)v) >> 52) & 0x7FF);
        };
        unsigned ez = 0, ey = 0;
#pragma unroll
        for (int q = 0; q < C; ++q)
          if (c + q * W < nu) {
            Zs[at + q * W] = own.v[q];
            Ys[at + q * W] = acc.v[q];
            if (ezy) {
              ez = max(ez, expo(own.v[q]));
              ey = max(ey, expo(acc.v[q]));
            }
          }
        if (ezy) {
          const unsigned lanes = W == 32 ? 0xffffffffu : ((1u << W) - 1) << (lane - cl);
          ez = __reduce_max_sync(lanes, ez);
          ey = __reduce_max_sync(lanes, ey);
          if (cl == 0) {
            const size_t k = (size_t)sc * nx + row;
            if (ez) atomicMax(&ezy[k], (int)ez);
            if (ey) atomicMax(&ezy[(size_t)N * nx + k], (int)ey);
          }
        }
      });
  sweep_rows<double, W, C, U, false>(
      1, [&](int l) { return l * nu; },
      [&](int j) { return RowDesc{j, S.ku_ptr[j], S.ku_ptr[j + 1] - S.ku_ptr[j]}; },
      [&](int f, int &col, int &slot) {
        col = S.ku_col[f];
        slot = S.ku_src[f];
      },
      [&](int slot) { return K[(size_t)slot * N + sc]; },
      [&](int p, bool &mine) {
        const P z = zi_read(p, mine);
        Pack<double, C> d;
#pragma unroll
        for (int q = 0; q < C; ++q) d.v[q] = (double)z.v[q];
        return d;
      },
      [](int) { return Pack<double, C>{}; },
      [&](int j, const Pack<double, C> &acc) {
#pragma unroll
        for (int q = 0; q < C; ++q)
          if (c + q * W < nu) Yus[(size_t)j * nu + c + q * W] = acc.v[q];
      });
}

// A CTA works through (scenario, panel) items blockIdx.x, blockIdx.x +
// gridDim.x, ... (the panels of a scenario side by side: they read the same
// factors), each in its own slice of the work buffer.  5 CTAs of 256 threads
// per SM (shared memory and registers sized for it).
template <int W, int C>
__global__ void __launch_bounds__(256, 5) k_zsolve64(DevSym S, int npan, const double *__restrict__ LU,
                                                  const double *__restrict__ rd,
                                                  const double *__restrict__ J,
                                                  const double *__restrict__ K, double *work, double *Z, double *Y,
                                                  double *Yu, const double *__restrict__ gvec,
                                                  double *bvec, int *ezy, int phase) {
  extern __shared__ __align__(16) unsigned char smz[];
  const size_t E = (size_t)S.nx * S.nu;
  for (int it = blockIdx.x; it < npan * S.N; it += gridDim.x) {
    const int sc = it / npan;
    zsolve_panel<double, W, C>(S, sc, it - sc * npan, LU + (size_t)sc * S.nnzLU, rd + (size_t)sc * S.nx, J, K, nullptr,
                               work + (size_t)blockIdx.x * S.nx * (W * C), Z + sc * E, Y + sc * E,
                               Yu + (size_t)sc * S.nu * S.nu, reinterpret_cast<double *>(smz), gvec,
                               bvec ? bvec + (size_t)sc * S.nx : nullptr, ezy, phase);
    __syncthreads();
  }
}

template <int W, int C>
__global__ void __launch_bounds__(256, 5) k_zsolve32(DevSym S, int npan, const float *__restrict__ LUf,
                                                  const float *__restrict__ rdf, const float *__restrict__ Kf,
                                                  const double *__restrict__ J,
                                                  const double *__restrict__ K, float *work, float *Z, float *Y,
                                                  double *Yu, int phase) {
  extern __shared__ __align__(16) unsigned char smz[];
  const size_t E = (size_t)S.nx * S.nu;
  for (int it = blockIdx.x; it < npan * S.N; it += gridDim.x) {
    const int sc = it / npan;
    zsolve_panel<float, W, C>(S, sc, it - sc * npan, LUf + (size_t)sc * round_lu_len(S), rdf + (size_t)sc * S.nx, J, K,
                              Kf, work + (size_t)blockIdx.x * S.nx * (W * C), Z + sc * E, Y + sc * E,
                              Yu + (size_t)sc * S.nu * S.nu, reinterpret_cast<float *>(smz), nullptr,
                              (float *)nullptr, nullptr, phase);
    __syncthreads();
  }
}

// FP32 copies of the factor values the mixed path's solve reads (the whole
// LU, or its sparse part when the trailing block has kernels of its own) and
// of the reciprocal pivots: one conversion per value (12 B each).
__global__ void k_round_factors(DevSym S, const double *__restrict__ LU, const double *__restrict__ rd, float *LUf,
                                float *rdf) {
  const int sc = blockIdx.y, n = round_lu_len(S), p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) LUf[(size_t)sc * n + p] = (float)LU[(size_t)sc * S.nnzLU + p];
  else if (p - n < S.nx) rdf[(size_t)sc * S.nx + p - n] = (float)rd[(size_t)sc * S.nx + p - n];
}

// FP32 copy of K in the order of the row lists of K_x, scenario-major (K
// itself is scenario-fastest): 32 x 32 tiles through shared memory.
__global__ void __launch_bounds__(256) k_round_k(DevSym S, int nk, const double *__restrict__ K, float *Kf) {
  __shared__ float tile[32][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, e0 = blockIdx.x * 32, s0 = blockIdx.y * 32;
  for (int q = w; q < 32; q += 8) {
    const int e = e0 + q, sc = s0 + lane;
    if (e < nk && sc < S.N) tile[q][lane] = (float)K[(size_t)S.kx2[e].y * S.N + sc];
  }
  __syncthreads();
  for (int q = w; q < 32; q += 8) {
    const int e = e0 + lane, sc = s0 + q;
    if (e < nk && sc < S.N) Kf[(size_t)sc * nk + e] = tile[lane][q];
  }
}

// The same factorization by a cluster of two CTAs per scenario (two SMs'
// FP64 units): the sparse part shared by index parity; the nd x nd
// trailing block is then split by column panels of 16, panel q
// held by CTA q mod 2 in its shared memory.  Per panel, factored by its owner
// and copied by the other CTA from the owner's shared memory, each CTA solves
// U12 = L11^{-1} A12 and updates A22 -= L21 U12 on its own columns (4 x 4
// register tiles), the next panel first.  Bound by the FP64 units in the
// updates and by latency elsewhere: 768 us at 1,000 buses x 64 (890 with the
// panels' factorization in turn with the updates and one load in flight in
// the copies: 179 init and sparse levels, 87 trailing-block products, 46 the
// block's load, ~50 per panel).
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(512, 1)
    k_lu_factor_pair(DevSym S, int nL, const double *__restrict__ J, double *LU, double *rd, int *flags,
                     double piv_tol) {
  constexpr int PB = 16;
  __shared__ double sh[32];
  extern __shared__ double Tl[];
  const unsigned rank = cluster_rank();
  const int sc = blockIdx.x >> 1, tid = threadIdx.x, bd = blockDim.x;
  double *A = LU + (size_t)sc * S.nnzLU;
  double *r = rd + (size_t)sc * S.nx;
  const int nd = S.nd, t0 = S.t0, ns = nd;
  const double amax = lu_sparse_part<true>(S, nL, J, A, r, flags, piv_tol, sc, sh, rank, 2);
  if (nd == 0) return;  // the same on both CTAs
  const int np = (ns + PB - 1) / PB, LDL = ((np + 1) / 2) * PB;
  double *Pb = Tl + (size_t)ns * LDL;  // the other CTA's panel [ns][PB]
  // own local column lc <-> block column (2 (lc / PB) + rank) PB + lc % PB;
  // the block is column-major in LU storage (whole column segments per warp,
  // four loads in flight per thread)
  double *D = A + S.dense_base;
  for (int e0 = tid; e0 < ns * LDL; e0 += 4 * bd) {
    double v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int e = e0 + q * bd, lc = e / ns, i = e - lc * ns;
      const int c = (2 * (lc / PB) + (int)rank) * PB + lc % PB;
      v[q] = e < ns * LDL && c < ns ? D[(size_t)c * nd + i] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int e = e0 + q * bd, lc = e / ns, i = e - lc * ns;
      if (e < ns * LDL) Tl[i * LDL + lc] = v[q];
    }
  }
  __syncthreads();
  // Panel p on its owner.  One barrier per column: thread 0 holds row k + 1,
  // so it forms the next pivot's reciprocal (a dependent FP64 division, ~565
  // cycles) as soon as its row has that entry, under the other rows' updates.
  const auto factor = [&](int p) {
    const int kb = p * PB, ke = min(kb + PB, ns), lc0 = (p >> 1) * PB;
    const auto pivot = [&](int k) {
      const double d = Tl[k * LDL + lc0 + (k - kb)];
      if (!(fabs(d) > piv_tol * amax)) flags[FLAG_SINGULAR] = 1;
      const double rk = 1.0 / d;
      r[t0 + k] = rk;
      sh[17 + (k & 1)] = rk;
    };
    if (tid == 0) pivot(kb);
    __syncthreads();
    for (int k = kb; k < ke; ++k) {
      const int lk = lc0 + (k - kb);
      const double rk = sh[17 + (k & 1)];
      for (int i = k + 1 + tid; i < ns; i += bd) {
        const double l = Tl[i * LDL + lk] * rk;
        Tl[i * LDL + lk] = l;
        int j = k + 1;
        if (j < ke) {
          Tl[i * LDL + lk + 1] -= l * Tl[k * LDL + lk + 1];
          if (i == k + 1) pivot(k + 1);
          for (++j; j < ke; ++j) Tl[i * LDL + lc0 + (j - kb)] -= l * Tl[k * LDL + lc0 + (j - kb)];
        }
      }
      __syncthreads();
    }
  };
  if (rank == 0) factor(0);
  cluster_sync_all();
  // Panel p is ready everywhere; the owner of panel p + 1 updates and factors
  // that first and arrives at the barrier, and both update their other
  // columns before waiting there: the factorization of a panel, a chain on
  // one SM, runs under the other SM's updates.
  for (int p = 0; p + 1 < np; ++p) {
    const int kb = p * PB, ke = kb + PB;
    const bool own = (p & 1) == (int)rank, next = !own;
    const double *Lp = Tl;
    int ldp = LDL, cp0 = (p >> 1) * PB;  // the panel's first local column in its owner
    if (!own) {
      for (int e = tid; e < (ns - kb) * PB; e += bd) {
        const int i = kb + e / PB, j = e % PB;
        Pb[i * PB + j] = ld_peer(&Tl[i * LDL + cp0 + j], rank ^ 1u);
      }
      __syncthreads();
      Lp = Pb;
      ldp = PB;
      cp0 = 0;
    }
    // own columns right of the panel: local panels from lcs on
    const int lcs = ((p + 2 - (int)rank) / 2) * PB;
    for (int lj = lcs + tid; lj < LDL; lj += bd) {  // a full panel: only the last can be ragged
      double x[PB];
#pragma unroll
      for (int k = 0; k < PB; ++k) x[k] = Tl[(kb + k) * LDL + lj];
#pragma unroll
      for (int k = 0; k < PB; ++k)
#pragma unroll
        for (int i = k + 1; i < PB; ++i) x[i] -= Lp[(kb + i) * ldp + cp0 + k] * x[k];
#pragma unroll
      for (int k = 1; k < PB; ++k) Tl[(kb + k) * LDL + lj] = x[k];
    }
    __syncthreads();
    // A22 -= L21 U12 on the own columns [j0s, j1)
    const auto update = [&](int j0s, int j1) {
      const int m = ns - ke, nt4r = (m + 3) / 4, nt4c = (j1 - j0s) / 4;
      for (int e = tid; e < nt4r * nt4c; e += bd) {
        const int i0 = ke + (e / nt4c) * 4, j0 = j0s + (e % nt4c) * 4;
        double c[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) c[a][b] = 0.0;
        for (int k = kb; k < ke; ++k) {
          double lv[4], uv[4];
#pragma unroll
          for (int a = 0; a < 4; ++a) lv[a] = i0 + a < ns ? Lp[(i0 + a) * ldp + cp0 + (k - kb)] : 0.0;
#pragma unroll
          for (int b = 0; b < 4; ++b) uv[b] = Tl[k * LDL + j0 + b];
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) c[a][b] = fma(lv[a], uv[b], c[a][b]);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (i0 + a < ns) Tl[(i0 + a) * LDL + j0 + b] -= c[a][b];
      }
    };
    if (next) {
      update(lcs, lcs + PB);
      __syncthreads();
      factor(p + 1);
    }
    cluster_arrive_all();
    update(next ? lcs + PB : lcs, LDL);
    __syncthreads();
    cluster_wait_all();
  }
  cluster_sync_all();  // no CTA leaves while the other may still read its panels
  for (int e = tid; e < ns * LDL; e += bd) {
    const int lc = e / ns, i = e - lc * ns;
    const int c = (2 * (lc / PB) + (int)rank) * PB + lc % PB;
    if (c < ns) D[(size_t)c * nd + i] = Tl[i * LDL + lc];
  }
}
}  // namespace

void launch_lu_factor(const DevSym &S, int nL, const double *J, double *LU, double *rd, int *flags,
                      cudaStream_t st, bool allow_pair, const EmuLuPlan *emu_lu) {
  // trailing sub-block held in shared memory: as large as fits next to the
  // kernel's static shared memory (170 x 170 doubles on GB300)
  static const int ns_max = [] {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    cudaFuncGetAttributes(&fa, k_lu_factor);
    int n = 1;
    while ((size_t)(n + 1) * (n + 1) * sizeof(double) + fa.sharedSizeBytes <= (size_t)optin) ++n;
    return n;
  }();
  // a cluster of two CTAs per scenario when the trailing block fits their
  // shared memory (own columns plus one panel of the other CTA)
  static const size_t pair_cap = [] {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, k_lu_factor_pair) != cudaSuccess) return (size_t)0;
    return raise_smem_cap(k_lu_factor_pair) ? (size_t)optin - fa.sharedSizeBytes : (size_t)0;
  }();
  if (S.big) {
    // sparse part (as many CTAs per scenario as fill the GPU twice, at most
    // 8), then the block by the batched kernels
    const int C = S.N <= 38 ? 8 : S.N <= 76 ? 4 : S.N <= 152 ? 2 : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(S.N * C);
    cfg.blockDim = dim3(512);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_lu_sparse, S, nL, J, LU, rd, flags, 1e-14, C); ipm_count_launch();
    launch_big_lu_dense(S, LU, rd, S.lu_amax, flags, st, emu_lu);
    launch_diag_inverse(S, LU, rd, st);
    return;
  }
  const int np = (S.nd + 15) / 16, ldl = ((np + 1) / 2) * 16;
  const size_t pair_smem = (size_t)S.nd * (ldl + 16) * sizeof(double);
  if (allow_pair && S.nd > 0 && pair_smem <= pair_cap) {
    k_lu_factor_pair<<<2 * S.N, 512, pair_smem, st>>>(S, nL, J, LU, rd, flags, 1e-14);
    ipm_count_launch();
    launch_diag_inverse(S, LU, rd, st);
    return;
  }
  const int ns = S.nd < ns_max ? S.nd : ns_max;
  const size_t smem = (size_t)ns * ns * sizeof(double);
  static const bool cap = raise_smem_cap(k_lu_factor);
  (void)cap;
  k_lu_factor<<<S.N, 512, smem, st>>>(S, nL, J, LU, rd, flags, 1e-14, ns); ipm_count_launch();
  launch_diag_inverse(S, LU, rd, st);
}
// b rides along unless the trailing block has kernels of its own
bool zsolve64_folds_b(const DevSym &S) { return !S.big; }

// CTAs of a multi-RHS solve that are on the GPU at once
constexpr int ZS_CTAS = 5 * 152;

// Columns per panel: 32, or 16 or 8 to spread a small problem over more SMs
// and to level the last wave of a larger one.  Every SM works through
// ceil(panels / 152) panels of w columns, so the width with the least
// w ceil(panels / 152) is taken, the wider at a tie within an eighth (its
// fetches serve more columns).
static int zsolve_width(const DevSym &S, int ncol) {
  if (S.big) return 32;
  int best = 32;
  long long cost = 0;
  for (int w : {32, 16, 8}) {
    const long long items = (long long)((ncol + w - 1) / w) * S.N, c = w * ((items + 151) / 152);
    if (w == 32 || 8 * c < 7 * cost) best = w, cost = c;
  }
  return best;
}
// 128 threads when more panels share an SM than five CTAs of 256 can hold
static int zsolve_cta(long long items, int w, int threads) { return w < 32 && items > ZS_CTAS ? 128 : threads; }
static int zsolve_grid(long long items, int threads) {
  return (int)(items < ZS_CTAS * (256 / threads) ? items : ZS_CTAS * (256 / threads));
}

size_t zsolve_work_bytes(const DevSym &S, size_t elem, int threads) {
  const int ncol = S.nu + (elem == sizeof(double) && zsolve64_folds_b(S) ? 1 : 0), w = zsolve_width(S, ncol);
  const long long items = (long long)((ncol + w - 1) / w) * S.N;
  return (size_t)zsolve_grid(items, zsolve_cta(items, w, threads)) * S.nx * w * elem;
}
// CTAs of a launch: what the GPU holds at once, no more than the work buffer
// has panels for (at least one: a buffer of fewer than 32 columns belongs to a
// problem of panels of 8)
static int zsolve_ctas(long long items, int threads, size_t panel_bytes, size_t work_bytes) {
  return (int)std::min((long long)zsolve_grid(items, threads), (long long)(work_bytes / panel_bytes));
}

template <int W, int C>
static void zsolve64_launch(const DevSym &S, const double *LU, const double *rd, const double *J, const double *K,
                            ZsolveWork work, double *Z, double *Y, double *Yu, cudaStream_t st, int threads,
                            const double *g, double *b, int *ezy, int phase) {
  // dynamic plus static shared memory may pass the 48 KB default
  static const bool cap = raise_smem_cap(k_zsolve64<W, C>);
  (void)cap;
  const int npan = (S.nu + (b ? 1 : 0) + W * C - 1) / (W * C);
  const size_t bytes = phase == 0 ? (size_t)S.nd * W * C * sizeof(double) : 0;
  threads = zsolve_cta((long long)npan * S.N, W * C, threads);
  k_zsolve64<W, C><<<zsolve_ctas((long long)npan * S.N, threads, sizeof(double) * S.nx * W * C, work.bytes), threads,
                     bytes, st>>>(S, npan, LU, rd, J, K, (double *)work.p, Z, Y, Yu, g, b, ezy, phase);
  ipm_count_launch();
}

void launch_zsolve64(const DevSym &S, const double *LU, const double *rd, const double *J,
                     const double *K, ZsolveWork work, double *Z, double *Y, double *Yu, cudaStream_t st, int threads,
                     const double *g, double *b, int *ezy) {
  if (S.big) {
    // the block's right-hand sides, the block by the batched triangular
    // solves, then the sparse rows and products
    zsolve64_launch<16, 2>(S, LU, rd, J, K, work, Z, Y, Yu, st, threads, nullptr, nullptr, ezy, 1);
    launch_big_trsm64(S, LU, rd, Z, st);
    zsolve64_launch<16, 2>(S, LU, rd, J, K, work, Z, Y, Yu, st, threads, nullptr, nullptr, ezy, 2);
    return;
  }
  switch (zsolve_width(S, S.nu + (b ? 1 : 0))) {
    case 8: zsolve64_launch<4, 2>(S, LU, rd, J, K, work, Z, Y, Yu, st, threads, g, b, ezy, 0); break;
    case 16: zsolve64_launch<8, 2>(S, LU, rd, J, K, work, Z, Y, Yu, st, threads, g, b, ezy, 0); break;
    default: zsolve64_launch<16, 2>(S, LU, rd, J, K, work, Z, Y, Yu, st, threads, g, b, ezy, 0);
  }
}

template <int W, int C>
static void zsolve32_launch(const DevSym &S, const RoundedFactors &f, const double *J, const double *K, ZsolveWork work,
                            float *Z, float *Y, double *Yu, cudaStream_t st, int threads, int phase) {
  static const bool cap = raise_smem_cap(k_zsolve32<W, C>);
  (void)cap;
  const int npan = (S.nu + W * C - 1) / (W * C);
  const size_t bytes = phase == 0 ? (size_t)S.nd * W * C * sizeof(float) : 0;
  threads = zsolve_cta((long long)npan * S.N, W * C, threads);
  k_zsolve32<W, C><<<zsolve_ctas((long long)npan * S.N, threads, sizeof(float) * S.nx * W * C, work.bytes), threads,
                     bytes, st>>>(S, npan, f.LUf, f.rdf, f.Kf, J, K, (float *)work.p, Z, Y, Yu, phase);
  ipm_count_launch();
}

void launch_zsolve32(const DevSym &S, const double *LU, const double *rd, const double *J,
                     const double *K, const RoundedFactors &f, ZsolveWork work, float *Z, float *Y, double *Yu,
                     cudaStream_t st, int threads, const TcsPlan *tcs, int *flags) {
  k_round_factors<<<dim3((round_lu_len(S) + S.nx + 255) / 256, S.N), 256, 0, st>>>(S, LU, rd, f.LUf, f.rdf);
  ipm_count_launch();
  k_round_k<<<dim3((f.nk + 31) / 32, (S.N + 31) / 32), 256, 0, st>>>(S, f.nk, K, f.Kf); ipm_count_launch();
  if (S.big) {
    zsolve32_launch<8, 4>(S, f, J, K, work, Z, Y, Yu, st, threads, 1);
    launch_big_trsm32(S, LU, rd, Z, st, tcs, flags);
    zsolve32_launch<8, 4>(S, f, J, K, work, Z, Y, Yu, st, threads, 2);
    return;
  }
  switch (zsolve_width(S, S.nu)) {
    case 8: zsolve32_launch<4, 2>(S, f, J, K, work, Z, Y, Yu, st, threads, 0); break;
    case 16: zsolve32_launch<8, 2>(S, f, J, K, work, Z, Y, Yu, st, threads, 0); break;
    default: zsolve32_launch<8, 4>(S, f, J, K, work, Z, Y, Yu, st, threads, 0);
  }
}
