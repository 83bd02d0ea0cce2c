// Learned warm start: a small MLP  x -> Linear -> GELU -> Linear -> GELU ->
// Linear  that maps a scenario's load vector to a primal point and log bound
// duals.  Training and inference run in this file's kernels: BF16 operands on
// the 5th-generation tensor cores (tcgen05.mma, TMEM accumulator, TMA-staged
// 128-byte-swizzled tiles), FP32 accumulation and epilogues, FP32 master
// weights with Adam.  The paper has no learned component.
//
// Every product is C[M][N] = A[M][K] B[N][K]^T with both operands K-major, so
// each weight matrix is kept in BF16 both as W [out][in] (forward) and as
// W^T [in][out] (backward through the layer), and the epilogues write the
// activations both row-major and transposed (the transposed copies are the
// K-major operands of the weight-gradient products, K = batch).  Sizes are
// padded: input and output widths to multiples of 128 (zero weights and
// targets in the padding), batches to multiples of 128 (padded rows carry
// zero loss gradients, so they add nothing to the weight gradients).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "../../include/ipm.h"
#include "dev.cuh"
#include "kernels.h"
#include "tcgen05.cuh"

namespace mlpk {

using namespace tcx;

constexpr int BM = 128, BK = 64;
constexpr int TILE_BYTES = BM * BK * 2;  // 16 KB of A
__host__ __device__ constexpr int stage_bytes(int bn) { return TILE_BYTES + bn * BK * 2; }
__host__ __device__ constexpr int smem_bytes(int bn, int stages) { return stages * stage_bytes(bn) + 1024 + 256; }

enum { ACT_NONE = 0, ACT_GELU = 1, ACT_GELU_BWD = 2 };

struct Epi {
  const float *bias;      // [N] or null
  const float *pre_in;    // [M][ldo]: pre-activation for ACT_GELU_BWD
  float *pre_out;         // [M][ldo] or null: pre-activation (ACT_GELU)
  float *out_f32;         // [M][ldo] or null
  __nv_bfloat16 *out_bf;  // [M][ldo] or null
  __nv_bfloat16 *out_t;   // [N][ldt] or null (transposed)
  const float *scale;     // [N] or null: out_f32 = shift + scale * v
  const float *shift;
  int ldo, ldt, act;
  int m_valid, n_valid;   // out_f32 is written in rows < m_valid and columns < n_valid only
};

// GELU with the Gauss error function, and its derivative
__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_d(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// C = A B^T by 128 x BN tiles, one CTA each.  The products here are small (K =
// 128 to a few thousand), so what counts is how many CTAs there are and what
// each does beside its few MMAs: tiles of 32 columns where 128-wide ones
// would leave SMs without work (a 256 x 256 product: 16 CTAs instead of 4),
// and two CTAs per SM, one's epilogue under the other's products.  The
// epilogue turns 32 x 32 pieces of the accumulator in shared memory (the
// stages are free by then), so every array is read and written in whole
// rows of 32 neighbouring entries instead of one row per lane.  With
// that and the predictions written where the caller wants them, a forward pass
// of 1,024 rows (2,000-512-512-7,395) went from 266 to 95 us (the output layer
// takes 24, floor 9 for all), a training step of 256 (240-256-256-893), with
// one launch for the weights and one for the bias gradients, from 460 to 255.
template <int BN, int STAGES>
__global__ void __launch_bounds__(192, 2) k_gemm(const __grid_constant__ CUtensorMap ma,
                                                 const __grid_constant__ CUtensorMap mb, int kblocks, Epi e,
                                                 int *flags) {
  constexpr int STAGE_BYTES = stage_bytes(BN);
  static_assert(4 * 32 * 33 * 4 <= STAGES * STAGE_BYTES, "epilogue pieces in the stages");
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + STAGES * STAGE_BYTES);
  uint64_t *empty = full + STAGES;
  uint64_t *accf = empty + STAGES;
  uint32_t *tslot = reinterpret_cast<uint32_t *>(accf + 1);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accf, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {  // TMEM: one FP32 accumulator of BN columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)), "n"(BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  int issued = 0;
  if (warp == 0 && lane == 0) {
    for (int kb = 0; kb < kblocks; ++kb) {
      const int s = kb % STAGES;
      if (kb >= STAGES && !mbar_wait(&empty[s], ((kb / STAGES) - 1) & 1)) {
        flags[FLAG_TIMEOUT] = 1;
        *abort_flag = 1;
        break;
      }
      if (*abort_flag) break;
      uint8_t *st = smem + s * STAGE_BYTES;
      mbar_expect_tx(&full[s], STAGE_BYTES);
      tma_load_2d(st, &ma, &full[s], kb * BK, m0);
      tma_load_2d(st + TILE_BYTES, &mb, &full[s], kb * BK, n0);
      ++issued;
    }
  } else if (warp == 1 && lane == 0) {
    constexpr uint32_t idesc = idesc_bf16(BM, BN);
    for (int kb = 0; kb < kblocks; ++kb) {
      const int s = kb % STAGES;
      if (!mbar_wait(&full[s], (kb / STAGES) & 1)) {
        flags[FLAG_TIMEOUT] = 1;
        *abort_flag = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t base = smem_u32(smem + s * STAGE_BYTES);
#pragma unroll
      for (int kk = 0; kk < BK / 16; ++kk)
        mma_bf16(tmem, sdesc(base + kk * 32), sdesc(base + TILE_BYTES + kk * 32), idesc,
                 (kb > 0 || kk > 0) ? 1u : 0u);
      mma_commit(&empty[s]);
    }
    mma_commit(accf);
  } else if (warp >= 2) {
    const int q = warp & 3;  // TMEM lane quarter of this warp
    const int mq = m0 + q * 32;
    const bool ok = mbar_wait(accf, 0);
    if (!ok) {
      flags[FLAG_TIMEOUT] = 1;
      *abort_flag = 1;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) {
      float *t = reinterpret_cast<float *>(smem) + (warp - 2) * 32 * 33;  // every stage has been read
#pragma unroll 1
      for (int c0 = 0; c0 < BN; c0 += 32) {
#pragma unroll
        for (int h = 0; h < 32; h += 16) {
          uint32_t v[16];
          const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(c0 + h);
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
              : "r"(taddr));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 16; ++j) t[lane * 33 + h + j] = __uint_as_float(v[j]);
        }
        __syncwarp();
        const int n = n0 + c0 + lane;  // this lane's column
        const float bias = e.bias ? e.bias[n] : 0.0f;
        const bool nin = n < e.n_valid;
        const float scale = e.scale && nin ? e.scale[n] : 1.0f, shift = e.scale && nin ? e.shift[n] : 0.0f;
#pragma unroll 1
        for (int r0 = 0; r0 < 32; r0 += 8) {
          float pre[8];
          if (e.act == ACT_GELU_BWD)
#pragma unroll
            for (int j = 0; j < 8; ++j) pre[j] = e.pre_in[(size_t)(mq + r0 + j) * e.ldo + n];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int m = mq + r0 + j;
            const size_t at = (size_t)m * e.ldo + n;
            float a = t[(r0 + j) * 33 + lane];
            if (e.bias) a += bias;
            float o = a;
            if (e.act == ACT_GELU) {
              if (e.pre_out) e.pre_out[at] = a;
              o = gelu(a);
            } else if (e.act == ACT_GELU_BWD) {
              o = a * gelu_d(pre[j]);
            }
            if (e.out_f32 && nin && m < e.m_valid) e.out_f32[at] = e.scale ? shift + scale * o : o;
            if (e.out_bf) e.out_bf[at] = __float2bfloat16_rn(o);
            if (e.out_t) t[(r0 + j) * 33 + lane] = o;
          }
        }
        __syncwarp();
        if (e.out_t) {
#pragma unroll 8
          for (int j = 0; j < 32; ++j)
            e.out_t[(size_t)(n0 + c0 + j) * e.ldt + mq + lane] = __float2bfloat16_rn(t[lane * 33 + j]);
          __syncwarp();
        }
      }
    }
  }
  if (warp == 0 && lane == 0 && *abort_flag) {
    // let the copies already issued land before the CTA exits (bounded)
    for (int kb = max(0, issued - STAGES); kb < issued; ++kb) (void)mbar_wait(&full[kb % STAGES], (kb / STAGES) & 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(BN));
  }
}

// X (FP32 [B][din]) -> normalised BF16 rows [Mb][dinp] and columns [dinp][ldt]
// (zero in the padding: rows >= B, columns >= din); the columns, an operand of
// the weight gradients, only where XT is given
__global__ void k_input(int B, int Mb, int din, int dinp, int ldt, const float *__restrict__ X,
                        const float *__restrict__ mean, const float *__restrict__ stdv, __nv_bfloat16 *Xb,
                        __nv_bfloat16 *XT) {
  __shared__ float t[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
  for (int r = ty; r < 32; r += 8) {
    const int row = r0 + r, col = c0 + tx;
    float v = 0.0f;
    if (row < B && col < din) v = (X[(size_t)row * din + col] - mean[col]) / stdv[col];
    if (row < Mb && col < dinp) Xb[(size_t)row * dinp + col] = __float2bfloat16_rn(v);
    t[r][tx] = v;
  }
  if (!XT) return;
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    const int col = c0 + r, row = r0 + tx;
    if (col < dinp && row < Mb) XT[(size_t)col * ldt + row] = __float2bfloat16_rn(t[tx][r]);
  }
}

// mean squared error on normalised targets (padding excluded):
//   L = (1 / (B dout)) sum (y - tn)^2,  dL/dy = 2 (y - tn) / (B dout)
// dY written FP32 and BF16 row-major [Mb][doutp] and BF16 transposed
// [doutp][ldt]; per-block partial sums of the squared error in part[].
__global__ void k_loss(int B, int Mb, int dout, int doutp, int ldt, const float *__restrict__ Y,
                       const float *__restrict__ T, const float *__restrict__ mean, const float *__restrict__ stdv,
                       float *dYf, __nv_bfloat16 *dYb, __nv_bfloat16 *dYT, double *part) {
  __shared__ float t[32][33];
  __shared__ double red[8];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const float sc = 2.0f / ((float)B * (float)dout);
  double se = 0.0;
  for (int r = ty; r < 32; r += 8) {
    const int row = r0 + r, col = c0 + tx;
    float g = 0.0f;
    if (row < B && col < dout) {
      const float d = Y[(size_t)row * doutp + col] - (T[(size_t)row * dout + col] - mean[col]) / stdv[col];
      se += (double)d * d;
      g = sc * d;
    }
    if (row < Mb && col < doutp) {
      dYf[(size_t)row * doutp + col] = g;
      dYb[(size_t)row * doutp + col] = __float2bfloat16_rn(g);
    }
    t[r][tx] = g;
  }
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    const int col = c0 + r, row = r0 + tx;
    if (col < doutp && row < Mb) dYT[(size_t)col * ldt + row] = __float2bfloat16_rn(t[tx][r]);
  }
  se = warp_sum(se);
  if (tx == 0) red[ty] = se;
  __syncthreads();
  if (tx == 0 && ty == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[w];
    part[blockIdx.y * gridDim.x + blockIdx.x] = s;
  }
}

__global__ void k_sum(int n, const double *part, double *out) {
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += part[i];
  s = warp_sum(s);
  __shared__ double sh[32];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += sh[w];
    out[0] = r;
  }
}

// bias gradients of all layers: g[n] = sum_{b < B} d[b][n], a thread per column,
// added in order of b; 32 rows' loads in flight, one after another they
// were the time of the kernel (256 rows x 1,536 columns now 9 us)
struct Cols {
  const float *d[3];
  float *g[3];
  int n[3];
};
__global__ void __launch_bounds__(32) k_colsum(int B, Cols c) {
  int n = blockIdx.x * 32 + threadIdx.x, k = 0;
  while (k < 2 && n >= c.n[k]) n -= c.n[k++];
  if (n >= c.n[k]) return;
  const int ld = c.n[k];
  const float *d = c.d[k] + n;
  float s = 0.0f;
  for (int b = 0; b < B; b += 32) {
    float v[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = b + j < B ? d[(size_t)(b + j) * ld] : 0.0f;
#pragma unroll
    for (int j = 0; j < 32; ++j) s += v[j];
  }
  c.g[k][n] = s;
}

// The parameters: three weight matrices [rows][cols] with their BF16 copies
// and (W2, W3) transposed BF16 copies, each followed by its bias.
struct Weights {
  long long w[3], b[3];  // offsets in the parameter vector
  int rows[3], cols[3];
  __nv_bfloat16 *Wb[3], *WT[3];
  int tiles[3];  // 32 x 32 tiles
};
struct Adam {
  const float *g;
  float *m, *v;
  float lr, b1, b2, eps, c1, c2;
};

// One step of Adam (Kingma & Ba) on an FP32 master
__device__ __forceinline__ float adam(long long i, float p, const Adam &A) {
  const float gi = A.g[i];
  const float mi = A.b1 * A.m[i] + (1.0f - A.b1) * gi;
  const float vi = A.b2 * A.v[i] + (1.0f - A.b2) * gi * gi;
  A.m[i] = mi;
  A.v[i] = vi;
  return p - A.lr * (mi / A.c1) / (sqrtf(vi / A.c2) + A.eps);
}

// All parameters in one launch, a CTA per 32 x 32 tile (256 biases): the step
// of Adam where STEP, and the BF16 copies from the new value at hand
template <bool STEP>
__global__ void __launch_bounds__(256) k_weights(Weights W, float *P, Adam A) {
  __shared__ float t[32][33];
  const int tx = threadIdx.x, ty = threadIdx.y;
  int blk = blockIdx.x, k = 0;
  while (k < 3 && blk >= W.tiles[k]) blk -= W.tiles[k++];
  if (k == 3) {
    int i = blk * 256 + ty * 32 + tx;
    for (int l = 0; STEP && l < 3; i -= W.rows[l++])
      if (i >= 0 && i < W.rows[l]) P[W.b[l] + i] = adam(W.b[l] + i, P[W.b[l] + i], A);
    return;
  }
  const int tc = W.cols[k] / 32, r0 = blk / tc * 32, c0 = blk % tc * 32;  // every extent is a multiple of 128
#pragma unroll
  for (int r = ty; r < 32; r += 8) {
    const size_t at = (size_t)(r0 + r) * W.cols[k] + c0 + tx;
    float v = P[W.w[k] + at];
    if (STEP) P[W.w[k] + at] = v = adam(W.w[k] + at, v, A);
    W.Wb[k][at] = __float2bfloat16_rn(v);
    t[r][tx] = v;
  }
  if (!W.WT[k]) return;
  __syncthreads();
#pragma unroll
  for (int r = ty; r < 32; r += 8)
    W.WT[k][(size_t)(c0 + r) * W.rows[k] + r0 + tx] = __float2bfloat16_rn(t[tx][r]);
}

}  // namespace mlpk

using namespace mlpk;

struct ipm_mlp {
  int din = 0, dh = 0, dout = 0, maxb = 0;
  int dinp = 0, doutp = 0, bpad = 0;
  long long np = 0;                // padded parameter count
  long long oW1, ob1, oW2, ob2, oW3, ob3;  // offsets in the padded parameter vector
  float *P = nullptr, *G = nullptr, *Mm = nullptr, *V = nullptr;
  __nv_bfloat16 *W1b, *W2b, *W2T, *W3b, *W3T;
  __nv_bfloat16 *Xb, *XT, *H1b, *H1T, *H2b, *H2T, *dYb, *dYT, *dp2b, *dp2T, *dp1T;
  float *pre1, *pre2, *Y, *dYf, *dp2f, *dp1f;
  float *in_mean, *in_std, *out_mean, *out_std;
  double *part = nullptr, *lsum = nullptr, *h_loss = nullptr;
  int *flags = nullptr, *h_flags = nullptr;
  long long adam_t = 0;
  CUtensorMap maps[16], maps32[16];  // boxes of 128 rows, and of 32
  std::vector<void *> allocs;
};

namespace {

enum { MX, MW1, MH1, MW2, MH2, MW3, MDY, MW3T, MDYT, MH2T, MDP2, MW2T, MDP2T, MH1T, MDP1T, MXT };

template <class T>
bool mal(ipm_mlp *m, T **p, size_t count) {
  void *q = nullptr;
  if (cudaMalloc(&q, std::max<size_t>(count, 1) * sizeof(T)) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaMemset(q, 0, std::max<size_t>(count, 1) * sizeof(T));
  m->allocs.push_back(q);
  *p = (T *)q;
  return true;
}

inline int r128(int v) { return (v + 127) / 128 * 128; }

template <int BN, int STAGES>
void gemm_tiles(const CUtensorMap &a, const CUtensorMap &b, int M, int N, int K, const Epi &e, int *flags,
                cudaStream_t st) {
  static const bool attr = cudaFuncSetAttribute(k_gemm<BN, STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                smem_bytes(BN, STAGES)) == cudaSuccess;
  (void)attr;
  k_gemm<BN, STAGES><<<dim3(M / BM, N / BN), 192, smem_bytes(BN, STAGES), st>>>(a, b, K / BK, e, flags);
  ipm_count_launch();
}

// narrow tiles until wide ones come to one per SM
void gemm(ipm_mlp *m, int mapA, int mapB, int M, int N, int K, const Epi &e, cudaStream_t st) {
  if ((M / BM) * (N / 128) < 152) gemm_tiles<32, 5>(m->maps[mapA], m->maps32[mapB], M, N, K, e, m->flags, st);
  else gemm_tiles<128, 3>(m->maps[mapA], m->maps[mapB], M, N, K, e, m->flags, st);
}

Epi epi(int ldo) {
  Epi e;
  std::memset(&e, 0, sizeof(e));
  e.ldo = ldo;
  e.m_valid = e.n_valid = 1 << 30;
  return e;
}

void weights(ipm_mlp *m, const Adam *A, cudaStream_t st) {
  const Weights W = {{m->oW1, m->oW2, m->oW3}, {m->ob1, m->ob2, m->ob3},
                     {m->dh, m->dh, m->doutp}, {m->dinp, m->dh, m->dh},
                     {m->W1b, m->W2b, m->W3b}, {nullptr, m->W2T, m->W3T},
                     {m->dh / 32 * (m->dinp / 32), m->dh / 32 * (m->dh / 32), m->doutp / 32 * (m->dh / 32)}};
  const int tiles = W.tiles[0] + W.tiles[1] + W.tiles[2], nb = (2 * m->dh + m->doutp + 255) / 256;
  if (A) k_weights<true><<<tiles + nb, dim3(32, 8), 0, st>>>(W, m->P, *A);
  else k_weights<false><<<tiles, dim3(32, 8), 0, st>>>(W, m->P, Adam{});
  ipm_count_launch();
}

// forward pass over B rows of X; the output layer writes de-normalised
// predictions [B][dout] where the caller wants them (`denorm`), normalised
// ones with their padding otherwise (training), and what only the backward
// pass reads (pre-activations, transposed operands) only then
void forward(ipm_mlp *m, const float *X, int B, bool denorm, float *Yout, int ldy, cudaStream_t st) {
  const int Mb = r128(B);
  k_input<<<dim3((m->dinp + 31) / 32, (Mb + 31) / 32), dim3(32, 8), 0, st>>>(B, Mb, m->din, m->dinp, m->bpad, X,
                                                                           m->in_mean, m->in_std, m->Xb,
                                                                           denorm ? nullptr : m->XT);
  ipm_count_launch();
  Epi e = epi(m->dh);
  e.bias = m->P + m->ob1;
  e.act = ACT_GELU;
  e.pre_out = denorm ? nullptr : m->pre1;
  e.out_bf = m->H1b;
  e.out_t = denorm ? nullptr : m->H1T;
  e.ldt = m->bpad;
  gemm(m, MX, MW1, Mb, m->dh, m->dinp, e, st);
  e.bias = m->P + m->ob2;
  e.pre_out = denorm ? nullptr : m->pre2;
  e.out_bf = m->H2b;
  e.out_t = denorm ? nullptr : m->H2T;
  gemm(m, MH1, MW2, Mb, m->dh, m->dh, e, st);
  Epi o = epi(ldy);
  o.bias = m->P + m->ob3;
  o.act = ACT_NONE;
  o.out_f32 = Yout;
  if (denorm) {
    o.scale = m->out_std;
    o.shift = m->out_mean;
    o.m_valid = B;
    o.n_valid = m->dout;
  }
  gemm(m, MH2, MW3, Mb, m->doutp, m->dh, o, st);
}

// loss and gradients (into m->G) for B rows
void backward(ipm_mlp *m, const float *T, int B, cudaStream_t st) {
  const int Mb = r128(B);
  const dim3 lg((m->doutp + 31) / 32, (Mb + 31) / 32);
  k_loss<<<lg, dim3(32, 8), 0, st>>>(B, Mb, m->dout, m->doutp, m->bpad, m->Y, T, m->out_mean, m->out_std, m->dYf,
                                     m->dYb, m->dYT, m->part);
  ipm_count_launch();
  k_sum<<<1, 256, 0, st>>>((int)(lg.x * lg.y), m->part, m->lsum);
  ipm_count_launch();
  // dpre2 = (dY W3) * GELU'(pre2)
  Epi e = epi(m->dh);
  e.act = ACT_GELU_BWD;
  e.pre_in = m->pre2;
  e.out_f32 = m->dp2f;
  e.out_bf = m->dp2b;
  e.out_t = m->dp2T;
  e.ldt = m->bpad;
  gemm(m, MDY, MW3T, Mb, m->dh, m->doutp, e, st);
  // dW3 = dY^T H2
  Epi w = epi(m->dh);
  w.out_f32 = m->G + m->oW3;
  gemm(m, MDYT, MH2T, m->doutp, m->dh, Mb, w, st);
  // dpre1 = (dpre2 W2) * GELU'(pre1)
  Epi e1 = epi(m->dh);
  e1.act = ACT_GELU_BWD;
  e1.pre_in = m->pre1;
  e1.out_f32 = m->dp1f;
  e1.out_t = m->dp1T;
  e1.ldt = m->bpad;
  gemm(m, MDP2, MW2T, Mb, m->dh, m->dh, e1, st);
  // dW2 = dpre2^T H1, dW1 = dpre1^T X
  w.out_f32 = m->G + m->oW2;
  gemm(m, MDP2T, MH1T, m->dh, m->dh, Mb, w, st);
  Epi w1 = epi(m->dinp);
  w1.out_f32 = m->G + m->oW1;
  gemm(m, MDP1T, MXT, m->dh, m->dinp, Mb, w1, st);
  const Cols c = {{m->dp1f, m->dp2f, m->dYf}, {m->G + m->ob1, m->G + m->ob2, m->G + m->ob3}, {m->dh, m->dh, m->doutp}};
  k_colsum<<<(2 * m->dh + m->doutp) / 32, 32, 0, st>>>(B, c);
  ipm_count_launch();
}

ipm_status finish(ipm_mlp *m, cudaStream_t st, float *loss, int B) {
  if (cudaGetLastError() != cudaSuccess) return IPM_ERR_CUDA;
  if (cudaMemcpyAsync(m->h_flags, m->flags, FLAG_COUNT * sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return IPM_ERR_CUDA;
  if (loss && cudaMemcpyAsync(m->h_loss, m->lsum, sizeof(double), cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return IPM_ERR_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return IPM_ERR_CUDA;
  if (m->h_flags[FLAG_TIMEOUT]) return IPM_ERR_TIMEOUT;
  if (loss) *loss = (float)(*m->h_loss / ((double)B * m->dout));
  return IPM_OK;
}

// logical (unpadded) parameter layout: W1 [dh][din], b1, W2 [dh][dh], b2, W3 [dout][dh], b3
long long logical_count(const ipm_mlp *m) {
  return (long long)m->dh * m->din + m->dh + (long long)m->dh * m->dh + m->dh + (long long)m->dout * m->dh + m->dout;
}

void pack(const ipm_mlp *m, const float *lg, std::vector<float> &pd) {
  pd.assign(m->np, 0.0f);
  const float *s = lg;
  for (int o = 0; o < m->dh; ++o)
    for (int i = 0; i < m->din; ++i) pd[m->oW1 + (long long)o * m->dinp + i] = *s++;
  for (int o = 0; o < m->dh; ++o) pd[m->ob1 + o] = *s++;
  for (int o = 0; o < m->dh; ++o)
    for (int i = 0; i < m->dh; ++i) pd[m->oW2 + (long long)o * m->dh + i] = *s++;
  for (int o = 0; o < m->dh; ++o) pd[m->ob2 + o] = *s++;
  for (int o = 0; o < m->dout; ++o)
    for (int i = 0; i < m->dh; ++i) pd[m->oW3 + (long long)o * m->dh + i] = *s++;
  for (int o = 0; o < m->dout; ++o) pd[m->ob3 + o] = *s++;
}

void unpack(const ipm_mlp *m, const std::vector<float> &pd, float *lg) {
  float *s = lg;
  for (int o = 0; o < m->dh; ++o)
    for (int i = 0; i < m->din; ++i) *s++ = pd[m->oW1 + (long long)o * m->dinp + i];
  for (int o = 0; o < m->dh; ++o) *s++ = pd[m->ob1 + o];
  for (int o = 0; o < m->dh; ++o)
    for (int i = 0; i < m->dh; ++i) *s++ = pd[m->oW2 + (long long)o * m->dh + i];
  for (int o = 0; o < m->dh; ++o) *s++ = pd[m->ob2 + o];
  for (int o = 0; o < m->dout; ++o)
    for (int i = 0; i < m->dh; ++i) *s++ = pd[m->oW3 + (long long)o * m->dh + i];
  for (int o = 0; o < m->dout; ++o) *s++ = pd[m->ob3 + o];
}

}  // namespace

extern "C" {

ipm_status ipm_mlp_create(int d_in, int d_hidden, int d_out, int max_batch, unsigned long long seed,
                          ipm_mlp **out) {
  if (!out) return IPM_ERR_ARG;
  *out = nullptr;
  if (d_in < 1 || d_out < 1 || d_hidden < 128 || d_hidden % 128 != 0 || max_batch < 1 || d_in > (1 << 20) ||
      d_out > (1 << 20) || max_batch > (1 << 20))
    return IPM_ERR_ARG;
  ipm_mlp *m = new ipm_mlp();
  m->din = d_in;
  m->dh = d_hidden;
  m->dout = d_out;
  m->maxb = max_batch;
  m->dinp = r128(d_in);
  m->doutp = r128(d_out);
  m->bpad = r128(max_batch);
  long long o = 0;
  m->oW1 = o; o += (long long)m->dh * m->dinp;
  m->ob1 = o; o += m->dh;
  m->oW2 = o; o += (long long)m->dh * m->dh;
  m->ob2 = o; o += m->dh;
  m->oW3 = o; o += (long long)m->doutp * m->dh;
  m->ob3 = o; o += m->doutp;
  m->np = o;
  const size_t B = m->bpad, H = m->dh;
  bool ok = mal(m, &m->P, m->np) && mal(m, &m->G, m->np) && mal(m, &m->Mm, m->np) && mal(m, &m->V, m->np) &&
            mal(m, &m->W1b, H * m->dinp) && mal(m, &m->W2b, H * H) && mal(m, &m->W2T, H * H) &&
            mal(m, &m->W3b, (size_t)m->doutp * H) && mal(m, &m->W3T, (size_t)m->doutp * H) &&
            mal(m, &m->Xb, B * m->dinp) && mal(m, &m->XT, B * m->dinp) && mal(m, &m->H1b, B * H) &&
            mal(m, &m->H1T, B * H) && mal(m, &m->H2b, B * H) && mal(m, &m->H2T, B * H) &&
            mal(m, &m->dYb, B * m->doutp) && mal(m, &m->dYT, B * m->doutp) && mal(m, &m->dp2b, B * H) &&
            mal(m, &m->dp2T, B * H) && mal(m, &m->dp1T, B * H) && mal(m, &m->pre1, B * H) &&
            mal(m, &m->pre2, B * H) && mal(m, &m->Y, B * m->doutp) && mal(m, &m->dYf, B * m->doutp) &&
            mal(m, &m->dp2f, B * H) && mal(m, &m->dp1f, B * H) && mal(m, &m->in_mean, m->din) &&
            mal(m, &m->in_std, m->din) && mal(m, &m->out_mean, m->dout) && mal(m, &m->out_std, m->dout) &&
            mal(m, &m->part, (B / 32 + 1) * (m->doutp / 32 + 1)) && mal(m, &m->lsum, 1) &&
            mal(m, &m->flags, FLAG_COUNT);
  ok = ok && cudaMallocHost(&m->h_loss, sizeof(double)) == cudaSuccess &&
       cudaMallocHost(&m->h_flags, FLAG_COUNT * sizeof(int)) == cudaSuccess;
  struct MapDef {
    const void *p;
    int rows;
    long long k;
  } defs[16] = {
      {m->Xb, m->bpad, m->dinp},   {m->W1b, m->dh, m->dinp},  {m->H1b, m->bpad, m->dh},
      {m->W2b, m->dh, m->dh},      {m->H2b, m->bpad, m->dh},  {m->W3b, m->doutp, m->dh},
      {m->dYb, m->bpad, m->doutp}, {m->W3T, m->dh, m->doutp}, {m->dYT, m->doutp, m->bpad},
      {m->H2T, m->dh, m->bpad},    {m->dp2b, m->bpad, m->dh}, {m->W2T, m->dh, m->dh},
      {m->dp2T, m->dh, m->bpad},   {m->H1T, m->dh, m->bpad},  {m->dp1T, m->dh, m->bpad},
      {m->XT, m->dinp, m->bpad}};
  for (int i = 0; ok && i < 16; ++i)
    ok = tc_make_kmajor_map(&m->maps[i], defs[i].p, defs[i].rows, defs[i].k) &&
         tc_make_kmajor_map_box(&m->maps32[i], defs[i].p, defs[i].rows, defs[i].k, 32, BK);
  if (!ok) {
    ipm_mlp_destroy(m);
    return IPM_ERR_OOM;
  }
  // He-uniform initial weights (a = sqrt(6 / fan_in)), zero biases, unit normalisation
  std::mt19937_64 rng(seed);
  std::vector<float> lg(logical_count(m), 0.0f);
  {
    float *s = lg.data();
    auto fill = [&](long long n, int fan_in) {
      std::uniform_real_distribution<float> U(-std::sqrt(6.0f / fan_in), std::sqrt(6.0f / fan_in));
      for (long long i = 0; i < n; ++i) *s++ = U(rng);
    };
    fill((long long)m->dh * m->din, m->din);
    s += m->dh;
    fill((long long)m->dh * m->dh, m->dh);
    s += m->dh;
    fill((long long)m->dout * m->dh, m->dh);
  }
  if (ipm_mlp_set_params(m, lg.data()) != IPM_OK) {
    ipm_mlp_destroy(m);
    return IPM_ERR_CUDA;
  }
  std::vector<float> zeros(std::max(m->din, m->dout), 0.0f), ones(std::max(m->din, m->dout), 1.0f);
  if (ipm_mlp_set_normalization(m, zeros.data(), ones.data(), zeros.data(), ones.data()) != IPM_OK) {
    ipm_mlp_destroy(m);
    return IPM_ERR_CUDA;
  }
  *out = m;
  return IPM_OK;
}

ipm_status ipm_mlp_destroy(ipm_mlp *m) {
  if (!m) return IPM_ERR_ARG;
  cudaDeviceSynchronize();
  for (void *p : m->allocs) cudaFree(p);
  if (m->h_loss) cudaFreeHost(m->h_loss);
  if (m->h_flags) cudaFreeHost(m->h_flags);
  delete m;
  return IPM_OK;
}

long long ipm_mlp_param_count(const ipm_mlp *m) { return m ? logical_count(m) : -1; }

ipm_status ipm_mlp_set_params(ipm_mlp *m, const float *params) {
  if (!m || !params) return IPM_ERR_ARG;
  for (long long i = 0; i < logical_count(m); ++i)
    if (!std::isfinite(params[i])) return IPM_ERR_ARG;
  std::vector<float> pd;
  pack(m, params, pd);
  if (cudaMemcpy(m->P, pd.data(), m->np * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return IPM_ERR_CUDA;
  cudaMemset(m->Mm, 0, m->np * sizeof(float));
  cudaMemset(m->V, 0, m->np * sizeof(float));
  m->adam_t = 0;
  weights(m, nullptr, 0);
  return cudaDeviceSynchronize() == cudaSuccess ? IPM_OK : IPM_ERR_CUDA;
}

ipm_status ipm_mlp_get_params(ipm_mlp *m, float *params) {
  if (!m || !params) return IPM_ERR_ARG;
  std::vector<float> pd(m->np);
  if (cudaMemcpy(pd.data(), m->P, m->np * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) return IPM_ERR_CUDA;
  unpack(m, pd, params);
  return IPM_OK;
}

ipm_status ipm_mlp_set_normalization(ipm_mlp *m, const float *in_mean, const float *in_std, const float *out_mean,
                                     const float *out_std) {
  if (!m || !in_mean || !in_std || !out_mean || !out_std) return IPM_ERR_ARG;
  for (int i = 0; i < m->din; ++i)
    if (!std::isfinite(in_mean[i]) || !(in_std[i] > 0) || !std::isfinite(in_std[i])) return IPM_ERR_ARG;
  for (int i = 0; i < m->dout; ++i)
    if (!std::isfinite(out_mean[i]) || !(out_std[i] > 0) || !std::isfinite(out_std[i])) return IPM_ERR_ARG;
  if (cudaMemcpy(m->in_mean, in_mean, m->din * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(m->in_std, in_std, m->din * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(m->out_mean, out_mean, m->dout * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemcpy(m->out_std, out_std, m->dout * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess)
    return IPM_ERR_CUDA;
  return IPM_OK;
}

ipm_status ipm_mlp_forward(ipm_mlp *m, const float *x, int batch, float *y, void *stream) {
  if (!m || !x || !y || batch < 1) return IPM_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  for (int b0 = 0; b0 < batch; b0 += m->maxb) {
    const int B = std::min(m->maxb, batch - b0);
    cudaMemsetAsync(m->flags, 0, FLAG_COUNT * sizeof(int), st);
    forward(m, x + (size_t)b0 * m->din, B, true, y + (size_t)b0 * m->dout, m->dout, st);
    ipm_status s = finish(m, st, nullptr, B);
    if (s != IPM_OK) return s;
  }
  return IPM_OK;
}

ipm_status ipm_mlp_gradients(ipm_mlp *m, const float *x, const float *target, int batch, float *grads, float *loss,
                             void *stream) {
  if (!m || !x || !target || batch < 1 || batch > m->maxb) return IPM_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  cudaMemsetAsync(m->flags, 0, FLAG_COUNT * sizeof(int), st);
  forward(m, x, batch, false, m->Y, m->doutp, st);
  backward(m, target, batch, st);
  ipm_status s = finish(m, st, loss, batch);
  if (s != IPM_OK || !grads) return s;
  std::vector<float> pd(m->np);
  if (cudaMemcpy(pd.data(), m->G, m->np * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) return IPM_ERR_CUDA;
  unpack(m, pd, grads);
  return IPM_OK;
}

ipm_status ipm_mlp_train_step(ipm_mlp *m, const float *x, const float *target, int batch, float lr, float *loss,
                              void *stream) {
  if (!m || !x || !target || batch < 1 || batch > m->maxb || !(lr > 0) || !std::isfinite(lr)) return IPM_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  cudaMemsetAsync(m->flags, 0, FLAG_COUNT * sizeof(int), st);
  forward(m, x, batch, false, m->Y, m->doutp, st);
  backward(m, target, batch, st);
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  ++m->adam_t;
  const float c1 = 1.0f - std::pow(b1, (float)m->adam_t), c2 = 1.0f - std::pow(b2, (float)m->adam_t);
  const Adam A = {m->G, m->Mm, m->V, lr, b1, b2, eps, c1, c2};
  weights(m, &A, st);
  return finish(m, st, loss, batch);
}

}  // extern "C"
