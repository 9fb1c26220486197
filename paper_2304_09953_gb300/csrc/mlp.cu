// Triage surrogate network on the tensor cores (paper Sec. 3.5: an affinity
// predictor on ligand features, trained on data the workflow generates).
//
// MLP 256 -> 512 -> 512 -> 512 -> 1, ReLU on hidden layers.  Weights and
// activations in BF16, products accumulated in FP32 by mma.sync m16n8k16,
// FP32 master weights updated by Adam.  Products of a training step:
//   forward      H_l = relu(H_{l-1} W_l + b_l)        A row-major, B row-major
//   data grad    dH_{l-1} = dZ_l W_l^T (then ReLU mask) A row-major, B = W^T
//   weight grad  dW_l = H_{l-1}^T dZ_l                 A = H^T,      B row-major
// The first two run on tcgen05 (mlp_tc05.cu) or, with LIGATE_MLP_GEMM=mma, on
// gemm_kernel here; the weight gradients of all layers are one launch
// (grads_kernel).  ldmatrix (.trans where the tile is stored k-major) feeds
// the fragments.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "ligate_internal.h"
#include "mlp.h"

namespace ligate {
namespace mlp {

constexpr int BM = 128, BN = 128, BKT = 32, PAD = 8;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void ldsm_x4(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3,
                                        const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(smem_u32(p)));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3,
                                          const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(smem_u32(p)));
}
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// C[M][N] = sum_k A(m,k) B(k,n).  A(m,k) = A[m*sAm + k], B(k,n) = B[k*sBk +
// n*sBn]; B's contiguous dimension (stride 1) is given by the template flag;
// contiguous dimensions must be multiples of 8 elements with 16 B aligned
// rows; the other dimension is bounds-checked (zero fill).
template <bool B_KCONTIG, int EPI>
__global__ void __launch_bounds__(256) gemm_kernel(GemmArgs g) {
  // B tile: [BN][BKT+PAD] if k-contiguous else [BKT][BN+PAD].
  __shared__ __align__(16) __nv_bfloat16 As[BM * (BKT + PAD)];
  __shared__ __align__(16) __nv_bfloat16 Bs[B_KCONTIG ? BN * (BKT + PAD) : BKT * (BN + PAD)];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp >> 2, wn = warp & 3;  // 2 x 4 warps, warp tile 64 x 32
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  float acc[4][4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;

  const __nv_bfloat16 *A = g.A, *B = g.B;
  for (int k0 = 0; k0 < g.K; k0 += BKT) {
    // ---- global -> shared
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int c = tid + r * 256;  // 512 16-byte chunks per tile
      uint4 v = make_uint4(0, 0, 0, 0);
      {
        const int row = c >> 2, kc = (c & 3) * 8;
        const int m = m0 + row, k = k0 + kc;
        if (m < g.M && k < g.K) v = *reinterpret_cast<const uint4 *>(A + (size_t)m * g.sAm + k);
        *reinterpret_cast<uint4 *>(&As[row * (BKT + PAD) + kc]) = v;
      }
      uint4 w = make_uint4(0, 0, 0, 0);
      if (B_KCONTIG) {
        const int row = c >> 2, kc = (c & 3) * 8;
        const int n = n0 + row, k = k0 + kc;
        if (n < g.N && k < g.K) w = *reinterpret_cast<const uint4 *>(B + (size_t)n * g.sBn + k);
        *reinterpret_cast<uint4 *>(&Bs[row * (BKT + PAD) + kc]) = w;
      } else {
        const int krow = c >> 4, nc = (c & 15) * 8;
        const int n = n0 + nc, k = k0 + krow;
        if (k < g.K && n < g.N) w = *reinterpret_cast<const uint4 *>(B + (size_t)k * g.sBk + n);
        *reinterpret_cast<uint4 *>(&Bs[krow * (BN + PAD) + nc]) = w;
      }
    }
    __syncthreads();
    // ---- tensor-core products over the two k16 steps of the tile
#pragma unroll
    for (int ks = 0; ks < BKT; ks += 16) {
      uint32_t af[4][4], bf[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int mb = wm * 64 + i * 16;
        const __nv_bfloat16 *p = &As[(mb + (lane & 15)) * (BKT + PAD) + ks + (lane >> 4) * 8];
        ldsm_x4(af[i][0], af[i][1], af[i][2], af[i][3], p);
      }
#pragma unroll
      for (int j = 0; j < 4; j += 2) {
        const int nb = wn * 32 + j * 8;
        if (B_KCONTIG) {
          // lanes 0-7: n 0-7 k0 | 8-15: n 0-7 k8 | 16-23: n 8-15 k0 | 24-31: n 8-15 k8
          const int r = lane & 7, ki = (lane >> 3) & 1, ni = lane >> 4;
          const __nv_bfloat16 *p = &Bs[(nb + ni * 8 + r) * (BKT + PAD) + ks + ki * 8];
          ldsm_x4(bf[j][0], bf[j][1], bf[j + 1][0], bf[j + 1][1], p);
        } else {
          const int r = lane & 7, ki = (lane >> 3) & 1, ni = lane >> 4;
          const __nv_bfloat16 *p = &Bs[(ks + ki * 8 + r) * (BN + PAD) + nb + ni * 8];
          ldsm_x4_t(bf[j][0], bf[j][1], bf[j + 1][0], bf[j + 1][1], p);
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], af[i], bf[j][0], bf[j][1]);
    }
    __syncthreads();
  }
  // ---- epilogue
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int m = m0 + wm * 64 + i * 16 + (lane >> 2) + h * 8;
        const int n = n0 + wn * 32 + j * 8 + (lane & 3) * 2;
        if (m >= g.M || n >= g.N) continue;
        float v0 = acc[i][j][2 * h], v1 = acc[i][j][2 * h + 1];
        if (EPI == EPI_BIAS_RELU) {
          v0 = fmaxf(v0 + g.bias[n], 0.f);
          v1 = fmaxf(v1 + g.bias[n + 1], 0.f);
          *reinterpret_cast<__nv_bfloat162 *>(g.Cb + (size_t)m * g.ldc + n) = __floats2bfloat162_rn(v0, v1);
        } else {
          const __nv_bfloat162 hm = *reinterpret_cast<const __nv_bfloat162 *>(g.mask + (size_t)m * g.ldc + n);
          if (!(__bfloat162float(hm.x) > 0.f)) v0 = 0.f;
          if (!(__bfloat162float(hm.y) > 0.f)) v1 = 0.f;
          *reinterpret_cast<__nv_bfloat162 *>(g.Cb + (size_t)m * g.ldc + n) = __floats2bfloat162_rn(v0, v1);
        }
      }
}

template <bool BKc, int EPI>
static cudaError_t gemm_t(const GemmArgs &g, cudaStream_t s) {
  dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM);
  gemm_kernel<BKc, EPI><<<grid, 256, 0, s>>>(g);
  return cudaGetLastError();
}

cudaError_t gemm(int kind, const GemmArgs &g, cudaStream_t s) {
  return kind == GEMM_FWD ? gemm_t<false, EPI_BIAS_RELU>(g, s) : gemm_t<true, EPI_RELU_MASK>(g, s);
}

// ---------------------------------------------------------------------------
// All parameter gradients of one training step in one launch: for each hidden
// layer the weight gradient dW = H^T dZ (128 x 64 tiles, mma.sync m16n8k16,
// rows as k) and the column sums of dZ (bias gradients), and the head's
// gw4[k] = sum_b H3[b][k] dy[b] and gb4 = sum_b dy[b].  Rows stream through a
// four-stage cp.async ring of 64-row slices.
//
// What bounds it: every sum runs over the rows in ascending order, so it is a
// serial chain per output (the MMA steps of a tile; one addition per row of a
// column sum), and the operands come from L2 once per tile row and column: 80
// tiles + 32 column CTAs, one wave, 31 MB at 1,024 rows (64 x 32 tiles, twice
// the traffic, took 17.7 us against 13.8).  Before, the sums ran as launches of
// their own on 2 and 4 CTAs with every load on the chain and the weight
// gradients on 8 to 16 CTAs without overlap: 87 + 3 x 61 + 3 x 37 us per step
// of 1,024 rows (serialised, cold).
constexpr int GK = 64, GM = 128, GN = 64, GC = 64, GSTAGES = 4;  // rows per slice, tile, columns of a sum CTA
constexpr int GT = 256;  // threads
constexpr int GA_LD = GM + 8, GB_LD = GN + 8, GC_LD = GC + 8;
constexpr int G_STAGE = GK * (GA_LD + GB_LD);  // elements per stage (a sum CTA's slice is smaller)
static_assert(GK * GC_LD <= G_STAGE, "column slices fit the stage");

__device__ __forceinline__ void cp16(void *dst, const void *src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src), "r"(in ? 16 : 0)
               : "memory");
}
// rows [k0, k0 + GK) x COLS columns from column c0 of src [rows][ld] into dst (zero past the last row)
template <int COLS, int LD>
__device__ __forceinline__ void load_slice(__nv_bfloat16 *dst, const __nv_bfloat16 *src, int ld, int c0, int k0,
                                           int rows) {
  constexpr int CH = COLS / 8;
#pragma unroll
  for (int c = threadIdx.x; c < GK * CH; c += GT) {
    const int r = c / CH, q = c % CH * 8;
    const bool in = k0 + r < rows;
    cp16(dst + r * LD + q, src + (size_t)(in ? k0 + r : 0) * ld + c0 + q, in);
  }
}

__global__ void __launch_bounds__(GT) grads_kernel(const GradArgs a) {
  extern __shared__ __align__(16) unsigned char graw[];
  __nv_bfloat16 *const ring = reinterpret_cast<__nv_bfloat16 *>(graw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int slices = (a.rows + GK - 1) / GK;
  pdl_wait();
  int t = blockIdx.x;
  int layer = 0;
  for (; layer < 3; ++layer) {  // a weight tile of this layer?
    const int n = (a.fan_in[layer] / GM) * (512 / GN);
    if (t < n) break;
    t -= n;
  }
  if (layer < 3) {
    const int m0 = t / (512 / GN) * GM, n0 = t % (512 / GN) * GN;
    const int mb = (warp >> 1) * 32, nb = (warp & 1) * 32;  // 4 x 2 warps of 32 x 32
    auto load = [&](int s) {
      __nv_bfloat16 *st = ring + (s % GSTAGES) * G_STAGE;
      load_slice<GM, GA_LD>(st, a.in[layer], a.fan_in[layer], m0, s * GK, a.rows);
      load_slice<GN, GB_LD>(st + GK * GA_LD, a.dz[layer], 512, n0, s * GK, a.rows);
    };
    float acc[2][4][4] = {};
    for (int s = 0; s < GSTAGES - 1; ++s) {
      if (s < slices) load(s);
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    for (int s = 0; s < slices; ++s) {
      asm volatile("cp.async.wait_group %0;\n" ::"n"(GSTAGES - 2) : "memory");
      __syncthreads();
      if (s + GSTAGES - 1 < slices) load(s + GSTAGES - 1);  // the stage read in the last iteration
      asm volatile("cp.async.commit_group;\n" ::: "memory");
      const __nv_bfloat16 *As = ring + (s % GSTAGES) * G_STAGE, *Bs = As + GK * GA_LD;
      const int r = lane & 7, q1 = (lane >> 3) & 1, q2 = lane >> 4;
#pragma unroll
      for (int ks = 0; ks < GK; ks += 16) {
        uint32_t af[2][4], bf[4][2];
#pragma unroll
        for (int i = 0; i < 2; ++i)
          ldsm_x4_t(af[i][0], af[i][1], af[i][2], af[i][3], As + (ks + q2 * 8 + r) * GA_LD + mb + i * 16 + q1 * 8);
#pragma unroll
        for (int j = 0; j < 4; j += 2)
          ldsm_x4_t(bf[j][0], bf[j][1], bf[j + 1][0], bf[j + 1][1], Bs + (ks + q1 * 8 + r) * GB_LD + nb + j * 8 + q2 * 8);
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], af[i], bf[j][0], bf[j][1]);
      }
    }
    float *dw = a.dw[layer];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int m = m0 + mb + i * 16 + (lane >> 2) + h * 8, n = n0 + nb + j * 8 + (lane & 3) * 2;
          *reinterpret_cast<float2 *>(dw + (size_t)m * 512 + n) = make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
        }
    return;
  }
  // column sums: 3 x 8 CTAs of the bias gradients, then 8 of the head
  const int what = t / (512 / GC), c0 = t % (512 / GC) * GC;
  const bool head = what == 3;
  const __nv_bfloat16 *src = head ? a.h3 : a.dz[what];
  __shared__ float dys[GSTAGES][GK];
  auto load = [&](int s) {
    load_slice<GC, GC_LD>(ring + (s % GSTAGES) * G_STAGE, src, 512, c0, s * GK, a.rows);
    if (head && tid < GK) dys[s % GSTAGES][tid] = s * GK + tid < a.rows ? a.dy[s * GK + tid] : 0.f;
  };
  float sum = 0.f;
  for (int s = 0; s < GSTAGES - 1; ++s) {
    if (s < slices) load(s);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  }
  for (int s = 0; s < slices; ++s) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(GSTAGES - 2) : "memory");
    __syncthreads();
    if (s + GSTAGES - 1 < slices) load(s + GSTAGES - 1);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    const __nv_bfloat16 *col = ring + (s % GSTAGES) * G_STAGE + tid;
    const float *dy = dys[s % GSTAGES];
    if (tid < GC) {
      if (head) {
#pragma unroll 16
        for (int r = 0; r < GK; ++r) sum = fmaf(__bfloat162float(col[r * GC_LD]), dy[r], sum);
      } else {
#pragma unroll 16
        for (int r = 0; r < GK; ++r) sum += __bfloat162float(col[r * GC_LD]);
      }
    } else if (tid == GC && head && c0 == 0) {
#pragma unroll 16
      for (int r = 0; r < GK; ++r) sum += dy[r];
    }
  }
  if (tid < GC) (head ? a.gw4 : a.db[what])[c0 + tid] = sum;
  else if (tid == GC && head && c0 == 0) a.gb4[0] = sum;
}

cudaError_t grads(const GradArgs &a, cudaStream_t s) {
  const int smem = GSTAGES * G_STAGE * 2;
  cudaError_t e = cudaFuncSetAttribute(grads_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  int ctas = 4 * (512 / GC);
  for (int l = 0; l < 3; ++l) ctas += (a.fan_in[l] / GM) * (512 / GN);
  return launch_pdl(grads_kernel, dim3(ctas), dim3(GT), smem, s, a);
}

// ---------------------------------------------------------------------------
// Small kernels of a training / inference step.

// Standardise gathered rows: x[b][f] = bf16((desc[idx[b]][f] - mu[f]) * inv_sd[f]).
__global__ void gather_std_kernel(const float *__restrict__ desc, const int *__restrict__ idx,
                                  int rows, int row0, const float *__restrict__ mu,
                                  const float *__restrict__ inv_sd, const float *__restrict__ labels,
                                  float ly_mu, float ly_inv, __nv_bfloat16 *__restrict__ x,
                                  float *__restrict__ t) {
  const int b = blockIdx.x;
  pdl_wait();
  if (b >= rows) return;
  const int src = idx ? idx[b] : row0 + b;
  for (int f = threadIdx.x; f < 256; f += blockDim.x)
    x[(size_t)b * 256 + f] = __float2bfloat16_rn((desc[(size_t)src * 256 + f] - mu[f]) * inv_sd[f]);
  if (t && threadIdx.x == 0) t[b] = (labels[src] - ly_mu) * ly_inv;
}

// Last layer y[b] = H3[b] . w4 + b4 (one warp per row); with targets, also
// dy = 2 (y - t) / B, the squared error sum, and dZ3 = dy w4^T masked by
// H3 > 0 (BF16).
__device__ __forceinline__ void head_row(const __nv_bfloat16 *__restrict__ h3, const __nv_bfloat16 *__restrict__ w4,
                                         const float *__restrict__ b4, const float *__restrict__ t,
                                         float *__restrict__ y, float *__restrict__ dy, float inv_b2,
                                         __nv_bfloat16 *__restrict__ dz3, int warp, int lane, double *sq) {
  const __nv_bfloat16 *h = h3 + (size_t)warp * 512;
  float hv[16], wv[16];  // columns lane, lane + 32, ...
#pragma unroll
  for (int k = 0; k < 16; ++k) { hv[k] = __bfloat162float(h[lane + 32 * k]); wv[k] = __bfloat162float(w4[lane + 32 * k]); }
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < 16; ++k) s = fmaf(hv[k], wv[k], s);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  s += b4[0];
  if (lane == 0 && y) y[warp] = s;
  if (!t) return;
  const float e = s - t[warp];
  const float d = inv_b2 * e;  // 2 (y - t) / B
  if (lane == 0) {
    dy[warp] = d;
    *sq = (double)e * e;
  }
#pragma unroll
  for (int k = 0; k < 16; ++k)
    dz3[(size_t)warp * 512 + lane + 32 * k] = __float2bfloat16_rn(hv[k] > 0.f ? d * wv[k] : 0.f);
}

__global__ void head_kernel(const __nv_bfloat16 *__restrict__ h3, const __nv_bfloat16 *__restrict__ w4,
                            const float *__restrict__ b4, int rows, const float *__restrict__ t,
                            float *__restrict__ y, float *__restrict__ dy, float inv_b2,
                            double *__restrict__ sse, __nv_bfloat16 *__restrict__ dz3) {
  __shared__ double sq[8];  // squared errors of the CTA's 8 rows: one atomic per CTA
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x < 8) sq[threadIdx.x] = 0.0;
  __syncthreads();
  pdl_wait();
  if (warp < rows) head_row(h3, w4, b4, t, y, dy, inv_b2, dz3, warp, lane, &sq[threadIdx.x >> 5]);
  if (!t) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    double e2 = 0.0;
    for (int q = 0; q < 8; ++q) e2 += sq[q];
    atomicAdd(sse, e2);
  }
}
// Adam (Kingma & Ba, Algorithm 1) on FP32 master weights, then their BF16
// copies: row-major wb and, for tcgen05, the transposed hidden weights wt.  A
// CTA of 256 threads owns a 32 x 32 tile of a hidden weight matrix (transposed
// through shared memory) or 1,024 of the remaining parameters; one launch in
// place of an elementwise pass and three transposes that read the weights
// again (6.2 + 10.6 us per step, serialised, to 6.3).
struct AdamArgs {
  float *w;
  const float *g;
  float *m, *v;
  __nv_bfloat16 *wb, *wt;
  int off[3], K[3], wt_off[3];  // hidden layers: weights at w + off, [K][512]
  int rest0[4], rest1[4];       // the other parameters' ranges
  float lr, b1, b2, eps, c1, c2;
};

__device__ __forceinline__ __nv_bfloat16 adam_one(const AdamArgs &a, int i) {
  const float gi = a.g[i];
  // products and sums written out: the rounding does not depend on how a
  // compiler contracts them
  const float mi = fmaf(1.f - a.b1, gi, __fmul_rn(a.b1, a.m[i]));
  const float vi = fmaf(__fmul_rn(1.f - a.b2, gi), gi, __fmul_rn(a.b2, a.v[i]));
  a.m[i] = mi;
  a.v[i] = vi;
  const float wi = a.w[i] - a.lr * (mi * a.c1) / (sqrtf(vi * a.c2) + a.eps);
  a.w[i] = wi;
  const __nv_bfloat16 b = __float2bfloat16_rn(wi);
  a.wb[i] = b;
  return b;
}

__global__ void __launch_bounds__(256) adam_kernel(const AdamArgs a) {
  __shared__ __nv_bfloat16 tile[32][34];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  pdl_wait();
  int t = blockIdx.x;
  for (int l = 0; l < 3; ++l) {
    const int n = a.K[l] / 32 * 16;
    if (t >= n) { t -= n; continue; }
    const int k0 = t / 16 * 32, n0 = t % 16 * 32;
#pragma unroll
    for (int q = 0; q < 4; ++q) tile[ty + 8 * q][tx] = adam_one(a, a.off[l] + (k0 + ty + 8 * q) * 512 + n0 + tx);
    if (!a.wt) return;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q)
      a.wt[a.wt_off[l] + (size_t)(n0 + ty + 8 * q) * a.K[l] + k0 + tx] = tile[tx][ty + 8 * q];
    return;
  }
  for (int r = 0; r < 4; ++r) {
    const int n = (a.rest1[r] - a.rest0[r] + 1023) / 1024;
    if (t >= n) { t -= n; continue; }
    for (int q = threadIdx.x; q < 1024; q += 256) {
      const int i = a.rest0[r] + t * 1024 + q;
      if (i < a.rest1[r]) adam_one(a, i);
    }
    return;
  }
}

__global__ void to_bf16_kernel(const float *__restrict__ a, __nv_bfloat16 *__restrict__ b, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    b[i] = __float2bfloat16_rn(a[i]);
}

// Per-feature mean and 1/std (population; zero spread -> 1) of desc[n][256],
// accumulated in FP64: one block per feature.
__global__ void feature_stats_kernel(const float *__restrict__ desc, int n, float *__restrict__ mu,
                                     float *__restrict__ inv_sd) {
  const int f = blockIdx.x;
  __shared__ double s1[256], s2[256];
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double v = desc[(size_t)i * 256 + f];
    a += v;
    b += v * v;
  }
  s1[threadIdx.x] = a;
  s2[threadIdx.x] = b;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) { s1[threadIdx.x] += s1[threadIdx.x + o]; s2[threadIdx.x] += s2[threadIdx.x + o]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double m = s1[0] / n;
    double var = s2[0] / n - m * m;
    if (var < 0) var = 0;
    const double sd = sqrt(var);
    mu[f] = (float)m;
    inv_sd[f] = sd > 1e-12 ? (float)(1.0 / sd) : 1.f;
  }
}

// Mean and std of labels[n] (FP64), single block.
__global__ void label_stats_kernel(const float *__restrict__ y, int n, double *__restrict__ out) {
  __shared__ double s1[256], s2[256];
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) { a += y[i]; b += (double)y[i] * y[i]; }
  s1[threadIdx.x] = a;
  s2[threadIdx.x] = b;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) { s1[threadIdx.x] += s1[threadIdx.x + o]; s2[threadIdx.x] += s2[threadIdx.x + o]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double m = s1[0] / n;
    double var = s2[0] / n - m * m;
    out[0] = m;
    out[1] = var > 0 ? sqrt(var) : 1.0;
  }
}

// Predictions back to label units.
__global__ void unstd_kernel(float *__restrict__ y, int n, float mu, float sd) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = y[i] * sd + mu;
}

// ---------------------------------------------------------------------------
// Ranking: the k smallest of n predictions in ascending order of (order-
// preserving key of the prediction, index), packed in 64 bits, so ties resolve
// by smaller index and all keys differ.  sort_tile_kernel sorts tiles of 2,048
// keys in shared memory; merge_kernel merges eight sorted runs at a time, each
// element finding its place by its rank in the seven sibling runs, and drops
// what cannot be among the first k.  A launch costs more than a tile's sort at
// these sizes, so the passes are what counts: 100,000 predictions with k =
// 5,000 take three launches where a bitonic sort of the whole array took 40
// (174 us serialised), a library of up to 2,048 one instead of 13.  A tile's
// strides below 64 stay in a warp's registers (20 -> 12.6 us), and a merge
// leaves elements that are beyond the first k at their first look (20 and 19 ->
// 14.8 and 12.3 us).
__device__ __forceinline__ uint32_t ordered_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

constexpr int SORT_TILE = 2048, MERGE_WAYS = 8;

// idx: the k smallest of a single tile; else the sorted tiles into keys[n].
__global__ void __launch_bounds__(1024) sort_tile_kernel(const float *__restrict__ pred, int n, int k,
                                                         unsigned long long *__restrict__ keys,
                                                         int32_t *__restrict__ idx) {
  __shared__ unsigned long long s[SORT_TILE];
  const int base = blockIdx.x * SORT_TILE;
  const int len = min(SORT_TILE, n - base);
  int size = 2;
  while (size < len) size <<= 1;
  pdl_wait();
  for (int q = threadIdx.x; q < size; q += blockDim.x) {
    unsigned long long key = ~0ull;
    if (q < len) {
      const float p = pred[base + q];
      key = ((unsigned long long)(isnan(p) ? 0xffffffffu : ordered_key(p)) << 32) | (uint32_t)(base + q);
    }
    s[q] = key;
  }
  // a warp keeps 64 consecutive keys (lane, lane + 32) in registers for the
  // strides up to 32; longer strides go through shared memory
  const int lane = threadIdx.x & 31, w0 = (threadIdx.x >> 5) * 64;
  unsigned long long k0 = ~0ull, k1 = ~0ull;
  auto near = [&](int kk, int j0) {  // strides j0, j0 / 2, ..., 1 of size kk
    for (int j = j0; j > 0; j >>= 1) {
      if (j == 32) {
        const bool up = ((w0 + lane) & kk) == 0;
        if ((k0 > k1) == up) { const unsigned long long t = k0; k0 = k1; k1 = t; }
      } else {
        const unsigned long long o0 = __shfl_xor_sync(0xffffffffu, k0, j), o1 = __shfl_xor_sync(0xffffffffu, k1, j);
        const bool low = (lane & j) == 0;
        const bool up0 = ((w0 + lane) & kk) == 0, up1 = ((w0 + 32 + lane) & kk) == 0;
        k0 = (low == up0) == (k0 < o0) ? k0 : o0;
        k1 = (low == up1) == (k1 < o1) ? k1 : o1;
      }
    }
  };
  __syncthreads();
  const bool on = w0 < size;  // sizes below 64 are sorted as 64
  if (on) { k0 = w0 + lane < size ? s[w0 + lane] : ~0ull; k1 = w0 + 32 + lane < size ? s[w0 + 32 + lane] : ~0ull; }
  for (int kk = 2; kk <= 64; kk <<= 1) near(kk, kk >> 1);
  for (int kk = 128; kk <= size; kk <<= 1) {
    if (on) { s[w0 + lane] = k0; s[w0 + 32 + lane] = k1; }
    for (int j = kk >> 1; j >= 64; j >>= 1) {
      __syncthreads();
      for (int t = threadIdx.x; t < size / 2; t += blockDim.x) {
        const int q = 2 * t - (t & (j - 1)), l = q + j;  // the pair of comparator t
        const unsigned long long x = s[q], y = s[l];
        if ((x > y) == ((q & kk) == 0)) { s[q] = y; s[l] = x; }
      }
    }
    __syncthreads();
    if (on) { k0 = s[w0 + lane]; k1 = s[w0 + 32 + lane]; near(kk, 32); }
  }
  __syncthreads();
  if (on) { s[w0 + lane] = k0; s[w0 + 32 + lane] = k1; }
  __syncthreads();
  for (int q = threadIdx.x; q < min(len, k); q += blockDim.x) {
    if (idx) idx[q] = (int32_t)(s[q] & 0xffffffffu);
    else keys[base + q] = s[q];
  }
}

// Runs of R keys (the last shorter) at in[run R], the first min(R, k) of each
// valid; out: runs of MERGE_WAYS R, or idx when one run remains.
__global__ void __launch_bounds__(256) merge_kernel(const unsigned long long *__restrict__ in, int n, int R, int k,
                                                    unsigned long long *__restrict__ out,
                                                    int32_t *__restrict__ idx) {
  pdl_wait();
  const int per = min(R, k);
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int run = (int)(t / per), p = (int)(t % per);
  const int i = run * R + p;
  if ((long long)run * R + p >= n) return;
  const unsigned long long key = in[i];
  const int g0 = run / MERGE_WAYS * MERGE_WAYS;
  int lo[MERGE_WAYS], len[MERGE_WAYS];
#pragma unroll
  for (int w = 0; w < MERGE_WAYS; ++w) {  // rank of key in each sibling run: the searches step side by side
    const long long b = (long long)(g0 + w) * R;
    lo[w] = 0;
    len[w] = g0 + w == run || b >= n ? 0 : (int)min((long long)per, n - b);
  }
  // most elements are beyond the first k: one is when every sibling's element
  // ceil((k - p) / siblings) - 1 is smaller
  int sib = 0;
#pragma unroll
  for (int w = 0; w < MERGE_WAYS; ++w) sib += len[w] > 0;
  if (sib > 0) {
    const int c = (k - p + sib - 1) / sib - 1;
    bool out_of_k = true;
#pragma unroll
    for (int w = 0; w < MERGE_WAYS; ++w)
      if (len[w] > 0) out_of_k &= c < len[w] && in[(long long)(g0 + w) * R + (c < len[w] ? c : 0)] < key;
    if (out_of_k) return;
  }
  for (int step = per; step > 0; step = step > 1 ? (step + 1) >> 1 : 0) {
    unsigned long long mid[MERGE_WAYS];
#pragma unroll
    for (int w = 0; w < MERGE_WAYS; ++w)
      mid[w] = len[w] > 0 ? in[(long long)(g0 + w) * R + lo[w] + (len[w] >> 1)] : 0ull;
#pragma unroll
    for (int w = 0; w < MERGE_WAYS; ++w) {
      const int half = len[w] >> 1;
      const bool right = len[w] > 0 && mid[w] < key;
      lo[w] += right ? half + 1 : 0;
      len[w] = right ? len[w] - half - 1 : half;
    }
  }
  int rank = p;
#pragma unroll
  for (int w = 0; w < MERGE_WAYS; ++w) rank += lo[w];
  if (rank >= k) return;
  if (idx) idx[rank] = (int32_t)(key & 0xffffffffu);
  else out[(long long)g0 * R + rank] = key;
}

cudaError_t sort_select(const float *pred, int n, int k, unsigned long long *keys, int32_t *idx, cudaStream_t s) {
  if (n <= 0 || k <= 0) return cudaSuccess;
  const int tiles = (n + SORT_TILE - 1) / SORT_TILE;
  cudaError_t e = launch_pdl(sort_tile_kernel, dim3(tiles), dim3(1024), 0, s, pred, n, k, keys, tiles == 1 ? idx : nullptr);
  unsigned long long *in = keys, *out = keys + n;
  long long runs = tiles;
  for (long long R = SORT_TILE; runs > 1 && e == cudaSuccess; R *= MERGE_WAYS) {
    const long long threads = runs * std::min<long long>(R, k);
    runs = (runs + MERGE_WAYS - 1) / MERGE_WAYS;
    e = launch_pdl(merge_kernel, dim3((unsigned)((threads + 255) / 256)), dim3(256), 0, s, in, n, (int)R, k, out,
                   runs == 1 ? idx : nullptr);
    std::swap(in, out);
  }
  return e;
}

// Mean prediction of an ensemble, accumulated in network order.
__global__ void mean_pred_kernel(const float *__restrict__ pred, int n_nets, int n, float a, float *__restrict__ mean) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_wait();
  if (i >= n) return;
  float v = a * pred[i];
  for (int m = 1; m < n_nets; ++m) v = fmaf(a, pred[(size_t)m * n + i], v);
  mean[i] = v;
}
cudaError_t mean_pred(const float *pred, int n_nets, int n, float *mean, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  return launch_pdl(mean_pred_kernel, dim3((n + 255) / 256), dim3(256), 0, s, pred, n_nets, n, 1.f / (float)n_nets, mean);
}

// Launch helpers used by the surrogate object.
cudaError_t gather_std(const float *desc, const int *idx, int rows, int row0, const float *mu,
                       const float *inv_sd, const float *labels, float ly_mu, float ly_inv,
                       __nv_bfloat16 *x, float *t, cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  return launch_pdl(gather_std_kernel, dim3(rows), dim3(128), 0, s, desc, idx, rows, row0, mu, inv_sd, labels, ly_mu,
                    ly_inv, x, t);
}
cudaError_t head(const __nv_bfloat16 *h3, const __nv_bfloat16 *w4, const float *b4, int rows,
                 const float *t, float *y, float *dy, float inv_b2, double *sse, __nv_bfloat16 *dz3,
                 cudaStream_t s) {
  return launch_pdl(head_kernel, dim3((rows * 32 + 255) / 256), dim3(256), 0, s, h3, w4, b4, rows, t, y, dy, inv_b2,
                    sse, dz3);
}
cudaError_t adam(float *w, const float *g, float *m, float *v, __nv_bfloat16 *wb, __nv_bfloat16 *wt, float lr,
                 float b1, float b2, float eps, float c1, float c2, cudaStream_t s) {
  AdamArgs a;
  a.w = w; a.g = g; a.m = m; a.v = v; a.wb = wb; a.wt = wt;
  a.lr = lr; a.b1 = b1; a.b2 = b2; a.eps = eps; a.c1 = c1; a.c2 = c2;
  int o = 0, tw = 0, ctas = 0;
  for (int l = 0; l < 3; ++l) {  // W1 [256][512], W2, W3 [512][512], each followed by its bias
    a.K[l] = l == 0 ? 256 : 512;
    a.off[l] = o;
    a.wt_off[l] = tw;
    o += a.K[l] * 512;
    tw += a.K[l] * 512;
    a.rest0[l] = o;
    a.rest1[l] = o += 512;
    ctas += a.K[l] / 32 * 16 + 1;
  }
  a.rest0[3] = o;  // W4 [512] and its bias
  a.rest1[3] = o + 513;
  return launch_pdl(adam_kernel, dim3(ctas + 1), dim3(256), 0, s, a);
}
cudaError_t to_bf16(const float *a, __nv_bfloat16 *b, int n, cudaStream_t s) {
  to_bf16_kernel<<<(n + 255) / 256 < 2048 ? (n + 255) / 256 : 2048, 256, 0, s>>>(a, b, n);
  return cudaGetLastError();
}
cudaError_t feature_stats(const float *desc, int n, float *mu, float *inv_sd, cudaStream_t s) {
  feature_stats_kernel<<<256, 256, 0, s>>>(desc, n, mu, inv_sd);
  return cudaGetLastError();
}
cudaError_t label_stats(const float *y, int n, double *out, cudaStream_t s) {
  label_stats_kernel<<<1, 256, 0, s>>>(y, n, out);
  return cudaGetLastError();
}
cudaError_t unstd(float *y, int n, float mu, float sd, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  unstd_kernel<<<(n + 255) / 256, 256, 0, s>>>(y, n, mu, sd);
  return cudaGetLastError();
}

}  // namespace mlp
}  // namespace ligate
