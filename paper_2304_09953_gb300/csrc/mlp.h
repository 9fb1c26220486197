// Kernels of the triage surrogate network (mlp.cu), used by surrogate.cu.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ligate {
namespace mlp {

// The kernels of a training step, and those of a ranking, follow one another on
// one stream, each a few microseconds long, so a launch's own latency counts:
// they are launched with programmatic stream serialisation.  A kernel's CTAs may
// start while the one before it drains, and pdl_wait (before the first access to
// memory that another kernel writes or reads) holds them until it has finished.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <class... P, class... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, P(args)...);
}
#endif

enum { EPI_BIAS_RELU = 0, EPI_RELU_MASK = 1 };
enum { GEMM_FWD = 0, GEMM_DGRAD = 1 };

struct GemmArgs {
  const __nv_bfloat16 *A, *B;
  int M, N, K;
  long long sAm, sBk, sBn;       // element strides (the contiguous ones are 1)
  const float *bias;             // EPI_BIAS_RELU
  const __nv_bfloat16 *mask;     // EPI_RELU_MASK: ReLU output of the forward layer
  __nv_bfloat16 *Cb;             // BF16 output
  int ldc;
};

cudaError_t gemm(int kind, const GemmArgs &g, cudaStream_t s);
cudaError_t gather_std(const float *desc, const int *idx, int rows, int row0, const float *mu,
                       const float *inv_sd, const float *labels, float ly_mu, float ly_inv,
                       __nv_bfloat16 *x, float *t, cudaStream_t s);
cudaError_t head(const __nv_bfloat16 *h3, const __nv_bfloat16 *w4, const float *b4, int rows,
                 const float *t, float *y, float *dy, float inv_b2, double *sse, __nv_bfloat16 *dz3,
                 cudaStream_t s);
// Parameter gradients of a step: hidden layers l = 0..2 with inputs in[l]
// [rows][fan_in[l]] and output gradients dz[l] [rows][512] -> dw[l]
// [fan_in][512] and db[l][512]; head inputs h3 [rows][512] and dy [rows] ->
// gw4[512], gb4[1].
struct GradArgs {
  const __nv_bfloat16 *in[3], *dz[3];
  float *dw[3], *db[3];
  int fan_in[3];
  const __nv_bfloat16 *h3;
  const float *dy;
  float *gw4, *gb4;
  int rows;
};
cudaError_t grads(const GradArgs &a, cudaStream_t s);
// Adam over the flat parameter vector (LIGATE_SURROGATE_PARAMS); wt: the
// transposed BF16 hidden weights, or NULL.
cudaError_t adam(float *w, const float *g, float *m, float *v, __nv_bfloat16 *wb, __nv_bfloat16 *wt, float lr,
                 float b1, float b2, float eps, float c1, float c2, cudaStream_t s);
cudaError_t to_bf16(const float *a, __nv_bfloat16 *b, int n, cudaStream_t s);
cudaError_t feature_stats(const float *desc, int n, float *mu, float *inv_sd, cudaStream_t s);
cudaError_t label_stats(const float *y, int n, double *out, cudaStream_t s);
cudaError_t unstd(float *y, int n, float mu, float sd, cudaStream_t s);
// Indices of the k smallest of pred[n] in ascending (value, index) order (NaN
// last) into idx; keys: scratch of 2 n entries.
cudaError_t sort_select(const float *pred, int n, int k, unsigned long long *keys, int32_t *idx, cudaStream_t s);

// tcgen05 path (mlp_tc05.cu) for K-major A [M][K] and B [N][K]:
// C[M][N] = epi(A B^T), epi EPI_BIAS_RELU or EPI_RELU_MASK; needs N % 256 == 0,
// K % 64 == 0, 16-byte aligned pointers.  *err is set to 1 when a bounded
// wait ran out (results then undefined).
bool tc05_supported(int M, int N, int K);
cudaError_t gemm_tc05(int epi, const __nv_bfloat16 *a, int M, int K, const __nv_bfloat16 *b, int N,
                      const float *bias, const __nv_bfloat16 *mask, __nv_bfloat16 *out, int *err,
                      cudaStream_t s);
// Inference of n_nets networks on desc [n][256] (FP32) in one launch per
// FWD_NETS networks: predictions in label units into pred [n] of each.
constexpr int FWD_NETS = 8;
struct FwdSpec {
  const __nv_bfloat16 *wt[3];  // transposed hidden weights, 16-byte aligned
  const float *b[3];           // 16-byte aligned
  const __nv_bfloat16 *w4;
  const float *b4, *mu, *inv_sd;
  float ly_mu, ly_sd;
  float *pred;
  int *err;
};
cudaError_t forward_tc05(const FwdSpec *nets, int n_nets, const float *desc, int n, cudaStream_t s);
// mean[i] = sum_m (1 / n_nets) pred[m][i], accumulated in network order.
cudaError_t mean_pred(const float *pred, int n_nets, int n, float *mean, cudaStream_t s);
// Test hook (err set, LIGATE_ERR_TIMEOUT at the next check): kind 1, the next
// CTA of a tcgen05 contraction issues no loads, so its bounded wait runs out;
// kind 2, one warp of the next forward_tc05 CTA takes its last layer's wait as
// run out while the warps beside it go on.
cudaError_t inject_fault_once(int kind);
// wt[n][k] = bf16(w[k][n]) for row-major FP32 w [K][N].
cudaError_t transpose_bf16(const float *w, int K, int N, __nv_bfloat16 *wt, cudaStream_t s);

}  // namespace mlp
}  // namespace ligate
