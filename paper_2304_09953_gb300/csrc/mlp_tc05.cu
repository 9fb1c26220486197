// K-major contractions of the triage surrogate on the 5th-generation tensor
// cores (paper Sec. 3.5: affinity predictor on ligand features).
//
//   C = epi(A B^T)  with A [M][K] BF16 and B [N][K] BF16 (K contiguous in
//   both), FP32 accumulation, BF16 output C [M][N].  Epilogues:
//     EPI_BIAS_RELU  forward layer   C = relu(acc + bias)   (B = W^T)
//     EPI_RELU_MASK  data gradient   C = acc * (mask > 0)   (B = W)
//
// One CTA computes a 128 x TN tile.  One elected thread streams 64-wide K
// slices of X and Wt into shared memory with TMA (128-byte swizzle, mbarrier
// transaction counts) and issues tcgen05.mma (kind::f16, M = 128, N = TN, K =
// 16 per instruction) into a TN-column FP32 accumulator in tensor memory;
// tcgen05.commit signals each stage's release and the final completion.  All
// four warps then read their 32 accumulator rows with tcgen05.ld, add the
// bias, apply ReLU and store BF16.
//
// TN and the stages follow the rows: a mini-batch of 1,024 rows has 8 row
// tiles, so 256-column tiles would leave 136 of 152 SMs idle; narrow tiles (64
// or 32 columns) fill them, and eight stages put the whole K = 512 in flight at
// once, which makes the launch one memory latency, the MMAs and a short
// epilogue.  Each output's sum runs over K in the same order for every TN.
//
// mlp_forward_kernel runs the whole network for inference: see there.
//
// Every mbarrier wait is bounded by the global timer: on a timeout the kernel
// records an error, drains what it issued (bounded again), frees its tensor
// memory and returns, so the host reports LIGATE_ERR_TIMEOUT instead of
// hanging.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "ligate_internal.h"
#include "mlp.h"

namespace ligate {
namespace mlp {
namespace {

constexpr int TM = 128, TK = 64;
constexpr int A_BYTES = TM * TK * 2;  // 16 KB per K slice
constexpr unsigned long long WAIT_NS = 2000000000ull;  // 2 s per wait

__device__ __forceinline__ uint32_t saddr(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(saddr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait on phase `parity`; false after WAIT_NS.
__device__ bool mbar_wait(uint64_t *bar, unsigned parity) {
  if (mbar_test(bar, parity)) return true;
  const unsigned long long t0 = now_ns();
  while (!mbar_test(bar, parity))
    if (now_ns() - t0 > WAIT_NS) return false;
  return true;
}
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x,
                                            int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(saddr(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(saddr(bar)), "r"(x), "r"(y)
      : "memory");
}
// Shared-memory matrix descriptor, K-major operand with 128-byte swizzle:
// start address >> 4 in bits [0,14), stride between 8-row groups (1024 B)
// >> 4 in [32,46), descriptor version 1 in [46,48), swizzle mode 2 in [61,64).
__device__ __forceinline__ uint64_t sdesc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// Instruction descriptor of kind::f16: FP32 accumulator (bits [4,6) = 1),
// BF16 A and B ([7,10) = 1, [10,13) = 1), both K-major, N >> 3 in [17,23),
// M >> 4 in [24,29).
constexpr uint32_t idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}

template <int N>
__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(tmem_d), "l"(a), "l"(b), "r"(idesc(N)), "r"(acc));
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   saddr(bar))
               : "memory");
}

// Fault for tests of the timeout path (ligate_debug_inject_fault's kind; the
// CTA that takes it resets it): nothing in normal operation sets it.
__device__ int g_fault = 0;

template <int TN, int STAGES>
struct __align__(1024) Smem {
  uint8_t a[STAGES][A_BYTES];
  uint8_t b[STAGES][TN * TK * 2];
  uint64_t full[STAGES];
  uint64_t empty[STAGES];
  uint64_t done;
  uint32_t tmem_base;
};

template <int EPI, int TN, int STAGES>
__global__ void __launch_bounds__(128, 1)
    gemm_tc05_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                     int M, int K, const float *__restrict__ bias,
                     const __nv_bfloat16 *__restrict__ mask, __nv_bfloat16 *__restrict__ out,
                     int ldc, int *__restrict__ err) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  typedef Smem<TN, STAGES> S;
  constexpr int B_BYTES = TN * TK * 2, TMEM_COLS = TN;
  S &s = *reinterpret_cast<S *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  const int nk = K / TK;

  if (threadIdx.x == 0) {
    for (int i = 0; i < STAGES; ++i) { mbar_init(&s.full[i], 1); mbar_init(&s.empty[i], 1); }
    mbar_init(&s.done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {  // one warp allocates the accumulator columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     saddr(&s.tmem_base)), "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s.tmem_base;
  pdl_wait();

  __shared__ int ok_shared;
  if (threadIdx.x == 0) {
    bool ok = true;
    int issued = 0;  // K slices whose loads were issued
    // test hook: a CTA that takes the fault flag issues no loads, so its
    // bounded wait on the first stage runs out and the error path runs
    const bool skip_loads = atomicCAS(&g_fault, 1, 0) == 1;
    for (int kb = 0; kb < nk && kb < STAGES && !skip_loads; ++kb, ++issued) {
      mbar_expect_tx(&s.full[kb], A_BYTES + B_BYTES);
      tma_load_2d(s.a[kb], &tm_a, &s.full[kb], kb * TK, m0);
      tma_load_2d(s.b[kb], &tm_b, &s.full[kb], kb * TK, n0);
    }
    int consumed = 0;
    for (int kb = 0; kb < nk && ok; ++kb) {
      const int st = kb % STAGES;
      const unsigned ph = (kb / STAGES) & 1u;
      if (!mbar_wait(&s.full[st], ph)) { ok = false; break; }
      consumed = kb + 1;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint64_t da = sdesc(saddr(s.a[st])), db = sdesc(saddr(s.b[st]));
#pragma unroll
      for (int kk = 0; kk < TK / 16; ++kk)  // 16 BF16 = 32 B per step: +2 in the address field
        mma_f16<TN>(tmem, da + 2 * kk, db + 2 * kk, (kb > 0 || kk > 0) ? 1u : 0u);
      mma_commit(&s.empty[st]);
      if (kb + STAGES < nk) {  // refill this stage once its MMAs are done
        if (!mbar_wait(&s.empty[st], ph)) { ok = false; break; }
        mbar_expect_tx(&s.full[st], A_BYTES + B_BYTES);
        tma_load_2d(s.a[st], &tm_a, &s.full[st], (kb + STAGES) * TK, m0);
        tma_load_2d(s.b[st], &tm_b, &s.full[st], (kb + STAGES) * TK, n0);
        ++issued;
      }
    }
    if (!ok) {  // drain loads still in flight (bounded), then report
      for (int kb = consumed; kb < issued; ++kb)
        (void)mbar_wait(&s.full[kb % STAGES], (kb / STAGES) & 1u);
      atomicExch(err, 1);
    }
    mma_commit(&s.done);  // arrives once every MMA issued so far has completed
    ok_shared = ok ? 1 : 0;
  }
  __syncthreads();
  const bool done_ok = mbar_wait(&s.done, 0);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!done_ok && lane == 0) atomicExch(err, 1);
  // block-uniform decision: tcgen05.ld is warp-collective
  if (__syncthreads_and(ok_shared && done_ok)) {
    // warp w owns accumulator rows 32 w .. 32 w + 31 (tensor-memory lanes)
    const int row = m0 + warp * 32 + lane;
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
    for (int c0 = 0; c0 < TN; c0 += 16) {
      uint32_t r[16];
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
            "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
            "=r"(r[14]), "=r"(r[15])
          : "r"(trow + (uint32_t)c0));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (row < M) {
        __align__(16) __nv_bfloat162 o[8];
        __align__(16) __nv_bfloat162 hm[8];
        if (EPI == EPI_RELU_MASK) {
          const uint4 *src = reinterpret_cast<const uint4 *>(mask + (size_t)row * ldc + n0 + c0);
          *reinterpret_cast<uint4 *>(&hm[0]) = src[0];
          *reinterpret_cast<uint4 *>(&hm[4]) = src[1];
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int n = n0 + c0 + 2 * q;
          float v0 = __uint_as_float(r[2 * q]), v1 = __uint_as_float(r[2 * q + 1]);
          if (EPI == EPI_BIAS_RELU) {
            v0 = fmaxf(v0 + bias[n], 0.f);
            v1 = fmaxf(v1 + bias[n + 1], 0.f);
          } else {
            if (!(__bfloat162float(hm[q].x) > 0.f)) v0 = 0.f;
            if (!(__bfloat162float(hm[q].y) > 0.f)) v1 = 0.f;
          }
          o[q] = __floats2bfloat162_rn(v0, v1);
        }
        uint4 *dst = reinterpret_cast<uint4 *>(out + (size_t)row * ldc + n0 + c0);
        dst[0] = *reinterpret_cast<const uint4 *>(&o[0]);
        dst[1] = *reinterpret_cast<const uint4 *>(&o[4]);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS)
                 : "memory");
}

// ---------------------------------------------------------------------------
// The whole network on 128 rows per CTA: standardised inputs, three hidden
// layers and the head, activations in shared memory, nothing but the rows'
// descriptors read and 4 bytes per row written.
//
// What bounds it: three layers that need one another, 0.17 GFLOP of tcgen05
// work per tile (11 us at the SM's share of the peak) between epilogues, with
// 1.3 MB of BF16 weights per tile from L2.  As layers of their own, each with a
// descriptor or activation pass through memory, 100,000 rows took gather + 3
// GEMM + head + unscale launches and 2 x 6 KB of activations per row: 590 us
// (serialised).  One kernel with the layers in a strict row of load, MMA and
// epilogue took 240, the pipeline below 161.  What it waits for is spread
// out: no loads of inputs -14 us, a quarter of the MMAs -14, no head -27; a
// quarter of the weight traffic, or pairs of CTAs sharing it by multicast, 0.
//
// A CTA keeps the layer input as eight 64-column K slices in the 128-byte
// swizzle the tensor core reads (128 KB) and streams the transposed weights as
// 256 x 64 tiles through a three-stage ring (six stages of 128 x 64: 231 us
// against 158 over two sizes); the 128 x 512 FP32 accumulator is the SM's whole
// tensor memory.  Warp 9 streams the weights of all tiles, warp 8 issues the
// MMAs, columns 0-255 of a layer before the others.  Warps 0-3 have columns
// 0-255: they read them, add the bias, apply ReLU and pack to BF16 in registers
// while the tensor core works on the other half, and write the next layer's
// slices 0-3 in place once that has read them.  Warps 4-7 do columns 256-511,
// while the next layer starts on slices 0-3.  After the last hidden layer warps
// 0-3 have the head and warps 4-7 write the next row tile's inputs.  Every
// output is the same bits as the layer-by-layer kernels': the same K order,
// rounding points, and head order (column l of each group of 32 in one chain,
// then the butterfly's tree).
constexpr int FW_THREADS = 384, FW_N = 256, FW_STAGES = 3, FW_B = FW_N * TK * 2;

struct FwdNet {
  CUtensorMap w[3];  // transposed hidden weights [512][256], [512][512], [512][512]
  const float *b[3];
  const __nv_bfloat16 *w4;
  const float *b4, *mu, *inv_sd;
  float ly_mu, ly_sd;
  float *pred;
  int *err;
};
struct FwdArgs {
  FwdNet net[FWD_NETS];
  const float *desc;
  int n, tiles, items, vec;  // rows, row tiles, tiles x networks, desc rows 16-byte aligned
};
struct __align__(1024) FwdSmem {
  uint8_t h[8][A_BYTES];
  uint8_t ring[FW_STAGES][FW_B];
  __nv_bfloat16 w4[512];
  uint64_t full[FW_STAGES], empty[FW_STAGES], in[2], acc[2], drain;
  uint32_t tmem_base;
  volatile int fault;  // test hook: warp 1 takes its last wait as run out
};
static_assert(sizeof(FwdSmem) + 1024 <= 227 * 1024, "one CTA's shared memory");

__device__ __forceinline__ void tmem_ld32(uint32_t (&r)[32], uint32_t addr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(bar)) : "memory");
}
// A warp's shared-memory writes and tensor-memory reads so far are done: tell
// the thread that issues the tensor-core work.
__device__ __forceinline__ void warp_arrive(uint64_t *bar, int lane) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}
// Whether all 128 threads of warps 0-3 are `ok`; a barrier among them.
__device__ __forceinline__ bool all_of_half(bool ok) {
  unsigned r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, 1, 128, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(ok ? 1u : 0u)
      : "memory");
  return r != 0;
}
// mbar_wait by a whole warp, the same answer in every lane.
__device__ __forceinline__ bool warp_wait(uint64_t *bar, unsigned parity) {
  const bool ok = __all_sync(0xffffffffu, mbar_wait(bar, parity));
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return ok;
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&v);
}

// A wait ran out: this CTA leaves its remaining tiles, of whichever network.
__device__ __forceinline__ void fw_report(const FwdArgs &a) {
  for (int q = 0; q < FWD_NETS; ++q) atomicExch(a.net[q].err, 1);
}
// Standardised inputs of NB x 8 rows (first, first + 4, ...) as packed BF16,
// eight columns per lane.
template <int NB, int U>
__device__ __forceinline__ void fw_load_rows(const FwdArgs &a, const FwdNet &net, int row0, int first, int lane,
                                             uint4 (&x)[NB * 8]) {
  float mu[8], sd[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) { mu[q] = __ldg(net.mu + 8 * lane + q); sd[q] = __ldg(net.inv_sd + 8 * lane + q); }
#pragma unroll
  for (int i = 0; i < NB * 8; i += U) {
    float v[U][8];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int row = row0 + first + 4 * (i + u);
      const float *src = a.desc + (size_t)(row < a.n ? row : 0) * 256 + 8 * lane;
      if (a.vec) {
#pragma unroll
        for (int q = 0; q < 8; q += 4)
          asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
                       : "=f"(v[u][q]), "=f"(v[u][q + 1]), "=f"(v[u][q + 2]), "=f"(v[u][q + 3])
                       : "l"(src + q));
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v[u][q]) : "l"(src + q));
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool in = row0 + first + 4 * (i + u) < a.n;
#pragma unroll
      for (int q = 0; q < 8; ++q) v[u][q] = (v[u][q] - mu[q]) * sd[q];
      x[i + u] = in ? make_uint4(pack_bf16(v[u][0], v[u][1]), pack_bf16(v[u][2], v[u][3]), pack_bf16(v[u][4], v[u][5]),
                                 pack_bf16(v[u][6], v[u][7]))
                    : make_uint4(0, 0, 0, 0);
      // packed here, not after the next rows' loads: registers
      asm volatile("" : "+r"(x[i + u].x), "+r"(x[i + u].y), "+r"(x[i + u].z), "+r"(x[i + u].w)::"memory");
    }
  }
}
template <int NB>
__device__ __forceinline__ void fw_store_rows(FwdSmem &s, int first, int lane, const uint4 (&x)[NB * 8]) {
#pragma unroll
  for (int i = 0; i < NB * 8; ++i) {
    const int r = first + 4 * i;
    *reinterpret_cast<uint4 *>(s.h[lane >> 3] + r * 128 + (((lane & 7) ^ (r & 7)) << 4)) = x[i];
  }
}
// The row's next-layer activations of one 256-column half, as packed BF16.
__device__ __forceinline__ void fw_activate(uint32_t trow, const float *bias, uint4 (&x)[32]) {
#pragma unroll
  for (int c0 = 0; c0 < 256; c0 += 32) {
    uint32_t r[32];
    tmem_ld32(r, trow + c0);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 b0 = __ldg(reinterpret_cast<const float4 *>(bias + c0 + 8 * q)),
                   b1 = __ldg(reinterpret_cast<const float4 *>(bias + c0 + 8 * q) + 1);
      const float bb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = fmaxf(__uint_as_float(r[8 * q + k]) + bb[k], 0.f);
      x[c0 / 8 + q] = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
    }
  }
}
__device__ __forceinline__ void fw_store_half(FwdSmem &s, int half, int row, const uint4 (&x)[32]) {
#pragma unroll
  for (int i = 0; i < 32; ++i)
    *reinterpret_cast<uint4 *>(s.h[half * 4 + (i >> 3)] + row * 128 + (((i & 7) ^ (row & 7)) << 4)) = x[i];
}

__global__ void __launch_bounds__(FW_THREADS, 1) mlp_forward_kernel(const __grid_constant__ FwdArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  FwdSmem &s = *reinterpret_cast<FwdSmem *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < FW_STAGES; ++i) { mbar_init(&s.full[i], 1); mbar_init(&s.empty[i], 1); }
    mbar_init(&s.in[0], 8);  // all layer warps
    mbar_init(&s.in[1], 4);  // one half's
    mbar_init(&s.acc[0], 1);
    mbar_init(&s.acc[1], 1);
    mbar_init(&s.drain, 1);
    s.fault = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 8) {  // the whole tensor memory: 512 columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(saddr(&s.tmem_base))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s.tmem_base;
  // an item: a network and a row tile
  const int first_item = blockIdx.x, step = gridDim.x;
  // registers: 384 threads start with 168; 128 x 40 + 256 x 232 is the same sum.
  // Compiled for the 168: a frame of 216 B, 852 B of spill stores, 284 of loads.
  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == 9) {  // the weight stream of all items, one thread
      const int fault = lane == 0 ? atomicExch(&g_fault, 0) : 1;  // test hook (see gemm_tc05_kernel)
      if (fault == 2) s.fault = 1;
      if (fault != 1) {
        int loaded = 0;
        bool go = true;
        for (int item = first_item; item < a.items && go; item += step) {
          const FwdNet &net = a.net[item / a.tiles];
          for (int l = 0; l < 3 && go; ++l) {
            const int slices = l == 0 ? 4 : 8;
            for (int r = 0; r < 2 * slices; ++r, ++loaded) {  // half of the columns, 64-wide K slice
              const int st = loaded % FW_STAGES;
              if (loaded >= FW_STAGES && !mbar_wait(&s.empty[st], (loaded / FW_STAGES - 1) & 1u)) { go = false; break; }
              mbar_expect_tx(&s.full[st], FW_B);
              const int x = r % slices * TK, y = r / slices * FW_N;
              tma_load_2d(s.ring[st], &net.w[l], &s.full[st], x, y);
            }
          }
        }
        // before the shared memory goes (bounded): loads in flight, the last commits
        for (int q = loaded < FW_STAGES ? 0 : loaded - FW_STAGES; q < loaded; ++q)
          if (mbar_wait(&s.full[q % FW_STAGES], (q / FW_STAGES) & 1u))
            (void)mbar_wait(&s.empty[q % FW_STAGES], (q / FW_STAGES) & 1u);
      }
      __syncwarp();
    } else if (warp == 8) {
      if (lane == 0) {  // the tensor-core work, one thread
        bool ok = true;
        int used = 0;
        unsigned layer = 0;
        for (int item = first_item; item < a.items && ok; item += step)
          for (int l = 0; l < 3 && ok; ++l, ++layer) {
            const int slices = l == 0 ? 4 : 8;
            for (int half = 0; half < 2 && ok; ++half) {
              for (int kb = 0; kb < slices; ++kb) {
                // in[0]: K slices 0-3 written, columns 0-255 read; in[1]: the others
                if (half == 0 && kb == 0 && !mbar_wait(&s.in[0], layer & 1u)) { ok = false; break; }
                if ((half == 0 ? kb == 4 : l == 0 && kb == 0) && !mbar_wait(&s.in[1], layer & 1u)) { ok = false; break; }
                const int st = used % FW_STAGES;
                if (!mbar_wait(&s.full[st], (used / FW_STAGES) & 1u)) { ok = false; break; }
                ++used;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t da = sdesc(saddr(s.h[kb])), db = sdesc(saddr(s.ring[st]));
#pragma unroll
                for (int kk = 0; kk < TK / 16; ++kk)
                  mma_f16<FW_N>(tmem + half * FW_N, da + 2 * kk, db + 2 * kk, (kb > 0 || kk > 0) ? 1u : 0u);
                mma_commit(&s.empty[st]);
              }
              if (ok) mma_commit(&s.acc[half]);  // arrives once every MMA issued so far has completed
            }
          }
        if (!ok) {
          fw_report(a);
          mma_commit(&s.drain);
          (void)mbar_wait(&s.drain, 0);
        }
      }
      __syncwarp();
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
    // warps 0-3 have accumulator columns 0-255 and the head, warps 4-7 the
    // other columns and the next tile's inputs
    const int half = warp >> 2, w = warp & 3, row = w * 32 + lane;
    const uint32_t trow = tmem + ((uint32_t)(w * 32) << 16);
    bool ok = true;
    unsigned layer = 0;
    if (first_item < a.items) {  // the first tile's inputs: half the rows each
      uint4 x[16];
      fw_load_rows<2, 8>(a, a.net[first_item / a.tiles], first_item % a.tiles * TM, half * 64 + w, lane, x);
      fw_store_rows<2>(s, half * 64 + w, lane, x);
      warp_arrive(&s.in[0], lane);
      if (half == 0) warp_arrive(&s.in[1], lane);
    }
    for (int item = first_item; item < a.items && ok; item += step) {
      const FwdNet &net = a.net[item / a.tiles];
      const int row0 = item % a.tiles * TM, next = item + step;
      if (half == 0) {
        // Warps 0-3 wait for the tensor core each by itself, and one's wait may run
        // out just before another's succeeds: each meets the others at the tile's
        // last barrier (all_of_half) all the same, and they leave together.
        for (int q = tid; q < 512; q += 128) s.w4[q] = net.w4[q];
        asm volatile("bar.sync 1, 128;" ::: "memory");
#pragma unroll 1
        for (int l = 0; l < 2 && ok; ++l, ++layer) {
          uint4 x[32];
          if (!(ok = warp_wait(&s.acc[0], layer & 1u))) break;
          fw_activate(trow, net.b[l], x);  // while the tensor core has the other columns
          if (!(ok = warp_wait(&s.acc[1], layer & 1u))) break;
          fw_store_half(s, 0, row, x);
          warp_arrive(&s.in[0], lane);
        }
        if (!ok || !(ok = warp_wait(&s.acc[0], layer & 1u) && !(warp == 1 && s.fault))) {
          all_of_half(false);
          break;
        }
        // head: chain c of 32 sums the columns c, c + 32, ..., then the
        // butterfly's tree
        float acc[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) acc[c] = 0.f;
#pragma unroll 1
        for (int j = 0; j < 512; j += 32) {
          if (j == 256) {
            warp_arrive(&s.in[0], lane);  // columns 0-255 read
            if (!(ok = warp_wait(&s.acc[1], layer & 1u))) break;
          }
          uint32_t r[32];
          tmem_ld32(r, trow + j);
#pragma unroll
          for (int c = 0; c < 32; c += 8) {
            const float4 b0 = __ldg(reinterpret_cast<const float4 *>(net.b[2] + j + c)),
                         b1 = __ldg(reinterpret_cast<const float4 *>(net.b[2] + j + c) + 1);
            const float bb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
            const uint4 wv = *reinterpret_cast<const uint4 *>(s.w4 + j + c);
            const uint32_t ww[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
            for (int k = 0; k < 8; k += 2) {
              const uint32_t h = pack_bf16(fmaxf(__uint_as_float(r[c + k]) + bb[k], 0.f),
                                           fmaxf(__uint_as_float(r[c + k + 1]) + bb[k + 1], 0.f));
              // a BF16 is the upper half of its FP32
              acc[c + k] = fmaf(__uint_as_float(h << 16), __uint_as_float(ww[k / 2] << 16), acc[c + k]);
              acc[c + k + 1] = fmaf(__uint_as_float(h & 0xffff0000u), __uint_as_float(ww[k / 2] & 0xffff0000u), acc[c + k + 1]);
            }
          }
        }
        if (!ok) {
          all_of_half(false);
          break;
        }
        ++layer;
        warp_arrive(&s.in[1], lane);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int c = 0; c < o; ++c) acc[c] += acc[c + o];
        if (row0 + row < a.n) net.pred[row0 + row] = fmaf(acc[0] + __ldg(net.b4), net.ly_sd, net.ly_mu);
        ok = all_of_half(true);  // w4 is read
      } else {
        const int nrow0 = next % a.tiles * TM;
        if (next < a.items)  // the next tile's rows towards L2
          for (int q = tid - 128; q < TM * 8; q += 128)
            if (nrow0 + (q >> 3) < a.n)
              asm volatile("prefetch.global.L2 [%0];" ::"l"(a.desc + (size_t)(nrow0 + (q >> 3)) * 256 + (q & 7) * 32));
#pragma unroll 1
        for (int l = 0; l < 2 && ok; ++l, ++layer) {
          uint4 x[32];
          if (!(ok = warp_wait(&s.acc[1], layer & 1u))) break;
          if (lane == 0) mbar_arrive(&s.in[0]);
          fw_activate(trow + 256, net.b[l] + 256, x);
          fw_store_half(s, 1, row, x);
          warp_arrive(&s.in[1], lane);
        }
        if (!ok) break;
        const FwdNet &nnet = a.net[next < a.items ? next / a.tiles : 0];
        uint4 x[16];  // half of the rows before the wait, the others after it: registers
        if (next < a.items) fw_load_rows<2, 8>(a, nnet, nrow0, w, lane, x);
        if (!(ok = warp_wait(&s.acc[1], layer & 1u))) break;
        ++layer;
        if (next < a.items) {
          fw_store_rows<2>(s, w, lane, x);
          fw_load_rows<2, 8>(a, nnet, nrow0, 64 + w, lane, x);
          fw_store_rows<2>(s, 64 + w, lane, x);
        }
        warp_arrive(&s.in[0], lane);
      }
    }
    if (!ok && lane == 0) fw_report(a);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 8)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// against the driver library).
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, []() {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// 2-D BF16 map of a row-major [rows][cols] matrix with a (64 x box_rows) box.
bool make_map(CUtensorMap *m, const void *base, int rows, int cols, int box_rows) {
  EncodeTiledFn f = encode_fn();
  if (!f) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  const cuuint32_t box[2] = {(cuuint32_t)TK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return f(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

bool tc05_supported(int M, int N, int K) {
  return M > 0 && N % 256 == 0 && K % TK == 0 && K >= TK && encode_fn() != nullptr;
}

namespace {
template <int EPI, int TN, int STAGES>
cudaError_t gemm_tile(const __nv_bfloat16 *a, int M, int K, const __nv_bfloat16 *b, int N, const float *bias,
                      const __nv_bfloat16 *mask, __nv_bfloat16 *out, int *err, cudaStream_t s) {
  CUtensorMap ta, tb;
  if (!make_map(&ta, a, M, K, TM) || !make_map(&tb, b, N, K, TN)) return cudaErrorInvalidValue;
  const int smem = (int)sizeof(Smem<TN, STAGES>) + 1024;
  // per-device attribute set-up is cheap; repeat it rather than cache per device
  cudaError_t e = cudaFuncSetAttribute(gemm_tc05_kernel<EPI, TN, STAGES>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(gemm_tc05_kernel<EPI, TN, STAGES>, dim3(N / TN, (M + TM - 1) / TM), dim3(128), smem, s, ta, tb, M, K,
                    bias, mask, out, N, err);
}

template <int EPI>
cudaError_t gemm_rows(const __nv_bfloat16 *a, int M, int K, const __nv_bfloat16 *b, int N, const float *bias,
                      const __nv_bfloat16 *mask, __nv_bfloat16 *out, int *err, cudaStream_t s) {
  // widest tile that still gives about two thirds of the 152 SMs a CTA
  const int tiles = (M + TM - 1) / TM;
  if (tiles * (N / 256) >= 96) return gemm_tile<EPI, 256, 3>(a, M, K, b, N, bias, mask, out, err, s);
  if (tiles * (N / 64) >= 96) return gemm_tile<EPI, 64, 8>(a, M, K, b, N, bias, mask, out, err, s);
  return gemm_tile<EPI, 32, 8>(a, M, K, b, N, bias, mask, out, err, s);
}
}  // namespace

cudaError_t gemm_tc05(int epi, const __nv_bfloat16 *a, int M, int K, const __nv_bfloat16 *b, int N,
                      const float *bias, const __nv_bfloat16 *mask, __nv_bfloat16 *out, int *err,
                      cudaStream_t s) {
  if (!tc05_supported(M, N, K) || (epi != EPI_BIAS_RELU && epi != EPI_RELU_MASK) ||
      (reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(out)) & 15)
    return cudaErrorInvalidValue;
  return epi == EPI_BIAS_RELU ? gemm_rows<EPI_BIAS_RELU>(a, M, K, b, N, bias, nullptr, out, err, s)
                              : gemm_rows<EPI_RELU_MASK>(a, M, K, b, N, nullptr, mask, out, err, s);
}

cudaError_t forward_tc05(const FwdSpec *nets, int n_nets, const float *desc, int n, cudaStream_t s) {
  if (n <= 0 || n_nets <= 0) return cudaSuccess;
  cudaError_t e;
  const int smem = (int)sizeof(FwdSmem) + 1024;
  if ((e = cudaFuncSetAttribute(mlp_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem))) return e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return e;
  for (int m0 = 0; m0 < n_nets; m0 += FWD_NETS) {
    const int m = n_nets - m0 < FWD_NETS ? n_nets - m0 : FWD_NETS;
    FwdArgs a;
    for (int q = 0; q < m; ++q) {
      const FwdSpec &f = nets[m0 + q];
      FwdNet &t = a.net[q];
      const int K[3] = {256, 512, 512};
      for (int l = 0; l < 3; ++l) {
        if (!make_map(&t.w[l], f.wt[l], 512, K[l], FW_N)) return cudaErrorInvalidValue;
        t.b[l] = f.b[l];
      }
      t.w4 = f.w4; t.b4 = f.b4; t.mu = f.mu; t.inv_sd = f.inv_sd;
      t.ly_mu = f.ly_mu; t.ly_sd = f.ly_sd;
      t.pred = f.pred; t.err = f.err;
    }
    for (int q = m; q < FWD_NETS; ++q) a.net[q] = a.net[0];
    a.desc = desc;
    a.n = n;
    a.tiles = (n + TM - 1) / TM;
    a.items = a.tiles * m;
    a.vec = (reinterpret_cast<uintptr_t>(desc) & 15) == 0;
    mlp_forward_kernel<<<std::min(a.items, sms), FW_THREADS, smem, s>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t inject_fault_once(int kind) { return cudaMemcpyToSymbol(g_fault, &kind, sizeof(int)); }

// Wt[n][k] = bf16(W[k][n]) for a row-major [K][N] FP32 weight matrix.
__global__ void transpose_bf16_kernel(const float *__restrict__ w, int K, int N,
                                      __nv_bfloat16 *__restrict__ wt) {
  __shared__ float tile[32][33];
  const int k0 = blockIdx.y * 32, n0 = blockIdx.x * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int k = k0 + r, n = n0 + threadIdx.x;
    tile[r][threadIdx.x] = (k < K && n < N) ? w[(size_t)k * N + n] : 0.f;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int n = n0 + r, k = k0 + threadIdx.x;
    if (n < N && k < K) wt[(size_t)n * K + k] = __float2bfloat16_rn(tile[threadIdx.x][r]);
  }
}

cudaError_t transpose_bf16(const float *w, int K, int N, __nv_bfloat16 *wt, cudaStream_t s) {
  dim3 grid((N + 31) / 32, (K + 31) / 32), block(32, 8);
  transpose_bf16_kernel<<<grid, block, 0, s>>>(w, K, N, wt);
  return cudaGetLastError();
}

}  // namespace mlp
}  // namespace ligate
