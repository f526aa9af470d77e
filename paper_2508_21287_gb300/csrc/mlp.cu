// Cardinality model: a 3-layer MLP (32 -> 128 -> 128 -> 1, ReLU) that predicts the log growth
// of the intermediate table for a candidate join step, trained on the cardinalities the
// executor logs. Matmuls run on the tensor cores as BF16 x BF16 -> FP32 (tcgen05.mma with the
// accumulator in tensor memory); the
// master weights, biases, the output layer and Adam's moments stay FP32. Activations that
// feed a matmul are rounded to BF16 (round to nearest even) right after they are produced.
//
// Flat parameter layout (FP32): W1[128][32] | b1[128] | W2[128][128] | b2[128] | w3[128] | b3.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "join_device.cuh"
#include "kernels.h"

namespace dmk {

constexpr int MLP_IN = 32, MLP_H = 128;

// C[M x N] (+)= sum_k A(m, k) * B(k, n); A(m, k) = A[m * am + k * ak], B(k, n) = B[k * bk + n * bn],
// M % 16 == 0, N = 32 or 128, K % 16 == 0: fifth-generation tensor cores (tcgen05). A CTA of 16
// warps owns 128 rows of C; its accumulator is 128 lanes x N FP32 columns of tensor memory. Per
// K chunk of up to 256 (a training batch of 256 samples is one chunk) the CTA stages A (its 128
// rows, zero past M) and B (N rows, as B^T) in shared memory in the canonical K-major layout
// without swizzle -- 8 x 8 BF16 core matrices of 128 contiguous bytes, 128 bytes apart along K
// and 4 KB apart along M / N -- and one thread issues the chunk's K / 16 MMAs (M = 128, K = 16
// each) and commits them to an mbarrier that every thread waits on before the next chunk is
// staged. Warp w then reads 32 columns (group w / 4) of the accumulator lanes 32 (w % 4) ..
// 32 (w % 4) + 31 (tcgen05.ld) and writes them to its rows of C. Every wait is bounded: a chunk
// whose MMAs do not complete within about a second raises *err, and the CTA still waits (bounded
// again) for them before it frees its tensor memory.
constexpr int TC_M = 128, TC_KC = 256, TC_THREADS = 512, TC_COLS = 128;
// shared memory of a CTA: A and B chunks (64 KB each; a whole training batch of 256 samples is
// one chunk). At 512 threads at most 4 CTAs could share an SM (2048 threads), so their tensor
// memory (4 x 128 of 512 columns) is always free to allocate.
constexpr int TC_SMEM = 2 * TC_M * TC_KC * 2;
static_assert(2048 / TC_THREADS * TC_COLS <= 512, "resident CTAs could exhaust tensor memory");
constexpr long long TC_WAIT_CYCLES = 2000000000ll;

__device__ __forceinline__ uint32_t tc_saddr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// BF16 offset of element (r, k) of a staged operand: core matrix (r / 8, k / 8), then row-major
// inside it.
__device__ __forceinline__ int tc_core_off(int r, int k) {
  return (((r >> 3) * (TC_KC >> 3) + (k >> 3)) << 6) + ((r & 7) << 3) + (k & 7);
}

// Shared-memory matrix descriptor: start address, leading (K) and stride (M / N) byte offsets
// between core matrices, descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t tc_sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major, N, M = 128.
__device__ __forceinline__ uint32_t tc_idesc(int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(TC_M >> 4) << 24);
}

// Spins with the non-blocking test (the MMAs of a chunk take microseconds; a suspending wait
// could sleep past their completion).
__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  while (true) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > TC_WAIT_CYCLES) return false;
  }
}

__global__ void __launch_bounds__(TC_THREADS) k_gemm_tc(int M, int N, int K, const __nv_bfloat16 *A, int am, int ak,
                                                        const __nv_bfloat16 *Bm, int bk, int bn, float *C, int ldc,
                                                        int accumulate, unsigned *err) {
  extern __shared__ __align__(1024) uint16_t tc_smem[];
  uint16_t *sA = tc_smem, *sB = tc_smem + TC_M * TC_KC;
  __shared__ __align__(8) unsigned long long bar;
  __shared__ uint32_t tmem_base;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * TC_M;
  const int kb = 0, ke = K;
  const uint32_t bar_a = tc_saddr(&bar);
  if (warp == 0) {  // the accumulator: 128 lanes x TC_COLS columns
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_saddr(&tmem_base)),
                 "r"(TC_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  const uint32_t idesc = tc_idesc(N);
  const bool vecA = ak == 1 && am % 8 == 0 && ((uintptr_t)A & 15) == 0;
  const bool vecB = bk == 1 && bn % 8 == 0 && ((uintptr_t)Bm & 15) == 0;
  const bool tA = am == 1 && ak % 8 == 0 && ((uintptr_t)A & 15) == 0;
  const bool tB = bn == 1 && bk % 8 == 0 && ((uintptr_t)Bm & 15) == 0;
  const uint32_t sbo = (TC_KC >> 3) * 128;  // bytes between 8-row groups
  uint32_t phase = 0;
  bool ok = true;
  for (int k0 = kb; k0 < ke && ok; k0 += TC_KC) {
    const int kc = min(TC_KC, ke - k0);  // a multiple of 16
    // an operand whose K is contiguous (16-byte aligned rows) moves as 16-byte pieces, one core
    // matrix row each; otherwise consecutive threads take consecutive elements of its contiguous
    // dimension
    // thread order: the 8 rows of a core matrix are 8 neighbouring threads (128 contiguous
    // bytes of shared memory: no bank conflict), then the core matrices along K, then along M
    if (vecA) {
      for (int i = tid; i < TC_M * (kc >> 3); i += TC_THREADS) {
        const int rest = i >> 3, kp = rest % (kc >> 3);
        const int r = ((rest / (kc >> 3)) << 3) | (i & 7), k = kp << 3;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (m0 + r < M) v = *(const uint4 *)(A + (int64_t)(m0 + r) * am + k0 + k);
        *(uint4 *)(sA + tc_core_off(r, k)) = v;
      }
    } else if (tA) {  // M contiguous: 16-byte pieces of 8 rows at one k, scattered to the rows
      for (int i = tid; i < kc * (TC_M >> 3); i += TC_THREADS) {  // neighbouring threads: neighbouring k
        const int r = (i / kc) << 3, k = i % kc;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (m0 + r < M) v = *(const uint4 *)(A + m0 + r + (int64_t)(k0 + k) * ak);  // M % 8 == 0
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 8; j++) sA[tc_core_off(r + j, k)] = (uint16_t)(w[j >> 1] >> (16 * (j & 1)));
      }
    } else {
      for (int i = tid; i < TC_M * kc; i += TC_THREADS) {
        const int r = am == 1 ? i % TC_M : i / kc, k = am == 1 ? i / TC_M : i % kc;
        sA[tc_core_off(r, k)] =
            m0 + r < M ? __bfloat16_as_ushort(A[(int64_t)(m0 + r) * am + (int64_t)(k0 + k) * ak]) : (uint16_t)0;
      }
    }
    if (vecB) {
      for (int i = tid; i < N * (kc >> 3); i += TC_THREADS) {
        const int rest = i >> 3, kp = rest % (kc >> 3);
        const int n = ((rest / (kc >> 3)) << 3) | (i & 7), k = kp << 3;
        *(uint4 *)(sB + tc_core_off(n, k)) = *(const uint4 *)(Bm + (int64_t)n * bn + k0 + k);
      }
    } else if (tB) {  // N contiguous: 16-byte pieces of 8 columns at one k
      for (int i = tid; i < kc * (N >> 3); i += TC_THREADS) {
        const int n = (i / kc) << 3, k = i % kc;
        const uint4 v = *(const uint4 *)(Bm + (int64_t)(k0 + k) * bk + n);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 8; j++) sB[tc_core_off(n + j, k)] = (uint16_t)(w[j >> 1] >> (16 * (j & 1)));
      }
    } else {
      for (int i = tid; i < N * kc; i += TC_THREADS) {
        const int n = bn == 1 ? i % N : i / kc, k = bn == 1 ? i / N : i % kc;
        sB[tc_core_off(n, k)] = __bfloat16_as_ushort(Bm[(int64_t)(k0 + k) * bk + (int64_t)n * bn]);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the tensor cores read what was stored
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int kk = 0; kk < kc; kk += 16) {
        const uint64_t ad = tc_sdesc(tc_saddr(sA) + (kk >> 3) * 128, 128, sbo);
        const uint64_t bd = tc_sdesc(tc_saddr(sB) + (kk >> 3) * 128, 128, sbo);
        const uint32_t acc = (k0 + kk) > kb;  // the CTA's first MMA overwrites the accumulator
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
            "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
            : "memory");
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar_a)
                   : "memory");
    }
    const bool landed = tc_wait(bar_a, phase);  // the chunk's MMAs are done with sA and sB
    phase ^= 1u;
    ok = __syncthreads_and(landed);
    if (!ok) {
      if (tid == 0) atomicOr(err, 1u);
      tc_wait(bar_a, phase ^ 1u);  // let them finish (bounded) before the memory is freed
    }
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const int quad = warp & 3, c0 = 32 * (warp >> 2);  // a warp reads its lane quadrant (warp % 4)
  if (ok && kb < ke && c0 < N) {  // rows m0 + 32 quad + lane, columns c0 .. c0 + 31
    const int row = m0 + 32 * quad + lane;
    {
      uint32_t v[32];
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
          "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
            "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
            "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]),
            "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
            "=r"(v[30]), "=r"(v[31])
          : "r"(tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)c0)
          : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (row < M) {  // the row's 32 columns as 16-byte pieces (ldc % 4 == 0, C 16-byte aligned)
        float4 *c = (float4 *)(C + (int64_t)row * ldc + c0);
#pragma unroll
        for (int j = 0; j < 8; j++) {
          float4 x = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                 __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
          if (accumulate) {
            const float4 o = c[j];
            x.x += o.x;
            x.y += o.y;
            x.z += o.z;
            x.w += o.w;
          }
          c[j] = x;
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_COLS) : "memory");
  if (tid == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar_a) : "memory");
}

__global__ void k_to_bf16(const float *x, __nv_bfloat16 *y, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = __float2bfloat16_rn(x[i]);
}

// H = relu(Z + b) rounded to BF16; Z keeps the pre-activation (its sign is the ReLU mask).
__global__ void k_bias_relu(float *Z, const float *b, __nv_bfloat16 *H, int rows, int cols) {
  int64_t n = (int64_t)rows * cols;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float z = Z[i] + b[i % cols];
    Z[i] = z;
    H[i] = __float2bfloat16_rn(z > 0.f ? z : 0.f);
  }
}

// y[r] = sum_o H2[r][o] * w3[o] + b3 (FP32); with targets, dy[r] = 2 (y - t) / n_valid for valid rows
// and the squared error is added to *loss.
__global__ void k_out_layer(const __nv_bfloat16 *H2, const float *w3, const float *b3, int rows, int n_valid,
                            const float *target, float *y, float *dy, float *loss) {
  int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  int lane = threadIdx.x & 31;
  if (r >= rows) return;
  float s = 0.f;
  for (int o = lane; o < MLP_H; o += 32) s += __bfloat162float(H2[(int64_t)r * MLP_H + o]) * w3[o];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if (lane == 0) {
    float v = s + b3[0];
    y[r] = v;
    if (target) {
      float e = r < n_valid ? v - target[r] : 0.f;
      dy[r] = 2.f * e / (float)n_valid;
      if (r < n_valid) atomicAdd(loss, e * e / (float)n_valid);
    }
  }
}

// Column sums of a rows x cols matrix, 32 columns a block: warp w of 8 adds rows w, w + 8, ...
// of its lane's column (coalesced), and the 8 partial sums are added in a fixed order.
template <typename T>
__device__ __forceinline__ float colsum32(const T *M, const float *wrow, int rows, int cols, int c,
                                          float *s_part) {
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  float s = 0.f;
  if (c < cols)
    for (int r = w; r < rows; r += 8) {
      float x;
      if constexpr (sizeof(T) == 2) x = __bfloat162float(M[(int64_t)r * cols + c]);
      else x = (float)M[(int64_t)r * cols + c];
      s += wrow ? wrow[r] * x : x;
    }
  s_part[w * 32 + l] = s;
  __syncthreads();
  float t = 0.f;
  if (w == 0)
    for (int k = 0; k < 8; k++) t += s_part[k * 32 + l];
  __syncthreads();
  return t;  // valid in warp 0
}

// dH2 = dy * w3 masked by Z2 > 0 (BF16), every block over its grid-stride share; blocks 0 .. 3
// also add dw3 (32 columns each) and block 0 db3 (FP32, accumulated). 256 threads a block.
__global__ void k_out_backward(const float *dy, const __nv_bfloat16 *H2, const float *Z2, const float *w3, int rows,
                               __nv_bfloat16 *dH2, float *dw3, float *db3) {
  __shared__ float s_part[256];
  if (blockIdx.x < MLP_H / 32) {
    const int c = blockIdx.x * 32 + (threadIdx.x & 31);
    const float t = colsum32(H2, dy, rows, MLP_H, c, s_part);
    if (threadIdx.x < 32) dw3[c] += t;
    if (blockIdx.x == 0) {
      const float u = colsum32(dy, (const float *)nullptr, rows, 1, threadIdx.x & 31, s_part);
      if (threadIdx.x == 0) db3[0] += u;
    }
  }
  int64_t n = (int64_t)rows * MLP_H;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int64_t r = i / MLP_H;
    int oo = (int)(i - r * MLP_H);
    float g = Z2[i] > 0.f ? dy[r] * w3[oo] : 0.f;
    dH2[i] = __float2bfloat16_rn(g);
  }
}

// dH = dA masked by Z > 0, rounded to BF16.
__global__ void k_relu_backward(const float *dA, const float *Z, __nv_bfloat16 *dH, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    dH[i] = __float2bfloat16_rn(Z[i] > 0.f ? dA[i] : 0.f);
}

// db[c] += sum_r dH[r][c]: 32 columns a block of 256 threads
__global__ void k_colsum(const __nv_bfloat16 *dH, int rows, int cols, float *db) {
  __shared__ float s_part[256];
  const int c = blockIdx.x * 32 + (threadIdx.x & 31);
  const float t = colsum32(dH, (const float *)nullptr, rows, cols, c, s_part);
  if (threadIdx.x < 32 && c < cols) db[c] += t;
}

// ------------------------------------------------------------------ training step ------
// One training step in two launches. k_train_rows: a block per 128 samples runs them forward and back
// to the gradients of the hidden layers, its activations in shared memory and its three products in
// tensor memory; only what the weight gradients need (the rounded activations and their gradients) goes
// to device memory. k_train_weights: a block per 32 columns of the weight gradients (or of a bias or
// output-layer sum) adds over the samples and applies Adam to its own parameters.
//
// A step is a chain of small dependent products and nothing else, so it costs what it waits. What is kept
// between the launches is kept as the next product reads it, so that a launch begins with bulk copies and
// no thread converts or transposes: the rounded weights in the canonical layout (written by the threads
// that apply Adam), and activations and gradients as sample-major 8 x 8 core matrices, whose 16-byte rows
// are what a thread of k_train_rows holds and which the weight gradients' products read as MN-major
// operands. The second layer's weights serve both directions from one copy: K-major forward, MN-major back.
//
// 256 samples: 170 us a step as fifteen launches with an upload, five allocations and a synchronisation of
// its own; 38 us as these two launches with every thread converting and transposing what it loads (a
// transposed copy of W2 alone cost 8000 clocks of bank conflicts); 18 us so. A call of 2048 samples, two
// epochs: 2.55 ms, 0.85, 0.44. What is left is waiting: two launches behind one another, a bulk copy and
// three dependent products in the first, one in the second. Products and sums run in the order of
// mlp_forward_backward, so a step's gradients are the bits that dm_model_grad returns.
constexpr int TR_THREADS = 512, TR_M = 128;

// Offset (in elements) of (r, k) in an operand of KC columns in the canonical layout (tc_core_off).
template <int KC>
__device__ __forceinline__ int tr_off(int r, int k) {
  return (((r >> 3) * (KC >> 3) + (k >> 3)) << 6) + ((r & 7) << 3) + (k & 7);
}

// K / 16 MMAs of a staged product, and the arrival of their completion at the barrier.
// An operand is its address, the bytes between core matrices along K and along M / N, and whether the
// 16-byte rows of a core matrix run along M / N (bits 15 and 16 of the instruction descriptor).
struct TrOp {
  const uint16_t *p;
  uint32_t k, mn;
  bool mn_major;
};
__device__ __forceinline__ void tr_mma(uint32_t tmem, const TrOp &A, const TrOp &B, int N, int K, bool first, uint32_t bar) {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t idesc = tc_idesc(N) | ((uint32_t)A.mn_major << 15) | ((uint32_t)B.mn_major << 16);
  for (int kk = 0; kk < K; kk += 16) {
    const uint64_t ad = tc_sdesc(tc_saddr(A.p) + (kk >> 3) * A.k, A.k, A.mn);
    const uint64_t bd = tc_sdesc(tc_saddr(B.p) + (kk >> 3) * B.k, B.k, B.mn);
    const uint32_t acc = !first || kk > 0;
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
  }
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tr_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Bulk copy into shared memory (16-byte aligned, a multiple of 16 bytes), counted at the barrier.
__device__ __forceinline__ void tr_bulk(void *dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(tc_saddr(dst)),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// 32 columns of this thread's accumulator row.
__device__ __forceinline__ void tr_ld32(uint32_t addr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
      "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]),
        "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
        "=r"(v[30]), "=r"(v[31])
      : "r"(addr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t tr_pack(float lo, float hi) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) |
         ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16);
}

struct TrainSmemA {
  uint16_t x[TR_M * 32], w1[MLP_H * 32];        // K = 32
  uint16_t h1[TR_M * MLP_H], w2[MLP_H * MLP_H]; // K = 128
  uint16_t d2[TR_M * MLP_H];
  uint16_t h2[TR_M * (MLP_H + 8)];              // row-major, padded
  float b1[MLP_H], b2[MLP_H], w3[MLP_H], dy[TR_M];
  unsigned long long bar, load[2];              // products; the first and the second layer's weights
  uint32_t tmem, stop;
};

// Block-wide wait for the MMAs committed to the barrier; false (and *err raised) when it ran out.
__device__ __forceinline__ bool tr_wait(uint32_t bar, uint32_t &phase, unsigned *err) {
  const bool landed = tc_wait(bar, phase);
  phase ^= 1u;
  const bool ok = __syncthreads_and(landed);
  if (!ok) {
    if (threadIdx.x == 0) atomicOr(err, 1u);
    tc_wait(bar, phase ^ 1u);  // let them finish (bounded) before the memory is freed
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  return ok;
}

__device__ __forceinline__ void tr_setup(unsigned long long *bar, int n_bar, uint32_t *tmem, int cols) {
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_saddr(tmem)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < n_bar; i++)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_saddr(bar + i)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tr_teardown(unsigned long long *bar, int n_bar, uint32_t tmem, int cols) {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
  if (threadIdx.x == 0)
    for (int i = 0; i < n_bar; i++) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(tc_saddr(bar + i)) : "memory");
}

// Wait of the thread that issues the products for a bulk copy; false (and *err raised) when it ran out,
// after a second bounded wait: the copy must not outlive the block.
__device__ __forceinline__ bool tr_landed(uint32_t bar, uint32_t phase, unsigned *err) {
  if (tc_wait(bar, phase)) return true;
  atomicOr(err, 1u);
  tc_wait(bar, phase);
  return false;
}

// Place (in elements) of column block c8 (eight columns) of sample r in a kept matrix of R samples.
__device__ __forceinline__ int64_t tr_at(int64_t R, int r, int c8) { return ((int64_t)c8 * R + r) * 8; }

// The rounded weights of both layers from the parameters, before the first step.
__global__ void __launch_bounds__(256) k_train_begin(const MlpTrain T) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  const float *W1 = T.params, *W2 = T.params + MLP_H * MLP_IN + MLP_H;
  auto bits = [](float x) { return __bfloat16_as_ushort(__float2bfloat16_rn(x)); };
  if (i < MLP_H * MLP_IN) T.W1b[tr_off<MLP_IN>(i / MLP_IN, i % MLP_IN)] = bits(W1[i]);
  if (i < MLP_H * MLP_H) T.W2b[tr_off<MLP_H>(i / MLP_H, i % MLP_H)] = bits(W2[i]);
}

__global__ void __launch_bounds__(TR_THREADS, 1) k_train_rows(const MlpTrain T, const int32_t *idx, int m, float *loss) {
  extern __shared__ __align__(1024) unsigned char tr_smem[];
  TrainSmemA &S = *(TrainSmemA *)tr_smem;
  constexpr int COLS = 512;  // three accumulators of 128 columns (allocations are powers of two)
  constexpr int OUT = TR_M / (TR_THREADS / 32);  // rows of the output layer a warp
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rows = (m + 15) / 16 * 16, m0 = blockIdx.x * TR_M;
  const float *b1 = T.params + MLP_H * MLP_IN, *b2 = b1 + MLP_H + MLP_H * MLP_H;
  const float *w3 = b2 + MLP_H, *b3 = w3 + MLP_H;
  tr_setup(&S.bar, 3, &S.tmem, COLS);
  const uint32_t tmem = S.tmem, bar = tc_saddr(&S.bar);
  uint32_t phase = 0;
  // the samples do not depend on the launch before; the parameters do
  static_assert(TR_M * 4 == TR_THREADS, "eight inputs of a row a thread");
  uint4 xin = make_uint4(0, 0, 0, 0);
  const int xr = tid >> 2, xk = tid & 3;
  if (m0 + xr < m) {
    const float4 *x = (const float4 *)(T.X + (int64_t)__ldg(idx + m0 + xr) * MLP_IN + 8 * xk);
    const float4 p = __ldg(x), q = __ldg(x + 1);
    xin = make_uint4(tr_pack(p.x, p.y), tr_pack(p.z, p.w), tr_pack(q.x, q.y), tr_pack(q.z, q.w));
  }
  *(uint4 *)(S.x + tr_off<32>(xr, 8 * xk)) = xin;
  const int ox = warp + (TR_THREADS / 32) * lane;  // the row of the output layer whose target this lane keeps
  const float target = lane < OUT && m0 + ox < m ? __ldg(T.target + __ldg(idx + m0 + ox)) : 0.f;
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  griddep_wait();
  griddep_launch_dependents();
  if (tid == 0) {
    asm volatile("fence.proxy.async.global;" ::: "memory");
    tr_expect(tc_saddr(&S.load[0]), sizeof(S.w1));
    tr_bulk(S.w1, T.W1b, sizeof(S.w1), tc_saddr(&S.load[0]));
    tr_expect(tc_saddr(&S.load[1]), sizeof(S.w2));
    tr_bulk(S.w2, T.W2b, sizeof(S.w2), tc_saddr(&S.load[1]));
  }
  if (tid < MLP_H) S.b1[tid] = b1[tid];
  else if (tid < 2 * MLP_H) S.b2[tid - MLP_H] = b2[tid - MLP_H];
  else if (tid < 3 * MLP_H) S.w3[tid - 2 * MLP_H] = w3[tid - 2 * MLP_H];
  else if (tid == 3 * MLP_H) S.stop = *(volatile unsigned *)T.err;  // a wait of an earlier step ran out: no more steps
  const float bias3 = b3[0];
  if (m0 + xr < rows) *(uint4 *)(T.Xb + tr_at(T.R, m0 + xr, xk)) = xin;  // kept for the weights of the first layer
  __syncthreads();
  const TrOp X{S.x, 128, 512, false}, L1{S.w1, 128, 512, false};
  const TrOp H1{S.h1, 128, 2048, false}, L2{S.w2, 128, 2048, false};  // h2 x h1, K = h1 ...
  const TrOp D2{S.d2, 128, 2048, false}, L2t{S.w2, 2048, 128, true};  // ... and backwards h1 x h2, K = h2
  const bool stop = S.stop != 0;
  if (tid == 0 && !stop && tr_landed(tc_saddr(&S.load[0]), 0, T.err)) tr_mma(tmem, X, L1, MLP_H, MLP_IN, true, bar);
  const int quad = warp & 3, c0 = 32 * (warp >> 2);  // a warp reads its lane quadrant (warp % 4)
  const int r = 32 * quad + lane;                    // this thread's row: columns c0 .. c0 + 31
  const bool live = m0 + r < rows;
  const uint32_t mine = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)c0;
  uint32_t v[32], on1 = 0, on2 = 0;  // signs of the pre-activations: the ReLU masks
  bool ok = !stop && tr_wait(bar, phase, T.err);
  if (ok) {
    tr_ld32(mine, v);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      uint32_t h[4];
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const int c = 8 * q + j;
        const float z = __uint_as_float(v[c]) + S.b1[c0 + c];
        on1 |= (uint32_t)(z > 0.f) << c;
        v[c] = __float_as_uint(z > 0.f ? z : 0.f);
      }
#pragma unroll
      for (int j = 0; j < 4; j++) h[j] = tr_pack(__uint_as_float(v[8 * q + 2 * j]), __uint_as_float(v[8 * q + 2 * j + 1]));
      const uint4 x = make_uint4(h[0], h[1], h[2], h[3]);
      *(uint4 *)(S.h1 + tr_off<MLP_H>(r, c0 + 8 * q)) = x;
      if (live) *(uint4 *)(T.H1 + tr_at(T.R, m0 + r, (c0 >> 3) + q)) = x;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0 && tr_landed(tc_saddr(&S.load[1]), 0, T.err)) tr_mma(tmem + 128, H1, L2, MLP_H, MLP_H, true, bar);
    ok = tr_wait(bar, phase, T.err);
  }
  if (ok) {
    tr_ld32(mine + 128, v);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      uint32_t h[4];
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const int c = 8 * q + j;
        const float z = __uint_as_float(v[c]) + S.b2[c0 + c];
        on2 |= (uint32_t)(z > 0.f) << c;
        v[c] = __float_as_uint(z > 0.f ? z : 0.f);
      }
#pragma unroll
      for (int j = 0; j < 4; j++) h[j] = tr_pack(__uint_as_float(v[8 * q + 2 * j]), __uint_as_float(v[8 * q + 2 * j + 1]));
      const uint4 x = make_uint4(h[0], h[1], h[2], h[3]);
      *(uint4 *)(S.h2 + r * (MLP_H + 8) + c0 + 8 * q) = x;
      if (live) *(uint4 *)(T.H2 + tr_at(T.R, m0 + r, (c0 >> 3) + q)) = x;
    }
    __syncthreads();
    float o[OUT];  // the output layer: a warp a row (as k_out_layer), its rows side by side
#pragma unroll
    for (int i = 0; i < OUT; i++) {
      const uint16_t *h = S.h2 + (warp + (TR_THREADS / 32) * i) * (MLP_H + 8) + lane;
      o[i] = 0.f;
#pragma unroll
      for (int k = 0; k < MLP_H; k += 32) o[i] += __bfloat162float(__ushort_as_bfloat16(h[k])) * S.w3[lane + k];
    }
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
      for (int i = 0; i < OUT; i++) o[i] += __shfl_down_sync(0xffffffffu, o[i], off);
    float y = 0.f;
#pragma unroll
    for (int i = 0; i < OUT; i++) {
      const float t = __shfl_sync(0xffffffffu, o[i], 0);
      if (lane == i) y = t;
    }
    if (lane < OUT) {
      y += bias3;
      const float e = m0 + ox < m ? y - target : 0.f;
      const float d = 2.f * e / (float)m;
      S.dy[ox] = d;
      if (m0 + ox < rows) T.dy[m0 + ox] = d;
      if (m0 + ox < m) atomicAdd(loss, e * e / (float)m);
    }
    __syncthreads();
    const float d = S.dy[r];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      uint32_t h[4];
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const int c = 8 * q + 2 * j;
        h[j] = tr_pack((on2 >> c) & 1u ? d * S.w3[c0 + c] : 0.f, (on2 >> (c + 1)) & 1u ? d * S.w3[c0 + c + 1] : 0.f);
      }
      const uint4 x = make_uint4(h[0], h[1], h[2], h[3]);
      *(uint4 *)(S.d2 + tr_off<MLP_H>(r, c0 + 8 * q)) = x;
      if (live) *(uint4 *)(T.dH2 + tr_at(T.R, m0 + r, (c0 >> 3) + q)) = x;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) tr_mma(tmem + 256, D2, L2t, MLP_H, MLP_H, true, bar);
    ok = tr_wait(bar, phase, T.err);
  }
  if (ok) {
    tr_ld32(mine + 256, v);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      uint32_t h[4];
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const int c = 8 * q + 2 * j;
        h[j] = tr_pack((on1 >> c) & 1u ? __uint_as_float(v[c]) : 0.f, (on1 >> (c + 1)) & 1u ? __uint_as_float(v[c + 1]) : 0.f);
      }
      if (live) *(uint4 *)(T.dH1 + tr_at(T.R, m0 + r, (c0 >> 3) + q)) = make_uint4(h[0], h[1], h[2], h[3]);
    }
  }
  else if (tid == 0) {  // given up: the copies have still to land
    tr_landed(tc_saddr(&S.load[0]), 0, T.err);
    tr_landed(tc_saddr(&S.load[1]), 0, T.err);
  }
  tr_teardown(&S.bar, 3, tmem, COLS);
}

__device__ __forceinline__ float adam_one(float w, float gi, float *m, float *v, float m0, float v0, float lr, float b1,
                                          float b2, float eps, float c1, float c2) {
  const float mi = b1 * m0 + (1.f - b1) * gi;
  const float vi = b2 * v0 + (1.f - b2) * gi * gi;
  *m = mi;
  *v = vi;
  return w - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

constexpr int TR_KC = 256;
struct TrainSmemB {
  uint16_t a[MLP_H * TR_KC], b[32 * TR_KC];  // gradients and inputs of up to 256 samples, as they are kept
  float g[MLP_H * 33];                       // the block's gradient
  float part[256];
  unsigned long long bar, load;
  uint32_t tmem, stop;
};

// Blocks 0 .. 3: columns 32 b .. of gW2; 4: gW1; then 4 blocks each for b1's, b2's and w3's gradients (32
// columns a block), the first of the last four b3's too.
constexpr int TR_BLOCKS = 17;
__global__ void __launch_bounds__(TR_THREADS, 1) k_train_weights(const MlpTrain T, int m, float lr, float c1, float c2) {
  extern __shared__ __align__(1024) unsigned char tr_smem[];
  TrainSmemB &S = *(TrainSmemB *)tr_smem;
  const float be1 = 0.9f, be2 = 0.999f, eps = 1e-8f;
  const int tid = threadIdx.x, b = blockIdx.x, rows = (m + 15) / 16 * 16;
  const int oW1 = 0, ob1 = MLP_H * MLP_IN, oW2 = ob1 + MLP_H, ob2 = oW2 + MLP_H * MLP_H, ow3 = ob2 + MLP_H, ob3 = ow3 + MLP_H;
  auto adam = [&](int at, float g) {
    T.params[at] = adam_one(T.params[at], g, T.m + at, T.v + at, T.m[at], T.v[at], lr, be1, be2, eps, c1, c2);
  };
  if (b >= 5) {
    griddep_wait();
    griddep_launch_dependents();
    const int what = (b - 5) >> 2, c = 32 * ((b - 5) & 3) + (tid & 31);
    const bool sums = tid < 256;  // colsum32's eight warps; all threads take its barriers
    const bool stop = *(volatile unsigned *)T.err != 0;
    float t = 0.f, u = 0.f;
    auto add = [&](const __nv_bfloat16 *M, const float *wrow) {
      float s = 0.f;
      const __nv_bfloat16 *col = M + tr_at(T.R, 0, c >> 3) + (c & 7);
      if (sums)
#pragma unroll 8
        for (int r = tid >> 5; r < rows; r += 8) {
          const float x = __bfloat162float(col[8 * r]);
          s += wrow ? wrow[r] * x : x;
        }
      if (sums) S.part[tid] = s;
      __syncthreads();
      float z = 0.f;
      if (tid < 32)
        for (int k = 0; k < 8; k++) z += S.part[k * 32 + tid];
      __syncthreads();
      return z;
    };
    if (what == 0) t = add(T.dH1, nullptr);
    else if (what == 1) t = add(T.dH2, nullptr);
    else t = add(T.H2, T.dy);
    if (b == 13) {  // the column sum of dy, as colsum32 on a matrix of one column
      float s = 0.f;
      if (sums && (tid & 31) == 0)
        for (int r = tid >> 5; r < rows; r += 8) s += T.dy[r];
      if (sums) S.part[tid] = s;
      __syncthreads();
      if (tid == 0) {
        for (int k = 0; k < 8; k++) u += S.part[k * 32];
        if (!stop) {
          adam(ob3, u);
          atomicAdd(T.err + 1, 1u);  // steps taken
        }
      }
    }
    if (tid < 32 && !stop) adam((what == 0 ? ob1 : what == 1 ? ob2 : ow3) + c, t);
    return;
  }
  constexpr int COLS = 32;
  if (tid == 0) S.stop = 0;
  tr_setup(&S.bar, 2, &S.tmem, COLS);
  const uint32_t tmem = S.tmem, bar = tc_saddr(&S.bar), load = tc_saddr(&S.load);
  griddep_wait();
  griddep_launch_dependents();
  // g[o][n] = sum over samples of dH[r][o] * In[r][n]
  const __nv_bfloat16 *dH = b < 4 ? T.dH2 : T.dH1, *In = b < 4 ? T.H1 + tr_at(T.R, 0, 4 * b) : T.Xb;
  const TrOp A{S.a, 128, TR_KC * 16, true}, B{S.b, 128, TR_KC * 16, true};
  constexpr int OWN = MLP_H * 32 / TR_THREADS;
  float w[OWN], am[OWN], av[OWN];  // the block's parameters, read while the copies and products run
  auto own = [&](int j) {
    const int i = tid + j * TR_THREADS, o = i >> 5, n = i & 31;
    return b < 4 ? oW2 + o * MLP_H + 32 * b + n : oW1 + o * MLP_IN + n;
  };
  uint32_t phase = 0, phase_l = 0;
  bool ok = true;
  for (int k0 = 0; k0 < rows && ok; k0 += TR_KC) {
    const int kc = min(TR_KC, rows - k0);  // a multiple of 16
    if (tid < 32) {
      if (tid == 0) {
        asm volatile("fence.proxy.async.global;" ::: "memory");
        tr_expect(load, (uint32_t)kc * 16 * (MLP_H / 8 + 4));
      }
      __syncwarp();
      if (tid < MLP_H / 8) tr_bulk(S.a + tid * TR_KC * 8, dH + tr_at(T.R, k0, tid), (uint32_t)kc * 16, load);
      else if (tid < MLP_H / 8 + 4)
        tr_bulk(S.b + (tid - MLP_H / 8) * TR_KC * 8, In + tr_at(T.R, k0, tid - MLP_H / 8), (uint32_t)kc * 16, load);
    }
    if (k0 == 0)
#pragma unroll
      for (int j = 0; j < OWN; j++) {
        const int at = own(j);
        w[j] = T.params[at];
        am[j] = T.m[at];
        av[j] = T.v[at];
      }
    if (tid == 0) {
      if (k0 == 0) S.stop = *(volatile unsigned *)T.err;  // this step's activations are void, or an earlier step's were
      const bool up = tr_landed(load, phase_l, T.err);
      if (S.stop) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
      else if (up) tr_mma(tmem, A, B, 32, kc, k0 == 0, bar);
    }
    phase_l ^= 1u;
    ok = tr_wait(bar, phase, T.err) && !S.stop;
  }
  if (ok) {
    if (tid < 128) {
      uint32_t v[32];
      const int row = tid;  // warps 0 .. 3 read their lane quadrants
      tr_ld32(tmem + ((uint32_t)(32 * (tid >> 5)) << 16), v);
#pragma unroll
      for (int j = 0; j < 32; j++) S.g[row * 33 + j] = __uint_as_float(v[j]);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int j = 0; j < OWN; j++) {
      const int i = tid + j * TR_THREADS, o = i >> 5, n = i & 31, at = own(j);
      const float x = adam_one(w[j], S.g[o * 33 + n], T.m + at, T.v + at, am[j], av[j], lr, be1, be2, eps, c1, c2);
      T.params[at] = x;
      const uint16_t h = __bfloat16_as_ushort(__float2bfloat16_rn(x));  // for the next step's products
      if (b < 4) T.W2b[tr_off<MLP_H>(o, 32 * b + n)] = h;
      else T.W1b[tr_off<MLP_IN>(o, n)] = h;
    }
  }
  tr_teardown(&S.bar, 2, tmem, COLS);
}

// He-uniform weights from SplitMix64 (draw d from the state seed + (d + 1) * step: W1, W2, w3 in that
// order, biases zero), and zero moments.
__global__ void __launch_bounds__(256) k_mlp_init(float *params, float *m, float *v, unsigned long long seed, double a1,
                                                  double a2, double a3) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  const int ob1 = MLP_H * MLP_IN, oW2 = ob1 + MLP_H, ob2 = oW2 + MLP_H * MLP_H, ow3 = ob2 + MLP_H, n = ow3 + MLP_H + 1;
  if (i >= n) return;
  int d = -1;  // which draw
  double a = 0.0;
  if (i < ob1) d = i, a = a1;
  else if (i >= oW2 && i < ob2) d = i - MLP_H, a = a2;
  else if (i >= ow3 && i < ow3 + MLP_H) d = i - 2 * MLP_H, a = a3;
  float x = 0.f;
  if (d >= 0) {
    unsigned long long z = seed + (unsigned long long)(d + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const double u = __dmul_rn(__dadd_rn((double)(z >> 11), 0.5), 2.0 / 9007199254740992.0);
    x = __double2float_rn(__dmul_rn(a, __dadd_rn(u, -1.0)));
  }
  params[i] = x;
  m[i] = 0.f;
  v[i] = 0.f;
}

cudaError_t mlp_init(float *params, float *m, float *v, uint64_t seed, cudaStream_t s) {
  g_launches++;
  k_mlp_init<<<(unsigned)((mlp_param_count() + 255) / 256), 256, 0, s>>>(params, m, v, seed, sqrt(6.0 / MLP_IN),
                                                                       sqrt(6.0 / MLP_H), sqrt(3.0 / MLP_H));
  return cudaGetLastError();
}

int64_t mlp_train_bytes(int batch) {
  const int64_t r = (batch + 15) / 16 * 16;
  return r * MLP_IN * 2 + 4 * r * MLP_H * 2 + r * 4 + (MLP_IN + MLP_H) * MLP_H * 2 + 8 * 256;
}

void mlp_train_layout(MlpTrain &T, void *work, int batch) {
  const int64_t r = (batch + 15) / 16 * 16;
  unsigned char *p = (unsigned char *)work;
  auto take = [&](int64_t bytes) {
    void *q = p;
    p += (bytes + 255) / 256 * 256;
    return (__nv_bfloat16 *)q;
  };
  T.Xb = take(r * MLP_IN * 2);
  T.H1 = take(r * MLP_H * 2);
  T.H2 = take(r * MLP_H * 2);
  T.dH2 = take(r * MLP_H * 2);
  T.dH1 = take(r * MLP_H * 2);
  T.dy = (float *)take(r * 4);
  T.W1b = (uint16_t *)take(MLP_H * MLP_IN * 2);
  T.W2b = (uint16_t *)take(MLP_H * MLP_H * 2);
  T.R = r;
}

cudaError_t mlp_train_begin(const MlpTrain &T, cudaStream_t s) {
  g_launches++;
  k_train_begin<<<MLP_H * MLP_H / 256, 256, 0, s>>>(T);
  return cudaGetLastError();
}

cudaError_t mlp_train_step(const MlpTrain &T, const int32_t *idx, int m, float *loss, float lr, int step, cudaStream_t s) {
  static std::atomic<unsigned long long> attr_set{0};  // one bit per device ordinal below 64
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
  if (!bit || !(attr_set.load() & bit)) {
    cudaFuncSetAttribute(k_train_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmemA));
    cudaFuncSetAttribute(k_train_weights, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmemB));
    attr_set.fetch_or(bit);
  }
  const float c1 = 1.f - powf(0.9f, (float)step), c2 = 1.f - powf(0.999f, (float)step);
  cudaError_t e = launch_pdl(k_train_rows, dim3((m + TR_M - 1) / TR_M), dim3(TR_THREADS), sizeof(TrainSmemA), s, T, idx, m,
                             loss);
  if (e == cudaSuccess)
    e = launch_pdl(k_train_weights, dim3(TR_BLOCKS), dim3(TR_THREADS), sizeof(TrainSmemB), s, T, m, lr, c1, c2);
  g_launches += 2;
  return e;
}

static int blocks_for(int64_t n, int per = 256) {
  int64_t b = (n + per - 1) / per;
  return (int)(b < 1 ? 1 : (b > 4096 ? 4096 : b));
}

static cudaError_t gemm(int M, int N, int K, const __nv_bfloat16 *A, int am, int ak, const __nv_bfloat16 *Bm, int bk,
                        int bn, float *C, int ldc, int acc, unsigned *err, cudaStream_t s) {
  if (M % 16 || K % 16 || (N != 32 && N != 128) || ldc % 4 || ((uintptr_t)C & 15)) return cudaErrorInvalidValue;
  static std::atomic<unsigned long long> attr_set{0};  // one bit per device ordinal below 64
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
  if (!bit || !(attr_set.load() & bit)) {
    cudaFuncSetAttribute(k_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    attr_set.fetch_or(bit);
  }
  g_launches++;
  k_gemm_tc<<<(M + TC_M - 1) / TC_M, TC_THREADS, TC_SMEM, s>>>(M, N, K, A, am, ak, Bm, bk, bn, C, ldc, acc, err);
  return cudaGetLastError();
}

int64_t mlp_param_count() { return (int64_t)MLP_H * MLP_IN + MLP_H + MLP_H * MLP_H + MLP_H + MLP_H + 1; }

int64_t mlp_work_bytes(int rows) {
  int64_t r = rows;
  return r * MLP_IN * 2 + 2 * (r * MLP_H * 4) + 2 * (r * MLP_H * 2) + 3 * r * 4 + 2 * (r * MLP_H * 2) +
         r * MLP_H * 4 + 2 * mlp_param_count() * 2 + 4096 + 256;
}

unsigned *mlp_error_flag(void *work, int rows) {
  return (unsigned *)((unsigned char *)work + (mlp_work_bytes(rows) - 256) / 256 * 256);
}

// Forward (and, with targets, backward into grads) for `rows` samples (rows % 16 == 0; the
// first n_valid are real). X: rows x 32 FP32 on the device; params / grads: flat FP32.
cudaError_t mlp_forward_backward(const float *params, const float *X, const float *target, int rows, int n_valid,
                                 float *y, float *grads, float *loss, void *work, cudaStream_t s) {
  const float *W1 = params, *b1 = W1 + MLP_H * MLP_IN, *W2 = b1 + MLP_H, *b2 = W2 + MLP_H * MLP_H;
  const float *w3 = b2 + MLP_H, *b3 = w3 + MLP_H;
  unsigned char *p = (unsigned char *)work;
  auto take = [&](int64_t bytes) {
    void *q = p;
    p += (bytes + 255) / 256 * 256;
    return q;
  };
  __nv_bfloat16 *Xb = (__nv_bfloat16 *)take((int64_t)rows * MLP_IN * 2);
  float *Z1 = (float *)take((int64_t)rows * MLP_H * 4);
  float *Z2 = (float *)take((int64_t)rows * MLP_H * 4);
  __nv_bfloat16 *H1 = (__nv_bfloat16 *)take((int64_t)rows * MLP_H * 2);
  __nv_bfloat16 *H2 = (__nv_bfloat16 *)take((int64_t)rows * MLP_H * 2);
  float *dy = (float *)take((int64_t)rows * 4);
  __nv_bfloat16 *dH2 = (__nv_bfloat16 *)take((int64_t)rows * MLP_H * 2);
  __nv_bfloat16 *dH1 = (__nv_bfloat16 *)take((int64_t)rows * MLP_H * 2);
  float *dA1 = (float *)take((int64_t)rows * MLP_H * 4);
  __nv_bfloat16 *W1b = (__nv_bfloat16 *)take((int64_t)MLP_H * MLP_IN * 2);
  __nv_bfloat16 *W2b = (__nv_bfloat16 *)take((int64_t)MLP_H * MLP_H * 2);
  unsigned *err = mlp_error_flag(work, rows);  // raised by a tensor-core wait that ran out
  cudaError_t e = cudaMemsetAsync(err, 0, sizeof(unsigned), s);
  if (e != cudaSuccess) return e;
  int launches = 0;
  k_to_bf16<<<blocks_for((int64_t)rows * MLP_IN), 256, 0, s>>>(X, Xb, (int64_t)rows * MLP_IN);
  k_to_bf16<<<blocks_for(MLP_H * MLP_IN), 256, 0, s>>>(W1, W1b, MLP_H * MLP_IN);
  k_to_bf16<<<blocks_for(MLP_H * MLP_H), 256, 0, s>>>(W2, W2b, MLP_H * MLP_H);
  launches += 3;
  // Z1 = X W1^T: A = X (row-major), B(k, n) = W1[n][k]
  e = gemm(rows, MLP_H, MLP_IN, Xb, MLP_IN, 1, W1b, 1, MLP_IN, Z1, MLP_H, 0, err, s);
  if (e != cudaSuccess) return e;
  k_bias_relu<<<blocks_for((int64_t)rows * MLP_H), 256, 0, s>>>(Z1, b1, H1, rows, MLP_H);
  e = gemm(rows, MLP_H, MLP_H, H1, MLP_H, 1, W2b, 1, MLP_H, Z2, MLP_H, 0, err, s);
  if (e != cudaSuccess) return e;
  k_bias_relu<<<blocks_for((int64_t)rows * MLP_H), 256, 0, s>>>(Z2, b2, H2, rows, MLP_H);
  k_out_layer<<<(rows + 7) / 8, 256, 0, s>>>(H2, w3, b3, rows, n_valid, target, y, dy, loss);
  launches += 3;
  if (target && grads) {
    float *gW1 = grads, *gb1 = gW1 + MLP_H * MLP_IN, *gW2 = gb1 + MLP_H, *gb2 = gW2 + MLP_H * MLP_H;
    float *gw3 = gb2 + MLP_H, *gb3 = gw3 + MLP_H;
    k_out_backward<<<blocks_for((int64_t)rows * MLP_H), 256, 0, s>>>(dy, H2, Z2, w3, rows, dH2, gw3, gb3);
    k_colsum<<<MLP_H / 32, 256, 0, s>>>(dH2, rows, MLP_H, gb2);
    launches += 2;
    // gW2[o][i] += sum_r dH2[r][o] H1[r][i]: A(m=o, k=r) = dH2[r][o], B(k=r, n=i) = H1[r][i]
    e = gemm(MLP_H, MLP_H, rows, dH2, 1, MLP_H, H1, MLP_H, 1, gW2, MLP_H, 1, err, s);
    if (e != cudaSuccess) return e;
    // dA1[r][i] = sum_o dH2[r][o] W2[o][i]: A = dH2 (row-major), B(k=o, n=i) = W2[o][i]
    e = gemm(rows, MLP_H, MLP_H, dH2, MLP_H, 1, W2b, MLP_H, 1, dA1, MLP_H, 0, err, s);
    if (e != cudaSuccess) return e;
    k_relu_backward<<<blocks_for((int64_t)rows * MLP_H), 256, 0, s>>>(dA1, Z1, dH1, (int64_t)rows * MLP_H);
    k_colsum<<<MLP_H / 32, 256, 0, s>>>(dH1, rows, MLP_H, gb1);
    launches += 2;
    // gW1[o][j] += sum_r dH1[r][o] X[r][j]
    e = gemm(MLP_H, MLP_IN, rows, dH1, 1, MLP_H, Xb, MLP_IN, 1, gW1, MLP_IN, 1, err, s);
    if (e != cudaSuccess) return e;
  }
  g_launches += launches;
  return cudaGetLastError();
}

}  // namespace dmk
