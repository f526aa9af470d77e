// The k best rows of a table by (score, row), k <= SEL_K, in three launches and without the host: the
// row count may be read from a counter on the device.
//
// k_sel_hist counts the scores by the top 13 bits of their order-preserving keys (16 bins an octave),
// k_sel_collect finds the bin that holds the k-th smallest and collects every row up to that bin, and
// k_sel_rank gives each collected row its rank (one warp a row counts the keys before its own; equal
// keys compare the rows themselves, or their positions in a canonically sorted table) and writes it to
// its place if that is below k. Layout scores are sums of ten or more error rates, so the bin of the
// k-th best of n rows holds a few percent of them at most; a table with more than SEL_CAP rows up to
// that bin (equal scores by the thousand) is reported instead of answered. Tables of up to SEL_DIRECT
// rows are collected whole.
//
// The work is a pass over the scores for each of the first two kernels (the first is left out where the
// joins count the scores as they write the rows: chain.cu, which also prunes by the bound it finds on
// the way) and m^2 / 32 steps of the third for m rows collected; on the tables of layout queries all of
// it is launch latency, 3 + 8 + 5 us. It replaces a radix select with a read-back of the histogram to
// the host after each of four passes, a canonical sort of the selected rows and four radix passes over
// them (30 launches, 7 synchronisations). Wall clock of whole calls: best 100 of the 26 258 layouts of a
// 22-qubit circuit 640 us -> 113 us, best 10 of 3.1 M 593 us -> 143 us (254 us without the pruning). Results
// of up to 64 KB are written to the host's pinned buffer by k_sel_rank itself, and the joins' counters by
// their last block: two copies fewer behind the kernels, 90 us -> 84 and 119 -> 113 on the same calls later.
#include <cuda_runtime.h>
#include <stdint.h>

#include "join_device.cuh"
#include "kernels.h"

namespace dmk {

constexpr int SEL_BINS = SelHist::FINE, SEL_SHIFT = SelHist::FINE_SHIFT, SEL_BLK = 256, SEL_DIRECT = 2048;

constexpr int SEL_U = 4;  // scores of a thread in flight

struct SelWork {
  SelHist h;
  uint32_t m;  // rows collected
  uint32_t key[SEL_CAP];
  int32_t idx[SEL_CAP];
};

int64_t select_work_bytes() { return sizeof(SelWork); }

__device__ __forceinline__ int64_t sel_n(const SelectArgs &a) {
  return a.n_dev ? imin64((int64_t)*a.n_dev, a.n) : a.n;
}

__global__ void __launch_bounds__(SEL_BLK) k_sel_hist(const SelectArgs a) {
  __shared__ uint32_t h[SEL_BINS];
  SelWork *W = (SelWork *)a.work;
  for (int i = threadIdx.x; i < SEL_BINS; i += SEL_BLK) h[i] = 0;
  __syncthreads();
  griddep_wait();
  griddep_launch_dependents();
  const int64_t n = sel_n(a);
  if (blockIdx.x == 0 && threadIdx.x == 0) W->m = n <= SEL_DIRECT ? (uint32_t)n : 0u;
  if (n <= SEL_DIRECT || a.counted) return;
  const int64_t step = (int64_t)gridDim.x * SEL_BLK;
  for (int64_t i = blockIdx.x * (int64_t)SEL_BLK + threadIdx.x; i < n; i += SEL_U * step) {
    float x[SEL_U];
#pragma unroll
    for (int u = 0; u < SEL_U; u++) x[u] = i + u * step < n ? __ldg(a.sc + i + u * step) : 0.f;
#pragma unroll
    for (int u = 0; u < SEL_U; u++)
      if (i + u * step < n) atomicAdd(&h[score_key(x[u]) >> SEL_SHIFT], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < SEL_BINS; i += SEL_BLK)
    if (h[i]) atomicAdd(&W->h.fine[i], h[i]);
}

__global__ void __launch_bounds__(SEL_BLK) k_sel_collect(const SelectArgs a) {
  __shared__ int s_warp[SEL_BLK / 32];
  __shared__ uint32_t s_top;
  SelWork *W = (SelWork *)a.work;
  griddep_wait();
  griddep_launch_dependents();
  const int64_t n = sel_n(a);
  const int lane = threadIdx.x & 31;
  uint32_t top = ~0u;  // the largest key collected
  if (n > SEL_DIRECT) {
    constexpr int PER = SEL_BINS / SEL_BLK;
    uint32_t c[PER];
    int sum = 0;
#pragma unroll
    for (int j = 0; j < PER / 4; j++) {
      const uint4 x = ((const uint4 *)W->h.fine)[threadIdx.x * (PER / 4) + j];
      c[4 * j] = x.x;
      c[4 * j + 1] = x.y;
      c[4 * j + 2] = x.z;
      c[4 * j + 3] = x.w;
      sum += (int)(x.x + x.y + x.z + x.w);
    }
    int total;
    int before = block_excl_scan<SEL_BLK>(sum, total, s_warp);
    const int kk = (int)imin64(a.k, n);
    if (before < kk && kk <= before + sum) {  // one thread: the bin of the kk-th smallest
      int j = 0;
      while (before + (int)c[j] < kk) before += (int)c[j++];
      s_top = ((uint32_t)(threadIdx.x * PER + j) << SEL_SHIFT) | ((1u << SEL_SHIFT) - 1);
    }
    __syncthreads();
    top = s_top;
  }
  const int64_t step = (int64_t)gridDim.x * SEL_BLK;
  for (int64_t i0 = blockIdx.x * (int64_t)SEL_BLK + threadIdx.x - lane; i0 < n; i0 += SEL_U * step) {
    float x[SEL_U];
#pragma unroll
    for (int u = 0; u < SEL_U; u++) x[u] = i0 + u * step + lane < n ? __ldg(a.sc + i0 + u * step + lane) : 0.f;
#pragma unroll
    for (int u = 0; u < SEL_U; u++) {
      const int64_t i = i0 + u * step + lane;
      const uint32_t key = score_key(x[u]);
      const bool take = i < n && key <= top;
      uint32_t at = (uint32_t)i;
      if (n > SEL_DIRECT) {
        const unsigned bal = __ballot_sync(FULL_MASK, take);
        if (bal == 0) continue;
        if (lane == 0) at = atomicAdd(&W->m, (uint32_t)__popc(bal));
        at = __shfl_sync(FULL_MASK, at, 0) + __popc(bal & lanemask_lt());
      }
      if (take && at < SEL_CAP) {
        W->key[at] = key;
        W->idx[at] = (int32_t)i;
      }
    }
  }
}

__device__ __forceinline__ bool sel_row_before(const SelectArgs &a, int32_t x, int32_t y) {
  if (!a.sorted) {
    const int32_t *rx = a.rows + (int64_t)x * a.w, *ry = a.rows + (int64_t)y * a.w;
    for (int c = 0; c < a.w; c++) {
      const int32_t p = __ldg(rx + c), q = __ldg(ry + c);
      if (p != q) return p < q;
    }
  }
  return x < y;
}

__global__ void __launch_bounds__(SEL_BLK) k_sel_rank(const SelectArgs a) {
  SelWork *W = (SelWork *)a.work;
  griddep_wait();
  griddep_launch_dependents();
  const int lane = threadIdx.x & 31;
  const uint32_t m = W->m;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ((uint32_t *)a.out)[0] = m;
    if (a.h_out) ((uint32_t *)a.h_out)[0] = m;
  }
  for (int i = blockIdx.x * SEL_BLK + threadIdx.x; i < SEL_BINS; i += gridDim.x * SEL_BLK) {
    W->h.fine[i] = 0;
    if (i < SelHist::COARSE) W->h.coarse[i] = 0;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) W->h.bound = SEL_NO_BOUND;
  if (m > SEL_CAP) return;
  float *osc = (float *)(a.out + 16);
  int32_t *orows = (int32_t *)(osc + a.k);
  float *hsc = (float *)(a.h_out + 16);
  int32_t *hrows = (int32_t *)(hsc + a.k);
  for (uint32_t i = (blockIdx.x * SEL_BLK + threadIdx.x) >> 5; i < m; i += (gridDim.x * SEL_BLK) >> 5) {
    const uint32_t key = W->key[i];
    const int32_t row = W->idx[i];
    unsigned rank = 0;
    for (uint32_t j = lane; j < m; j += 32) {
      const uint32_t o = W->key[j];
      if (o < key || (o == key && j != i && sel_row_before(a, W->idx[j], row))) rank++;
    }
    rank = __reduce_add_sync(FULL_MASK, rank);
    if (rank >= (unsigned)a.k) continue;
    const float sc = __ldg(a.sc + row);
    if (lane == 0) osc[rank] = sc;
    if (lane == 0 && a.h_out) hsc[rank] = sc;
    for (int c = lane; c < a.w; c += 32) {
      const int64_t at = (int64_t)rank * a.w + c;
      const int32_t v = __ldg(a.rows + (int64_t)row * a.w + c);
      orows[at] = v;
      if (a.h_out) hrows[at] = v;
    }
  }
}

cudaError_t topk_select(const SelectArgs &a, int num_sms, cudaStream_t s) {
  const int64_t most = 2ll * num_sms, need = (a.n + 4 * SEL_BLK - 1) / (4 * SEL_BLK);
  const int grid = (int)(need < 1 ? 1 : need < most ? need : most);
  launch_pdl(k_sel_hist, dim3(grid), dim3(SEL_BLK), 0, s, a);
  launch_pdl(k_sel_collect, dim3(grid), dim3(SEL_BLK), 0, s, a);
  launch_pdl(k_sel_rank, dim3(num_sms), dim3(SEL_BLK), 0, s, a);
  g_launches += 3;
  return cudaGetLastError();
}

}  // namespace dmk
