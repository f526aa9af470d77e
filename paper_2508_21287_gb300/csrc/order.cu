// Canonical (lexicographic) order of a table of embeddings whose row count is known on the device only:
// four launches that can follow the joins without the host.
//
// A row's key is exact and short. In lexicographic order a column is compared only between rows that
// agree on all columns before it; if one of those, c', holds the image of a pattern neighbour, the
// column is a neighbour of f(c') in the data graph, and its place in that sorted neighbour list (below
// the largest degree) orders like its id. Columns without an earlier neighbour keep their id. The digits
// are packed with their exact radices into up to ORD_KW words: a line's row of 15 ids on 3999 vertices is
// a number below 3999 * 3^14, one word instead of 180 bits. Columns past the words are compared in the
// rows themselves.
//
// Such keys spread well over their range (all columns after a vertex's image are near it, so a scrambled
// pattern's keys crowd somewhat), so the rows are dealt by them into buckets: one to ORD_PER rows up to
// ORD_FEW buckets, and one to 64 rows in larger tables (11.8 M rows do not fit ORD_FEW buckets of ORD_BUCKET
// rows, and the merge sort that ordered them instead took 9 ms).
// k_ord_keys packs the keys, sums the rows' checksum and takes every row's number in its bucket,
// k_ord_scan finds the buckets' places, k_ord_deal puts the rows' indices there, and k_ord_rank orders
// each bucket's rows in shared memory (a warp a bucket; a block for the few large ones) and copies rows and
// scores to their final places. A bucket of more than ORD_BUCKET rows is reported. The caller tries large tables again with
// the row count in hand, buckets of ORD_FINE and blocks that order up to ORD_CROWDED rows by keys they leave
// in memory, and sorts another way where that is not enough.
//
// What bounds it: instructions of k_ord_keys (the checksum's 16 a column above all) and k_ord_rank, about
// 50 us each for 745 000 rows of 15 ids, 10 and 8 us for the two between. It replaces a merge sort on
// 180-bit keys (a tile sort and ten merge passes over three-word keys, 480 us); the whole call, joins and
// the caller's copy included, went from 740 to 407 us. Ranking every bucket by comparing all pairs took
// 180 us with 64-bit keys and three times as long on the crowded keys of layout queries. Large tables, the
// call with the merge sort and so: 11.8 M rows of a 19-vertex path on heavy-hex 53x59 9.3 -> 5.1 ms, 61 M of a
// 12-vertex path on a random 3-regular graph 48 -> 15 ms; 15 M rows of a 20-vertex path on heavy-hex 53x59
// with its columns scrambled in two ways (finer buckets at once) 13.1 -> 12.0 and 12.5 -> 7.3 ms. Finer buckets for scrambled columns at the
// first attempt cost tables of a million rows half as much again (382 -> 580 us: four times the empty
// buckets), and one addition a bucket and warp instead of one a row 1 % on layout queries.
#include <cuda_runtime.h>
#include <stdint.h>

#include "join_device.cuh"
#include "kernels.h"

namespace dmk {

constexpr int ORD_WARPS = 4, ORD_BLK = 32 * ORD_WARPS, ORD_SCAN = 1024;
constexpr int ORD_FEW = 16384, ORD_PER = 4;  // buckets of ORD_PER rows, up to ORD_FEW of them
constexpr int ORD_SMALL = ORD_BUCKET / ORD_WARPS;  // rows of a bucket that one warp ranks

__device__ __forceinline__ int64_t ord_n(const OrderArgs &a) {
  const int64_t n = a.n_dev ? (int64_t)*a.n_dev : a.n;
  return n <= a.cap ? n : 0;  // a table that does not fit is left alone
}

__device__ __forceinline__ int ord_buckets(const OrderArgs &a, int64_t n) {
  return (int)imax64(1, imin64(ORD_MAX, imax64(imin64(ORD_FEW, n / ORD_PER), n >> a.log2_many)));
}

// Bucket of a row by the first word of its key: a fraction of the word's range.
__device__ __forceinline__ int ord_bucket(const OrderArgs &a, unsigned long long key0, int nb) {
  return (int)__umul64hi(key0 * a.scale, (unsigned long long)nb);
}

template <int KW>
__global__ void __launch_bounds__(ORD_BLK) k_ord_keys(const __grid_constant__ OrderArgs a) {
  extern __shared__ int32_t tile[];
  __shared__ unsigned long long s_red[ORD_WARPS];
  griddep_wait();
  griddep_launch_dependents();
  const int64_t n = ord_n(a);
  const int nb = ord_buckets(a, n), w = a.w, ws = w | 1;  // odd stride: a column's reads fall on all banks
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t *T = tile + wid * 32 * ws;
  unsigned long long hs = 0;
  for (int64_t i0 = (blockIdx.x * (int64_t)ORD_WARPS + wid) * 32; i0 < n; i0 += (int64_t)gridDim.x * ORD_BLK) {
    const int nr = (int)imin64(32, n - i0);
    const int32_t *src = a.rows + i0 * w;
    int r = lane / w, c = lane - r * w;  // word e = r * w + c, advanced with carry
    const int dr = 32 / w, dc = 32 % w;
    for (int e = lane; e < nr * w; e += 32) {
      T[r * ws + c] = __ldg(src + e);
      r += dr;
      c += dc;
      if (c >= w) {
        c -= w;
        r++;
      }
    }
    __syncwarp();
    if (lane < nr) {
      const int32_t *row = T + lane * ws;
      unsigned long long key[KW], k = 0, p = 0;
      int word = 0;
#pragma unroll
      for (int j = 0; j < KW; j++) key[j] = 0;
      for (int x = 0; x < w; x++) {
        const int32_t v = row[x];
        p += col_term(x, v);
        if (x >= a.packed) continue;
        if (a.word[x] != word) {
#pragma unroll
          for (int j = 0; j < KW; j++)
            if (word == j) key[j] = k;
          word++;
          k = 0;
        }
        if (a.ref[x] == ORD_NONE) {
          k = k * (unsigned)a.radix_id + (unsigned)v;
        } else {  // its place among the neighbours of an earlier column's vertex
          const uint2 q = __ldg(a.adj4 + row[a.ref[x]]);  // ascending, 0xFFFF past the degree
          const unsigned code = ((q.x & 0xFFFFu) < (unsigned)v) + ((q.x >> 16) < (unsigned)v) + ((q.y & 0xFFFFu) < (unsigned)v);
          k = k * (unsigned)a.radix_place + code;
        }
      }
#pragma unroll
      for (int j = 0; j < KW; j++) {
        if (word == j) key[j] = k;
        a.key[j * a.cap + i0 + lane] = key[j];
      }
      hs += dmix64(p + (unsigned long long)(uint32_t)w);
      a.num[i0 + lane] = (int32_t)atomicAdd(&a.work->count[ord_bucket(a, key[0], nb)], 1u);
    }
    __syncwarp();
  }
  const unsigned long long t = block_sum_u64<ORD_BLK>(hs, s_red);
  if (threadIdx.x == 0 && t) atomicAdd(a.ctr + CTR_SUM, t);
}

// Exclusive scan of the bucket counts (which are zeroed for the next call).
__global__ void __launch_bounds__(ORD_SCAN) k_ord_scan(const __grid_constant__ OrderArgs a) {
  __shared__ int s_warp[ORD_SCAN / 32];
  __shared__ int s_most;
  if (threadIdx.x == 0) s_most = 0;
  griddep_wait();
  griddep_launch_dependents();
  const int64_t n = ord_n(a);
  const int nb = ord_buckets(a, n);
  constexpr int PER = ORD_FEW / ORD_SCAN;  // counts past nb are zero
  int most = 0, carry = 0;
  for (int b0 = 0; b0 < nb; b0 += ORD_FEW) {
    const int b = b0 + threadIdx.x * PER;
    uint4 *count = (uint4 *)(a.work->count + b);
    uint4 x[PER / 4];
    int sum = 0;
#pragma unroll
    for (int i = 0; i < PER / 4; i++) {
      x[i] = b + 4 * i < nb ? count[i] : make_uint4(0, 0, 0, 0);
      sum += (int)(x[i].x + x[i].y + x[i].z + x[i].w);
      most = max(max(most, max((int)x[i].x, (int)x[i].y)), max((int)x[i].z, (int)x[i].w));
    }
    int total;
    int at = carry + block_excl_scan<ORD_SCAN>(sum, total, s_warp);
    carry += total;
#pragma unroll
    for (int i = 0; i < PER / 4; i++) {
      if (b + 4 * i >= nb) break;
      uint4 s;
      s.x = (uint32_t)at;
      s.y = s.x + x[i].x;
      s.z = s.y + x[i].y;
      s.w = s.z + x[i].z;
      at = (int)(s.w + x[i].w);
      ((uint4 *)(a.work->start + b))[i] = s;
      count[i] = make_uint4(0, 0, 0, 0);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) a.work->start[nb] = (uint32_t)carry;
  atomicMax(&s_most, most);
  __syncthreads();
  if (threadIdx.x == 0) a.ctr[CTR_OVF] = (n != (a.n_dev ? (int64_t)*a.n_dev : a.n)) || s_most > (a.n_dev ? ORD_BUCKET : ORD_CROWDED);
}

__global__ void __launch_bounds__(256) k_ord_deal(const __grid_constant__ OrderArgs a) {
  griddep_wait();
  griddep_launch_dependents();
  if (a.ctr[CTR_OVF]) return;
  const int64_t n = ord_n(a);
  const int nb = ord_buckets(a, n);
  for (int64_t i = blockIdx.x * (int64_t)256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
    a.idx[a.work->start[ord_bucket(a, a.key[i], nb)] + a.num[i]] = (int32_t)i;
}

template <int KW>
struct OrdSmem {
  __align__(16) unsigned long long key[KW][ORD_BUCKET];
  int32_t idx[ORD_BUCKET];
  uint16_t order[ORD_BUCKET];  // rank -> row of the bucket
};

// The order of rows by key (read through key(j, x), of row number x) and then by the columns past it.
template <int KW, class Key, class Row>
__device__ __forceinline__ bool ord_before(const OrderArgs &a, Key key, Row row, int x, int y) {
#pragma unroll
  for (int j = 0; j < KW; j++) {
    const unsigned long long p = key(j, x), q = key(j, y);
    if (p != q) return p < q;
  }
  const int32_t ix = row(x), iy = row(y);
  if (a.packed != a.w) {
    const int32_t *rx = a.rows + (int64_t)ix * a.w, *ry = a.rows + (int64_t)iy * a.w;
    for (int c = a.packed; c < a.w; c++) {
      const int32_t p = __ldg(rx + c), q = __ldg(ry + c);
      if (p != q) return p < q;
    }
  }
  return ix < iy;
}

// A bitonic network of T threads over order[0 .. P), P the power of two from m up: numbers of rows by
// before(x, y), with m and above past every row.
template <int T, class Before>
__device__ __forceinline__ void ord_network(uint16_t *order, int t, int m, Before before) {
  int P = 1;
  while (P < m) P *= 2;
  for (int i = t; i < P; i += T) order[i] = (uint16_t)i;
  if (T == 32) __syncwarp();
  else __syncthreads();
  for (int k = 2; k <= P; k *= 2)
    for (int j = k / 2; j > 0; j /= 2) {
      for (int e = t; e < P / 2; e += T) {
        const int i = 2 * e - (e & (j - 1));
        const uint16_t x = order[i], y = order[i + j];
        const bool up = x >= m || y >= m ? y < x : before(y, x);
        if (up == ((i & k) == 0)) {
          order[i] = y;
          order[i + j] = x;
        }
      }
      if (T == 32) __syncwarp();
      else __syncthreads();
    }
}

// Rows and scores of the m rows row(0) .. row(m - 1) to their places from lo on, by T threads: a thread
// keeps its column (of several rows at a time where they are narrow).
template <int T, class Row>
__device__ __forceinline__ void ord_write(const OrderArgs &a, int t, int64_t lo, int m, Row row) {
  const int w = a.w, per = max(1, T / w), r0 = t / w;
  if (w <= T) {
    const int c = t - r0 * w;
    if (r0 < per) {
      int32_t *out = a.out + lo * w + c;
#pragma unroll 4
      for (int r = r0; r < m; r += per) out[r * w] = __ldg(a.rows + (int64_t)row(r) * w + c);
    }
  } else {
    for (int r = 0; r < m; r++) {
      const int32_t *src = a.rows + (int64_t)row(r) * w;
      for (int c = t; c < w; c += T) a.out[(lo + r) * w + c] = __ldg(src + c);
    }
  }
  if (a.sc)
    for (int i = t; i < m; i += T) a.outs[lo + i] = __ldg(a.sc + row(i));
  if (T == 32) __syncwarp();
  else __syncthreads();
}

// Order the m rows of the bucket that starts at lo, by T threads (a warp or the block) that share the
// places from `at` on (a multiple of 4), and write them out. LOCAL: the bucket's keys are not below `base`,
// are below base + 2^32 - 1 and decide alone.
template <int KW, int T, bool LOCAL>
__device__ __forceinline__ void ord_bucket_out(const OrderArgs &a, OrdSmem<KW> &S, int at, int64_t lo, int m,
                                               unsigned long long base) {
  const int t = T == 32 ? threadIdx.x & 31 : threadIdx.x;
  uint32_t *local = (uint32_t *)S.key[0] + at;
  for (int i = t; i < (LOCAL ? (m + 3) / 4 * 4 : m); i += T) {
    if (LOCAL && i >= m) {
      local[i] = ~0u;
      continue;
    }
    const int32_t x = __ldg(a.idx + lo + i);
    S.idx[at + i] = x;
    if (LOCAL) {
      local[i] = (uint32_t)(__ldg(a.key + x) - base);
    } else {
#pragma unroll
      for (int j = 0; j < KW; j++) S.key[j][at + i] = __ldg(a.key + j * a.cap + x);
    }
  }
  if (T == 32) __syncwarp();
  else __syncthreads();
  if (LOCAL) {
    const uint4 *l4 = (const uint4 *)local;
    for (int i = t; i < m; i += T) {
      const uint32_t k = local[i];
      int rank = 0;
#pragma unroll 4
      for (int o = 0; o < (m + 3) / 4; o++) {
        const uint4 x = l4[o];
        rank += (x.x < k) + (x.y < k) + (x.z < k) + (x.w < k);
      }
      S.order[at + rank] = (uint16_t)i;
    }
  } else {
    auto key = [&](int j, int x) { return S.key[j][at + x]; };
    auto row = [&](int x) { return S.idx[at + x]; };
    ord_network<T>(S.order + at, t, m, [&](int x, int y) { return ord_before<KW>(a, key, row, x, y); });
  }
  if (T == 32) __syncwarp();
  else __syncthreads();
  ord_write<T>(a, t, lo, m, [&](int r) { return S.idx[at + S.order[at + r]]; });
}

// The same for a bucket of more rows than shared memory holds keys of: the block reads them where they lie.
// Such buckets are few (a 20-vertex path with scrambled columns on 16 082 vertices: 24 % of its rows).
template <int KW>
__device__ __forceinline__ void ord_crowded_out(const OrderArgs &a, OrdSmem<KW> &S, int64_t lo, int m) {
  static_assert(sizeof(S) >= 2 * ORD_CROWDED, "the order of a crowded bucket takes the place of the keys");
  uint16_t *order = (uint16_t *)&S;
  auto row = [&](int x) { return __ldg(a.idx + lo + x); };
  auto key = [&](int j, int x) { return __ldg(a.key + j * a.cap + row(x)); };
  ord_network<ORD_BLK>(order, threadIdx.x, m, [&](int x, int y) { return ord_before<KW>(a, key, row, x, y); });
  ord_write<ORD_BLK>(a, threadIdx.x, lo, m, [&](int r) { return row(order[r]); });
}

// CROWDED: buckets of more than ORD_BUCKET rows are ordered, too.
template <int KW, bool CROWDED>
__global__ void __launch_bounds__(ORD_BLK) k_ord_rank(const __grid_constant__ OrderArgs a) {
  __shared__ OrdSmem<KW> S;
  __shared__ int s_large;
  griddep_wait();
  griddep_launch_dependents();
  const int64_t n = ord_n(a);
  if (n == 0 || a.ctr[CTR_OVF]) return;
  const int nb = ord_buckets(a, n), wid = threadIdx.x >> 5;
  // bucket b holds the keys k with b <= k * scale * nb / 2^64 < b + 1, at most 2^64 / (nb * scale) + 1 of them:
  // none below b * width, and width less than b + 2 short of a bucket (a division for each bucket instead took
  // 2 us of 20 here, and 8 of a call)
  const unsigned long long width = a.unit / nb;  // floor((2^64 - 1) / (nb * scale))
  const bool local = KW == 1 && a.packed == a.w && width < 0xFFFFFFFFull - 2 * ORD_MAX;
  auto base = [&](int b) { return width * (unsigned long long)b; };
  if (threadIdx.x == 0) s_large = 0;
  __syncthreads();
  for (int b = blockIdx.x * ORD_WARPS + wid; b < nb; b += gridDim.x * ORD_WARPS) {
    const int64_t lo = a.work->start[b];
    const int m = (int)((int64_t)a.work->start[b + 1] - lo);
    if (m > ORD_SMALL) s_large = 1;
    else if (m > 0 && local) ord_bucket_out<KW, 32, true>(a, S, wid * ORD_SMALL, lo, m, base(b));
    else if (m > 0) ord_bucket_out<KW, 32, false>(a, S, wid * ORD_SMALL, lo, m, 0);
  }
  __syncthreads();
  if (!s_large) return;
  for (int b0 = blockIdx.x * ORD_WARPS; b0 < nb; b0 += gridDim.x * ORD_WARPS)
    for (int b = b0; b < b0 + ORD_WARPS && b < nb; b++) {
      const int64_t lo = a.work->start[b];
      const int m = (int)((int64_t)a.work->start[b + 1] - lo);
      if (CROWDED && m > ORD_BUCKET) ord_crowded_out<KW>(a, S, lo, m);
      else if (m > ORD_SMALL) ord_bucket_out<KW, ORD_BLK, false>(a, S, 0, lo, m, 0);
    }
}

int64_t order_work_bytes() { return sizeof(OrderWork); }

// The words of the columns, and the scale of the first one; returns the words (at least 1).
int order_layout(OrderArgs &a, unsigned radix_id, unsigned radix_place) {
  a.radix_id = (int32_t)radix_id;
  a.radix_place = (int32_t)radix_place;
  a.packed = a.w;
  bool skewed = false;  // ids of several columns in the first word: they lie near each other
  int word = 0;
  unsigned long long range[ORD_KW] = {1, 1, 1, 1};
  for (int c = 0; c < a.w; c++) {
    const unsigned r = a.ref[c] == ORD_NONE ? radix_id : radix_place;
    if (range[word] > ~0ull / r) {
      if (word + 1 == ORD_KW) {
        a.packed = c;
        break;
      }
      word++;
    }
    range[word] *= r;
    a.word[c] = (uint8_t)word;
    skewed |= c && word == 0 && a.ref[c] == ORD_NONE;
  }
  a.scale = ~0ull / range[0];
  a.unit = ~0ull / a.scale;
  a.log2_many = skewed && !a.n_dev ? ORD_FINE : 6;
  return word + 1;
}

template <int KW>
static void order_launch(const OrderArgs &a, int num_sms, cudaStream_t s) {
  const size_t smem = (size_t)ORD_BLK * (a.w | 1) * 4;  // at most 66 KB
  static std::atomic<unsigned long long> attr{0};       // one bit per device ordinal below 64
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
  if (!bit || !(attr.load() & bit)) {
    cudaFuncSetAttribute(k_ord_keys<KW>, cudaFuncAttributeMaxDynamicSharedMemorySize, ORD_BLK * (MAXW | 1) * 4);
    attr.fetch_or(bit);
  }
  launch_pdl(k_ord_keys<KW>, dim3(6 * num_sms), dim3(ORD_BLK), smem, s, a);
  launch_pdl(k_ord_scan, dim3(1), dim3(ORD_SCAN), 0, s, a);
  launch_pdl(k_ord_deal, dim3(4 * num_sms), dim3(256), 0, s, a);
  launch_pdl(a.n_dev ? k_ord_rank<KW, false> : k_ord_rank<KW, true>, dim3(8 * num_sms), dim3(ORD_BLK), 0, s, a);
}

cudaError_t order_rows(const OrderArgs &a, int kw, int num_sms, cudaStream_t s) {
  switch (kw) {
    case 1: order_launch<1>(a, num_sms, s); break;
    case 2: order_launch<2>(a, num_sms, s); break;
    case 3: order_launch<3>(a, num_sms, s); break;
    default: order_launch<4>(a, num_sms, s); break;
  }
  g_launches += 4;
  return cudaGetLastError();
}

}  // namespace dmk
