// A plan's join chain (Alg. 1, one step after the other) without tables in device memory: the
// rows between the steps live in shared memory, several steps (often the whole plan) a launch.
//
// Every warp owns a stack of small tiles, one per step, that hold the rows waiting to be joined
// by that step. It takes a few rows of the launch's input at a time, and always joins the deepest
// tile that holds 32 rows (one row per lane, each lane walking its own key group), so lanes stay
// full and the stack stays bounded: a step is interrupted as soon as the next tile holds 32 rows
// and resumed when those are done. Only when the input is used up are partly filled tiles joined,
// shallowest first. Warps share nothing but the counter that deals out the input and the totals.
//
// A tile row is 16-bit ids (V <= 65 534) in chunks of four, chunk k of slot s at 512 k + 8 s: a
// lane's loads and stores of whole chunks are free of bank conflicts, and a survivor's row is its
// parent's chunks, still in registers, with the new ids put over them. A row keeps what later
// steps still read: a counted plan carries the sum of the row's checksum terms instead of its
// columns, a column's place is given to a new vertex after its last use, and chunks past the last
// place in use are not kept. (A stale id is that of a mapped vertex all the same, so comparing a
// new vertex with it rejects nothing wrongly.)
//
// FilterOverlappingNodes compares a new vertex p only with the columns q it can collide with.
// Let d be the distance of p and q along the pattern edges enforced so far and suppose
// f(p) = f(q) with d smallest among all colliding pairs: the images of a shortest path from p to
// q are then a closed walk whose inner vertices are distinct, that is d = 2 (the walk turns
// back) or a simple cycle of length d in the data graph. Pairs with d = 1, 2 < d < girth, or
// d odd in a bipartite data graph need no test, nor do pairs inside one motif row. In a bipartite
// graph the two colour classes of the pattern have their places in different chunks, so that a
// new vertex meets the chunks of its own class only.
//
// What the candidates of a key bring is written before the chain by k_chain_tables, in groups of one
// size per key, so that a lane finds its group without a lookup and reads four candidates with one load:
// a lane's group is another line than its neighbour's, and the tag lookups of such loads are what the
// first-level cache spends most of its time on. One new vertex: four ids (8 bytes) a key. Three: 8
// bytes a candidate (three ids and the group's length), and apart from them, read by survivors only,
// the sum of the candidate's checksum terms.
//
// What bounds it: instructions and the latency of the candidates' loads (second-level cache) at 16 warps
// an SM, whose tiles take all shared memory; about 130 warp instructions for 32 candidates and 2 a
// cycle and SM, where the launch-per-step kernel (k_joinw) needs about 450 and moves every table
// through device memory. Counts, wall clock, that kernel against this one: 24-vertex path on heavy-hex
// 53x59 5.21 ms -> 2.28 ms (53 M embeddings, 251 M candidates), 37-vertex patch there 1.60 -> 0.86 ms,
// 10-vertex path on the 60x60 grid 1.81 -> 0.66 ms, 13-vertex path on a random 3-regular graph of 4096
// vertices 0.58 -> 0.30 ms. Steps on the way (24-vertex path): columns of half-words copied one by one
// 9.0 ms, chunks of four 5.0, candidates in groups of one size 2.9, chunks by colour class and the last
// step counted on the spot 2.5, the key's own neighbours left out 2.2. Unrolling every step for every
// number of chunks in one kernel cost more in instruction-cache misses than it saved (3.0).
#include <cuda_runtime.h>
#include <stdint.h>

#include "join_device.cuh"
#include "kernels.h"

namespace dmk {

constexpr int CH_WARPS = CH_CTA_WARPS, CH_BLK = 32 * CH_WARPS;

__global__ void k_chain_tables(const __grid_constant__ ChainTables R) {
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
  griddep_launch_dependents();
  for (int64_t i = t0; i < R.n_ctr; i += nt) R.ctr[i] = 0ull;
  int j = 0;
  for (int64_t e = t0; e < R.total; e += nt) {
    while (e >= R.tab[j].end) j++;
    const ChainTables::Tab &s = R.tab[j];
    const int64_t o = e - (j ? R.tab[j - 1].end : 0);  // the entry's place
    int64_t m = o;                                     // and its motif row
    uint32_t len = 1;
    if (s.group) {
      const int64_t key = o / s.group, c = o - key * s.group;
      const int32_t first = __ldg(s.offsets + key);
      m = first + c;
      len = (uint32_t)(__ldg(s.offsets + key + 1) - first);
      if (c >= len) m = -1;
    }
    const int32_t *row = s.rows + m * s.mw;
    if (s.kind == CH_TAB_ID) {
      ((uint16_t *)s.out)[o] = m < 0 ? 0xFFFF : (uint16_t)__ldg(row + s.mpos[0]);
      continue;
    }
    if (s.kind == CH_TAB_ID3) {
      uint2 v = make_uint2(~0u, (len << 16) | 0xFFFFu);
      if (m >= 0) {
        v.x = (uint32_t)__ldg(row + s.mpos[0]) | ((uint32_t)__ldg(row + s.mpos[1]) << 16);
        v.y = (uint32_t)__ldg(row + s.mpos[2]) | (len << 16);
      }
      ((uint2 *)s.out)[o] = v;
      continue;
    }
    if (m < 0) continue;
    uint32_t h[4] = {0, 0, 0, 0};  // ids, two a word
    unsigned long long p = 0;
    float sc = s.score ? __ldg(s.score + m) : 0.f;
    for (int i = 0; i < s.n_new; i++) {
      const int32_t v = __ldg(row + s.mpos[i]);
      const uint32_t x = (uint32_t)v << (16 * (i & 1));
#pragma unroll
      for (int k = 0; k < 4; k++)
        if (i >> 1 == k) h[k] |= x;
      if (s.npos[i]) {
        p += pos_term(s.npos[i], v);
        if (R.qerr) sc += __ldg(R.qerr + v);
      }
    }
    if (s.kind == CH_TAB_SUM) {
      ((unsigned long long *)s.out)[o] = p;
    } else if (s.kind == CH_TAB_SCORE) {
      ((float *)s.out)[o] = sc;
    } else {
      const unsigned long long tail = R.mode == 1 ? p : (unsigned long long)__float_as_uint(sc);
      uint4 *d = (uint4 *)s.out + o * s.units;
      if (s.units == 1) {
        d[0] = make_uint4(h[0], h[1], (uint32_t)tail, (uint32_t)(tail >> 32));
      } else {
        d[0] = make_uint4(h[0], h[1], h[2], h[3]);
        d[1] = make_uint4((uint32_t)tail, (uint32_t)(tail >> 32), 0u, 0u);
      }
    }
  }
}

// Index lookup of a step: the lane's key group.
__device__ __forceinline__ void ch_lookup(const ChainStep &s, uint32_t ka, uint32_t kb, int32_t &start, int32_t &len) {
  if (s.nkeys == 1) {
    start = __ldg(s.offsets + ka);
    len = __ldg(s.offsets + ka + 1) - start;
    return;
  }
  const unsigned long long key = ((unsigned long long)ka << 32) | kb;
  const unsigned long long mask = (1ull << s.log2cap) - 1;
  unsigned long long h = (key * 0x9E3779B97F4A7C15ull) >> (64 - s.log2cap);
  start = 0;
  len = 0;
  for (unsigned long long probe = 0; probe <= mask; probe++) {
    const HashSlot *sl = s.slots + h;
    const unsigned long long k = sl->key;
    if (k == key) {
      start = sl->start;
      len = sl->len;
      break;
    }
    if (k == HASH_EMPTY) break;
    h = (h + 1) & mask;
  }
}

__device__ __forceinline__ bool ch_adjacent(const ChainArgs &A, int32_t u, int32_t v) {
  const unsigned long long word = __ldg(A.adj + (int64_t)u * A.adj_words + (v >> 6));
  return (word >> (v & 63)) & 1ull;
}

__device__ __forceinline__ float ch_edge_weight(const ChainArgs &A, int32_t u, int32_t v) {
  int32_t lo = __ldg(A.row_ptr + u), hi = __ldg(A.row_ptr + u + 1);
  while (lo < hi) {
    const int32_t mid = (lo + hi) >> 1, x = __ldg(A.col_idx + mid);
    if (x == v) return __ldg(A.eerr + mid);
    if (x < v) lo = mid + 1;
    else hi = mid;
  }
  return 0.f;
}

// A tile of the warp's memory: per slot the checksum sum or score (8 bytes), the state of an
// interrupted step per lane (start of its key group, and its length in the top byte), the chunks.
constexpr int CH_ROWS = 512 + 128;  // byte offset of a tile's rows
__device__ __forceinline__ unsigned long long *ch_tail(unsigned char *L) { return (unsigned long long *)L; }
__device__ __forceinline__ uint32_t *ch_state(unsigned char *L) { return (uint32_t *)(L + 512); }
__device__ __forceinline__ unsigned char *ch_rows(unsigned char *L) { return L + CH_ROWS; }

struct ChainWarp {
  // lane l holds the state of the tile that feeds the launch's step l
  int cnt;    // rows in it; the top 32 are in work
  int prog;   // > 0: the step is interrupted before candidate `prog` of each lane's group
  unsigned long long rows, cand;  // rows step l wrote, candidates it saw
  unsigned long long sum;         // checksum of the lane's embeddings
  unsigned long long last_rows, last_cand;  // the lane's embeddings and candidates, where ch_count took them
  unsigned spent;                 // candidates of this warp so far (uniform)
  float prune;                    // rows of a higher score are dropped (uniform)
  int part;                       // of the rows in the first tile, which share of the candidates is this
                                  // warp's: those at places = part modulo A.parts
};

// Whether one of the NV new ids (16 bits) of a candidate is among the row's ids it is compared with.
template <int NV, int NC>
__device__ __forceinline__ bool ch_hit(const uint32_t *nv, const uint32_t *cm, const uint2 *r) {
  uint32_t hit = 0;
#pragma unroll
  for (int i = 0; i < NV; i++) {
    const uint32_t vv = nv[i] * 0x10001u;
    uint32_t acc = ~0u;  // a zero half: some id equals
#pragma unroll
    for (int k = 0; k < NC; k++)
      if ((cm[i] >> k) & 1u) acc = __vimin3_u16x2(acc, r[k].x ^ vv, r[k].y ^ vv);
    hit |= (acc - 0x00010001u) & ~acc;
  }
  return (hit & 0x80008000u) != 0;
}

// Back-edges of a candidate that passed the overlap test; adds their errors to the score.
template <int MODE, int NV>
__device__ __forceinline__ bool ch_back_edges(const ChainArgs &A, const ChainStep &s, const unsigned char *row,
                                              const uint32_t *nv, float &sc) {
  bool ok = true;
  for (int b = 0; b < s.n_be && ok; b++) {
    const unsigned ca = s.be_a[b], cb = s.be_b[b];
    uint32_t va = 0, vb = 0;
    if (ca < 0x8000u) va = *(const uint16_t *)(row + ca);
    if (cb < 0x8000u) vb = *(const uint16_t *)(row + cb);
#pragma unroll
    for (int i = 0; i < NV; i++) {
      if (ca == 0x8000u + i) va = nv[i];
      if (cb == 0x8000u + i) vb = nv[i];
    }
    ok = ch_adjacent(A, va, vb);
    if (MODE == 0 && ok && A.scored && A.eerr) sc += ch_edge_weight(A, va, vb);
  }
  return ok;
}

// A row's chunks in registers, for a step whose new vertex 0 has colour class q: a are the chunks of
// that class and b those of the other one (TWO; chunk 2 k + class), or a are all chunks (!TWO).
template <int NC, bool TWO>
struct ChainRow {
  static constexpr int N = TWO ? NC / 2 : NC;
  uint2 a[N], b[TWO ? N : 1];
  __device__ __forceinline__ void load(const unsigned char *row, int q, int nc) {
    const uint2 none = make_uint2(~0u, ~0u);
#pragma unroll
    for (int k = 0; k < N; k++) {
      if (TWO) {
        const bool in = 2 * k < nc;
        a[k] = in ? *(const uint2 *)(row + 512 * q + 1024 * k) : none;
        b[k] = in ? *(const uint2 *)(row + 512 * (1 - q) + 1024 * k) : none;
      } else {
        a[k] = k < nc ? *(const uint2 *)(row + 512 * k) : none;
      }
    }
  }
  __device__ __forceinline__ void store(unsigned char *d, int q, int nc) const {
#pragma unroll
    for (int k = 0; k < N; k++) {
      if (TWO) {
        if (2 * k < nc) {
          *(uint2 *)(d + 512 * q + 1024 * k) = a[k];
          *(uint2 *)(d + 512 * (1 - q) + 1024 * k) = b[k];
        }
      } else if (k < nc) {
        *(uint2 *)(d + 512 * k) = a[k];
      }
    }
  }
  // Whether new ids pass the overlap test, each given twice in a word: v0 (and v1) against a, v2 against
  // b (a if `same`). The empty place 0xFFFF fails, and so does every id where in is 0.
  __device__ __forceinline__ uint32_t meets_a(uint32_t acc, uint32_t v) const {
#pragma unroll
    for (int k = 0; k < N; k++) acc = __vimin3_u16x2(acc, a[k].x ^ v, a[k].y ^ v);
    return acc;
  }
  __device__ __forceinline__ bool passes(uint32_t in, uint32_t v) const { return !zero_half(meets_a(~v & in, v)); }
  __device__ __forceinline__ bool passes(uint32_t in, uint32_t v0, uint32_t v1, uint32_t v2, bool same) const {
    uint32_t acc = meets_a(meets_a(~v0 & in, v0), v1);
    if (!TWO || same) {
      acc = meets_a(acc, v2);
    } else {
#pragma unroll
      for (int k = 0; k < N; k++) acc = __vimin3_u16x2(acc, b[k].x ^ v2, b[k].y ^ v2);
    }
    return !zero_half(acc);
  }
  static __device__ __forceinline__ bool zero_half(uint32_t x) { return ((x - 0x00010001u) & ~x & 0x80008000u) != 0; }
};

// Half i (0 or 1) of w, twice.
__device__ __forceinline__ uint32_t ch_twice(uint32_t w, int i) { return __byte_perm(w, 0, i ? 0x3232 : 0x1010); }

// 32 bytes of a group, read-only path.
__device__ __forceinline__ void ch_load4(const uint2 *p, uint2 (&x)[4]) {
  asm("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
      : "=r"(x[0].x), "=r"(x[0].y), "=r"(x[1].x), "=r"(x[1].y), "=r"(x[2].x), "=r"(x[2].y), "=r"(x[3].x), "=r"(x[3].y)
      : "l"(p));
}

// Checksum term of id v < 2^16 at the output position of a step of one new vertex: pos_term with the
// products of the position taken out (s.mul = (p << 32) * C1, s.pos2 = p << 2).
__device__ __forceinline__ unsigned long long ch_term(unsigned long long mul, uint32_t pos2, uint32_t v) {
  unsigned long long z = (unsigned long long)(v ^ pos2) * 0xBF58476D1CE4E5B9ull + mul;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// The candidates of a step of one new vertex (at most four ids), less those that are images of the key's
// pattern neighbours in the row: the data edges to them are among the key's, so each of them would be
// a candidate that fails (n_ex of them; the last place in use moves up). Returns the places in use, and
// in len how many candidates the group has.
__device__ __forceinline__ int ch_ids(const ChainStep &s, const unsigned char *row, uint2 x, uint32_t (&id)[4],
                                      unsigned &len) {
  id[0] = x.x & 0xFFFFu;
  id[1] = x.x >> 16;
  id[2] = x.y & 0xFFFFu;
  id[3] = x.y >> 16;
  len = (id[0] != 0xFFFFu) + (id[1] != 0xFFFFu) + (id[2] != 0xFFFFu) + (id[3] != 0xFFFFu);
  int n = s.group;
  const int n_ex = s.n_ex;
#pragma unroll 1
  for (int e = 0; e < n_ex; e++) {
    const uint32_t v = *(const uint16_t *)(row + s.ex_off[e]);
    n--;
    const uint32_t last = n == 3 ? id[3] : n == 2 ? id[2] : id[1];
#pragma unroll
    for (int u = 0; u < 3; u++)
      if (id[u] == v) id[u] = last;
  }
  return n;
}

// Count rows base .. base + t - 1 (t <= 32) of the last step's tile L: a step of one key, NN new
// vertices and no back-edges whose candidates lie in groups of one size.
template <int NN, int NC, bool TWO>
__device__ __forceinline__ void ch_count(const ChainArgs &A, const ChainStep &s, unsigned char *L, int base, int t,
                                         ChainWarp &w) {
  const int lane = threadIdx.x & 31;
  const uint32_t in = lane < t ? ~0u : 0u;
  const unsigned char *slot = L + 8 * (base + lane);
  const uint32_t key = *(const uint16_t *)(slot + CH_ROWS + s.key_off[0]) & in;
  const uint2 *ids = s.ids + key * (uint32_t)s.stride;
  uint2 x[4];
  if (NN == 1) x[0] = __ldg(ids);
  else ch_load4(ids, x);
  ChainRow<NC, TWO> r;
  r.load(slot + CH_ROWS, s.q, s.nc_in);
  const unsigned long long tail = *(const unsigned long long *)slot + (unsigned long long)(uint32_t)A.wo;
  unsigned rows = 0, cand = 0;
  if (NN == 1) {
    const unsigned long long mul = s.mul;
    const uint32_t pos2 = s.pos2;
    uint32_t id[4];
    const int n = ch_ids(s, slot + CH_ROWS, x[0], id, cand);
#pragma unroll
    for (int u = 0; u < 4; u++) {
      if (u >= n) break;  // uniform
      const bool ok = r.passes(in, id[u] * 0x10001u);
      const unsigned long long f = dmix64(tail + ch_term(mul, pos2, id[u]));
      if (ok) {
        w.sum += f;
        rows++;
      }
    }
    cand &= in;
  } else {
    const bool same = s.same;
    cand = (x[0].y >> 16) & in;
    const int longest = __reduce_max_sync(FULL_MASK, cand);
    const unsigned long long *sums = (const unsigned long long *)s.extra + key * (uint32_t)s.stride;
#pragma unroll 1
    for (int c = 0; c < longest; c += 4) {
#pragma unroll
      for (int u = 0; u < 4; u++) {
        if (c + u >= longest) break;  // uniform
        const bool ok = r.passes(in, ch_twice(x[u].x, 0), ch_twice(x[u].x, 1), ch_twice(x[u].y, 0), same);
        if (ok) {
          w.sum += dmix64(tail + __ldg(sums + c + u));
          rows++;
        }
      }
      if (c + 4 < longest) ch_load4(ids + c + 4, x);
    }
  }
  w.last_rows += rows;
  w.last_cand += cand;
}

// A candidate's part of the score. Of one new vertex: ids move about in a group (ch_ids), so its place
// is looked for.
template <int NN>
__device__ __forceinline__ float ch_part(const ChainStep &s, uint32_t first, int c, uint2 x, uint32_t id) {
  if (NN == 1) {
    c = (x.x & 0xFFFFu) == id ? 0 : x.x >> 16 == id ? 1 : (x.y & 0xFFFFu) == id ? 2 : 3;
  }
  return __ldg((const float *)s.extra + first + c);
}

// Join (or go on joining) the top rows of step j's tile, for a step of one key and NN new vertices
// whose candidates lie in groups of one size, empty places at a group's end marked. NC: chunks of a
// row, at most. Not for a counted step. Where the next step is the last of a count (CN: its new vertices,
// if ch_count takes it), every 32 survivors are counted on the spot: the two last steps of a plan see
// most of its rows, and to leave a tile and come back costs as much as a candidate of every lane.
template <int MODE, int NN, int NC, bool TWO, int CN>
__device__ __forceinline__ void ch_step_dense(const ChainArgs &A, unsigned char *W, ChainWarp &w, int j) {
  const ChainStep &s = A.st[j];
  const int lane = threadIdx.x & 31;
  unsigned char *L = W + (unsigned)s.in_off * 8u, *D = W + (unsigned)s.out_off * 8u;
  const int nc_out = s.nc_out, n_be = s.n_be, q = s.q;
  const int n = __shfl_sync(FULL_MASK, w.cnt, j), t = min(n, 32), base = n - t;
  int c = __shfl_sync(FULL_MASK, w.prog, j);
  const uint32_t in = lane < t ? ~0u : 0u;
  const unsigned char *slot = L + 8 * (base + lane);
  const uint32_t key = *(const uint16_t *)(slot + CH_ROWS + s.key_off[0]) & in;
  const uint2 *ids = s.ids + key * (uint32_t)s.stride;
  uint2 x[4];
  if (NN == 1) x[0] = __ldg(ids);
  else ch_load4(ids + (c & ~3), x);
  ChainRow<NC, TWO> r;
  r.load(slot + CH_ROWS, q, s.nc_in);
  const unsigned long long tail = *(const unsigned long long *)slot;
  unsigned to[NN];
#pragma unroll
  for (int i = 0; i < NN; i++) to[i] = s.new_off[i];
  int longest;
  unsigned len = 0;
  uint32_t id[4];
  if (NN == 3) {
    len = (x[0].y >> 16) & in;
    longest = __reduce_max_sync(FULL_MASK, len);
  } else {
    longest = ch_ids(s, slot + CH_ROWS, x[0], id, len);
    len &= in;
  }
  const bool then = CN && j + 1 == A.n_steps;
  // the places that are this warp's, modulo 4 (with a remainder for each candidate instead, a 24-vertex
  // path took 2.36 ms against 2.28)
  const unsigned own = j > 1 || A.parts == 1 ? 0xFu : (A.parts == 2 ? 0x5u : 0x1u) << w.part;
  const unsigned seen = c == 0 && (j > 1 || w.part == 0) ? __reduce_add_sync(FULL_MASK, len) : 0u;
  const int nch0 = __shfl_sync(FULL_MASK, w.cnt, j + 1);
  int nch = nch0;
  const unsigned long long mul = s.mul;
  const uint32_t pos2 = s.pos2, first = key * (uint32_t)s.stride * (NN == 1 ? 4u : 1u);  // place of the group in s.extra
  // the candidate at place c of every lane's group: its id in h0, or its three in h0 and h1
  auto one = [&](uint32_t h0, uint32_t h1, bool same) {
    bool ok = NN == 1 ? r.passes(in, h0 * 0x10001u)
                      : r.passes(in, ch_twice(h0, 0), ch_twice(h0, 1), ch_twice(h1, 0), same);
    const uint32_t id0 = NN == 1 ? h0 : h0 & 0xFFFFu;
    float sc = 0.f;
    if (MODE == 0 && A.scored && ok) sc = __uint_as_float((uint32_t)tail) + ch_part<NN>(s, first, c, x[0], id0);
    if (n_be && ok) {
      const uint32_t nv[3] = {id0, h0 >> 16, h1 & 0xFFFFu};
      ok = ch_back_edges<MODE, NN>(A, s, slot + CH_ROWS, nv, sc);
    }
    if (MODE == 0 && A.scored && sc > w.prune) ok = false;
    const unsigned bal = __ballot_sync(FULL_MASK, ok);
    if (ok) {
      unsigned char *d = D + 8 * (nch + __popc(bal & lanemask_lt()));
      unsigned long long out = (unsigned long long)__float_as_uint(sc);
      if (MODE == 1) out = tail + (NN == 1 ? ch_term(mul, pos2, id0) : __ldg((const unsigned long long *)s.extra + first + c));
      *(unsigned long long *)d = out;
      r.store(d + CH_ROWS, q, nc_out);
      if (to[0] != CH_DEAD) *(uint16_t *)(d + CH_ROWS + to[0]) = (uint16_t)id0;
      if (NN == 3) {
        if (to[NN / 2] != CH_DEAD) *(uint16_t *)(d + CH_ROWS + to[NN / 2]) = (uint16_t)(h0 >> 16);
        if (to[NN - 1] != CH_DEAD) *(uint16_t *)(d + CH_ROWS + to[NN - 1]) = (uint16_t)h1;
      }
    }
    nch += __popc(bal);
  };
  const bool same = s.same;
  unsigned counted = 0;
  while (true) {
    if (NN == 1) {
#pragma unroll
      for (int u = 0; u < 4; u++) {
        if (c > u) continue;                   // done before (uniform)
        if (u >= longest || nch >= 32) break;  // 32 rows in the next tile: that one first
        if (own >> u & 1u) one(id[u], 0u, true);
        c = u + 1;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 4; u++) {
        if ((c & 3) != u) continue;
        if (c >= longest || nch >= 32) break;
        if (own >> u & 1u) one(x[u].x, x[u].y, same);
        c++;
      }
      if ((c & 3) == 0 && c < longest) ch_load4(ids + c, x);
    }
    if (nch >= 32) {
      if (!CN || !then) break;
      nch -= 32;
      counted += 32;
      __syncwarp();
      ch_count<CN ? CN : 1, NC, TWO>(A, A.st[j + 1], D, nch, 32, w);
      __syncwarp();
    }
    if (c >= longest) break;
  }
  w.spent += seen;
  if (lane == j) {
    if (c >= longest) w.cnt = base;
    w.prog = c >= longest ? 0 : c;
    w.rows += (unsigned)(nch - nch0) + counted;
    w.cand += seen;
  }
  if (lane == j + 1) w.cnt = nch;
}

// The same for any other step: the group of a key (or two) is looked up, up to CH_NEW new vertices and
// further keys are read at run time. The state of an interrupted step is kept in shared memory.
template <int MODE, int NC>
__device__ __forceinline__ void ch_step(const ChainArgs &A, unsigned char *W, ChainWarp &w, int j) {
  const ChainStep &s = A.st[j];
  const int lane = threadIdx.x & 31;
  unsigned char *L = W + (unsigned)s.in_off * 8u, *D = W + (unsigned)s.out_off * 8u;
  const bool count = MODE == 1 && j == A.n_steps && A.out_kind == 0;
  const int nn = s.n_new, units = s.units, nc_in = s.nc_in, nc_out = s.nc_out;
  const int n = __shfl_sync(FULL_MASK, w.cnt, j), t = min(n, 32), base = n - t;
  int c = __shfl_sync(FULL_MASK, w.prog, j);
  const unsigned char *row = ch_rows(L) + 8 * (base + lane);
  int start = 0, len = 0;
  if (c == 0) {
    if (lane < t)
      ch_lookup(s, *(const uint16_t *)(row + s.key_off[0]), s.nkeys == 2 ? *(const uint16_t *)(row + s.key_off[1]) : 0u,
                start, len);
    const unsigned tot = __reduce_add_sync(FULL_MASK, (unsigned)len);
    ch_state(L)[lane] = (uint32_t)start | ((uint32_t)len << 24);
    w.spent += tot;
    if (lane == j && (j > 1 || w.part == 0)) w.cand += tot;
  } else {
    const uint32_t v = ch_state(L)[lane];
    start = (int)(v & 0xFFFFFFu);
    len = (int)(v >> 24);
  }
  const int maxlen = __reduce_max_sync(FULL_MASK, (unsigned)len);
  uint2 r[NC];
#pragma unroll
  for (int k = 0; k < NC; k++) r[k] = k < nc_in ? *(const uint2 *)(row + 512 * k) : make_uint2(~0u, ~0u);
  const unsigned long long tail = ch_tail(L)[base + lane];
  uint32_t cm[CH_NEW];
#pragma unroll
  for (int i = 0; i < CH_NEW; i++) cm[i] = i < nn ? s.cm[i] : 0u;
  const uint4 *rec = s.rec + (int64_t)start * units;
  int nch = count ? 0 : __shfl_sync(FULL_MASK, w.cnt, j + 1);
  unsigned K = 0;
  while (c < maxlen) {
    if (j == 1 && A.parts > 1 && c % A.parts != w.part) {  // another warp's share
      c++;
      continue;
    }
    bool ok = c < len;
    const uint4 x = ok ? __ldg(rec + c * units) : make_uint4(0, 0, 0, 0);
    uint4 y = make_uint4(x.z, x.w, 0, 0);
    if (units == 2) y = ok ? __ldg(rec + c * units + 1) : make_uint4(0, 0, 0, 0);
    const unsigned long long add = y.x | ((unsigned long long)y.y << 32);
    uint32_t nv[CH_NEW];
    {
      const uint32_t h[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int i = 0; i < CH_NEW; i++) nv[i] = (h[i >> 1] >> (16 * (i & 1))) & 0xFFFFu;
    }
    for (int e = 0; e < s.n_chk; e++) {  // further keys: behind the new ids
      uint32_t v = 0;
#pragma unroll
      for (int i = 0; i < CH_NEW; i++)
        if (i == nn + e) v = nv[i];
      ok &= *(const uint16_t *)(row + s.chk_off[e]) == v;
    }
    ok = ok && !ch_hit<CH_NEW, NC>(nv, cm, r);
    float sc = 0.f;
    if (MODE == 0) sc = __uint_as_float((uint32_t)tail) + __uint_as_float((uint32_t)add);
    if (s.n_be && ok) ok = ch_back_edges<MODE, CH_NEW>(A, s, row, nv, sc);
    if (MODE == 0 && A.scored && sc > w.prune) ok = false;
    const unsigned bal = __ballot_sync(FULL_MASK, ok);
    c++;
    if (bal == 0) continue;
    const int k_ok = __popc(bal);
    K += k_ok;
    if (count) {
      if (ok) w.sum += dmix64(tail + add + (unsigned long long)(uint32_t)A.wo);
      continue;
    }
    if (ok) {
      const int pos = nch + __popc(bal & lanemask_lt());
      unsigned char *d = ch_rows(D) + 8 * pos;
      ch_tail(D)[pos] = MODE == 1 ? tail + add : (unsigned long long)__float_as_uint(sc);
#pragma unroll
      for (int k = 0; k < NC; k++)
        if (k < nc_out) *(uint2 *)(d + 512 * k) = r[k];
#pragma unroll
      for (int i = 0; i < CH_NEW; i++)
        if (i < nn && s.new_off[i] != CH_DEAD) *(uint16_t *)(d + s.new_off[i]) = (uint16_t)nv[i];
    }
    nch += k_ok;
    if (nch >= 32) break;  // the next tile first
  }
  const bool done = c >= maxlen;
  if (lane == j) {
    if (done) w.cnt = base;
    w.prog = done ? 0 : c;
    w.rows += K;
  }
  if (!count && lane == j + 1) w.cnt = nch;
}

// Rows [lo, lo + nr) of the first motif table into the first tile.
template <int MODE>
__device__ __forceinline__ void ch_seed(const ChainArgs &A, unsigned char *W, ChainWarp &w, int64_t lo, int nr) {
  const int lane = threadIdx.x & 31;
  bool ok = lane < nr;
  const int32_t *trow = A.seed_rows + (lo + (ok ? lane : 0)) * A.seed_mw;
  if (A.n_shards > 1) ok = ok && (uint32_t)__ldg(trow) % (uint32_t)A.n_shards == (uint32_t)A.shard;
  float sc = 0.f;
  if (MODE == 0 && A.scored && ok) {
    if (A.seed_score) sc += __ldg(A.seed_score + lo + lane);
    if (A.qerr)
      for (int i = 0; i < A.seed_k; i++) sc += __ldg(A.qerr + __ldg(trow + i));
  }
  for (int b = 0; b < A.seed_nbe; b++) {
    if (ok) {
      const int32_t va = __ldg(trow + A.seed_be[b][0]), vb = __ldg(trow + A.seed_be[b][1]);
      ok = ch_adjacent(A, va, vb);
      if (MODE == 0 && ok && A.scored && A.eerr) sc += ch_edge_weight(A, va, vb);
    }
  }
  if (MODE == 0 && A.scored && sc > w.prune) ok = false;
  const unsigned bal = __ballot_sync(FULL_MASK, ok);
  const int n = __shfl_sync(FULL_MASK, w.cnt, 1);
  unsigned char *D = W + (unsigned)A.st[1].in_off * 8u;
  if (ok) {
    const int pos = n + __popc(bal & lanemask_lt());
    unsigned char *d = ch_rows(D) + 8 * pos;
    for (int k = 0; k < A.st[1].nc_in; k++) *(uint2 *)(d + 512 * k) = make_uint2(~0u, ~0u);
    unsigned long long p = 0;
    for (int i = 0; i < A.seed_k; i++) {
      const int32_t v = __ldg(trow + i);
      if (MODE == 1) p += pos_term(A.seed_npos[i], v);
      if (A.seed_off[i] != CH_DEAD) *(uint16_t *)(d + A.seed_off[i]) = (uint16_t)v;
    }
    ch_tail(D)[pos] = MODE == 1 ? p : (unsigned long long)__float_as_uint(sc);
  }
  if (lane == 1) w.cnt = n + __popc(bal);
  if (lane == 0 && w.part == 0) {
    w.rows += __popc(bal);
    w.cand += nr;
  }
}

// The rows of block b of the input table whose number is part modulo parts (a power of two) into the
// first tile.
__device__ __forceinline__ void ch_fetch(const ChainArgs &A, unsigned char *W, ChainWarp &w, int64_t b, int part,
                                         int parts) {
  const int lane = threadIdx.x & 31, nc = A.st[1].nc_in;
  const int nr = (__ldg(A.in_rows + b) - part + parts - 1) >> (__ffs(parts) - 1), n = __shfl_sync(FULL_MASK, w.cnt, 1);
  const uint2 *src = (const uint2 *)(A.in + b * (nc + 1) * 256) + part + parts * lane;
  unsigned char *D = W + (unsigned)A.st[1].in_off * 8u;
  if (lane < nr) {
    unsigned char *d = ch_rows(D) + 8 * (n + lane);
    *(uint2 *)(ch_tail(D) + n + lane) = __ldg(src);
    for (int k = 0; k < nc; k++) *(uint2 *)(d + 512 * k) = __ldg(src + 32 * (k + 1));
  }
  if (lane == 1) w.cnt = n + nr;
}

// The top rows of the output tile (at most 32) as one block of the table the next launch reads.
// False when the table is full: the caller's result is void then, and the warp ends.
__device__ __forceinline__ bool ch_put(const ChainArgs &A, unsigned char *W, ChainWarp &w) {
  const int lane = threadIdx.x & 31, nc = A.st[A.n_steps].nc_out, l = A.n_steps + 1;
  unsigned char *L = W + (unsigned)A.st[A.n_steps].out_off * 8u;
  const int cnt = __shfl_sync(FULL_MASK, w.cnt, l), n = min(cnt, 32), base = cnt - n;
  long long b = 0;
  if (lane == 0) b = (long long)atomicAdd(A.ctr_last + CTR_BLOCKS, 1ull);
  b = __shfl_sync(FULL_MASK, b, 0);
  if (lane == l) w.cnt = base;
  if (b >= A.out_cap) {
    if (lane == 0) atomicOr(A.ctr_last + CTR_OVF, 1ull);
    return false;
  }
  if (lane == 0) A.out_rows[b] = n;
  uint2 *dst = (uint2 *)((unsigned char *)A.out + b * (nc + 1) * 256) + lane;
  if (lane < n) {
    const unsigned char *row = ch_rows(L) + 8 * (base + lane);
    dst[0] = *(const uint2 *)(ch_tail(L) + base + lane);
    for (int k = 0; k < nc; k++) dst[32 * (k + 1)] = *(const uint2 *)(row + 512 * k);
  }
  return true;
}

// Lower the bound of a top-k run: the upper end of the bin that holds the k-th best of the rows written
// so far by anyone. Rows above it, and partial rows above it where no weight is negative, cannot be
// among the k best.
__device__ __forceinline__ void ch_bound(const ChainArgs &A, ChainWarp &w) {
  constexpr int PER = SelHist::COARSE / 32;
  const int lane = threadIdx.x & 31;
  unsigned c[PER], sum = 0;
#pragma unroll
  for (int i = 0; i < PER; i++) sum += c[i] = *(volatile unsigned *)&A.sel->coarse[lane * PER + i];
  unsigned incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(FULL_MASK, incl, o);
    if (lane >= o) incl += v;
  }
  const unsigned k = (unsigned)A.sel_k;
  if (__shfl_sync(FULL_MASK, incl, 31) < k) return;
  // the first lane that reaches k, its bin, and how many of that bin are needed
  const int at = __ffs(__ballot_sync(FULL_MASK, incl >= k)) - 1;
  unsigned before = incl - sum;
  int bin = lane * PER;
  for (int i = 0; i + 1 < PER && before + c[i] < k; i++) {
    before += c[i];
    bin++;
  }
  before = __shfl_sync(FULL_MASK, before, at);
  bin = __shfl_sync(FULL_MASK, bin, at);
  constexpr int SUB = SelHist::FINE / SelHist::COARSE;  // 32
  incl = *(volatile unsigned *)&A.sel->fine[bin * SUB + lane];
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(FULL_MASK, incl, o);
    if (lane >= o) incl += v;
  }
  const unsigned hit = __ballot_sync(FULL_MASK, before + incl >= k);
  if (!hit) return;  // the counts moved on between the two reads
  const uint32_t top = ((uint32_t)(bin * SUB + __ffs(hit) - 1) << SelHist::FINE_SHIFT) | ((1u << SelHist::FINE_SHIFT) - 1);
  // scores are not negative where this runs, so their bits order like their keys
  const int bits = (int)(top & 0x7FFFFFFFu);
  if (lane == 0) atomicMin(&A.sel->bound, bits);
  w.prune = fminf(w.prune, __int_as_float(bits));
}

// All rows of the output tile to the packed result in pattern-vertex order. False when they do
// not fit, as above.
__device__ __forceinline__ bool ch_flush(const ChainArgs &A, unsigned char *W, ChainWarp &w, const uint16_t *ooff) {
  const int lane = threadIdx.x & 31, l = A.n_steps + 1, wo = A.wo;
  unsigned char *L = W + (unsigned)A.st[A.n_steps].out_off * 8u;
  const int n = __shfl_sync(FULL_MASK, w.cnt, l);
  long long at = 0;
  if (lane == 0) at = (long long)atomicAdd(A.ctr_last + CTR_ROWS, (unsigned long long)n);
  at = __shfl_sync(FULL_MASK, at, 0);
  if (lane == l) w.cnt = 0;
  if (at + n > A.out_cap) {
    if (lane == 0) atomicOr(A.ctr_last + CTR_OVF, 1ull);
    return false;
  }
  if (A.scored)
    for (int i0 = 0; i0 < n; i0 += 32) {
      const int i = i0 + lane;
      const float sc = i < n ? __uint_as_float((uint32_t)ch_tail(L)[i]) : 0.f;
      if (i < n) A.outs[at + i] = sc;
      if (A.sel) {  // scores crowd in a few bins: one addition a bin and warp
        const uint32_t key = i < n ? score_key(sc) : ~0u;
        const unsigned f = __match_any_sync(FULL_MASK, key >> SelHist::FINE_SHIFT);
        const unsigned c = __match_any_sync(FULL_MASK, key >> SelHist::COARSE_SHIFT);
        if (i < n) {
          if ((f & lanemask_lt()) == 0) atomicAdd(&A.sel->fine[key >> SelHist::FINE_SHIFT], (unsigned)__popc(f));
          if ((c & lanemask_lt()) == 0) atomicAdd(&A.sel->coarse[key >> SelHist::COARSE_SHIFT], (unsigned)__popc(c));
        }
      }
    }
  if (A.sel) ch_bound(A, w);
  int32_t *out = A.out + at * wo;
  const unsigned char *rows = ch_rows(L);
  int r = lane / wo, q = lane - r * wo;
  const int dr = 32 / wo, dq = 32 % wo;
  for (int e = lane; e < n * wo; e += 32) {
    out[e] = *(const uint16_t *)(rows + 8 * r + ooff[q]);
    r += dr;
    q += dq;
    if (q >= wo) {
      q -= wo;
      r++;
    }
  }
  return true;
}

template <int MODE, bool TWO, int NC, int CN>
__global__ void __launch_bounds__(CH_BLK, 4) k_chain(const __grid_constant__ ChainArgs A) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long red[2 * 32 + 1];
  __shared__ uint16_t ooff[MAXW];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned char *W = smem + (size_t)wid * A.warp_bytes;
  for (int i = threadIdx.x; i < 65; i += CH_BLK) red[i] = 0;
  if (MODE == 0 && A.out_kind == 1)
    for (int q = threadIdx.x; q < A.wo; q += CH_BLK) ooff[q] = A.out_off[q];
  __syncthreads();
  griddep_wait();  // the candidate tables, the counters and the input table come from the launches before
  griddep_launch_dependents();
  ChainWarp w{};
  w.prune = A.prune;
  float best = A.prune;  // the bound as it was asked for last
  const int64_t nw = (int64_t)gridDim.x * CH_WARPS;
  const int64_t n_in = A.in ? imin64((int64_t)*A.in_blocks, A.in_cap) - A.lo : (A.seed_n - A.lo + A.chunk - 1) / A.chunk;
  // a table of few blocks is dealt out in shares of a block: every warp of the launch before leaves a
  // partly filled one, so a share is every second or fourth row. 23-vertex path on heavy-hex 9x11: 169 us
  // in quarters of 8 rows, 111 in twos, 104 in fours; 27-vertex patch on 17x19: 225, 210, 226, by this
  // line 209
  const int parts = !A.in || n_in >= 8 * nw ? 1 : n_in < 4 * nw ? 4 : 2;
  const int64_t n_items = n_in * parts * A.parts;
  // items 0 .. nw - 1 are the warps' first; the counter deals out the rest. The next item's number
  // is asked for before the present one is joined.
  long long nxt = (int64_t)blockIdx.x * CH_WARPS + wid;
  bool more = true;
  while (true) {
    __syncwarp();
    if (MODE == 0 && A.sel) {  // used from the next turn on: nothing waits for it
      w.prune = fminf(w.prune, best);
      best = __int_as_float(*(volatile int *)&A.sel->bound);
    }
    const unsigned act = __ballot_sync(FULL_MASK, w.cnt >= 32 || w.prog > 0);
    int j;
    if (act) {
      j = 31 - __clz(act);
    } else if (A.parts > 1 && __shfl_sync(FULL_MASK, w.cnt, 1) > 0) {
      j = 1;  // the first tile holds one share only
    } else {
      if (more) {
        const long long it = __shfl_sync(FULL_MASK, nxt, 0);
        more = it < n_items;
        if (more) {
          if (n_items <= nw || (w.spent > A.limit && parts == 1)) nxt = n_items;  // one each; or the rest is left to another launch
          else if (lane == 0) nxt = nw + (long long)atomicAdd(A.ctr_last + CTR_ITEM, 1ull);
          if (A.in) {
            ch_fetch(A, W, w, A.lo + it / parts, (int)(it % parts), parts);
          } else {
            w.part = (int)(it % A.parts);
            const int64_t lo = A.lo + it / A.parts * A.chunk;
            ch_seed<MODE>(A, W, w, lo, (int)imin64(A.chunk, A.seed_n - lo));
          }
        }
        continue;
      }
      const unsigned ne = __ballot_sync(FULL_MASK, w.cnt > 0);
      if (!ne) break;
      j = __ffs(ne) - 1;
    }
    if (j > A.n_steps) {
      if (!(MODE == 0 && A.out_kind == 1 ? ch_flush(A, W, w, ooff) : ch_put(A, W, w))) break;
      continue;
    }
    const ChainStep &s = A.st[j];
    if (CN && j == A.n_steps) {
      const int n = __shfl_sync(FULL_MASK, w.cnt, j), t = min(n, 32);
      ch_count<CN ? CN : 1, NC, TWO>(A, s, W + (unsigned)s.in_off * 8u, n - t, t, w);
      if (lane == j) w.cnt = n - t;
    } else if (s.group && s.n_new == 1) {
      ch_step_dense<MODE, 1, NC, TWO, CN>(A, W, w, j);
    } else if (s.group) {
      ch_step_dense<MODE, 3, NC, TWO, CN>(A, W, w, j);
    } else {
      ch_step<MODE, NC>(A, W, w, j);
    }
  }
  // totals: step l of the launch is step first + l of the plan
  if (MODE == 0 && A.out_kind == 1 && lane == A.n_steps) w.rows = 0;  // counted as they were written
  if (lane <= A.n_steps) {
    if (w.rows) atomicAdd(&red[2 * lane], w.rows);
    if (w.cand) atomicAdd(&red[2 * lane + 1], w.cand);
  }
  if (MODE == 1 && A.out_kind == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      w.sum += __shfl_down_sync(FULL_MASK, w.sum, o);
      w.last_rows += __shfl_down_sync(FULL_MASK, w.last_rows, o);
      w.last_cand += __shfl_down_sync(FULL_MASK, w.last_cand, o);
    }
    if (lane == 0) {
      atomicAdd(&red[64], w.sum);
      atomicAdd(&red[2 * A.n_steps], w.last_rows);
      atomicAdd(&red[2 * A.n_steps + 1], w.last_cand);
    }
  }
  __syncthreads();
  unsigned long long *ctr = A.ctr_last - (int64_t)A.n_steps * CTR_N;
  for (int i = threadIdx.x; i < 2 * (A.n_steps + 1); i += CH_BLK)
    if (red[i]) atomicAdd(ctr + (int64_t)(i >> 1) * CTR_N + ((i & 1) ? CTR_CAND : CTR_ROWS), red[i]);
  if (MODE == 1 && A.out_kind == 0 && threadIdx.x == 0) atomicAdd(A.ctr_last + CTR_SUM, red[64]);
  if (A.h_out) {  // the last block hands the totals over: a copy behind the launch costs 4 us
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(A.done, 1ull) == gridDim.x - 1;
    __syncthreads();
    if (last) {
      __threadfence();
      const unsigned long long *c0 = A.done - (A.n_out - CTR_N);
      for (int i = threadIdx.x; i < A.n_out; i += CH_BLK) A.h_out[i] = __ldcg(c0 + i);
    }
  }
}

typedef void (*ChainKernel)(ChainArgs);

// Chunks of a row: as many as the launch's widest tile has.
constexpr int CH_NC[3] = {2, 4, CH_CHUNKS};
// [row mode, count with a last step for ch_count of 1 or 3 new vertices, with any other][classes]
template <int I>
static void chain_kernels(ChainKernel (*k)[2]) {
  k[0][0] = k_chain<0, false, CH_NC[I], 0>;
  k[0][1] = k_chain<0, true, CH_NC[I], 0>;
  k[1][0] = k_chain<1, false, CH_NC[I], 1>;
  k[1][1] = k_chain<1, true, CH_NC[I], 1>;
  k[2][0] = k_chain<1, false, CH_NC[I], 3>;
  k[2][1] = k_chain<1, true, CH_NC[I], 3>;
  k[3][0] = k_chain<1, false, CH_NC[I], 0>;
  k[3][1] = k_chain<1, true, CH_NC[I], 0>;
}
struct ChainKernels {
  ChainKernel k[3][4][2];
  ChainKernels() {
    chain_kernels<0>(k[0]);
    chain_kernels<1>(k[1]);
    chain_kernels<2>(k[2]);
  }
};

static const ChainKernels &all_chain_kernels() {
  static const ChainKernels ks;
  return ks;
}

static ChainKernel pick_chain(const ChainArgs &a) {
  int nc = 0;
  for (int j = 1; j <= a.n_steps; j++) nc = a.st[j].nc_in > nc ? a.st[j].nc_in : nc;
  nc = a.st[a.n_steps].nc_out > nc ? a.st[a.n_steps].nc_out : nc;
  const int kind = a.mode == 0 ? 0 : a.count_new == 1 ? 1 : a.count_new == 3 ? 2 : 3;
  return all_chain_kernels().k[nc <= CH_NC[0] ? 0 : nc <= CH_NC[1] ? 1 : 2][kind][a.two != 0];
}

static cudaError_t chain_attrs() {
  static std::atomic<unsigned long long> done{0};  // one bit per device ordinal below 64
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
  if (bit && (done.load() & bit)) return cudaSuccess;
  for (auto &kind : all_chain_kernels().k)
    for (auto &row : kind)
      for (ChainKernel k : row) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, CH_SMEM_MAX);
        if (e != cudaSuccess) return e;
      }
  if (bit) done.fetch_or(bit);
  return cudaSuccess;
}

int chain_grid(const ChainArgs &a, int num_sms) {
  int per_sm = 0;
  chain_attrs();
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pick_chain(a), CH_BLK, (size_t)CH_WARPS * a.warp_bytes);
  return num_sms * (per_sm < 1 ? 1 : per_sm);
}

cudaError_t launch_chain(const ChainArgs &a, int grid, cudaStream_t s) {
  const cudaError_t e = chain_attrs();
  if (e != cudaSuccess) return e;
  g_launches++;
  return launch_pdl(pick_chain(a), dim3(grid), dim3(CH_BLK), (size_t)CH_WARPS * a.warp_bytes, s, a);
}

cudaError_t launch_chain_tables(const ChainTables &r, cudaStream_t s) {
  g_launches++;
  const int64_t n = r.total > r.n_ctr ? r.total : r.n_ctr;
  k_chain_tables<<<(int)imin64((n + 255) / 256, 2048), 256, 0, s>>>(r);
  return cudaGetLastError();
}

}  // namespace dmk
