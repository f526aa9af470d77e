// Launchers of the library's sm_103a kernels (kernels.cu). All take the stream to run on;
// none synchronises. Sizes are in elements unless the name says bytes.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "dm_internal.h"

namespace dmk {

// Launch with programmatic dependent launch: the kernel may be scheduled while the previous
// kernel in the stream is finishing; it must execute griddep_wait() (join_device.cuh) before
// touching global memory that the previous kernel reads or writes. Used only where the
// previous stream operation is itself a kernel of the same chain.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Number of kernels this library has launched from the calling thread so far (a context's
// calls run on the calling thread, so per-call differences stay exact when several threads
// drive their own contexts at once).
int64_t launch_count();
extern thread_local int64_t g_launches;

// Fused join step of Alg. 1 (InnerJoin + FilterOverlappingNodes + back-edge filter + score
// + compaction, or count + checksum in the last step), warp-centric (join_warp.cu). The grid
// fills the GPU at the kernel's occupancy, or covers the rows of R when they are fewer.
// pdl: launched with programmatic dependent launch (the previous stream operation must be a
// kernel of the same chain).
cudaError_t launch_wjoin(const dmi::JoinArgs &a, int grid, cudaStream_t s, bool pdl = false);
// One full wave for a launch that reads its input row count on the device (n_dev), else the
// blocks its rows need, at most one wave.
int wjoin_grid(const dmi::JoinArgs &a, int num_sms);
// The last two steps of a counted plan in one kernel (join_warp.cu): a = the second-to-last
// step (writes, identity column order), b = the last (counted); b's rows are a's survivors,
// which never reach global memory (b.R is ignored). Counts go to a.ctr (a's survivors and
// candidates) and b.ctr (the count, checksum and b's candidates). fused_ok tells whether the
// pair qualifies (1 to 4 new vertices each, no scores, no shards, shared memory fits).
bool fused_ok(const dmi::JoinArgs &a, const dmi::JoinArgs &b);
cudaError_t launch_fused(const dmi::JoinArgs &a, const dmi::JoinArgs &b, int num_sms, cudaStream_t s, bool pdl);

// Scores of a table's rows by the leading bits of their order-preserving keys (select.cu), and the bound
// that a top-k run of the joins lowers as it goes (bits of a non-negative score).
struct SelHist {
  static constexpr int FINE = 8192, FINE_SHIFT = 32 - 13, COARSE = 256, COARSE_SHIFT = 32 - 8;
  uint32_t fine[FINE], coarse[COARSE];
  int32_t bound;
};

// Several steps of a plan, often all of them, in one launch (chain.cu).
constexpr int CH_STEPS = 24;          // steps of a launch besides the seed, at most
constexpr int CH_NEW = 8;             // new vertices and further keys of a step, at most
constexpr int CH_CHUNKS = 8;          // chunks of four ids in a row, at most
constexpr uint16_t CH_DEAD = 0xFFFF;  // a new vertex that no later step reads
constexpr int CH_SMEM_MAX = 220 * 1024;
constexpr int CH_CTA_WARPS = 4;
constexpr int CH_MAX_GROUP = 255;     // longest key group, and rows of a motif table: what the
constexpr int64_t CH_MAX_ROWS = (1 << 24) - 1;  // state of an interrupted step holds
// A warp's tile of 64 rows of nc chunks: checksum sums or scores, state of an interrupted step, rows.
constexpr int chain_tile_bytes(int nc) { return 64 * 8 + 32 * 4 + nc * 512; }
struct ChainStep {
  // steps of grouped candidates (one key, 1 or 3 new vertices; group > 0: candidates of a key, at
  // most): the ids, `stride` words of 8 bytes a key, and what else a candidate brings (three new
  // vertices: sum of the checksum terms; scored rows: part of the score)
  const uint2 *ids;
  const void *extra;
  unsigned long long mul;        // one new vertex: its checksum term's constants (ch_term)
  uint32_t pos2;
  int32_t group, stride;
  uint8_t n_ex;                  // one new vertex: columns that are the key's pattern neighbours
  uint16_t ex_off[2];
  uint8_t q, same;               // colour class of new vertices 0 and 1, and whether 2 is of it too
  // any other step: one record a motif row in index order
  uint8_t units;
  uint8_t nkeys, n_new, n_chk, n_be, nc_in, nc_out;
  uint8_t cm[CH_NEW];            // chunks new vertex i is compared with
  const uint4 *rec;
  const int32_t *offsets;        // nkeys == 1
  const dmi::HashSlot *slots;    // nkeys == 2
  uint32_t log2cap;
  uint16_t in_off, out_off;      // its tile and the next one, in 8-byte words of the warp's memory
  uint16_t key_off[2], chk_off[4], new_off[CH_NEW];  // byte offsets from a row's first chunk
  uint16_t be_a[8], be_b[8];     // byte offset, or 0x8000 + index of the new vertex
};
struct ChainArgs {
  ChainStep st[CH_STEPS + 1];    // 1 .. n_steps; st[0] is the seed or the input table
  int32_t n_steps, mode, wo, warp_bytes;
  int32_t two;                   // two colour classes: chunk 2 k + class
  int32_t count_new;             // 1 or 3: new vertices of a counted last step that ch_count takes, else 0
  int32_t out_kind;              // 0: count and checksum, 1: packed rows, 2: table for another launch
  const unsigned long long *adj;
  int32_t adj_words;
  const int32_t *row_ptr, *col_idx;
  const float *eerr, *qerr;
  int32_t scored;
  float prune;
  const int32_t *seed_rows;
  const float *seed_score;
  int32_t seed_mw, seed_k, seed_nbe, shard, n_shards;
  // chunk <= 32 rows of the first table are one work item, or with parts > 1 as many: every warp then
  // takes one share of their first step's candidates
  int64_t seed_n, chunk;
  int32_t parts;
  int64_t lo;                    // input already joined by earlier launches: rows of the first table, or blocks
  uint8_t seed_npos[dmi::MAXM], seed_be[8][2];
  uint16_t seed_off[dmi::MAXM];
  const unsigned char *in;       // instead of the seed: blocks of up to 32 rows, in_rows[b] rows in block b
  const int32_t *in_rows;
  const unsigned long long *in_blocks;
  int64_t in_cap;
  unsigned limit;                // candidates after which a warp takes no further items (first launch only)
  unsigned long long *ctr_last;  // CTR_N counters of the launch's last step, behind those of its others
  unsigned long long *h_out;     // where set (pinned host memory), the last block writes the n_out
  unsigned long long *done;      // counters there whose last CTR_N begin at done (one of them, zero
  int32_t n_out;                 // before the launch, tells which block is the last)
  int32_t *out;                  // packed rows in pattern-vertex order, or blocks
  float *outs;
  int32_t *out_rows;
  int64_t out_cap;               // rows, or blocks
  SelHist *sel;                  // rows are wanted for their k best only: counted here, pruned by its bound
  int32_t sel_k;
  uint16_t out_off[dmi::MAXW];   // output position -> byte offset in the last tile's rows
};
int chain_grid(const ChainArgs &a, int num_sms);  // blocks of a full launch
cudaError_t launch_chain(const ChainArgs &a, int grid, cudaStream_t s);
// What the candidates of a plan's steps bring, and n_ctr zeroed counters. Kinds of tables: records (per
// motif row, `units` of 16 bytes), and per place of a grouped step an id, three ids and the group's
// length, the sum of checksum terms, the part of the score.
enum { CH_TAB_REC = 0, CH_TAB_ID = 1, CH_TAB_ID3 = 2, CH_TAB_SUM = 3, CH_TAB_SCORE = 4 };
constexpr int CH_TABS = 96;
struct ChainTables {
  struct Tab {
    const int32_t *rows;
    const float *score;
    const int32_t *offsets;
    void *out;
    int64_t end;                 // entries of the tables up to this one
    int32_t kind, group, mw, n_new, units;
    uint8_t mpos[CH_NEW], npos[CH_NEW];  // npos: 1 + output position (0: a further key, not a new vertex)
  } tab[CH_TABS];
  int64_t total, n_ctr;
  unsigned long long *ctr;
  const float *qerr;
  int32_t mode;
};
cudaError_t launch_chain_tables(const ChainTables &r, cudaStream_t s);

// Data-graph preparation.
cudaError_t launch_csr_to_m2(const int32_t *row_ptr, const int32_t *col_idx, const float *eerr,
                             int32_t V, int64_t nnz, int32_t *rows, float *score, cudaStream_t s);
// *girth = min(*girth, a lower bound of the graph's girth); the caller sets it to GIRTH_MAX or more before.
// adj4 (nullable): the neighbours of every vertex, ascending, 16 bits each, 0xFFFF past its degree (at most
// 4; V <= 65 534).
constexpr int GIRTH_MAX = 32;
cudaError_t launch_girth(const int32_t *row_ptr, const int32_t *col_idx, int32_t V, int32_t *girth, uint2 *adj4,
                         cudaStream_t s);
cudaError_t launch_vertex_table(int32_t V, int32_t *rows, float *score, cudaStream_t s);
cudaError_t launch_bitmap(const int32_t *row_ptr, const int32_t *col_idx, int32_t V, int64_t nnz,
                          int32_t words, unsigned long long *adj, cudaStream_t s);

// Exclusive scan of n values into out[0..n], out[n] = total. tmp must hold
// scan_tmp_elems(n) int64 values: per level of the scan over tile sums, the sums and their scan.
constexpr int SCAN_BLK = 256, SCAN_ITEMS = 8, SCAN_TILE = 2048;
constexpr int64_t scan_tmp_elems(int64_t n) {
  return (n + SCAN_TILE - 1) / SCAN_TILE <= 1
             ? 1
             : 2 * ((n + SCAN_TILE - 1) / SCAN_TILE) + 1 + scan_tmp_elems((n + SCAN_TILE - 1) / SCAN_TILE);
}
cudaError_t scan_i64(const int64_t *in, int64_t *out, int64_t n, int64_t *tmp, cudaStream_t s);
cudaError_t scan_i32(const int32_t *in, int64_t *out, int64_t n, int64_t *tmp, cudaStream_t s);

// One stable LSD pass: perm_out = perm_in stably sorted by the 8-bit digit
// (key >> shift) & 255 of key = keys[perm_in[i] * stride]. hist must hold
// radix_hist_elems(n) int64, tmp scan_tmp_elems(radix_hist_elems(n)).
constexpr int RS_BLK = 256, RS_ITEMS = 8, RS_TILE = 2048;
constexpr int64_t radix_hist_elems(int64_t n) { return 256 * ((n + RS_TILE - 1) / RS_TILE); }
cudaError_t radix_pass(const uint32_t *keys, int64_t stride, const int32_t *perm_in,
                       int32_t *perm_out, int64_t n, int shift, int64_t *hist, int64_t *hist_scan,
                       int64_t *tmp, cudaStream_t s);
cudaError_t launch_iota(int32_t *p, int64_t n, cudaStream_t s);
// In place: w[i] = -log(1 - w[i]) (error rate -> negative log fidelity).
cudaError_t launch_neg_log1m(float *w, int64_t n, cudaStream_t s);
// Packed join keys of a table's rows: (row[kp0] << 32) | row[kp1], or row[kp0] when kp1 < 0.
cudaError_t launch_join_keys(const int32_t *rows, int32_t w, int32_t kp0, int32_t kp1, int64_t n,
                             unsigned long long *keys, cudaStream_t s);
// Streaming chunk boundaries over a prefix array pre[0..n] (non-decreasing): bounds[t] is the
// largest i with pre[i] <= t * step for 0 < t < nch, bounds[0] = 0, bounds[nch] = n; bpre[t] =
// pre[bounds[t]]. Both outputs hold nch + 1 entries.
cudaError_t launch_chunk_bounds(const int64_t *pre, int64_t n, int64_t step, int64_t nch, int64_t *bounds,
                                int64_t *bpre, cudaStream_t s);
cudaError_t launch_gather_rows(const int32_t *in, const float *ins, const int32_t *perm, int64_t n,
                               int32_t w, int32_t *out, float *outs, cudaStream_t s);

// Motif-table indices.
cudaError_t launch_offsets_direct(const int32_t *rows, int32_t mw, int32_t kpos, int64_t n,
                                  int32_t V, int32_t *offsets, cudaStream_t s);
cudaError_t launch_hash_build(const int32_t *rows, int32_t mw, int32_t kp0, int32_t kp1, int64_t n,
                              dmi::HashSlot *slots, uint32_t log2cap, unsigned long long *ctr,
                              cudaStream_t s);

// Top-k support: histogram of the 8-bit digit at `shift` of the scores' order-preserving keys, over the
// scores whose keys agree with `prefix` on `pmask`; and compaction of indices with key <= T.
cudaError_t launch_score_hist(const float *sc, int64_t n, uint32_t prefix, uint32_t pmask, int shift,
                              unsigned long long *hist, cudaStream_t s);
cudaError_t launch_select_le(const float *sc, int64_t n, uint32_t T, int32_t *out_idx,
                             unsigned long long *ctr, cudaStream_t s);
// Direction-aware scores (Sec. 5.4 footnote): out[i] = sum_e sw[e] * edir[slot of
// rows[i][sp[e]] -> rows[i][sq[e]]] (+ sum_u qerr[rows[i][u]] when qerr is set), FP32.
cudaError_t launch_rescore_directed(const int32_t *rows, int64_t n, int32_t np, const int32_t *sp, const int32_t *sq,
                                    const float *sw, int32_t nslots, const int32_t *row_ptr, const int32_t *col_idx,
                                    const float *edir, const float *qerr, float *out, cudaStream_t s);
// keys[i] = order-preserving unsigned key of sc[i] (the bits of both functions above are
// these keys, not the raw FP32 bits).
cudaError_t launch_score_keys(const float *sc, int64_t n, uint32_t *keys, cudaStream_t s);

// Sum over rows of the checksum hash H(row) into ctr[CTR_SUM] (count = n).
cudaError_t launch_hash_rows(const int32_t *rows, int64_t n, int32_t w, unsigned long long *ctr, cudaStream_t s);

// Canonical row order by comparison sort (sort.cu): *perm_out (inside tmp) receives the
// row indices in ascending lexicographic order; ids are below 2^bits. tmp holds
// msort_tmp_bytes(n) bytes.
int64_t msort_tmp_bytes(int64_t n);
// Tables of at most msort_into_max_rows() rows: the canonical order written straight into
// out_rows / out_scores (nullable) in three launches (key packing with the optional checksum,
// tile sort, rank scatter, the last on at most max_blocks blocks); tmp as for msort_rows.
int64_t msort_into_max_rows();
cudaError_t msort_rows_into(const int32_t *rows, const float *scores, int64_t n, int32_t w, int bits, void *tmp,
                            int32_t *out_rows, float *out_scores, unsigned long long *sum, int max_blocks,
                            cudaStream_t s);
// When sum is set, the row checksums (sum of H(row), as the count-mode join) are added to it.
cudaError_t msort_rows(const int32_t *rows, int64_t n, int32_t w, int bits, void *tmp, int32_t **perm_out,
                       unsigned long long *sum, cudaStream_t s);

// Canonical order of a table of embeddings whose row count is on the device (order.cu). The counters
// ctr[CTR_SUM] (zeroed by the caller) and ctr[CTR_OVF] receive the rows' checksum and whether the order
// was given up (more than cap rows, or a bucket too full; no rows are written then, and the checksum only in the
// second case).
constexpr int ORD_KW = 4, ORD_MAX = 1 << 20;             // words of a key, buckets
constexpr int ORD_BUCKET = 1024, ORD_CROWDED = 4096;     // most rows of a bucket, with n_dev and without
constexpr int64_t ORD_ROWS = (int64_t)ORD_MAX * ORD_BUCKET;
constexpr int ORD_FINE = 2;                              // log2 rows a bucket, for keys that crowd
constexpr uint8_t ORD_NONE = 255;
struct OrderWork {
  uint32_t count[ORD_MAX];           // zero between calls
  uint32_t start[ORD_MAX + 1];
};
struct OrderArgs {
  const int32_t *rows;
  const float *sc;                   // nullable
  int64_t n;                         // rows, unless n_dev says it
  const unsigned long long *n_dev;
  int64_t cap;                       // rows key, num, idx, out and outs have room for, at most ORD_ROWS
  int32_t w, packed;                 // packed: columns held in the key
  int32_t log2_many;                 // rows a bucket of large tables (order_layout), fewer where keys crowd
  const uint2 *adj4;                 // neighbour lists of the data graph, for columns with ref
  int32_t radix_id, radix_place;     // of a column's id, and of its place among an earlier one's neighbours
  unsigned long long scale, unit;    // the first word times scale is its fraction of 2^64; 2^64 - 1 over scale
  uint8_t ref[dmi::MAXW];            // an earlier column that is a pattern neighbour, or ORD_NONE
  uint8_t word[dmi::MAXW];
  OrderWork *work;
  unsigned long long *key;           // kw x cap
  int32_t *num, *idx;                // row -> its number in its bucket; place -> row
  int32_t *out;
  float *outs;
  unsigned long long *ctr;
};
int64_t order_work_bytes();
int order_layout(OrderArgs &a, unsigned radix_id, unsigned radix_place);  // returns kw
cudaError_t order_rows(const OrderArgs &a, int kw, int num_sms, cudaStream_t s);

// The min(k, n) best rows of a table by (score, row), k <= SEL_K (select.cu). out: the number of rows
// collected on the way (4 bytes, padded to 16; above SEL_CAP nothing else was written and the caller
// takes another way), k scores, k rows. work: select_work_bytes(), zeroed once before the first call.
constexpr int SEL_K = 1024, SEL_CAP = 16384;
struct SelectArgs {
  const int32_t *rows;
  const float *sc;
  int64_t n;                         // rows, or with n_dev the most *n_dev may say
  const unsigned long long *n_dev;
  int32_t w, k, sorted;              // sorted: the rows are in canonical order
  int32_t counted;                   // the scores are in the work buffer's histogram already
  void *work;
  unsigned char *out, *h_out;        // the result; where set, pinned host memory that receives it as well
};
constexpr int64_t select_out_bytes(int64_t k, int64_t w) { return 16 + 4 * k + 4 * k * w; }
int64_t select_work_bytes();
// (the work buffer starts with a SelHist, all zero but bound = the bits of +infinity between calls)
constexpr int32_t SEL_NO_BOUND = 0x7F800000;
cudaError_t topk_select(const SelectArgs &a, int num_sms, cudaStream_t s);

// Images (sort.cu): sort the ids inside each row in place; then, on canonically sorted rows,
// keep the first row of every run of equal rows (pos[n] receives the number kept; flag holds n
// ints, pos n + 1, tmp scan_tmp_elems(n)).
cudaError_t images_prepare(int32_t *rows, int64_t n, int32_t w, cudaStream_t s);
cudaError_t unique_rows(const int32_t *rows, int64_t n, int32_t w, int32_t *flag, int64_t *pos, int64_t *tmp,
                        int32_t *out, cudaStream_t s);

// Persistent batch kernel (batch.cu).
struct BatchPlan {
  int32_t n_steps;
  int32_t args_off;  // index of the plan's first step in BatchParams::args
  int32_t seed_direct;  // warp walks: the first step keeps every motif row as it stands (no check, columns
                        // in table order) and is not the last; the second reads the table
};
struct BatchItem {
  int32_t plan;
  int32_t pad;
  int64_t lo, hi;    // rows of the first slice's motif table
};
struct BatchParams {
  const dmi::JoinArgs *args;
  const BatchPlan *plans;
  const BatchItem *items;
  int64_t n_items;
  unsigned long long *next_item;  // work counter (zeroed before the launch)
  unsigned long long *out;        // count, checksum per plan (zeroed before the launch)
  unsigned long long *ovf;
  unsigned char *scratch;         // grid * cta_bytes (warp walks: one cta_bytes slice per warp)
  int64_t cta_bytes;
  int64_t lvl_off[dmi::MAXSTEPS]; // byte offset of level j inside a CTA's scratch
  int64_t lvl_cap[dmi::MAXSTEPS]; // rows level j can hold
  int TR;                         // rows per tile
  int ws_max;                     // shared-memory row stride covering every step
  int bm_words;                   // > 0: per tile row, a bitmap of its ids (ids < 64 * bm_words) for
                                  // the injectivity test of steps with many new vertices
  unsigned long long *plan_left;  // work items still open per plan (set before the launch)
  unsigned long long *plan_done;  // GPU global-timer time at which each plan's last item ended
  unsigned long long *start_ns;   // GPU global-timer time at the start of the launch
  int max_steps;                  // warp walks: the most steps of a plan (per-warp level state)
  int tile_words;                 // warp walks: words of each walk's shared tile (a multiple of 4)
  // warp walks: items of plans that k_batch_wide runs (two steps, the second deciding many new vertices
  // by injectivity alone), and per entry of args the id bitmaps (sig_units x 256 bits a row) of the
  // motif rows such a plan reads, or null
  const BatchItem *wide;
  int64_t n_wide;
  unsigned long long *next_wide;  // work counter (zeroed before the launch)
  const uint32_t *const *sigs;
  int sig_units;
};
// threads: 128 or 256 per CTA. batch_grid: SMs x resident CTAs per SM (at most max_per_sm when
// it is > 0).
size_t batch_smem_bytes(int tile_rows, int ws_max, int bm_words, int threads);
int batch_grid(int tile_rows, int ws_max, int bm_words, int num_sms, int threads, int max_per_sm);
cudaError_t launch_batch(const BatchParams &p, int grid, int threads, cudaStream_t s);
// The same batch with one depth-first walk per warp (k_batchw, 64-thread CTAs): tiles of up to
// 32 rows (TR = 32; a step of row stride s takes min(32, tile_words / s)), the levels of each warp
// in its own cta_bytes slice of scratch, rows of level j of stride args[j].rs_out (padded,
// working-column order) or args[j].wo. walk_grid: SMs x resident CTAs per SM (at most max_per_sm
// when it is > 0); BW_WALK_WARPS warps a CTA. BW_WALK_TILE_STRIDE: the row stride (words) that a
// walk's tile holds 32 rows of.
constexpr int BW_WALK_WARPS = 2, BW_WALK_TILE_STRIDE = 28;
// The wide plans of a batch of warp walks, on graphs of up to 256 * BATCH_SIG_UNITS vertices; and the
// id bitmaps of a motif table (su units of 256 bits a row).
constexpr int BATCH_SIG_UNITS = 4;
cudaError_t launch_batch_wide(const BatchParams &p, int num_sms, cudaStream_t s);
cudaError_t launch_row_bits(const int32_t *rows, int mw, int64_t n, int su, uint32_t *out, cudaStream_t s);
size_t walk_smem_bytes(int tile_words, int max_steps);
int walk_grid(int tile_words, int max_steps, int num_sms, int max_per_sm);
cudaError_t launch_batch_walk(const BatchParams &p, int grid, cudaStream_t s);

// Cardinality model (mlp.cu): flat FP32 parameters, BF16 tensor-core forward / backward.
int64_t mlp_param_count();
int64_t mlp_work_bytes(int rows);
// Word of the work buffer that the forward/backward pass sets when a tensor-core wait ran out
// (the pass's outputs are then invalid); zeroed at the start of every pass.
unsigned *mlp_error_flag(void *work, int rows);
cudaError_t mlp_forward_backward(const float *params, const float *X, const float *target, int rows, int n_valid,
                                 float *y, float *grads, float *loss, void *work, cudaStream_t s);
// Training (mlp.cu): one Adam step on m samples (rows idx[0 .. m) of X and target) in two launches. The
// launches before must be this stream's kernels or copies. err[0] is raised as mlp_error_flag is, and no step is
// taken once it is up; err[1] counts the steps taken. *loss is added to.
struct MlpTrain {
  float *params, *m, *v;
  const float *X, *target;   // standardised samples, n x 32, and their targets
  __nv_bfloat16 *Xb, *H1, *H2, *dH2, *dH1;  // kept for the weight gradients: column blocks of 8 x R samples
  float *dy;
  uint16_t *W1b, *W2b;       // the rounded weights, in the products' layout
  int64_t R;
  unsigned *err;
};
// Fresh parameters from a seed, and zero moments.
cudaError_t mlp_init(float *params, float *m, float *v, uint64_t seed, cudaStream_t s);
int64_t mlp_train_bytes(int batch);
void mlp_train_layout(MlpTrain &T, void *work, int batch);  // places the buffers of a batch in work
cudaError_t mlp_train_begin(const MlpTrain &T, cudaStream_t s);  // before the first step: W1b, W2b from params
cudaError_t mlp_train_step(const MlpTrain &T, const int32_t *idx, int m, float *loss, float lr, int step, cudaStream_t s);

}  // namespace dmk
