// Shared declarations of the FASA CUDA library (sm_100a only).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include "fasa.h"

#define FASA_HEAD_DIM 128
#define FASA_MAX_GROUP 8
#define FASA_MAX_DOM 64

// Context: the normalised configuration plus a small device table.
struct fasa_ctx {
  fasa_config_t cfg;      // strides and softmax_scale filled in
  int group;              // query heads per KV head
  int sel_heads;          // query heads that share one index set (a divisor of group)
  int n_sets;             // index sets (selection units) per sequence = n_q_heads / sel_heads
  int chunks;             // 16-byte chunks per proxy row = ceil(n_dom / 4)
  int row_elems;          // bf16 elements per proxy row = 8 * chunks
  int device;
  int n_sm;
  const int32_t* block_table;  // paged caches: device [batch][pages_per_seq], caller-owned; null until set
  int page_shift;         // log2(page_size), 0 for contiguous caches
  int pages_per_seq;      // ceil(max_len / page_size)
  int16_t* d_chan;        // device [n_kv_heads][row_elems]: K channel of each proxy element, -1 = padding
  void* m_resident;       // memory-optimised variant: the caller's buffer of GPU-resident sink / recent rows (null: none)
  int16_t* d_ndchan;      // device [n_kv_heads][128 - 2 n_dom]: the other channels of each head, ascending (null
                          // unless n_dom is a multiple of 4: the split key cache of the memory-optimised variant)
  int32_t* d_status;      // device status word (FASA_DEV_* bits)
  int32_t* d_arrive;      // device [batch]: CTAs of a sequence that have read its length (append-then-step)
  int fused_cs;           // cluster size of the cluster kernel (step and top-k), 0 = not available
  int fused_step_ok;      // the one-launch step supports this configuration
  size_t fused_smem;      // its dynamic shared memory
  int step_threads;       // the decode step's own shape: 512 threads with fused_cs CTAs per cluster, or the wide
  int step_cs;            // form (1024 threads, one CTA per SM, half the cluster) where that evens out the stream
  size_t step_smem;
  int step_resident;      // clusters of the step's shape that the device holds at once
  int use_fused;          // fasa_decode_step takes the one-launch kernel when it is available
  int topk_rows;          // fasa_topk and fasa_topk_batched by the one-CTA-per-row kernel whatever the rows (fasa_set_step_mode 2)
  long long launches;     // kernels launched through this context
  char cuda_err[256];
};

// Records a CUDA failure in the context and returns FASA_ERR_CUDA from the caller.
#define FASA_CUDA_TRY(ctx, expr)                                                       \
  do {                                                                                 \
    cudaError_t e_ = (expr);                                                           \
    if (e_ != cudaSuccess) {                                                           \
      snprintf((ctx)->cuda_err, sizeof((ctx)->cuda_err), "%.120s: %.100s", #expr,      \
               cudaGetErrorString(e_));                                                \
      return FASA_ERR_CUDA;                                                            \
    }                                                                                  \
  } while (0)

#define FASA_LAUNCH_CHECK(ctx)                                                         \
  do {                                                                                 \
    (ctx)->launches += 1;                                                              \
    FASA_CUDA_TRY(ctx, cudaGetLastError());                                            \
  } while (0)

// How the attention kernels cut a list of at most n_upper rows per unit into splits, given
// the number of units (grid.y) of the launch.
struct fasa_split_plan {
  int n_splits;   // grid.x
  int chunk;      // rows per split (multiple of 32)
};
fasa_split_plan fasa_plan_splits(const fasa_ctx* ctx, int n_upper, int units);
// CTAs of the dense pass over long contexts: what the device holds at once (six per SM, four on pages), and how many are
// launched: 1.8 times that where contiguous caches can hold 64 tiles of 16 rows for each (see dense_deal).
constexpr int kDenseTiles = 64;
static inline int fasa_dense_resident(const fasa_ctx* ctx) { return (ctx->cfg.page_size > 0 ? 4 : 6) * (ctx->n_sm > 0 ? ctx->n_sm : 148); }
static inline int fasa_dense_ctas(const fasa_ctx* ctx) {
  const int res = fasa_dense_resident(ctx);
  const long long tiles = (long long)ctx->cfg.batch * ctx->cfg.n_kv_heads * ((ctx->cfg.max_len + 15) / 16);
  return ctx->cfg.page_size == 0 && tiles >= (long long)kDenseTiles * res ? res * 9 / 5 : res;
}

// One-launch decode step (fasa_fused.cu): plan at context creation, launch per step.
int fasa_fused_plan(fasa_ctx* ctx);
int32_t fasa_fused_launch(fasa_ctx* ctx, const void* q, const void* k_cache, const void* v_cache,
                          const void* proxy_k, const int32_t* seq_lens, int32_t budget,
                          int32_t n_sel_max, float* scores, int32_t* idx, int32_t* n_sel,
                          float* out, float* lse, const void* k_new, const void* v_new,
                          cudaStream_t stream, bool with_attention = true, float* out_mirror = nullptr,
                          bool split_keys = false);
// Whether the attention of a step is a launch of its own, the split-K tensor-core kernel, rather than the last phase of the
// cluster kernel.  A grid whose clusters are all resident attends in its own launch, whatever the selection: the hand-over
// costs two launches (batch 8 x 8 heads at 64 K: 58 against 52 us at budget 256, 68 / 62 at 1024, 90 / 80 at 4096; 32 x 4
// heads with 7 query heads each at 9 K: 58 / 53 at 1700; 12 x 8 in pages at 3-28 K: 103 / 91 at 4096; batch 4 x 8 at 9 K and
// 4096: 37 / 39 us, the one loss).  A grid of several rounds pays for the attention in every round while HBM waits for the next
// round's streams: there one launch for all units is better (16 x 8 heads at 64-128 K: 154 against 166 us at budget 64, 175 /
// 189 at 1024, 214 / 228 at 4096), except for 512 rows or more where two CTAs share an SM and one's attention runs beside the
// other's stream (48 x 8 at 16 K: 105 / 107 us at 256, 143 / 133 at 1024; 64 x 4 x 7 at 20 K 86 / 89, 107 / 103).
// A resident grid of barely more CTAs than SMs leaves most SMs with one CTA beside some with two.  One or two heads per set
// do not make up for that: clusters of one attend separately from 1024 rows on (160 units of two heads at 10 K, 2048 rows: 71
// against 79 us, at 3 K and 1455 51 / 55; 256 units 95 / 91), larger ones below that on long slices (96 units at 10 K, 512
// rows: 33 / 34.5; 2048 rows: 59 / 52.5).
// From some thousand rows on the attention itself decides.  Clusters of four 512-thread CTAs, each alone on its SM, have 16
// warps an SM to gather with, the split-K kernel 20 and more (4 x 8 at 16 K: 25.5 / 26.4 us at 1024, 35.7 / 40.7 at 4096, 50.2 /
// 59.1 at 8192).  And where several sets read the rows of one KV head they come from L2, and what counts is the instructions
// per row, of which 16-row tiles need fewer: four sets or more to a KV head from 1024 rows on (a set per head, 16 x 32 at 16 K:
// 209 / 226 us at 3072, 352 / 444 at 8192; 4 x 28 at 32 K 97 / 116 at 6144), two sets of several heads once they hold a fifth
// of the context (16 x 16 sets of two heads at 16 K: 201 / 233 at 8192, 32 x 16 at 8 K 208 / 236 at 4096).
// Up to eight units on short caches keep the two launches that they are documented with (2 x 4 x 7 at 5.4 K, 1800 rows: 23.9
// us; one launch would take 20.7).
static inline bool fasa_attend_separately(const fasa_ctx* ctx, int n_sel_max, const void* workspace) {
  const bool pairs = (long long)ctx->step_resident * ctx->step_cs > ctx->n_sm;
  const long long units = (long long)ctx->cfg.batch * ctx->n_sets;
  const bool documented = units <= 8 && ctx->cfg.max_len <= 8192 && (long long)n_sel_max * ((ctx->sel_heads + 3) / 4) >= 2048;
  const long long ctas = units * ctx->step_cs;
  const bool uneven = ctx->sel_heads <= 2 && ctx->step_threads == 512 && ctas > ctx->n_sm && 10 * ctas <= 13ll * ctx->n_sm &&
                      (ctx->step_cs == 1 ? n_sel_max >= 1024 : n_sel_max >= 64 && n_sel_max < 1024 && ctx->cfg.max_len / ctx->step_cs >= 4096);
  const bool lone = ctx->step_threads == 512 && ctx->step_cs == 4 && ctas <= ctx->n_sm && 8 * units >= ctx->n_sm && n_sel_max >= 1024;
  const int sharing = ctx->group / ctx->sel_heads;
  const bool from_l2 = (sharing >= 4 && units >= 96 && n_sel_max >= 1024) ||
                       (sharing >= 2 && ctx->sel_heads >= 2 && n_sel_max >= 2048 && 5ll * n_sel_max >= ctx->cfg.max_len);
  return workspace != nullptr && (uneven || lone || from_l2 || (units > ctx->step_resident && n_sel_max >= 64 && !(pairs && n_sel_max >= 512)) || documented);
}

// Whether the attention of a step that runs on 16-row tiles (a launch of its own, or select-and-attend) keeps all 24 bits of a
// probability.  The cluster kernel does; the split-K kernel's 17 bits are for lists that are long, or of which there are so many
// that the gather decides (the third term costs 1 to 4 % there: 16 x 32 sets of 4096 rows 325 -> 332 us).
static inline bool fasa_full_probabilities(const fasa_ctx* ctx, int n_sel_max) {
  const long long rows = (long long)n_sel_max * ((ctx->sel_heads + 3) / 4), units = (long long)ctx->cfg.batch * ctx->n_sets;
  return !(rows >= 2048 || (rows >= 256 && units * ctx->fused_cs > 2ll * ctx->n_sm) || (rows >= 512 && rows * units >= 24576));
}

cudaError_t fasa_stage_from_mapped(void* dq, const void* sq, size_t q_bytes, void* dk, const void* sk, void* dv,
                                   const void* sv, size_t kv_bytes, cudaStream_t stream);

int32_t fasa_sparse_attn_mirrored(fasa_ctx* ctx, const void* q, const void* k_cache, const void* v_cache,
                                  const int32_t* idx, const int32_t* n_sel, int32_t n_sel_max, float* out,
                                  float* lse, void* workspace, cudaStream_t stream, float* out_mirror, bool* mirrored, bool full_p);

// Split key cache (memory-optimised variant): what the attention kernels need besides k_nondom.
// The rows every step attends to (the sink positions and the recent window) can stay on the GPU:
// a slot per sink position and a ring of n_recent slots for the positions behind them, each
// tagged with the position it holds.  A slot holds the key row as the attention kernel
// assembles it (non-dominant channels, then the dominant pairs in proxy order) and the value row.
struct fasa_resident {
  int32_t* tags;                // [batch * n_kv_heads][slots_pad]: position held by each slot, -1 = none
  uint16_t* rows;               // [batch * n_kv_heads][slots][2][128]
  int slots, slots_pad, n_sink, n_recent;   // tags == nullptr: no resident rows
};
__host__ __device__ inline int fasa_resident_slot(const fasa_resident& r, int tok) {
  if (tok < r.n_sink) return tok;
  return r.n_recent > 0 ? r.n_sink + (tok - r.n_sink) % r.n_recent : -1;
}
struct fasa_ksplit {
  const unsigned char* proxy;   // the dominant part, on the GPU
  const int16_t* ndchan;        // [n_kv_heads][nd]
  const int16_t* chan;          // [n_kv_heads][2 n_dom]
  int chunks, nd;               // 16-byte chunks per proxy row; non-dominant channels per key
  fasa_resident res;            // rows that need not cross the host link
};
fasa_resident fasa_resident_of(const fasa_ctx* ctx);
int32_t fasa_attn_split_keys(fasa_ctx* ctx, const void* q, const void* k_nondom, const void* v_cache, const void* proxy_k,
                             const int32_t* idx, const int32_t* n_sel, int32_t n_sel_max, float* out, float* lse,
                             void* workspace, cudaStream_t stream);
bool fasa_on_host(const void* p);

bool fasa_topk_row_ok(const fasa_ctx* ctx);
// Calibration: the single-FC rows of a (sequence, query head) are not stored, they are computed from the KV head's
// channel pairs: pairs [batch * n_kv_heads][64][stride], two bf16 values per position.
struct fasa_calib_rows {
  const uint32_t* pairs;
  const uint16_t* q;        // [samples][128]
  int64_t stride;           // positions per row, a multiple of 4 (also of the full-head score rows)
  int group, pairing;       // query heads per KV head; rope_pairing
};
// TopK-I over rows_per_seq score rows per sequence (row r of the buffer belongs to sequence
// r / rows_per_seq), with the given forced positions.  q_len > 1: the rows of a sequence are (query, set)
// pairs, query-major, and query t of the block sees seq_lens[b] - (q_len - 1 - t) positions.
int32_t fasa_topk_row_launch(fasa_ctx* ctx, const float* scores, const int32_t* seq_lens, int32_t budget,
                             int32_t n_sel_max, int32_t* idx, int32_t* n_sel, int rows_per_seq, int n_sink,
                             int n_recent, cudaStream_t stream, int q_len = 1, const struct fasa_calib_rows* calib = nullptr,
                             const struct fasa_row_maxima* given = nullptr);
// Where the scoring pass leaves the maxima of groups of 1 << gs scores, a row of `stride` of them for each score row; the size
// of the groups that a selection of n_rows rows would use (0: it would not).
struct fasa_row_maxima {
  float* gm;
  int gs, stride;
};
size_t fasa_block_maxima_bytes(const fasa_ctx* ctx);   // of the largest block of queries, a set to a KV head
int fasa_row_maxima_shift(const fasa_ctx* ctx, int budget, long long n_rows);
// Floats per row of such a buffer with groups of 8.
int fasa_stream_gm_stride(const fasa_ctx* ctx);
// The same by the selection phases of the cluster kernel (fasa_fused.cu), for contexts that it can serve (fused_cs > 0).
int32_t fasa_topk_cluster_launch(fasa_ctx* ctx, const float* scores, const int32_t* seq_lens, int32_t budget, int32_t n_sel_max,
                                 int32_t* idx, int32_t* n_sel, int rows_per_seq, int n_sink, int n_recent, cudaStream_t stream,
                                 int q_len);
// Paged caches: how a (sequence, token) pair finds its page.  All zero = contiguous caches.
struct PageMap {
  const int32_t* table;   // [batch][pages_per_seq]: physical page of each logical page
  int shift;              // log2(tokens per page)
  int pages_per_seq;
  int n_pages;
};
static inline PageMap fasa_page_map(const fasa_ctx* ctx) {
  PageMap m;
  m.table = ctx->block_table;
  m.shift = ctx->page_shift;
  m.pages_per_seq = ctx->pages_per_seq;
  m.n_pages = ctx->cfg.n_pages;
  return m;
}
// Paged contexts need their block table before any call that touches a cache.
static inline bool fasa_pages_ready(const fasa_ctx* ctx) { return ctx->cfg.page_size == 0 || ctx->block_table != nullptr; }

static inline size_t fasa_align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

#ifdef __CUDACC__

// Two bf16 packed in a 32-bit word -> two fp32 (exact).
__device__ __forceinline__ float2 bf16x2_to_f32x2(uint32_t w) {
  return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}

__device__ __forceinline__ float bf16_bits_to_f32(uint16_t b) {
  return __uint_as_float(((uint32_t)b) << 16);
}

// 128-bit read-only load that does not allocate in L1 (streamed once).
__device__ __forceinline__ uint4 ld_stream_u4(const void* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// Dot product of 8 fp32 (as 4 float2) with 8 bf16 (one uint4), packed FMAs.
__device__ __forceinline__ float dot8(const float2 (&q)[4], const uint4& k) {
  float2 a = make_float2(0.f, 0.f);
  a = __ffma2_rn(q[0], bf16x2_to_f32x2(k.x), a);
  a = __ffma2_rn(q[1], bf16x2_to_f32x2(k.y), a);
  a = __ffma2_rn(q[2], bf16x2_to_f32x2(k.z), a);
  a = __ffma2_rn(q[3], bf16x2_to_f32x2(k.w), a);
  return a.x + a.y;
}

__device__ __forceinline__ bool page_ok(const PageMap& m, int page) { return page >= 0 && page < m.n_pages; }
__device__ __forceinline__ int page_of(const PageMap& m, int b, int tok) {
  // (not through the read-only path: the table may change in stream order, and kernels wait for their predecessor inside)
  return m.table[(int64_t)b * m.pages_per_seq + (tok >> m.shift)];
}
// Element offset of row `tok` of (sequence b, KV head h) in a K or V cache, for reading: an
// entry outside the pool reads page 0 and raises the status bit.
__device__ __forceinline__ int64_t cache_row(const PageMap& m, int b, int h, int tok, int64_t sb, int64_t sh,
                                             int64_t st, int32_t* status) {
  if (m.table == nullptr) return b * sb + h * sh + (int64_t)tok * st;
  int page = page_of(m, b, tok);
  if (!page_ok(m, page)) {
    atomicOr(status, FASA_DEV_PAGE_CLAMPED);
    page = 0;
  }
  return page * sb + h * sh + (int64_t)(tok & ((1 << m.shift) - 1)) * st;
}
// The pool's row of token `tok` of sequence b: its page, and the row within the page in the low bits (a pool holds fewer
// than 2^31 rows: they are at least 512 bytes each).
__device__ __forceinline__ int pool_row(const PageMap& m, int b, int tok, int32_t* status) {
  int page = page_of(m, b, tok);
  if (!page_ok(m, page)) {
    atomicOr(status, FASA_DEV_PAGE_CLAMPED);
    page = 0;
  }
  return (page << m.shift) | (tok & ((1 << m.shift) - 1));
}
// Byte offset of the proxy tile of token tile T (tokens 16 T .. 16 T + 15) of (b, h).
// status == nullptr: a speculative read (a tile that may lie past the sequence's end, where no
// page need be mapped) - page 0 is read and nothing is reported.
__device__ __forceinline__ int64_t proxy_tile_offset(const PageMap& m, int b, int h, int n_kv_heads, int T,
                                                     int tiles_per_unit, int tile_bytes, int32_t* status) {
  if (m.table == nullptr) return ((int64_t)(b * n_kv_heads + h) * tiles_per_unit + T) * tile_bytes;
  int page = (T >> (m.shift - 4)) < m.pages_per_seq ? page_of(m, b, T << 4) : -1;
  if (!page_ok(m, page)) {
    if (status) atomicOr(status, FASA_DEV_PAGE_CLAMPED);
    page = 0;
  }
  const int tpp = 1 << (m.shift - 4);           // tiles per page
  return (((int64_t)page * n_kv_heads + h) * tpp + (T & (tpp - 1))) * tile_bytes;
}

// Reports (status bit) a token tile whose page is not in the pool; for tiles that were read
// speculatively and turned out to be part of the sequence.
__device__ __forceinline__ void proxy_tile_check(const PageMap& m, int b, int T, int32_t* status) {
  if (m.table != nullptr && !page_ok(m, page_of(m, b, T << 4))) atomicOr(status, FASA_DEV_PAGE_CLAMPED);
}

// A selection unit: `heads` consecutive query heads of one sequence that share an index set
// (Sec. 4.1 keeps a set per head; by default all heads of a KV head share one).  Unit u of
// the grid is set hs = u % n_sets of sequence b = u / n_sets.
struct SelUnit {
  int b;        // sequence
  int h;        // KV head whose cache the unit reads
  int kv;       // b * n_kv_heads + h: index of that cache (K, V, proxy, appended rows)
  int64_t q0;   // b * n_q_heads + first query head of the unit: row of q, out and lse
};
__device__ __forceinline__ SelUnit sel_unit(int u, int n_sets, int heads, int n_q_heads, int n_kv_heads) {
  SelUnit s;
  const int hs = u % n_sets;
  s.b = u / n_sets;
  s.h = hs / (n_sets / n_kv_heads);
  s.kv = s.b * n_kv_heads + s.h;
  s.q0 = (int64_t)s.b * n_q_heads + (int64_t)hs * heads;
  return s;
}

__device__ __forceinline__ int clamp_len(int len, int max_len, int32_t* status) {
  if (len < 0 || len > max_len) {
    atomicOr(status, FASA_DEV_LEN_CLAMPED);
    len = len < 0 ? 0 : max_len;
  }
  return len;
}

#endif  // __CUDACC__
