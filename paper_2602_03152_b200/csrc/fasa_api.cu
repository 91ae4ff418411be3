// Context, validation, workspace sizing and the composite calls of the C ABI.
#include <algorithm>
#include <new>
#include <vector>

#include "fasa_common.cuh"
#include "fasa_select.cuh"
#include "fasa_stream.cuh"

namespace {

bool valid_cfg(const fasa_config_t& c, int32_t* why) {
  *why = FASA_ERR_INVALID_ARG;
  if (c.batch <= 0 || c.n_q_heads <= 0 || c.n_kv_heads <= 0 || c.max_len <= 0) return false;
  if (c.n_sink < 0 || c.n_recent < 0) return false;
  if (c.softmax_scale < 0.f || c.softmax_scale != c.softmax_scale) return false;
  *why = FASA_ERR_UNSUPPORTED;
  if (c.head_dim != FASA_HEAD_DIM) return false;
  if (c.n_dom < 1 || c.n_dom > FASA_MAX_DOM) return false;
  if (c.n_q_heads % c.n_kv_heads != 0) return false;
  if (c.n_q_heads / c.n_kv_heads > FASA_MAX_GROUP) return false;
  if (c.rope_pairing != 0 && c.rope_pairing != 1) return false;
  if (c.group_reduce != 0 && c.group_reduce != 1) return false;
  if (c.page_size != 0) {
    if (c.page_size < 16 || (c.page_size & (c.page_size - 1)) != 0 || c.n_pages < 1) return false;
  }
  if (c.select_heads < 0) return false;
  const int group = c.n_q_heads / c.n_kv_heads;
  const int per_set = c.select_heads > 0 ? c.select_heads : group;
  if (group % per_set != 0) return false;
  if ((long long)c.batch * (c.n_q_heads / per_set) > 65535) return false;  // grid.y
  return true;
}

bool fill_strides(int64_t& sb, int64_t& sh, int64_t& st, const fasa_config_t& c) {
  if (sb == 0 && sh == 0 && st == 0) {
    st = FASA_HEAD_DIM;
    sh = (int64_t)(c.page_size > 0 ? c.page_size : c.max_len) * FASA_HEAD_DIM;   // rows per head of a page / a sequence
    sb = sh * c.n_kv_heads;
    return true;
  }
  // rows are read with 16-byte loads
  return st >= FASA_HEAD_DIM && st % 8 == 0 && sh % 8 == 0 && sb % 8 == 0 && sh > 0 && sb > 0;
}

}  // namespace

extern "C" int32_t fasa_proxy_row_elems(int32_t n_dom) {
  if (n_dom < 1 || n_dom > FASA_MAX_DOM) return 0;
  return 8 * ((n_dom + 3) / 4);
}

extern "C" int32_t fasa_proxy_bytes(const fasa_ctx_t* ctx, size_t* out_bytes) {
  if (!ctx || !out_bytes) return FASA_ERR_INVALID_ARG;
  const fasa_config_t& c = ctx->cfg;
  const size_t rows = (size_t)((c.max_len + 15) / 16) * 16;
  *out_bytes = c.page_size > 0 ? (size_t)c.n_pages * c.n_kv_heads * c.page_size * ctx->row_elems * 2
                               : (size_t)c.batch * c.n_kv_heads * rows * ctx->row_elems * 2;
  return FASA_OK;
}

extern "C" int32_t fasa_create(const fasa_config_t* cfg, const int32_t* dom_fc_host,
                               fasa_ctx_t** out) {
  if (!cfg || !dom_fc_host || !out) return FASA_ERR_INVALID_ARG;
  *out = nullptr;
  int32_t why;
  if (!valid_cfg(*cfg, &why)) return why;

  fasa_ctx* ctx = new (std::nothrow) fasa_ctx();
  if (!ctx) return FASA_ERR_INVALID_ARG;
  memset(ctx, 0, sizeof(*ctx));
  ctx->cfg = *cfg;
  fasa_config_t& c = ctx->cfg;
  if (!fill_strides(c.k_stride_b, c.k_stride_h, c.k_stride_t, c) ||
      !fill_strides(c.v_stride_b, c.v_stride_h, c.v_stride_t, c)) {
    delete ctx;
    return FASA_ERR_INVALID_ARG;
  }
  if (c.softmax_scale == 0.f) c.softmax_scale = 0.08838834764831845f;  // 1/sqrt(128)
  ctx->group = c.n_q_heads / c.n_kv_heads;
  ctx->sel_heads = c.select_heads > 0 ? c.select_heads : ctx->group;
  ctx->n_sets = c.n_q_heads / ctx->sel_heads;
  if (c.page_size > 0) {
    while ((1 << ctx->page_shift) < c.page_size) ++ctx->page_shift;
    ctx->pages_per_seq = (c.max_len + c.page_size - 1) / c.page_size;
  }
  ctx->chunks = (c.n_dom + 3) / 4;
  ctx->row_elems = 8 * ctx->chunks;

  // Channel table: dominant FCs sorted ascending, FC r of head h at elements 2r, 2r+1.
  std::vector<int16_t> chan((size_t)c.n_kv_heads * ctx->row_elems, (int16_t)-1);
  for (int h = 0; h < c.n_kv_heads; ++h) {
    std::vector<int32_t> fcs(dom_fc_host + (size_t)h * c.n_dom, dom_fc_host + (size_t)(h + 1) * c.n_dom);
    std::sort(fcs.begin(), fcs.end());
    for (int r = 0; r < c.n_dom; ++r) {
      bool bad = fcs[r] < 0 || fcs[r] >= FASA_HEAD_DIM / 2 || (r > 0 && fcs[r] == fcs[r - 1]);
      if (bad) {
        delete ctx;
        return FASA_ERR_INVALID_ARG;
      }
      int c0 = c.rope_pairing == 0 ? fcs[r] : 2 * fcs[r];
      int c1 = c.rope_pairing == 0 ? fcs[r] + FASA_HEAD_DIM / 2 : 2 * fcs[r] + 1;
      chan[(size_t)h * ctx->row_elems + 2 * r] = (int16_t)c0;
      chan[(size_t)h * ctx->row_elems + 2 * r + 1] = (int16_t)c1;
    }
  }

  // the complement of each head's dominant channels, ascending (split key cache)
  std::vector<int16_t> ndchan;
  if (c.n_dom % 4 == 0 && c.n_dom < FASA_HEAD_DIM / 2 && c.page_size == 0) {
    const int nd = FASA_HEAD_DIM - 2 * c.n_dom;
    ndchan.resize((size_t)c.n_kv_heads * nd);
    for (int h = 0; h < c.n_kv_heads; ++h) {
      bool dom[FASA_HEAD_DIM] = {false};
      for (int i = 0; i < 2 * c.n_dom; ++i) dom[chan[(size_t)h * ctx->row_elems + i]] = true;
      int n = 0;
      for (int ch = 0; ch < FASA_HEAD_DIM; ++ch)
        if (!dom[ch]) ndchan[(size_t)h * nd + n++] = (int16_t)ch;
    }
  }

  cudaError_t e = cudaGetDevice(&ctx->device);
  cudaDeviceProp prop;
  if (e == cudaSuccess) e = cudaGetDeviceProperties(&prop, ctx->device);
  if (e == cudaSuccess && prop.major != 10) {
    delete ctx;
    return FASA_ERR_UNSUPPORTED;  // built for sm_100a only
  }
  if (e == cudaSuccess) ctx->n_sm = prop.multiProcessorCount;
  if (e == cudaSuccess) e = cudaMalloc(&ctx->d_chan, chan.size() * sizeof(int16_t));
  if (e == cudaSuccess) e = cudaMalloc(&ctx->d_status, 256);
  if (e == cudaSuccess) e = cudaMalloc(&ctx->d_arrive, (size_t)c.batch * sizeof(int32_t));
  if (e == cudaSuccess) e = cudaMemset(ctx->d_arrive, 0, (size_t)c.batch * sizeof(int32_t));
  if (e == cudaSuccess)
    e = cudaMemcpy(ctx->d_chan, chan.data(), chan.size() * sizeof(int16_t), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(ctx->d_status, 0, 256);
  if (e == cudaSuccess && !ndchan.empty()) {
    e = cudaMalloc(&ctx->d_ndchan, ndchan.size() * sizeof(int16_t));
    if (e == cudaSuccess) e = cudaMemcpy(ctx->d_ndchan, ndchan.data(), ndchan.size() * sizeof(int16_t), cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    cudaFree(ctx->d_chan);
    cudaFree(ctx->d_ndchan);
    cudaFree(ctx->d_status);
    cudaFree(ctx->d_arrive);
    delete ctx;
    return FASA_ERR_CUDA;
  }
  fasa_fused_plan(ctx);
  ctx->use_fused = 1;
  *out = ctx;
  return FASA_OK;
}

// Whether a K/V cache pointer is host memory (the memory-optimised variant keeps the caches in page-locked host memory).  The
// driver is asked each time, 60 ns: an answer kept by address would be wrong for what is allocated there next.
bool fasa_on_host(const void* p) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) == cudaSuccess) return at.type == cudaMemoryTypeHost;
  cudaGetLastError();
  return false;
}

extern "C" int32_t fasa_set_block_table(fasa_ctx_t* ctx, const int32_t* block_table) {
  if (!ctx || !block_table || ctx->cfg.page_size == 0) return FASA_ERR_INVALID_ARG;
  ctx->block_table = block_table;
  return FASA_OK;
}

extern "C" int32_t fasa_destroy(fasa_ctx_t* ctx) {
  if (!ctx) return FASA_ERR_INVALID_ARG;
  cudaFree(ctx->d_chan);
  cudaFree(ctx->d_ndchan);
  cudaFree(ctx->d_status);
  cudaFree(ctx->d_arrive);
  delete ctx;
  return FASA_OK;
}

extern "C" const char* fasa_status_string(int32_t s) {
  switch (s) {
    case FASA_OK: return "ok";
    case FASA_ERR_INVALID_ARG: return "invalid argument";
    case FASA_ERR_UNSUPPORTED: return "unsupported configuration";
    case FASA_ERR_WORKSPACE: return "workspace too small for this selection size";
    case FASA_ERR_CUDA: return "CUDA runtime error";
    case FASA_ERR_TIMEOUT: return "timeout";
    default: return "unknown status";
  }
}

extern "C" const char* fasa_last_cuda_error(const fasa_ctx_t* ctx) {
  return ctx ? ctx->cuda_err : "";
}

extern "C" int32_t fasa_set_step_mode(fasa_ctx_t* ctx, int32_t mode) {
  if (!ctx || mode < 0 || mode > 2) return FASA_ERR_INVALID_ARG;
  ctx->use_fused = mode != 0;
  ctx->topk_rows = mode == 2;
  return FASA_OK;
}

extern "C" int32_t fasa_step_cluster_size(const fasa_ctx_t* ctx) {
  return ctx && ctx->use_fused && ctx->fused_step_ok ? (ctx->fused_cs > 0 ? ctx->step_cs : 0) : 0;
}

extern "C" int64_t fasa_launch_count(const fasa_ctx_t* ctx) { return ctx ? ctx->launches : 0; }

extern "C" int32_t fasa_get_device_status(fasa_ctx_t* ctx, void* stream, int32_t* host_out) {
  if (!ctx || !host_out) return FASA_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  FASA_CUDA_TRY(ctx, cudaMemcpyAsync(host_out, ctx->d_status, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  FASA_CUDA_TRY(ctx, cudaMemsetAsync(ctx->d_status, 0, sizeof(int32_t), s));
  FASA_CUDA_TRY(ctx, cudaStreamSynchronize(s));
  return FASA_OK;
}

// Splits: enough CTAs to fill the GPU a few times over, between 64 and 2048 rows each.
static int split_count_bound(const fasa_ctx* ctx, int n_upper, int units) {
  const int target = 4 * (ctx->n_sm > 0 ? ctx->n_sm : 148);
  const int want = std::max((target + units - 1) / units, (n_upper + 2047) / 2048);
  const int most = (n_upper + 63) / 64;
  return std::max(1, std::min(want, most));   // non-decreasing in n_upper, non-increasing in units
}

fasa_split_plan fasa_plan_splits(const fasa_ctx* ctx, int n_upper, int units) {
  const int n = split_count_bound(ctx, n_upper, units);
  int chunk = (n_upper + n - 1) / n;
  chunk = (chunk + 31) / 32 * 32;
  fasa_split_plan p;
  p.chunk = chunk;
  p.n_splits = std::max(1, (n_upper + chunk - 1) / chunk);  // <= n
  return p;
}

// Workspace: split-K partial results, then (contexts whose steps can run as two launches) what the first half passes to the
// second, a score row and a row of group maxima per index set.  A block of queries has its group maxima there before it attends:
// 4 bytes to a position and KV head.  The partial-result area is sized for the largest
// split count any call can use (the bound at max_len for the fewest units a launch can have, one per KV head), so
// nothing here depends on the selection size.
static bool set_per_head(const fasa_ctx* ctx) { return ctx->sel_heads == 1 && ctx->group > 1; }
// Whether the clusters of the one-launch step run in rounds, or some SMs hold two CTAs of it and others one.
static bool clusters_crowd(const fasa_ctx* ctx) {
  const long long units = (long long)ctx->cfg.batch * ctx->n_sets;
  return ctx->fused_cs > 0 && (units * ctx->step_cs > ctx->n_sm || units > ctx->step_resident);
}
// Scratch that grows with batch x max_len is for caches that do: of a page pool, those that hold half of it or more.  (Pages are there
// to give many long sequences room that they share: 64 sequences of up to 128 K, 8 heads, in a pool of 1 M tokens would have 370 MB
// of scratch beside 4.8 GB of cache and proxy, and have 68.)
static bool cache_covers_max_len(const fasa_ctx* ctx) {
  const fasa_config_t& c = ctx->cfg;
  return c.page_size == 0 || 2ll * c.n_pages * c.page_size >= (long long)c.batch * c.max_len;
}
// Whether any step of this context can run as two launches (see two_launches).
static bool two_launches_possible(const fasa_ctx* ctx) {
  if (ctx->cfg.max_len < 2048 || !fasa_select_attend_ok(ctx, 1)) return false;
  if (set_per_head(ctx)) return ctx->group >= 4 || (long long)ctx->cfg.batch * ctx->n_sets >= 192;
  return ctx->sel_heads == ctx->group && clusters_crowd(ctx) && cache_covers_max_len(ctx);
}
struct fasa_ws {
  size_t scores, gm, total;
};
static fasa_ws ws_layout(const fasa_ctx* ctx) {
  const fasa_config_t& c = ctx->cfg;
  const int n = split_count_bound(ctx, c.max_len, c.batch * c.n_kv_heads);
  const size_t per_split = (size_t)c.batch * c.n_q_heads * (FASA_HEAD_DIM + 2) * sizeof(float), rows = two_launches_possible(ctx) ? (size_t)c.batch * ctx->n_sets : 0;
  fasa_ws w;
  const size_t dense = ((size_t)fasa_dense_ctas(ctx) + (size_t)c.batch * c.n_kv_heads) * ctx->group * (FASA_HEAD_DIM + 2) * sizeof(float);
  w.scores = fasa_align_up(std::max(per_split * (size_t)n, dense), 256) + 256;
  w.gm = w.scores + fasa_align_up(rows * (size_t)c.max_len * sizeof(float), 256);
  w.total = w.gm + fasa_align_up(rows * (size_t)fasa_stream_gm_stride(ctx) * sizeof(float), 256);
  // (a block of queries keeps its group maxima here between scoring and selection, before any partial result)
  if (cache_covers_max_len(ctx)) w.total = std::max(w.total, fasa_block_maxima_bytes(ctx));
  return w;
}
extern "C" int32_t fasa_workspace_bytes(const fasa_ctx_t* ctx, int32_t n_sel_max, size_t* out_bytes) {
  if (!ctx || !out_bytes || n_sel_max < 0) return FASA_ERR_INVALID_ARG;
  *out_bytes = ws_layout(ctx).total;
  return FASA_OK;
}

// Whether a step over index sets per query head runs as two launches (score stream, then selection and attention)
// instead of the cluster kernel, which streams a KV head's proxy once per set.  Measured (32 / 8 heads): batch 4 at
// 50 K 92 -> 43 us with 128 rows a set, 99 -> 58 us with 1024; batch 16 at 16 K 123 -> 66 and 153 -> 121 us; batch 4 at
// 4 K 24 -> 19 us; 28 / 4 heads, batch 4 at 50 K 89 -> 33 us.  Few sets with long lists stay with the cluster kernel, whose
// CTAs share one selection (batch 1 at 16 K, 1024 rows a set: 24 against 28 us), as do groups of two or three, where the
// stream saves less (16 / 8 heads, batch 4 at 50 K: 40 against 42 us; batch 16 at 16 K: 71 -> 50 us), and rows shorter
// than 2048, which are one launch whatever the batch.  Every CTA of the second launch selects for itself, which large selections do
// not repay: beyond a sixteenth of the context nothing narrows a row down (batch 16 at 16 K, 1536 rows a set: 180 against
// 166 us by cluster kernel and split-K attention, 4096: 324 / 238; rows of up to 4096 are cheap to take whole, and of up to
// 8192 in larger groups: batch 16 at 4 K, 2048 rows 103 / 116; batch 8, 28 / 4 heads, at 8 K, 1024 rows 43 / 47), and beyond 2048
// rows a set has several such CTAs (batch 4 at 64 K: 2048 89 / 129, 3072 130 / 140, 8192 376 / 189).
//
// A set for all heads of a KV head takes two launches where the one-launch step's clusters run in rounds or lie unevenly on the
// SMs: the score stream shares every sequence's tokens out to all SMs, and all sets are selected at once.  Batch 12, 32 / 8 heads,
// 40-60 K, 256 rows 83.4 -> 64.2 us, 4 K in caches of 64 K 40.6 -> 22.8; 3-28 K on pages of 64, 512 rows 46.7 -> 38.0; batch 32 at 16-28 K
// 102 -> 80; batch 16 at 3-7 K 27.3 -> 24.8.  Resident clusters with an SM to each CTA are faster (batch 8 at 57 K 52 / 57, batch 4 at
// 60-120 K 47 / 53).  The lines are drawn through 12000 pairs of both routes (60 to 400 sets, 1 to 8 heads, 4 to 64 FCs, 2 K to 128 K
// full and a quarter full, 64 to 1024 rows, contiguous and paged; times of one launch over times of two, mean and worst twentieth):
//   - Clusters of one CTA end by themselves, two to an SM, and one's attention runs beside the other's stream.  Lists of up to 256
//     repay the second launch (1.29, 1.08), of 512 too (1.19, 1.01), of 1024 not (1.07, 0.89; in rounds 0.99, 0.86).
//   - Larger ones: up to 512 rows 1.41, 1.12, and 1024 up to two sets to an SM (1.30, 1.06; beyond 1.04, 0.92).
//   - Few sets (long rows, whose clusters of eight run in rounds) leave SMs idle while each CTA selects a whole row for itself: 16 sets,
//     128 rows 1.54, 1.33, 256 1.10, 0.90, 512 0.94, 0.73; 24 sets, 256 rows 1.34, 1.15, 512 1.18, 1.05, 1024 0.90, 0.81; 40 sets, 1024 rows
//     1.24, 0.94; 48 sets 1.26, 1.03 (3800 pairs of 16 to 72 sets).
//   - A single round that fills four fifths of the SMs or more leaves little to even out, and the other route attends long lists with
//     a CTA to a set, of half the threads beyond a set to an SM: from 256 rows and 8 K to each CTA of a cluster 1.08, 0.90, full caches
//     alone 1.01, 0.87 (256 sets of 15 K, 512 rows 70 / 82; 136 of 21 K, 1024 rows 60 / 69); 1.26, 1.05 below.  Not so with large
//     proxies (24 FCs and more 1.10, 0.97), whose stream decides.
static bool two_launches(fasa_ctx* ctx, const void* k_cache, int n_sel_max, const void* workspace) {
  const fasa_config_t& c = ctx->cfg;
  const long long sets = (long long)c.batch * ctx->n_sets;
  if (workspace == nullptr || !two_launches_possible(ctx) || n_sel_max > (sets <= ctx->n_sm ? 3072 : 2048)) return false;
  if (!set_per_head(ctx)) {
    const int cs = ctx->step_cs;
    const bool full = sets <= ctx->step_resident && 5 * sets >= 4ll * ctx->step_resident && c.n_dom <= 20;
    const long long most = std::min(cs == 1 || sets > 2ll * ctx->n_sm ? 512ll : 1024ll, 24 * (sets - 8));
    if (n_sel_max > most || 8ll * n_sel_max > c.max_len || (full && n_sel_max >= 256 * cs && c.max_len > 8192 * cs)) return false;
    return !(c.page_size == 0 && fasa_on_host(k_cache));
  }
  if (ctx->group < 4 ? n_sel_max > 1024 : sets < 96 && n_sel_max > 512) return false;
  if (16ll * n_sel_max > c.max_len && c.max_len > (ctx->group > 4 ? 8192 : 4096)) return false;
  return !(c.page_size == 0 && fasa_on_host(k_cache));
}

// A workspace that is not 256-byte aligned is refused where the list is one for the split-K kernel, and goes unused by steps
// that can do without: one launch.
static bool usable_workspace(const fasa_ctx* ctx, int n_sel_max, void** workspace) {
  if (((uintptr_t)*workspace & 255) == 0) return true;
  *workspace = nullptr;
  return fasa_full_probabilities(ctx, n_sel_max);
}

// The groups whose maxima the first half takes: those that suit a row of max_len.
static int stream_group_shift(const fasa_ctx* ctx, int budget) {
  const long long n = ctx->cfg.max_len, k = budget > 0 ? budget : ((long long)-budget * n + 999) / 1000;
  return sel_group_shift((int)n, (int)(k < n ? k : n), 16386);
}

static int32_t two_launch_step(fasa_ctx* ctx, const void* q, const void* k_new, const void* v_new, void* k_cache, void* v_cache,
                               void* proxy_k, const int32_t* seq_lens, int32_t budget, int32_t n_sel_max, float* scores,
                               int32_t* idx, int32_t* n_sel, float* out, float* lse, void* workspace, float* out_mirror,
                               cudaStream_t stream) {
  const fasa_ws w = ws_layout(ctx);
  fasa_stream_args a{};
  a.q = q; a.proxy_k = proxy_k; a.seq_lens = seq_lens;
  a.scores = scores ? scores : (float*)((char*)workspace + w.scores);
  a.maxima.gm = (float*)((char*)workspace + w.gm);
  a.maxima.gs = stream_group_shift(ctx, budget);
  a.maxima.stride = fasa_stream_gm_stride(ctx);
  a.k_new = k_new; a.v_new = v_new; a.k_cache = k_cache; a.v_cache = v_cache;
  int32_t st = fasa_stream_launch(ctx, a, stream);
  if (st != FASA_OK) return st;
  // (a probability keeps as many bits as on the route that this one replaces)
  const bool full_p = fasa_full_probabilities(ctx, n_sel_max) || (!set_per_head(ctx) && !fasa_attend_separately(ctx, n_sel_max, workspace));
  return fasa_select_attend_launch(ctx, q, k_cache, v_cache, a.scores, a.maxima.gm, a.maxima.gs, seq_lens, budget, n_sel_max, idx, n_sel, out, lse,
                                   out_mirror, k_new != nullptr, full_p, stream);
}

// What fasa_fc_score, fasa_topk and fasa_sparse_decode_attn require of the arguments they share
// with the composite calls.
static bool three_kernel_args_ok(const fasa_ctx* ctx, const void* q, const void* k_cache, const void* v_cache,
                                 const void* proxy_k, const float* scores, const void* workspace) {
  return scores && workspace && fasa_pages_ready(ctx) && !((uintptr_t)proxy_k & 15) && !((uintptr_t)q & 15) &&
         !((uintptr_t)scores & 3) && !((uintptr_t)k_cache & 15) && !((uintptr_t)v_cache & 15) &&
         !((uintptr_t)workspace & 255);
}

extern "C" int32_t fasa_decode_step(fasa_ctx_t* ctx, const void* q, const void* k_cache,
                                    const void* v_cache, const void* proxy_k,
                                    const int32_t* seq_lens, int32_t budget, int32_t n_sel_max,
                                    float* scores, int32_t* idx, int32_t* n_sel, float* out,
                                    float* lse, void* workspace, void* stream) {
  if (!ctx || !q || !k_cache || !v_cache || !proxy_k || !seq_lens || !idx || !n_sel || !out ||
      budget == 0 || budget < -1000 || n_sel_max <= 0)
    return FASA_ERR_INVALID_ARG;
  if (ctx->use_fused && ctx->fused_step_ok && ctx->fused_cs > 0) {
    if (((uintptr_t)proxy_k & 15) || ((uintptr_t)q & 15) || ((uintptr_t)k_cache & 15) ||
        ((uintptr_t)v_cache & 15) || (scores && ((uintptr_t)scores & 3)))
      return FASA_ERR_INVALID_ARG;
    if (!fasa_pages_ready(ctx)) return FASA_ERR_INVALID_ARG;
    if (!usable_workspace(ctx, n_sel_max, &workspace)) return FASA_ERR_INVALID_ARG;
    if (two_launches(ctx, k_cache, n_sel_max, workspace))
      return two_launch_step(ctx, q, nullptr, nullptr, const_cast<void*>(k_cache), const_cast<void*>(v_cache), const_cast<void*>(proxy_k),
                             seq_lens, budget, n_sel_max, scores, idx, n_sel, out, lse, workspace, nullptr, (cudaStream_t)stream);
    if (fasa_attend_separately(ctx, n_sel_max, workspace)) {
      int32_t st2 = fasa_fused_launch(ctx, q, k_cache, v_cache, proxy_k, seq_lens, budget, n_sel_max, scores,
                                      idx, n_sel, out, lse, nullptr, nullptr, (cudaStream_t)stream, false);
      if (st2 != FASA_OK) return st2;
      bool mirrored;
      return fasa_sparse_attn_mirrored(ctx, q, k_cache, v_cache, idx, n_sel, n_sel_max, out, lse, workspace, (cudaStream_t)stream,
                                       nullptr, &mirrored, fasa_full_probabilities(ctx, n_sel_max));
    }
    return fasa_fused_launch(ctx, q, k_cache, v_cache, proxy_k, seq_lens, budget, n_sel_max, scores,
                             idx, n_sel, out, lse, nullptr, nullptr, (cudaStream_t)stream);
  }
  // three kernels: everything any of them would refuse is refused before the first is enqueued
  if (!three_kernel_args_ok(ctx, q, k_cache, v_cache, proxy_k, scores, workspace)) return FASA_ERR_INVALID_ARG;
  int32_t st = fasa_fc_score(ctx, q, proxy_k, seq_lens, scores, stream);
  if (st != FASA_OK) return st;
  st = fasa_topk(ctx, scores, seq_lens, budget, n_sel_max, idx, n_sel, workspace, stream);
  if (st != FASA_OK) return st;
  return fasa_sparse_decode_attn(ctx, q, k_cache, v_cache, idx, n_sel, n_sel_max, out, lse,
                                 workspace, stream);
}

// out_mirror (nullable): device-accessible second destination of `out`; *mirrored tells whether
// the path taken wrote it.
static int32_t append_decode_step_impl(fasa_ctx_t* ctx, const void* q, const void* k_new,
                                       const void* v_new, void* k_cache, void* v_cache,
                                       void* proxy_k, int32_t* seq_lens, int32_t budget,
                                       int32_t n_sel_max, float* scores, int32_t* idx,
                                       int32_t* n_sel, float* out, float* lse, void* workspace,
                                       void* stream, float* out_mirror, bool* mirrored) {
  *mirrored = false;
  if (!ctx || !q || !k_new || !v_new || !k_cache || !v_cache || !proxy_k || !seq_lens || !idx ||
      !n_sel || !out || budget == 0 || budget < -1000 || n_sel_max <= 0)
    return FASA_ERR_INVALID_ARG;
  if (ctx->use_fused && ctx->fused_step_ok && ctx->fused_cs > 0) {
    if (((uintptr_t)proxy_k & 15) || ((uintptr_t)q & 15) || ((uintptr_t)k_cache & 15) ||
        ((uintptr_t)v_cache & 15) || ((uintptr_t)k_new & 15) || ((uintptr_t)v_new & 15) ||
        (scores && ((uintptr_t)scores & 3)))
      return FASA_ERR_INVALID_ARG;
    if (!fasa_pages_ready(ctx)) return FASA_ERR_INVALID_ARG;
    if (!usable_workspace(ctx, n_sel_max, &workspace)) return FASA_ERR_INVALID_ARG;
    if (two_launches(ctx, k_cache, n_sel_max, workspace)) {
      *mirrored = out_mirror != nullptr;
      return two_launch_step(ctx, q, k_new, v_new, k_cache, v_cache, proxy_k, seq_lens, budget, n_sel_max, scores, idx, n_sel,
                             out, lse, workspace, out_mirror, (cudaStream_t)stream);
    }
    if (fasa_attend_separately(ctx, n_sel_max, workspace)) {
      int32_t st2 = fasa_fused_launch(ctx, q, k_cache, v_cache, proxy_k, seq_lens, budget, n_sel_max, scores,
                                      idx, n_sel, out, lse, k_new, v_new, (cudaStream_t)stream, false);
      if (st2 != FASA_OK) return st2;
      return fasa_sparse_attn_mirrored(ctx, q, k_cache, v_cache, idx, n_sel, n_sel_max, out, lse, workspace,
                                       (cudaStream_t)stream, out_mirror, mirrored, fasa_full_probabilities(ctx, n_sel_max));
    }
    *mirrored = out_mirror != nullptr;
    return fasa_fused_launch(ctx, q, k_cache, v_cache, proxy_k, seq_lens, budget, n_sel_max, scores,
                             idx, n_sel, out, lse, k_new, v_new, (cudaStream_t)stream, true, out_mirror);
  }
  // append + three kernels: the arguments of all four calls are checked before the cache grows,
  // so that a caller who repairs an argument and retries does not append the token twice
  if (!three_kernel_args_ok(ctx, q, k_cache, v_cache, proxy_k, scores, workspace) || ((uintptr_t)k_new & 15) ||
      ((uintptr_t)v_new & 15))
    return FASA_ERR_INVALID_ARG;
  int32_t st = fasa_kv_append(ctx, k_cache, v_cache, proxy_k, seq_lens, k_new, v_new, 1, stream);
  if (st != FASA_OK) return st;
  return fasa_decode_step(ctx, q, k_cache, v_cache, proxy_k, seq_lens, budget, n_sel_max, scores, idx,
                          n_sel, out, lse, workspace, stream);
}

extern "C" int32_t fasa_append_decode_step(fasa_ctx_t* ctx, const void* q, const void* k_new,
                                           const void* v_new, void* k_cache, void* v_cache,
                                           void* proxy_k, int32_t* seq_lens, int32_t budget,
                                           int32_t n_sel_max, float* scores, int32_t* idx,
                                           int32_t* n_sel, float* out, float* lse, void* workspace,
                                           void* stream) {
  bool mirrored;
  return append_decode_step_impl(ctx, q, k_new, v_new, k_cache, v_cache, proxy_k, seq_lens, budget, n_sel_max,
                                 scores, idx, n_sel, out, lse, workspace, stream, nullptr, &mirrored);
}

extern "C" int32_t fasa_select_step(fasa_ctx_t* ctx, const void* q, const void* k_new,
                                    const void* v_new, void* k_cache, void* v_cache, void* proxy_k,
                                    int32_t* seq_lens, int32_t budget, int32_t n_sel_max,
                                    float* scores, int32_t* idx, int32_t* n_sel, void* stream) {
  if (!ctx || !q || !k_cache || !v_cache || !proxy_k || !seq_lens || !idx || !n_sel || budget == 0 ||
      budget < -1000 || n_sel_max <= 0 || (k_new == nullptr) != (v_new == nullptr))
    return FASA_ERR_INVALID_ARG;
  if (!(ctx->use_fused && ctx->fused_step_ok && ctx->fused_cs > 0)) return FASA_ERR_UNSUPPORTED;
  if (((uintptr_t)proxy_k & 15) || ((uintptr_t)q & 15) || ((uintptr_t)k_cache & 15) || ((uintptr_t)v_cache & 15) ||
      ((uintptr_t)k_new & 15) || ((uintptr_t)v_new & 15) || (scores && ((uintptr_t)scores & 3)) ||
      !fasa_pages_ready(ctx))
    return FASA_ERR_INVALID_ARG;
  return fasa_fused_launch(ctx, q, k_cache, v_cache, proxy_k, seq_lens, budget, n_sel_max, scores, idx, n_sel,
                           nullptr, nullptr, k_new, v_new, (cudaStream_t)stream, false);
}

extern "C" int32_t fasa_stage_bytes(const fasa_ctx_t* ctx, size_t* out_bytes) {
  if (!ctx || !out_bytes) return FASA_ERR_INVALID_ARG;
  const fasa_config_t& c = ctx->cfg;
  size_t qb = fasa_align_up((size_t)c.batch * c.n_q_heads * FASA_HEAD_DIM * 2, 256);
  size_t kb = fasa_align_up((size_t)c.batch * c.n_kv_heads * FASA_HEAD_DIM * 2, 256);
  *out_bytes = qb + 2 * kb;
  return FASA_OK;
}

extern "C" int32_t fasa_decode_step_host(fasa_ctx_t* ctx, const void* q_host,
                                         const void* k_new_host, const void* v_new_host,
                                         void* dev_stage, void* k_cache, void* v_cache,
                                         void* proxy_k, int32_t* seq_lens, int32_t budget,
                                         int32_t n_sel_max, float* scores, int32_t* idx,
                                         int32_t* n_sel, float* out, float* out_host,
                                         void* workspace, void* stream) {
  if (!ctx || !q_host || !k_new_host || !v_new_host || !dev_stage || !out_host || !out)
    return FASA_ERR_INVALID_ARG;
  const fasa_config_t& c = ctx->cfg;
  cudaStream_t s = (cudaStream_t)stream;
  size_t q_bytes = (size_t)c.batch * c.n_q_heads * FASA_HEAD_DIM * 2;
  size_t kv_bytes = (size_t)c.batch * c.n_kv_heads * FASA_HEAD_DIM * 2;
  char* dq = (char*)dev_stage;
  char* dk = dq + fasa_align_up(q_bytes, 256);
  char* dv = dk + fasa_align_up(kv_bytes, 256);
  // Pinned (page-locked, mapped) host buffers need no copy call: where the step is a single wave
  // of one launch its kernel reads them in place (the few KB cross the host link inside the
  // launch); where it is several launches or several waves of CTAs, one small kernel first
  // brings all three to the staging area, so that no CTA's start waits on the link.  Anything
  // else is copied to the staging area with cudaMemcpyAsync.  The driver is asked about each
  // pointer in every call (see fasa_on_host; a buffer that is no longer pinned must not be touched by a kernel).
  auto mapped = [](const void* hp) -> void* {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, hp) == cudaSuccess) return at.type == cudaMemoryTypeHost ? at.devicePointer : nullptr;
    cudaGetLastError();
    return nullptr;
  };
  const void* mq = mapped(q_host);
  const void* mk = mapped(k_new_host);
  const void* mv = mapped(v_new_host);
  const bool all_mapped = mq && mk && mv && !((uintptr_t)mq & 15) && !((uintptr_t)mk & 15) && !((uintptr_t)mv & 15);
  // (a set per query head at 16 K, batch 1: every warp of the score stream would fetch its query over the link, 105 us against 45)
  const bool one_wave_one_launch = ctx->use_fused && ctx->fused_cs > 0 && !two_launches(ctx, k_cache, n_sel_max, workspace) &&
                                   !fasa_attend_separately(ctx, n_sel_max, workspace) &&
                                   (long long)c.batch * ctx->n_sets * ctx->fused_cs <= 2ll * ctx->n_sm;
  if (all_mapped && one_wave_one_launch) {
    dq = (char*)mq; dk = (char*)mk; dv = (char*)mv;
  } else if (all_mapped) {
    FASA_CUDA_TRY(ctx, fasa_stage_from_mapped(dq, mq, q_bytes, dk, mk, dv, mv, kv_bytes, s));
    ctx->launches += 1;
  } else {
    FASA_CUDA_TRY(ctx, cudaMemcpyAsync(dq, q_host, q_bytes, cudaMemcpyHostToDevice, s));
    FASA_CUDA_TRY(ctx, cudaMemcpyAsync(dk, k_new_host, kv_bytes, cudaMemcpyHostToDevice, s));
    FASA_CUDA_TRY(ctx, cudaMemcpyAsync(dv, v_new_host, kv_bytes, cudaMemcpyHostToDevice, s));
  }
  // A pinned out_host is written by the step's kernel itself (next to `out`), where the path
  // taken has a single kernel to do it; otherwise `out` is copied back.
  float* mo = (float*)mapped(out_host);
  if ((uintptr_t)mo & 3) mo = nullptr;
  bool mirrored = false;
  int32_t st = append_decode_step_impl(ctx, dq, dk, dv, k_cache, v_cache, proxy_k, seq_lens, budget, n_sel_max,
                                       scores, idx, n_sel, out, nullptr, workspace, stream, mo, &mirrored);
  if (st != FASA_OK) return st;
  size_t o_bytes = (size_t)c.batch * c.n_q_heads * FASA_HEAD_DIM * sizeof(float);
  if (!mirrored) FASA_CUDA_TRY(ctx, cudaMemcpyAsync(out_host, out, o_bytes, cudaMemcpyDeviceToHost, s));
  FASA_CUDA_TRY(ctx, cudaStreamSynchronize(s));
  return FASA_OK;
}
