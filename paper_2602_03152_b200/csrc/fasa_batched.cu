// Blocks of query tokens (q_len = T > 1 per sequence: speculative or multi-token decoding).
//
// The method is defined per query q_t (Sec. 4.1: S_t and T_t; Sec. 4.2, Eq. 6-7: the output of
// q_t), so a block of T queries is T decode steps that happen to read the same cache: query t of
// the block sits at cache position L - T + t (L = seq_lens[b] counts the block's own keys, already
// appended), sees the rows up to its own, and gets its own scores, index set and output.  What
// the T steps share is the proxy-K stream: scoring all of them is ONE pass over it, for every head of a set
//     S[T x L] = Q[T x 2F] . P^T[2F x L],
// whose heads are then summed (or their maximum taken), by the kernel of fasa_stream.cu: the block's queries are the rows of its
// products, two heads to one.
//
// Selection and attention of the block are those of fasa_topk and fasa_sparse_decode_attn over (sequence, query) pairs.
#include "fasa_common.cuh"
#include "fasa_stream.cuh"

namespace {

bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

}  // namespace

size_t fasa_block_maxima_bytes(const fasa_ctx* ctx) {
  return (size_t)ctx->cfg.batch * FASA_MAX_QLEN * ctx->cfg.n_kv_heads * fasa_stream_gm_stride(ctx) * sizeof(float);
}

static int32_t block_score(fasa_ctx_t* ctx, const void* q, const void* proxy_k, const int32_t* seq_lens, int32_t q_len, float* scores,
                           const fasa_row_maxima& m, cudaStream_t stream) {
  if (!ctx || !q || !proxy_k || !seq_lens || !scores || !fasa_pages_ready(ctx)) return FASA_ERR_INVALID_ARG;
  if (!aligned16(proxy_k) || ((uintptr_t)q & 1) || ((uintptr_t)scores & 3)) return FASA_ERR_INVALID_ARG;
  if (q_len < 1 || q_len > FASA_MAX_QLEN) return FASA_ERR_UNSUPPORTED;
  if ((long long)ctx->cfg.batch * q_len * ctx->n_sets > 65535) return FASA_ERR_UNSUPPORTED;
  fasa_stream_args a{};
  a.q = q; a.proxy_k = proxy_k; a.seq_lens = seq_lens; a.scores = scores; a.maxima = m; a.q_len = q_len;
  return fasa_stream_launch(ctx, a, stream);
}

extern "C" int32_t fasa_fc_score_batched(fasa_ctx_t* ctx, const void* q, const void* proxy_k,
                                         const int32_t* seq_lens, int32_t q_len, float* scores, void* stream) {
  return block_score(ctx, q, proxy_k, seq_lens, q_len, scores, fasa_row_maxima{}, (cudaStream_t)stream);
}

// TopK-I of every query of the block: rows (sequence, query, index set) of the score buffer,
// each with the length its query sees.
extern "C" int32_t fasa_topk_batched(fasa_ctx_t* ctx, const float* scores, const int32_t* seq_lens, int32_t q_len,
                                     int32_t budget, int32_t n_sel_max, int32_t* idx, int32_t* n_sel, void* stream) {
  if (!ctx || !scores || !seq_lens || !idx || !n_sel || budget == 0 || budget < -1000 || n_sel_max <= 0)
    return FASA_ERR_INVALID_ARG;
  if (q_len < 1 || q_len > FASA_MAX_QLEN) return FASA_ERR_UNSUPPORTED;
  if (!(ctx->fused_cs > 0)) return FASA_ERR_UNSUPPORTED;            // needs the cluster kernel's selection phases
  if ((long long)ctx->cfg.batch * q_len * ctx->n_sets > 65535) return FASA_ERR_UNSUPPORTED;
  return fasa_topk_row_launch(ctx, scores, seq_lens, budget, n_sel_max, idx, n_sel, q_len * ctx->n_sets,
                              ctx->cfg.n_sink, ctx->cfg.n_recent, (cudaStream_t)stream, q_len);
}

extern "C" int32_t fasa_decode_step_batched(fasa_ctx_t* ctx, const void* q, const void* k_cache, const void* v_cache,
                                            const void* proxy_k, const int32_t* seq_lens, int32_t q_len, int32_t budget,
                                            int32_t n_sel_max, float* scores, int32_t* idx, int32_t* n_sel, float* out,
                                            float* lse, void* workspace, void* stream) {
  if (!scores || !workspace) return FASA_ERR_INVALID_ARG;
  if (!ctx || !q || !k_cache || !v_cache || !idx || !n_sel || !out || !aligned16(q) || !aligned16(k_cache) ||
      !aligned16(v_cache) || ((uintptr_t)workspace & 255) || n_sel_max <= 0 || budget == 0 || budget < -1000)
    return FASA_ERR_INVALID_ARG;                                    // (everything the later calls would refuse)
  if (!(ctx->fused_cs > 0)) return FASA_ERR_UNSUPPORTED;
  const fasa_config_t& c = ctx->cfg;
  // Where the selection goes by group maxima, the scoring pass takes them from its registers: the selection then reads an
  // eighth of a row (or less) and the few groups that it looks at.  They lie in the workspace, which is free until attention
  // writes partial results there.  (320 rows of 40-65 K, 512 of each: 34.8 -> 23.8 us, and 3 us more to score.)
  const long long rows = (long long)c.batch * q_len * ctx->n_sets;
  fasa_row_maxima m;
  m.gm = (float*)workspace;
  m.gs = q_len >= 1 && q_len <= FASA_MAX_QLEN ? fasa_row_maxima_shift(ctx, budget, rows) : 0;
  m.stride = ((c.max_len >> m.gs) + 8) & ~3;
  size_t room = 0;
  if (fasa_workspace_bytes(ctx, n_sel_max, &room) != FASA_OK || (size_t)rows * m.stride * sizeof(float) > room) m.gs = 0;   // (many sets to a KV head)
  int32_t st = block_score(ctx, q, proxy_k, seq_lens, q_len, scores, m, (cudaStream_t)stream);
  if (st != FASA_OK) return st;
  st = m.gs > 0 ? fasa_topk_row_launch(ctx, scores, seq_lens, budget, n_sel_max, idx, n_sel, q_len * ctx->n_sets, c.n_sink, c.n_recent,
                                       (cudaStream_t)stream, q_len, nullptr, &m)
                : fasa_topk_batched(ctx, scores, seq_lens, q_len, budget, n_sel_max, idx, n_sel, stream);
  if (st != FASA_OK) return st;
  return fasa_sparse_decode_attn_batched(ctx, q, k_cache, v_cache, idx, n_sel, q_len, n_sel_max, out, lse, workspace, stream);
}
