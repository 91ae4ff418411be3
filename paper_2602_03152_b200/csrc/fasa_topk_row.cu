// TopK-I (Sec. 4.1) for score rows, one CTA per row: one pass over the row for the maxima of its groups
// (4 bytes per position, the only time the whole row is read), then the selection of fasa_select.cuh.
//
// The pass is a stream of 16-byte loads with one max per score; what follows works on a few thousand
// values and costs instructions and block barriers.  Measured (ncu), against a select that histograms
// every key: 320 rows of 40-65 K positions, 512 of each: 67 -> 34 us; 2080 rows of 24 K, 256 of each:
// 200 -> 72 us (44 M warp instructions, a fifth of what the histogram form issued).
#include "fasa_common.cuh"
#include "fasa_launch.cuh"
#include "fasa_score_core.cuh"
#include "fasa_select.cuh"

namespace {

struct RowParams {
  const float* scores;                  // [rows][max_len]; CALIB: [samples][stride], the full-head scores
  fasa_calib_rows calib;                // (CALIB) the other 64 rows of a sample
  const int32_t* seq_lens;
  int32_t* idx;
  int32_t* n_sel;
  int32_t* status;
  int rows_per_seq, max_len, n_sink, n_recent, budget, n_sel_max, q_len;
  SelLayout lay;
  fasa_row_maxima given;                // (MAXIMA) what the scoring pass has left
};

// One row: unit u = blockIdx.x of sequence b.
template <int NT, bool MAXIMA, typename Src>
__device__ __forceinline__ void topk_row(const RowParams& p, const Src& src, int b, SelShared& sm, unsigned char* rsm) {
  const int tid = threadIdx.x, lane = tid & 31, u = blockIdx.x;
  int len_raw = p.seq_lens[b];
  if (p.q_len > 1) {                                // rows of a block of queries: query t sees q_len - 1 - t fewer positions
    const int t = (u % p.rows_per_seq) / (p.rows_per_seq / p.q_len);
    if (len_raw >= 0 && len_raw <= p.max_len) len_raw = max(0, len_raw - (p.q_len - 1 - t));
  }
  const int len = clamp_len(len_raw, p.max_len, p.status);
  const SelPlan plan = sel_plan(len, p.budget, p.n_sink, p.n_recent, p.n_sel_max);
  if (tid == 0) {
    if (plan.clamped) atomicOr(p.status, FASA_DEV_NSEL_CLAMPED);
    p.n_sel[u] = plan.ktot;
  }
  SelRow<Src> row;
  row.src = src;
  row.lo = plan.lo;
  row.hi = plan.hi;
  row.k = plan.k;
  int gs = row.k > 0 && row.k < row.hi - row.lo ? sel_group_shift(row.hi - row.lo, row.k, p.lay.gm_cap) : 0;
  // (given maxima are of the groups that suit max_len, which a short row may do without)
  const bool given = MAXIMA && gs > 0 && (long long)row.k * (p.given.gs == 3 ? 12 : 43) <= row.hi - row.lo;
  if (given) gs = p.given.gs;
  auto maxima = [&](float* gm, float& gm_lo, float& gm_hi) {
    if (given) {
      sel_copy_maxima<NT>(gm, p.given.gm + (int64_t)u * p.given.stride, row.lo >> gs, ((row.hi - 1) >> gs) + 1, gm_lo, gm_hi);
      return;
    }
    // A thread takes eight consecutive positions: their maximum needs no other lane (groups of 32: two shuffles).
    const int g0 = row.lo >> gs, first = g0 << gs;
    const bool vec_ok = src.aligned();
    constexpr int UNR = 2, STEP = NT * 8;
    for (int w0 = first + (tid - lane) * 8; w0 < row.hi; w0 += STEP * UNR) {       // uniform over the warp
      const int i0 = w0 + lane * 8;
      float m[UNR];
      if (vec_ok && w0 >= row.lo && w0 + STEP * (UNR - 1) + 256 <= row.hi) {        // plain positions only
#pragma unroll
        for (int j = 0; j < UNR; ++j) m[j] = src.max8(i0 + j * STEP);
      } else {
#pragma unroll
        for (int j = 0; j < UNR; ++j) {
          m[j] = -INFINITY;
          for (int e = 0; e < 8; ++e) {
            const int i = i0 + j * STEP + e;
            if (i >= row.lo && i < row.hi) m[j] = max_nan(m[j], src(i));
          }
        }
      }
#pragma unroll
      for (int j = 0; j < UNR; ++j) {
        const int i = i0 + j * STEP;
        if (gs == 5) {
          m[j] = max_nan(m[j], __shfl_xor_sync(0xffffffffu, m[j], 1));
          m[j] = max_nan(m[j], __shfl_xor_sync(0xffffffffu, m[j], 2));
        }
        if (i < row.hi && (gs == 3 || (lane & 3) == 0)) {
          gm[(i >> gs) - g0] = m[j];
          gm_lo = fminf(gm_lo, m[j]);
          gm_hi = max_nan(gm_hi, m[j]);
        }
      }
    }
  };
  int32_t* out = p.idx + (int64_t)u * p.n_sel_max;
  sel_row<NT>(row, gs, maxima, sm, rsm, p.lay, [&](int r, int pos) { out[plan.sink + r] = pos; });
  for (int i = tid; i < plan.n_forced; i += NT) {
    int rank, pos;
    sel_forced(plan, i, &rank, &pos);
    if (rank < plan.ktot) out[rank] = pos;
  }
}

// CALIB: row r < 64 of a sample (sequence, query head) is FC r alone, computed from the channel pairs as it is read, row
// 64 the full head: the 64 rows of the four to eight query heads of a KV head share 4 bytes per position and FC
// instead of having 4 bytes each.
template <int NT, bool CALIB, bool MAXIMA = false>
__global__ void __launch_bounds__(NT, 1024 / NT)
topk_row_kernel(const RowParams p) {
  extern __shared__ __align__(16) unsigned char rsm[];
  __shared__ SelShared sm;
  sel_begin<NT>(sm);
  pdl_wait_for_predecessor();
  pdl_release_successor();
  const int b = blockIdx.x / p.rows_per_seq;
  if constexpr (CALIB) {
    const int sample = blockIdx.x / 65, fc = blockIdx.x - 65 * sample;
    if (fc < 64) {
      const int kv = sample / p.calib.group;        // (sequence, KV head)
      const uint16_t* q = p.calib.q + (int64_t)sample * FASA_HEAD_DIM;
      SelPairs src;
      src.p = p.calib.pairs + ((int64_t)kv * 64 + fc) * p.calib.stride;
      src.q0 = bf16_bits_to_f32(q[p.calib.pairing == 0 ? fc : 2 * fc]);
      src.q1 = bf16_bits_to_f32(q[p.calib.pairing == 0 ? fc + 64 : 2 * fc + 1]);
      topk_row<NT, false>(p, src, b, sm, rsm);
    } else {
      topk_row<NT, false>(p, SelScores{p.scores + (int64_t)sample * p.calib.stride}, b, sm, rsm);
    }
  } else {
    topk_row<NT, MAXIMA>(p, SelScores{p.scores + (int64_t)blockIdx.x * p.max_len}, b, sm, rsm);
  }
}

}  // namespace

// Longest row the kernel takes: its group maxima and their list must fit in shared memory.
static constexpr int kTopkRowMaxLen = 524288;

bool fasa_topk_row_ok(const fasa_ctx* ctx) { return ctx->cfg.max_len <= kTopkRowMaxLen; }

// A cluster per row keeps the row's keys in shared memory and selects by their bits, whatever their distribution.  One CTA per
// row pays for every position that it looks at again, the more, the larger the selection.  Measured (us, clusters / one CTA, budgets
// of 64, 256, 1024, 4096):
//   8 to 16 rows     of 12 K 7.6 / 7.3, 8.0 / 8.6, 8.4 / 13.5 (of 8 K, after their scoring, 512: 12.9 / 12.2)
//   32 rows          of 32 K 10.2 / 9.4, 11.3 / 9.8, 11.9 / 14.3, 13.8 / 22.6; of 128 K 15.0 / 13.9, 15.7 / 16.7, 16.6 / 30.8, 17.6 / 69
//   64 rows          of 32 K 11.7 / 9.4, 13.1 / 9.9, 12.9 / 14.4, 15.2 / 22.7; of 64 K 15 / 12, 16 / 12, 17 / 15, 18 / 31; of 128 K 29 / 14,
//                    30 / 17, 33 / 31, 33 / 73
//   74 rows          of 32 K 18 / 10, 19 / 10, 20 / 14, 24 / 23; of 50 K 20 / 11, 22 / 12, 23 / 14, 26 / 31; of 128 K 37 / 14, 40 / 17, 43 / 31, 44 / 73
// Rows that are not aligned are read 4 bytes at a time by one CTA: scoring and selection of 40 rows of 50001, 256 of each, 33.2 / 34.5,
// 1024 33.8 / 37.8; 48 of 119943, 512, with its attention 63.5 / 69.8; 72 of 65535, 2048: 46.2 / 48.4.
// One CTA's bins are spread evenly over the scores, and outliers can spoil that (they are clamped into the last bin where the rest is
// far below): one score in 500 thirty times as large, 24 to 32 rows beyond 64 K, 64 of each, 13 / 18 to 14 / 21 us; sums over seven heads
// with outlier channels do it too (24 rows of 100 K, 64: 13.5 / 21.8), so rows of that length go to clusters although scores that are
// spread evenly would take 14 / 13.
// Where nothing narrows a row down (96 rows at 65 K, 12387 of each: 35 / 48 us; 320 rows: 102 / 172; 320 rows at 16 K, 2048 of each:
// 29 / 42) a row held in shared memory is read once, here three times.
// block: of a block of queries; given: the scoring pass has left the rows' maxima, which spares the pass over the row (blocks of queries, 64 rows of 120 K,
// 128: 64 us a block by clusters, 48; 16 rows of 64 K 34.7 / 31.5; 16 K, 1024: 31.4 / 35.5; 32 rows of 120 K, 512: 43.0 / 45.8).
static bool topk_by_clusters(const fasa_ctx* ctx, long long n_rows, int budget, bool block, bool given) {
  const fasa_config_t& c = ctx->cfg;
  const int k = budget > 0 ? budget : (int)(((long long)-budget * c.max_len + 999) / 1000);
  const bool narrowed = sel_group_shift(c.max_len, k < c.max_len ? k : c.max_len, 16386) > 0, whole = !narrowed && c.max_len > 8192;
  if (ctx->topk_rows) return false;
  if (whole && ctx->fused_cs > 0) return true;
  if (ctx->fused_cs <= 1) return false;
  // up to 16, 32, 64 and 74 of 148 SMs' rows
  const bool r16 = n_rows <= 16, r32 = 9 * n_rows <= 2ll * ctx->n_sm, r64 = 9 * n_rows <= 4ll * ctx->n_sm, r74 = 2 * n_rows <= ctx->n_sm;
  const bool odd = (c.max_len & 3) != 0;
  const bool few = r16 && c.max_len >= 2048 && (c.max_len > 16384 || (k >= 128 && (narrowed || whole) && (n_rows <= 12 || c.max_len > 8192)));
  const bool large = r32   ? c.max_len > 8192 && (k >= 1024 || (c.max_len > 32768 && k >= 256) || c.max_len > 65536)
                     : r64 ? c.max_len > 8192 && (k >= 2048 || (k >= 1024 && (c.max_len <= 32768 || c.max_len > 65536)) || (odd && k >= 256 && c.max_len > 32768))
                           : r74 && (c.max_len > 65536 ? k >= 2048 : c.max_len > 32768 && k >= (odd ? 2048 : 4096));
  if (given && !(k >= 1024 && (r32 || (r74 && c.max_len <= 32768))) && !(r32 && k >= 512 && c.max_len > 65536)) return false;
  // (a block's rows have smaller clusters of their own)
  return few || large || (block && r74 && k >= 1024 && c.max_len > 8192 && c.max_len <= 32768);
}

// Group maxima that fit: groups of 8 up to 65536 positions, groups of 32 beyond (16 KB + 8 KB to 64 KB + 32 KB of shared memory).
static int row_maxima_cap(const fasa_ctx* ctx) {
  const int by32 = (ctx->cfg.max_len >> 5) + 2, by8 = (ctx->cfg.max_len >> 3) + 2;
  return by32 > 8194 ? by32 : (by8 < 8194 ? by8 : 8194);
}

int fasa_row_maxima_shift(const fasa_ctx* ctx, int budget, long long n_rows) {
  const long long n = ctx->cfg.max_len, k = budget > 0 ? budget : ((long long)-budget * n + 999) / 1000;
  if (!fasa_topk_row_ok(ctx) || topk_by_clusters(ctx, n_rows, budget, true, true)) return 0;
  return sel_group_shift((int)n, (int)(k < n ? k : n), row_maxima_cap(ctx));
}

int32_t fasa_topk_row_launch(fasa_ctx* ctx, const float* scores, const int32_t* seq_lens, int32_t budget,
                             int32_t n_sel_max, int32_t* idx, int32_t* n_sel, int rows_per_seq, int n_sink,
                             int n_recent, cudaStream_t stream, int q_len, const fasa_calib_rows* calib, const fasa_row_maxima* given) {
  const fasa_config_t& c = ctx->cfg;
  if (!calib && !given && topk_by_clusters(ctx, (long long)c.batch * rows_per_seq, budget, rows_per_seq > ctx->n_sets, false))
    return fasa_topk_cluster_launch(ctx, scores, seq_lens, budget, n_sel_max, idx, n_sel, rows_per_seq, n_sink, n_recent, stream, q_len);
  RowParams p;
  p.scores = scores; p.seq_lens = seq_lens; p.idx = idx; p.n_sel = n_sel; p.status = ctx->d_status;
  p.rows_per_seq = rows_per_seq; p.max_len = c.max_len; p.n_sink = n_sink; p.n_recent = n_recent;
  p.budget = budget; p.n_sel_max = n_sel_max; p.q_len = q_len;
  p.calib = calib ? *calib : fasa_calib_rows{};
  p.given = given ? *given : fasa_row_maxima{};
  p.lay.gm_cap = row_maxima_cap(ctx);
  const int rows = c.batch * rows_per_seq;
  p.lay.word_cap = (c.max_len >> 5) + 2;
  const int room = 2 * p.lay.gm_cap > 8192 ? 2 * p.lay.gm_cap : 8192, need = (c.max_len + 63) & ~31;
  p.lay.uni_cap = need < room ? need : room;
  auto go = [&](auto kernel, int threads) -> int32_t {
    FASA_CUDA_TRY(ctx, cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    ctx->launches += 1;
    FASA_CUDA_TRY(ctx, launch_after_predecessor(kernel, dim3((unsigned)rows), dim3((unsigned)threads), (size_t)p.lay.bytes(), stream, 0, p));
    return FASA_OK;
  };
  // Threads: a row ends soonest with many where it is long, and all rows should be resident: rows of 128 K, 256 of each, 17 us with
  // 1024 threads, 20 with 512, 30 with 256; 160 of 32 K 18 / 13 / 13; 320 of 64 K, two rounds of 512 threads 27.5, one of 256 23.9; 512 of
  // 16 K 33 / 20 / 15.
  if (calib) return go(topk_row_kernel<256, true>, 256);
  if (given) {
    if (rows <= ctx->n_sm && c.max_len > 16384) return go(topk_row_kernel<1024, false, true>, 1024);
    if (rows <= 2 * ctx->n_sm) return go(topk_row_kernel<512, false, true>, 512);
    return go(topk_row_kernel<256, false, true>, 256);
  }
  if (rows <= ctx->n_sm && c.max_len > 16384) return go(topk_row_kernel<1024, false>, 1024);
  if (rows <= 2 * ctx->n_sm) return go(topk_row_kernel<512, false>, 512);
  return go(topk_row_kernel<256, false>, 256);
}
