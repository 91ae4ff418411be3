// Decode step in two launches, second half: TopK-I of every index set from its scores and group maxima
// (fasa_select.cuh), then exact attention over the selected rows (Sec. 4.2, Eq. 6-7), in one launch.
//
// A cluster of 1 to 8 CTAs serves an index set.  Every CTA selects for itself - the maxima and the few groups it
// looks at come from L2, which is cheaper than one CTA selecting and the others waiting for its list - and
// attends to its share of the list on tensor cores; the partial results merge through distributed shared
// memory, the launch's only cluster barrier.  The kernel waits for the first half by programmatic dependent
// launch, so its own start-up overlaps that kernel's tail.
#include "fasa_attn_core.cuh"
#include "fasa_cluster_merge.cuh"
#include "fasa_common.cuh"
#include "fasa_launch.cuh"
#include "fasa_select.cuh"
#include "fasa_stream.cuh"

namespace cg = cooperative_groups;

namespace {

struct SelAttnParams {
  const uint16_t* q;
  const uint16_t* k;
  const uint16_t* v;
  const float* scores;                    // [units][max_len]
  const float* gm;                        // [units][gm_stride]
  const int32_t* seq_lens;
  int32_t* idx;
  int32_t* n_sel;
  float* out;
  float* out_mirror;
  float* lse;
  int32_t* status;
  int32_t* seq_lens_w;                    // append: the lengths grow here
  int32_t* arrive;
  int append, batch;
  int n_q_heads, n_kv_heads, n_sets, group, max_len, n_sink, n_recent, budget, n_sel_max;   // group: query heads of a unit
  int gs, gm_stride;                      // groups of 1 << gs positions (0: no maxima)
  SelLayout lay;
  int idx_off;                            // of the CTA's share of the list in dynamic shared memory
  int64_t ksb, ksh, kst, vsb, vsh, vst;
  PageMap pm;
  float scale_log2;
  fasa_ksplit ks;                         // (unused: attn_load_query's general form)
};

template <int NT, bool PAGED, int TERMS>
__global__ void __launch_bounds__(NT, NT == 256 ? 2 : 1)
select_attend_kernel(const SelAttnParams p) {
  constexpr int WARPS = NT / 32;
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ SelShared sm;
  __shared__ ClusterMergeSmem s_merge;
  __shared__ int s_last;
  const int tid = threadIdx.x, lane = tid & 31;
  // (the merge writes into the peers' shared memory: each CTA says that it runs, and waits for that much at the end)
  cluster_arrive_running();
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks(), crank = (int)cluster.block_rank();
  const int u = blockIdx.y;
  const SelUnit su = sel_unit(u, p.n_sets, p.group, p.n_q_heads, p.n_kv_heads);
  // Before the first half has ended: its inputs alone, the lengths and the query, are read, and no result is written.  The
  // first half lets this kernel start after its own wait, so what is older than it is complete, and these loads take it
  // from L2: nothing says that an L1 line of that age is current before this kernel's own wait.  (The appended token's
  // length is stored below.)
  const int old_len = clamp_len(__ldcg(p.seq_lens + su.b), p.max_len, p.status);
  const int len = p.append && old_len < p.max_len ? old_len + 1 : old_len;
  uint32_t qb[8][2];
  attn_load_query<false, true>(qb, p, su, lane);
  sel_begin<NT>(sm);
  const SelPlan plan = sel_plan(len, p.budget, p.n_sink, p.n_recent, p.n_sel_max);
  // this CTA's share of the list
  const int a0 = (int)(((long long)plan.ktot * crank) / cs), a1 = (int)(((long long)plan.ktot * (crank + 1)) / cs);
  int32_t* s_idx = reinterpret_cast<int32_t*>(dsm + p.idx_off);
  int32_t* out_idx = p.idx + (int64_t)u * p.n_sel_max;
  auto take = [&](int rank, int pos) {
    if (rank >= a0 && rank < a1) {
      s_idx[rank - a0] = pos;
      out_idx[rank] = pos;
    }
  };
  SelRow<SelScores> row;
  row.src = SelScores{p.scores + (int64_t)u * p.max_len};
  row.lo = plan.lo;
  row.hi = plan.hi;
  row.k = plan.k;
  // (the maxima were taken in groups of the size that suits max_len; a short row may be better off whole)
  const int n_free = row.hi - row.lo;
  int gs = p.gs;
  if (gs > 0 && !(row.k > 0 && row.k < n_free && (long long)row.k * (gs == 3 ? 12 : 43) <= n_free)) gs = 0;
  pdl_wait_for_predecessor();
  pdl_release_successor();
  auto maxima = [&](float* gm, float& gm_lo, float& gm_hi) {
    sel_copy_maxima<NT>(gm, p.gm + (int64_t)u * p.gm_stride, row.lo >> gs, ((row.hi - 1) >> gs) + 1, gm_lo, gm_hi);
  };
  sel_row<NT>(row, gs, maxima, sm, dsm, p.lay, [&](int r, int pos) { take(plan.sink + r, pos); });
  for (int i = tid; i < plan.n_forced; i += NT) {
    int rank, pos;
    sel_forced(plan, i, &rank, &pos);
    take(rank, pos);
  }
  if (crank == 0 && tid == 0) {
    if (plan.clamped) atomicOr(p.status, FASA_DEV_NSEL_CLAMPED);
    p.n_sel[u] = plan.ktot;
  }
  __syncthreads();                                   // the list is complete, the selection's memory free
  if constexpr (PAGED) {
    // from here on as rows of the pool: a table entry is looked up once, not for each copy of a row's K and V (12 sequences of
    // 3-28 K on pages of 64, 512 rows: 18 -> 13 thousand cycles of attention)
#pragma unroll 4
    for (int i = tid; i < a1 - a0; i += NT) s_idx[i] = pool_row(p.pm, su.b, s_idx[i], p.status);
    __syncthreads();
  }
  float (*s_part)[kMergePartStride] = mma_part<WARPS>(dsm);
  attn_rows<WARPS, true, PAGED, false, false, TERMS>(p, su, su.b, qb, a0, a1, s_idx, dsm, [&](int gl) { return &s_part[gl][0]; });
  // append: every CTA of the launch has read the old length by the time that it arrives here; the last one stores the
  // new ones, below
  if (p.append && tid == 0) s_last = atomicAdd(p.arrive, 1) == (int)(gridDim.x * gridDim.y) - 1;
  __syncthreads();
  cluster_wait();
  if constexpr (TERMS == 3)
    cluster_merge_store<NT>(cluster, s_part, s_merge, p.group, su.q0, p.out, p.out_mirror, p.lse, [&](int g) {
      const int u = unit_again();
      const SelUnit s = sel_unit(u, p.n_sets, p.group, p.n_q_heads, p.n_kv_heads);
      ExactOutput<PAGED> e;
      e.q = p.q + (s.q0 + g) * FASA_HEAD_DIM;
      e.k = p.k + s.h * p.ksh + (PAGED ? 0 : s.b * p.ksb);
      e.v = p.v + s.h * p.vsh + (PAGED ? 0 : s.b * p.vsb);
      e.list = p.idx + (int64_t)u * p.n_sel_max;
      e.n = p.n_sel[u];
      e.status = p.status; e.pm = p.pm; e.ksb = p.ksb; e.kst = p.kst; e.vsb = p.vsb; e.vst = p.vst;
      e.b = s.b; e.max_len = p.max_len; e.scale_log2 = p.scale_log2;
      return e;
    });
  else   // (long lists go without: see fasa_attn.cu)
    cluster_merge_store<NT>(cluster, s_part, s_merge, p.group, su.q0, p.out, p.out_mirror, p.lse);
  if (p.append && tid < 32 && s_last) {
    if (tid == 0) *p.arrive = 0;
    for (int b = tid; b < p.batch; b += 32) {
      const int l = clamp_len(p.seq_lens_w[b], p.max_len, p.status);
      if (l == p.max_len) atomicOr(p.status, FASA_DEV_APPEND_FULL);
      p.seq_lens_w[b] = l < p.max_len ? l + 1 : l;
    }
  }
}

constexpr int kSelAttnMaxShare = 2048;    // rows of one CTA
constexpr int kSelAttnMaxLen = 262144;    // positions: groups of 8 up to 65536 listed, mask words, both in shared memory

// CTAs per index set.
int sel_attn_cluster(const fasa_ctx* ctx, int units, int n_sel_max) {
  int cs = 1;
  while (cs < 8 && units * cs * 2 <= ctx->n_sm && n_sel_max / (2 * cs) >= 32) cs *= 2;
  while (cs < 8 && (n_sel_max + cs - 1) / cs > kSelAttnMaxShare) cs *= 2;
  return cs;
}

}  // namespace

bool fasa_select_attend_ok(const fasa_ctx* ctx, int n_sel_max) {
  const int n = n_sel_max < ctx->cfg.max_len ? n_sel_max : ctx->cfg.max_len;
  return n <= 8 * kSelAttnMaxShare && ctx->cfg.max_len <= kSelAttnMaxLen;
}

int32_t fasa_select_attend_launch(fasa_ctx* ctx, const void* q, const void* k_cache, const void* v_cache, const float* scores,
                                  const float* gm, int gs, const int32_t* seq_lens, int32_t budget, int32_t n_sel_max,
                                  int32_t* idx, int32_t* n_sel, float* out, float* lse, float* out_mirror, bool append, bool full_p,
                                  cudaStream_t stream) {
  const fasa_config_t& c = ctx->cfg;
  SelAttnParams p;
  memset(&p, 0, sizeof(p));
  p.q = (const uint16_t*)q; p.k = (const uint16_t*)k_cache; p.v = (const uint16_t*)v_cache;
  p.scores = scores; p.gm = gm; p.seq_lens = seq_lens; p.idx = idx; p.n_sel = n_sel;
  p.out = out; p.out_mirror = out_mirror; p.lse = lse; p.status = ctx->d_status;
  p.append = append ? 1 : 0; p.batch = c.batch; p.arrive = ctx->d_arrive; p.seq_lens_w = const_cast<int32_t*>(seq_lens);
  p.n_q_heads = c.n_q_heads; p.n_kv_heads = c.n_kv_heads; p.n_sets = ctx->n_sets; p.group = ctx->sel_heads; p.max_len = c.max_len;
  p.n_sink = c.n_sink; p.n_recent = c.n_recent; p.budget = budget; p.n_sel_max = n_sel_max;
  p.gs = gs; p.gm_stride = fasa_stream_gm_stride(ctx);
  p.ksb = c.k_stride_b; p.ksh = c.k_stride_h; p.kst = c.k_stride_t;
  p.vsb = c.v_stride_b; p.vsh = c.v_stride_h; p.vst = c.v_stride_t;
  p.pm = fasa_page_map(ctx);
  p.scale_log2 = c.softmax_scale * 1.4426950408889634f;
  const int units = c.batch * ctx->n_sets;
  const int n_upper = n_sel_max < c.max_len ? n_sel_max : c.max_len;
  const int cs = sel_attn_cluster(ctx, units, n_upper);
  const int share_cap = (n_upper + cs - 1) / cs + 1;
  const bool wide = units * cs <= ctx->n_sm;
  p.lay.gm_cap = gs == 0 ? 4 : (c.max_len >> gs) + 2;
  // (the bins of about k groups are kept; a row that is taken whole keeps as many as there is room for)
  const int need = (c.max_len + 63) & ~31, room = 2 * p.lay.gm_cap > (wide ? 24576 : 12288) ? 2 * p.lay.gm_cap : (wide ? 24576 : 12288);
  p.lay.uni_cap = need < room ? need : room;
  p.lay.word_cap = (c.max_len >> 5) + 2;
  const size_t stage = wide ? sizeof(MmaSmem<16, 3>) : sizeof(MmaSmem<8, 3>);
  p.idx_off = (int)fasa_align_up(stage > (size_t)p.lay.bytes() ? stage : (size_t)p.lay.bytes(), 16);
  const size_t smem = (size_t)p.idx_off + (size_t)share_cap * 4;
  auto go = [&](auto kernel, int threads) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 208 * 1024);
    if (e != cudaSuccess) return e;
    return launch_after_predecessor(kernel, dim3((unsigned)cs, (unsigned)units), dim3((unsigned)threads), smem, stream, cs, p);
  };
  const bool paged = c.page_size > 0;
  ctx->launches += 1;
  auto form = [&](auto terms_tag) -> cudaError_t {
    constexpr int T = decltype(terms_tag)::value;
    if (wide) return paged ? go(select_attend_kernel<512, true, T>, 512) : go(select_attend_kernel<512, false, T>, 512);
    return paged ? go(select_attend_kernel<256, true, T>, 256) : go(select_attend_kernel<256, false, T>, 256);
  };
  FASA_CUDA_TRY(ctx, full_p ? form(std::integral_constant<int, 3>{}) : form(std::integral_constant<int, 2>{}));
  return FASA_OK;
}
