// Blocks of query tokens (q_len = T > 1 per sequence: speculative or multi-token decoding).
//
// The method is defined per query q_t (Sec. 4.1: S_t and T_t; Sec. 4.2, Eq. 6-7: the output of
// q_t), so a block of T queries is T decode steps that happen to read the same cache: query t of
// the block sits at cache position L - T + t (L = seq_lens[b] counts the block's own keys, already
// appended), sees the rows up to its own, and gets its own scores, index set and output.  What
// the T steps share is the proxy-K stream: scoring all of them is ONE pass over it,
//     S[L x (G T)] = P[L x 2F] . Q[2F x (G T)],
// a matrix product with up to 64 columns, after which the G columns of each query are reduced.
//
// block_score_kernel: what bounds it is the stream (the proxy once, 4 T bytes of scores per token), so the rest is arranged to
// take few instructions and no barrier between warps.  The proxy lies in HBM in the fragment order of mma.m16n8k16's operand A,
// 16 tokens by 16 channels; the same registers are two operands B, of tokens 0-7 (words 0, 2) and 8-15 (words 1, 3).  So the
// query is operand A: rows 0-7 are the T queries of one head, rows 8-15 those of the next, whose scores then meet in one
// thread.  The heads are reduced without a shuffle; a lane holds two consecutive tokens of one query, and eight tokens' maximum
// is two shuffles away.  A warp goes from its loads to its stores alone.
//
// Measured (batch 8, 32 / 8 heads, 40-65 K, 16 FCs, T = 5): 46.4 us, 6.1 TB/s.  Before, tcgen05.mma with both operands in shared
// memory took 71.8 us: the proxy had to be scattered into its operand layout, four warps met at a barrier for each 128 tokens,
// 250 instructions per 32 tokens and warp against 146 here.  The tensor pipe is no limit: 16 products of 8 cycles per 32 tokens
// and scheduler, a quarter of the time that the tokens take to arrive.  At 8 FCs and five heads a set 59.8 -> 34.2 us, 32 FCs
// 50.4 -> 40.8, 64 FCs 53.5 -> 44.6, 12 FCs (no whole blocks) 86 -> 46.7; the same bits throughout.
//
// Selection and attention of the block are those of fasa_topk and fasa_sparse_decode_attn over (sequence, query) pairs.
#include <algorithm>
#include <type_traits>

#include "fasa_common.cuh"
#include "fasa_launch.cuh"
#include "fasa_score_core.cuh"
#include "fasa_select.cuh"

namespace {

constexpr int kBlockThreads = 256;
constexpr int kBlockWarps = kBlockThreads / 32;
constexpr int kBlockMaxTiles = 1024;          // proxy tiles of a CTA at most (its page entries lie in shared memory)
// Tiles that a warp holds in registers (positions are finished 32 at a time), and CTAs on an SM.  About 32 KB of loads in flight
// on an SM are enough; more CTAs with fewer tiles each beat fewer with more (batch 8, 40-65 K, 16 FCs, 5 queries: 47 us with 4
// CTAs of two tiles a warp, 51 with 2 or 3 of four).
template <int KB, int HP>
struct BlockShape {
  static constexpr int tiles = KB == 1 ? 4 : (KB == 8 ? 1 : 2);
  static constexpr int step = tiles < 2 ? 2 : tiles;        // tiles per warp and iteration
  static constexpr int ctas = KB <= 2 && HP <= 2 ? 4 : 3;
};

struct BlockParams {
  const uint16_t* q;            // [batch][q_len][n_q_heads][128]
  const unsigned char* proxy;
  const int32_t* seq_lens;
  const int16_t* chan;
  float* scores;                // [batch][q_len][n_sets][max_len]
  float* gm;                    // gs > 0: maxima of groups of 1 << gs positions, a row of gm_stride per score row
  int32_t* status;
  int n_q_heads, n_kv_heads, n_sets, group, max_len, chunks, q_len, tiles_per_cta, max_reduce;
  int gs, gm_stride, n_sink, n_recent;
  PageMap pm;
};

// (volatile: read where it is used, not kept in registers around the loop)
__device__ __forceinline__ uint4 lds_u4(const void* p) {
  uint4 r;
  asm volatile("ld.volatile.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"((uint32_t)__cvta_generic_to_shared(p)));
  return r;
}
// c (FIRST: a new one, zero before) + the product of the query's block and eight tokens'
template <bool FIRST>
__device__ __forceinline__ void mma_q_tokens(float (&c)[4], const uint4& q, uint32_t b0, uint32_t b1) {
  if constexpr (FIRST)
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(q.x), "r"(q.y), "r"(q.z), "r"(q.w), "r"(b0), "r"(b1), "f"(0.f));
  else
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(q.x), "r"(q.y), "r"(q.z), "r"(q.w), "r"(b0), "r"(b1));
}

// KB: 16-channel blocks per tile rounded up to 1, 2, 4 or 8.  HP: pairs of query heads of a set.
// The query's fragments are read from shared memory for each tile: in registers they cost CTAs (47 against 46 us).
template <int KB, int HP, bool PAGED>
__global__ void __launch_bounds__(kBlockThreads, BlockShape<KB, HP>::ctas)
block_score_kernel(const BlockParams p) {
  constexpr int NT = BlockShape<KB, HP>::tiles, STEP = BlockShape<KB, HP>::step;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int u = blockIdx.y;
  const SelUnit su = sel_unit(u, p.n_sets, p.group, p.n_q_heads, p.n_kv_heads);
  const int b = su.b, h = su.h, hs = u % p.n_sets;
  __shared__ __align__(16) uint32_t s_q[HP * KB][32][4];
  extern __shared__ uint32_t s_first[];                       // (PAGED) the pool's index of the first tile of each page
  pdl_wait_for_predecessor();
  pdl_release_successor();
  const ProxyGeom pg = proxy_geom(p.chunks);
  const int n_blocks = pg.n16 + pg.n8;
  const int tiles_alloc = (p.max_len + 15) >> 4;
  const int tile0 = blockIdx.x * p.tiles_per_cta, tile1 = min(tiles_alloc, tile0 + p.tiles_per_cta);
  const unsigned char* unit = p.proxy + (int64_t)su.kv * tiles_alloc * pg.tile_bytes;
  int T = tile0 + warp * STEP;
  uint4 a[NT][KB];
  // (every tile up to max_len is allocated: the first loads do not wait for the length)
  if constexpr (!PAGED) {
#pragma unroll
    for (int j = 0; j < NT; ++j) load_tile<KB>(a[j], unit + (int64_t)(T + j) * pg.tile_bytes, pg, lane, T + j < tile1);
  }
  // (nor do those of the channel pairs that this thread's words of the query operand take: a thread meets every second block,
  // or the only one)
  constexpr int NW = KB < 2 ? 1 : KB / 2;
  const int qe = tid & 3, ql = (tid >> 2) & 31, qkb = KB < 2 ? 0 : tid >> 7;
  uint32_t pair[NW];
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    const int w = (qkb + 2 * i) * 8 + (qe >> 1) * 4 + (ql & 3);
    pair[i] = w < 4 * p.chunks ? *reinterpret_cast<const uint32_t*>(p.chan + (h * p.chunks * 8 + 2 * w)) : 0xffffffffu;
  }
  const int len = clamp_len(p.seq_lens[b], p.max_len, p.status);
  if (tile0 * 16 >= len) return;
  const int row1 = min(len, tile1 * 16);
  const int sh = p.pm.shift - 4, page0 = PAGED ? tile0 >> sh : 0;
  if constexpr (PAGED) {
    for (int i = tid; i <= ((row1 - 1) >> p.pm.shift) - page0; i += kBlockThreads) {
      int page = page_of(p.pm, b, (page0 + i) << p.pm.shift);
      if (!page_ok(p.pm, page)) {
        atomicOr(p.status, FASA_DEV_PAGE_CLAMPED);
        page = 0;
      }
      s_first[i] = (uint32_t)(page * p.n_kv_heads + h) << sh;
    }
  }
  // The query as operand A: rows 0-7 are the queries of head 2 hp, rows 8-15 those of head 2 hp + 1.
#pragma unroll
  for (int n = 0; n < (KB < 2 ? (HP + 1) / 2 : HP * NW); ++n) {
    const int hp = KB < 2 ? 2 * n + (tid >> 7) : n / NW, i = n % NW, kb = KB < 2 ? 0 : qkb + 2 * i;
    const int head = 2 * hp + (qe & 1), query = ql >> 2;
    uint32_t x = 0u;
    if (head < p.group && query < p.q_len) {
      const uint16_t* qrow = p.q + (((int64_t)b * p.q_len + query) * p.n_q_heads + hs * p.group + head) * FASA_HEAD_DIM;
      const int c0 = (int16_t)(pair[i] & 0xffffu), c1 = (int16_t)(pair[i] >> 16);
      x = (c0 >= 0 ? (uint32_t)qrow[c0] : 0u) | ((c1 >= 0 ? (uint32_t)qrow[c1] : 0u) << 16);
    }
    if (hp < HP) s_q[hp * KB + kb][ql][qe] = x;
  }
  __syncthreads();
  auto tile_at = [&](int TT) -> const unsigned char* {
    if constexpr (PAGED) {
      const uint32_t first = s_first[(min(TT, (row1 - 1) >> 4) >> sh) - page0];
      return p.proxy + (int64_t)(first + (uint32_t)(TT & ((1 << sh) - 1))) * pg.tile_bytes;
    } else {
      return unit + (int64_t)TT * pg.tile_bytes;
    }
  };
  if constexpr (PAGED) {
#pragma unroll
    for (int j = 0; j < NT; ++j) load_tile<KB>(a[j], tile_at(T + j), pg, lane, (T + j) * 16 < row1);
  }
  // this lane's row: query g of the set, and the positions that compete there
  const bool mine = g < p.q_len;
  const int64_t row = ((int64_t)b * p.q_len + (mine ? g : 0)) * p.n_sets + hs;
  float* const srow = p.scores + row * p.max_len + 2 * t;
  float* const gmrow = p.gm + row * p.gm_stride;
  const int len_q = max(0, len - (p.q_len - 1 - g)), lo = min(len_q, p.n_sink), hi = len_q - min(p.n_recent, len_q - lo);
  const int all = max(0, len - (p.q_len - 1));                // positions that every query sees
  const bool pairs_ok = ((p.max_len & 1) == 0) && (reinterpret_cast<uintptr_t>(p.scores) & 7) == 0;

  auto stream = [&](auto exact_tag) {
    constexpr bool EXACT = decltype(exact_tag)::value;        // the dominant channels fill exactly KB whole blocks
    const unsigned char* ahead = unit + (int64_t)T * (KB * 512) + lane * 16;    // (EXACT, contiguous) of the tile at T
    while (T * 16 < row1) {                                   // uniform over the warp
      const int next = T + kBlockWarps * STEP;
#pragma unroll
      for (int jp = 0; jp < STEP / 2; ++jp) {
        float v[4][2];                                        // octet o of the pair of tiles, positions 2 t and 2 t + 1
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int j = (2 * jp + e) % NT;                    // (one register tile: both tiles of a pair go through it)
          float c[HP][2][4];
#pragma unroll
          for (int hp = 0; hp < HP; ++hp) {
            const uint4 qa = lds_u4(s_q[hp * KB][lane]);
            mma_q_tokens<true>(c[hp][0], qa, a[j][0].x, a[j][0].z);
            mma_q_tokens<true>(c[hp][1], qa, a[j][0].y, a[j][0].w);
          }
#pragma unroll
          for (int kb = 1; kb < KB; ++kb) {
            if (EXACT || kb < n_blocks) {
#pragma unroll
              for (int hp = 0; hp < HP; ++hp) {
                const uint4 qa = lds_u4(s_q[hp * KB + kb][lane]);
                mma_q_tokens<false>(c[hp][0], qa, a[j][kb].x, a[j][kb].z);
                mma_q_tokens<false>(c[hp][1], qa, a[j][kb].y, a[j][kb].w);
              }
            }
          }
          {                                                   // the registers are free again
            const int TN = NT == 1 && e == 0 ? T + 1 : next + 2 * jp + (NT == 1 ? 0 : e);
            const bool ok = TN * 16 < row1;                   // (otherwise they keep what they held: scored, and not stored)
            if constexpr (EXACT) {
              const unsigned char* tile;
              if constexpr (PAGED) tile = tile_at(TN) + lane * 16;
              else tile = ahead + (NT == 1 && e == 0 ? 1 : kBlockWarps * STEP + 2 * jp + (NT == 1 ? 0 : e)) * KB * 512;
#pragma unroll
              for (int kb = 0; kb < KB; ++kb)
                if (ok) a[j][kb] = ld_proxy_u4(tile + kb * 512);
            } else {
              load_tile<KB>(a[j], tile_at(TN), pg, lane, ok);
            }
          }
#pragma unroll
          for (int o = 0; o < 2; ++o) {
            float2 s;                                         // (-0 becomes +0)
            if (p.max_reduce) {                               // uniform
              s = make_float2(c[0][o][0], c[0][o][1]);
#pragma unroll
              for (int hp = 0; hp < HP; ++hp) {
                if (hp > 0) s = make_float2(fmaxf(s.x, c[hp][o][0]), fmaxf(s.y, c[hp][o][1]));
                if (2 * hp + 1 < p.group) s = make_float2(fmaxf(s.x, c[hp][o][2]), fmaxf(s.y, c[hp][o][3]));
              }
              s = __fadd2_rn(s, make_float2(0.f, 0.f));
            } else {
              s = make_float2(0.f, 0.f);
#pragma unroll
              for (int hp = 0; hp < HP; ++hp)
                s = __fadd2_rn(s, __fadd2_rn(make_float2(c[hp][o][0], c[hp][o][1]), make_float2(c[hp][o][2], c[hp][o][3])));
            }
            v[2 * e + o][0] = s.x;
            v[2 * e + o][1] = s.y;
          }
        }
        const int pos = (T + 2 * jp) * 16;                    // of the pair of tiles
        if (mine) {
          if (pos + 32 <= all && pairs_ok) {
#pragma unroll
            for (int o = 0; o < 4; ++o) *reinterpret_cast<float2*>(srow + pos + 8 * o) = make_float2(v[o][0], v[o][1]);
          } else {
#pragma unroll
            for (int o = 0; o < 4; ++o)
#pragma unroll
              for (int x = 0; x < 2; ++x)
                if (pos + 8 * o + 2 * t + x < len_q) srow[pos + 8 * o + x] = v[o][x];
          }
        }
        if (p.gs > 0) {                                       // uniform
          if (pos < p.n_sink || pos + 32 > all - p.n_recent) {
#pragma unroll
            for (int o = 0; o < 4; ++o)
#pragma unroll
              for (int x = 0; x < 2; ++x) {
                const int i = pos + 8 * o + 2 * t + x;
                if (!(i >= lo && i < hi)) v[o][x] = -INFINITY;
              }
          }
          float m[4];
#pragma unroll
          for (int o = 0; o < 4; ++o) m[o] = max_nan(v[o][0], v[o][1]);
          if (p.gs == 3) {
            // lane t of a quad ends with the maximum of octet t
            const bool t2 = (t & 2) != 0, t1 = (t & 1) != 0;
            const float k0 = max_nan(t2 ? m[2] : m[0], __shfl_xor_sync(0xffffffffu, t2 ? m[0] : m[2], 2));
            const float k1 = max_nan(t2 ? m[3] : m[1], __shfl_xor_sync(0xffffffffu, t2 ? m[1] : m[3], 2));
            const float k = max_nan(t1 ? k1 : k0, __shfl_xor_sync(0xffffffffu, t1 ? k0 : k1, 1));
            if (mine) gmrow[(pos >> 3) + t] = k;
          } else {
            float k = max_nan(max_nan(m[0], m[1], m[2]), m[3]);
            k = max_nan(k, __shfl_xor_sync(0xffffffffu, k, 1));
            k = max_nan(k, __shfl_xor_sync(0xffffffffu, k, 2));
            if (mine && t == 0) gmrow[pos >> 5] = k;
          }
        }
      }
      T = next;
      ahead += kBlockWarps * STEP * KB * 512;
    }
  };
  if (pg.n8 == 0 && pg.n16 == KB) stream(std::true_type{});
  else stream(std::false_type{});
}

template <int KB, int HP>
cudaError_t launch_block_score(fasa_ctx* ctx, BlockParams& p, cudaStream_t stream) {
  constexpr int kStep = kBlockWarps * BlockShape<KB, HP>::step;
  const fasa_config_t& c = ctx->cfg;
  const int units = c.batch * ctx->n_sets, tiles = (c.max_len + 15) / 16;
  // Ten CTAs to an SM, so that the SMs end together (they pull at different rates); but six iterations to a CTA, whose start
  // costs one or two, as long as every SM still gets all it can hold.
  const long long total = (long long)units * tiles, fine = total / (10ll * ctx->n_sm), one_wave = total / (BlockShape<KB, HP>::ctas * (long long)ctx->n_sm);
  long long per_ll = std::max(fine, std::min(6ll * kStep, one_wave));
  per_ll = std::min((long long)kBlockMaxTiles, std::max(1ll, (per_ll + kStep - 1) / kStep) * kStep);
  const int per = (int)per_ll;
  p.tiles_per_cta = per;
  const dim3 grid((unsigned)((tiles + per - 1) / per), (unsigned)units);
  const bool paged = c.page_size > 0;
  const size_t smem = paged ? (size_t)((per >> (p.pm.shift - 4)) + 2) * 4 : 0;
  return paged ? launch_after_predecessor(block_score_kernel<KB, HP, true>, grid, dim3(kBlockThreads), smem, stream, 0, p)
               : launch_after_predecessor(block_score_kernel<KB, HP, false>, grid, dim3(kBlockThreads), smem, stream, 0, p);
}

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
  const fasa_config_t& c = ctx->cfg;
  if ((long long)c.batch * q_len * ctx->n_sets > 65535) return FASA_ERR_UNSUPPORTED;
  BlockParams p;
  memset(&p, 0, sizeof(p));
  p.q = (const uint16_t*)q; p.proxy = (const unsigned char*)proxy_k; p.seq_lens = seq_lens; p.chan = ctx->d_chan;
  p.scores = scores; p.gm = m.gm; p.gs = m.gs; p.gm_stride = m.stride; p.status = ctx->d_status;
  p.n_q_heads = c.n_q_heads; p.n_kv_heads = c.n_kv_heads; p.n_sets = ctx->n_sets; p.group = ctx->sel_heads;
  p.max_len = c.max_len; p.chunks = ctx->chunks; p.q_len = q_len;
  p.max_reduce = c.group_reduce; p.n_sink = c.n_sink; p.n_recent = c.n_recent;
  p.pm = fasa_page_map(ctx);
  const int nb = (ctx->chunks + 1) / 2;                // 16-channel blocks per tile, the 8-channel one included
  auto pick = [&](auto kb_tag) -> cudaError_t {
    constexpr int K = decltype(kb_tag)::value;
    switch ((ctx->sel_heads + 1) / 2) {
      case 1: return launch_block_score<K, 1>(ctx, p, stream);
      case 2: return launch_block_score<K, 2>(ctx, p, stream);
      case 3: return launch_block_score<K, 3>(ctx, p, stream);
      default: return launch_block_score<K, 4>(ctx, p, stream);
    }
  };
  cudaError_t e;
  if (nb <= 1) e = pick(std::integral_constant<int, 1>{});
  else if (nb <= 2) e = pick(std::integral_constant<int, 2>{});
  else if (nb <= 4) e = pick(std::integral_constant<int, 4>{});
  else e = pick(std::integral_constant<int, 8>{});
  FASA_CUDA_TRY(ctx, e);
  FASA_LAUNCH_CHECK(ctx);
  return FASA_OK;
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
