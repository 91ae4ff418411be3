// Scores of every cached token (TIP, Sec. 4.1) for several score rows to a KV head from one pass over its proxy: the first half
// of the decode step in two launches (the appended token's rows first, Algorithm 2's UpdateCache), and the blocks of queries
// of fasa_batched.cu; with the maxima of groups of 8 or 32 scores that the selection goes by (fasa_select.cuh).
//
// score_stream_kernel: what bounds it is the stream (the proxy once, 4 T bytes of scores per token), so the rest is arranged to
// take few instructions and no barrier between warps.  The proxy lies in HBM in the fragment order of mma.m16n8k16's operand A,
// 16 tokens by 16 channels; the same registers are two operands B, of tokens 0-7 (words 0, 2) and 8-15 (words 1, 3).  So the
// query is operand A: rows 0-7 are the T queries of one head (or the heads of a KV head that have a row each), rows 8-15 those of
// the next head of the sum, whose scores then meet in one thread.  The heads are reduced without a shuffle; a lane holds two
// consecutive tokens of one row, and eight tokens' maximum is two shuffles away.  A warp goes from its loads to its stores alone.
//
// The tokens of a unit are shared out to its CTAs by its length, read from the device: a batch of short sequences in long caches
// takes as many CTAs as it has work for, and nothing is read past a length.  With shares cut from max_len, 4 K tokens of four
// sequences in caches of 64 K lay on two or three CTAs of several iterations each, and the others read 21 MB of nothing: a step with a
// set per head 24.4 us, now 18.4; 16 sequences of 2 K in 32 K 45.6 -> 35.6; blocks of five, 8 sequences of 4 K in 64 K 44.6 -> 34.6.
//
// Measured (batch 8, 32 / 8 heads, 40-65 K, 16 FCs, T = 5): 45.1 us, 6.0 TB/s.  Before, tcgen05.mma with both operands in shared
// memory took 71.0 us: the proxy had to be scattered into its operand layout, four warps met at a barrier for each 128 tokens,
// 250 instructions per 32 tokens and warp against 146 here.  The tensor pipe is no limit: 16 products of 8 cycles per 32 tokens
// and scheduler, a quarter of the time that the tokens take to arrive.  At 8 FCs and five heads a set 59.6 -> 32.9 us, 32 FCs
// 97.5 -> 77.7, 64 FCs 189 -> 141, 12 FCs (no whole blocks) 82.6 -> 41.0; the same bits throughout.
//
// A set per query head took another kernel, a persistent grid with rings of bulk copies whose every warp had an equal share, 171
// instructions per 32 tokens and heads in columns that shuffles brought together; its SMs were busy for 31 to 50 thousand cycles.
// The step (scoring, then selection and attention), 32 / 8 heads, batch 4, 30-56 K: 42.7 -> 31.3 us, on pages of 64 53.4 -> 32.5,
// with 32 FCs 65.2 -> 43.9, 64 FCs and batch 2 74.6 -> 41.8; batch 16, 12-16 K 74.3 -> 56.9.
//
// The new token's row is scored from k_new itself: the CTA whose share it ends writes the K, V and proxy rows before it streams
// and keeps the row's channel pairs in shared memory, where the warp that owns its tile takes them for its fragments; nothing waits
// for those writes.  (Written by that warp in its loop, the row's addresses cost 8 to 40 bytes of spills around it at 64 registers:
// batch 4, 30-56 K, a set per head, 36.3 us a step, 31.8 without; default sets, batch 8, 60-90 K, 8 FCs 53.6, 46.4.)  What is left: 8 to
// 72 bytes where the sums of six heads and more fill the registers.  The lengths themselves grow in the second half, which reads the
// old ones before this one ends.
#include <algorithm>
#include <type_traits>

#include "fasa_common.cuh"
#include "fasa_launch.cuh"
#include "fasa_score_core.cuh"
#include "fasa_select.cuh"
#include "fasa_stream.cuh"

namespace {

constexpr int kStreamThreads = 256;
constexpr int kStreamWarps = kStreamThreads / 32;
constexpr int kStreamMaxTiles = 1024;          // proxy tiles of a CTA at most (its page entries lie in shared memory)
// Tiles that a warp holds in registers (positions are finished 32 at a time), and CTAs on an SM.  About 32 KB of loads in flight
// on an SM are enough; more CTAs with fewer tiles each beat fewer with more (batch 8, 40-65 K, 16 FCs, 5 queries: 47 us with 4
// CTAs of two tiles a warp, 51 with 2 or 3 of four).
// HP 0: a single row, whose heads are the rows of the product.
template <int KB, int HP>
struct StreamShape {
  static constexpr int tiles = KB == 1 ? 4 : (KB == 8 ? 1 : 2);
  static constexpr int step = tiles < 2 ? 2 : tiles;        // tiles per warp and iteration
  static constexpr int ctas = KB <= 2 && HP <= 2 ? 4 : 3;
  static constexpr int pairs = HP > 0 ? HP : 1;
};

// A unit is what one pass over a KV head's proxy serves: `rows` score rows (up to 8), each the sum (or the maximum) over `heads`
// query heads.
struct StreamParams {
  const uint16_t* q;
  const unsigned char* proxy;
  const int32_t* seq_lens;
  const int16_t* chan;
  float* scores;                // rows of max_len
  float* gm;                    // gs > 0: maxima of groups of 1 << gs positions, a row of gm_stride per score row
  int32_t* status;
  int n_kv_heads, n_units, rows, heads, max_len, chunks, max_reduce;      // n_units: to a sequence
  int q_seq, q_unit, q_row;     // elements of q from one sequence / unit / row to the next (a head's 128 follow each other)
  int row_seq, row_unit, row_step;   // score rows likewise
  int causal;                   // row r sees rows - 1 - r fewer positions (a block of queries)
  int gs, gm_stride, n_sink, n_recent;
  // (APPEND) the new token's rows, and where they go
  const uint16_t* k_new;
  const uint16_t* v_new;
  uint16_t* k_w;
  uint16_t* v_w;
  unsigned char* proxy_w;
  int64_t ksb, ksh, kst, vsb, vsh, vst;
  PageMap pm;
};

// Tiles of each of n shares of a unit with `tiles` of them: as even as a warp's tiles allow (blocks of four, 7 sequences of 12-18 K, 28 / 4
// heads, 8 FCs 8.3 -> 7.4 us against whole iterations of a CTA; 19 of 3-7 K, 64 FCs 37.6 -> 35.5), but at least an iteration.  A single row
// per unit takes whole iterations (a default step, 12 sequences of 40-60 K, 64.4 us, 65.9 with even shares).
template <int KB, int HP>
__host__ __device__ __forceinline__ int stream_share(int tiles, int n) {
  constexpr int kStep = kStreamWarps * StreamShape<KB, HP>::step, kUnit = HP > 0 ? StreamShape<KB, HP>::step : kStep;
  const int share = ((tiles + n - 1) / n + kUnit - 1) / kUnit * kUnit;
  return share > kStep ? share : kStep;
}

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

// KB: 16-channel blocks per tile (the last one may be half), from five on rounded up to 8.  Up to four blocks the loop knows how
// many bytes a tile has; with tests of the geometry and loads under them, 12 FCs took 72.1 us a default step (12 sequences of
// 40-60 K) where 57.0 are enough, 16 FCs 65.6; 24 FCs, in a loop for four blocks, 88.7 -> 84.5; blocks of seven at 61-73 K, 24 FCs
// 133.6 -> 123.2.
// HP: pairs of heads that are reduced; 0: one row, whose up to eight heads are rows 0-7 of the product (an eighth of the products
// that HP > 0 takes for a single row).  Their sum is a tree over lanes in which every step also halves the tokens a lane holds:
// ((0 + 1) + (2 + 3)) + ((4 + 5) + (6 + 7)), as everywhere else.
// The query's fragments are read from shared memory for each tile: in registers they cost CTAs (47 against 46 us).
// APPEND: the sequence grows by a token first.
template <int KB, int HP, bool PAGED, bool APPEND>
__global__ void __launch_bounds__(kStreamThreads, StreamShape<KB, HP>::ctas)
score_stream_kernel(const StreamParams p) {
  constexpr int NT = StreamShape<KB, HP>::tiles, STEP = StreamShape<KB, HP>::step, HQ = StreamShape<KB, HP>::pairs;
  constexpr bool TREE = HP == 0;
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (known to be uniform)
  const int g = lane >> 2, t = lane & 3;
  const int u = blockIdx.y;
  const int b = u / p.n_units, hs = u - b * p.n_units, h = hs / (p.n_units / p.n_kv_heads), kv = b * p.n_kv_heads + h;
  __shared__ __align__(16) uint32_t s_q[HQ * KB][32][4];
  __shared__ uint32_t s_new[APPEND ? 64 : 1];                 // the appended row's channel pairs
  extern __shared__ uint32_t s_first[];                       // (PAGED) the pool's index of the first tile of each page
  pdl_wait_for_predecessor();
  pdl_release_successor();
  const ProxyGeom pg = proxy_geom(p.chunks);
  const int n_blocks = pg.n16 + pg.n8;
  const int tiles_alloc = (p.max_len + 15) >> 4;
  // The channel pairs that this thread's words of the query operand take: a thread meets every second block, or the only one.
  constexpr int NW = (KB + 1) / 2;
  const int qe = tid & 3, ql = (tid >> 2) & 31, qkb = KB < 2 ? 0 : tid >> 7;
  uint32_t chan2[NW];
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    const int w = (qkb + 2 * i) * 8 + (qe >> 1) * 4 + (ql & 3);
    chan2[i] = w < 4 * p.chunks ? *reinterpret_cast<const uint32_t*>(p.chan + (h * p.chunks * 8 + 2 * w)) : 0xffffffffu;
  }
  // The unit's tokens are shared out to the CTAs of its row of the grid as its length stands on the device: nothing is read past
  // it, and a short sequence in a long cache takes as many CTAs as it has work for.
  const int old_len = clamp_len(p.seq_lens[b], p.max_len, p.status);
  const int new_row = APPEND && old_len < p.max_len ? old_len : -1, len = new_row >= 0 ? old_len + 1 : old_len;
  const int share = stream_share<KB, HP>((len + 15) >> 4, (int)gridDim.x), tile0 = blockIdx.x * share;
  if (tile0 * 16 >= len) return;
  const int row1 = min(len, (tile0 + share) * 16);
  const unsigned char* unit = p.proxy + (int64_t)kv * tiles_alloc * pg.tile_bytes;
  int T = tile0 + warp * STEP;
  uint4 a[NT][KB];
  if constexpr (!PAGED) {
#pragma unroll
    for (int j = 0; j < NT; ++j) load_tile<KB>(a[j], unit + (int64_t)(T + j) * pg.tile_bytes, pg, lane, (T + j) * 16 < row1);
  }
  const int sh = p.pm.shift - 4, page0 = PAGED ? tile0 >> sh : 0;
  if constexpr (PAGED) {
    for (int i = tid; i <= ((row1 - 1) >> p.pm.shift) - page0; i += kStreamThreads) {
      int page = page_of(p.pm, b, (page0 + i) << p.pm.shift);
      if (!page_ok(p.pm, page)) {
        atomicOr(p.status, FASA_DEV_PAGE_CLAMPED);
        page = 0;
      }
      s_first[i] = (uint32_t)(page * p.n_kv_heads + h) << sh;
    }
  }
  // The appended row is in this CTA's share: its K, V and proxy rows (a CTA of every unit that reads this KV head writes them, the
  // same bytes), and its channel pairs from their source for the warp that scores its tile.
  if (APPEND && new_row >= tile0 * 16 && new_row < row1) {    // uniform
    bool mapped = true;
    int64_t koff = b * p.ksb + h * p.ksh + (int64_t)new_row * p.kst, voff = b * p.vsb + h * p.vsh + (int64_t)new_row * p.vst;
    int64_t poff = (int64_t)kv * tiles_alloc * pg.tile_bytes;
    int prow = new_row;
    if constexpr (PAGED) {
      const int page = page_of(p.pm, b, new_row);
      mapped = page_ok(p.pm, page);
      if (!mapped && tid == 0) atomicOr(p.status, FASA_DEV_PAGE_CLAMPED);
      prow = new_row & ((1 << p.pm.shift) - 1);
      koff = page * p.ksb + h * p.ksh + (int64_t)prow * p.kst;
      voff = page * p.vsb + h * p.vsh + (int64_t)prow * p.vst;
      poff = ((int64_t)page * p.n_kv_heads + h) * (1 << sh) * pg.tile_bytes;
    }
    if (tid < 4 * p.chunks) {
      const uint16_t* kn = p.k_new + (int64_t)kv * FASA_HEAD_DIM;
      const int16_t* ch = p.chan + h * p.chunks * 8;
      const int c0 = ch[2 * tid], c1 = ch[2 * tid + 1];
      const uint32_t x = (c0 >= 0 ? (uint32_t)kn[c0] : 0u) | ((c1 >= 0 ? (uint32_t)kn[c1] : 0u) << 16);
      s_new[tid] = x;
      if (mapped) *reinterpret_cast<uint32_t*>(p.proxy_w + poff + proxy_word_offset(pg, prow, tid)) = x;
    } else if (tid >= kStreamThreads - 32 && mapped) {
      const uint16_t* from = (lane < 16 ? p.k_new : p.v_new) + (int64_t)kv * FASA_HEAD_DIM + (lane & 15) * 8;
      uint16_t* to = (lane < 16 ? p.k_w + koff : p.v_w + voff) + (lane & 15) * 8;
      *reinterpret_cast<uint4*>(to) = *reinterpret_cast<const uint4*>(from);
    }
  }
  // The query as operand A: rows 0-7 are the rows of head 2 hp, rows 8-15 those of head 2 hp + 1.
#pragma unroll
  for (int n = 0; n < (KB < 2 ? (HQ + 1) / 2 : HQ * NW); ++n) {
    const int hp = KB < 2 ? 2 * n + (tid >> 7) : n / NW, i = n % NW, kb = KB < 2 ? 0 : qkb + 2 * i;
    // (TREE: up to four heads are there twice, so that a lane's first halving of its tokens needs no other lane)
    const int head = TREE ? ((qe & 1) ? p.heads : (p.heads <= 4 ? (ql >> 2) & 3 : ql >> 2)) : 2 * hp + (qe & 1), query = TREE ? 0 : ql >> 2;
    uint32_t x = 0u;
    if (head < p.heads && query < p.rows) {
      const uint16_t* qrow = p.q + (int64_t)b * p.q_seq + hs * p.q_unit + query * p.q_row + head * FASA_HEAD_DIM;
      const int c0 = (int16_t)(chan2[i] & 0xffffu), c1 = (int16_t)(chan2[i] >> 16);
      x = (c0 >= 0 ? (uint32_t)qrow[c0] : 0u) | ((c1 >= 0 ? (uint32_t)qrow[c1] : 0u) << 16);
    }
    if (hp < HQ && kb < KB) s_q[hp * KB + kb][ql][qe] = x;
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
  // this lane's row, and the positions that compete there
  const bool mine = TREE || g < p.rows;
  const int64_t row = (int64_t)b * p.row_seq + hs * p.row_unit + (mine && !TREE ? g : 0) * p.row_step;
  float* const srow = p.scores + row * p.max_len + (TREE ? 0 : 2 * t);
  float* const gmrow = p.gm + row * p.gm_stride;
  const int len_q = TREE ? len : max(0, len - (p.causal ? p.rows - 1 - g : 0)), lo = min(len_q, p.n_sink), hi = len_q - min(p.n_recent, len_q - lo);
  const int all = max(0, len - (p.causal ? p.rows - 1 : 0));  // positions that every row sees
  const bool even_heads = (p.heads & 1) == 0;
  // TREE: the octet of a pair of tiles and the position that this lane ends with
  const bool four = p.heads <= 4, b0 = (lane & 4) != 0, b1 = (lane & 8) != 0, b2 = (lane & 16) != 0;
  const int octet = four ? 2 * (int)b2 + (int)b0 : 2 * (int)b0 + (int)b1, mine_at = 8 * octet + 2 * t + (int)(four ? b1 : b2);
  const bool no_head = TREE && p.max_reduce && (four ? g & 3 : g) >= p.heads;
  const bool pairs_ok = ((p.max_len & 1) == 0) && (reinterpret_cast<uintptr_t>(p.scores) & 7) == 0;

  // The appended row's words in place of its tile's: nothing waits for the proxy row that is written above.
  auto take_new = [&](uint4 (&x)[KB]) {
    const int r = new_row & 15;
    if (g == (r & 7)) {
#pragma unroll
      for (int kb = 0; kb < KB; ++kb) {
        if (kb < n_blocks) {
          const uint32_t w0 = s_new[kb * 8 + t], w1 = kb < pg.n16 ? s_new[kb * 8 + t + 4] : 0u;
          if (r < 8) { x[kb].x = w0; x[kb].z = w1; }
          else { x[kb].y = w0; x[kb].w = w1; }
        }
      }
    }
  };

  auto stream = [&](auto geometry) {
    constexpr int GEO = decltype(geometry)::value;            // the dominant channels fill KB whole blocks (2), the last one by half (1)
    constexpr bool EXACT = GEO != 0;
    constexpr int kTile = GEO == 1 ? KB * 512 - 256 : KB * 512;
    const unsigned char* ahead = unit + (int64_t)T * kTile + lane * 16;   // (EXACT, contiguous) of the tile at T
    while (T * 16 < row1) {                                   // uniform over the warp
      const int next = T + kStreamWarps * STEP;
#pragma unroll
      for (int jp = 0; jp < STEP / 2; ++jp) {
        float v[4][2];                                        // octet o of the pair of tiles, positions 2 t and 2 t + 1
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int j = (2 * jp + e) % NT;                    // (one register tile: both tiles of a pair go through it)
          if (APPEND && T + 2 * jp + e == (new_row >> 4)) take_new(a[j]);     // (-1: none) uniform
          float c[HQ][2][4];
#pragma unroll
          for (int hp = 0; hp < HQ; ++hp) {
            const uint4 qa = lds_u4(s_q[hp * KB][lane]);
            mma_q_tokens<true>(c[hp][0], qa, a[j][0].x, a[j][0].z);
            mma_q_tokens<true>(c[hp][1], qa, a[j][0].y, a[j][0].w);
          }
#pragma unroll
          for (int kb = 1; kb < KB; ++kb) {
            if (EXACT || kb < n_blocks) {
#pragma unroll
              for (int hp = 0; hp < HQ; ++hp) {
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
              else tile = ahead + (NT == 1 && e == 0 ? 1 : kStreamWarps * STEP + 2 * jp + (NT == 1 ? 0 : e)) * kTile;
#pragma unroll
              for (int kb = 0; kb < KB; ++kb) {
                if (GEO == 1 && kb == KB - 1) {
                  if (ok) {
                    const uint2 w = ld_proxy_u2(tile + kb * 512 - lane * 8);
                    a[j][kb].x = w.x;
                    a[j][kb].y = w.y;
                  }
                } else if (ok) {
                  a[j][kb] = ld_proxy_u4(tile + kb * 512);
                }
              }
            } else {
              load_tile<KB>(a[j], tile_at(TN), pg, lane, ok);
            }
          }
#pragma unroll
          for (int o = 0; o < 2; ++o) {
            float2 s;                                         // (-0 becomes +0)
            if constexpr (TREE) {
              s = no_head ? make_float2(-INFINITY, -INFINITY) : make_float2(c[0][o][0], c[0][o][1]);
            } else if (p.max_reduce) {                               // uniform
              s = make_float2(c[0][o][0], c[0][o][1]);
#pragma unroll
              for (int hp = 0; hp < HP; ++hp) {
                if (hp > 0) s = make_float2(fmaxf(s.x, c[hp][o][0]), fmaxf(s.y, c[hp][o][1]));
                if (2 * hp + 1 < p.heads) s = make_float2(fmaxf(s.x, c[hp][o][2]), fmaxf(s.y, c[hp][o][3]));
              }
              s = __fadd2_rn(s, make_float2(0.f, 0.f));
            } else {
              s = make_float2(0.f, 0.f);
#pragma unroll
              for (int hp = 0; hp < HP; ++hp) {
                float2 pair = make_float2(c[hp][o][0], c[hp][o][1]);
                // (an absent head's zeros make NaN of a key that is not finite)
                if (hp + 1 < HP || even_heads) pair = __fadd2_rn(pair, make_float2(c[hp][o][2], c[hp][o][3]));
                s = __fadd2_rn(s, pair);
              }
            }
            v[2 * e + o][0] = s.x;
            v[2 * e + o][1] = s.y;
          }
        }
        const int pos = (T + 2 * jp) * 16;                    // of the pair of tiles
        if constexpr (TREE) {
          float s;
          auto tree = [&](auto op) {
            float x[2][2];                                    // [octet of the kept tile][position]
#pragma unroll
            for (int o = 0; o < 2; ++o)
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                if (four) x[o][i] = b2 ? v[2 + o][i] : v[o][i];
                else x[o][i] = op(b0 ? v[2 + o][i] : v[o][i], __shfl_xor_sync(0xffffffffu, b0 ? v[o][i] : v[2 + o][i], 4));
              }
            const bool bo = four ? b0 : b1, bi = four ? b1 : b2;
            const int lo_ = four ? 4 : 8, li = four ? 8 : 16;
            const float y0 = op(bo ? x[1][0] : x[0][0], __shfl_xor_sync(0xffffffffu, bo ? x[0][0] : x[1][0], lo_));
            const float y1 = op(bo ? x[1][1] : x[0][1], __shfl_xor_sync(0xffffffffu, bo ? x[0][1] : x[1][1], lo_));
            s = op(bi ? y1 : y0, __shfl_xor_sync(0xffffffffu, bi ? y0 : y1, li));
          };
          if (p.max_reduce) tree([](float u, float w) { return fmaxf(u, w); });     // uniform
          else tree([](float u, float w) { return u + w; });
          s += 0.0f;                                          // (-0 becomes +0)
          const int i = pos + mine_at;
          if (i < len) srow[i] = s;
          if (p.gs > 0) {                                     // uniform
            float m = i >= lo && i < hi ? s : -INFINITY;
            m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, 1));
            m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, 2));
            m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, four ? 8 : 16));
            if (p.gs == 3) {
              if (t == 0 && !(four ? b1 : b2)) gmrow[(pos >> 3) + octet] = m;
            } else {
              m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, 4));
              m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, four ? 16 : 8));
              if (lane == 0) gmrow[pos >> 5] = m;
            }
          }
          continue;
        }
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
      ahead += kStreamWarps * STEP * kTile;
    }
  };
  if constexpr (KB <= 4) {                                   // (KB blocks, the last one whole or half: see fasa_stream_launch)
    if (pg.n8 == 0) stream(std::integral_constant<int, 2>{});
    else stream(std::integral_constant<int, 1>{});
  } else {
    if (pg.n8 == 0 && pg.n16 == KB) stream(std::integral_constant<int, 2>{});
    else stream(std::integral_constant<int, 0>{});
  }
}

template <int KB, int HP>
cudaError_t launch_stream(fasa_ctx* ctx, StreamParams& p, cudaStream_t stream) {
  constexpr int kStep = kStreamWarps * StreamShape<KB, HP>::step;
  const fasa_config_t& c = ctx->cfg;
  const int units = c.batch * p.n_units, tiles = (c.max_len + 15) / 16;
  // CTAs to a unit: as many as fit in one to eight waves, whichever a full cache is scored in soonest.  A CTA's start costs two
  // iterations or so, and the last ones end up to a fifth of their time apart.  One wave against two, three and four (with the append
  // still in the loop, shares of whole iterations): a set per head, batch 4, 30-56 K, 36.5 us a step / 37.1 / 38.9 / 39.6; batch 16, 20-30 K
  // 92.2 / 86.7 / 86.8 / 87.3; default sets, batch 12, 40-60 K 70.0 / 66.1 / 66.9 / 68.3; batch 14, 72 K 126 / 99 / 100 / 99; batch 32, 16-28 K
  // 86.8 / 85.4 / 85.3 / 81.7 (two CTAs to each of 256 units leave a seventh of a wave empty); blocks of three, batch 3, 84-108 K 49.1 /
  // 52.0 / 52.8 / 55.1.  Against the best of ten counts the rule loses 1 % over 173 shapes.
  const int least = (tiles + kStreamMaxTiles - 1) / kStreamMaxTiles, most = (tiles + kStep - 1) / kStep;
  const long long slots = (long long)StreamShape<KB, HP>::ctas * ctx->n_sm;
  int n = least;
  float best = INFINITY;
  for (int w = 1; w <= 8; ++w) {
    const int m = std::max(least, (int)std::min((long long)most, w * slots / units));
    const float each = std::max(1.f, (float)tiles / (float)(m * kStep)), waves = (float)((m * (long long)units + slots - 1) / slots);
    const float time = waves * (each + 2.f) + 0.2f * each;
    if (time < best) {
      best = time;
      n = m;
    }
  }
  const dim3 grid((unsigned)n, (unsigned)units);
  auto go = [&](auto kernel, size_t smem) { return launch_after_predecessor(kernel, grid, dim3(kStreamThreads), smem, stream, 0, p); };
  if (c.page_size > 0) {
    const size_t smem = (size_t)((stream_share<KB, HP>(tiles, n) >> (p.pm.shift - 4)) + 2) * 4;
    if constexpr (HP <= 1)
      if (p.k_new) return go(score_stream_kernel<KB, HP, true, true>, smem);
    return go(score_stream_kernel<KB, HP, true, false>, smem);
  }
  if constexpr (HP <= 1)                             // (a step appends: sets of one row, or of one head)
    if (p.k_new) return go(score_stream_kernel<KB, HP, false, true>, 0);
  return go(score_stream_kernel<KB, HP, false, false>, 0);
}

}  // namespace

int fasa_stream_gm_stride(const fasa_ctx* ctx) { return (ctx->cfg.max_len / 8 + 8) & ~3; }

int32_t fasa_stream_launch(fasa_ctx* ctx, const fasa_stream_args& a, cudaStream_t stream) {
  const fasa_config_t& c = ctx->cfg;
  StreamParams p;
  memset(&p, 0, sizeof(p));
  p.q = (const uint16_t*)a.q; p.proxy = (const unsigned char*)a.proxy_k; p.seq_lens = a.seq_lens; p.chan = ctx->d_chan;
  p.scores = a.scores; p.gm = a.maxima.gm; p.gs = a.maxima.gs; p.gm_stride = a.maxima.stride; p.status = ctx->d_status;
  p.n_kv_heads = c.n_kv_heads; p.max_len = c.max_len; p.chunks = ctx->chunks; p.n_sink = c.n_sink; p.n_recent = c.n_recent;
  p.max_reduce = c.group_reduce;
  if (a.q_len == 0 && ctx->sel_heads == 1) {           // a row per query head
    p.n_units = c.n_kv_heads; p.rows = ctx->group; p.heads = 1;
    p.q_seq = c.n_q_heads * FASA_HEAD_DIM; p.q_unit = ctx->group * FASA_HEAD_DIM; p.q_row = FASA_HEAD_DIM;
    p.row_seq = c.n_q_heads; p.row_unit = ctx->group; p.row_step = 1;
  } else {                                             // a row per query
    const int T = a.q_len > 0 ? a.q_len : 1;
    p.n_units = ctx->n_sets; p.rows = T; p.heads = ctx->sel_heads;
    p.q_seq = T * c.n_q_heads * FASA_HEAD_DIM; p.q_unit = ctx->sel_heads * FASA_HEAD_DIM; p.q_row = c.n_q_heads * FASA_HEAD_DIM;
    p.row_seq = T * ctx->n_sets; p.row_unit = 1; p.row_step = ctx->n_sets;
    p.causal = 1;
  }
  if (a.k_new != nullptr) {
    p.k_new = (const uint16_t*)a.k_new; p.v_new = (const uint16_t*)a.v_new;
    p.k_w = (uint16_t*)a.k_cache; p.v_w = (uint16_t*)a.v_cache; p.proxy_w = (unsigned char*)const_cast<void*>(a.proxy_k);
    p.ksb = c.k_stride_b; p.ksh = c.k_stride_h; p.kst = c.k_stride_t;
    p.vsb = c.v_stride_b; p.vsh = c.v_stride_h; p.vst = c.v_stride_t;
  }
  p.pm = fasa_page_map(ctx);
  const int nb = (ctx->chunks + 1) / 2;                // 16-channel blocks per tile, the 8-channel one included
  auto pick = [&](auto kb_tag) -> cudaError_t {
    constexpr int K = decltype(kb_tag)::value;
    if (p.rows == 1 && a.q_len == 0 && p.heads > 1) return launch_stream<K, 0>(ctx, p, stream);
    switch ((p.heads + 1) / 2) {
      case 1: return launch_stream<K, 1>(ctx, p, stream);
      case 2: return launch_stream<K, 2>(ctx, p, stream);
      case 3: return launch_stream<K, 3>(ctx, p, stream);
      default: return launch_stream<K, 4>(ctx, p, stream);
    }
  };
  cudaError_t e;
  if (nb <= 1) e = pick(std::integral_constant<int, 1>{});
  else if (nb <= 2) e = pick(std::integral_constant<int, 2>{});
  else if (nb <= 3) e = pick(std::integral_constant<int, 3>{});
  else if (nb <= 4) e = pick(std::integral_constant<int, 4>{});
  else e = pick(std::integral_constant<int, 8>{});
  ctx->launches += 1;
  FASA_CUDA_TRY(ctx, e);
  return FASA_OK;
}
