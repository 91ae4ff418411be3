// Decode step in two launches, first half: the appended token's rows and the importance scores of every cached
// token (Algorithm 2's UpdateCache, then TIP, Sec. 4.1), with the maxima of groups of 8 or 32 scores that the
// second half (fasa_select_attend.cu) selects with.
//
// The pass is a stream of the proxy (2 * chunks * 8 bytes per token): what bounds it is HBM.  Two CTAs per SM for
// the whole launch; the tokens of all sequences and KV heads are dealt out to their warps evenly, in pairs of
// 16-token tiles, by the lengths as they stand on the device, so ragged batches end together.  A warp keeps its
// own ring of bulk copies (cp.async.bulk, one copy per page of a paged cache) in flight and scores what has
// arrived with mma.sync straight from shared memory (the proxy's tiles are stored in fragment order, so a lane
// reads its 16 bytes without conflicts): no barrier between warps, and a rate that depends neither on the tile
// geometry nor on the pages.
//
// A score row per query head: the accumulators hold every head in a column of its own and no reduction over the heads
// follows, so one pass over the proxy serves all index sets of a KV head (the cluster kernel streams it once per set).
// Scores go to a buffer (4 bytes per token and head: the caller's, or scratch), which the second half reads back from
// L2 for a few groups per index set.
//
// Measured (ncu, batch 4, 32 / 8 heads, 30-56 K): 31 us for 88 MB of proxy and 22 MB of scores, and 23 us for the second
// half, against 79 + 10 us for a cluster per set.
//
// With at most four query heads to a KV head the eight columns of an instruction hold the four heads twice: of a pair of tiles
// the lanes t < 2 of a quad keep the first one's scores and t >= 2 the second's, which halves the work after the products.
//
// The new token's row is scored from k_new itself: the warp that owns its tile writes the K, V and proxy rows
// and replaces the row in its fragments, so nothing waits for those writes.  The lengths themselves grow in the
// second half, which reads the old ones before this one ends.
#include "fasa_common.cuh"
#include "fasa_launch.cuh"
#include "fasa_score_core.cuh"
#include "fasa_select.cuh"
#include "fasa_stream.cuh"

namespace {

constexpr int kSlots = 3;                 // bulk copies a warp has in flight
constexpr long long kSpinCycles = 400000000ll;   // bound of a wait for a copy, in SM clocks (~0.2 s)

struct StreamParams {
  const uint16_t* q;
  const unsigned char* proxy;
  const int32_t* seq_lens;
  const int16_t* chan;
  float* scores;                          // [batch][n_q_heads][max_len]
  float* gm;                              // [batch * n_q_heads][gm_stride]
  int32_t* status;
  int batch, n_q_heads, n_kv_heads, group, max_len, chunks, n_sink, n_recent;
  int gs, gm_stride;                      // groups of 1 << gs positions; gs 0: no maxima
  int slot_pairs, slot_bytes;             // a copy: pairs of tiles, bytes
  // append (null: none)
  const uint16_t* k_new;
  const uint16_t* v_new;
  uint16_t* k_w;
  uint16_t* v_w;
  unsigned char* proxy_w;
  int64_t ksb, ksh, kst, vsb, vsh, vst;
  PageMap pm;
};

__device__ __forceinline__ uint32_t sptr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(unsigned long long* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(sptr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_expect(unsigned long long* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(sptr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_try(unsigned long long* bar, uint32_t parity) {
  uint32_t done;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.b32 %0, 1, 0, p;\n\t}"
               : "=r"(done) : "r"(sptr(bar)), "r"(parity) : "memory");
  return done != 0;
}
// One warp, all lanes with the same answer.  false: the bound ran out.
__device__ __forceinline__ bool bar_wait(unsigned long long* bar, uint32_t parity) {
  bool done = bar_try(bar, parity);
  if (!__all_sync(0xffffffffu, done)) {
    const long long t0 = clock64();
    while (!done && clock64() - t0 <= kSpinCycles) done = bar_try(bar, parity);
  }
  return __all_sync(0xffffffffu, done);
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(sptr(dst)), "l"(src), "r"(bytes), "r"(sptr(bar)) : "memory");
}

// Walks a warp's share of all pairs of tiles: sequence after sequence, KV head after KV head.
struct Walk {
  int b, h, len, pairs, pair, left;       // of the current (sequence, KV head): grown length, pairs, next pair; pairs left in the share
};
__device__ __forceinline__ int walk_len(const StreamParams& p, int b, int* old_len) {
  const int l = clamp_len(p.seq_lens[b], p.max_len, p.status);
  *old_len = l;
  return p.k_new != nullptr && l < p.max_len ? l + 1 : l;
}
// Share i of n: [total * i / n, total * (i + 1) / n) of the pairs.
__device__ __forceinline__ Walk walk_start(const StreamParams& p, int i, int n, int lane) {
  int old_len;
  long long total = 0;
  for (int b0 = 0; b0 < p.batch; b0 += 32) {
    const int np = b0 + lane < p.batch ? (walk_len(p, b0 + lane, &old_len) + 31) >> 5 : 0;
    total += __reduce_add_sync(0xffffffffu, np);
  }
  total *= p.n_kv_heads;
  const long long first = total * i / n, end = total * (i + 1) / n;
  Walk w{0, 0, 0, 0, 0, (int)(end - first)};
  if (w.left == 0) return w;
  long long before = 0;
  for (int b0 = 0; b0 < p.batch; b0 += 32) {
    const int len = b0 + lane < p.batch ? walk_len(p, b0 + lane, &old_len) : 0;
    const uint32_t np = (uint32_t)(len + 31) >> 5, incl = sel_scan(np, lane);
    const uint32_t hits = __ballot_sync(0xffffffffu, before + (long long)incl * p.n_kv_heads > first);
    if (hits) {
      const int l = __ffs(hits) - 1;
      w.b = b0 + l;
      w.len = __shfl_sync(0xffffffffu, len, l);
      w.pairs = (w.len + 31) >> 5;
      const int off = (int)(first - before - (long long)(__shfl_sync(0xffffffffu, incl, l) - w.pairs) * p.n_kv_heads);
      w.h = off / w.pairs;
      w.pair = off - w.h * w.pairs;
      return w;
    }
    before += (long long)__shfl_sync(0xffffffffu, incl, 31) * p.n_kv_heads;
  }
  w.left = 0;
  return w;
}
// On to the next (sequence, KV head) with pairs once this one is finished (w.left > 0).
__device__ __forceinline__ void walk_next(const StreamParams& p, Walk& w) {
  w.pair = 0;
  if (++w.h < p.n_kv_heads) return;
  w.h = 0;
  do {
    int old_len;
    w.len = walk_len(p, ++w.b, &old_len);
    w.pairs = (w.len + 31) >> 5;
  } while (w.pairs == 0 && w.b + 1 < p.batch);
}

// KB: 16-channel blocks per tile rounded up to 1, 2, 4 or 8.  G4: at most four query heads to a KV head.
template <int KB, bool G4, bool PAGED>
__global__ void __launch_bounds__(KB > 4 ? 128 : 256, 2)
score_stream_kernel(const StreamParams p) {
  constexpr int WARPS = KB > 4 ? 4 : 8;
  extern __shared__ __align__(128) unsigned char ring[];
  __shared__ __align__(8) unsigned long long s_bar[WARPS][kSlots];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (lane == 0) {
    for (int i = 0; i < kSlots; ++i) bar_init(&s_bar[warp][i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  pdl_wait_for_predecessor();
  pdl_release_successor();
  const ProxyGeom pg = proxy_geom(p.chunks);
  const int tiles_alloc = (p.max_len + 15) >> 4;
  const int pair_bytes = 2 * pg.tile_bytes;
  unsigned char* const my_ring = ring + warp * kSlots * p.slot_bytes;
  Walk w = walk_start(p, blockIdx.x * WARPS + warp, gridDim.x * WARPS, lane);
  // ---- the copies run kSlots ahead of the scoring, on a walk of their own ---------------------------
  Walk ahead = w;
  int ahead_run = min(ahead.left, ahead.pairs - ahead.pair);           // pairs left of its (sequence, KV head)
  const unsigned char* ahead_src = nullptr;
  auto locate = [&]() {
    ahead_src = p.proxy + ((int64_t)(ahead.b * p.n_kv_heads + ahead.h) * tiles_alloc + 2 * ahead.pair) * pg.tile_bytes;
  };
  if (!PAGED) locate();
  auto issue = [&](int slot) {
    if (ahead_run <= 0) return;
    const int n = min(p.slot_pairs, ahead_run);
    uint32_t bytes = (uint32_t)(n * pair_bytes);
    if (2 * (ahead.pair + n) * 16 - 16 >= ahead.len) bytes -= pg.tile_bytes;      // the last pair has one tile
    unsigned char* dst = my_ring + slot * p.slot_bytes;
    unsigned long long* bar = &s_bar[warp][slot];
    if (lane == 0) bar_expect(bar, bytes);
    if constexpr (PAGED) {
      __syncwarp();
      const int T0 = 2 * ahead.pair, T1 = T0 + (int)(bytes / (uint32_t)pg.tile_bytes);
      const int sh = p.pm.shift - 4, first = T0 >> sh, pages = ((T1 - 1) >> sh) - first + 1;
      for (int i = lane; i < pages; i += 32) {
        const int a = max(T0, (first + i) << sh), e = min(T1, (first + i + 1) << sh);
        bulk_copy(dst + (a - T0) * pg.tile_bytes, p.proxy + proxy_tile_offset(p.pm, ahead.b, ahead.h, p.n_kv_heads, a, tiles_alloc, pg.tile_bytes, p.status),
                  (uint32_t)((e - a) * pg.tile_bytes), bar);
      }
    } else {
      if (lane == 0) bulk_copy(dst, ahead_src, bytes, bar);
      ahead_src += bytes;
    }
    ahead_run -= n;
    ahead.pair += n;
    if (ahead_run == 0) {
      ahead.left -= ahead.pair;                      // (kept as what is left counted from pair 0 of this unit)
      if (ahead.left > 0) {
        walk_next(p, ahead);
        ahead_run = min(ahead.left, ahead.pairs);
        if (!PAGED) locate();
      }
    }
  };
  ahead.left += ahead.pair;
  for (int i = 0; i < kSlots; ++i) issue(i);

  const int g = lane >> 2, t = lane & 3;
  const bool exact = pg.n8 == 0 && pg.n16 == KB;     // whole 16-channel blocks: no test of the geometry in the loop
  int slot = 0;
  uint32_t parity = 0;
  bool ok = true;
  while (w.left > 0 && ok) {
    const int run = min(w.left, w.pairs - w.pair);   // pairs of this (sequence, KV head)
    // Operand: column n of the product is query head n; G4: head n mod 4.
    ScoreFrag<KB> f;
    load_score_b<KB>(f, p.q + ((int64_t)w.b * p.n_q_heads + (int64_t)w.h * p.group) * FASA_HEAD_DIM, p.chan + w.h * p.chunks * 8, p.chunks, p.group,
                     G4 ? (lane & 15) : lane);
    const int64_t row0 = (int64_t)w.b * p.n_q_heads + w.h * p.group;                    // its first score row
    float* const srow0 = p.scores + row0 * p.max_len;
    float* const gm0 = p.gm + row0 * p.gm_stride;
    const int lo = min(w.len, p.n_sink), hi = w.len - min(p.n_recent, w.len - lo);      // positions that compete
    int new_row = -1;                                // the appended row, if the sequence grows
    if (p.k_new != nullptr) {
      int old_len;
      if (walk_len(p, w.b, &old_len) > old_len) new_row = old_len;
    }
    // channel pair i of the appended row, from its source
    auto new_word = [&](int i) -> uint32_t {
      if (i >= 4 * p.chunks) return 0u;
      const uint16_t* kn = p.k_new + (int64_t)(w.b * p.n_kv_heads + w.h) * FASA_HEAD_DIM;
      const int16_t* ch = p.chan + w.h * p.chunks * 8;
      const int c0 = ch[2 * i], c1 = ch[2 * i + 1];
      return (c0 >= 0 ? (uint32_t)kn[c0] : 0u) | ((c1 >= 0 ? (uint32_t)kn[c1] : 0u) << 16);
    };
    // its K, V and proxy rows (one warp)
    auto store_new = [&]() {
      const int64_t kv = (int64_t)(w.b * p.n_kv_heads + w.h);
      int64_t koff = w.b * p.ksb + w.h * p.ksh + (int64_t)new_row * p.kst, voff = w.b * p.vsb + w.h * p.vsh + (int64_t)new_row * p.vst;
      int64_t poff = kv * tiles_alloc * pg.tile_bytes;
      int prow = new_row;
      if constexpr (PAGED) {
        const int page = page_of(p.pm, w.b, new_row);
        if (!page_ok(p.pm, page)) {
          if (lane == 0) atomicOr(p.status, FASA_DEV_PAGE_CLAMPED);
          return;
        }
        prow = new_row & ((1 << p.pm.shift) - 1);
        koff = page * p.ksb + w.h * p.ksh + (int64_t)prow * p.kst;
        voff = page * p.vsb + w.h * p.vsh + (int64_t)prow * p.vst;
        poff = ((int64_t)page * p.n_kv_heads + w.h) * (1 << (p.pm.shift - 4)) * pg.tile_bytes;
      }
      const uint16_t* from = (lane < 16 ? p.k_new : p.v_new) + kv * FASA_HEAD_DIM + (lane & 15) * 8;
      uint16_t* to = (lane < 16 ? p.k_w + koff : p.v_w + voff) + (lane & 15) * 8;
      *reinterpret_cast<uint4*>(to) = *reinterpret_cast<const uint4*>(from);
      for (int i = lane; i < 4 * p.chunks; i += 32)
        *reinterpret_cast<uint32_t*>(p.proxy_w + poff + proxy_word_offset(pg, prow, i)) = new_word(i);
    };
    constexpr int NC = G4 ? 1 : 2;                    // fragments of a pair
    // Maxima of the groups of a head's scores in the fragments of one column: v[o] = octet 2 (t >> 1) + o (G4), or octet o
    auto store_max_head = [&](const float (&v)[2 * NC], float* hgm, bool mine, int pair) {
      const bool u16 = (lane & 16) != 0, u8 = (lane & 8) != 0;
      float m;
      int octet;
      if constexpr (G4) {
        m = max_nan(u16 ? v[1] : v[0], __shfl_xor_sync(0xffffffffu, u16 ? v[0] : v[1], 16));
        m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, 8));
        octet = 2 * (t >> 1) + (u16 ? 1 : 0);
      } else {
        const float x0 = max_nan(u16 ? v[2 * NC - 2] : v[0], __shfl_xor_sync(0xffffffffu, u16 ? v[0] : v[2 * NC - 2], 16));
        const float x1 = max_nan(u16 ? v[2 * NC - 1] : v[1], __shfl_xor_sync(0xffffffffu, u16 ? v[1] : v[2 * NC - 1], 16));
        m = max_nan(u8 ? x1 : x0, __shfl_xor_sync(0xffffffffu, u8 ? x0 : x1, 8));
        octet = 2 * (u16 ? 1 : 0) + (u8 ? 1 : 0);
      }
      m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, 4));
      if (p.gs == 3) {
        if (mine && (lane & (G4 ? 12 : 4)) == 0) hgm[pair * 4 + octet] = m;
      } else {
        m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, 16));
        m = max_nan(m, __shfl_xor_sync(0xffffffffu, m, G4 ? 2 : 8));
        if (mine && g == 0 && (!G4 || t < 2)) hgm[pair] = m;
      }
    };

    // where this lane's values go: rows g, g + 8, ... of its two heads' score rows
    const int head0 = G4 ? 2 * (t & 1) : 2 * t;
    float* const lane_row = srow0 + (int64_t)head0 * p.max_len + (G4 ? 16 * (t >> 1) : 0) + g;
    float* const lane_gm = gm0 + (int64_t)head0 * p.gm_stride;
    // Pairs whose 32 positions exist and compete, and whose tiles are whole 16-channel blocks: no test in the loop.
    auto plain = [&](auto np_tag, const unsigned char* src, int pair0) {
      constexpr int NP = decltype(np_tag)::value;
      uint4 a[NP][2][KB];
#pragma unroll
      for (int i = 0; i < NP; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
          for (int kb = 0; kb < KB; ++kb) a[i][e][kb] = *reinterpret_cast<const uint4*>(src + ((i * 2 + e) * KB + kb) * 512 + lane * 16);
      float c[NP][2][4];                             // (a fragment for each tile: in a common one, each tile meeting zeros in the other's
                                                     // columns, a key that is not finite made scores of the other tile NaN)
#pragma unroll
      for (int i = 0; i < NP; ++i)
#pragma unroll
        for (int e = 0; e < 2; ++e) c[i][e][0] = c[i][e][1] = c[i][e][2] = c[i][e][3] = 0.f;
#pragma unroll
      for (int kb = 0; kb < KB; ++kb)
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
          for (int i = 0; i < NP; ++i) mma_bf16_16816(c[i][e], a[i][e][kb], f.b[kb]);
      if constexpr (G4) {
#pragma unroll
        for (int i = 0; i < NP; ++i)
#pragma unroll
          for (int k = 0; k < 4; ++k) c[i][0][k] = t < 2 ? c[i][0][k] : c[i][1][k];
      }
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const int pair = pair0 + i;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const bool mine = head0 + e < p.group;
          float* hrow = lane_row + (int64_t)e * p.max_len + pair * 32;
          float v[2 * NC];
#pragma unroll
          for (int o = 0; o < 2 * NC; ++o) {
            v[o] = c[i][o >> 1][(o & 1) * 2 + e] + 0.0f;               // (-0 becomes +0)
            if (mine) hrow[8 * o] = v[o];
          }
          if (p.gs > 0) store_max_head(v, lane_gm + (int64_t)e * p.gm_stride, mine, pair);
        }
      }
    };
    // The general form, a pair at a time.  PATCH: the pair holds the appended row, which is taken from its source.
    auto general = [&](auto patch_tag, const unsigned char* src, int pair) {
      constexpr bool PATCH = decltype(patch_tag)::value;
      uint4 a[2][KB];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const unsigned char* tile = src + e * pg.tile_bytes;
#pragma unroll
        for (int kb = 0; kb < KB; ++kb) {
          a[e][kb] = make_uint4(0u, 0u, 0u, 0u);
          if (kb < pg.n16) {
            a[e][kb] = *reinterpret_cast<const uint4*>(tile + kb * 512 + lane * 16);
          } else if (kb == pg.n16 && pg.n8) {
            const uint2 x = *reinterpret_cast<const uint2*>(tile + pg.n16 * 512 + lane * 8);
            a[e][kb] = make_uint4(x.x, x.y, 0u, 0u);
          }
        }
        if constexpr (PATCH) {
          const int r = new_row & 15;
          if ((new_row >> 4) == 2 * pair + e && g == (r & 7)) {
#pragma unroll
            for (int kb = 0; kb < KB; ++kb) {
              if (kb < pg.n16 + pg.n8) {
                const uint32_t x0 = new_word(kb * 8 + t), x1 = kb < pg.n16 ? new_word(kb * 8 + t + 4) : 0u;
                if (r < 8) { a[e][kb].x = x0; a[e][kb].z = x1; }
                else { a[e][kb].y = x0; a[e][kb].w = x1; }
              }
            }
          }
        }
      }
      float c[2][4];
#pragma unroll
      for (int e = 0; e < 2; ++e) c[e][0] = c[e][1] = c[e][2] = c[e][3] = 0.f;
#pragma unroll
      for (int kb = 0; kb < KB; ++kb) {
        if (kb < pg.n16 + pg.n8) {
#pragma unroll
          for (int e = 0; e < 2; ++e) mma_bf16_16816(c[e], a[e][kb], f.b[kb]);
        }
      }
      if constexpr (G4) {
#pragma unroll
        for (int i = 0; i < 4; ++i) c[0][i] = t < 2 ? c[0][i] : c[1][i];
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const bool mine = head0 + e < p.group;
        float* hrow = lane_row + (int64_t)e * p.max_len + pair * 32;
        float v[2 * NC];
#pragma unroll
        for (int o = 0; o < 2 * NC; ++o) {
          v[o] = c[o >> 1][(o & 1) * 2 + e] + 0.0f;
          const int row = pair * 32 + 8 * ((G4 ? 2 * (t >> 1) : 0) + o) + g;
          if (mine && row < w.len) hrow[8 * o] = v[o];
          if (!(row >= lo && row < hi)) v[o] = -INFINITY;
        }
        if (p.gs > 0) store_max_head(v, lane_gm + (int64_t)e * p.gm_stride, mine, pair);
      }
    };
    // pairs [plain0, plain1) are plain: all their positions compete, and none holds the appended row
    const int plain0 = exact ? (lo + 31) >> 5 : w.pairs, plain1 = min(hi, new_row >= 0 ? new_row : w.len) >> 5;
    using One = std::integral_constant<int, 1>;
    using Two = std::integral_constant<int, (KB > 4) ? 1 : 2>;           // (64 FCs: the tiles of one pair fill the registers)
    for (int off = 0; off < run; off += p.slot_pairs) {
      const int n = min(p.slot_pairs, run - off);
      ok = bar_wait(&s_bar[warp][slot], parity);
      if (!ok) break;
      const unsigned char* src = my_ring + slot * p.slot_bytes;
      const int first = w.pair + off;
      int j = 0;
      while (j < n) {
        const int pair = first + j;
        if (pair >= plain0 && pair < plain1) {
          if (Two::value == 2 && j + 1 < n && pair + 1 < plain1) {
            plain(Two{}, src + j * pair_bytes, pair);
            j += 2;
            continue;
          }
          plain(One{}, src + j * pair_bytes, pair);
        } else if ((new_row >> 5) == pair) {         // (new_row -1: none)
          general(std::true_type{}, src + j * pair_bytes, pair);
          store_new();
        } else {
          general(std::false_type{}, src + j * pair_bytes, pair);
        }
        ++j;
      }
      __syncwarp();                                  // every lane is done with the slot
      issue(slot);
      if (++slot == kSlots) { slot = 0; parity ^= 1u; }
    }
    w.left -= run;
    w.pair += run;
    if (w.left > 0) walk_next(p, w);
  }
  if (!ok) {                                         // (uniform over the warp) leave no copy behind that still writes here
    if (lane == 0) atomicOr(p.status, FASA_DEV_TIMEOUT);
    for (int i = 0; i < kSlots; ++i) {
      bar_wait(&s_bar[warp][slot], parity);
      if (++slot == kSlots) { slot = 0; parity ^= 1u; }
    }
  }
}

}  // namespace

int fasa_stream_gm_stride(const fasa_ctx* ctx) { return (ctx->cfg.max_len / 8 + 8) & ~3; }

int32_t fasa_stream_launch(fasa_ctx* ctx, const fasa_stream_args& a, cudaStream_t stream) {
  const fasa_config_t& c = ctx->cfg;
  StreamParams p;
  memset(&p, 0, sizeof(p));
  p.q = (const uint16_t*)a.q; p.proxy = (const unsigned char*)a.proxy_k; p.seq_lens = a.seq_lens; p.chan = ctx->d_chan;
  p.scores = a.scores; p.gm = a.gm; p.status = ctx->d_status;
  p.batch = c.batch; p.n_q_heads = c.n_q_heads; p.n_kv_heads = c.n_kv_heads;
  p.group = ctx->group; p.max_len = c.max_len; p.chunks = ctx->chunks; p.n_sink = c.n_sink; p.n_recent = c.n_recent;
  p.gs = a.gs; p.gm_stride = fasa_stream_gm_stride(ctx);
  if (a.k_new != nullptr) {
    p.k_new = (const uint16_t*)a.k_new; p.v_new = (const uint16_t*)a.v_new;
    p.k_w = (uint16_t*)a.k_cache; p.v_w = (uint16_t*)a.v_cache; p.proxy_w = (unsigned char*)const_cast<void*>(a.proxy_k);
    p.ksb = c.k_stride_b; p.ksh = c.k_stride_h; p.kst = c.k_stride_t;
    p.vsb = c.v_stride_b; p.vsh = c.v_stride_h; p.vst = c.v_stride_t;
  }
  p.pm = fasa_page_map(ctx);
  const bool paged = c.page_size > 0, g4 = ctx->group <= 4;
  const int nb = (ctx->chunks + 1) / 2, kb = nb <= 1 ? 1 : (nb <= 2 ? 2 : (nb <= 4 ? 4 : 8)), warps = kb > 4 ? 4 : 8;
  p.slot_bytes = kb > 4 ? 8192 : 4096;                               // of a copy (64 FCs: one pair)
  p.slot_pairs = p.slot_bytes / (512 * ctx->chunks);                 // a pair takes 512 bytes per 16-byte chunk of a token
  const size_t smem = (size_t)warps * kSlots * p.slot_bytes;
  auto go = [&](auto kernel) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 98304);
    if (e != cudaSuccess) return e;
    return launch_after_predecessor(kernel, dim3((unsigned)(2 * ctx->n_sm)), dim3((unsigned)(32 * warps)), smem, stream, 0, p);
  };
  auto form = [&](auto kb_tag) -> cudaError_t {
    constexpr int K = decltype(kb_tag)::value;
    if (g4) return paged ? go(score_stream_kernel<K, true, true>) : go(score_stream_kernel<K, true, false>);
    return paged ? go(score_stream_kernel<K, false, true>) : go(score_stream_kernel<K, false, false>);
  };
  cudaError_t e;
  if (kb == 1) e = form(std::integral_constant<int, 1>{});
  else if (kb == 2) e = form(std::integral_constant<int, 2>{});
  else if (kb == 4) e = form(std::integral_constant<int, 4>{});
  else e = form(std::integral_constant<int, 8>{});
  ctx->launches += 1;
  FASA_CUDA_TRY(ctx, e);
  return FASA_OK;
}
