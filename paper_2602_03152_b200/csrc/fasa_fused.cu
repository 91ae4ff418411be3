// One decode step in one launch: UpdateCache -> TIP scoring -> TopK-I -> FAC (Algorithm 2's
// order; Sec. 4.1-4.2, Eq. 6-7).
//
// One thread-block cluster per selection unit: a (batch, KV head) pair, or the part of a KV
// head's query heads that shares an index set.  The CTAs of the cluster cut the unit's cached
// tokens into contiguous slices and
//   0. (append form) the CTA whose slice ends the sequence writes the new K, V and proxy rows;
//   1. stream their slice of the tiled proxy-K buffer once (16-byte loads in tensor-core
//      fragment order, scored with mma.sync), keep every token's selection key in shared
//      memory and histogram its top 11 bits;
//   2. find the budget-th largest key by an MSB-first radix select.  A radix pass (11, 11, 10
//      bits) costs one cluster barrier: before it every CTA PUSHES the sums of its 32-bin
//      groups into every peer's shared memory, after it every warp locates the group from its
//      local copy, fetches that group's 32 bins from the peers through distributed shared
//      memory and locates the bin, redundantly and without a block barrier.  As soon as the
//      bin that holds the budget-th key has few keys cluster-wide (normally after the first
//      pass), every CTA pushes its keys of that bin to all peers (second barrier) and each CTA
//      finishes the selection on its own copy with block-level passes;
//   3. write the selected positions in ascending order (ballot masks + prefix sums, equal keys
//      lowest index first, so the result equals a stable sort).  The number of selected tokens
//      in lower-ranked CTAs follows from what step 2 has already fetched (their bin counts and
//      their pushed keys), so no barrier is needed here;
//   4. attend, each CTA over an equal share of the index list (one barrier makes the peers'
//      parts of the list visible): K/V rows gathered by index with an online softmax;
//   5. push their partial results into the shared memory of the CTA that finishes each output
//      (one last barrier), which merges them locally.
// Scores, histograms and split-K partials never travel through HBM: the launch moves the
// proxy rows of every token, the K/V rows of the selected tokens, q and the outputs.
//
// Cluster barriers per launch: the split set-up barrier, then normally four (first histogram,
// candidate keys, index list, merge); up to six when many keys share the leading bits of the
// budget-th key.  Each is reached by all
// threads of all CTAs of a cluster the same number of times: every decision around one is taken
// from cluster-wide integer sums that are identical in every warp of every CTA.  The whole-step
// form ends with the merge barrier; the select-only forms end with the last barrier of the
// selection, after which no CTA touches a peer's shared memory.  No thread spins on anything.
#include <cooperative_groups.h>

#include <type_traits>

#include "fasa_attn_core.cuh"
#include "fasa_common.cuh"
#include "fasa_launch.cuh"
#include "fasa_score_core.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int kFT = 512;               // threads per CTA; two CTAs share an SM (64 registers per thread):
                                       // what one SM can pull from HBM grows with its resident warps
constexpr int kFBins = 2048;           // bins of the widest radix pass
constexpr int kPartStride = kMergePartStride - 2;   // m, l, acc[128] (+ 2 words of padding in shared memory)
constexpr int kCapMax = 22528;         // keys a CTA can hold (88 KB of shared memory)
constexpr int kCapPair = 16384;        // ... and still leave room for a second CTA on the SM
constexpr int kMaxCs = kMergeMaxCs;     // CTAs per cluster at most
constexpr int kGroups = kFBins / 32;   // 32-bin groups of the widest radix pass
constexpr int kCandCap = 4096;         // keys of one bin that the cluster finishes locally
constexpr int kFinBits = 7;            // bits per block-level pass of that local finish
constexpr int kFinBins = 1 << kFinBits;
// A warp's part of the attention phase: 8 K and 8 V rows, afterwards 8 accumulators of 128 channels.
constexpr int kAttSlot = 16 * kRowPad * 2;
static_assert(kAttSlot >= 8 * kAccStride * 4 && kAttSlot % 16 == 0, "a warp's accumulators take over its rows");

// Dynamic shared memory of one CTA holding `cap` keys (bytes from the start):
//   keys[cap] | hist1 (8 KB) | sums1 (4 KB) | 4 KB | sums0 (4 KB) | hist0 (8 KB) | masks
// hist0 / hist1: the histograms of even / odd radix passes; sums0 / sums1: the group sums that
// every CTA of the cluster pushes here before the barrier of an even / odd pass, [rank][group].
// The candidate keys pushed after pass 0 land in hist1 .. the spare 4 KB (nothing else uses
// them then), those pushed after pass 1 in the spare 4 KB .. hist0 (read by peers during pass
// 0 only).  The attention phase reuses the area from its start (keys, histograms and masks are
// dead by then; no peer writes here after the last barrier of the selection).
struct FusedSmem {
  int keys, hist1, sums1, spare, sums0, hist0, mask, sel_end;
  int ring, part, m, l, att_end;
  int total;
};
__host__ __device__ inline FusedSmem fused_smem_layout(int cap, int kFW = kFT / 32) {   // kFW: warps per CTA
  FusedSmem L;
  L.keys = 0;
  L.hist1 = cap * 4;
  L.sums1 = L.hist1 + kFBins * 4;
  L.spare = L.sums1 + kMaxCs * kGroups * 4;
  L.sums0 = L.spare + 4096;
  L.hist0 = L.sums0 + kMaxCs * kGroups * 4;
  L.mask = L.hist0 + kFBins * 4;
  L.sel_end = L.mask + 2 * (cap / 32 + 1) * 4;     // one bit per key: above / equal to the threshold
  L.ring = 0;                                      // [kFW] slots of the attention phase
  L.part = L.ring + kFW * kAttSlot;                // [8][kPartStride + 2]
  L.m = L.part + FASA_MAX_GROUP * (kPartStride + 2) * 4;   // [kFW][8]
  L.l = L.m + kFW * FASA_MAX_GROUP * 4;
  L.att_end = L.l + kFW * FASA_MAX_GROUP * 4;
  L.total = L.sel_end > L.att_end ? L.sel_end : L.att_end;
  return L;
}
static_assert(kFBins * 4 + kMaxCs * kGroups * 4 + 4096 == kCandCap * 4, "candidate area");

struct FusedParams {
  const uint16_t* q;
  const uint16_t* k;
  const uint16_t* v;
  const unsigned char* proxy;
  const int32_t* seq_lens;
  const int16_t* chan;
  // append-then-step form (all null / unused otherwise): the new token's rows, the buffers
  // they are written to, the length to update and a per-sequence arrival counter
  const uint16_t* k_new;
  const uint16_t* v_new;
  uint16_t* k_w;
  uint16_t* v_w;
  unsigned char* proxy_w;
  int32_t* seq_lens_w;
  int32_t* arrive;
  // split key cache (append form; ndchan null otherwise): k_w holds the nd non-dominant channels of every key
  const int16_t* ndchan;
  int nd;
  fasa_resident res;
  int early;               // at most one CTA per SM, all resident at once: launched early, and lets its successor be
  int shift_clusters, shift_ctas;   // phase shift of grids that run in rounds: clusters / CTAs resident at once (0: none)
  float* scores;           // nullable
  int32_t* idx;
  int32_t* n_sel;
  float* out;
  float* out_mirror;       // nullable: a second copy of out (mapped host memory of the host-buffer step)
  float* lse;              // nullable
  int32_t* status;
  int n_q_heads, n_kv_heads, n_sets, group, max_len, chunks, n_sink, n_recent, budget, n_sel_max;   // group: query heads of a unit
  int max_reduce;          // score of a KV head = max over its query heads instead of their sum
  int64_t ksb, ksh, kst, vsb, vsh, vst;
  float scale_log2;        // softmax_scale * log2(e)
  int q_len;               // (SCORES) blocks of queries: the rows of a sequence are (query, set) pairs, query t sees q_len - 1 - t
                           // fewer positions (1: plain rows)
  int host_rows;           // K and V rows lie in host memory
  PageMap pm;              // paged caches (all zero: contiguous)
};

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Among per-lane counts v (lane 0 first), finds the lane where the running sum reaches kth.
// Returns true when found; *hit_lane and *residual (= kth minus the sum before that lane) are
// then uniform over the warp.  *total is the sum over the warp.
__device__ __forceinline__ bool warp_find_kth(uint32_t v, uint32_t kth, int lane, int* hit_lane,
                                              uint32_t* residual, uint32_t* total) {
  const uint32_t incl = warp_incl_scan(v, lane);
  *total = __shfl_sync(0xffffffffu, incl, 31);
  const uint32_t hits = __ballot_sync(0xffffffffu, incl >= kth);
  if (hits == 0u) return false;
  const int first = __ffs(hits) - 1;
  const uint32_t before = __shfl_sync(0xffffffffu, incl - v, first);
  *hit_lane = first;
  *residual = kth - before;
  return true;
}

// A tile's 16-channel blocks are taken NG groups of KB at a time (KB = 1, 2, 4; NG = 2 only with
// KB = 4, for more than 4 blocks), which bounds the registers the loads in flight need.
// ATTEND: the whole step; otherwise the step without its attention phase (large selections are
// attended by the split-K tensor-core kernel instead).
// PAGED: K, V and the proxy are page pools behind a block table (compiled separately, so that
// the contiguous form keeps its plain address arithmetic within 64 registers).
// NT: threads per CTA: 512 (two CTAs per SM) or 1024 (one CTA per SM with twice the slice).
// SCORES: TopK-I alone: the keys come from a score buffer instead of the proxy stream, and the kernel ends after the list.
template <int KB, int NG, bool ATTEND, bool PAGED = false, int NT = 512, bool SCORES = false>
__global__ void __launch_bounds__(NT, NT == 512 ? 2 : 1)
fused_decode_kernel(const FusedParams p) {
  constexpr int kFT = NT;                  // (shadow the file-level constants inside this kernel)
  constexpr int kFW = NT / 32;
  cg::cluster_group cluster = cg::this_cluster();
  const int cs = (int)cluster.num_blocks();
  const int crank = (int)cluster.block_rank();
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int u = blockIdx.y;
  const SelUnit su = sel_unit(u, p.n_sets, p.group, p.n_q_heads, p.n_kv_heads);
  const int h = su.h;
  const int b = su.b;

  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned long long s_wcnt[kFW];
  __shared__ uint32_t s_fin[3][kFinBins];          // histograms of the local finish (one per pass)
  __shared__ __align__(8) uint32_t s_gsum[3][2][kGroups];   // per radix pass: cluster-wide group sums, and those of the lower ranks (added by the peers)
  __shared__ uint32_t s_fine[3][2][32];            // per radix pass: the bins of the group that holds the kth key, same two sums
  __shared__ uint32_t s_mine[kGroups];             // this CTA's group sums of the current pass
  __shared__ uint32_t s_ncand, s_cgt, s_ceq;       // candidates found here; pushed keys of lower ranks above / equal to the threshold
  __shared__ int s_len_old;
  constexpr int GP = FASA_MAX_GROUP;     // query heads a KV head can serve
  __shared__ __align__(16) uint16_t s_qraw[GP][kRowPad];   // the unit's query rows as stored (operand of scoring and attention)
  __shared__ int16_t s_chan[8 * FASA_MAX_DOM / 4];               // the head's channel table
  __shared__ ClusterMergeSmem s_merge;                            // pushed by the cluster: the partial results this CTA finishes

  const int cap = (((p.max_len + cs - 1) / cs) + 31) & ~31;
  const FusedSmem sl = fused_smem_layout(cap, kFW);
  uint32_t* keys = reinterpret_cast<uint32_t*>(smem_raw + sl.keys);
  uint32_t* hist0 = reinterpret_cast<uint32_t*>(smem_raw + sl.hist0);
  uint32_t* hist1 = reinterpret_cast<uint32_t*>(smem_raw + sl.hist1);
  uint32_t* s_mask = reinterpret_cast<uint32_t*>(smem_raw + sl.mask);
  for (int i = tid; i < kFBins; i += kFT) { hist0[i] = 0u; hist1[i] = 0u; }
  for (int i = tid; i < 3 * kFinBins; i += kFT) (&s_fin[0][0])[i] = 0u;
  for (int i = tid; i < 3 * 2 * kGroups; i += kFT) (&s_gsum[0][0][0])[i] = 0u;
  for (int i = tid; i < 3 * 2 * 32; i += kFT) (&s_fine[0][0][0])[i] = 0u;
  if (tid == 0) { s_ncand = 0u; s_cgt = 0u; s_ceq = 0u; }
  // (all of this before the kernel ahead on the stream has ended: it touches this CTA's shared memory alone)
  pdl_wait_for_predecessor();

  // ---- slices -------------------------------------------------------------------------
  // Append-then-step: one thread reads the length for the whole CTA, so that the CTA's arrival
  // (below) certifies that it no longer needs the old value; the last CTA of the sequence to
  // arrive stores the new length.  Nothing waits on the counter.
  // Loads that depend on nothing are issued first, so their (cold) latencies overlap: the
  // length, this thread's 16 bytes of the unit's query rows and its entry of the channel table.
  // The scoring operand (query values at the dominant channels) is gathered from the staged
  // copies in shared memory after the set-up barrier: no load waits on another load's result.
  const bool append = !SCORES && p.k_new != nullptr;
  int len_raw = 0;
  if (!append || tid == 0) len_raw = p.seq_lens[b];
  uint4 q_stage = make_uint4(0u, 0u, 0u, 0u);
  if (!SCORES && tid < FASA_MAX_GROUP * (FASA_HEAD_DIM / 8) && tid / (FASA_HEAD_DIM / 8) < p.group)
    q_stage = *reinterpret_cast<const uint4*>(p.q + su.q0 * FASA_HEAD_DIM + tid * 8);
  int16_t chan_stage = -1;
  if (!SCORES && tid < p.chunks * 8) chan_stage = p.chan[h * p.chunks * 8 + tid];
  if (SCORES && p.q_len > 1) {
    const int t = (u % p.n_sets) / (p.n_sets / p.q_len);        // the query of this row
    if (len_raw >= 0 && len_raw <= p.max_len) len_raw = max(0, len_raw - (p.q_len - 1 - t));   // (a bad length is left for clamp_len to flag)
  }
  int len_old;
  if (append) {
    if (tid == 0) s_len_old = clamp_len(len_raw, p.max_len, p.status);
    __syncthreads();
    len_old = s_len_old;
  } else {
    len_old = clamp_len(len_raw, p.max_len, p.status);
  }
  const bool grows = append && len_old < p.max_len;
  const int len = len_old + (grows ? 1 : 0);
  if (append && tid == 0) {
    if (!grows && crank == 0) atomicOr(p.status, FASA_DEV_APPEND_FULL);
    __threadfence();
    const int total = p.n_sets * cs;
    if (atomicAdd(&p.arrive[b], 1) == total - 1) {
      p.seq_lens_w[b] = len;
      p.arrive[b] = 0;
    }
  }
  const int per = (((len + cs - 1) / cs) + 31) & ~31;          // <= the capacity the host sized
  const int c0 = min(len, crank * per);
  const int c1 = min(len, c0 + per);
  const int nloc = c1 - c0;
  // Phase shift.  A grid of several rounds of CTAs runs in lock-step: streams that run side by side
  // share HBM evenly and end together, after which all their CTAs select at the same time and HBM
  // idles for the length of a select chain, round after round.  Every second cluster of the FIRST
  // round therefore starts late by a little under half the time the round's streams take (its own
  // slice stands for the average; 6.4 bytes per ns is about what the memory delivers), which puts
  // the two halves of the machine out of phase for the rest of the launch: one half streams while
  // the other selects.  Measured: batch 16 at 64-128 K 177.9 -> 167.9 us, batch 32 at 64 K
  // 225.9 -> 189.2 us.  The wait is a sleep bounded by the clock; nothing is waited for.
  if (!SCORES && p.shift_ctas > 0 && (int)blockIdx.y < p.shift_clusters && (blockIdx.y & 1)) {
    const float ns = 0.45f * (float)p.shift_ctas * (float)nloc * (float)(p.chunks * 16) * (1.0f / 6400.0f);
    const unsigned long long want = (unsigned long long)fminf(ns, 200000.0f);
    unsigned long long t0, t1;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    do {
      __nanosleep(1000);
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
    } while (t1 - t0 < want);
  }

  const long long k_budget =
      p.budget > 0 ? (long long)p.budget : ((long long)(-p.budget) * len + 999) / 1000;
  const int sink = min(len, p.n_sink);
  const int n_forced = sink + min(p.n_recent, len - sink);
  long long ktot_ll = min((long long)len, (long long)n_forced + k_budget);
  if (ktot_ll > p.n_sel_max) {
    ktot_ll = p.n_sel_max;
    if (crank == 0 && tid == 0) atomicOr(p.status, FASA_DEV_NSEL_CLAMPED);
  }
  const uint32_t ktot = (uint32_t)ktot_ll;

  // The first proxy loads leave before the rest of the set-up (histogram clearing, query
  // staging, its barrier), whose latency they then hide.  A warp keeps about four 16-byte
  // loads per lane in flight (more do not raise what a warp can pull); the SM's bandwidth
  // comes from its 32 resident warps.  Only the CTA that is about to write the new token's
  // rows has to wait for them.
  constexpr int TPI = KB == 1 ? 4 : 2;                        // tiles per warp iteration (even)
  const ProxyGeom pg = proxy_geom(p.chunks);
  const int n_blocks = pg.n16 + pg.n8;
  const unsigned char* unit = p.proxy + (int64_t)su.kv * ((p.max_len + 15) >> 4) * pg.tile_bytes;
  float* srow = p.scores ? p.scores + (int64_t)u * p.max_len : nullptr;
  const int tiles_alloc = (p.max_len + 15) >> 4;
  // Paged caches: the block-table entries of the slice's pages go to shared memory first (over the selection's bit masks,
  // which come later), as the index in the pool of the page's first tile; only the first batch, which leaves before they are
  // there, reads the table itself.  (Looking each tile up in the table, a batch ahead of its loads, took 8 registers and the
  // issue slots of two 64-bit products per tile: 12 sequences of 3-28 K tokens in pages of 64 58.8 -> 52.0 us, 16 of 64-126 K
  // 218 -> 174 us; contiguous caches of those lengths 47.4 and 175 us.)
  uint32_t* s_pages = s_mask;
  const int page0 = PAGED ? (crank * per) >> p.pm.shift : 0;
  auto tile_at = [&](int T) {
    if constexpr (PAGED) {
      const int s = p.pm.shift - 4;
      const uint32_t first = s_pages[(min(T, (c1 - 1) >> 4) >> s) - page0];
      return p.proxy + (int64_t)(first + (uint32_t)(T & ((1 << s) - 1))) * pg.tile_bytes;
    } else {
      return unit + (int64_t)T * pg.tile_bytes;
    }
  };
  auto fetch = [&](uint4 (&a)[TPI][KB], int T, int grp) {
#pragma unroll
    for (int j = 0; j < TPI; ++j) load_tile<KB>(a[j], tile_at(T + j), pg, lane, (T + j) * 16 < c1, grp * KB);
  };
  const int step = kFW * TPI;
  int T = ((crank * per) >> 4) + warp * TPI;                  // slices start on a tile boundary
  const bool own_new = grows && c0 <= len_old && len_old < c1;
  uint4 a[TPI][KB];
  if (!SCORES && !own_new) {
    if constexpr (PAGED) {
#pragma unroll
      for (int j = 0; j < TPI; ++j)
        load_tile<KB>(a[j], p.proxy + proxy_tile_offset(p.pm, b, h, p.n_kv_heads, min(T + j, tiles_alloc - 1), tiles_alloc, pg.tile_bytes, nullptr),
                      pg, lane, (T + j) * 16 < c1);
    } else {
      fetch(a, T, 0);
    }
  }
  if constexpr (PAGED) {
    for (int i = tid; i < (nloc > 0 ? ((c1 - 1) >> p.pm.shift) - page0 + 1 : 0); i += kFT) {
      int page = page_of(p.pm, b, (page0 + i) << p.pm.shift);
      if (!page_ok(p.pm, page)) {
        atomicOr(p.status, FASA_DEV_PAGE_CLAMPED);
        page = 0;
      }
      s_pages[i] = (uint32_t)(page * p.n_kv_heads + h) << (p.pm.shift - 4);
    }
  }

  if (own_new) {
    // this CTA's slice holds the new row: K and V copies (16 lanes each) and the packed
    // dominant-FC pairs of the key (one lane per 16-byte chunk), as in fasa_kv_append.  When
    // several units share a KV head each writes the same values, and reads back its own.
    const uint16_t* ksrc = p.k_new + (int64_t)su.kv * FASA_HEAD_DIM;
    const ProxyGeom pg = proxy_geom(p.chunks);
    // where the row goes: the sequence's own cache, or (paged) the page of position len_old; a
    // table entry outside the pool drops the row
    int64_t koff = b * p.ksb + h * p.ksh + (int64_t)len_old * p.kst;
    int64_t voff = b * p.vsb + h * p.vsh + (int64_t)len_old * p.vst;
    int64_t poff = (int64_t)su.kv * ((p.max_len + 15) >> 4) * pg.tile_bytes;
    int prow = len_old;
    bool row_ok = true;
    if constexpr (PAGED) {
      const int page = page_of(p.pm, b, len_old);
      row_ok = page_ok(p.pm, page);
      if (!row_ok && tid == 0) atomicOr(p.status, FASA_DEV_PAGE_CLAMPED);
      prow = len_old & ((1 << p.pm.shift) - 1);
      koff = page * p.ksb + h * p.ksh + (int64_t)prow * p.kst;
      voff = page * p.vsb + h * p.vsh + (int64_t)prow * p.vst;
      poff = ((int64_t)page * p.n_kv_heads + h) * (1 << (p.pm.shift - 4)) * pg.tile_bytes;
    }
    if (!PAGED && p.ndchan != nullptr) {
      // Split (Algorithm 2), as in fasa_m_kv_append: the rows may lie in host memory, and cross the link while this kernel
      // selects.  A sink position, and every new one while a recent window is kept, goes to its resident slot too.
      const int slot = p.res.tags != nullptr && (len_old < p.res.n_sink || p.res.n_recent > 0) ? fasa_resident_slot(p.res, len_old) : -1;
      uint16_t* res_row = slot >= 0 ? p.res.rows + ((int64_t)su.kv * p.res.slots + slot) * 2 * FASA_HEAD_DIM : nullptr;
      uint16_t* k_row = p.k_w + ((int64_t)su.kv * p.max_len + len_old) * p.nd;
      const int16_t* nch = p.ndchan + h * p.nd;
      for (int i = tid; i < p.nd / 2; i += kFT) {
        const uint32_t w = ksrc[nch[2 * i]] | ((uint32_t)ksrc[nch[2 * i + 1]] << 16);
        *reinterpret_cast<uint32_t*>(k_row + 2 * i) = w;
        if (res_row) *reinterpret_cast<uint32_t*>(res_row + 2 * i) = w;
      }
      for (int i = tid; i < 4 * p.chunks; i += kFT) {
        const int16_t* ch = p.chan + h * p.chunks * 8 + 2 * i;
        const uint32_t w = ksrc[ch[0]] | ((uint32_t)ksrc[ch[1]] << 16);
        *reinterpret_cast<uint32_t*>(p.proxy_w + poff + proxy_word_offset(pg, prow, i)) = w;
        if (res_row) *reinterpret_cast<uint32_t*>(res_row + p.nd + 2 * i) = w;
      }
      if (tid < 16) {
        const uint4 x = *reinterpret_cast<const uint4*>(p.v_new + (int64_t)su.kv * FASA_HEAD_DIM + tid * 8);
        *reinterpret_cast<uint4*>(p.v_w + voff + tid * 8) = x;
        if (res_row) *reinterpret_cast<uint4*>(res_row + FASA_HEAD_DIM + tid * 8) = x;
      }
      if (tid == 0 && slot >= 0) p.res.tags[(int64_t)su.kv * p.res.slots_pad + slot] = len_old;
    } else if (!row_ok) {
    } else if (tid < 16) {
      *reinterpret_cast<uint4*>(p.k_w + koff + tid * 8) = *reinterpret_cast<const uint4*>(ksrc + tid * 8);
    } else if (tid < 32) {
      const int c = tid - 16;
      *reinterpret_cast<uint4*>(p.v_w + voff + c * 8) =
          *reinterpret_cast<const uint4*>(p.v_new + (int64_t)su.kv * FASA_HEAD_DIM + c * 8);
    } else if (tid - 32 < 4 * p.chunks) {
      const int w = tid - 32;                       // one dominant FC = one 4-byte channel pair
      const int16_t* ch = p.chan + h * p.chunks * 8 + 2 * w;
      const int ch0 = ch[0], ch1 = ch[1];
      const uint32_t lo = ch0 >= 0 ? ksrc[ch0] : 0u;
      const uint32_t hi = ch1 >= 0 ? ksrc[ch1] : 0u;
      *reinterpret_cast<uint32_t*>(p.proxy_w + poff + proxy_word_offset(pg, prow, w)) = lo | (hi << 16);
    }
  }
  if (!SCORES && tid < GP * (FASA_HEAD_DIM / 8))
    *reinterpret_cast<uint4*>(&s_qraw[tid / (FASA_HEAD_DIM / 8)][(tid % (FASA_HEAD_DIM / 8)) * 8]) = q_stage;
  if (!SCORES && tid < p.chunks * 8) s_chan[tid] = chan_stage;
  __syncthreads();
  // This CTA runs and its totals are cleared: the peers may add to them from now on.  Each CTA
  // waits for the others' arrival only when it is about to touch them, after its stream.
  cluster_arrive();
  ScoreFrag<KB> f[NG];
#pragma unroll
  for (int grp = 0; !SCORES && grp < NG; ++grp)
    load_score_b<KB>(f[grp], &s_qraw[0][0], s_chan, p.chunks, p.group, lane, grp * KB, kRowPad);

  // ---- 1. scoring stream -> keys + first histogram ------------------------------------------
  if constexpr (SCORES) {
    // four consecutive positions per thread
    const float* sin = p.scores + (int64_t)u * p.max_len;
    const bool vec_ok = (reinterpret_cast<uintptr_t>(sin) & 15) == 0;
    for (int i = c0 + tid * 4; i < c1; i += kFT * 4) {
      float sv[4] = {0.f, 0.f, 0.f, 0.f};
      if (vec_ok && i + 3 < c1) {
        const float4 v4 = *reinterpret_cast<const float4*>(sin + i);
        sv[0] = v4.x; sv[1] = v4.y; sv[2] = v4.z; sv[3] = v4.w;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (i + e < c1) sv[e] = sin[i + e];
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (i + e < c1) {
          const uint32_t key = fasa_item_key(sv[e], i + e, len, p.n_sink, p.n_recent);
          atomicAdd(&hist0[key >> 21], 1u);
          keys[i + e - c0] = key;
        }
      }
    }
  } else {
    if (own_new) fetch(a, T, 0);                              // (the new row is in place now)
    // The loop exists twice.  When the head's dominant channels fill whole 16-channel blocks and
    // exactly the KB x NG blocks this kernel is compiled for (4 n_dom = 32 KB NG: 8, 16, 32 or 64
    // FCs), a tile's loads and products need no run-time test of the geometry: the loads of a batch
    // then leave back to back, which is worth a quarter of what one SM can pull on its own.
    auto stream = [&](auto exact_tag) {
      constexpr bool EXACT = decltype(exact_tag)::value;
      auto fetch_x = [&](uint4 (&aa)[TPI][KB], int TT, int grp) {
        if constexpr (EXACT) {
#pragma unroll
          for (int j = 0; j < TPI; ++j) {
            const unsigned char* tile;
            if constexpr (PAGED) tile = tile_at(TT + j);
            else tile = unit + (int64_t)(TT + j) * (KB * NG * 512);
            const bool ok = (TT + j) * 16 < c1;
#pragma unroll
            for (int i = 0; i < KB; ++i)
              aa[j][i] = ok ? ld_proxy_u4(tile + (grp * KB + i) * 512 + lane * 16) : make_uint4(0u, 0u, 0u, 0u);
          }
        } else {
          fetch(aa, TT, grp);
        }
      };
      while (T * 16 < c1) {       // uniform over the warp
        float c[TPI][4];
#pragma unroll
        for (int j = 0; j < TPI; ++j) c[j][0] = c[j][1] = c[j][2] = c[j][3] = 0.f;
#pragma unroll
        for (int grp = 0; grp < NG; ++grp) {
#pragma unroll
          for (int j = 0; j < TPI; ++j) {
            if constexpr (EXACT) {
#pragma unroll
              for (int kb = 0; kb < KB; ++kb) mma_bf16_16816(c[j], a[j][kb], f[grp].b[kb]);
            } else {
              mma_tile<KB>(c[j], a[j], f[grp], n_blocks - grp * KB);
            }
          }
          // the registers are free again: the next group, or the next batch of tiles, at once
          if (grp + 1 < NG) fetch_x(a, T, grp + 1);
          else if ((T + step) * 16 < c1) fetch_x(a, T + step, 0);
        }
#pragma unroll
        for (int pr = 0; pr < TPI / 2; ++pr) {
          float a_lo, a_hi, b_lo, b_hi, sc;
          if (p.max_reduce) {     // uniform
            reduce_heads<true>(c[2 * pr], p.group, lane, a_lo, a_hi);
            reduce_heads<true>(c[2 * pr + 1], p.group, lane, b_lo, b_hi);
          } else {
            reduce_heads<false>(c[2 * pr], p.group, lane, a_lo, a_hi);
            reduce_heads<false>(c[2 * pr + 1], p.group, lane, b_lo, b_hi);
          }
          const int row = (T + 2 * pr) * 16 + pick_row_of_pair(lane, a_lo, a_hi, b_lo, b_hi, sc);
          if (row < c1) {
            const uint32_t key = fasa_item_key(sc, row, len, p.n_sink, p.n_recent);
            atomicAdd(&hist0[key >> 21], 1u);
            keys[row - c0] = key;
            if (srow) srow[row] = sc;
          }
        }
        T += step;
      }
    };
    if (pg.n8 == 0 && pg.n16 == KB * NG) stream(std::true_type{});
    else stream(std::false_type{});
  }
  // At most one CTA per SM: the next kernel's launch and set-up may overlap what follows, which leaves most of the SM idle.
  // (With more rounds its CTAs would take the places of those still to come: 174 -> 203 us at batch 16, 64-128 K.)
  if (ATTEND && p.early) pdl_release_successor();
  __syncthreads();

  // ---- 2. radix select of the ktot-th largest key ------------------------------------------
  // Every value that steers this phase (the bin found, the keys still wanted from it, the
  // number of keys it holds) is computed by every warp of every CTA from the same cluster-wide
  // integer sums, hence identical everywhere: loops and barriers end for the whole cluster at
  // once.  `lower_gt` / `lower_eq` count, over the lower-ranked CTAs, the keys above the
  // threshold found so far and the keys equal to it: the compaction's cluster-wide prefix.
  cluster_wait();               // (set-up barrier, second half: every peer has started and cleared its totals)
  uint32_t prefix = 0, kth = ktot, thr = 0, tie_quota = 0, lower_gt = 0, lower_eq = 0;
  bool done = false;            // thr and tie_quota are final
  bool peers_idle = false;      // a barrier has passed since the last access to a peer's memory
  bool have_masks = false;      // s_mask already holds (higher bins, candidates) per block of 128 keys
  // Bit masks over the keys: word w covers keys 32 w .. 32 w + 31.  A warp owns a contiguous run
  // of words, a lane one word of every 32 of them: after the first pass over the keys all work
  // is per word, without ballots.
  const int n_words = (nloc + 31) >> 5;
  const int words_per_warp = (n_words + kFW - 1) / kFW;
  const int w0 = min(n_words, warp * words_per_warp), w1 = min(n_words, w0 + words_per_warp);
  uint32_t* s_mg = s_mask;                       // keys above the threshold (first: in higher bins)
  uint32_t* s_me = s_mask + (cap / 32 + 1);      // keys equal to it (first: the candidates)
#pragma unroll 1
  for (int pass = 0; pass < 3 && !done; ++pass) {
    const int bits = pass == 2 ? 10 : 11;
    const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
    const int nb = 1 << bits;
    const int ng = nb / 32;
    uint32_t* buf = (pass & 1) ? hist1 : hist0;
    if (pass > 0) {
      if (pass == 2) {          // (hist0: its remote readers of pass 0 are past the barrier of pass 1)
        for (int i = tid; i < nb; i += kFT) buf[i] = 0u;
        __syncthreads();
      }
#pragma unroll 4
      for (int i = tid * 4; i < nloc; i += kFT * 4) {
        const uint4 kq = *reinterpret_cast<const uint4*>(&keys[i]);
        const uint32_t kv[4] = {kq.x, kq.y, kq.z, kq.w};
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (i + e < nloc && (kv[e] >> (shift + bits)) == prefix)
            atomicAdd(&buf[(kv[e] >> shift) & (uint32_t)(nb - 1)], 1u);
      }
      __syncthreads();
    }
    {
      // Group sums: each warp reduces its groups side by side; after a block barrier warp r
      // ADDS them into CTA r's totals (coalesced remote atomics, zeros skipped: scores crowd
      // into few groups), and into CTA r's totals of lower ranks if this CTA ranks below r.
      // After the cluster barrier every CTA holds the cluster-wide sums, already reduced.
      constexpr int GPW = kGroups / kFW;
      uint32_t v[GPW];
#pragma unroll
      for (int j = 0; j < GPW; ++j) {
        const int g = warp + j * kFW;
        v[j] = g < ng ? buf[g * 32 + lane] : 0u;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < GPW; ++j) v[j] += __shfl_xor_sync(0xffffffffu, v[j], o);
      if (lane == 0) {
#pragma unroll
        for (int j = 0; j < GPW; ++j) s_mine[warp + j * kFW] = v[j];
      }
      __syncthreads();
      if (warp < cs) {
        uint32_t* tot = cluster.map_shared_rank(&s_gsum[pass][0][0], warp);
        uint32_t* low = cluster.map_shared_rank(&s_gsum[pass][1][0], warp);
#pragma unroll
        for (int j = 0; j < kGroups / 32; ++j) {
          const uint32_t x = s_mine[lane + 32 * j];
          if (x) {
            atomicAdd(tot + lane + 32 * j, x);
            if (crank < warp) atomicAdd(low + lane + 32 * j, x);
          }
        }
      }
    }
    cluster.sync();   // one per radix pass: all group sums have arrived, all histograms are complete

    // (a) every warp finds the group of 32 bins that holds the kth key from the local totals:
    // lane l owns groups 63 - 2 l and 62 - 2 l (highest first)
    uint32_t res, above_lower;                 // above_lower: keys of lower ranks in higher bins
    int group_id;
    {
      const uint2 t2 = *reinterpret_cast<const uint2*>(&s_gsum[pass][0][kGroups - 2 - 2 * lane]);   // (.y, .x) = (first, second)
      const uint2 l2 = *reinterpret_cast<const uint2*>(&s_gsum[pass][1][kGroups - 2 - 2 * lane]);
      int hit = 31;
      uint32_t tot = 0;
      res = 1;
      if (!warp_find_kth(t2.x + t2.y, kth, lane, &hit, &res, &tot)) { hit = 31; res = 1; }   // cannot fail: kth <= number of keys
      above_lower = __reduce_add_sync(0xffffffffu, lane < hit ? l2.x + l2.y : 0u);
      const uint32_t first = __shfl_sync(0xffffffffu, t2.y, hit), first_low = __shfl_sync(0xffffffffu, l2.y, hit);
      group_id = kGroups - 1 - 2 * hit;
      if (first < res) {
        res -= first;
        above_lower += first_low;
        --group_id;
      }
    }
    // (b) warp r fetches the 32 bins of that group from CTA r (one transaction) and adds them to
    // the block's totals; after a block barrier every warp locates the bin
    if (warp < cs) {
      const uint32_t x = cluster.map_shared_rank(buf, warp)[group_id * 32 + 31 - lane];   // lane 0 = highest bin
      if (x) {
        atomicAdd(&s_fine[pass][0][lane], x);
        if (warp < crank) atomicAdd(&s_fine[pass][1][lane], x);
      }
    }
    __syncthreads();
    uint32_t in_bin, bin_lower;                // keys in the bin: cluster-wide / in lower ranks
    {
      const uint32_t v = s_fine[pass][0][lane], vl = s_fine[pass][1][lane];
      int hit = 31;
      uint32_t tot = 0, res2 = 1;
      if (!warp_find_kth(v, res, lane, &hit, &res2, &tot)) { hit = 31; res2 = 1; }
      in_bin = __shfl_sync(0xffffffffu, v, hit);
      bin_lower = __shfl_sync(0xffffffffu, vl, hit);
      above_lower += __reduce_add_sync(0xffffffffu, lane < hit ? vl : 0u);
      prefix = (prefix << bits) | (uint32_t)(group_id * 32 + 31 - hit);
      kth = res2;
    }
    lower_gt += above_lower;
    peers_idle = false;

    if (in_bin == kth) {            // every key of this bin is selected: its other bits do not matter
      thr = prefix << shift;
      tie_quota = 0xffffffffu;
      lower_gt += bin_lower;
      done = true;
    } else if (pass == 2) {         // all 32 bits are fixed: the bin holds the keys equal to the threshold
      thr = prefix;
      tie_quota = kth;
      lower_eq = bin_lower;
      done = true;
    } else if (in_bin <= (uint32_t)kCandCap) {
      // ---- few keys share this prefix: every CTA gets all of them and finishes on its own ----
      // CTA r's keys occupy [sum of lower ranks' counts, + its own count) of every copy.
      uint32_t* cand = reinterpret_cast<uint32_t*>(smem_raw + (pass == 0 ? sl.hist1 : sl.spare));
      // One pass over the keys: masks of the keys in higher bins (selected for certain) and of
      // the keys in this bin (the candidates, decided once the threshold is known); then the
      // candidates themselves are appended, with one counter update per warp.
      have_masks = true;
      {
        uint32_t cnt = 0;
#pragma unroll 4
        for (int w = w0; w < w1; ++w) {
          const int i = 32 * w + lane;
          const uint32_t top = keys[i] >> shift;
          const uint32_t ma = __ballot_sync(0xffffffffu, i < nloc && top > prefix);
          const uint32_t mc = __ballot_sync(0xffffffffu, i < nloc && top == prefix);
          if (lane == 0) { s_mg[w] = ma; s_me[w] = mc; }
          cnt += __popc(mc);
        }
        uint32_t base = 0;
        if (lane == 0 && cnt) base = atomicAdd(&s_ncand, cnt);
        base = __shfl_sync(0xffffffffu, base, 0) + bin_lower;
        __syncwarp();
        for (int wb = w0; wb < w1; wb += 32) {     // uniform over the warp
          const int w = wb + lane;
          uint32_t m = w < w1 ? s_me[w] : 0u;
          const uint32_t c = __popc(m), incl = warp_incl_scan(c, lane);
          uint32_t slot = base + incl - c;
          base += __shfl_sync(0xffffffffu, incl, 31);
          while (m) {
            const int j = __ffs(m) - 1;
            m &= m - 1;
            if (slot < (uint32_t)kCandCap) cand[slot] = keys[32 * w + j];
            ++slot;
          }
        }
      }
      __syncthreads();
      if (warp < cs && warp != crank) {          // this CTA's run of keys, to CTA `warp`, coalesced
        const uint32_t n_own = min(s_ncand, (uint32_t)kCandCap - min(bin_lower, (uint32_t)kCandCap));
        uint32_t* dst = cluster.map_shared_rank(cand, warp) + bin_lower;
        for (uint32_t i = lane; i < n_own; i += 32) dst[i] = cand[bin_lower + i];
      }
      cluster.sync();   // every CTA holds every candidate; no peer is touched from here to the merge
      peers_idle = true;
      // block-level radix passes over the remaining `shift` bits, kFinBits at a time; every
      // warp scans the small histogram itself, so a pass costs one block barrier
      int rem = shift;
#pragma unroll 1
      for (int fp = 0; rem > 0 && !done; ++fp) {
        const int wbits = rem < kFinBits ? rem : kFinBits;
        const int sh = rem - wbits;
        uint32_t* fh = s_fin[fp];
        for (int i = tid; i < (int)in_bin; i += kFT) {
          const uint32_t key = cand[i];
          if ((key >> rem) == prefix) atomicAdd(&fh[(key >> sh) & (uint32_t)((1 << wbits) - 1)], 1u);
        }
        __syncthreads();
        // lane l owns the four bins 127 - 4 l .. 124 - 4 l (highest first)
        uint32_t c4[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) c4[j] = fh[kFinBins - 1 - 4 * lane - j];
        int hit = 0;
        uint32_t res2 = 1, tot = 0;
        if (!warp_find_kth(c4[0] + c4[1] + c4[2] + c4[3], kth, lane, &hit, &res2, &tot)) { hit = 0; res2 = 1; }
        uint32_t digit = 0, cnt = 0;
        bool found = false;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t c = __shfl_sync(0xffffffffu, c4[j], hit);
          if (!found) {
            if (c >= res2) { digit = (uint32_t)(kFinBins - 1 - 4 * hit - j); cnt = c; found = true; }
            else res2 -= c;
          }
        }
        prefix = (prefix << wbits) | digit;
        kth = res2;
        rem = sh;
        if (cnt == kth && rem > 0) {     // the rest of this bin is selected whole
          thr = prefix << rem;
          tie_quota = 0xffffffffu;
          done = true;
        }
      }
      if (!done) {
        thr = prefix;
        tie_quota = kth;
        done = true;
      }
      // pushed keys of the lower-ranked CTAs against the threshold (they lie in [0, bin_lower))
      {
        uint32_t ngt = 0, neq = 0;
        for (int i = tid; i < (int)bin_lower; i += kFT) {
          const uint32_t key = cand[i];
          ngt += key > thr ? 1u : 0u;
          neq += key == thr ? 1u : 0u;
        }
        ngt = __reduce_add_sync(0xffffffffu, ngt);
        neq = __reduce_add_sync(0xffffffffu, neq);
        if (lane == 0 && (ngt | neq)) { atomicAdd(&s_cgt, ngt); atomicAdd(&s_ceq, neq); }
      }
    }
  }
  // The attention phase reuses the histograms, and a CTA of the select-only forms may leave:
  // both only once no peer can still be reading this CTA's bins.
  if (!peers_idle) cluster.sync();

  // ---- 3. ascending compaction ---------------------------------------------------------------
  // (a) the masks of the keys above / equal to the threshold: from the keys (ballots), or,
  // where the select phase has left the masks of the higher bins and of the candidates, by
  // looking at the candidates alone, each lane at the bits of its own words; (b) the warps'
  // totals give each warp its offset (one block barrier); (c) every lane turns the set bits of
  // its words into positions of the index list (prefix over the lanes by shuffles).  Equal
  // keys are taken lowest index first, so the result equals a stable sort.
  {
    uint32_t g_tot = 0, e_tot = 0;
    if (have_masks) {
      for (int w = w0 + lane; w < w1; w += 32) {
        uint32_t mc = s_me[w], mg = s_mg[w], me = 0u;
        while (mc) {
          const int j = __ffs(mc) - 1;
          mc &= mc - 1;
          const uint32_t key = keys[32 * w + j];
          if (key > thr) mg |= 1u << j;
          else if (key == thr) me |= 1u << j;
        }
        s_mg[w] = mg;
        s_me[w] = me;
        g_tot += __popc(mg);
        e_tot += __popc(me);
      }
      g_tot = __reduce_add_sync(0xffffffffu, g_tot);
      e_tot = __reduce_add_sync(0xffffffffu, e_tot);
    } else {
#pragma unroll 4
      for (int w = w0; w < w1; ++w) {
        const int i = 32 * w + lane;
        const uint32_t key = keys[i];
        const uint32_t mg = __ballot_sync(0xffffffffu, i < nloc && key > thr);
        const uint32_t me = __ballot_sync(0xffffffffu, i < nloc && key == thr);
        if (lane == 0) { s_mg[w] = mg; s_me[w] = me; }
        g_tot += __popc(mg);
        e_tot += __popc(me);
      }
    }
    if (lane == 0) s_wcnt[warp] = ((unsigned long long)g_tot << 32) | e_tot;
  }
  __syncthreads();            // the warps' totals; the candidate counts of the select phase
  uint32_t g_run, e_run;        // selected keys before this warp's run: above / equal to the threshold
  {
    static_assert(kFW <= 32, "one lane per warp total");
    const unsigned long long mine = lane < kFW ? s_wcnt[lane] : 0ull;
    unsigned long long incl = mine;
#pragma unroll
    for (int o = 1; o < kFW; o <<= 1) {
      const unsigned long long t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    const unsigned long long before = __shfl_sync(0xffffffffu, incl - mine, warp);
    const unsigned long long all = __shfl_sync(0xffffffffu, incl, kFW - 1);
    // selected tokens of the lower-ranked CTAs: from the bin counts and the pushed keys that
    // the select phase has seen, no barrier needed
    const uint32_t gb = lower_gt + s_cgt, eb = lower_eq + s_ceq;
    g_run = gb + (uint32_t)(before >> 32);
    e_run = eb + (uint32_t)before;
  }
  {
    int32_t* out_idx = p.idx + (int64_t)u * p.n_sel_max;
    for (int wb = w0; wb < w1; wb += 32) {         // uniform over the warp
      const int w = wb + lane;
      const uint32_t mg = w < w1 ? s_mg[w] : 0u, me = w < w1 ? s_me[w] : 0u;
      // counts of the lower lanes' words, packed (a word holds at most 32 keys, a CTA < 65536)
      const uint32_t cnt = (__popc(mg) << 16) | __popc(me), incl = warp_incl_scan(cnt, lane);
      uint32_t g_before = g_run + ((incl - cnt) >> 16), e_before = e_run + ((incl - cnt) & 0xffffu);
      const uint32_t all = __shfl_sync(0xffffffffu, incl, 31);
      g_run += all >> 16;
      e_run += all & 0xffffu;
      uint32_t m = mg | me;
      while (m) {
        const int j = __ffs(m) - 1;
        m &= m - 1;
        // (positions are < ktot by construction; the comparison keeps a write inside the
        // list whatever the scores hold)
        uint32_t pos = 0xffffffffu;
        if ((mg >> j) & 1u) { pos = g_before + min(e_before, tie_quota); ++g_before; }
        else { if (e_before < tie_quota) pos = g_before + e_before; ++e_before; }
        if (pos < ktot) out_idx[pos] = c0 + 32 * w + j;
      }
    }
    if (crank == 0 && tid == 0) p.n_sel[u] = (int32_t)ktot;
  }
  if constexpr (!ATTEND) return;   // (no peer reads this CTA's memory after the selection's last barrier)

  // ---- 4. attention over this CTA's share of the selected rows -----------------------------
  // Tensor cores, eight rows per warp step, 64 registers per thread.  What bounds this phase is the gather itself once the
  // instructions are out of the way: an FMA form (four rows and four heads per step, so two passes for groups of 5-8) spent
  // ~250 instructions per step and was bound by their issue.
  //   - K and V rows go to the warp's two buffers in shared memory (cp.async, rows padded so that ldmatrix is free of bank
  //     conflicts): the next step's K rows leave when this step's logits are done, its V rows after the output product.
  //   - logits: A = q, bf16 as stored (heads in rows 0-7), B = K rows; the softmax scale is applied to the fp32 result, whose
  //     fragment (head lane / 4, rows 2 t and 2 t + 1) is already the B operand of
  //   - out^T: A = V^T (ldmatrix.trans), B = P^T, with p split into three bf16 terms that add up to all its 24 bits: the
  //     first two as the two halves of one k = 16 product (A holds the same eight rows twice), the third with k = 8.
  constexpr int R = 8;
  // The selected tokens are dealt out evenly: CTA r attends to rows [r, r + 1) * ktot / cs of the
  // index list, whoever selected them (scores cluster by position, so the CTAs' own selections
  // can differ several times in size); this costs one cluster barrier, after which the list
  // written by the peers is visible.
  cluster.sync();               // the index list is complete
  const int a0 = (int)(((long long)ktot * crank) / cs);
  const int a1 = (int)(((long long)ktot * (crank + 1)) / cs);
  // The attention phase's working arrays take over the key / histogram area: every read of
  // it, local or remote, happened before the selection's last barrier or the block barrier above.
  unsigned char* ring = smem_raw + sl.ring + warp * kAttSlot;      // K rows, then V rows; at the end the warp's [8][kAccStride] accumulators
  uint16_t (*k_rows)[kRowPad] = reinterpret_cast<uint16_t (*)[kRowPad]>(ring);
  uint16_t (*v_rows)[kRowPad] = k_rows + R;
  float (*s_part)[kPartStride + 2] = reinterpret_cast<float (*)[kPartStride + 2]>(smem_raw + sl.part);
  float (*s_m)[GP] = reinterpret_cast<float (*)[GP]>(smem_raw + sl.m);
  float (*s_l)[GP] = reinterpret_cast<float (*)[GP]>(smem_raw + sl.l);
  const int n_active = min(kFW, (a1 - a0 + R - 1) / R);           // warps that get rows
  if (warp < n_active) {
    const int g = lane >> 2, t = lane & 3;
    const int32_t* irow = p.idx + (int64_t)u * p.n_sel_max;
    const uint16_t* kbase = p.k + h * p.ksh + (PAGED ? 0 : b * p.ksb) + (lane & 15) * 8;
    const uint16_t* vbase = p.v + h * p.vsh + (PAGED ? 0 : b * p.vsb) + (lane & 15) * 8;
    float acc[FASA_HEAD_DIM / 16][4];         // out^T: [16-channel block][frag], heads 2 t and 2 t + 1
#pragma unroll
    for (int cb = 0; cb < FASA_HEAD_DIM / 16; ++cb) acc[cb][0] = acc[cb][1] = acc[cb][2] = acc[cb][3] = 0.f;
    float m_run = -INFINITY, l_run = 0.f;     // of head g (the sum: over this lane's rows only)
    // 32 entries of the list at a time, lane 8 s + r holding row r of the warp's s-th step from here on (rows past the end
    // repeat the last one and are masked below); on paged caches as the row of the pool.
    int listed = 0;
    auto list_rows = [&](int base) {
      const int i = __ldcg(irow + min(base + (lane >> 3) * (kFW * R) + (lane & 7), a1 - 1));
      listed = min(max(i, 0), p.max_len - 1);
      if constexpr (PAGED) listed = pool_row(p.pm, b, listed, p.status);
    };
    // lane l copies the 16 bytes l % 16 of rows 2 i + l / 16 of step s
    auto stage = [&](uint16_t (*dst)[kRowPad], const uint16_t* unit_rows, int64_t sb, int64_t st, int s) {
#pragma unroll
      for (int i = 0; i < R / 2; ++i) {
        const int r = __shfl_sync(0xffffffffu, listed, (s & 3) * R + 2 * i + (lane >> 4));
        const int64_t off = PAGED ? (r >> p.pm.shift) * sb + (r & ((1 << p.pm.shift) - 1)) * st : r * st;
        uint16_t* to = &dst[2 * i + (lane >> 4)][(lane & 15) * 8];
        if (!PAGED && p.host_rows) cp_async16_ca(to, unit_rows + off);
        else cp_async16(to, unit_rows + off);
      }
    };
    int base = a0 + warp * R;
    list_rows(base);
    stage(k_rows, kbase, p.ksb, p.kst, 0);
    cp_async_commit();
    stage(v_rows, vbase, p.vsb, p.vst, 0);
    cp_async_commit();
    for (int s = 0; base < a1; ++s, base += kFW * R) {
      const bool more = base + kFW * R < a1;                       // uniform over the warp
      cp_async_wait<1>();                                          // the K rows
      __syncwarp();
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int i = 0; i < FASA_HEAD_DIM / 32; ++i) {
        uint32_t qa[4], kb[4];
        ldmatrix_x4(qa, &s_qraw[lane & 7][(4 * i + (lane >> 3)) * 8]);
        ldmatrix_x4(kb, &k_rows[lane & 7][(4 * i + (lane >> 3)) * 8]);
        const uint32_t a_lo[4] = {qa[0], 0u, qa[1], 0u}, a_hi[4] = {qa[2], 0u, qa[3], 0u};
        mma16816(c, a_lo, kb[0], kb[1]);
        mma16816(c, a_hi, kb[2], kb[3]);
      }
      __syncwarp();
      if (more) {
        if (((s + 1) & 3) == 0) list_rows(base + kFW * R);
        stage(k_rows, kbase, p.ksb, p.kst, s + 1);
      }
      cp_async_commit();
      const float x0 = base + 2 * t < a1 ? c[0] * p.scale_log2 : -INFINITY;
      const float x1 = base + 2 * t + 1 < a1 ? c[1] * p.scale_log2 : -INFINITY;
      float bmax = fmaxf(x0, x1);
      bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, 1));
      bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, 2));
      const float m_new = fmaxf(m_run, bmax);
      const float m_safe = m_new == -INFINITY ? 0.f : m_new;
      const float alpha = exp2f(m_run - m_safe);
      const float p0 = exp2f(x0 - m_safe), p1 = exp2f(x1 - m_safe);
      l_run = l_run * alpha + (p0 + p1);
      if (__any_sync(0xffffffffu, m_new != m_run)) {
        const float al0 = __shfl_sync(0xffffffffu, alpha, 8 * t), al1 = __shfl_sync(0xffffffffu, alpha, 8 * t + 4);
#pragma unroll
        for (int cb = 0; cb < FASA_HEAD_DIM / 16; ++cb) {
          acc[cb][0] *= al0; acc[cb][1] *= al1; acc[cb][2] *= al0; acc[cb][3] *= al1;
        }
      }
      m_run = m_new;
      const uint32_t p_1 = pack_bf16(p0, p1);
      const float2 f1 = bf16x2_to_f32x2(p_1);
      const float r0 = p0 - f1.x, r1 = p1 - f1.y;
      const uint32_t p_2 = pack_bf16(r0, r1);
      const float2 f2 = bf16x2_to_f32x2(p_2);
      const uint32_t p_3 = pack_bf16(r0 - f2.x, r1 - f2.y);
      cp_async_wait<1>();                                          // the V rows
      __syncwarp();
#pragma unroll
      for (int i = 0; i < FASA_HEAD_DIM / 32; ++i) {
        uint32_t va[4];
        ldmatrix_x4_trans(va, &v_rows[lane & 7][(4 * i + (lane >> 3)) * 8]);
        const uint32_t a_lo[4] = {va[0], va[1], va[0], va[1]}, a_hi[4] = {va[2], va[3], va[2], va[3]};
        mma16816(acc[2 * i], a_lo, p_1, p_2);
        mma16816(acc[2 * i + 1], a_hi, p_1, p_2);
        mma1688(acc[2 * i], va[0], va[1], p_3);
        mma1688(acc[2 * i + 1], va[2], va[3], p_3);
      }
      __syncwarp();
      if (more) stage(v_rows, vbase, p.vsb, p.vst, s + 1);
      cp_async_commit();
    }
    cp_async_wait<0>();
    // ---- 5a. combine the warps of this CTA -------------------------------------------------
    float* s_acc = reinterpret_cast<float*>(ring);
#pragma unroll
    for (int cb = 0; cb < FASA_HEAD_DIM / 16; ++cb) {
      float* o = s_acc + 2 * t * kAccStride + cb * 16 + g;
      o[0] = acc[cb][0];
      o[kAccStride] = acc[cb][1];
      o[8] = acc[cb][2];
      o[kAccStride + 8] = acc[cb][3];
    }
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
    l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
    if (t == 0) {
      s_m[warp][g] = m_run;
      s_l[warp][g] = l_run;
    }
  }
  __syncthreads();
  for (int o = tid; o < p.group * FASA_HEAD_DIM; o += kFT) {
    const int g = o / FASA_HEAD_DIM, c = o % FASA_HEAD_DIM;       // (g: uniform over the warp)
    // lane w: the weight of warp w's partial result
    const float ms = lane < n_active ? s_m[lane][g] : -INFINITY;
    float mx = ms;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    const float wt = ms == -INFINITY ? 0.f : exp2f(ms - mx);
    float av = 0.f;
    const float* acc_o = reinterpret_cast<const float*>(smem_raw + sl.ring) + g * kAccStride + c;
    for (int w = 0; w < n_active; ++w) av += __shfl_sync(0xffffffffu, wt, w) * acc_o[w * (kAttSlot / 4)];
    s_part[g][2 + c] = av;
    if (c < 32) {
      float l = lane < n_active ? wt * s_l[lane][g] : 0.f;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
      if (c == 0) {
        s_part[g][0] = mx;
        s_part[g][1] = l;
      }
    }
  }
  __syncthreads();
  // ---- 5b. merge across the cluster (one barrier; see fasa_cluster_merge.cuh) -------------------
  cluster_merge_store<kFT>(cluster, s_part, s_merge, p.group, su.q0, p.out, p.out_mirror, p.lse, [&](int g) {
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
}

size_t fused_smem_bytes(int cap) { return (size_t)fused_smem_layout(cap).total; }

using FusedFn = void (*)(const FusedParams);

template <bool ATTEND, bool PAGED>
FusedFn fused_variant(int chunks) {
  const int nb = (chunks + 1) / 2;      // 16-channel blocks per tile, the 8-channel one included
  if (nb <= 1) return fused_decode_kernel<1, 1, ATTEND, PAGED>;
  if (nb <= 2) return fused_decode_kernel<2, 1, ATTEND, PAGED>;
  if (nb <= 4) return fused_decode_kernel<4, 1, ATTEND, PAGED>;
  return fused_decode_kernel<4, 2, ATTEND, PAGED>;
}

FusedFn fused_fn(int chunks, bool paged = false) {
  return paged ? fused_variant<true, true>(chunks) : fused_variant<true, false>(chunks);
}

// The wide form of the step: 1024 threads, one CTA per SM.
template <bool ATTEND, bool PAGED>
FusedFn wide_variant(int chunks) {
  const int nb = (chunks + 1) / 2;
  if (nb <= 1) return fused_decode_kernel<1, 1, ATTEND, PAGED, 1024>;
  if (nb <= 2) return fused_decode_kernel<2, 1, ATTEND, PAGED, 1024>;
  if (nb <= 4) return fused_decode_kernel<4, 1, ATTEND, PAGED, 1024>;
  return fused_decode_kernel<4, 2, ATTEND, PAGED, 1024>;
}
FusedFn wide_fn(int chunks, bool paged) { return paged ? wide_variant<true, true>(chunks) : wide_variant<true, false>(chunks); }
FusedFn wide_select_fn(int chunks, bool paged) { return paged ? wide_variant<false, true>(chunks) : wide_variant<false, false>(chunks); }
FusedFn topk_fn() { return fused_decode_kernel<1, 1, false, false, 512, true>; }
constexpr int kCapWide = 40960;        // keys a 1024-thread CTA can hold (one CTA per SM)

FusedFn select_fn(int chunks, bool paged = false) {         // the step without attention
  return paged ? fused_variant<false, true>(chunks) : fused_variant<false, false>(chunks);
}

}  // namespace

// Decides once per context whether and how the fused kernel runs: the smallest cluster whose
// CTAs can hold their slice of max_len keys, grown while that leaves SMs idle, then shrunk
// again if the device cannot co-schedule a cluster of that size.
int fasa_fused_plan(fasa_ctx* ctx) {
  const fasa_config_t& c = ctx->cfg;
  ctx->fused_cs = 0;
  ctx->fused_smem = 0;
  ctx->fused_step_ok = 1;
  const int units = c.batch * ctx->n_sets;
  const bool paged = c.page_size > 0;
  FusedFn fn = fused_fn(ctx->chunks, paged);
  auto cap_of = [&](int cs) { return (((c.max_len + cs - 1) / cs) + 31) & ~31; };
  // Two CTAs per SM can be resident; a cluster is doubled while the whole grid still fits in one wave of them and the slices
  // are worth it: at least 512 tokens, 2560 for clusters of 16, whose barriers cost more than their stream saves (8 units at
  // 12 K: 18.6 us with 16, 16.1 with 8; at 25 K 20.5 / 18.9; at 60 K 24.0 / 25.5), and beyond one CTA per SM only from slices
  // of 4608 on (20 units: at 6 K 23.1 us with 8 CTAs each or half as many wide ones, 20.2 with 4; at 12 K 24.5 / 22.4; at
  // 25 K 27.5 / 27.2; at 50 K 33.0 / 34.7).
  const int slots = 2 * ctx->n_sm;
  int want = 1;
  while (want < 16 && cap_of(want) > kCapPair) want *= 2;
  while (want < 16 && units * want * 2 <= slots && c.max_len / (2 * want) >= (want == 8 ? 2560 : 512) &&
         (units * want * 2 <= ctx->n_sm || c.max_len / want >= 4608))
    want *= 2;
  if (cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    if (want > 8) want = 8;
  }
  // Clusters of the wide form with half of cs CTAs that the device holds at once; 0 where it is not available.
  auto wide_clusters = [&](int cs) -> int {
    if (cs < 4 || cap_of(cs / 2) > kCapWide) return 0;
    const int limit_w = (int)fused_smem_layout(kCapWide, 32).total;
    FusedFn fw = wide_fn(ctx->chunks, paged), fs = wide_select_fn(ctx->chunks, paged);
    cudaLaunchConfig_t cw;
    memset(&cw, 0, sizeof(cw));
    cw.gridDim = dim3((unsigned)(cs / 2), (unsigned)units, 1);
    cw.blockDim = dim3(1024, 1, 1);
    cw.dynamicSmemBytes = (size_t)fused_smem_layout(cap_of(cs / 2), 32).total;
    cudaLaunchAttribute aw[1];
    aw[0].id = cudaLaunchAttributeClusterDimension;
    aw[0].val.clusterDim.x = (unsigned)(cs / 2);
    aw[0].val.clusterDim.y = 1;
    aw[0].val.clusterDim.z = 1;
    cw.attrs = aw;
    cw.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute((const void*)fw, cudaFuncAttributeMaxDynamicSharedMemorySize, limit_w) == cudaSuccess &&
        cudaFuncSetAttribute((const void*)fs, cudaFuncAttributeMaxDynamicSharedMemorySize, limit_w) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n, (const void*)fw, &cw) == cudaSuccess)
      return n;
    cudaGetLastError();
    return 0;
  };
  for (int cs = want; cs >= 1; cs /= 2) {
    const int cap = cap_of(cs);
    if (cap > kCapMax) break;
    const size_t smem = fused_smem_bytes(cap);
    // The opt-in limit is a property of the kernel, shared by every context of the process:
    // it is set to the most any context can ask for, not to what this one needs.
    const int smem_limit = (int)fused_smem_bytes(kCapMax);
    if (cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)cs, (unsigned)units, 1);
    cfg.blockDim = dim3(kFT, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n_clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&n_clusters, (const void*)fn, &cfg) != cudaSuccess || n_clusters < 1) {
      cudaGetLastError();
      continue;
    }
    // A grid meant for one wave whose clusters do not all fit at once (a cluster lives on one GPC, so wide ones leave
    // SMs over) would run a second round for the last few: half the cluster size instead.  Likewise the wide form below is
    // taken only if it holds every unit or the narrow one does not either.  16 units at 25 K (wide clusters of 8, 14 or 15
    // of them at once): 41.9 -> 22.8 us with 512-thread CTAs; at 60 K 50 -> 30 us; 36 units at 6 K 48 -> 26 us.
    if (n_clusters < units && (long long)units * cs <= slots && cs > 1 && cap_of(cs / 2) <= kCapPair &&
        !((long long)units * cs > ctx->n_sm && wide_clusters(cs) >= units))
      continue;
    // the forms without attention run with the same cluster shape
    bool ok = true;
    for (FusedFn other : {select_fn(ctx->chunks, paged), topk_fn()})
      ok = ok && cudaFuncSetAttribute((const void*)other, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_limit) == cudaSuccess &&
           (cs <= 8 || cudaFuncSetAttribute((const void*)other, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess);
    if (!ok) {
      cudaGetLastError();
      continue;
    }
    ctx->fused_cs = cs;
    ctx->fused_smem = smem;
    // The wide form.  When the 512-thread grid has more CTAs than SMs, SMs hold pairs of CTAs that
    // share their ~44 GB/s while lone CTAs (in a single wave: batch 8 x 8 heads at 64 K) end their
    // stream at 28 us against 50 us, and grids of several rounds run twice as many select chains.
    // Half as many CTAs of 1024 threads with twice the slice each sit alone on their SMs and
    // stream at the same rate: 74 -> 70 us there, 68 -> 57 us for batch 5, 210 -> 203 us for the
    // four-round grid of batch 16 at 64-128 K.
    ctx->step_threads = kFT;
    ctx->step_cs = cs;
    ctx->step_smem = smem;
    ctx->step_resident = n_clusters;
    // (not down to clusters of one CTA: batch 32 x 4 heads of 7 query heads at 16 K lost 3-6 % that way)
    const int n_w = (long long)units * cs > ctx->n_sm ? wide_clusters(cs) : 0;
    if (n_w >= 1 && (n_w >= units || n_clusters < units)) {
      ctx->step_threads = 1024;
      ctx->step_cs = cs / 2;
      ctx->step_smem = (size_t)fused_smem_layout(cap_of(cs / 2), 32).total;
      ctx->step_resident = n_w;
    }
    return cs;
  }
  return 0;
}

int32_t fasa_fused_launch(fasa_ctx* ctx, const void* q, const void* k_cache, const void* v_cache,
                          const void* proxy_k, const int32_t* seq_lens, int32_t budget,
                          int32_t n_sel_max, float* scores, int32_t* idx, int32_t* n_sel,
                          float* out, float* lse, const void* k_new, const void* v_new,
                          cudaStream_t stream, bool with_attention, float* out_mirror, bool split_keys) {
  const fasa_config_t& c = ctx->cfg;
  FusedParams p;
  p.out_mirror = out_mirror;
  p.q = (const uint16_t*)q; p.k = (const uint16_t*)k_cache; p.v = (const uint16_t*)v_cache;
  p.proxy = (const unsigned char*)proxy_k; p.seq_lens = seq_lens; p.chan = ctx->d_chan;
  p.k_new = (const uint16_t*)k_new; p.v_new = (const uint16_t*)v_new;
  p.k_w = (uint16_t*)k_cache; p.v_w = (uint16_t*)v_cache; p.proxy_w = (unsigned char*)proxy_k;
  p.seq_lens_w = (int32_t*)seq_lens; p.arrive = ctx->d_arrive;
  p.shift_clusters = 0; p.shift_ctas = 0;
  p.q_len = 1;
  p.ndchan = split_keys ? ctx->d_ndchan : nullptr;
  p.nd = FASA_HEAD_DIM - 2 * c.n_dom;
  p.res = split_keys ? fasa_resident_of(ctx) : fasa_resident{};
  p.scores = scores; p.idx = idx; p.n_sel = n_sel; p.out = out; p.lse = lse; p.status = ctx->d_status;
  p.n_q_heads = c.n_q_heads; p.n_kv_heads = c.n_kv_heads; p.n_sets = ctx->n_sets; p.group = ctx->sel_heads; p.max_len = c.max_len;
  p.chunks = ctx->chunks; p.n_sink = c.n_sink; p.n_recent = c.n_recent; p.budget = budget;
  p.n_sel_max = n_sel_max;
  p.max_reduce = c.group_reduce;
  p.ksb = c.k_stride_b; p.ksh = c.k_stride_h; p.kst = c.k_stride_t;
  p.vsb = c.v_stride_b; p.vsh = c.v_stride_h; p.vst = c.v_stride_t;
  p.scale_log2 = c.softmax_scale * 1.4426950408889634f;
  p.pm = fasa_page_map(ctx);
  p.host_rows = with_attention && c.page_size == 0 && fasa_on_host(k_cache);
  if (!fasa_pages_ready(ctx)) return FASA_ERR_INVALID_ARG;
  const bool paged = c.page_size > 0;
  FusedFn fn = with_attention ? fused_fn(ctx->chunks, paged) : select_fn(ctx->chunks, paged);
  // (the step's own shape: 512 threads and the context's cluster size, or the wide form)
  const bool wide = ctx->step_threads == 1024;
  if (wide) fn = with_attention ? wide_fn(ctx->chunks, paged) : wide_select_fn(ctx->chunks, paged);
  const int threads = wide ? 1024 : kFT, cs_l = wide ? ctx->step_cs : ctx->fused_cs;
  const size_t smem_l = wide ? ctx->step_smem : ctx->fused_smem;

  p.early = (long long)c.batch * ctx->n_sets <= ctx->step_resident && (long long)c.batch * ctx->n_sets * cs_l <= ctx->n_sm;
  // (from one and a half rounds of CTAs on: see the kernel)
  if (ctx->step_resident > 0 && 2ll * c.batch * ctx->n_sets >= 3ll * ctx->step_resident) {
    p.shift_clusters = ctx->step_resident;
    p.shift_ctas = ctx->step_resident * cs_l;
  }
  // Only a grid of at most one CTA per SM is launched early, and gains the launch latency (steps back to back, batch 1 at
  // 32 K: 24.9 -> 21.9 us, batch 8 at 64 K: 59.6 -> 56.3 us).  The clusters of a larger one would be placed around the CTAs
  // of the kernel ahead, which leaves SMs with two CTAs beside SMs with none (96 units on pages: 67.7 -> 69.9 us) and,
  // over several rounds, gaps that stay (batch 16 at 64-128 K: 177 -> 211 us).
  const fasa_launch_shape shape{dim3((unsigned)cs_l, (unsigned)(c.batch * ctx->n_sets)), dim3((unsigned)threads), smem_l, cs_l, p.early != 0};
  const cudaError_t e = fasa_launch(fn, shape, stream, p);
  ctx->launches += 1;
  FASA_CUDA_TRY(ctx, e);
  return FASA_OK;
}

int32_t fasa_topk_cluster_launch(fasa_ctx* ctx, const float* scores, const int32_t* seq_lens, int32_t budget, int32_t n_sel_max,
                                 int32_t* idx, int32_t* n_sel, int rows_per_seq, int n_sink, int n_recent, cudaStream_t stream,
                                 int q_len) {
  const fasa_config_t& c = ctx->cfg;
  FusedParams p;
  memset(&p, 0, sizeof(p));
  p.seq_lens = seq_lens; p.scores = const_cast<float*>(scores); p.idx = idx; p.n_sel = n_sel; p.status = ctx->d_status;
  // (this form uses the unit index for its score row and its sequence alone)
  p.n_q_heads = rows_per_seq; p.n_kv_heads = 1; p.n_sets = rows_per_seq; p.group = 1; p.max_len = c.max_len;
  p.chunks = ctx->chunks; p.n_sink = n_sink; p.n_recent = n_recent; p.budget = budget;
  p.n_sel_max = n_sel_max;
  p.q_len = q_len;
  // The context's cluster size suits its own number of rows; a block of queries has more, and takes the smallest that holds
  // a row two CTAs to an SM.
  int cs = ctx->fused_cs;
  auto cap_of = [&](int n) { return (((c.max_len + n - 1) / n) + 31) & ~31; };
  if (rows_per_seq > ctx->n_sets) {
    cs = 1;
    while (cs < ctx->fused_cs && cap_of(cs) > kCapPair) cs *= 2;
  }
  p.early = (long long)c.batch * rows_per_seq * cs <= ctx->n_sm;
  const fasa_launch_shape shape{dim3((unsigned)cs, (unsigned)(c.batch * rows_per_seq)), dim3(kFT), fused_smem_bytes(cap_of(cs)), cs, p.early != 0};
  const cudaError_t e = fasa_launch(topk_fn(), shape, stream, p);
  ctx->launches += 1;
  FASA_CUDA_TRY(ctx, e);
  return FASA_OK;
}
