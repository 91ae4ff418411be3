// TopK-I (Sec. 4.1) of one score row by one thread block: the k best positions of a row in
// ascending order, equal scores lowest index first (= a stable sort).
//
// A row of L scores is not sorted or histogrammed as a whole.  It is cut into groups of 8 or 32
// consecutive positions whose maxima bound the k-th largest score from below: at least k groups have a
// maximum at or above the k-th largest maximum, so at least k scores do, and a group whose maximum lies
// below it holds none of the k best.  With k well below the number of groups only those k groups are
// looked at again (k = 256 of 65536 positions: 2100 of them); otherwise the row is taken whole.
//   1. the k-th largest group maximum, to the resolution of one histogram of 1024 bins spread evenly
//      over the range of the maxima (values, not their bit patterns: real scores crowd into a few
//      exponents, which makes the atomics of a radix histogram collide and its bins useless);
//   2. the list of the groups at or above that bin, ascending;
//   3. one more such histogram, over the scores of these groups from the bound up, gives the bin of the
//      k-th largest score; its few members are ranked against each other by (score, index), which
//      settles which of them are taken;
//   4. the bit masks of the selected positions become ranks (a block-wide prefix sum).
// What bounds this is latency, instructions and block barriers (ten), not bytes: a pass touches a score with a dozen
// instructions per 32 of them, so the fewer positions a pass visits the better.  A row of 53 K with its maxima given, 256 of it,
// 512 threads, in thousands of cycles: the maxima 2.6, their histogram 3.4 with the search, the list 2.7, the scores of its
// groups 3.5, their threshold 1.1, classes 1.3, ties 1.2, ranks 1.7; before loads went in batches without a serial rest, shares of
// the bins were summed by warps, and ranks went by bytes: 4.0, 3.6, 2.8, 5.1 for scores and threshold, 3.5, 2.2.  Bins are
// monotone in the score, whatever the rounding, so the result is exact.  A few scores far above the others (outlier keys,
// sinks) would leave the rest in one or two bins: where some warp's largest value is far below the largest of all, the bins
// end a little above it, and what lies beyond falls into the last one.  A histogram whose bin of interest is crowded all the
// same is taken again over that bin's range, what lies above or below falling into the outermost bins.  Scores that this cannot spread either (infinities and
// NaNs, hundreds of equal scores at the threshold) are settled by an 11 / 11 / 10-bit radix select on order-preserving keys.
#pragma once

#include "fasa_common.cuh"
#include "fasa_score_core.cuh"

#ifdef __CUDACC__

constexpr int kSelBins = 1024;
constexpr int kSelRank = 256;            // members of the threshold's bin that are ranked against each other
constexpr int kSelRadixBins = 2048;

struct SelShared {
  alignas(16) uint32_t hist[2][kSelBins];   // (read 16 bytes at a time) group maxima; scores.  Together: the bins of a radix pass
  uint32_t ckey[kSelRank], cpos[kSelRank];
  uint32_t wlo[32], whi[32], wcnt[32], share[32];
  uint32_t n_cand;
};
static_assert(2 * kSelBins == kSelRadixBins, "the radix passes use both histograms");

// A block's dynamic shared memory for a row: the maxima of the groups (float; later their bins) and, once the
// groups are listed, the bins of the positions looked at in their place; the list of groups; one bit per position
// looked at.
struct SelLayout {
  int gm_cap, uni_cap, word_cap;         // group maxima (and list entries) / positions' bins / mask words that fit
  __host__ __device__ int list_off() const { return ((gm_cap * 4 > uni_cap * 2 ? gm_cap * 4 : uni_cap * 2) + 15) & ~15; }
  __host__ __device__ int word_off() const { return list_off() + ((gm_cap * 2 + 15) & ~15); }
  __host__ __device__ int bytes() const { return word_off() + word_cap * 4; }
};

// max and min that keep NaNs, so that one in the row is noticed
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

__device__ __forceinline__ float max_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ float sel_key_value(uint32_t k) {       // inverse of fasa_order_key
  return __uint_as_float((k & 0x80000000u) ? k ^ 0x80000000u : ~k);
}

// Evenly spread bins 1 .. kSelBins - 1 from `lo` up; 0 is what lies below.
struct SelBinning {
  float lo, scale;
  __device__ __forceinline__ int bin(float x) const {              // non-decreasing in x
    return min(kSelBins - 1, max(0, __float2int_rz(fmaf(x - lo, scale, 1.0f))));
  }
};
__device__ __forceinline__ SelBinning sel_binning(float lo, float hi) {
  SelBinning b;
  b.lo = lo;
  b.scale = (float)(kSelBins - 1) / (hi - lo);                      // hi == lo, or a range past the largest float: one bin
  if (!(b.scale < 3.0e38f)) b.scale = 0.f;
  return b;
}

// Bins over the range of one bin alone (and a little to either side; the last one reaches up to `hi`, the largest value);
// scale 0 where that is too narrow.
constexpr int kSelTries = 3;             // histograms taken at most
__device__ __forceinline__ SelBinning sel_narrower(const SelBinning& b, int bin, float hi) {
  const float lo = b.lo + ((float)bin - 1.0625f) / b.scale;
  return sel_binning(lo, bin == kSelBins - 1 ? hi : lo + 1.125f / b.scale);
}
// Where the bins of values in [lo, hi] end if they are to spread the kth largest: mid = the least of the warps' largest values.
template <int NT>
__device__ __forceinline__ float sel_reach(float lo, float hi, float mid, int k) {
  const float r = 1.25f * (mid - lo);
  return k >= NT / 16 && r > 0.f && hi - lo > 4.f * r ? lo + r : hi;
}

__device__ __forceinline__ uint32_t sel_scan(uint32_t v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// One warp: the bin of hist[0 .. NB) that holds the kth largest entry (counted from the highest bin
// down; kth <= entries), its rank inside the bin and the bin's count.
template <int NB>
__device__ __forceinline__ void sel_find(const uint32_t* hist, uint32_t kth, int lane, int* bin, uint32_t* rank, uint32_t* count) {
  constexpr int PER = NB / 32;
  uint32_t v = 0;
#pragma unroll
  for (int j = 0; j < PER / 4; ++j) {
    // (the start of a lane's run rotates with the lane, so that the lanes' 16-byte reads spread over the banks)
    const uint4 q = *reinterpret_cast<const uint4*>(hist + NB - PER * (lane + 1) + 4 * ((j + lane) & (PER / 4 - 1)));
    v += q.x + q.y + q.z + q.w;
  }
  const uint32_t incl = sel_scan(v, lane);
  const uint32_t hits = __ballot_sync(0xffffffffu, incl >= kth);
  const int hit = hits ? __ffs(hits) - 1 : 31;
  uint32_t left = kth - __shfl_sync(0xffffffffu, incl - v, hit);
  int top = NB - PER * hit;                                         // one past the run's highest bin
#pragma unroll
  for (int part = 0; part < PER; part += 32) {
    const uint32_t c = hist[top - 1 - lane];
    const uint32_t ci = sel_scan(c, lane);
    const uint32_t h2 = __ballot_sync(0xffffffffu, ci >= left);
    if (h2 || part + 32 >= PER) {
      const int first = h2 ? __ffs(h2) - 1 : 31;
      *bin = top - 1 - first;
      *rank = left - __shfl_sync(0xffffffffu, ci - c, first);
      *count = __shfl_sync(0xffffffffu, c, first);
      return;
    }
    left -= __shfl_sync(0xffffffffu, ci, 31);
    top -= 32;
  }
}

// The same for the histograms of kSelBins bins, by the whole block: every warp sums its share of the bins, then looks at the
// sums and at one share alone.  (Every warp scanning all bins moves 4 KB of shared memory for each: 1200 cycles with 16 warps,
// 450 this way.)  One barrier, behind the one that completes the histogram.
template <int NT>
__device__ __forceinline__ void sel_find_block(SelShared& sm, const uint32_t* hist, uint32_t kth, int warp, int lane, int* bin, uint32_t* rank,
                                               uint32_t* count) {
  constexpr int NW = NT / 32, PER = kSelBins / NW, EACH = PER / 32;  // bins of a share / of a lane: 1, 2 or 4
  static_assert(EACH == 1 || EACH == 2 || EACH == 4, "a lane reads its bins at once");
  auto share = [&](int w, uint32_t (&c)[EACH]) {                    // the lane's bins of share w, highest first (share 0 is the highest)
    const uint32_t* p = hist + kSelBins - PER * w - EACH * (lane + 1);
    if constexpr (EACH == 4) {
      const uint4 q = *reinterpret_cast<const uint4*>(p);
      c[0] = q.w; c[1] = q.z; c[2] = q.y; c[3] = q.x;
    } else if constexpr (EACH == 2) {
      const uint2 q = *reinterpret_cast<const uint2*>(p);
      c[0] = q.y; c[1] = q.x;
    } else {
      c[0] = *p;
    }
  };
  uint32_t c[EACH], sum = 0;
  share(warp, c);
#pragma unroll
  for (int j = 0; j < EACH; ++j) sum += c[j];
  sum = __reduce_add_sync(0xffffffffu, sum);
  if (lane == 0) sm.share[warp] = sum;
  __syncthreads();
  const uint32_t v = lane < NW ? sm.share[lane] : 0u, incl = sel_scan(v, lane);
  const uint32_t hits = __ballot_sync(0xffffffffu, incl >= kth);
  const int w = hits ? __ffs(hits) - 1 : NW - 1;
  const uint32_t left = kth - __shfl_sync(0xffffffffu, incl - v, w);
  share(w, c);
  sum = 0;
#pragma unroll
  for (int j = 0; j < EACH; ++j) sum += c[j];
  const uint32_t ci = sel_scan(sum, lane);
  const uint32_t h2 = __ballot_sync(0xffffffffu, ci >= left);
  const int at = h2 ? __ffs(h2) - 1 : 31;
  uint32_t r = left - (ci - sum);                                   // (of the lane `at`)
  int j = 0;
  uint32_t n = c[0];
#pragma unroll
  for (int i = 1; i < EACH; ++i) {
    if (j == i - 1 && r > n) { r -= n; n = c[i]; j = i; }
  }
  *bin = __shfl_sync(0xffffffffu, kSelBins - PER * w - EACH * lane - 1 - j, at);
  *rank = __shfl_sync(0xffffffffu, r, at);
  *count = __shfl_sync(0xffffffffu, n, at);
}

// Block-wide min and max of the threads' values, and the least of the warps' maxima (of those that have values: the others
// come with -inf); one barrier.  false when a value is not finite.
template <int NT>
__device__ __forceinline__ bool sel_minmax(SelShared& sm, float& lo, float& hi, float& mid, int warp, int lane) {
  const uint32_t kl = __reduce_min_sync(0xffffffffu, fasa_order_key(lo)), kh = __reduce_max_sync(0xffffffffu, fasa_order_key(hi));
  if (lane == 0) { sm.wlo[warp] = kl; sm.whi[warp] = kh; }
  __syncthreads();
  lo = sel_key_value(__reduce_min_sync(0xffffffffu, lane < NT / 32 ? sm.wlo[lane] : 0xffffffffu));
  const uint32_t w = lane < NT / 32 ? sm.whi[lane] : 0u;
  hi = sel_key_value(__reduce_max_sync(0xffffffffu, w));
  mid = sel_key_value(__reduce_min_sync(0xffffffffu, w > fasa_order_key(-INFINITY) ? w : 0xffffffffu));
  return hi - lo < 3.0e38f;                                         // (false for NaN)
}

// Block-wide exclusive prefix of v over the threads and the total (one barrier; sm.wcnt is used).
template <int NT>
__device__ __forceinline__ uint32_t sel_block_prefix(SelShared& sm, uint32_t v, int warp, int lane, uint32_t* total) {
  const uint32_t incl = sel_scan(v, lane);
  if (lane == 31) sm.wcnt[warp] = incl;
  __syncthreads();
  const uint32_t w = lane < NT / 32 ? sm.wcnt[lane] : 0u, wi = sel_scan(w, lane);
  *total = __shfl_sync(0xffffffffu, wi, 31);
  return __shfl_sync(0xffffffffu, wi - w, warp) + incl - v;
}

// Where the scores of a row come from: a buffer, or (calibration) the channel pairs of one FC, two bf16 values to a
// position, with the query's values at these two channels: fl(q0 k0 + q1 k1), the products of bf16 values being exact.
struct SelScores {
  const float* p;
  __device__ __forceinline__ float operator()(int i) const { return p[i]; }
  __device__ __forceinline__ float4 four(int i) const { return *reinterpret_cast<const float4*>(p + i); }
  __device__ __forceinline__ float max8(int i) const {              // of eight positions; i: as four wants it
    const float4 a = four(i), b = four(i + 4);
    return max_nan(max_nan(a.x, a.y, a.z), max_nan(a.w, b.x, b.y), max_nan(b.z, b.w));
  }
  __device__ __forceinline__ bool aligned() const { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
};
struct SelPairs {
  const uint32_t* p;
  float q0, q1;
  __device__ __forceinline__ float score(uint32_t w) const {
    const float2 k = bf16x2_to_f32x2(w);
    return fmaf(q0, k.x, q1 * k.y) + 0.0f;                          // (-0 becomes +0)
  }
  __device__ __forceinline__ float operator()(int i) const { return score(p[i]); }
  __device__ __forceinline__ float4 four(int i) const {
    const uint4 w = *reinterpret_cast<const uint4*>(p + i);
    return make_float4(score(w.x), score(w.y), score(w.z), score(w.w));
  }
  // Two positions to an instruction (the values are the same; a maximum needs no +0).
  __device__ __forceinline__ float2 two(uint32_t a, uint32_t b) const {
    const float2 x = make_float2(__uint_as_float(a << 16), __uint_as_float(b << 16));
    const float2 y = make_float2(__uint_as_float(a & 0xffff0000u), __uint_as_float(b & 0xffff0000u));
    return __ffma2_rn(make_float2(q0, q0), x, __fmul2_rn(make_float2(q1, q1), y));
  }
  __device__ __forceinline__ float max8(int i) const {
    const uint4 a = *reinterpret_cast<const uint4*>(p + i), b = *reinterpret_cast<const uint4*>(p + i + 4);
    const float2 s = two(a.x, a.y), t = two(a.z, a.w), u = two(b.x, b.y), v = two(b.z, b.w);
    return max_nan(max_nan(s.x, s.y, t.x), max_nan(t.y, u.x, u.y), max_nan(v.x, v.y));
  }
  __device__ __forceinline__ bool aligned() const { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
};

// The positions a row may be selected from, and how many of them are.
template <typename Src>
struct SelRow {
  Src src;
  int lo, hi;                            // positions [lo, hi) compete (the others are forced or past the end)
  int k;                                 // 0 <= k <= hi - lo
};

// Before a row: clears what the row's histograms add to.
template <int NT>
__device__ __forceinline__ void sel_begin(SelShared& sm) {
  for (int i = threadIdx.x; i < kSelRadixBins / 4; i += NT) reinterpret_cast<uint4*>(&sm.hist[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
  if (threadIdx.x == 0) sm.n_cand = 0u;
}

// Groups of 1 << shift positions narrow a row of n positions down; 0: take the row whole.  Groups of 8 leave
// the fewest positions to look at, those of 32 have the fewest maxima: with about 1.5 instructions per 32
// maxima and pass and 5 per 32 positions the larger ones pay below k = n / 1024.
__host__ __device__ __forceinline__ int sel_group_shift(int n, int k, int gm_cap) {
  const bool by8 = (long long)k * 12 <= n && (n >> 3) + 2 <= gm_cap;
  const bool by32 = (long long)k * 43 <= n && (n >> 5) + 2 <= gm_cap;
  if (by32 && ((long long)k * 1024 <= n || !by8)) return 5;
  return by8 ? 3 : 0;
}

// Calls emit(r, position) for the r-th selected position in ascending order, r = 0 .. k - 1.
// gs > 0: fill(gm, lo, hi), called by all threads, once or up to kSelTries times, writes the maxima (float) of the groups
// (r.lo >> gs) .. ((r.hi - 1) >> gs), positions outside [lo, hi) left out, and the least and the largest of those that this
// thread has written to lo and hi.  sel_begin comes before (the first barrier is behind the first reads of the row, so that
// nothing delays them); all threads call.
template <int NT, typename Src, typename Fill, typename Emit>
__device__ __forceinline__ void sel_row(const SelRow<Src>& r, int gs, Fill fill, SelShared& sm, unsigned char* dyn,
                                        const SelLayout& lay, Emit emit) {
  constexpr int NW = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (r.k <= 0) return;                                             // (uniform)
  if (r.k == r.hi - r.lo) {
    for (int i = tid; i < r.k; i += NT) emit(i, r.lo + i);
    return;
  }
  float* gm = reinterpret_cast<float*>(dyn);
  uint16_t* list = reinterpret_cast<uint16_t*>(dyn + lay.list_off());
  uint16_t* bins16 = reinterpret_cast<uint16_t*>(dyn);
  uint32_t* words = reinterpret_cast<uint32_t*>(dyn + lay.word_off());
  const uint32_t below = (1u << lane) - 1u;

  bool radix = false;                    // the even bins do not apply
  bool equal_maxima = false;             // the threshold lies among many equal scores, it seems
  int n_list = 0;
  float bound = 0.f, top = 0.f, reach = 0.f;                       // the largest value; where the bins end
  int g0 = 0;
  if (gs > 0) {
    // ---- 1, 2: the groups that can hold one of the k best -------------------------------------
    g0 = r.lo >> gs;
    const int n_groups = ((r.hi - 1) >> gs) + 1 - g0;
    SelBinning first{0.f, 0.f};
    int b0 = 0;
    uint32_t rank, count = 0;
#pragma unroll 1
    for (int t = 0; t < kSelTries; ++t) {
      float lo = INFINITY, hi = -INFINITY, mid;
      fill(gm, lo, hi);
      if (t == 0) {
        if (!sel_minmax<NT>(sm, lo, hi, mid, warp, lane)) {              // (the maxima are complete after its barrier)
          radix = true;
          gs = 0;
          break;
        }
        top = hi;
        reach = sel_reach<NT>(lo, hi, mid, r.k);
        first = sel_binning(lo, reach);
      } else {
        __syncthreads();
      }
      for (int i0 = tid; i0 < n_groups; i0 += NT * 4) {
        float m[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) m[j] = gm[min(i0 + j * NT, n_groups - 1)];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (i0 + j * NT < n_groups) {
            const int bin = first.bin(m[j]);
            atomicAdd(&sm.hist[0][bin], 1u);
            gm[i0 + j * NT] = __int_as_float(bin);
          }
        }
      }
      __syncthreads();
      const uint32_t was = count;
      sel_find_block<NT>(sm, sm.hist[0], (uint32_t)r.k, warp, lane, &b0, &rank, &count);
      // crowded: its groups would all be listed, and 8 or 32 positions of each visited
      if (count <= 64u + (uint32_t)r.k / 2u || t + 1 == kSelTries || !(first.scale > 0.f)) break;
      // a thousandth of the range with half the maxima in it: no bins spread these (the same token again and again)
      equal_maxima = 2u * count > was && t > 0;
      if (equal_maxima) break;
      const SelBinning nb = sel_narrower(first, b0, top);
      if (!(nb.scale > 0.f)) break;
      first = nb;
      __syncthreads();                   // (every warp has read the histogram)
      for (int i = tid; i < kSelBins / 4; i += NT) reinterpret_cast<uint4*>(&sm.hist[0][0])[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    if (!radix) {
      const int per = ((n_groups + NW - 1) / NW + 31) & ~31;        // a warp takes a run of groups
      const int s0 = min(n_groups, warp * per), s1 = min(n_groups, s0 + per);
      uint32_t mine = 0;
#pragma unroll 4
      for (int i = s0 + lane; i < s1; i += 32) mine += __float_as_int(gm[i]) >= b0 ? 1u : 0u;
      mine = __reduce_add_sync(0xffffffffu, mine);
      if (lane == 0) sm.wcnt[warp] = mine;
      __syncthreads();
      const uint32_t w = lane < NW ? sm.wcnt[lane] : 0u, incl = sel_scan(w, lane);
      n_list = (int)__shfl_sync(0xffffffffu, incl, 31);
      uint32_t at = __shfl_sync(0xffffffffu, incl - w, warp);
      for (int i = s0; i < s1; i += 128) {                          // uniform over the warp
        bool in[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) in[j] = __float_as_int(gm[min(i + 32 * j + lane, n_groups - 1)]) >= b0 && i + 32 * j + lane < s1;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t m = __ballot_sync(0xffffffffu, in[j]);
          if (in[j]) list[at + __popc(m & below)] = (uint16_t)(i + 32 * j + lane);
          at += __popc(m);
        }
      }
      // (a little below the bin's edge, so that rounding leaves none of the listed maxima under it)
      bound = first.scale > 0.f ? first.lo + ((float)b0 - 1.0625f) / first.scale : first.lo;
      __syncthreads();
    }
  }
  // The universe: positions base + 0, 1, ... or those of the listed groups, 32 to a chunk; a warp owns a
  // run of chunks throughout.
  const bool listed = gs > 0;
  const int base = listed ? g0 << gs : r.lo & ~31;
  const int n_uni = listed ? n_list << gs : r.hi - base;
  const int n_chunks = (n_uni + 31) >> 5;
  const int cper = (n_chunks + NW - 1) / NW;
  const int c0 = min(n_chunks, warp * cper), c1 = min(n_chunks, c0 + cper);
  const bool held = n_chunks * 32 <= lay.uni_cap;
  auto pos_at = [&](int c, int l) -> int {                          // position l of chunk c (it may not compete)
    if (!listed) return base + 32 * c + l;
    const int e = (c << (5 - gs)) + (l >> gs);
    return e < n_list ? base + ((int)list[e] << gs) + (l & ((1 << gs) - 1)) : -1;
  };
  constexpr int UNR = 4;
  // visits this warp's chunks, UNR loads in flight: f(chunk, competes, score)
  auto visit = [&](auto f) {
    for (int c = c0; c < c1; c += UNR) {                            // uniform over the warp
      float x[UNR];
      bool ok[UNR];
#pragma unroll
      for (int j = 0; j < UNR; ++j) {
        const int p = pos_at(c + j, lane);
        ok[j] = c + j < c1 && p >= r.lo && p < r.hi;
        x[j] = ok[j] ? r.src(p) : -INFINITY;
      }
#pragma unroll
      for (int j = 0; j < UNR; ++j)
        if (c + j < c1) f(c + j, ok[j], x[j]);
    }
  };
  // Listed groups of 8 are visited by a thread each where they occupy 128 of 256 threads, or all of more: two 16-byte loads, eight
  // bins kept as 16 bytes, a byte of the masks.  Against positions in chunks of 32 to a warp, 1024 rows a set: batch 4 at 30-56 K, a
  // set per query head 51.8 -> 49.3 us a step, batch 32 at 16-31 K 122 -> 117; calibration, 512 of 8-16 K 80 -> 67.5, 128 of 12-24 K 44.5
  // -> 42.6.  With fewer groups than threads the chunks are more parallel: 512 threads, 256 of 3-7 K 26.3 / 27.2.  So they are for
  // 1024 threads on rows that are not aligned, whose groups take eight loads of 4 bytes: 128 rows of 43765 after their scoring, 1024
  // of each: 81.3 / 83.5 us in all (aligned rows of 40960 that have left the caches: 15.8 / 14.8).
  const bool octets = gs == 3 && held && (NT == 256 ? 2 : 1) * n_list >= NT && (NT < 1024 || r.src.aligned());
  SelBinning second{0.f, 0.f};
  if (listed) {
    second = sel_binning(bound, reach > bound ? reach : top);
  } else if (!radix) {
    float lo = INFINITY, hi = -INFINITY, mid;
    visit([&](int, bool ok, float x) {
      if (ok) { lo = fminf(lo, x); hi = max_nan(hi, x); }           // (a NaN shows in hi)
    });
    if (!sel_minmax<NT>(sm, lo, hi, mid, warp, lane)) radix = true;
    else second = sel_binning(lo, sel_reach<NT>(lo, hi, mid, r.k));
    top = hi;
  }
  uint32_t rank = 0, count = 0;
  int b1 = 0;
  if (!radix) {
#pragma unroll 1
    for (int t = 0; t < kSelTries; ++t) {
      if (octets) {
        const bool whole = r.src.aligned();
#pragma unroll 2
        for (int e = tid; e < n_list; e += NT) {
          const int p = base + ((int)list[e] << 3);
          // (all eight are loaded before the first is used, also where a row is not aligned: one after another, 128 rows of 43765
          // that have left the caches cost 4 us more)
          float v[8];
          if (whole && p >= r.lo && p + 8 <= r.hi) {
            const float4 x = r.src.four(p), y = r.src.four(p + 4);
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
            v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = p + i >= r.lo && p + i < r.hi ? r.src(p + i) : -INFINITY;
          }
          uint32_t bin[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            bin[i] = p + i >= r.lo && p + i < r.hi ? (uint32_t)second.bin(v[i]) : 0u;
            if (bin[i] > 0u) atomicAdd(&sm.hist[1][bin[i]], 1u);
          }
          *reinterpret_cast<uint4*>(bins16 + e * 8) =
              make_uint4(bin[0] | bin[1] << 16, bin[2] | bin[3] << 16, bin[4] | bin[5] << 16, bin[6] | bin[7] << 16);
        }
      } else {
        visit([&](int c, bool ok, float x) {
          const int bin = ok ? second.bin(x) : 0;
          if (bin > 0) atomicAdd(&sm.hist[1][bin], 1u);
          if (held) bins16[c * 32 + lane] = (uint16_t)bin;
        });
      }
      __syncthreads();
      const uint32_t was = count;
      sel_find_block<NT>(sm, sm.hist[1], (uint32_t)r.k, warp, lane, &b1, &rank, &count);
      if (count <= (uint32_t)kSelRank && b1 > 0) break;
      const SelBinning nb = sel_narrower(second, b1, top);
      // (half as many as before: equal scores)
      radix = b1 == 0 || t + 1 == kSelTries || (t > 0 && 2u * count > was) || equal_maxima || !(second.scale > 0.f) || !(nb.scale > 0.f);
      __syncthreads();                   // (every warp has read the histogram)
      if (radix) break;
      second = nb;
      for (int i = tid; i < kSelBins / 4; i += NT) reinterpret_cast<uint4*>(&sm.hist[1][0])[i] = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
    }
  }

  // ---- 3: one bit per position of the universe: selected or not ----------------------------------
  if (!radix) {
    auto classify = [&](int c, int bin) {
      const uint32_t ma = __ballot_sync(0xffffffffu, bin > b1), mc = __ballot_sync(0xffffffffu, bin == b1);
      if (lane == 0) words[c] = ma;
      if (mc) {
        uint32_t at = 0;
        if (lane == 0) at = atomicAdd(&sm.n_cand, (uint32_t)__popc(mc));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(mc & below);
        if (bin == b1 && at < (uint32_t)kSelRank) {
          sm.cpos[at] = (uint32_t)(c * 32 + lane);
          sm.ckey[at] = fasa_order_key(r.src(pos_at(c, lane)));
        }
      }
    };
    if (octets) {
      for (int e = tid; e < 4 * n_chunks; e += NT) {
        uint32_t mask = 0u, equal = 0u;
        if (e < n_list) {
          const uint4 q = *reinterpret_cast<const uint4*>(bins16 + e * 8);
          const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int lo = (int)(w[i] & 0xffffu), hi = (int)(w[i] >> 16);
            mask |= (lo > b1 ? 1u : 0u) << (2 * i) | (hi > b1 ? 2u : 0u) << (2 * i);
            equal |= (lo == b1 ? 1u : 0u) << (2 * i) | (hi == b1 ? 2u : 0u) << (2 * i);
          }
        }
        reinterpret_cast<uint8_t*>(words)[e] = (uint8_t)mask;
        while (equal) {
          const int i = __ffs(equal) - 1;
          equal &= equal - 1;
          const uint32_t at = atomicAdd(&sm.n_cand, 1u);
          if (at < (uint32_t)kSelRank) {
            sm.cpos[at] = (uint32_t)(e * 8 + i);
            sm.ckey[at] = fasa_order_key(r.src(base + ((int)list[e] << 3) + i));
          }
        }
      }
    } else if (held) {
#pragma unroll 4
      for (int c = c0; c < c1; ++c) classify(c, bins16[c * 32 + lane]);
    } else {
      visit([&](int c, bool ok, float x) { classify(c, ok ? second.bin(x) : 0); });
    }
    __syncthreads();
    // four threads to a member, each comparing it with a quarter of the others (the minimum: no entry that nobody wrote is
    // looked at, whatever becomes of the scores meanwhile)
    count = min(count, sm.n_cand);
    for (int i = tid >> 2; i < (int)count; i += NT / 4) {           // (uniform over the four)
      const uint32_t key = sm.ckey[i], pos = sm.cpos[i];
      uint32_t ahead = 0;
      for (int j = tid & 3; j < (int)count; j += 4) {
        const uint32_t kj = sm.ckey[j];
        ahead += kj > key || (kj == key && sm.cpos[j] < pos) ? 1u : 0u;
      }
      const uint32_t quad = 0xfu << (lane & ~3);
      ahead += __shfl_xor_sync(quad, ahead, 1);
      ahead += __shfl_xor_sync(quad, ahead, 2);
      if ((tid & 3) == 0 && ahead < rank) atomicOr(&words[pos >> 5], 1u << (pos & 31));
    }
  } else {
    uint32_t* bins = &sm.hist[0][0];
    uint32_t prefix = 0, kth = (uint32_t)r.k;
    int shift = 32;
#pragma unroll 1
    for (int level = 0; level < 3; ++level) {
      const int bits = level == 2 ? 10 : 11, above = shift;
      for (int i = tid; i < kSelRadixBins; i += NT) bins[i] = 0u;
      __syncthreads();
      shift -= bits;
      visit([&](int, bool ok, float x) {
        const uint32_t key = fasa_order_key(x);
        if (ok && (level == 0 || (key >> above) == prefix)) atomicAdd(&bins[(key >> shift) & ((1u << bits) - 1u)], 1u);
      });
      __syncthreads();
      int bin;
      uint32_t in_bin;
      sel_find<kSelRadixBins>(bins, kth, lane, &bin, &kth, &in_bin);
      prefix = (prefix << bits) | (uint32_t)bin;
      __syncthreads();
    }
    // prefix = the threshold, kth = how many of the scores equal to it are taken, lowest index first
    uint32_t equal = 0;
    visit([&](int, bool ok, float x) { equal += __popc(__ballot_sync(0xffffffffu, ok && fasa_order_key(x) == prefix)); });
    uint32_t total, e_run = sel_block_prefix<NT>(sm, lane == 0 ? equal : 0u, warp, lane, &total);
    e_run = __shfl_sync(0xffffffffu, e_run, 0);
    visit([&](int c, bool ok, float x) {
      const uint32_t key = fasa_order_key(x);
      const uint32_t me = __ballot_sync(0xffffffffu, ok && key == prefix);
      const bool in = ok && (key > prefix || (key == prefix && e_run + __popc(me & below) < kth));
      const uint32_t m = __ballot_sync(0xffffffffu, in);
      if (lane == 0) words[c] = m;
      e_run += __popc(me);
    });
  }
  __syncthreads();

  // ---- 4: ranks in ascending order ---------------------------------------------------------------
  // A thread takes a run of bytes of the masks (a byte is a group of 8), or of words where there are enough of them: as few bits
  // after one another as there are threads for.
  const bool bytes = 2 * n_chunks <= NT;
  const uint8_t* mask8 = reinterpret_cast<const uint8_t*>(words);
  const int n_parts = bytes ? 4 * n_chunks : n_chunks, each = (n_parts + NT - 1) / NT;
  const int w0 = min(n_parts, tid * each), w1 = min(n_parts, w0 + each);
  uint32_t mine = 0;
  for (int c = w0; c < w1; ++c) mine += __popc(bytes ? (uint32_t)mask8[c] : words[c]);
  uint32_t total, at = sel_block_prefix<NT>(sm, mine, warp, lane, &total);
  for (int c = w0; c < w1; ++c) {
    uint32_t m = bytes ? (uint32_t)mask8[c] : words[c];
    if (m == 0u) continue;
    const int first = bytes ? pos_at(c >> 2, (c & 3) * 8) : 0;
    while (m) {
      const int j = __ffs(m) - 1;
      m &= m - 1;
      if (at < (uint32_t)r.k) emit((int)at, bytes ? first + j : pos_at(c, j));     // (the comparison keeps a write inside the list)
      ++at;
    }
  }
}

// fill for sel_row where the maxima of groups [g0, g1) of a row were left in memory by the scoring pass.  Eight or sixteen loads in flight
// per thread, the last ones predicated: a loop that takes what is left over one by one waits for memory each time.
template <int NT>
__device__ __forceinline__ void sel_copy_maxima(float* gm, const float* src, int g0, int g1, float& lo, float& hi) {
  constexpr int UNR = NT == 256 ? 8 : 16;         // (64 registers)
  const int n = g1 - g0;
  src += g0;
  for (int i0 = threadIdx.x; i0 < n; i0 += NT * UNR) {
    float m[UNR];
#pragma unroll
    for (int j = 0; j < UNR; ++j)
      if (i0 + j * NT < n) m[j] = src[i0 + j * NT];
#pragma unroll
    for (int j = 0; j < UNR; ++j) {
      if (i0 + j * NT < n) {
        gm[i0 + j * NT] = m[j];
        lo = fminf(lo, m[j]);
        hi = max_nan(hi, m[j]);
      }
    }
  }
}

// The selection of a row of `len` positions with forced ones: how the budget, the forced positions and
// the size of the list combine (the forced ones are taken first, in ascending order).
struct SelPlan {
  int ktot;                              // positions selected
  int sink, n_forced;
  int lo, hi, k;                         // the free positions and how many of them are taken
  bool clamped;                          // the list was too small
};
__device__ __forceinline__ SelPlan sel_plan(int len, int budget, int n_sink, int n_recent, int n_sel_max) {
  SelPlan s;
  const long long kb = budget > 0 ? (long long)budget : ((long long)(-budget) * len + 999) / 1000;
  s.sink = min(len, n_sink);
  s.lo = s.sink;
  s.hi = len - min(n_recent, len - s.sink);
  s.n_forced = len - (s.hi - s.lo);
  long long kt = min((long long)len, (long long)s.n_forced + kb);
  s.clamped = kt > n_sel_max;
  if (s.clamped) kt = n_sel_max;
  s.ktot = (int)kt;
  s.k = max(0, s.ktot - s.n_forced);
  return s;
}
// Rank of the i-th forced position (ascending) in the list, and the position itself.
__device__ __forceinline__ void sel_forced(const SelPlan& s, int i, int* rank, int* pos) {
  *rank = i < s.sink ? i : i + s.k;
  *pos = i < s.sink ? i : s.hi + (i - s.sink);
}

#endif  // __CUDACC__
