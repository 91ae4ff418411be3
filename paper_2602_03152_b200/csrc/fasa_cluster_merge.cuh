// Merge of split-K attention partials inside one thread-block cluster (the second half of
// flash decoding: m* = max_s m_s, out = sum_s 2^(m_s - m*) acc_s / sum_s 2^(m_s - m*) l_s),
// shared by the one-launch decode step and by the split-K attention kernel.
//
// CTA r of a cluster of cs finishes channels [r, r + 1) * 128 / cs of every head.  Every CTA PUSHES its partial
// values for those into r's shared memory (consecutive threads write runs of consecutive words of one
// peer, so the distributed-shared-memory traffic is a few wide transactions); after ONE cluster barrier r
// combines from local memory only: no CTA reads a peer afterwards, so none has to wait for the others to leave.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "fasa_common.cuh"

constexpr int kMergePartStride = FASA_HEAD_DIM + 4;   // a head's partial in shared memory: m, l, acc[128], padding
constexpr int kMergeMaxCs = 16;                        // CTAs per cluster at most

// The two halves of a cluster barrier (cluster.sync() = arrive + wait), for all threads of all CTAs alike: what a thread
// wrote before its arrive is visible to every thread after its wait.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
// (the first half where nothing was written that a peer may touch: the CTA only says that it runs, without a fence)
__device__ __forceinline__ void cluster_arrive_running() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// What the peers write into: must not share memory with anything the owning CTA still uses
// when the first peer finishes its part.
struct ClusterMergeSmem {
  float racc[FASA_MAX_GROUP * FASA_HEAD_DIM + kMergeMaxCs];   // [rank][per_o]: accumulators of this CTA's outputs
  alignas(8) float rml[kMergeMaxCs][FASA_MAX_GROUP][2];                 // every CTA's (m, l) per head
};

// Infinite values.  A probability enters the output products of the tensor-core forms as a sum of bf16 terms, of which the
// later ones may be zero or negative, and rows past the end of a tile repeat the last one with probability zero: an infinite
// entry of V then gives NaN where its sum with the other rows is an infinity.  An output that is not finite is therefore
// computed once more by a warp, row by row with multiply-adds.  (Here, because the attention loops have no register to
// spare: a test at their end, a branch in them or a second copy of them cost 2 to 10 % of a step; this costs 0.2 us of the
// smallest ones, 13.4 -> 13.6 us, nothing that shows of most others, and 3 % of the cluster kernel's lists of 4096 rows.)
template <bool PAGED>
struct ExactOutput {
  const uint16_t* q;              // the query head
  const uint16_t* k;              // (of the KV head; contiguous caches: of the sequence)
  const uint16_t* v;
  const int32_t* list;            // n rows
  int32_t* status;
  PageMap pm;
  int64_t ksb, kst, vsb, vst;
  int n, b, max_len;
  float scale_log2;
};
// One warp: channel c of the output.
template <bool PAGED>
__device__ __forceinline__ float exact_output(const ExactOutput<PAGED>& r, int c) {
  const int lane = threadIdx.x & 31;
  const uint2 qw = *reinterpret_cast<const uint2*>(r.q + lane * 4);
  const float2 q0 = bf16x2_to_f32x2(qw.x), q1 = bf16x2_to_f32x2(qw.y);
  float m = -INFINITY, l = 0.f, a = 0.f;
#pragma unroll 1
  for (int i = 0; i < r.n; ++i) {
    const int tok = min(max(r.list[i], 0), r.max_len - 1);
    const int row = PAGED ? pool_row(r.pm, r.b, tok, r.status) : tok;
    const int page = PAGED ? row >> r.pm.shift : 0, in = PAGED ? row & ((1 << r.pm.shift) - 1) : row;
    const uint16_t* kr = r.k + page * r.ksb + in * r.kst;
    const uint16_t* vr = r.v + page * r.vsb + in * r.vst;
    const uint2 kw = *reinterpret_cast<const uint2*>(kr + lane * 4);
    const float2 k0 = bf16x2_to_f32x2(kw.x), k1 = bf16x2_to_f32x2(kw.y);
    float x = q0.x * k0.x + q0.y * k0.y + q1.x * k1.x + q1.y * k1.y;
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    x *= r.scale_log2;
    const float m_new = fmaxf(m, x), m_safe = m_new == -INFINITY ? 0.f : m_new;
    const float alpha = exp2f(m - m_safe), pr = exp2f(x - m_safe);
    l = l * alpha + pr;
    a = fmaf(pr, bf16_bits_to_f32(vr[c]), a * alpha);
    m = m_new;
  }
  return l > 0.f ? a / l : 0.f;
}
struct NoExactOutput {};
// The CTA's unit, read anew: what is derived from it where exact_output is called shall not be kept since the kernel's start.
__device__ __forceinline__ int unit_again() {
  int u;
  asm volatile("mov.u32 %0, %%ctaid.y;" : "=r"(u));
  return u;
}

// part[g] = (m, l, acc[128]) of head g of this CTA, base-2 logit domain, complete and visible to
// the whole block.  NT threads call this together, in every CTA of the cluster (the cluster
// size must be a power of two <= 16).  out / lse rows start at query head q0; out_mirror and
// lse may be null.  The peers must be known to run before this is called (their shared memory is written): a cluster barrier
// since the kernel's start, or cluster_arrive_running() at the start and cluster_wait() before the call.  exact(g): what is needed to
// compute the outputs of head g of this unit row by row (ExactOutput), for those that are not finite.
template <int NT, typename Exact = NoExactOutput>
__device__ __forceinline__ void cluster_merge_store(cooperative_groups::cluster_group& cluster,
                                                    const float (*part)[kMergePartStride], ClusterMergeSmem& sm,
                                                    int group, int64_t q0, float* out, float* out_mirror, float* lse,
                                                    Exact exact = Exact()) {
  // a warp: the value of a lane that has one at (g, c), computed anew where it is not finite
  auto settled = [&](float ov, bool has, int g, int c) -> float {
    if constexpr (!std::is_same<Exact, NoExactOutput>::value) {
#pragma unroll 1
      for (uint32_t odd = __ballot_sync(0xffffffffu, has && !(fabsf(ov) < INFINITY)); odd != 0u; odd &= odd - 1u) {
        const int l = __ffs(odd) - 1;
        const auto e = exact(__shfl_sync(0xffffffffu, g, l));
        const float x = exact_output(e, __shfl_sync(0xffffffffu, c, l));
        if ((int)(threadIdx.x & 31) == l) ov = x;
      }
    }
    return ov;
  };
  const int cs = (int)cluster.num_blocks();
  const int crank = (int)cluster.block_rank();
  const int tid = threadIdx.x;
  constexpr int GP = FASA_MAX_GROUP;
  const int n_out = group * FASA_HEAD_DIM;
  if (cs == 1) {                              // nothing to merge
    for (int o = tid; o < n_out; o += NT) {
      const int g = o / FASA_HEAD_DIM, c = o % FASA_HEAD_DIM;
      const float l = part[g][1], ov = settled(l > 0.f ? part[g][2 + c] / l : 0.f, true, g, c);
      out[q0 * FASA_HEAD_DIM + o] = ov;
      if (out_mirror) out_mirror[q0 * FASA_HEAD_DIM + o] = ov;
      if (lse && c == 0) lse[q0 + g] = l > 0.f ? (part[g][0] + log2f(l)) * 0.6931471805599453f : -INFINITY;
    }
    return;
  }
  const int lc = 31 - __clz(cs), lw = 7 - lc, cw = 1 << lw;   // channels of a head that a CTA finishes: 128 / cs = 1 << lw
  const int per_o = group << lw;
  for (int o = tid; o < n_out; o += NT) {
    const int c = o % FASA_HEAD_DIM, g = o / FASA_HEAD_DIM;
    float* dst = cluster.map_shared_rank(&sm.racc[0], c >> lw);
    dst[crank * per_o + (g << lw) + (c & (cw - 1))] = part[g][2 + c];
  }
  for (int i = tid; i < cs * GP; i += NT) {
    const int r = i / GP, g = i % GP;
    if (g < group) *reinterpret_cast<float2*>(cluster.map_shared_rank(&sm.rml[crank][g][0], r)) = make_float2(part[g][0], part[g][1]);
  }
  cluster.sync();   // the merge barrier: every CTA's partial results have arrived
  const int opp = NT >> lc;                  // outputs per pass
  const int r = tid & (cs - 1), tl = tid >> lc;
  for (int t0 = 0; t0 < per_o; t0 += opp) {  // uniform trip count
    const int t = t0 + tl;
    const bool ok = t < per_o;
    const int g = ok ? t >> lw : 0;
    const float ms = sm.rml[r][g][0], ls = sm.rml[r][g][1];
    const float as = ok ? sm.racc[r * per_o + t] : 0.f;
    float mx = ms;
    for (int off = cs >> 1; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    const float wt = ms == -INFINITY ? 0.f : exp2f(ms - mx);
    float av = wt * as, l = wt * ls;
    for (int off = cs >> 1; off > 0; off >>= 1) {
      av += __shfl_xor_sync(0xffffffffu, av, off);
      l += __shfl_xor_sync(0xffffffffu, l, off);
    }
    const int c = (crank << lw) + (t & (cw - 1));
    const float ov = settled(l > 0.f ? av / l : 0.f, ok && r == 0, g, c);
    if (ok && r == 0) {
      const int64_t hq = q0 + g;
      out[hq * FASA_HEAD_DIM + c] = ov;
      if (out_mirror) out_mirror[hq * FASA_HEAD_DIM + c] = ov;
      if (lse && c == 0) lse[hq] = l > 0.f ? (mx + log2f(l)) * 0.6931471805599453f : -INFINITY;
    }
  }
}
