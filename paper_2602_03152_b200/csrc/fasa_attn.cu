// FAC (Sec. 4.2, Eq. 6-7) and the dense FKV path (Sec. 5.1): split-K flash decoding with an
// online softmax, rows gathered by index for the sparse form, followed by a merge pass.
//
// Two kernels compute the partial results of a split.
//   decode_attn_mma_kernel (the default): the GQA group (<= 8 query heads) is the N = 8 of
//     mma.m16n8k16, so both products of the step run on tensor cores; described above the
//     kernel.
//   decode_attn_kernel (step mode 0, the first version): a KV row (128 bf16 = 256 bytes) is
//     read by a half-warp, 16 bytes per lane; a lane owns 8 channels of every row it sees and
//     keeps, for up to 4 query heads of the group, its slice of q and of the output
//     accumulator in registers, so one K/V row serves the whole group from a single load.
//     Groups of 5-8 heads use both half-warps of a warp on the same row (the second load is
//     merged by the coalescer).  Logits of a batch of 8 rows are completed with a transposing
//     xor-shuffle reduction (8 shuffles per head per batch); probabilities travel back to all
//     lanes through shared memory.  All multiply-adds are packed two-wide fp32 FMAs.
// decode_attn_merge_kernel then combines the splits of every (sequence, query head).  Where a
// unit needs at most 8 splits (selections up to 16384 rows), the splits of a unit form one
// thread-block cluster instead and merge through distributed shared memory inside the same
// launch: no partial result touches HBM, no second launch, no workspace.
#include <mutex>

#include "fasa_attn_core.cuh"
#include "fasa_cluster_merge.cuh"
#include "fasa_common.cuh"
#include "fasa_launch.cuh"
#include "fasa_score_core.cuh"

namespace cg = cooperative_groups;

namespace {

// Split-K partials of fasa_sparse_decode_attn_static: lives in the library image, so every
// GPU that loads the library holds these bytes until the process exits.
constexpr size_t kStaticScratchBytes = FASA_STATIC_SCRATCH_BYTES;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

constexpr int kAttnThreads = 128;
constexpr int kAttnHalfWarps = kAttnThreads / 16;  // 8
constexpr int kRB = 8;                              // rows per half-warp batch
constexpr int kPartialStride = FASA_HEAD_DIM + 2;   // m, l, acc[128] (base-2 domain)

struct AttnParams {
  const uint16_t* q;
  const uint16_t* k;
  const uint16_t* v;
  const int32_t* idx;      // sparse: [units][n_sel_max]
  const int32_t* n_rows;   // sparse: n_sel [units]; dense: seq_lens [batch]
  float* partial;          // [batch][n_q_heads][n_splits][kPartialStride]
  float* out;              // (cluster form: merged in the same launch)
  float* out_mirror;       // (cluster form, nullable: a second copy of out, e.g. mapped host memory)
  float* lse;
  int32_t* status;
  int n_q_heads, n_kv_heads, n_sets, group, max_len, n_sel_max, n_cap, chunk, n_splits;   // a unit = `group` query heads; n_sets units per sequence
  int64_t ksb, ksh, kst, vsb, vsh, vst;
  PageMap pm;              // paged caches (all zero: contiguous)
  float scale_log2;        // softmax_scale * log2(e)
  fasa_ksplit ks;          // split key cache (KSPLIT kernels): k holds the non-dominant channels only
  int q_len;               // blocks of queries (tensor-core kernel, sparse form): a "sequence" of the grid is a
                           // (sequence, query) pair and reads the cache of sequence b / q_len; 1 otherwise
};

// GP: heads per half-warp (1..4).  HWS: half-warps sharing a row (1: group <= 4, 2: group <= 8).
template <int GP, int HWS, bool SPARSE>
__global__ void __launch_bounds__(kAttnThreads)
decode_attn_kernel(const AttnParams p) {
  const int u = blockIdx.y;
  const SelUnit su = sel_unit(u, p.n_sets, p.group, p.n_q_heads, p.n_kv_heads);
  const int h = su.h;
  const int b = su.b;
  int n;
  if (SPARSE) {
    n = p.n_rows[u];
    if (n < 0 || n > p.n_cap) {
      atomicOr(p.status, FASA_DEV_NSEL_CLAMPED);
      n = n < 0 ? 0 : p.n_cap;
    }
  } else {
    n = clamp_len(p.n_rows[b], p.max_len, p.status);
  }
  const int split = blockIdx.x;
  const int r0 = split * p.chunk;
  if (r0 >= n) return;
  const int r1 = min(n, r0 + p.chunk);

  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int l16 = lane & 15;
  const int hw = lane >> 4;
  const int hwid = warp * 2 + hw;                          // half-warp within the CTA
  constexpr int kSlots = kAttnHalfWarps / HWS;             // row-batch streams per CTA
  constexpr int kWarpRows = kRB * (2 / HWS);               // rows one warp covers per iteration
  const int g0 = HWS == 1 ? 0 : hw * GP;                   // first head (within the group) of this half-warp

  __shared__ __align__(16) float s_p[kAttnHalfWarps][kRB][4];
  __shared__ __align__(16) float s_acc[kAttnHalfWarps][GP][FASA_HEAD_DIM];
  __shared__ float s_m[kAttnHalfWarps][GP];
  __shared__ float s_l[kAttnHalfWarps][GP];

  // q slice of this lane, pre-multiplied by scale * log2(e): logits live in the base-2 domain.
  float2 qf[GP][4];
#pragma unroll
  for (int g = 0; g < GP; ++g) {
    const bool head_ok = g0 + g < p.group;
    const uint16_t* qp =
        p.q + (su.q0 + (head_ok ? g0 + g : 0)) * FASA_HEAD_DIM + l16 * 8;
    uint4 w = *reinterpret_cast<const uint4*>(qp);
    const float sc = head_ok ? p.scale_log2 : 0.f;
    float2 t;
    t = bf16x2_to_f32x2(w.x); qf[g][0] = make_float2(t.x * sc, t.y * sc);
    t = bf16x2_to_f32x2(w.y); qf[g][1] = make_float2(t.x * sc, t.y * sc);
    t = bf16x2_to_f32x2(w.z); qf[g][2] = make_float2(t.x * sc, t.y * sc);
    t = bf16x2_to_f32x2(w.w); qf[g][3] = make_float2(t.x * sc, t.y * sc);
  }

  float2 acc[GP][4];
  float m[GP], lsum[GP];
#pragma unroll
  for (int g = 0; g < GP; ++g) {
    m[g] = -INFINITY;
    lsum[g] = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[g][e] = make_float2(0.f, 0.f);
  }

  const uint16_t* kbase = p.k + l16 * 8;
  const uint16_t* vbase = p.v + l16 * 8;
  const int32_t* irow = SPARSE ? p.idx + (int64_t)u * p.n_sel_max : nullptr;
  // The row of the batch whose finished logit lands in this lane after the reduction.
  const int my_row = ((l16 >> 3) & 1) * 4 + ((l16 >> 2) & 1) * 2 + ((l16 >> 1) & 1);

  // The trip count is the same for both half-warps of a warp (the shuffles below name all
  // 32 lanes); a half-warp whose batch starts past r1 runs it fully masked.
  for (int wbase = r0 + warp * kWarpRows; wbase < r1; wbase += (kAttnThreads / 32) * kWarpRows) {
    const int base = wbase + (HWS == 1 ? hw * kRB : 0);
    // all row indices first, then all row loads, so that no load waits on a previous row
    int tok[kRB];
#pragma unroll
    for (int i = 0; i < kRB; ++i) {
      const int r = base + i;
      tok[i] = SPARSE ? (r < r1 ? __ldg(irow + r) : 0) : r;
    }
    uint4 kk[kRB], vv[kRB];
#pragma unroll
    for (int i = 0; i < kRB; ++i) {
      const int r = base + i;
      if (r < r1) {
        int t = tok[i];
        if (SPARSE && (t < 0 || t >= p.max_len)) {
          atomicOr(p.status, FASA_DEV_IDX_CLAMPED);
          t = 0;
        }
        if (p.pm.table != nullptr) {
          kk[i] = ld_stream_u4(kbase + cache_row(p.pm, b, h, t, p.ksb, p.ksh, p.kst, p.status));
          vv[i] = ld_stream_u4(vbase + cache_row(p.pm, b, h, t, p.vsb, p.vsh, p.vst, p.status));
        } else {
          kk[i] = ld_stream_u4(kbase + b * p.ksb + h * p.ksh + (int64_t)t * p.kst);
          vv[i] = ld_stream_u4(vbase + b * p.vsb + h * p.vsh + (int64_t)t * p.vst);
        }
      } else {
        kk[i] = make_uint4(0u, 0u, 0u, 0u);
        vv[i] = make_uint4(0u, 0u, 0u, 0u);
      }
    }

    float alpha[GP];
#pragma unroll
    for (int g = 0; g < GP; ++g) {
      // partial logits of the 8 rows over this lane's 8 channels
      float part[kRB];
#pragma unroll
      for (int i = 0; i < kRB; ++i) part[i] = dot8(qf[g], kk[i]);
      // transposing reduction over the 16 lanes: 8 -> 4 -> 2 -> 1 rows per lane
      float p4[4], p2[2], p1;
      {
        const bool up = (l16 & 8) != 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float send = up ? part[i] : part[i + 4];
          const float keep = up ? part[i + 4] : part[i];
          p4[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
        }
      }
      {
        const bool up = (l16 & 4) != 0;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float send = up ? p4[i] : p4[i + 2];
          const float keep = up ? p4[i + 2] : p4[i];
          p2[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
        }
      }
      {
        const bool up = (l16 & 2) != 0;
        const float send = up ? p2[0] : p2[1];
        const float keep = up ? p2[1] : p2[0];
        p1 = keep + __shfl_xor_sync(0xffffffffu, send, 2);
      }
      p1 += __shfl_xor_sync(0xffffffffu, p1, 1);
      const float logit = (base + my_row < r1) ? p1 : -INFINITY;
      float bmax = logit;
      bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, 8));
      bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, 4));
      bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, 2));
      const float m_new = fmaxf(m[g], bmax);
      // m_new is finite here: the batch holds at least one real row with finite inputs.
      const float m_safe = m_new == -INFINITY ? 0.f : m_new;
      alpha[g] = exp2f(m[g] - m_safe);
      const float pr = exp2f(logit - m_safe);
      lsum[g] = lsum[g] * alpha[g] + ((l16 & 1) ? 0.f : pr);
      m[g] = m_new;
      if ((l16 & 1) == 0) s_p[hwid][my_row][g] = pr;
    }
    __syncwarp();

#pragma unroll
    for (int g = 0; g < GP; ++g) {
      const float2 a2 = make_float2(alpha[g], alpha[g]);
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[g][e] = __ffma2_rn(acc[g][e], a2, make_float2(0.f, 0.f));
    }
#pragma unroll
    for (int i = 0; i < kRB; ++i) {
      const float4 pi = *reinterpret_cast<const float4*>(&s_p[hwid][i][0]);
      const float pg[4] = {pi.x, pi.y, pi.z, pi.w};
      float2 vf[4];
      vf[0] = bf16x2_to_f32x2(vv[i].x);
      vf[1] = bf16x2_to_f32x2(vv[i].y);
      vf[2] = bf16x2_to_f32x2(vv[i].z);
      vf[3] = bf16x2_to_f32x2(vv[i].w);
#pragma unroll
      for (int g = 0; g < GP; ++g) {
        const float2 p2 = make_float2(pg[g], pg[g]);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[g][e] = __ffma2_rn(p2, vf[e], acc[g][e]);
      }
    }
    __syncwarp();  // s_p is rewritten by the next batch
  }

  // ---- combine the half-warps of this CTA, then write one partial per head -----------
#pragma unroll
  for (int g = 0; g < GP; ++g) {
    float l = lsum[g];
    l += __shfl_xor_sync(0xffffffffu, l, 8);
    l += __shfl_xor_sync(0xffffffffu, l, 4);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    if (l16 == 0) {
      s_m[hwid][g] = m[g];
      s_l[hwid][g] = l;
    }
    float4* dst = reinterpret_cast<float4*>(&s_acc[hwid][g][l16 * 8]);
    dst[0] = make_float4(acc[g][0].x, acc[g][0].y, acc[g][1].x, acc[g][1].y);
    dst[1] = make_float4(acc[g][2].x, acc[g][2].y, acc[g][3].x, acc[g][3].y);
  }
  __syncthreads();

  const int c = threadIdx.x;  // one channel per thread
  for (int gl = 0; gl < p.group; ++gl) {
    const int gi = HWS == 1 ? gl : gl % GP;      // index inside the half-warp
    const int hsel = HWS == 1 ? 0 : gl / GP;     // which half of each warp holds it
    float mx = -INFINITY;
#pragma unroll
    for (int s = 0; s < kSlots; ++s) {
      const int hwi = HWS == 1 ? s : s * 2 + hsel;
      mx = fmaxf(mx, s_m[hwi][gi]);
    }
    float a = 0.f, l = 0.f;
#pragma unroll
    for (int s = 0; s < kSlots; ++s) {
      const int hwi = HWS == 1 ? s : s * 2 + hsel;
      const float ms = s_m[hwi][gi];
      const float w = ms == -INFINITY ? 0.f : exp2f(ms - mx);
      a += w * s_acc[hwi][gi][c];
      l += w * s_l[hwi][gi];
    }
    float* dst = p.partial +
                 ((su.q0 + gl) * p.n_splits + split) * kPartialStride;
    dst[2 + c] = a;
    if (c == 0) {
      dst[0] = mx;
      dst[1] = l;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Tensor-core form: see fasa_attn_core.cuh.
constexpr int kMmaThreads = 128;
constexpr int kMmaWarps = kMmaThreads / 32;

// CLUSTER: the splits of a unit are the CTAs of one cluster (grid.x = cluster size) and merge
// in the same launch; otherwise each split writes its partial result for the merge kernel.
// HOSTMEM: K and V rows are copied through L1 (caches in page-locked host memory).  KSPLIT
// (Algorithm 2's Combine; sparse, contiguous, HOSTMEM): a key row is assembled in shared memory
// from its non-dominant channels (p.k, ascending channel order, the part that crosses the host
// link) followed by its dominant channels in proxy order (from the GPU-resident proxy); the
// query operand is loaded in the same channel order, so the logits are the same dot products
// summed in another order.
// (CTAs per SM: as many as the registers allow)
// TERMS: of a probability (see fasa_attn_core.cuh).
template <bool SPARSE, bool PAGED, bool CLUSTER, bool HOSTMEM = false, bool KSPLIT = false, int TERMS = 2>
__global__ void __launch_bounds__(kMmaThreads, KSPLIT || PAGED ? 4 : 5)
decode_attn_mma_kernel(const AttnParams p) {
  __shared__ ClusterMergeSmem s_merge;              // (CLUSTER only: written by the peers)
  if constexpr (CLUSTER) cluster_arrive_running();  // each waits for that much before it writes to a peer
  pdl_wait_for_predecessor();
  pdl_release_successor();
  const int u = blockIdx.y;
  const SelUnit su = sel_unit(u, p.n_sets, p.group, p.n_q_heads, p.n_kv_heads);
  const int b = su.b;
  int n;
  if (SPARSE) {
    n = p.n_rows[u];
    if (n < 0 || n > p.n_cap) {
      atomicOr(p.status, FASA_DEV_NSEL_CLAMPED);
      n = n < 0 ? 0 : p.n_cap;
    }
  } else {
    n = clamp_len(p.n_rows[b], p.max_len, p.status);
  }
  const int split = blockIdx.x;
  // In a cluster the splits share the rows the unit actually has (every CTA stays for the merge
  // anyway, and with rows far below the bound a fixed split size would leave most of them idle
  // while they hold their place on an SM); otherwise the split size is the planned one, which
  // the merge kernel knows.
  const int chunk = CLUSTER ? min(p.chunk, max(32, ((n + (int)gridDim.x - 1) / (int)gridDim.x + 31) & ~31)) : p.chunk;
  const int r0 = min(n, split * chunk);
  if (!CLUSTER && r0 >= n) return;
  const int r1 = min(n, r0 + chunk);

  const int lane = threadIdx.x & 31;
  extern __shared__ __align__(16) unsigned char attn_smem_raw[];
  uint32_t qb[8][2];
  attn_load_query<KSPLIT>(qb, p, su, lane);

  const int32_t* irow = SPARSE ? p.idx + (int64_t)u * p.n_sel_max : nullptr;

  // The CTA's slice of the index list goes to shared memory in one coalesced read (checked
  // once): a tile then costs one memory round trip (its rows), not two (its indices first).
  int32_t* s_idx = reinterpret_cast<int32_t*>(attn_smem_raw + sizeof(MmaSmem<kMmaWarps, TERMS>));
  if (SPARSE) {
    // Four entries in flight per thread: they are plain loads, as the kernel ahead may have written the list, which the compiler
    // does not move over the check's atomic (13 x 8 lists of 9-12 K rows: one at a time, and a fence at the start, 207.4 us a
    // step, now 203.6).
    constexpr int kAhead = 4;
    for (int i0 = threadIdx.x; i0 < r1 - r0; i0 += kAhead * kMmaThreads) {
      int ahead[kAhead];
#pragma unroll
      for (int j = 0; j < kAhead; ++j) ahead[j] = i0 + j * kMmaThreads < r1 - r0 ? irow[r0 + i0 + j * kMmaThreads] : 0;
      int pages[kAhead];                            // (looked up here once, not for each copy of a row's K and V)
      if constexpr (PAGED) {
#pragma unroll
        for (int j = 0; j < kAhead; ++j) pages[j] = page_of(p.pm, b / p.q_len, ahead[j] < 0 || ahead[j] >= p.max_len ? 0 : ahead[j]);
      }
#pragma unroll
      for (int j = 0; j < kAhead; ++j) {
        const int i = i0 + j * kMmaThreads;
        if (i >= r1 - r0) break;
        int tok = ahead[j];
        if (tok < 0 || tok >= p.max_len) {
          atomicOr(p.status, FASA_DEV_IDX_CLAMPED);
          tok = 0;
        }
        if constexpr (PAGED) {
          int page = pages[j];
          if (!page_ok(p.pm, page)) {
            atomicOr(p.status, FASA_DEV_PAGE_CLAMPED);
            page = 0;
          }
          tok = (page << p.pm.shift) | (tok & ((1 << p.pm.shift) - 1));
        }
        if constexpr (KSPLIT) {
          // a row that is resident on the GPU is entered as -1 - slot: it is then copied from there
          if (p.ks.res.tags != nullptr) {
            const int slot = fasa_resident_slot(p.ks.res, tok);
            if (slot >= 0 && p.ks.res.tags[(int64_t)su.kv * p.ks.res.slots_pad + slot] == tok) tok = -1 - slot;
          }
        }
        s_idx[i] = tok;
      }
    }
    __syncthreads();
  }

  float (*s_part)[kMergePartStride] = mma_part<kMmaWarps>(attn_smem_raw);
  attn_rows<kMmaWarps, SPARSE, PAGED, HOSTMEM, KSPLIT, TERMS>(p, su, b / p.q_len, qb, r0, r1, s_idx, attn_smem_raw, [&](int gl) {
    return CLUSTER ? &s_part[gl][0] : p.partial + ((su.q0 + gl) * p.n_splits + split) * kPartialStride;
  });
  if constexpr (CLUSTER) {
    __syncthreads();
    cluster_wait();
    cg::cluster_group cluster = cg::this_cluster();
    if constexpr (TERMS == 3)
      cluster_merge_store<kMmaThreads>(cluster, s_part, s_merge, p.group, su.q0, p.out, p.out_mirror, p.lse, [&](int g) {
        const int u = unit_again();
        const SelUnit s = sel_unit(u, p.n_sets, p.group, p.n_q_heads, p.n_kv_heads);
        ExactOutput<PAGED> e;
        e.q = p.q + (s.q0 + g) * FASA_HEAD_DIM;
        e.k = p.k + s.h * p.ksh + (PAGED ? 0 : (s.b / p.q_len) * p.ksb);
        e.v = p.v + s.h * p.vsh + (PAGED ? 0 : (s.b / p.q_len) * p.vsb);
        e.list = p.idx + (int64_t)u * p.n_sel_max;
        e.n = min(max(p.n_rows[u], 0), p.n_cap);
        e.status = p.status; e.pm = p.pm; e.ksb = p.ksb; e.kst = p.kst; e.vsb = p.vsb; e.vst = p.vst;
        e.b = (s.b / p.q_len); e.max_len = p.max_len; e.scale_log2 = p.scale_log2;
        return e;
      });
    else   // (long lists, the dense pass and split key caches go without, as ever)
      cluster_merge_store<kMmaThreads>(cluster, s_part, s_merge, p.group, su.q0, p.out, p.out_mirror, p.lse);
  }
}

// Merge pass: one CTA per (batch, query head); thread (c, j) takes channels 2 c and 2 c + 1 of the splits s = j, j + 8, ...,
// eight of them in flight at a time, then the eight partial merges are merged.  (Four ways and a channel per thread, the
// maxima read in a pass of their own: 8 us at 32 splits against 5 us.)
constexpr int kMergeWays = 8, kMergeThreads = FASA_HEAD_DIM / 2 * kMergeWays;
// ns partial results (m, l, acc[128]), `stride` floats apart (an even number), to out[128] and *lse (nullable).
__device__ __forceinline__ void merge_partials(const float* src, int64_t stride, int ns, float* out, float* lse) {
  const int c = threadIdx.x % (FASA_HEAD_DIM / 2), j = threadIdx.x / (FASA_HEAD_DIM / 2);
  __shared__ float s_m[kMergeWays], s_l[kMergeWays];
  __shared__ float2 s_a[kMergeWays][FASA_HEAD_DIM / 2];
  float mx = -INFINITY, l = 0.f;
  float2 a = make_float2(0.f, 0.f);
  for (int s0 = j; s0 < ns; s0 += 8 * kMergeWays) {
    float2 ml[8], as[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int s = s0 + i * kMergeWays;
      const float* row = src + (s < ns ? s : s0) * stride;
      ml[i] = *reinterpret_cast<const float2*>(row);
      as[i] = *reinterpret_cast<const float2*>(row + 2 + 2 * c);
      if (s >= ns) ml[i].x = -INFINITY;
    }
    float mn = mx;
#pragma unroll
    for (int i = 0; i < 8; ++i) mn = fmaxf(mn, ml[i].x);
    const float keep = mx == -INFINITY ? 0.f : exp2f(mx - mn);
    a.x *= keep;
    a.y *= keep;
    l *= keep;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float w = ml[i].x == -INFINITY ? 0.f : exp2f(ml[i].x - mn);
      a.x += w * as[i].x;
      a.y += w * as[i].y;
      l += w * ml[i].y;
    }
    mx = mn;
  }
  s_a[j][c] = a;
  if (c == 0) {
    s_m[j] = mx;
    s_l[j] = l;
  }
  __syncthreads();
  if (j != 0) return;
  float m_all = -INFINITY, l_all = 0.f;
#pragma unroll
  for (int k = 0; k < kMergeWays; ++k) m_all = fmaxf(m_all, s_m[k]);
  float2 a_all = make_float2(0.f, 0.f);
#pragma unroll
  for (int k = 0; k < kMergeWays; ++k) {
    const float w = s_m[k] == -INFINITY ? 0.f : exp2f(s_m[k] - m_all);
    a_all.x += w * s_a[k][c].x;
    a_all.y += w * s_a[k][c].y;
    l_all += w * s_l[k];
  }
  const bool any = ns > 0 && l_all > 0.f;
  out[2 * c] = any ? a_all.x / l_all : 0.f;
  out[2 * c + 1] = any ? a_all.y / l_all : 0.f;
  if (lse && c == 0) *lse = any ? (m_all + log2f(l_all)) * 0.6931471805599453f : -INFINITY;
}

template <bool SPARSE>
__global__ void __launch_bounds__(kMergeThreads)
decode_attn_merge_kernel(const float* partial, const int32_t* n_rows,
                         float* __restrict__ out, float* __restrict__ lse,
                         int32_t* __restrict__ status, int n_q_heads, int n_sets, int group,
                         int max_len, int n_cap, int chunk, int n_splits) {
  pdl_wait_for_predecessor();
  const int bh = blockIdx.x;
  const int b = bh / n_q_heads;
  const int hq = bh % n_q_heads;
  int n;
  if (SPARSE) {
    n = n_rows[b * n_sets + hq / group];
    n = n < 0 ? 0 : (n > n_cap ? n_cap : n);
  } else {
    n = n_rows[b];
    n = n < 0 ? 0 : (n > max_len ? max_len : n);
  }
  const int ns = min(n_splits, (n + chunk - 1) / chunk);
  merge_partials(partial + (int64_t)bh * n_splits * kPartialStride, kPartialStride, ns, out + (int64_t)bh * FASA_HEAD_DIM, lse ? lse + bh : nullptr);
}

// ---- dense pass over long contexts -----------------------------------------------------------------
// The rows of all (sequence, KV head) units, laid end to end in tiles of 16, are dealt out to the CTAs evenly by the lengths on
// the device, so ragged batches end together.
// A CTA whose share spans several units writes a partial result for each; segment (CTA i, unit u) is number i + u of
// the partial results (from one segment to the next exactly one of the two grows).  Bound by HBM.  Measured (back to back,
// with the merge) against splits of a fixed size: batch 4 at 20-60 K 131 -> 116 us, batch 16 x 4 heads at 9-18 K 94 -> 88 us,
// batch 1 at 30 K 32.2 -> 27.9 us, batch 8 at 64 K 336 -> 330 us; batch 4, 40 / 8 heads, 12-22 K 54.2 / 55.9 us.
struct DenseDeal {
  long long total;         // tiles of all units
  int n;                   // CTAs that take part
  int mine;                // tiles of a KV head of sequence `lane`
};
// (Products of tiles and CTAs are formed in 32 bits where they fit: a 64-bit division costs more than the rest of the set-up.)
__device__ __forceinline__ int dense_tiles(const int32_t* seq_lens, int b, int batch, int max_len, int32_t* status) {
  return b < batch ? (clamp_len(seq_lens[b], max_len, status) + 15) >> 4 : 0;
}
// One warp.  n_ctas: CTAs launched, of which the device holds `resident` at once; n_sm: 0 on pages.
__device__ __forceinline__ DenseDeal dense_deal(const int32_t* seq_lens, int batch, int n_kv_heads, int max_len, int n_ctas, int resident, int n_sm,
                                                int lane, int32_t* status) {
  DenseDeal d;
  d.mine = dense_tiles(seq_lens, lane, batch, max_len, status);
  d.total = __reduce_add_sync(0xffffffffu, d.mine);
  for (int b0 = 32; b0 < batch; b0 += 32) d.total += __reduce_add_sync(0xffffffffu, dense_tiles(seq_lens, b0 + lane, batch, max_len, status));
  d.total *= n_kv_heads;
  // Long contexts: 1.8 times as many shares as CTAs are resident.  With one share to each, the slowest SM ends last by a
  // twentieth of the launch (batch 8 x 8 heads at 64 K: 350 us, 330 with 1.8; batch 16 at 32 K 355 / 334; batch 4 at 64 K 184 /
  // 176); a number of shares just above a whole multiple leaves most SMs idle at the end (1.4: 348 us, 1.9: 346, 2.3: 339).
  // Less than 64 tiles to each: as many CTAs to each SM as get 64 (batch 1 at 73 K 60 -> 57 us, batch 4 at 17 K 55.7 -> 53.5).
  // Pages keep one share to each resident CTA (batch 8 at 64 K: 374 us, 414 with 1.8), and short contexts a few tiles to
  // each of a third of the CTAs, then 32 tiles to each before the others join: below that a CTA's start and its partial
  // result cost more than its share (70 MB of 2 x 4 heads at 17 K: 24.6 us with all CTAs, 22.2 with a third).
  if (n_sm > 0 && d.total >= (long long)kDenseTiles * resident) d.n = n_ctas;
  else if (n_sm > 0 && d.total >= 2ll * kDenseTiles * n_sm) d.n = (int)(d.total / ((long long)kDenseTiles * n_sm)) * n_sm;
  else d.n = (int)max(1ll, min((long long)resident, max(d.total >> 5, min(d.total >> 2, (long long)(resident / 3)))));
  return d;
}

template <bool PAGED, bool HOSTMEM>
__global__ void __launch_bounds__(kMmaThreads, PAGED ? 4 : 6)
dense_attn_kernel(const AttnParams p) {
  pdl_wait_for_predecessor();
  pdl_release_successor();
  const int lane = threadIdx.x & 31;
  const int batch = p.n_cap;                        // (the launch's number of sequences)
  const DenseDeal d = dense_deal(p.n_rows, batch, p.n_kv_heads, p.max_len, (int)gridDim.x, p.n_splits, p.chunk, lane, p.status);
  const int i = blockIdx.x;
  if (i >= d.n) return;
  long long x = d.total < (1 << 21) ? (uint32_t)d.total * (uint32_t)i / (uint32_t)d.n : d.total * i / d.n;
  const long long end = d.total < (1 << 21) ? (uint32_t)d.total * (uint32_t)(i + 1) / (uint32_t)d.n : d.total * (i + 1) / d.n;
  if (x >= end) return;
  // the sequence that tile x lies in
  int b = 0, tiles = 0;
  long long before = 0;                             // tiles of the sequences ahead of it
  for (int b0 = 0; b0 < batch; b0 += 32) {
    const int mine = b0 == 0 ? d.mine : dense_tiles(p.n_rows, b0 + lane, batch, p.max_len, p.status);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const uint32_t hits = __ballot_sync(0xffffffffu, before + (long long)incl * p.n_kv_heads > x);
    if (hits) {
      const int l = __ffs(hits) - 1;
      b = b0 + l;
      tiles = __shfl_sync(0xffffffffu, mine, l);
      before += (long long)(__shfl_sync(0xffffffffu, incl, l) - tiles) * p.n_kv_heads;
      break;
    }
    before += (long long)__shfl_sync(0xffffffffu, incl, 31) * p.n_kv_heads;
  }
  extern __shared__ __align__(16) unsigned char attn_smem_raw[];
  int h = (int)(x - before) / tiles, t0 = (int)(x - before) - h * tiles;      // (within a sequence: 32 bits)
  while (x < end) {                                 // uniform over the CTA: a segment per unit
    const int n = (int)min((long long)(tiles - t0), end - x);
    const int len = clamp_len(p.n_rows[b], p.max_len, p.status);
    const SelUnit su = sel_unit(b * p.n_kv_heads + h, p.n_kv_heads, p.group, p.n_q_heads, p.n_kv_heads);
    uint32_t qb[8][2];
    attn_load_query<false>(qb, p, su, lane);
    float* const dst = p.partial + (int64_t)(i + b * p.n_kv_heads + h) * p.group * kPartialStride;
    attn_rows<kMmaWarps, false, PAGED, HOSTMEM, false, 2>(p, su, b, qb, t0 * 16, min(len, (t0 + n) * 16), nullptr, attn_smem_raw,
                                                       [&](int gl) { return dst + gl * kPartialStride; });
    x += n;
    if (x < end) {
      t0 = 0;
      if (++h == p.n_kv_heads) {
        h = 0;
        do tiles = dense_tiles(p.n_rows, ++b, batch, p.max_len, p.status);
        while (tiles == 0 && b + 1 < batch);
      }
      __syncthreads();                              // the next segment's rows take over the combine area
    }
  }
}

// Merge of the segments of every (sequence, query head): one CTA each, as decode_attn_merge_kernel.
__global__ void __launch_bounds__(kMergeThreads)
dense_merge_kernel(const AttnParams p, int n_ctas) {
  pdl_wait_for_predecessor();
  const int bh = blockIdx.x, b = bh / p.n_q_heads, hq = bh % p.n_q_heads, h = hq / p.group;
  const int lane = threadIdx.x & 31, batch = p.n_cap;
  const DenseDeal d = dense_deal(p.n_rows, batch, p.n_kv_heads, p.max_len, n_ctas, p.n_splits, p.chunk, lane, p.status);
  long long first = 0;                              // this unit's first tile
  for (int b0 = 0; b0 < b; b0 += 32)
    first += __reduce_add_sync(0xffffffffu, b0 + lane < b ? (b0 == 0 ? d.mine : dense_tiles(p.n_rows, b0 + lane, batch, p.max_len, p.status)) : 0);
  const int tiles = b < 32 ? __shfl_sync(0xffffffffu, d.mine, b & 31) : dense_tiles(p.n_rows, b, batch, p.max_len, p.status);
  first = first * p.n_kv_heads + (long long)h * tiles;
  // tile x belongs to CTA ((x + 1) n - 1) / total
  auto cta_of = [&](long long y) {                  // y = x + 1
    return d.total < (1 << 21) ? (int)(((uint32_t)y * (uint32_t)d.n - 1u) / (uint32_t)d.total) : (int)((y * d.n - 1) / d.total);
  };
  const int i0 = tiles > 0 ? cta_of(first + 1) : 0;
  const int ns = tiles > 0 ? cta_of(first + tiles) - i0 + 1 : 0;
  merge_partials(p.partial + ((int64_t)(i0 + b * p.n_kv_heads + h) * p.group + hq % p.group) * kPartialStride, (int64_t)p.group * kPartialStride, ns,
                 p.out + (int64_t)bh * FASA_HEAD_DIM, p.lse ? p.lse + bh : nullptr);
}

// out_mirror (nullable): a second destination of out; *mirrored tells whether it was written
// (only the form that merges inside the attention launch can do that).  full_p: three terms of a probability (that form too).
template <bool SPARSE>
int32_t launch_attn(fasa_ctx* ctx, const void* q, const void* k, const void* v,
                    const int32_t* idx, const int32_t* n_rows, int n_upper, int n_sel_max,
                    float* out, float* lse, void* workspace, cudaStream_t s, float* out_mirror = nullptr,
                    bool* mirrored = nullptr, int q_len = 1, const fasa_ksplit* ksplit = nullptr, bool full_p = false) {
  if (mirrored) *mirrored = false;
  const fasa_config_t& c = ctx->cfg;
  if (!fasa_pages_ready(ctx)) return FASA_ERR_INVALID_ARG;
  // the dense pass treats a KV head with all its query heads as the unit
  const int n_sets = SPARSE ? ctx->n_sets : c.n_kv_heads;
  const int G = SPARSE ? ctx->sel_heads : ctx->group;
  const int n_seq = c.batch * q_len;                // rows of the grid's "batch" axis
  const fasa_split_plan plan = fasa_plan_splits(ctx, n_upper, n_seq * n_sets);
  AttnParams p;
  p.q_len = q_len;
  memset(&p.ks, 0, sizeof(p.ks));
  if (ksplit) p.ks = *ksplit;
  // caches in page-locked host memory are copied through L1 (contiguous caches, tensor-core kernel)
  const bool host = c.page_size == 0 && ctx->use_fused && (ksplit != nullptr || fasa_on_host(k));
  p.q = (const uint16_t*)q; p.k = (const uint16_t*)k; p.v = (const uint16_t*)v;
  p.idx = idx; p.n_rows = n_rows; p.partial = (float*)workspace; p.out = nullptr; p.out_mirror = nullptr; p.lse = nullptr; p.status = ctx->d_status;
  p.n_q_heads = c.n_q_heads; p.n_kv_heads = c.n_kv_heads; p.n_sets = n_sets; p.group = G;
  p.max_len = c.max_len; p.n_sel_max = n_sel_max; p.n_cap = n_upper; p.chunk = plan.chunk; p.n_splits = plan.n_splits;
  p.ksb = c.k_stride_b; p.ksh = c.k_stride_h; p.kst = c.k_stride_t;
  p.vsb = c.v_stride_b; p.vsh = c.v_stride_h; p.vst = c.v_stride_t;
  p.pm = fasa_page_map(ctx);
  p.scale_log2 = c.softmax_scale * 1.4426950408889634f;
  dim3 grid((unsigned)plan.n_splits, (unsigned)(n_seq * n_sets));
  if (ctx->use_fused) {   // default: the tensor-core kernel (mode 0 keeps the scalar one)
    const int max_smem = (int)(sizeof(MmaSmem<kMmaWarps, 3>) + 2080 * sizeof(int32_t));
    // One launch where the splits of a unit fit a portable cluster: the split count becomes a
    // power of two <= 8 (the nearest to the planned one) and the cluster merges by itself.
    int cs = 1;
    while (cs < 8 && cs * 3 < plan.n_splits * 2) cs *= 2;          // nearest power of two, ties up
    int cchunk = ((n_upper + cs - 1) / cs + 31) / 32 * 32;
    while (cs < 8 && cchunk > 2048) { cs *= 2; cchunk = ((n_upper + cs - 1) / cs + 31) / 32 * 32; }
    if (cchunk <= 2048) {
      p.chunk = cchunk; p.n_splits = cs; p.out = out; p.out_mirror = out_mirror; p.lse = lse;
      if (mirrored) *mirrored = out_mirror != nullptr;
      auto fn = c.page_size > 0 ? decode_attn_mma_kernel<SPARSE, true, true> : decode_attn_mma_kernel<SPARSE, false, true>;
      if (host) fn = decode_attn_mma_kernel<SPARSE, false, true, true>;
      if constexpr (SPARSE) {
        if (full_p) {
          fn = c.page_size > 0 ? decode_attn_mma_kernel<true, true, true, false, false, 3> : decode_attn_mma_kernel<true, false, true, false, false, 3>;
          if (host) fn = decode_attn_mma_kernel<true, false, true, true, false, 3>;
        }
        if (ksplit) fn = decode_attn_mma_kernel<true, false, true, true, true>;
      }
      const size_t smem = (full_p ? sizeof(MmaSmem<kMmaWarps, 3>) : sizeof(MmaSmem<kMmaWarps>)) + (SPARSE ? (size_t)cchunk * sizeof(int32_t) : 0);
      FASA_CUDA_TRY(ctx, cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem));
      FASA_CUDA_TRY(ctx, launch_after_predecessor(fn, dim3((unsigned)cs, grid.y), dim3(kMmaThreads), smem, s, cs, p));
      FASA_LAUNCH_CHECK(ctx);
      return FASA_OK;
    }
    if constexpr (!SPARSE) {
      p.out = out; p.lse = lse; p.n_cap = c.batch;
      p.n_splits = fasa_dense_resident(ctx); p.chunk = c.page_size > 0 ? 0 : ctx->n_sm;   // (what dense_deal asks for)
      auto fn = c.page_size > 0 ? dense_attn_kernel<true, false> : dense_attn_kernel<false, false>;
      if (host) fn = dense_attn_kernel<false, true>;
      const int n_ctas = fasa_dense_ctas(ctx);
      FASA_CUDA_TRY(ctx, cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem));
      FASA_CUDA_TRY(ctx, launch_after_predecessor(fn, dim3((unsigned)n_ctas), dim3(kMmaThreads), sizeof(MmaSmem<kMmaWarps>), s, 0, p));
      FASA_LAUNCH_CHECK(ctx);
      FASA_CUDA_TRY(ctx, launch_after_predecessor(dense_merge_kernel, dim3((unsigned)(c.batch * c.n_q_heads)), dim3(kMergeThreads),
                                                  (size_t)0, s, 0, p, n_ctas));
      FASA_LAUNCH_CHECK(ctx);
      return FASA_OK;
    } else {
    auto fn = c.page_size > 0 ? decode_attn_mma_kernel<true, true, false> : decode_attn_mma_kernel<true, false, false>;
    if (host) fn = decode_attn_mma_kernel<true, false, false, true>;
    if (ksplit) fn = decode_attn_mma_kernel<true, false, false, true, true>;
    // (+ the slice of the index list: chunk <= 2048 rows)
    const size_t smem = sizeof(MmaSmem<kMmaWarps>) + (size_t)plan.chunk * sizeof(int32_t);
    FASA_CUDA_TRY(ctx, cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem));
    FASA_CUDA_TRY(ctx, launch_after_predecessor(fn, grid, dim3(kMmaThreads), smem, s, 0, p));
    }
  } else if (G == 1) decode_attn_kernel<1, 1, SPARSE><<<grid, kAttnThreads, 0, s>>>(p);
  else if (G == 2) decode_attn_kernel<2, 1, SPARSE><<<grid, kAttnThreads, 0, s>>>(p);
  else if (G == 3) decode_attn_kernel<3, 1, SPARSE><<<grid, kAttnThreads, 0, s>>>(p);
  else if (G == 4) decode_attn_kernel<4, 1, SPARSE><<<grid, kAttnThreads, 0, s>>>(p);
  else if (G <= 6) decode_attn_kernel<3, 2, SPARSE><<<grid, kAttnThreads, 0, s>>>(p);
  else decode_attn_kernel<4, 2, SPARSE><<<grid, kAttnThreads, 0, s>>>(p);
  FASA_LAUNCH_CHECK(ctx);
  FASA_CUDA_TRY(ctx, launch_after_predecessor(
      decode_attn_merge_kernel<SPARSE>, dim3((unsigned)(n_seq * c.n_q_heads)), dim3(kMergeThreads),
      (size_t)0, s, 0, (const float*)workspace, n_rows, out, lse, ctx->d_status, (int)c.n_q_heads, (int)n_sets,
      (int)G, (int)c.max_len, (int)n_upper, (int)plan.chunk, (int)plan.n_splits));
  FASA_LAUNCH_CHECK(ctx);
  return FASA_OK;
}

bool aligned(const void* p, uintptr_t a) { return ((uintptr_t)p & (a - 1)) == 0; }

}  // namespace

extern "C" int32_t fasa_sparse_decode_attn(fasa_ctx_t* ctx, const void* q, const void* k_cache,
                                           const void* v_cache, const int32_t* idx,
                                           const int32_t* n_sel, int32_t n_sel_max, float* out,
                                           float* lse, void* workspace, void* stream) {
  if (!ctx || !q || !k_cache || !v_cache || !idx || !n_sel || !out || !workspace || n_sel_max <= 0)
    return FASA_ERR_INVALID_ARG;
  if (!aligned(q, 16) || !aligned(k_cache, 16) || !aligned(v_cache, 16) || !aligned(workspace, 256))
    return FASA_ERR_INVALID_ARG;
  const int n_upper = n_sel_max < ctx->cfg.max_len ? n_sel_max : ctx->cfg.max_len;
  return launch_attn<true>(ctx, q, k_cache, v_cache, idx, n_sel, n_upper, n_sel_max, out, lse,
                           workspace, (cudaStream_t)stream);
}

// fasa_sparse_decode_attn with a second destination for the output (the host-buffer step).
int32_t fasa_sparse_attn_mirrored(fasa_ctx* ctx, const void* q, const void* k_cache, const void* v_cache,
                                  const int32_t* idx, const int32_t* n_sel, int32_t n_sel_max, float* out,
                                  float* lse, void* workspace, cudaStream_t stream, float* out_mirror, bool* mirrored, bool full_p) {
  const int n_upper = n_sel_max < ctx->cfg.max_len ? n_sel_max : ctx->cfg.max_len;
  return launch_attn<true>(ctx, q, k_cache, v_cache, idx, n_sel, n_upper, n_sel_max, out, lse, workspace, stream,
                           out_mirror, mirrored, 1, nullptr, full_p);
}

// FAC over a split key cache (Algorithm 2: Combine, then Eq. 6-7): k_nondom holds the non-dominant
// channels of every key, the proxy their dominant ones.
int32_t fasa_attn_split_keys(fasa_ctx* ctx, const void* q, const void* k_nondom, const void* v_cache, const void* proxy_k,
                             const int32_t* idx, const int32_t* n_sel, int32_t n_sel_max, float* out, float* lse,
                             void* workspace, cudaStream_t stream) {
  const fasa_config_t& c = ctx->cfg;
  fasa_ksplit ks;
  ks.proxy = (const unsigned char*)proxy_k; ks.ndchan = ctx->d_ndchan; ks.chan = ctx->d_chan;
  ks.chunks = ctx->chunks; ks.nd = FASA_HEAD_DIM - 2 * c.n_dom;
  ks.res = fasa_resident_of(ctx);
  // (the kernel addresses k_nondom with the K strides: rows of nd elements, dense per unit)
  fasa_ctx tmp = *ctx;
  tmp.cfg.k_stride_t = ks.nd;
  tmp.cfg.k_stride_h = (int64_t)c.max_len * ks.nd;
  tmp.cfg.k_stride_b = tmp.cfg.k_stride_h * c.n_kv_heads;
  const int n_upper = n_sel_max < c.max_len ? n_sel_max : c.max_len;
  int32_t st = launch_attn<true>(&tmp, q, k_nondom, v_cache, idx, n_sel, n_upper, n_sel_max, out, lse, workspace, stream,
                                 nullptr, nullptr, 1, &ks);
  ctx->launches = tmp.launches;
  memcpy(ctx->cuda_err, tmp.cuda_err, sizeof(ctx->cuda_err));
  return st;
}

extern "C" int32_t fasa_sparse_decode_attn_batched(fasa_ctx_t* ctx, const void* q, const void* k_cache,
                                                   const void* v_cache, const int32_t* idx, const int32_t* n_sel,
                                                   int32_t q_len, int32_t n_sel_max, float* out, float* lse,
                                                   void* workspace, void* stream) {
  if (!ctx || !q || !k_cache || !v_cache || !idx || !n_sel || !out || !workspace || n_sel_max <= 0)
    return FASA_ERR_INVALID_ARG;
  if (!aligned(q, 16) || !aligned(k_cache, 16) || !aligned(v_cache, 16) || !aligned(workspace, 256))
    return FASA_ERR_INVALID_ARG;
  if (q_len < 1 || q_len > FASA_MAX_QLEN || !ctx->use_fused) return FASA_ERR_UNSUPPORTED;   // (tensor-core kernel only)
  if ((long long)ctx->cfg.batch * q_len * ctx->n_sets > 65535) return FASA_ERR_UNSUPPORTED;
  const int n_upper = n_sel_max < ctx->cfg.max_len ? n_sel_max : ctx->cfg.max_len;
  // (beyond 16384 rows per unit the splits no longer merge inside one cluster, and the workspace
  // is sized for single queries)
  if (q_len > 1 && n_upper > 16384) return FASA_ERR_UNSUPPORTED;
  return launch_attn<true>(ctx, q, k_cache, v_cache, idx, n_sel, n_upper, n_sel_max, out, lse, workspace,
                           (cudaStream_t)stream, nullptr, nullptr, q_len);
}

extern "C" int32_t fasa_full_decode_attn(fasa_ctx_t* ctx, const void* q, const void* k_cache,
                                         const void* v_cache, const int32_t* seq_lens, float* out,
                                         float* lse, void* workspace, void* stream) {
  if (!ctx || !q || !k_cache || !v_cache || !seq_lens || !out || !workspace)
    return FASA_ERR_INVALID_ARG;
  if (!aligned(q, 16) || !aligned(k_cache, 16) || !aligned(v_cache, 16) || !aligned(workspace, 256))
    return FASA_ERR_INVALID_ARG;
  return launch_attn<false>(ctx, q, k_cache, v_cache, nullptr, seq_lens, ctx->cfg.max_len, 0, out,
                            lse, workspace, (cudaStream_t)stream);
}

// ---- variant for callers that cannot allocate device memory --------------------------------

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_scratch_mutex;
void* g_scratch_ptr[kMaxDevices];   // device address of g_static_scratch, per device ordinal
}  // namespace

extern "C" int32_t fasa_sparse_decode_attn_static(fasa_ctx_t* ctx, const void* q,
                                                  const void* k_cache, const void* v_cache,
                                                  const int32_t* idx, const int32_t* n_sel,
                                                  int32_t n_sel_max, float* out, float* lse,
                                                  void* stream) {
  if (!ctx || !q || !k_cache || !v_cache || !idx || !n_sel || !out || n_sel_max <= 0)
    return FASA_ERR_INVALID_ARG;
  if (!aligned(q, 16) || !aligned(k_cache, 16) || !aligned(v_cache, 16)) return FASA_ERR_INVALID_ARG;
  const fasa_config_t& c = ctx->cfg;
  const int n_upper = n_sel_max < c.max_len ? n_sel_max : c.max_len;
  const fasa_split_plan plan = fasa_plan_splits(ctx, n_upper, c.batch * ctx->n_sets);
  const size_t need = (size_t)c.batch * c.n_q_heads * (size_t)plan.n_splits * kPartialStride * sizeof(float);
  if (need > kStaticScratchBytes) return FASA_ERR_WORKSPACE;

  // The symbol names a different copy of the array on each device: its address is looked up
  // once per device, with that device current (the name itself is not a device pointer).
  int dev = -1;
  FASA_CUDA_TRY(ctx, cudaGetDevice(&dev));
  if (dev != ctx->device || dev < 0 || dev >= kMaxDevices) return FASA_ERR_INVALID_ARG;
  void* scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (!g_scratch_ptr[dev]) {
      void* p = nullptr;
      FASA_CUDA_TRY(ctx, cudaGetSymbolAddress(&p, g_static_scratch));
      g_scratch_ptr[dev] = p;
    }
    scratch = g_scratch_ptr[dev];
  }
  return launch_attn<true>(ctx, q, k_cache, v_cache, idx, n_sel, n_upper, n_sel_max, out, lse,
                           scratch, (cudaStream_t)stream);
}
