// Offline calibration of the dominant FCs (Algorithm 1): the contextual agreement CA of every
// FC with the full head (Sec. 3.3, Eq. 4), accumulated over samples, and the choice of the F
// FCs with the highest mean.
//
// One call takes a batch of (query, key cache) pairs laid out as for a decode step.  A sample
// is a (sequence, query head) pair.  Three stages, all on the caller's stream:
//   1. calib_score_kernel: the keys' channel pairs, FC-major (4 bytes per position, FC and KV head), and the
//      full-head raw scores alpha[j] (Eq. 2) of every query head;
//   2. TopK-I of each of a sample's 65 rows (one CTA per row, no forced positions): the single-FC raw
//      scores alpha^(i)[j] (Eq. 3) are evaluated from the channel pairs as the row is read, so the query heads
//      of a group share one row of pairs and no single-FC score travels through memory;
//   3. calib_intersect_kernel: |TopK-I(alpha) n TopK-I(alpha^(i))| for every i, added to the
//      caller's running counts.
// Measured (ncu), 32 samples of 24 K positions (8 KV heads): stage 1 70 -> 27 us (it wrote 65 score rows per
// sample), stage 2 94 -> 72 us, stage 3 57 -> 6.6 us (binary searches by 32 CTAs -> bit maps in 256).
// Which index enters a top-k set is decided by fp32 values with a fixed evaluation order:
// alpha^(i) = fl(q_c0 k_c0 + q_c1 k_c1) (the products of bf16 values are exact in fp32, so a fused
// multiply-add rounds the same once) and alpha = ((alpha^(0) + alpha^(1)) + alpha^(2)) + ...; equal
// scores keep the lower index.
#include <algorithm>
#include <vector>

#include "fasa_common.cuh"
#include "fasa_launch.cuh"

namespace {

constexpr int kFc = FASA_HEAD_DIM / 2;        // FCs per head
constexpr int kRows = kFc + 1;                // score rows per sample: the FCs, then the full head
constexpr int kTok = 128;                     // positions per CTA of the first stage
constexpr int kRowWords = kFc + 4;            // words of a staged key: 64 pairs, padded so that 16-byte accesses spread over the banks

// grid (ceil(max_len / 128), batch * n_kv_heads), 128 threads.  Bound by HBM: the keys are read once, a copy of the
// same size (the pairs) is written.  A key's 64 pairs are staged in shared memory in FC order, whatever the pairing;
// then a thread owns a position: it writes its pairs (a warp 128 consecutive bytes of one FC at a time) and sums the
// FCs of four query heads at a time.
template <bool PAGED>
__global__ void __launch_bounds__(kTok)
calib_score_kernel(const uint16_t* __restrict__ q, const uint16_t* __restrict__ k, const int32_t* __restrict__ seq_lens,
                   uint32_t* __restrict__ pairs, float* __restrict__ full, int32_t* __restrict__ status, int n_q_heads,
                   int n_kv_heads, int max_len, int64_t stride, int pairing, int64_t ksb, int64_t ksh, int64_t kst, const PageMap pm) {
  const int u = blockIdx.y, b = u / n_kv_heads, h = u % n_kv_heads, group = n_q_heads / n_kv_heads;
  const int tid = threadIdx.x;
  const int len = clamp_len(seq_lens[b], max_len, status);
  const int base = blockIdx.x * kTok;
  if (base >= len) return;
  __shared__ __align__(16) uint32_t s_k[kTok][kRowWords];
  __shared__ __align__(16) float2 s_q[kFc][FASA_MAX_GROUP];
  for (int i = tid; i < kFc * group; i += kTok) {
    const int fc = i % kFc, g = i / kFc;
    const uint16_t* qrow = q + ((int64_t)b * n_q_heads + h * group + g) * FASA_HEAD_DIM;
    s_q[fc][g] = make_float2(bf16_bits_to_f32(qrow[pairing == 0 ? fc : 2 * fc]), bf16_bits_to_f32(qrow[pairing == 0 ? fc + kFc : 2 * fc + 1]));
  }
  const bool whole = (reinterpret_cast<uintptr_t>(k) & 15) == 0;    // (the strides are multiples of 16 bytes)
  auto load8 = [&](const uint16_t* p) -> uint4 {
    if (whole) return *reinterpret_cast<const uint4*>(p);
    return make_uint4(p[0] | (uint32_t)p[1] << 16, p[2] | (uint32_t)p[3] << 16, p[4] | (uint32_t)p[5] << 16, p[6] | (uint32_t)p[7] << 16);
  };
  // eight threads to a key: 16 bytes from each half of the row (pairing 0), or 32 consecutive bytes
#pragma unroll 4
  for (int r = tid >> 3; r < kTok; r += kTok / 8) {
    const int c = (tid & 7) * 8, tok = min(base + r, len - 1);
    const uint16_t* row = PAGED ? k + cache_row(pm, b, h, tok, ksb, ksh, kst, status) : k + b * ksb + h * ksh + (int64_t)tok * kst;
    const uint4 x = load8(row + (pairing == 0 ? c : 2 * c)), y = load8(row + (pairing == 0 ? c + kFc : 2 * c + 8));
    uint4 lo = x, hi = y;
    if (pairing == 0) {                                             // (x's element i, y's element i)
      lo = make_uint4(__byte_perm(x.x, y.x, 0x5410), __byte_perm(x.x, y.x, 0x7632), __byte_perm(x.y, y.y, 0x5410), __byte_perm(x.y, y.y, 0x7632));
      hi = make_uint4(__byte_perm(x.z, y.z, 0x5410), __byte_perm(x.z, y.z, 0x7632), __byte_perm(x.w, y.w, 0x5410), __byte_perm(x.w, y.w, 0x7632));
    }
    *reinterpret_cast<uint4*>(&s_k[r][c]) = lo;
    *reinterpret_cast<uint4*>(&s_k[r][c + 4]) = hi;
  }
  __syncthreads();
  const int tok = base + tid;
  uint32_t* dst = pairs + (int64_t)u * kFc * stride + tok;
  for (int g0 = 0; g0 < group; g0 += 4) {                           // four query heads at a time
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int f4 = 0; f4 < kFc; f4 += 4) {
      const uint4 w4 = *reinterpret_cast<const uint4*>(&s_k[tid][f4]);
      const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
      if (g0 == 0 && tok < len) {
#pragma unroll
        for (int e = 0; e < 4; ++e) dst[(f4 + e) * stride] = w[e];
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 kv = bf16x2_to_f32x2(w[e]);
        const float4 qa = *reinterpret_cast<const float4*>(&s_q[f4 + e][g0]), qb = *reinterpret_cast<const float4*>(&s_q[f4 + e][g0 + 2]);
        acc[0] = __fadd_rn(acc[0], fmaf(qa.x, kv.x, qa.y * kv.y));
        acc[1] = __fadd_rn(acc[1], fmaf(qa.z, kv.x, qa.w * kv.y));
        acc[2] = __fadd_rn(acc[2], fmaf(qb.x, kv.x, qb.y * kv.y));
        acc[3] = __fadd_rn(acc[3], fmaf(qb.z, kv.x, qb.w * kv.y));
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (g0 + e < group && tok < len) full[((int64_t)b * n_q_heads + h * group + g0 + e) * stride + tok] = acc[e] + 0.0f;   // (-0 becomes +0)
  }
}

// grid (samples, kParts): a CTA marks the positions of the full head's list in a bit map and every warp counts the
// marked positions of an FC list at a time.
constexpr int kParts = 8;
__global__ void __launch_bounds__(256)
calib_intersect_kernel(const int32_t* idx, const int32_t* seq_lens, unsigned long long* counts, unsigned long long* n_used,
                       int n_q_heads, int max_len, int top_k) {
  extern __shared__ uint32_t marked[];
  const int u = blockIdx.x;
  const int b = u / n_q_heads, hq = u % n_q_heads;
  for (int i = threadIdx.x; i < (max_len + 31) >> 5; i += blockDim.x) marked[i] = 0u;
  pdl_wait_for_predecessor();
  pdl_release_successor();
  int len = seq_lens[b];
  len = len > max_len ? max_len : len;
  if (len <= top_k) return;                   // every position is selected: not a sample
  const int32_t* lists = idx + (int64_t)u * kRows * top_k;
  __syncthreads();
  for (int i = threadIdx.x; i < top_k; i += blockDim.x) {
    const int pos = lists[(int64_t)kFc * top_k + i];
    atomicOr(&marked[pos >> 5], 1u << (pos & 31));
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  for (int i = blockIdx.y * n_warps + warp; i < kFc; i += kParts * n_warps) {
    const int32_t* mine = lists + (int64_t)i * top_k;
    uint32_t common = 0;
#pragma unroll 4
    for (int e = lane; e < top_k; e += 32) common += (marked[mine[e] >> 5] >> (mine[e] & 31)) & 1u;
    common = __reduce_add_sync(0xffffffffu, common);
    if (lane == 0 && common > 0) atomicAdd(&counts[(int64_t)hq * kFc + i], (unsigned long long)common);
  }
  if (blockIdx.y == 0 && threadIdx.x == 0) atomicAdd(&n_used[hq], 1ull);
}

struct CalibLayout {
  size_t pairs, full, idx, n_sel, total;
  int64_t stride;                             // positions per row
};

CalibLayout calib_layout(const fasa_ctx* ctx, int top_k) {
  const fasa_config_t& c = ctx->cfg;
  const size_t samples = (size_t)c.batch * c.n_q_heads;
  CalibLayout l;
  l.stride = ((int64_t)c.max_len + 3) & ~3ll;
  l.pairs = 0;
  l.full = fasa_align_up((size_t)c.batch * c.n_kv_heads * kFc * (size_t)l.stride * sizeof(uint32_t), 256);
  l.idx = l.full + fasa_align_up(samples * (size_t)l.stride * sizeof(float), 256);
  l.n_sel = l.idx + fasa_align_up(samples * kRows * (size_t)top_k * sizeof(int32_t), 256);
  l.total = l.n_sel + fasa_align_up(samples * kRows * sizeof(int32_t), 256);
  return l;
}

bool calib_args_ok(const fasa_ctx* ctx, int top_k) {
  const fasa_config_t& c = ctx->cfg;
  return top_k >= 1 && top_k <= c.max_len && top_k <= 8192 &&
         (long long)c.batch * c.n_q_heads * kRows <= 65535;      // grid.y of the select launch
}

}  // namespace

extern "C" int32_t fasa_calib_workspace_bytes(const fasa_ctx_t* ctx, int32_t top_k, size_t* out_bytes) {
  if (!ctx || !out_bytes) return FASA_ERR_INVALID_ARG;
  if (!calib_args_ok(ctx, top_k)) return FASA_ERR_UNSUPPORTED;
  *out_bytes = calib_layout(ctx, top_k).total;
  return FASA_OK;
}

extern "C" int32_t fasa_calib_accumulate(fasa_ctx_t* ctx, const void* q, const void* k_cache,
                                         const int32_t* seq_lens, int32_t top_k, int64_t* ca_counts,
                                         int64_t* n_used, void* workspace, void* stream) {
  if (!ctx || !q || !k_cache || !seq_lens || !ca_counts || !n_used || !workspace) return FASA_ERR_INVALID_ARG;
  if (((uintptr_t)workspace & 255) != 0 || ((uintptr_t)ca_counts & 7) != 0 || ((uintptr_t)n_used & 7) != 0)
    return FASA_ERR_INVALID_ARG;
  if (!fasa_pages_ready(ctx)) return FASA_ERR_INVALID_ARG;
  if (!calib_args_ok(ctx, top_k) || ctx->fused_cs <= 0) return FASA_ERR_UNSUPPORTED;
  const fasa_config_t& c = ctx->cfg;
  cudaStream_t s = (cudaStream_t)stream;
  const CalibLayout l = calib_layout(ctx, top_k);
  uint32_t* pairs = reinterpret_cast<uint32_t*>((char*)workspace + l.pairs);
  float* full = reinterpret_cast<float*>((char*)workspace + l.full);
  int32_t* idx = reinterpret_cast<int32_t*>((char*)workspace + l.idx);
  int32_t* n_sel = reinterpret_cast<int32_t*>((char*)workspace + l.n_sel);
  const int samples = c.batch * c.n_q_heads;

  dim3 grid((unsigned)((c.max_len + kTok - 1) / kTok), (unsigned)(c.batch * c.n_kv_heads));
  auto score = c.page_size > 0 ? calib_score_kernel<true> : calib_score_kernel<false>;
  score<<<grid, kTok, 0, s>>>((const uint16_t*)q, (const uint16_t*)k_cache, seq_lens, pairs, full, ctx->d_status, c.n_q_heads,
                              c.n_kv_heads, c.max_len, l.stride, c.rope_pairing, c.k_stride_b, c.k_stride_h, c.k_stride_t,
                              fasa_page_map(ctx));
  FASA_LAUNCH_CHECK(ctx);
  fasa_calib_rows rows;
  rows.pairs = pairs; rows.q = (const uint16_t*)q; rows.stride = l.stride; rows.group = ctx->group; rows.pairing = c.rope_pairing;
  const int32_t st = fasa_topk_row_launch(ctx, full, seq_lens, top_k, top_k, idx, n_sel, c.n_q_heads * kRows, 0, 0, s, 1, &rows);
  if (st != FASA_OK) return st;
  FASA_CUDA_TRY(ctx, launch_after_predecessor(calib_intersect_kernel, dim3((unsigned)samples, kParts), dim3(256),
                                              (size_t)((c.max_len + 31) / 32) * sizeof(uint32_t), s, 0, (const int32_t*)idx, seq_lens,
                                              reinterpret_cast<unsigned long long*>(ca_counts),
                                              reinterpret_cast<unsigned long long*>(n_used), (int)c.n_q_heads, (int)c.max_len, (int)top_k));
  FASA_LAUNCH_CHECK(ctx);
  return FASA_OK;
}

extern "C" int32_t fasa_calib_select(int32_t n_q_heads, int32_t n_kv_heads, const int64_t* ca_counts_host,
                                     const int64_t* n_used_host, int32_t top_k, int32_t n_dom,
                                     int32_t* dom_fc_host, double* mean_ca_host) {
  if (!ca_counts_host || !n_used_host || !dom_fc_host) return FASA_ERR_INVALID_ARG;
  if (n_q_heads <= 0 || n_kv_heads <= 0 || n_q_heads % n_kv_heads != 0 || top_k < 1) return FASA_ERR_INVALID_ARG;
  if (n_dom < 1 || n_dom > kFc) return FASA_ERR_UNSUPPORTED;
  const int group = n_q_heads / n_kv_heads;
  for (int h = 0; h < n_kv_heads; ++h) {
    // the query heads of a KV head read the same keys: their samples are pooled
    int64_t sum[kFc] = {0}, samples = 0;
    for (int g = h * group; g < (h + 1) * group; ++g) {
      samples += n_used_host[g];
      for (int i = 0; i < kFc; ++i) sum[i] += ca_counts_host[(int64_t)g * kFc + i];
    }
    int order[kFc];
    for (int i = 0; i < kFc; ++i) order[i] = i;
    std::stable_sort(order, order + kFc, [&](int a, int b) { return sum[a] > sum[b]; });   // equal means: lower FC first
    std::sort(order, order + n_dom);
    for (int r = 0; r < n_dom; ++r) dom_fc_host[(int64_t)h * n_dom + r] = order[r];
    if (mean_ca_host)
      for (int i = 0; i < kFc; ++i)
        mean_ca_host[(int64_t)h * kFc + i] = samples > 0 ? (double)sum[i] / ((double)samples * (double)top_k) : 0.0;
  }
  return FASA_OK;
}
