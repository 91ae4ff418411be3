// The tensor-core core of attention over a list of rows, shared by the split-K attention kernel and by the
// kernel that selects and attends in one launch.
#pragma once

#include "fasa_cluster_merge.cuh"
#include "fasa_common.cuh"
#include "fasa_score_core.cuh"

#ifdef __CUDACC__

// ---------------------------------------------------------------------------------------------
// Tensor-core form.  With a GQA group of G query heads the two products of a decode step are
// [rows x 128] . [128 x G] (logits) and [128 x rows] . [rows x G] (output, transposed): G <= 8
// is exactly the N = 8 of mma.m16n8k16.  The scalar kernel of fasa_attn.cu spends ~60 instructions per
// K/V row per four heads and is bound by instruction issue (0.67 of the copy bandwidth at
// G = 4, 0.3 at G = 7); here a warp handles 16 rows with 8 + 16 MMAs.
//   - K and V rows go to shared memory with 16-byte cp.async copies (row stride padded by 16
//     bytes, so ldmatrix reads them without bank conflicts);
//   - logits: A = K tile via ldmatrix.x4, B = q (bf16, exact) in registers; the softmax scale
//     is applied to the fp32 result;
//   - online softmax per head on the accumulator fragment (a thread owns heads 2t, 2t+1 of
//     rows g, g+8; row maxima and sums by xor-shuffles over g);
//   - output: A = V^T via ldmatrix.x4.trans, B = P^T, split into bf16 terms; a MMA per block and term.
//     Two terms hold 17 bits of a probability, three all 24 (outputs of 64 to 256 rows: 1.6e-6 and
//     2.5e-7 of their norm); fasa_full_probabilities says where the third is taken.
constexpr int kRowPad = FASA_HEAD_DIM + 8;          // bf16 elements per staged row (272 bytes)

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
// The same through L1 ("cache all levels"): rows that live in page-locked HOST memory cross the
// host link in full 128-byte requests this way, at twice the rate of the L2-only form (measured:
// 50 vs 25 GB/s of a 55 GB/s link); for rows in HBM the L2-only form above is the faster one.
__device__ __forceinline__ void cp_async16_ca(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// waits until at most N of this thread's committed groups are still in flight
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], const void* row) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(row)));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], const void* row) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(row)));
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// the same with k = 8
__device__ __forceinline__ void mma1688(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(b));
}
// two fp32 values rounded to nearest bf16, x in the low half
__device__ __forceinline__ uint32_t pack_bf16(float x, float y) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(y), "f"(x));
  return r;
}
// round-to-nearest-even fp32 -> bf16 bits (finite inputs)
__device__ __forceinline__ uint32_t f32_to_bf16_bits(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u + 0x7fffu + ((u >> 16) & 1u)) >> 16;
}

template <int WARPS, int TERMS = 2>
struct MmaSmem {
  uint16_t k[WARPS][16][kRowPad];
  uint16_t v[WARPS][16][kRowPad];
  uint16_t p[TERMS][WARPS][8][16];                  // terms of P^T: [head][row]
};
// After the last row the staging memory becomes the combine area: [WARPS][8] accumulators of 128 channels, then
// [WARPS][8][2] running maxima and sums, then one partial result per head.  (The stride of an accumulator keeps a
// warp's stores, four heads two apart by eight channels, on 32 banks.)
constexpr int kAccStride = FASA_HEAD_DIM + 4;
template <int WARPS>
__host__ __device__ constexpr size_t mma_combine_bytes() {
  return ((size_t)WARPS * 8 * (kAccStride + 2) + 8 * kMergePartStride) * sizeof(float);
}
template <int WARPS>
__device__ __forceinline__ float (*mma_part(unsigned char* smem))[kMergePartStride] {
  return reinterpret_cast<float (*)[kMergePartStride]>(smem + (size_t)WARPS * 8 * (kAccStride + 2) * sizeof(float));
}

// B operand of the logits: q[head g][channels], bf16 as stored, for the 8 blocks of 16 channels.
// P: launch parameters with the fields of the attention kernels (q, k, v and their strides, group, ks ...).  FROM_L2: the
// loads bypass L1 (a kernel that has not waited for its predecessor yet).
template <bool KSPLIT, bool FROM_L2 = false, typename P>
__device__ __forceinline__ void attn_load_query(uint32_t (&qb)[8][2], const P& p, const SelUnit& su, int lane) {
  const int g = lane >> 2, t = lane & 3, h = su.h;
  const uint16_t* qh = p.q + (su.q0 + (g < p.group ? g : 0)) * FASA_HEAD_DIM;
  // position c of an assembled key row holds channel ndchan[c] (c < nd) or chan[c - nd]
  auto q_at = [&](int c) -> uint32_t {
    const int ch = c < p.ks.nd ? p.ks.ndchan[h * p.ks.nd + c] : p.ks.chan[h * p.ks.chunks * 8 + c - p.ks.nd];
    return qh[ch];
  };
#pragma unroll
  for (int kb = 0; kb < 8; ++kb) {
    uint32_t w0, w1;
    if constexpr (KSPLIT) {
      w0 = q_at(kb * 16 + 2 * t) | (q_at(kb * 16 + 2 * t + 1) << 16);
      w1 = q_at(kb * 16 + 2 * t + 8) | (q_at(kb * 16 + 2 * t + 9) << 16);
    } else {
      const uint32_t* qw = reinterpret_cast<const uint32_t*>(qh + kb * 16 + 2 * t);
      w0 = FROM_L2 ? __ldcg(qw) : qw[0];
      w1 = FROM_L2 ? __ldcg(qw + 4) : qw[4];
    }
    qb[kb][0] = g < p.group ? w0 : 0u;
    qb[kb][1] = g < p.group ? w1 : 0u;
  }
}

// Attention of the unit's query heads over rows [r0, r1): a warp takes 16 rows at a time.  SPARSE: row r is token
// s_idx[r - r0] (shared memory; on pages that token's row of the pool), else token r.  bc: the sequence whose cache is read.  part(head) receives the
// block's partial result (m, l, acc[128]); the threads must be synchronised before another reads it.  smem: at least
// MmaSmem<WARPS, TERMS>; it must not be in use by anything else when the first warp arrives.  HOSTMEM: K and V rows are
// copied through L1 (caches in page-locked host memory).  KSPLIT: Algorithm 2's Combine, see fasa_attn.cu.
template <int WARPS, bool SPARSE, bool PAGED, bool HOSTMEM, bool KSPLIT, int TERMS, typename P, typename Part>
__device__ __forceinline__ void attn_rows(const P& p, const SelUnit& su, int bc, const uint32_t (&qb)[8][2], int r0, int r1,
                                          const int32_t* s_idx, unsigned char* smem, Part part) {
  static_assert(sizeof(MmaSmem<WARPS, TERMS>) >= mma_combine_bytes<WARPS>(), "combine area");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3, h = su.h;
  MmaSmem<WARPS, TERMS>& sm = *reinterpret_cast<MmaSmem<WARPS, TERMS>*>(smem);
  float acc[8][4];                                  // out^T: [16-channel block][frag], heads 2t, 2t+1
#pragma unroll
  for (int cb = 0; cb < 8; ++cb) acc[cb][0] = acc[cb][1] = acc[cb][2] = acc[cb][3] = 0.f;
  float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f};

  // Staging of a tile's 16 K rows (or V rows): lane l copies chunk (l % 16) of rows 2j + l / 16.
  // The K and the V buffer of a warp are two pipeline stages: the next tile's K rows are
  // requested as soon as this tile's logits are done (they travel during the output
  // product), its V rows as soon as the output product is done (they travel during the next
  // logits), so memory stays busy while the warp computes.  One cp.async group per buffer
  // fill, an empty group when there is no next tile, so "all but the newest group" always
  // names the buffer that is needed next.
  const uint16_t* kunit = PAGED ? p.k : p.k + bc * p.ksb + h * p.ksh;
  const uint16_t* vunit = PAGED ? p.v : p.v + bc * p.vsb + h * p.vsh;
  auto stage = [&](uint16_t (*dst)[kRowPad], const uint16_t* unit, int64_t sb, int64_t sh, int64_t st, int base) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int row = 2 * j + (lane >> 4);
      const int r = min(base + row, r1 - 1);        // rows past the end repeat the last one (masked below)
      const int tok = SPARSE ? s_idx[r - r0] : r;
      const int c8 = (lane & 15) * 8;
      // (contiguous caches keep the plain address arithmetic: the page map costs registers)
      if constexpr (PAGED && SPARSE)
        cp_async16(&dst[row][c8], unit + (tok >> p.pm.shift) * sb + h * sh + (tok & ((1 << p.pm.shift) - 1)) * st + c8);
      else if constexpr (PAGED) cp_async16(&dst[row][c8], unit + cache_row(p.pm, bc, h, tok, sb, sh, st, p.status) + c8);
      else if constexpr (HOSTMEM) cp_async16_ca(&dst[row][c8], unit + (int64_t)tok * st + c8);
      else cp_async16(&dst[row][c8], unit + (int64_t)tok * st + c8);
    }
  };
  // Combine: the 16 key rows of a tile from their two homes
  const ProxyGeom ks_pg = proxy_geom(KSPLIT ? p.ks.chunks : 1);
  const unsigned char* ks_proxy = KSPLIT ? p.ks.proxy + (int64_t)su.kv * ((p.max_len + 15) >> 4) * ks_pg.tile_bytes : nullptr;
  const uint16_t* res_rows = KSPLIT && p.ks.res.tags ? p.ks.res.rows + (int64_t)su.kv * p.ks.res.slots * 2 * FASA_HEAD_DIM : nullptr;
  auto stage_split_k = [&](uint16_t (*dst)[kRowPad], int base) {
    const int nd_chunks = p.ks.nd >> 3, words = 4 * p.ks.chunks;
    for (int c = lane; c < 16 * nd_chunks; c += 32) {                 // the part that crosses the link
      const int row = c / nd_chunks, ch = c % nd_chunks;
      const int tok = s_idx[min(base + row, r1 - 1) - r0];
      if (tok >= 0) cp_async16_ca(&dst[row][ch * 8], kunit + (int64_t)tok * p.kst + ch * 8);
    }
    for (int c = lane; c < 16 * words; c += 32) {                     // the dominant pairs, from the proxy
      const int row = c / words, w = c % words;
      const int tok = s_idx[min(base + row, r1 - 1) - r0];
      if (tok >= 0) cp_async4(&dst[row][p.ks.nd + 2 * w], ks_proxy + proxy_word_offset(ks_pg, tok, w));
    }
    if (res_rows != nullptr) {                                        // resident rows: whole assembled key rows
      for (int c = lane; c < 16 * 16; c += 32) {
        const int row = c >> 4, ch = c & 15;
        const int tok = s_idx[min(base + row, r1 - 1) - r0];
        if (tok < 0) cp_async16(&dst[row][ch * 8], res_rows + (int64_t)(-1 - tok) * 2 * FASA_HEAD_DIM + ch * 8);
      }
    }
  };
  // value rows of a tile with a split key cache: from the host, or from the resident rows
  auto stage_split_v = [&](uint16_t (*dst)[kRowPad], int base) {
    for (int c = lane; c < 16 * 16; c += 32) {
      const int row = c >> 4, ch = c & 15;
      const int tok = s_idx[min(base + row, r1 - 1) - r0];
      if (tok >= 0) cp_async16_ca(&dst[row][ch * 8], vunit + (int64_t)tok * p.vst + ch * 8);
      else cp_async16(&dst[row][ch * 8], res_rows + (int64_t)(-1 - tok) * 2 * FASA_HEAD_DIM + FASA_HEAD_DIM + ch * 8);
    }
  };
  auto stage_v = [&](int base) {
    if constexpr (KSPLIT) stage_split_v(sm.v[warp], base);
    else stage(sm.v[warp], vunit, p.vsb, p.vsh, p.vst, base);
  };
  auto stage_k = [&](int base) {
    if constexpr (KSPLIT) stage_split_k(sm.k[warp], base);
    else stage(sm.k[warp], kunit, p.ksb, p.ksh, p.kst, base);
  };
  constexpr int kTileStep = WARPS * 16;
  if (r0 + warp * 16 < r1) stage_k(r0 + warp * 16);
  cp_async_commit();
  if (r0 + warp * 16 < r1) stage_v(r0 + warp * 16);
  cp_async_commit();

  for (int base = r0 + warp * 16; base < r1; base += kTileStep) {   // uniform over the warp
    const bool more = base + kTileStep < r1;
    cp_async_wait<1>();                             // this tile's K rows have landed
    __syncwarp();

    // ---- logits: D[16 rows x 8 heads] ---------------------------------------------------------
    float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int kb = 0; kb < 8; ++kb) {
      uint32_t a[4];
      // matrices: (rows 0-7, ch 0-7), (rows 8-15, ch 0-7), (rows 0-7, ch 8-15), (rows 8-15, ch 8-15)
      ldmatrix_x4(a, &sm.k[warp][(lane & 7) + 8 * ((lane >> 3) & 1)][kb * 16 + 8 * (lane >> 4)]);
      mma16816(c, a, qb[kb][0], qb[kb][1]);
    }
    // thread: c0, c1 = row g, heads 2t, 2t+1; c2, c3 = row g + 8
    const bool ok_lo = base + g < r1, ok_hi = base + g + 8 < r1;
    float lg[4];
    lg[0] = ok_lo ? c[0] * p.scale_log2 : -INFINITY;
    lg[1] = ok_lo ? c[1] * p.scale_log2 : -INFINITY;
    lg[2] = ok_hi ? c[2] * p.scale_log2 : -INFINITY;
    lg[3] = ok_hi ? c[3] * p.scale_log2 : -INFINITY;
    float alpha[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float bm = fmaxf(lg[e], lg[2 + e]);
      bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 4));
      bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 8));
      bm = fmaxf(bm, __shfl_xor_sync(0xffffffffu, bm, 16));
      const float m_new = fmaxf(m_run[e], bm);
      const float m_safe = m_new == -INFINITY ? 0.f : m_new;
      alpha[e] = exp2f(m_run[e] - m_safe);
      lg[e] = exp2f(lg[e] - m_safe);
      lg[2 + e] = exp2f(lg[2 + e] - m_safe);
      l_run[e] = l_run[e] * alpha[e] + lg[e] + lg[2 + e];   // this thread's rows; the g lanes are added at the end
      m_run[e] = m_new;
    }
    // P^T[head][row] as bf16 terms
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int head = 2 * t + (e & 1), row = g + 8 * (e >> 1);
      float rest = lg[e];
#pragma unroll
      for (int i = 0; i < TERMS; ++i) {
        const uint32_t term = f32_to_bf16_bits(rest);
        sm.p[i][warp][head][row] = (uint16_t)term;
        rest -= __uint_as_float(term << 16);
      }
    }
    __syncwarp();                                   // P is visible; every lane is done with the K buffer
    if (more) stage_k(base + kTileStep);
    cp_async_commit();
    cp_async_wait<1>();                             // this tile's V rows have landed
    __syncwarp();
    // B operand of the output product: B[k = row][n = head g]: rows 2t, 2t+1 and 2t+8, 2t+9
    uint32_t pt[TERMS][2];
#pragma unroll
    for (int i = 0; i < TERMS; ++i) {
      pt[i][0] = *reinterpret_cast<const uint32_t*>(&sm.p[i][warp][g][2 * t]);
      pt[i][1] = *reinterpret_cast<const uint32_t*>(&sm.p[i][warp][g][2 * t + 8]);
    }

    // ---- output: out^T[16 ch x 8 heads] += V^T[16 ch x 16 rows] . P^T[16 rows x 8 heads] ------
#pragma unroll
    for (int cb = 0; cb < 8; ++cb) {
      acc[cb][0] *= alpha[0]; acc[cb][1] *= alpha[1]; acc[cb][2] *= alpha[0]; acc[cb][3] *= alpha[1];
      uint32_t a[4];
      // source blocks (token rows x channels), transposed on load:
      // (rows 0-7, ch 0-7), (rows 0-7, ch 8-15), (rows 8-15, ch 0-7), (rows 8-15, ch 8-15)
      ldmatrix_x4_trans(a, &sm.v[warp][(lane & 7) + 8 * (lane >> 4)][cb * 16 + 8 * ((lane >> 3) & 1)]);
#pragma unroll
      for (int i = 0; i < TERMS; ++i) mma16816(acc[cb], a, pt[i][0], pt[i][1]);
    }
    __syncwarp();                                   // every lane is done with the V buffer
    if (more) stage_v(base + kTileStep);
    cp_async_commit();
  }
  cp_async_wait<0>();

  // ---- this warp's (m, l, acc) per head; the g lanes add their sums -------------------------------
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    l_run[e] += __shfl_xor_sync(0xffffffffu, l_run[e], 4);
    l_run[e] += __shfl_xor_sync(0xffffffffu, l_run[e], 8);
    l_run[e] += __shfl_xor_sync(0xffffffffu, l_run[e], 16);
  }
  __syncthreads();                                  // staging memory becomes the combine area
  const int n_warps = min(WARPS, max(1, (r1 - r0 + 15) >> 4));         // warps that had rows
  float* s_acc = reinterpret_cast<float*>(smem);
  float* s_ml = s_acc + WARPS * 8 * kAccStride;
  if (warp < n_warps && 2 * t < p.group) {          // (an odd group's last column is written and not read)
    float* dst = s_acc + (warp * 8 + 2 * t) * kAccStride + g;
#pragma unroll
    for (int cb = 0; cb < 8; ++cb) {
      dst[cb * 16] = acc[cb][0];
      dst[kAccStride + cb * 16] = acc[cb][1];
      dst[cb * 16 + 8] = acc[cb][2];
      dst[kAccStride + cb * 16 + 8] = acc[cb][3];
    }
    if (g == 0) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        s_ml[(warp * 8 + 2 * t + e) * 2 + 0] = m_run[e];
        s_ml[(warp * 8 + 2 * t + e) * 2 + 1] = l_run[e];
      }
    }
  }
  __syncthreads();
  for (int o = threadIdx.x; o < p.group * FASA_HEAD_DIM; o += WARPS * 32) {
    const int gl = o / FASA_HEAD_DIM, cch = o % FASA_HEAD_DIM;
    float mx = -INFINITY;
#pragma unroll 4
    for (int w = 0; w < n_warps; ++w) mx = fmaxf(mx, s_ml[(w * 8 + gl) * 2]);
    float a = 0.f, l = 0.f;
#pragma unroll 4
    for (int w = 0; w < n_warps; ++w) {
      const float2 ml = *reinterpret_cast<const float2*>(&s_ml[(w * 8 + gl) * 2]);
      const float wt = ml.x == -INFINITY ? 0.f : exp2f(ml.x - mx);
      a += wt * s_acc[(w * 8 + gl) * kAccStride + cch];
      l += wt * ml.y;
    }
    float* dst = part(gl);
    dst[2 + cch] = a;
    if (cch == 0) {
      dst[0] = mx;
      dst[1] = l;
    }
  }
}

#endif  // __CUDACC__
