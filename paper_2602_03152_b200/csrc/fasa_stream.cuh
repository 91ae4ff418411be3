// The two halves of the two-launch decode step; the first one also scores blocks of queries.
#pragma once

#include <type_traits>

#include "fasa_common.cuh"

// First half: scores [batch][n_sets][max_len] (and group maxima, gs > 0) of every cached token; k_new != null: the appended
// token first.  q_len > 0: of a block of queries, [batch][q_len][n_sets][max_len].  Index sets of one head or of as many as a
// block takes.
struct fasa_stream_args {
  const void* q;
  const void* proxy_k;
  const int32_t* seq_lens;
  float* scores;
  fasa_row_maxima maxima;
  int q_len;
  const void* k_new;
  const void* v_new;
  void* k_cache;
  void* v_cache;
};
int32_t fasa_stream_launch(fasa_ctx* ctx, const fasa_stream_args& a, cudaStream_t stream);

// Second half: selection and attention (append: of the grown sequences, whose lengths it stores); n_sel_max beyond
// fasa_select_attend_ok is not taken.
bool fasa_select_attend_ok(const fasa_ctx* ctx, int n_sel_max);
int32_t fasa_select_attend_launch(fasa_ctx* ctx, const void* q, const void* k_cache, const void* v_cache, const float* scores,
                                  const float* gm, int gs, const int32_t* seq_lens, int32_t budget, int32_t n_sel_max,
                                  int32_t* idx, int32_t* n_sel, float* out, float* lse, float* out_mirror, bool append, bool full_p,
                                  cudaStream_t stream);
