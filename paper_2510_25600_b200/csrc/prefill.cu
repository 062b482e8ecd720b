// purekv_st_sparse_prefill: argument checks and dispatch to the tensor-core or CUDA-core kernel.
#include <algorithm>

#include "prefill.cuh"

using namespace purekv;

// The checks of a call and its launches; `name` is the entry point's.
static purekv_status prefill(const char* name, const void* q, const void* k, const void* v, void* o, float* lse, int64_t q_stride,
                             int64_t kv_stride, int64_t o_stride, int64_t lse_stride, int32_t n_layers, const purekv_batch* batch,
                             void* plan, const purekv_plan_info* info, int32_t n_q_heads, int32_t n_kv_heads, int32_t head_dim,
                             purekv_dtype dtype, float softmax_scale, void* ws, size_t ws_bytes, int32_t* status, void* stream) {
  purekv_status st = check_batch(batch, false);
  if (st != PUREKV_OK) return st;
  if (batch->total_tokens == 0 || batch->n_req == 0) return PUREKV_OK;  // empty batch: nothing to do
  PK_REQUIRE(q && k && v && o && plan && info, PUREKV_ERR_INVALID_ARG, "%s: null pointer", name);
  PK_REQUIRE(n_q_heads >= 1 && n_kv_heads >= 1 && n_q_heads % n_kv_heads == 0 && n_q_heads <= 65535,
             PUREKV_ERR_INVALID_ARG, "n_q_heads %d must be a positive multiple of n_kv_heads %d", n_q_heads,
             n_kv_heads);
  PK_REQUIRE(dtype == PUREKV_BF16 || dtype == PUREKV_FP32, PUREKV_ERR_INVALID_ARG, "unknown dtype");
  PK_REQUIRE(info->dtype == (int32_t)dtype && info->head_dim == head_dim, PUREKV_ERR_INVALID_ARG,
             "plan was built for dtype %d head_dim %d, call has dtype %d head_dim %d", info->dtype, info->head_dim,
             (int)dtype, head_dim);
  PK_REQUIRE(info->n_q_heads == n_q_heads && info->n_kv_heads == n_kv_heads, PUREKV_ERR_INVALID_ARG,
             "plan was built for %d/%d heads, call has %d/%d", info->n_q_heads, info->n_kv_heads, n_q_heads,
             n_kv_heads);
  PK_REQUIRE(info->ws_bytes == 0 || (ws != nullptr && ws_bytes >= (size_t)info->ws_bytes && (uintptr_t)ws % 16 == 0),
             PUREKV_ERR_WORKSPACE, "prefill workspace: need %lld bytes (16-byte aligned), got %zu",
             (long long)info->ws_bytes, ws_bytes);
  PK_REQUIRE(((uintptr_t)q | (uintptr_t)k | (uintptr_t)v | (uintptr_t)o | (uintptr_t)plan) % 16 == 0,
             PUREKV_ERR_INVALID_ARG, "Q/K/V/O/plan must be 16-byte aligned");
  if (info->n_qtiles == 0) return PUREKV_OK;
  PrefillArgs a{q, k, v, o, lse, batch, plan, info, n_q_heads, n_kv_heads, head_dim, dtype,
                softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)head_dim), ws, ws_bytes, status,
                (cudaStream_t)stream, n_layers, q_stride, kv_stride, o_stride, lse_stride};
  const bool tc = dtype == PUREKV_BF16 && head_dim == 128 && info->tile_q == 128;
  // Several layers are one launch of the tensor-core kernel where lists are whole (the chunks of a split list meet in counters
  // and workspace slots that the plan has for one layer at a time).  31 layers of 2432 tokens: 40 us each as launches of their
  // own, a third of it start, merges and the uneven end.
  // Layers that overlap (one Q for all of them, say) are launches of their own too, and so are strides that a tensor map cannot
  // hold.
  const int64_t esz = dtype == PUREKV_BF16 ? 2 : 4, t = batch->total_tokens, o_align = tc ? 32 : 16;
  PK_REQUIRE(n_layers == 1 || (q_stride * esz % 16 == 0 && kv_stride * esz % 16 == 0 && o_stride * esz % o_align == 0),
             PUREKV_ERR_INVALID_ARG, "layer strides must be multiples of 16 bytes, O's of %lld", (long long)o_align);
  const bool apart = q_stride >= t * n_q_heads * head_dim && o_stride >= t * n_q_heads * head_dim &&
                     kv_stride >= t * n_kv_heads * head_dim && (lse == nullptr || lse_stride >= t * n_q_heads) &&
                     std::max({q_stride, kv_stride, o_stride}) < (1ll << 38);
  if (n_layers == 1 || (tc && apart && info->max_chunks == 1 && (int64_t)info->n_units * n_layers <= INT32_MAX / 2))
    return tc ? launch_prefill_tc(a) : launch_prefill_simt(a);
  a.n_layers = 1;
  for (int32_t n = 0; n < n_layers; ++n) {
    a.q = (const char*)q + n * q_stride * esz;
    a.k = (const char*)k + n * kv_stride * esz;
    a.v = (const char*)v + n * kv_stride * esz;
    a.o = (char*)o + n * o_stride * esz;
    a.lse = lse ? lse + n * lse_stride : nullptr;
    const purekv_status one = tc ? launch_prefill_tc(a) : launch_prefill_simt(a);
    if (one != PUREKV_OK) return one;
  }
  return PUREKV_OK;
}

extern "C" purekv_status purekv_st_sparse_prefill(const void* q, const void* k, const void* v, void* o, float* lse,
                                                  const purekv_batch* batch, void* plan,
                                                  const purekv_plan_info* info, int32_t n_q_heads, int32_t n_kv_heads,
                                                  int32_t head_dim, purekv_dtype dtype, float softmax_scale, void* ws,
                                                  size_t ws_bytes, int32_t* status, void* stream) {
  return prefill("purekv_st_sparse_prefill", q, k, v, o, lse, 0, 0, 0, 0, 1, batch, plan, info, n_q_heads, n_kv_heads, head_dim,
                 dtype, softmax_scale, ws, ws_bytes, status, stream);
}

extern "C" purekv_status purekv_st_sparse_prefill_layers(const void* q, const void* k, const void* v, void* o, float* lse,
                                                         int64_t q_layer_stride, int64_t kv_layer_stride, int64_t o_layer_stride,
                                                         int64_t lse_layer_stride, int32_t n_layers, const purekv_batch* batch,
                                                         void* plan, const purekv_plan_info* info, int32_t n_q_heads,
                                                         int32_t n_kv_heads, int32_t head_dim, purekv_dtype dtype,
                                                         float softmax_scale, void* ws, size_t ws_bytes, int32_t* status,
                                                         void* stream) {
  PK_REQUIRE(n_layers >= 0, PUREKV_ERR_INVALID_ARG, "n_layers %d is negative", n_layers);
  if (n_layers == 0) return PUREKV_OK;
  return prefill("purekv_st_sparse_prefill_layers", q, k, v, o, lse, q_layer_stride, kv_layer_stride, o_layer_stride,
                 lse_layer_stride, n_layers, batch, plan, info, n_q_heads, n_kv_heads, head_dim, dtype, softmax_scale, ws, ws_bytes,
                 status, stream);
}
