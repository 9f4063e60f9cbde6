// C ABI of libq4kv.so: host-side validation, sizing and dispatch.  See include/q4kv.h for
// the contract of every entry point.
#include "q4kv_layout.cuh"

using namespace q4kv;

namespace {

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int check_spec(const q4kv_spec* s) {
  if (!s) return Q4KV_EINVAL;
  if (s->n_layers <= 0 || s->n_q_heads <= 0 || s->n_kv_heads <= 0 || s->d_qk <= 0 || s->d_v <= 0) return Q4KV_EINVAL;
  if (s->group != 64 || s->block_tokens != 256 || (s->sb_dtype != 0 && s->sb_dtype != 1)) return Q4KV_EUNSUPPORTED;
  if (s->exact_products != 0 && s->exact_products != 1) return Q4KV_EINVAL;
  if (s->d_qk % 64 || s->d_v % 64 || s->n_q_heads % s->n_kv_heads) return Q4KV_EUNSUPPORTED;
  if (s->d_qk > 1024 || s->d_v > 512) return Q4KV_EUNSUPPORTED;
  if (s->v_aliases_k && s->d_v > s->d_qk) return Q4KV_EUNSUPPORTED;
  return Q4KV_OK;
}

int check_batch(const q4kv_batch* b) {
  if (!b || b->n_agents < 0 || b->max_blocks <= 0) return Q4KV_EINVAL;
  if (b->n_agents > 0 && !b->block_tables) return Q4KV_EINVAL;
  return Q4KV_OK;
}

// Every decode kernel keeps its partial records behind a header of fixed size (the arrival counters
// of the kernels that merge in the same launch), so that one workspace serves any sequence of calls.
size_t workspace_need(const Layout& y, int n_agents, int max_kv_len, int total_q) {
  if (total_q > 0) return 16;   // the prefill kernels need none; what they make use of is prefill_workspace
  const DecodePlan p = plan_decode(y, n_agents, max_kv_len, 0);
  size_t need = (size_t)n_agents * y.Hq * p.n_splits * (y.Dv + 2) * sizeof(float) + 16;
  if (decode_mla_supported(y)) {
    const size_t mla = decode_mla_workspace_bytes(y, n_agents, max_kv_len);
    if (mla > need) need = mla;
  }
  if (decode_mma_supported(y)) {
    const size_t mma = decode_mma_workspace_bytes(y, n_agents);
    if (mma > need) need = mma;
  }
  return kWorkspaceHeaderBytes + need;
}

// The tcgen05 prefill kernels: the query rows of a CTA and the CTAs that share them (0: no such kernel for the shape).
int prefill_rows(const Layout& y) { return prefill_umma_supported(y) ? 256 : prefill_umma_1tile_supported(y) || prefill_mla_supported(y) ? 128 : 0; }
int prefill_tile_q(const Layout& y) { return prefill_rows(y) == 256 ? 2 * (128 / y.n_rep) : 128 / y.n_rep; }
size_t align256(size_t n) { return (n + 255) & ~(size_t)255; }

// Agents that bring one query while others bring more go to the decode kernel.  The counts are on the device; what the host
// sees is that one such agent leaves the batch max_q_len - 1 rows short of n_agents * max_q_len.  A launch that finds none
// costs 2 us, so it is made only where an average agent brings at most a third of the longest: chunks of one schedule lie
// closer together, decoding agents pull the average down.
bool may_decode_singles(const Layout& y, int n_agents, int max_blocks, int total_q, int max_q_len) {
  const long long all = (long long)n_agents * max_q_len;
  return max_q_len > 1 && all - total_q >= max_q_len - 1 && 3ll * total_q <= all && decode_mma_supported(y) &&
         decode_mma_fits(y, n_agents, max_blocks);
}
size_t singles_bytes(const Layout& y, int n_agents) {
  return align256(sizeof(int32_t) * decode_mma_tickets(y, n_agents)) + decode_mma_workspace_bytes(y, n_agents);
}

// What a prefill call can make use of: the records of the query tiles whose keys it cuts into parts, and the workspace of
// the decode launch for agents with one query.  The call makes do with less, so this size is not a condition.
size_t prefill_workspace(const Layout& y, int n_agents, int max_kv_len, int total_q) {
  if (!prefill_rows(y)) return 16;
  const int splits = plan_prefill_splits(y, prefill_tile_q(y), prefill_mla_supported(y) ? 2 : 1, n_agents, total_q, total_q, max_kv_len, 0, (size_t)-1);
  size_t need = splits > 1 ? align256(prefill_record_bytes(y, total_q, splits)) : 0;
  if (n_agents > 1 && total_q > n_agents && decode_mma_supported(y)) need += align256(singles_bytes(y, n_agents));
  return need > 0 ? kWorkspaceHeaderBytes + need : 16;
}

// The part of a workspace that a prefill call may write: what lies behind the arrival counters, which every decode call on
// the same workspace expects to find at zero.
struct Scratch { uint8_t* at; size_t bytes; };
Scratch prefill_scratch(void* workspace, size_t bytes) {
  if (bytes <= kWorkspaceHeaderBytes) return {nullptr, 0};
  return {(uint8_t*)workspace + kWorkspaceHeaderBytes, bytes - kWorkspaceHeaderBytes};
}

// The kernels that expand the cache into binary16 tiles round each dequantized element once; they are taken only when
// the spec allows it and the softmax scale is at most 2 / sqrt(d_qk) (the error a rounded key leaves in a score grows
// with the scale).  Everything else multiplies the codes exactly.  Bfloat16 scales and biases are converted to binary16
// once per key block by those kernels (exact for every magnitude a cache written by this library can hold; a magnitude
// beyond binary16's largest number, which only a foreign cache can hold, raises Q4KV_FLAG_SB_RANGE).
bool tiles_allowed(const q4kv_spec* s, float softmax_scale) {
  return s->exact_products == 0 && softmax_scale > 0.f && softmax_scale * softmax_scale * (float)s->d_qk <= 4.f;
}

}  // namespace

extern "C" {

const char* q4kv_status_string(int code) {
  switch (code) {
    case Q4KV_OK: return "ok";
    case Q4KV_EINVAL: return "invalid argument (null, negative or misaligned)";
    case Q4KV_EUNSUPPORTED: return "spec not supported by this library";
    case Q4KV_EWORKSPACE: return "workspace or destination buffer too small";
    case Q4KV_ECUDA: return "CUDA launch or runtime error";
    default: return "unknown status";
  }
}

size_t q4kv_pool_bytes(const q4kv_spec* spec, int32_t n_blocks) {
  if (check_spec(spec) != Q4KV_OK || n_blocks <= 0) return 0;
  const Layout y = make_layout(*spec, n_blocks);
  return (size_t)y.L * y.layer_bytes;
}

size_t q4kv_packed_bytes(const q4kv_spec* spec, int32_t n_tokens) {
  if (check_spec(spec) != Q4KV_OK || n_tokens < 0) return 0;
  const Layout y = make_layout(*spec, 1);
  const uint64_t nblk = ((uint64_t)n_tokens + kBlockTokens - 1) / kBlockTokens;
  return (size_t)(y.L * nblk * persisted_block_bytes(y));
}

size_t q4kv_workspace_bytes(const q4kv_spec* spec, int32_t n_agents, int32_t max_kv_len, int32_t total_q) {
  if (check_spec(spec) != Q4KV_OK || n_agents < 0 || max_kv_len < 0 || total_q < 0) return 0;
  const Layout y = make_layout(*spec, 1);
  if (n_agents == 0) n_agents = 1;
  if (max_kv_len == 0) max_kv_len = 1;
  return total_q > 0 ? prefill_workspace(y, n_agents, max_kv_len, total_q) : workspace_need(y, n_agents, max_kv_len, 0);
}

int q4kv_quantize_append(const q4kv_spec* spec, void* pool, int32_t n_blocks, int32_t layer,
                         const q4kv_batch* batch, const int32_t* pos, const int32_t* new_offs,
                         int32_t total_new, const void* k_new, const void* v_new,
                         int32_t* status_flags, void* stream) {
  int rc = check_spec(spec);
  if (rc) return rc;
  if ((rc = check_batch(batch))) return rc;
  if (!pool || n_blocks <= 0 || layer < 0 || layer >= spec->n_layers || total_new < 0) return Q4KV_EINVAL;
  if (total_new == 0 || batch->n_agents == 0) return Q4KV_OK;
  if (!pos || !new_offs || !k_new) return Q4KV_EINVAL;
  if ((spec->v_aliases_k != 0) != (v_new == nullptr)) return Q4KV_EINVAL;
  if (!aligned16(pool) || !aligned16(k_new) || !aligned16(v_new)) return Q4KV_EINVAL;
  const Layout y = make_layout(*spec, n_blocks);
  const cudaError_t e = launch_quantize_append(y, pool, n_blocks, layer, *batch, pos, new_offs, total_new, k_new,
                                               v_new, status_flags, (cudaStream_t)stream);
  return e == cudaSuccess ? Q4KV_OK : Q4KV_ECUDA;
}

int q4kv_decode_attention(const q4kv_spec* spec, const void* pool, int32_t n_blocks, int32_t layer,
                          const q4kv_batch* batch, const int32_t* kv_lens, int32_t max_kv_len,
                          int32_t window, const void* q, float softmax_scale,
                          void* out, int32_t out_dtype, float* lse,
                          void* workspace, size_t workspace_bytes,
                          int32_t* status_flags, void* stream) {
  int rc = check_spec(spec);
  if (rc) return rc;
  if ((rc = check_batch(batch))) return rc;
  if (!pool || n_blocks <= 0 || layer < 0 || layer >= spec->n_layers || window < 0 || max_kv_len < 0) return Q4KV_EINVAL;
  if (out_dtype != Q4KV_OUT_F32 && out_dtype != Q4KV_OUT_BF16) return Q4KV_EINVAL;
  if (batch->n_agents == 0) return Q4KV_OK;
  if (!kv_lens || !q || !out || !workspace) return Q4KV_EINVAL;
  if (!aligned16(pool) || !aligned16(q) || !aligned16(out) || !aligned16(workspace)) return Q4KV_EINVAL;
  const int cap = batch->max_blocks * kBlockTokens;
  if (max_kv_len == 0 || max_kv_len > cap) max_kv_len = cap;
  const Layout y = make_layout(*spec, n_blocks);
  if (workspace_bytes < workspace_need(y, batch->n_agents, max_kv_len, 0)) return Q4KV_EWORKSPACE;
  void* records = (uint8_t*)workspace + kWorkspaceHeaderBytes;
  cudaError_t e;
  if (decode_mla_supported(y))
    e = launch_decode_mla(y, pool, n_blocks, layer, *batch, kv_lens, max_kv_len, window, q, softmax_scale, out, out_dtype,
                          lse, records, status_flags, (cudaStream_t)stream, nullptr, !tiles_allowed(spec, softmax_scale));
  else if (decode_mma_supported(y) && decode_mma_fits(y, batch->n_agents, batch->max_blocks))
    e = launch_decode_mma(y, pool, n_blocks, layer, *batch, kv_lens, max_kv_len, &window, 1, q, softmax_scale, out,
                          out_dtype, lse, workspace, status_flags, (cudaStream_t)stream);
  else
    e = launch_attention_generic(y, pool, n_blocks, layer, *batch, kv_lens, nullptr, 0, 1, max_kv_len, window, q,
                                 softmax_scale, out, out_dtype, lse, records, status_flags, (cudaStream_t)stream);
  return e == cudaSuccess ? Q4KV_OK : Q4KV_ECUDA;
}

int q4kv_append_decode_attention(const q4kv_spec* spec, void* pool, int32_t n_blocks, int32_t layer,
                                 const q4kv_batch* batch, const int32_t* kv_lens, int32_t max_kv_len,
                                 int32_t window, const void* k_new, const void* v_new,
                                 const void* q, float softmax_scale,
                                 void* out, int32_t out_dtype, float* lse,
                                 void* workspace, size_t workspace_bytes,
                                 int32_t* status_flags, void* stream) {
  int rc = check_spec(spec);
  if (rc) return rc;
  if ((rc = check_batch(batch))) return rc;
  if (!pool || n_blocks <= 0 || layer < 0 || layer >= spec->n_layers || window < 0 || max_kv_len < 0) return Q4KV_EINVAL;
  if (out_dtype != Q4KV_OUT_F32 && out_dtype != Q4KV_OUT_BF16) return Q4KV_EINVAL;
  if (batch->n_agents == 0) return Q4KV_OK;
  const bool need_v = !spec->v_aliases_k;                  // an aliased cache stores no V rows
  if (!kv_lens || !q || !out || !workspace || !k_new || (need_v && !v_new)) return Q4KV_EINVAL;
  if (!aligned16(pool) || !aligned16(q) || !aligned16(out) || !aligned16(workspace) || !aligned16(k_new) ||
      (need_v && !aligned16(v_new)))
    return Q4KV_EINVAL;
  const int cap = batch->max_blocks * kBlockTokens;
  if (max_kv_len == 0 || max_kv_len > cap) max_kv_len = cap;
  const Layout y = make_layout(*spec, n_blocks);
  if (decode_mla_supported(y)) {
    if (workspace_bytes < workspace_need(y, batch->n_agents, max_kv_len, 0)) return Q4KV_EWORKSPACE;
    const cudaError_t e = launch_decode_mla(y, pool, n_blocks, layer, *batch, kv_lens, max_kv_len, window, q, softmax_scale,
                                            out, out_dtype, lse, (uint8_t*)workspace + kWorkspaceHeaderBytes, status_flags,
                                            (cudaStream_t)stream, k_new, !tiles_allowed(spec, softmax_scale));
    return e == cudaSuccess ? Q4KV_OK : Q4KV_ECUDA;
  }
  if (!decode_mma_supported(y) || y.n_rep > 4 || !decode_mma_fits(y, batch->n_agents, batch->max_blocks))
    return Q4KV_EUNSUPPORTED;
  if (workspace_bytes < workspace_need(y, batch->n_agents, max_kv_len, 0)) return Q4KV_EWORKSPACE;
  const cudaError_t e = launch_decode_mma(y, pool, n_blocks, layer, *batch, kv_lens, max_kv_len, &window, 1, q, softmax_scale,
                                          out, out_dtype, lse, workspace, status_flags, (cudaStream_t)stream, k_new, v_new);
  return e == cudaSuccess ? Q4KV_OK : Q4KV_ECUDA;
}

size_t q4kv_workspace_bytes_layers(const q4kv_spec* spec, int32_t n_agents, int32_t max_kv_len, int32_t layer_count) {
  if (check_spec(spec) != Q4KV_OK || n_agents < 0 || max_kv_len < 0 || layer_count < 1) return 0;
  const Layout y = make_layout(*spec, 1);
  if (!decode_mma_supported(y) || y.n_rep > 4) return 0;
  const size_t one = workspace_need(y, n_agents > 0 ? n_agents : 1, max_kv_len > 0 ? max_kv_len : 1, 0);
  const size_t all = kWorkspaceHeaderBytes + decode_mma_workspace_bytes(y, n_agents > 0 ? n_agents : 1, layer_count);
  return all > one ? all : one;
}

int q4kv_decode_attention_layers(const q4kv_spec* spec, void* pool, int32_t n_blocks, int32_t layer_begin,
                                 int32_t layer_count, const q4kv_batch* batch, const int32_t* kv_lens, int32_t max_kv_len,
                                 const int32_t* windows, const void* k_new, const void* v_new, const void* q,
                                 float softmax_scale, void* out, int32_t out_dtype, float* lse,
                                 void* workspace, size_t workspace_bytes, int32_t* status_flags, void* stream) {
  int rc = check_spec(spec);
  if (rc) return rc;
  if ((rc = check_batch(batch))) return rc;
  if (!pool || n_blocks <= 0 || layer_begin < 0 || layer_count < 1 || layer_begin + layer_count > spec->n_layers ||
      max_kv_len < 0 || !windows)
    return Q4KV_EINVAL;
  for (int i = 0; i < layer_count; ++i)
    if (windows[i] < 0) return Q4KV_EINVAL;
  if (out_dtype != Q4KV_OUT_F32 && out_dtype != Q4KV_OUT_BF16) return Q4KV_EINVAL;
  if (batch->n_agents == 0) return Q4KV_OK;
  if (!kv_lens || !q || !out || !workspace || ((k_new == nullptr) != (v_new == nullptr))) return Q4KV_EINVAL;
  if (!aligned16(pool) || !aligned16(q) || !aligned16(out) || !aligned16(workspace) || !aligned16(k_new) || !aligned16(v_new))
    return Q4KV_EINVAL;
  const int cap = batch->max_blocks * kBlockTokens;
  if (max_kv_len == 0 || max_kv_len > cap) max_kv_len = cap;
  const Layout y = make_layout(*spec, n_blocks);
  if (!decode_mma_supported(y) || y.n_rep > 4 || !decode_mma_fits(y, batch->n_agents, batch->max_blocks, layer_count))
    return Q4KV_EUNSUPPORTED;
  if (workspace_bytes < kWorkspaceHeaderBytes + decode_mma_workspace_bytes(y, batch->n_agents, layer_count)) return Q4KV_EWORKSPACE;
  const cudaError_t e = launch_decode_mma(y, pool, n_blocks, layer_begin, *batch, kv_lens, max_kv_len, windows, layer_count, q,
                                          softmax_scale, out, out_dtype, lse, workspace, status_flags, (cudaStream_t)stream,
                                          k_new, v_new);
  return e == cudaSuccess ? Q4KV_OK : Q4KV_ECUDA;
}

int q4kv_prefill_attention(const q4kv_spec* spec, const void* pool, int32_t n_blocks, int32_t layer,
                           const q4kv_batch* batch, const int32_t* kv_lens, const int32_t* q_offs,
                           int32_t total_q, int32_t max_q_len, int32_t max_kv_len,
                           int32_t window, const void* q, float softmax_scale,
                           void* out, int32_t out_dtype, float* lse,
                           void* workspace, size_t workspace_bytes,
                           int32_t* status_flags, void* stream) {
  int rc = check_spec(spec);
  if (rc) return rc;
  if ((rc = check_batch(batch))) return rc;
  if (!pool || n_blocks <= 0 || layer < 0 || layer >= spec->n_layers || window < 0 || max_kv_len < 0 ||
      total_q < 0 || max_q_len < 0)
    return Q4KV_EINVAL;
  if (out_dtype != Q4KV_OUT_F32 && out_dtype != Q4KV_OUT_BF16) return Q4KV_EINVAL;
  if (batch->n_agents == 0 || total_q == 0) return Q4KV_OK;
  if (!kv_lens || !q_offs || !q || !out || !workspace) return Q4KV_EINVAL;
  if (!aligned16(pool) || !aligned16(q) || !aligned16(out) || !aligned16(workspace)) return Q4KV_EINVAL;
  const int cap = batch->max_blocks * kBlockTokens;
  if (max_kv_len == 0 || max_kv_len > cap) max_kv_len = cap;
  if (max_q_len == 0 || max_q_len > total_q) max_q_len = total_q;
  const Layout y = make_layout(*spec, n_blocks);
  if (workspace_bytes < workspace_need(y, batch->n_agents, max_kv_len, total_q)) return Q4KV_EWORKSPACE;
  const Scratch scratch = prefill_scratch(workspace, workspace_bytes);
  cudaError_t e;
  if ((prefill_umma_supported(y) || prefill_umma_1tile_supported(y)) && tiles_allowed(spec, softmax_scale)) {
    PrefillExtra x = {};
    uint8_t* at = scratch.at;
    size_t left = scratch.bytes;
    if (may_decode_singles(y, batch->n_agents, batch->max_blocks, total_q, max_q_len) && left >= singles_bytes(y, batch->n_agents)) {
      x.tickets = (int32_t*)at;
      x.n_tickets = decode_mma_tickets(y, batch->n_agents);
      at += align256(singles_bytes(y, batch->n_agents));
      left -= left < align256(singles_bytes(y, batch->n_agents)) ? left : align256(singles_bytes(y, batch->n_agents));
    }
    x.n_splits = plan_prefill_splits(y, prefill_tile_q(y), 1, batch->n_agents, total_q, max_q_len, max_kv_len, window, left,
                                     x.tickets != nullptr);
    x.records = (float*)at;
    const auto launch = prefill_umma_supported(y) ? launch_prefill_umma : launch_prefill_umma_1tile;
    e = launch(y, pool, n_blocks, layer, *batch, kv_lens, q_offs, max_q_len, window, q, softmax_scale, out, out_dtype, lse,
               status_flags, (cudaStream_t)stream, x);
    if (e == cudaSuccess && x.n_splits > 1)
      e = launch_merge_prefill(y, total_q, x.n_splits, x.records, out, out_dtype, lse, (cudaStream_t)stream,
                               x.tickets ? q_offs : nullptr, batch->n_agents);
    if (e == cudaSuccess && x.tickets)
      e = launch_decode_mma(y, pool, n_blocks, layer, *batch, kv_lens, cap, &window, 1, q, softmax_scale, out, out_dtype, lse,
                            (uint8_t*)x.tickets + align256(sizeof(int32_t) * x.n_tickets) - kWorkspaceHeaderBytes, status_flags,
                            (cudaStream_t)stream, nullptr, nullptr, q_offs, x.tickets);
  }
  else if (prefill_mla_supported(y) && tiles_allowed(spec, softmax_scale))
    e = launch_prefill_mla(y, pool, n_blocks, layer, *batch, kv_lens, q_offs, total_q, max_q_len, max_kv_len, window, q,
                           softmax_scale, out, out_dtype, lse, scratch.at, scratch.bytes, status_flags, (cudaStream_t)stream);
  else if (prefill_mma_supported(y))
    e = launch_prefill_mma(y, pool, n_blocks, layer, *batch, kv_lens, q_offs, max_q_len, window, q, softmax_scale, out,
                           out_dtype, lse, status_flags, (cudaStream_t)stream);
  else
    e = launch_attention_generic(y, pool, n_blocks, layer, *batch, kv_lens, q_offs, total_q, max_q_len, max_kv_len,
                                 window, q, softmax_scale, out, out_dtype, lse, workspace, status_flags,
                                 (cudaStream_t)stream);
  return e == cudaSuccess ? Q4KV_OK : Q4KV_ECUDA;
}

int q4kv_pack(const q4kv_spec* spec, const void* pool, int32_t n_blocks,
              const int32_t* block_table_row, int32_t n_tokens,
              void* dst, size_t dst_bytes, int32_t* status_flags, void* stream) {
  int rc = check_spec(spec);
  if (rc) return rc;
  if (!pool || n_blocks <= 0 || n_tokens < 0) return Q4KV_EINVAL;
  if (n_tokens == 0) return Q4KV_OK;
  if (!block_table_row || !dst || !aligned16(pool) || !aligned16(dst)) return Q4KV_EINVAL;
  if (dst_bytes < q4kv_packed_bytes(spec, n_tokens)) return Q4KV_EWORKSPACE;
  const Layout y = make_layout(*spec, n_blocks);
  const cudaError_t e = launch_pack(y, pool, n_blocks, block_table_row, n_tokens, dst, status_flags, (cudaStream_t)stream);
  return e == cudaSuccess ? Q4KV_OK : Q4KV_ECUDA;
}

int q4kv_unpack(const q4kv_spec* spec, const void* src, size_t src_bytes, int32_t n_tokens,
                void* pool, int32_t n_blocks, const int32_t* block_table_row,
                int32_t* status_flags, void* stream) {
  int rc = check_spec(spec);
  if (rc) return rc;
  if (!pool || n_blocks <= 0 || n_tokens < 0) return Q4KV_EINVAL;
  if (n_tokens == 0) return Q4KV_OK;
  if (!block_table_row || !src || !aligned16(pool) || !aligned16(src)) return Q4KV_EINVAL;
  if (src_bytes < q4kv_packed_bytes(spec, n_tokens)) return Q4KV_EWORKSPACE;
  const Layout y = make_layout(*spec, n_blocks);
  const cudaError_t e = launch_unpack(y, src, n_tokens, pool, n_blocks, block_table_row, status_flags, (cudaStream_t)stream);
  return e == cudaSuccess ? Q4KV_OK : Q4KV_ECUDA;
}

}  // extern "C"
