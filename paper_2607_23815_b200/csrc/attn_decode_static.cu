// attn_decode_static: decode attention for callers that are not allowed to allocate device memory.
//
// attn_decode takes a workspace of attn_workspace_bytes(); code that runs where cudaMalloc is off limits (inside a
// framework's captured or memory-planned region, in a plugin that was handed fixed buffers, in a process whose allocator
// is frozen after start-up) cannot produce one.  The decode kernel keeps its partial results on chip, so this entry
// point is the same launch; the limit on the batch (what 8 MiB of partials would hold) is part of its contract.
#include "common.cuh"

namespace kvattn {
size_t decode_workspace_bytes(int n_q_heads, int head_dim, int batch, int max_ctx_len);
kv_status_t launch_decode(kv_pool_t* p, const void* q, int n_q_heads, const int* block_tables, int max_pages,
                          const int* ctx_lens, int batch, int max_ctx_len, float scale, void* out, float* lse,
                          cudaStream_t st, bool beside = false);

constexpr size_t kStaticScratchBytes = size_t(8) << 20;
}  // namespace kvattn

using namespace kvattn;

extern "C" kv_status_t attn_decode_static(kv_pool_t* p, const void* q, int n_q_heads, const int* block_tables,
                                          int max_pages, const int* ctx_lens, int batch, int max_ctx_len,
                                          float scale, void* out, float* lse, void* stream) {
  if (p == nullptr || batch < 0 || max_pages < 0 || max_ctx_len < 0) return KV_ERR_INVALID;
  if (n_q_heads <= 0 || n_q_heads % p->n_kv_heads != 0) return KV_ERR_UNSUPPORTED;
  const int g = n_q_heads / p->n_kv_heads;
  if (!(g == 1 || g == 2 || g == 4 || g == 8)) return KV_ERR_UNSUPPORTED;
  if (batch == 0) return KV_OK;
  if (q == nullptr || block_tables == nullptr || ctx_lens == nullptr || out == nullptr || lse == nullptr)
    return KV_ERR_INVALID;
  if ((((uintptr_t)q) | ((uintptr_t)out)) & 15) return KV_ERR_INVALID;
  if (max_ctx_len > (int64_t)max_pages * kPageSize) return KV_ERR_INVALID;
  if (!on_pool_device(p)) return KV_ERR_INVALID;
  if (max_ctx_len == 0) max_ctx_len = 1;
  // beyond the documented limit: refuse
  if (decode_workspace_bytes(n_q_heads, p->head_dim, batch, max_ctx_len) > kStaticScratchBytes) return KV_ERR_WORKSPACE;
  return launch_decode(p, q, n_q_heads, block_tables, max_pages, ctx_lens, batch, max_ctx_len, scale, out, lse,
                       (cudaStream_t)stream);
}

extern "C" size_t attn_decode_static_scratch_bytes(void) { return kStaticScratchBytes; }
