// Small-tile extend attention: the in-library cross-check of the tensor-core kernel and the path for what that one does
// not take.
//
// One warp owns one work item = (sequence, KV head, tile of 8 query rows) and streams the visible pages straight from
// HBM into registers with coalesced 16-byte loads.  The 8 query rows are 8/G consecutive suffix tokens times the G query
// heads that share the KV head (page_mma.cuh holds the arithmetic on a page).
#include "common.cuh"
#include "page_mma.cuh"
#include "sm100_ptx.cuh"

namespace kvattn {

constexpr int kSmallWarps = 8;
constexpr int kSmallBoundTokens = 1024;  // the host-side bound on a sequence's length is taken up to a multiple of this

struct SmallArgs {
  PoolView pool;
  const __nv_bfloat16* q;  // [rows][Hq][D]
  const int* block_tables;
  int max_pages;
  const int* prefix_lens;
  const int* extend_lens;
  const int* cu_q;
  int n_q_heads, group;
  int max_row_tiles;  // ceil(max_extend_len / (8/G))
  int64_t len_bound;
  float scale_log2;   // scale * log2(e)
  __nv_bfloat16* out;
  float* lse;
};

template <int D>
__global__ void __launch_bounds__(kSmallWarps * 32, 1) attn_small_kernel(SmallArgs a, int64_t total_items) {
  constexpr int NJ = D / 32;  // K chunk loads per token row per lane
  constexpr int NU = D / 64;  // 64-dim halves
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = lane >> 2, c = lane & 3;
  const int64_t item = (int64_t)blockIdx.x * kSmallWarps + warp;
  if (item >= total_items) return;

  const int Hkv = a.pool.n_kv_heads, G = a.group, Hq = a.n_q_heads;
  const int rt = (int)(item % a.max_row_tiles);
  const int64_t rest = item / a.max_row_tiles;
  const int kvh = (int)(rest % Hkv), seq = (int)(rest / Hkv);

  const int P = __ldg(a.prefix_lens + seq), E = __ldg(a.extend_lens + seq), L = P + E;
  const int row0 = __ldg(a.cu_q + seq);
  const int tpt = 8 / G;  // query tokens per tile
  // more suffix tokens than the host-side bound the grid covers: the rows beyond it would never be written
  if (rt == 0 && lane == 0 && (int64_t)E > (int64_t)a.max_row_tiles * tpt) report(a.pool.status, KV_ERR_BOUNDS);
  const int t_first = rt * tpt;
  if (t_first >= E || L <= 0 || P < 0) return;
  if (L > a.max_pages * kPageSize) { report(a.pool.status, KV_ERR_BOUNDS); return; }
  const int t_last = min(E, t_first + tpt) - 1;
  const int tile_limit = P + t_last + 1;  // keys visible to the tile's last token
  // the host-side bound (max_total_len) was too small for this sequence
  if ((int64_t)tile_limit > a.len_bound) { report(a.pool.status, KV_ERR_BOUNDS); return; }

  // the two query rows whose scores this lane holds (n = 2c, 2c+1) and the row it loads (n = r)
  auto row_token = [&](int n) { return t_first + n / G; };
  auto row_head = [&](int n) { return kvh * G + n % G; };
  auto row_valid = [&](int n) { return row_token(n) < E; };
  const int n0 = 2 * c, n1 = 2 * c + 1;
  const bool valid0 = row_valid(n0), valid1 = row_valid(n1);
  const int limit0 = valid0 ? P + row_token(n0) + 1 : 0;
  const int limit1 = valid1 ? P + row_token(n1) + 1 : 0;

  uint4 qf[NJ];
  {
    const bool vr = row_valid(r);
    const __nv_bfloat16* qp = a.q + ((int64_t)(row0 + row_token(r)) * Hq + row_head(r)) * D;
#pragma unroll
    for (int j = 0; j < NJ; ++j)
      qf[j] = vr ? __ldg(reinterpret_cast<const uint4*>(qp) + 4 * j + c) : make_uint4(0, 0, 0, 0);
  }

  RowState<D> st;
  st.clear();
  const size_t blk = block_bytes(D);
  const char* kbase = reinterpret_cast<const char*>(a.pool.k) + (size_t)kvh * blk;
  const char* vbase = reinterpret_cast<const char*>(a.pool.v) + (size_t)kvh * blk;
  const size_t page_stride = (size_t)Hkv * blk;
  const int* bt_row = a.block_tables + (int64_t)seq * a.max_pages;
  const int n_pages = (tile_limit + 15) >> 4;
  for (int pb = 0; pb < n_pages; pb += 32) {
    const int np = min(32, n_pages - pb);
    int my_page = 0;
    if (lane < np) {
      my_page = __ldg(bt_row + pb + lane);
      if ((unsigned)my_page >= (unsigned)a.pool.num_pages) {
        report(a.pool.status, KV_ERR_BOUNDS);
        my_page = 0;  // stay inside the pool; the result of this row is flagged, not trusted
      }
    }
    auto fetch = [&](PageRegs<D>& pr, int p) {
      const int pg = __shfl_sync(0xffffffffu, my_page, p);
      load_page<D>(pr, kbase + (size_t)pg * page_stride, vbase + (size_t)pg * page_stride, r, c);
    };
    auto process = [&](PageRegs<D>& pr, int p) {
      page_step<D>(st, pr, qf, (pb + p) << 4, limit0, limit1, L, a.scale_log2, r, c);
    };
    // two register sets alternate: the next page's loads are in flight while this one is consumed
    PageRegs<D> ra, rb;
    fetch(ra, 0);
    for (int p = 0; p < np; p += 2) {
      if (p + 1 < np) fetch(rb, p + 1);
      process(ra, p);
      if (p + 1 < np) {
        if (p + 2 < np) fetch(ra, p + 2);
        process(rb, p + 1);
      }
    }
  }

  // ---- finish: reduce the row sums over the token lanes, normalise, store
#pragma unroll
  for (int off = 4; off < 32; off <<= 1) {
    st.l0 += __shfl_xor_sync(0xffffffffu, st.l0, off);
    st.l1 += __shfl_xor_sync(0xffffffffu, st.l1, off);
  }
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    if (!(half ? valid1 : valid0)) continue;
    const int n = half ? n1 : n0;
    const float l = half ? st.l1 : st.l0, m = half ? st.m1 : st.m0;
    const float inv = l > 0.f ? 1.f / l : 0.f;
    const int64_t orow = (int64_t)(row0 + row_token(n)) * Hq + row_head(n);
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      uint4 o;
      o.x = pack_bf16x2(st.acc[u][0][half] * inv, st.acc[u][0][half + 2] * inv);
      o.y = pack_bf16x2(st.acc[u][1][half] * inv, st.acc[u][1][half + 2] * inv);
      o.z = pack_bf16x2(st.acc[u][2][half] * inv, st.acc[u][2][half + 2] * inv);
      o.w = pack_bf16x2(st.acc[u][3][half] * inv, st.acc[u][3][half + 2] * inv);
      *reinterpret_cast<uint4*>(a.out + orow * D + (8 * u + r) * 8) = o;
    }
    if (r == 0) a.lse[orow] = l > 0.f ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
  }
}

// Every tile of 8 query rows walks its whole visible KV range, so K/V are re-read once per 8/G suffix tokens.
kv_status_t launch_extend_small(kv_pool_t* p, const void* q, int n_q_heads, const int* cu_q, const int* block_tables,
                                int max_pages, const int* prefix_lens, const int* extend_lens, int batch,
                                int max_extend_len, int max_total_len, float scale, void* out, float* lse,
                                cudaStream_t st) {
  SmallArgs a{};
  a.pool = p->view();
  a.q = (const __nv_bfloat16*)q;
  a.block_tables = block_tables;
  a.max_pages = max_pages;
  a.prefix_lens = prefix_lens;
  a.extend_lens = extend_lens;
  a.cu_q = cu_q;
  a.n_q_heads = n_q_heads;
  a.group = n_q_heads / p->n_kv_heads;
  a.scale_log2 = scale * 1.4426950408889634f;
  a.out = (__nv_bfloat16*)out;
  a.lse = lse;
  const int tpt = 8 / a.group;
  a.max_row_tiles = (max_extend_len + tpt - 1) / tpt;
  a.len_bound = ((int64_t)max_total_len + kSmallBoundTokens - 1) / kSmallBoundTokens * kSmallBoundTokens;
  const int64_t items = (int64_t)batch * p->n_kv_heads * a.max_row_tiles;
  if (items == 0) return KV_OK;
  const int64_t blocks = (items + kSmallWarps - 1) / kSmallWarps;
  if (blocks > 0x7fffffffLL) return KV_ERR_UNSUPPORTED;
  if (p->head_dim == 128)
    attn_small_kernel<128><<<(int)blocks, kSmallWarps * 32, 0, st>>>(a, items);
  else
    attn_small_kernel<64><<<(int)blocks, kSmallWarps * 32, 0, st>>>(a, items);
  count_launch();
  KV_CUDA_OK(cudaGetLastError());
  return KV_OK;
}

}  // namespace kvattn
