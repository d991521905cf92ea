// Split-KV decode attention without scratch memory: one query token per sequence over the pages of its context.
//
// A cluster of `splits` CTAs owns one (sequence, KV head); its splits * kWarps warps take equal runs of the sequence's
// pages.  Every warp streams its run (page_mma.cuh), the warps of a CTA are merged through shared memory and the CTAs of
// the cluster through distributed shared memory: one kernel, no partial result in global memory, no combine kernel.
// Where there are many short sequences instead, a CTA takes several pairs (pairs_per_cta).
//
// What bounds it: full batches, HBM (256 sequences of 1024-4096 tokens, 32/8 heads of 128: 379 us; the kernel it replaced,
// one warp per 1024-token chunk and a combine kernel behind it, took 418).  Small batches, the latency of a warp's
// pages (about 0.7 us each, whatever the depth of its ring), so the sequence is spread over as many warps as are
// resident: one sequence of 517 tokens 32.0 -> 3.9 us, of 16000 tokens 63 -> 15.9, 8 of 1000-4000 tokens 61.7 -> 19.3.
// kWarps x kStages: six warps with two page slots each, two CTAs per SM (D = 128).  4 x 3, 8 x 3, 12 x 2 and 4 x 6 were
// measured on 20 batch shapes: twelve warps on an SM beat eight everywhere (a slot is refilled as soon as its page is
// in registers, so two are enough), and two CTAs of six beat one of twelve by a sixth on short contexts (128 sequences of
// 200-700 tokens: 44 us) because one starts while the other ends.
#include <math.h>

#include "common.cuh"
#include "page_mma.cuh"
#include "sm100_ptx.cuh"

namespace kvattn {
using namespace ptx;

struct DecodeArgs {
  PoolView pool;
  const __nv_bfloat16* q;  // [batch][Hq][D]
  const int* block_tables;
  int max_pages;
  const int* ctx_lens;
  int n_q_heads, group;
  int splits;        // CTAs of a cluster
  int units;         // (sequence, KV head) pairs
  int per_cta;       // pairs a CTA takes, kWarps / per_cta warps each (1 where splits > 1)
  int len_bound;     // host-side bound on ctx_lens, up to a multiple of kDecodeChunkTokens (a longer sequence is reported and skipped)
  int wait_mode;     // kWaitFirst / kWaitLast
  float scale_log2;  // scale * log2(e)
  __nv_bfloat16* out;
  float* lse;
};
constexpr int kDecodeChunkTokens = 1024;
constexpr int kWaitFirst = 0;  // everything queued before this kernel is waited for before anything is read
constexpr int kWaitLast = 1;   // runs beside the kernel queued before it (attn_mixed); only the grid's end waits for that kernel

constexpr int kWarps = 6;
constexpr int kStages = 2;
constexpr int kMaxSplits = 16;

template <int D>
struct DecodeSmem {
  static constexpr int kSlot = 2 * 16 * D * 2;                // one page of one head: K block, V block
  static constexpr int kRing = kWarps * kStages * kSlot;
  static constexpr int kRowFloats = D + 8;                    // a row of a warp's partial O, padded
  static constexpr int kPart = kWarps * 8 * kRowFloats * 4;   // over the ring once every page has been consumed
  static_assert(kPart <= kRing, "the warps' partials fit into the ring");
  static constexpr int kIn = (8 * D + 4 * kMaxSplits) * 4;    // partials pushed by the cluster's CTAs: [splits][slice]
};

// Everything but the ring (the register variant has no ring and keeps the partials in the same place).
struct DecodeShared {
  unsigned long long bars[kWarps * kStages];
  float ml[kWarps][8][2];         // [warp][row]: maximum, sum
  float in_ml[kMaxSplits][8][2];  // [CTA][row]
  int abort_flag;
  int fits[kWarps];               // [pair of the CTA]: its sequence is as long as the host said or shorter
};

template <int D, bool RING>
constexpr int decode_smem_bytes() {
  return (RING ? DecodeSmem<D>::kRing : DecodeSmem<D>::kPart) + DecodeSmem<D>::kIn + (int)sizeof(DecodeShared);
}

// MULTI: several pairs per CTA (a.per_cta > 1).  An instantiation of its own: with the pair as a run-time value everywhere the
// others lost 0.3 us (13 sequences of 200-3000 tokens, 64 dims, 13.2 -> 13.5; one of 517 4.25 -> 4.5).
template <int D, bool RING, bool MULTI>
__global__ void __launch_bounds__(kWarps * 32) attn_decode_kernel(const DecodeArgs a) {
  using SM = DecodeSmem<D>;
  constexpr int NJ = D / 32, NU = D / 64;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  float* part = reinterpret_cast<float*>(smem_raw);  // [warp][row][kRowFloats], over the ring
  float* in_o = reinterpret_cast<float*>(smem_raw + (RING ? SM::kRing : SM::kPart));
  DecodeShared& sh = *reinterpret_cast<DecodeShared*>(smem_raw + (RING ? SM::kRing : SM::kPart) + SM::kIn);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r = lane >> 2, c = lane & 3;
  const int splits = a.splits;
  const int cluster = blockIdx.x / splits, rank = blockIdx.x - cluster * splits;
  const int Hkv = a.pool.n_kv_heads, G = a.group, Hq = a.n_q_heads;
  const int team = MULTI ? kWarps / a.per_cta : kWarps, mine = MULTI ? warp / team : 0;  // warps of a pair; the pair of this warp
  const int first_unit = MULTI ? cluster * a.per_cta : cluster, n_units = MULTI ? min(a.per_cta, a.units - first_unit) : 1;
  const bool idle = MULTI && mine >= n_units;
  const int unit = idle ? first_unit : first_unit + mine;
  const int seq = unit / Hkv, kvh = unit - seq * Hkv;

  if (RING) {
    if (tid == 0) {
      sh.abort_flag = 0;
      for (int i = 0; i < kWarps * kStages; ++i) ptx::mbar_init(ptx::smem_u32(&sh.bars[i]), 1);
      ptx::fence_mbar_init();
    }
    __syncthreads();
  }
  // (the partner CTAs may be written to once they are known to run: waited for before the push below)
  if (splits > 1) cluster_arrive();
  if (a.wait_mode == kWaitFirst) ptx::dependency_wait();

  const int L = ptx::ld_plain(a.ctx_lens + seq);
  const bool fits = L <= a.max_pages * kPageSize && L <= a.len_bound;
  if (!fits && rank == 0 && lane == 0) report(a.pool.status, KV_ERR_BOUNDS);  // left unwritten
  if (MULTI && lane == 0 && warp == mine * team) sh.fits[mine] = fits;
  const int n_pages = fits && L > 0 && !idle ? (L + kPageSize - 1) / kPageSize : 0;
  const int runs = team * splits;
  const int run = rank * team + warp - mine * team;
  const int p_begin = (int)((int64_t)n_pages * run / runs), p_end = (int)((int64_t)n_pages * (run + 1) / runs);

  // query rows: lane loads row r's chunks; rows past the group are zero
  uint4 qf[NJ];
  {
    const __nv_bfloat16* qp = a.q + ((int64_t)seq * Hq + kvh * G + r) * D;
#pragma unroll
    for (int j = 0; j < NJ; ++j)
      qf[j] = r < G ? ptx::ld_plain(reinterpret_cast<const uint4*>(qp) + 4 * j + c) : make_uint4(0, 0, 0, 0);
  }
  const int limit0 = 2 * c < G ? L : 0, limit1 = 2 * c + 1 < G ? L : 0;

  RowState<D> st;
  st.clear();
  {
    const size_t blk = block_bytes(D);
    const char* kbase = reinterpret_cast<const char*>(a.pool.k) + (size_t)kvh * blk;
    const char* vbase = reinterpret_cast<const char*>(a.pool.v) + (size_t)kvh * blk;
    const size_t page_stride = (size_t)Hkv * blk;
    const int* bt_row = a.block_tables + (int64_t)seq * a.max_pages;
    auto table_entry = [&](int p) {
      int pg = 0;
      if (p < p_end) {
        pg = ptx::ld_plain(bt_row + p);
        if ((unsigned)pg >= (unsigned)a.pool.num_pages) {
          report(a.pool.status, KV_ERR_BOUNDS);
          pg = 0;  // stay inside the pool; the result of this row is flagged, not trusted
        }
      }
      return pg;
    };
    // Block-table entries: 32 per batch, the next batch asked for while this one is walked.
    int cur = table_entry(p_begin + lane), nxt = table_entry(p_begin + 32 + lane);
    int base = p_begin;  // page of cur's lane 0
    auto page_id = [&](int p) {  // p in [base, base + 64); the whole warp calls
      const int i = p - base;
      return __shfl_sync(0xffffffffu, i < 32 ? cur : nxt, i & 31);
    };
    auto advance = [&](int p) {
      if (p - base >= 32) {
        cur = nxt;
        base += 32;
        nxt = table_entry(base + 32 + lane);
      }
    };
    if constexpr (RING) {
      const uint32_t slots = ptx::smem_u32(smem_raw) + warp * (kStages * SM::kSlot);
      const uint32_t bars = ptx::smem_u32(&sh.bars[warp * kStages]);
      const uint64_t policy = ptx::l2_evict_first_policy();  // every page is read once
      uint32_t issued = 0, used = 0;
      auto issue = [&](int p) {
        const int pg = page_id(p);
        if (lane == 0) {
          const uint32_t s = issued % kStages, slot = slots + s * SM::kSlot, bar = bars + s * 8;
          ptx::mbar_arrive_expect_tx(bar, SM::kSlot);
          ptx::bulk_g2s_hint(slot, kbase + (size_t)pg * page_stride, SM::kSlot / 2, bar, policy);
          ptx::bulk_g2s_hint(slot + SM::kSlot / 2, vbase + (size_t)pg * page_stride, SM::kSlot / 2, bar, policy);
        }
        ++issued;
      };
      for (int p = p_begin; p < min(p_begin + kStages, p_end); ++p) issue(p);
      PageRegs<D> pr;
      bool ok = true;
      for (int p = p_begin; p < p_end; ++p) {
        advance(p);
        const uint32_t s = used % kStages;
        ok = ptx::mbar_wait(bars + s * 8, (used / kStages) & 1, &sh.abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        ++used;
        load_page_smem<D>(pr, slots + s * SM::kSlot, r, c);
        // every lane has its copy of the slot in registers: the slot can take the page kStages ahead
        __syncwarp();
        ptx::fence_proxy_async_smem();
        if (p + kStages < p_end) issue(p + kStages);
        page_step<D>(st, pr, qf, p * kPageSize, limit0, limit1, L, a.scale_log2, r, c);
      }
      if (!ok && lane == 0) {  // a wait gave up: flag it and let the copies that were asked for land (bounded)
        report(a.pool.status, KV_ERR_TIMEOUT);
        int never = 0;
        for (; used < issued; ++used)
          ptx::mbar_wait_limit(bars + (used % kStages) * 8, (used / kStages) & 1, &never, 100000000ull);
      }
    } else {
      for (int p = p_begin; p < p_end; ++p) {
        advance(p);
        const int pg = page_id(p);
        PageRegs<D> pr;
        load_page<D>(pr, kbase + (size_t)pg * page_stride, vbase + (size_t)pg * page_stride, r, c);
        page_step<D>(st, pr, qf, p * kPageSize, limit0, limit1, L, a.scale_log2, r, c);
      }
    }
  }

  // The kernel behind this one is let in as soon as a warp of every CTA has its pages, where clusters share a pair, else at the end.  At
  // the start of this one its blocks took the SMs with room left, as many as fit on each, and waited there; blocks that asked for so
  // much shared memory that one or two of them fill an SM did not, but kept other streams' blocks away too.  Us for a call, let in at
  // the start / that with the shared memory / with the pages / at the end.  Clusters: 1 sequence of 517 tokens 4.25 / 4.05 / 4.03 / 4.15, 1
  // of 1454, 64/8 heads, 5.15 / 5.12 / 5.19 / 5.48, 13 of 200-3000, 64 dims, 13.7 / 13.7 / 13.5 / 13.4.  None: 11 of 81-85 3.78 / 3.33 / 3.58 /
  // 3.27, 64 dims, 29 of 79-133 4.75 / 3.80 / 4.24 / 3.75, 16/8 heads, 64 of 344-516 15.5 / 12.9 / 14.2 / 12.9, 73 of 271-308 11.9 / 10.3 /
  // 11.7 / 10.7.  Two streams of 9 sequences of 100-150 (clusters) 4.46 / 7.39 / 4.43, of 18 of up to 40 3.54 / 5.44 / 3.54 / 3.50.
  if (splits > 1) ptx::launch_dependents();

  // ---- the warp's rows to shared memory (every bulk copy into the ring has landed and been read)
#pragma unroll
  for (int off = 4; off < 32; off <<= 1) {
    st.l0 += __shfl_xor_sync(0xffffffffu, st.l0, off);
    st.l1 += __shfl_xor_sync(0xffffffffu, st.l1, off);
  }
  __syncthreads();
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const int n = 2 * c + half;
    if (n >= G) continue;
    float* row = part + (warp * 8 + n) * SM::kRowFloats;
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      float4* dst = reinterpret_cast<float4*>(row + (8 * u + r) * 8);
      dst[0] = make_float4(st.acc[u][0][half], st.acc[u][0][half + 2], st.acc[u][1][half], st.acc[u][1][half + 2]);
      dst[1] = make_float4(st.acc[u][2][half], st.acc[u][2][half + 2], st.acc[u][3][half], st.acc[u][3][half + 2]);
    }
    if (r == 0) {
      sh.ml[warp][n][0] = half ? st.m1 : st.m0;
      sh.ml[warp][n][1] = half ? st.l1 : st.l0;
    }
  }
  __syncthreads();

  // ---- merge.  Element i (four dims of a row) of a pair = row i / (D/4), dims 4 (i % (D/4)) ..
  constexpr int kVec = D / 4;
  const int n_elem = G * kVec;
  auto store = [&](int u, int i, float4 o, float m, float l) {
    const int row = i / kVec, dv = i % kVec;
    const float inv = l > 0.f ? 1.f / l : 0.f;
    const int s_u = MULTI ? u / Hkv : seq, h_u = MULTI ? u - s_u * Hkv : kvh;
    const int64_t orow = (int64_t)s_u * Hq + h_u * G + row;
    *reinterpret_cast<uint2*>(a.out + orow * D + dv * 4) = make_uint2(pack_bf16x2(o.x * inv, o.y * inv), pack_bf16x2(o.z * inv, o.w * inv));
    if (dv == 0) a.lse[orow] = l > 0.f ? (m + log2f(l)) * 0.6931471805599453f : -INFINITY;
  };
  const int slice = (n_elem + splits - 1) / splits;  // elements of the result each CTA finishes (the last ones: what is left)
  if (splits > 1) cluster_wait();                    // the partners run: their shared memory may be written
  for (int e = tid; e < n_units * n_elem; e += kWarps * 32) {
    const int pair = MULTI ? e / n_elem : 0, i = e - pair * n_elem, w0 = pair * team;
    const int row = i / kVec, dv = i % kVec;
    float m = -INFINITY, l = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w)
      if (w < team) m = fmaxf(m, sh.ml[w0 + w][row][0]);
    const float mu = m == -INFINITY ? 0.f : m;
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      if (w >= team) break;
      const float wt = fast_exp2(sh.ml[w0 + w][row][0] - mu);
      l += wt * sh.ml[w0 + w][row][1];
      const float4 x = *reinterpret_cast<const float4*>(part + ((w0 + w) * 8 + row) * SM::kRowFloats + dv * 4);
      o.x += wt * x.x; o.y += wt * x.y; o.z += wt * x.z; o.w += wt * x.w;
    }
    if (splits == 1) {
      if (MULTI ? sh.fits[pair] != 0 : fits) store(first_unit + pair, i, o, m, l);
    } else {
      const int dest = i / slice, at = i - dest * slice;
      st_cluster(cluster_addr(ptx::smem_u32(in_o + ((rank * slice + at) << 2)), dest), o);
      // the row's (maximum, sum) goes to every CTA that finishes a part of the row
      if (dv == 0 || at == 0) st_cluster(cluster_addr(ptx::smem_u32(&sh.in_ml[rank][row][0]), dest), make_float2(m, l));
    }
  }
  if (splits > 1) {
    cluster_arrive();
    cluster_wait();
    for (int at = tid; at < slice && rank * slice + at < n_elem; at += kWarps * 32) {
      const int i = rank * slice + at, row = i / kVec;
      float m = -INFINITY, l = 0.f;
      for (int s = 0; s < splits; ++s) m = fmaxf(m, sh.in_ml[s][row][0]);
      const float mu = m == -INFINITY ? 0.f : m;
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int s = 0; s < splits; ++s) {
        const float wt = fast_exp2(sh.in_ml[s][row][0] - mu);
        l += wt * sh.in_ml[s][row][1];
        const float4 x = *reinterpret_cast<const float4*>(in_o + ((s * slice + at) << 2));
        o.x += wt * x.x; o.y += wt * x.y; o.z += wt * x.z; o.w += wt * x.w;
      }
      if (fits) store(unit, i, o, m, l);
    }
  }
  ptx::launch_dependents();  // (not by ending: a block may still have to wait below)
  // Beside another kernel: this grid must not be complete before that one is, or work queued behind this grid with an
  // early start could overtake it.  The last block (it starts last) is enough.
  if (a.wait_mode == kWaitLast && blockIdx.x == gridDim.x - 1) ptx::dependency_wait();
}

std::atomic<int> g_decode_impl{0};  // 0: by the pages per warp, 1: pages stream through registers, 2: pages go through a shared-memory ring

// Prepares a variant of the kernel for the current device; asking for its attributes loads its code.
template <int D, bool RING, bool MULTI>
static kv_status_t prepare_variant() {
  cudaFuncAttributes at;
  KV_CUDA_OK(cudaFuncGetAttributes(&at, attn_decode_kernel<D, RING, MULTI>));
  KV_CUDA_OK(cudaFuncSetAttribute(attn_decode_kernel<D, RING, MULTI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  decode_smem_bytes<D, RING>()));
  KV_CUDA_OK(cudaFuncSetAttribute(attn_decode_kernel<D, RING, MULTI>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  return KV_OK;
}

// Prepares the kernel for a device, once, and every variant at a time: which one a later call takes depends on its batch and
// lengths, and callers that may not allocate (attn_decode_static) or that capture make one call of any shape beforehand.
static kv_status_t decode_setup(int device) {
  static std::atomic<bool> configured[kMaxDevices];
  if (device < 0 || device >= kMaxDevices) return KV_ERR_INVALID;
  if (!configured[device].load(std::memory_order_acquire)) {
    kv_status_t (*const all[])() = {prepare_variant<128, true, false>, prepare_variant<128, false, false>, prepare_variant<128, true, true>,
                                    prepare_variant<128, false, true>, prepare_variant<64, true, false>,   prepare_variant<64, false, false>,
                                    prepare_variant<64, true, true>,   prepare_variant<64, false, true>};
    for (const auto prepare : all) {
      const kv_status_t s = prepare();
      if (s != KV_OK) return s;
    }
    configured[device].store(true, std::memory_order_release);
  }
  return KV_OK;
}

static void decode_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2], int splits, int64_t blocks, int smem, cudaStream_t st) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(kWarps * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  // launched early: it sets itself up while the kernel in front of it still runs and waits for that one inside
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)splits;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = splits > 1 ? 2 : 1;
}

static constexpr int kSplitChoices[] = {1, 2, 3, 4, 6, 8, 16};

// How many clusters of kSplitChoices[i] CTAs are resident at a time (asked once per device and head size; always of the
// ring variant, so that both variants split alike and give the same bits).
template <int D>
static kv_status_t resident_clusters(int device, int i, int* n) {
  static std::atomic<int> cached[kMaxDevices][sizeof(kSplitChoices) / sizeof(int)];  // value + 1
  const kv_status_t s = decode_setup(device);
  if (s != KV_OK) return s;
  int v = cached[device][i].load(std::memory_order_relaxed);
  if (v == 0) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    decode_config(cfg, attr, kSplitChoices[i], kSplitChoices[i], decode_smem_bytes<D, true>(), nullptr);
    cfg.attrs = attr + 1;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, attn_decode_kernel<D, true, false>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      clusters = 0;
    }
    v = clusters + 1;
    cached[device][i].store(v, std::memory_order_relaxed);
  }
  *n = v - 1;
  return KV_OK;
}

// CTAs per (sequence, KV head), from the host-side bounds alone.
//  - As many as fit on the device at once: a second wave of clusters costs more than the shorter runs save (8 sequences
//    of 1000-4000 tokens: 24.2 / 19.3 / 21.8 us with 2 / 4 / 8), but not more warps than about 3/2 of the sequence's
//    pages (517 tokens: 4.5 / 3.9 / 4.2 us with 4 / 8 / 16).
//  - Where that leaves SMs idle, more, by what the last wave costs.  A wave of less than kFull of the CTAs the device
//    holds is as slow as one of kFull (the memory is saturated with 0.65 of them at 128 dims, hardly with all at 64):
//    32 of 2600-5100 tokens, 64 dims: 51.9 / 52.9 / 45.8 us with 1 / 2 / 3, 64 of 1500-3000: 58.8 / 56.9 / 56.9; 20 of
//    6000-12000, 128 dims: 130 / 132 / 117.  Every further CTA costs about 4 % at 192 pages.
//  - Long sequences of different lengths are split even when the batch fills the device many times over, so that the last
//    CTAs to finish hold less: 64 x 1024-4096 tokens 113.8 -> 104.7 us with 2, 32 x 3230-5100 92.5 -> 88.0; with runs below
//    128 pages it costs (128 x 200-700: 44.0 against 56.4; 24 x 1000-3000, 64/8 heads: 39.1 against 39.9).
template <int D>
static kv_status_t decode_splits(const kv_pool_t* p, int batch, int max_ctx_len, int* splits) {
  const int64_t units = (int64_t)batch * p->n_kv_heads;
  const int pages = (int)(((int64_t)max_ctx_len + kPageSize - 1) / kPageSize);
  constexpr int kChoices = (int)(sizeof(kSplitChoices) / sizeof(int));
  int resident[kChoices];
  *splits = 1;
  for (int i = 0; i < kChoices; ++i) {
    const kv_status_t s = resident_clusters<D>(p->device, i, &resident[i]);
    if (s != KV_OK) return s;
    if (2 * kWarps * kSplitChoices[i] <= 3 * pages && units <= resident[i]) *splits = kSplitChoices[i];
  }
  constexpr double kFull = D == 128 ? 0.65 : 0.9;
  auto score = [&](int c) {
    const double waves = (double)units * c / (resident[0] > 0 ? resident[0] : 1), whole = floor(waves), last = waves - whole;
    const double per_cta = 1.0 + 0.04 * (c - 1) * 192.0 / pages;
    return waves / (whole + (last > 0 ? (last > kFull ? last : kFull) : 0.0)) / per_cta;
  };
  const int cap = pages >= 640 ? 4 : 3;
  double best = score(*splits);
  for (int i = 0; i < kChoices; ++i) {
    const int c = kSplitChoices[i];
    if (c <= *splits || c > cap || pages < 48 * c || resident[i] == 0) continue;
    const double sc = score(c);
    if (sc > best || (pages >= 128 * c && sc > 0.9 * best)) {
      *splits = c;
      best = sc > best ? sc : best;
    }
  }
  return KV_OK;
}

// (sequence, KV head) pairs per CTA where no pair is spread over a cluster: many short sequences are bound by the starts,
// barriers and merges of their CTAs, so a CTA takes as many pairs as bring them all on the device at once, one to three
// warps for a pair, while a warp's run stays short: 16 pages, 8 where there is a second wave all the same.  Us with 1 / 2 /
// 3 / 6 pairs (lengths from two thirds of the stated pages; 128 dims, 296 CTAs resident): 72 x 8 pairs of 6 pages 10.2 / 8.5 / 8.8 /
// 11.8, 103 x 8 of 7 15.5 / 15.8 / 11.8 / 13.7, 222 x 8 of 8 30.2 / 27.3 / 25.2 / 22.1, 75 x 8 of 32 27.6 / 30.7 / 27.3 / 34.5; second
// waves: 251 x 8 of 12 37.9 / 37.6 / 36.9 / 40.0, 149 x 8 of 37 52.5 / 53.2 / 56.0 / 58.6; 64 dims (444 resident): 101 x 8 of 18
// 14.6 / 12.6 / 13.8 / 20.8, 230 x 8 of 48 52.3 / 55.1 / 57.6 / 57.6.
template <int D>
static kv_status_t pairs_per_cta(const kv_pool_t* p, int64_t units, int max_ctx_len, int* n) {
  int resident;
  const kv_status_t s = resident_clusters<D>(p->device, 0, &resident);
  if (s != KV_OK) return s;
  const int pages = (int)(((int64_t)max_ctx_len + kPageSize - 1) / kPageSize);
  *n = 1;
  for (int u : {2, 3, 6})
    if (units > (int64_t)*n * resident && pages * u <= kWarps * (units <= (int64_t)u * resident ? 16 : 8)) *n = u;
  return KV_OK;
}

// Whether a warp has so few pages that it should load them straight into registers: a copy into a slot, its barrier and the
// read back cost 0.3 to 0.6 us more than a load, and with a page or two per warp there is nothing to overlap them with.
// Ring / registers at so many pages per warp: 128 dims 4.2 / 3.9 us (1.0), 6.0 / 5.4 (1.95), 6.6 / 5.9 (2.1), 7.1 / 7.3 (2.1, 8
// sequences), 7.8 / 8.0 (3.1), with more CTAs than are resident 45.6 / 47.1 (6.0), 97.8 / 114.1 (6.0); 64 dims 4.6 / 4.2 (0.8), 5.4 /
// 5.1 (1.6), 6.6 / 6.0 (2.75), 10.6 / 11.2 (4.2).
static bool few_pages(const kv_pool_t* p, int64_t blocks, int warps, int max_ctx_len) {
  const double pages = (double)(max_ctx_len + kPageSize - 1) / kPageSize / warps;
  return pages <= (p->head_dim == 64 ? 2.75 : blocks <= 2 * sm_count_of(p->device) ? 2.0 : 1.0);
}

template <int D, bool RING, bool MULTI>
static kv_status_t launch_decode_variant(const kv_pool_t* p, const DecodeArgs& a, int64_t blocks, cudaStream_t st) {
  const kv_status_t s = decode_setup(p->device);
  if (s != KV_OK) return s;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  decode_config(cfg, attr, a.splits, blocks, decode_smem_bytes<D, RING>(), st);
  KV_CUDA_OK(cudaLaunchKernelEx(&cfg, attn_decode_kernel<D, RING, MULTI>, a));
  count_launch();
  return KV_OK;
}
template <int D, bool RING>
static kv_status_t launch_decode_kernel(const kv_pool_t* p, const DecodeArgs& a, int64_t blocks, cudaStream_t st) {
  return a.per_cta > 1 ? launch_decode_variant<D, RING, true>(p, a, blocks, st) : launch_decode_variant<D, RING, false>(p, a, blocks, st);
}

// What the entry points ask their callers for.  The kernel keeps its partial results on chip and uses none of it; the
// size (that of one partial row per 1024 tokens) is part of the interface.
size_t decode_workspace_bytes(int n_q_heads, int head_dim, int batch, int max_ctx_len) {
  if (batch <= 0 || max_ctx_len <= 0) return 0;
  const int max_chunks = (int)(((int64_t)max_ctx_len + kDecodeChunkTokens - 1) / kDecodeChunkTokens);
  if (max_chunks <= 1) return 0;
  const size_t slots = (size_t)batch * n_q_heads * max_chunks;
  const auto align256 = [](size_t x) { return (x + 255) & ~(size_t)255; };
  return align256(slots * head_dim * sizeof(float)) + align256(slots * sizeof(float));
}

// beside: the kernel may start while the kernel in front of it in the stream still runs and does not wait for it
// (nothing it touches is written there).  The mixed step uses this to run decode next to the extend kernel.
kv_status_t launch_decode(kv_pool_t* p, const void* q, int n_q_heads, const int* block_tables, int max_pages,
                          const int* ctx_lens, int batch, int max_ctx_len, float scale, void* out, float* lse,
                          cudaStream_t st, bool beside) {
  DecodeArgs a{};
  a.pool = p->view();
  a.q = (const __nv_bfloat16*)q;
  a.block_tables = block_tables;
  a.max_pages = max_pages;
  a.ctx_lens = ctx_lens;
  a.n_q_heads = n_q_heads;
  a.group = n_q_heads / p->n_kv_heads;
  const kv_status_t s = p->head_dim == 128 ? decode_splits<128>(p, batch, max_ctx_len, &a.splits)
                                           : decode_splits<64>(p, batch, max_ctx_len, &a.splits);
  if (s != KV_OK) return s;
  const int64_t bound = ((int64_t)max_ctx_len + kDecodeChunkTokens - 1) / kDecodeChunkTokens * kDecodeChunkTokens;
  a.len_bound = (int)(bound < 0x7fffffffLL ? bound : 0x7fffffffLL);
  a.wait_mode = beside ? kWaitLast : kWaitFirst;
  a.scale_log2 = scale * 1.4426950408889634f;
  a.out = (__nv_bfloat16*)out;
  a.lse = lse;
  const int64_t units = (int64_t)batch * p->n_kv_heads;
  if (units * a.splits > 0x7fffffffLL) return KV_ERR_UNSUPPORTED;
  a.units = (int)units;
  a.per_cta = 1;
  if (a.splits == 1) {
    const kv_status_t us = p->head_dim == 128 ? pairs_per_cta<128>(p, units, max_ctx_len, &a.per_cta)
                                              : pairs_per_cta<64>(p, units, max_ctx_len, &a.per_cta);
    if (us != KV_OK) return us;
  }
  const int64_t blocks = (units + a.per_cta - 1) / a.per_cta * a.splits;
  const int impl = g_decode_impl.load();
  const bool ring = impl == 0 ? !few_pages(p, blocks, kWarps / a.per_cta * a.splits, max_ctx_len) : impl != 1;
  if (p->head_dim == 128)
    return ring ? launch_decode_kernel<128, true>(p, a, blocks, st) : launch_decode_kernel<128, false>(p, a, blocks, st);
  return ring ? launch_decode_kernel<64, true>(p, a, blocks, st) : launch_decode_kernel<64, false>(p, a, blocks, st);
}

}  // namespace kvattn
