// Tensor-core extend attention for sm_100a: suffix queries over reused prefix pages.
//
// Work item = (sequence, KV head, pair of 128-row query tiles).  The rows of a tile are the
// (suffix token, query head of the KV head's group) pairs, token-major, so the G query heads that
// share a KV head share every K/V tile that is brought on chip (GQA) and the causal diagonal is
// only 128/G tokens wide.  One persistent CTA per SM; the items are sorted by cost and taken heaviest
// first from a global counter, so a CTA that finishes early simply takes more.
// Besides extend, the kernel has a prefix-only mode and a fan-out mode (see TcArgs::mode).
//
// Roles (warp-specialised, 16 warps):
//   warps 0-3   softmax of query tile 0: one thread per row (= TMEM lane): masks, running max and
//   warps 4-7   softmax of query tile 1: sum, exp2, P as bf16 back to TMEM, lazy rescale of O.
//   warps 8-11  epilogue of both tiles: O / l -> bf16 -> global, while the softmax warps are already
//               at the next item.
//   warp 12     producer: per 128-token KV tile, one 1-D bulk copy per 16-token page block
//               (the pool keeps blocks in the MMA's 128-byte-swizzle operand layout) into a ring of
//               shared-memory stages; completion is signalled on mbarriers.
//   warp 13     MMA issuer (one elected lane): S = Q K^T and O += P V on tcgen05 with accumulators in
//               tensor memory; P is read straight from tensor memory (it overwrites S in place).
//   warp 14     Q loader: one tensor-map (TMA) copy per 64-dim half brings a query tile into shared
//               memory in the swizzled operand layout, as soon as the MMAs that read the previous
//               item's tile have finished.
//   warp 15     span scheduling: finds the CTA's span and announces its items; else idle (launched for the registers it
//               hands to the others).
// The two query tiles ping-pong: while one tile's softmax runs, the tensor core works on the other.
// All waits are bounded; on expiry the CTA records KV_ERR_TIMEOUT, drains its copies, frees its
// tensor memory and returns.
#include <math.h>

#include <type_traits>

#include <cuda.h>  // CUtensorMap and its enums (types only: the encoder is looked up at run time)

#include "append.cuh"
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace kvattn {
using namespace ptx;

// The roles' register budgets are set with setmaxnreg.  What the warps hold afterwards must not exceed what the
// CTA was launched with (512 threads x 128 registers), in total and per scheduler (warp index mod 4):
// 8 x 192 (softmax) + 4 x 72 (epilogue) + 56 + 56 + 40 + 24 = 2000 <= 2048 per lane.
constexpr int kTcThreads = 512;
constexpr int kWarpEpilogue = 8, kWarpProducer = 12, kWarpMma = 13, kWarpQ = 14, kWarpSched = 15;
constexpr int kPlanBuckets = 2048;
constexpr int kPlanSeqBuckets = 1024;   // length buckets for ranking the sequences (one per plan thread)
constexpr int kPlanMaxRanked = 8192;    // batches up to this size are ranked by length; larger ones keep their order
constexpr float kRescaleThreshold = 8.0f;  // log2 units: O is rescaled only when the max grows by more than this
constexpr int kOptimisticMinLen = 4096;     // batches with a sequence this long use the kernel that skips the maximum search
constexpr float kOptimisticSum = 65536.0f;  // a row sum of one tile beyond this sends the step to the exact maximum

// Span scheduling, for batches with few work items per SM.  The KV steps of all items, laid end to end, are cut into
// at most n_spans spans of equal length, one CTA takes one (in attn_mixed: a few neighbouring ones), and an item that a
// cut goes through leaves partial results that span_combine_kernel merges.  Every CTA finds its span by itself from the
// length arrays, so no plan kernel runs in front.  The cuts depend on the lengths and on n_spans alone.
struct SpanArgs {
  int n_spans, per_cta;  // spans at most; neighbouring spans one CTA takes
  int max_tp, total_q;   // host-side bounds: tile pairs of a sequence, rows of Q
  int plan_early;        // the kernel in front is this call's own append: lengths, tables and Q may be read before it is done
  int4* desc;            // [n_spans][3]: the cut at the start of a span: (first step of the item it goes through among all
                         // steps, or -1; step of the item; KV head; tile pair), (rows, first row, KV steps of the two tiles)
  int rows;              // rows a slot of partial results holds (no item of the batch has more)
  float* part_o;         // [slot][D / 8][rows][8]: a cut item's rows, normalised within the chunk (nullptr: no item is cut);
                         // eight dims of a row, then the next row, so that a warp's rows are contiguous.  Slots: two per
                         // span, or one per CTA of the clusters
  float* part_lse;       // [slot][rows]: log2-domain log-sum-exp of the chunk (clusters: the maximum and the sum)
};
constexpr int kSpanMinSteps = 2;  // KV steps of a span at least
constexpr int kSpanSnap = 1;      // a cut this close to the edge of an item moves to the edge

// Who takes which items.
//  kSchedList: the plan's list, through a work counter (any number of items).
//  kSchedSpans: equal spans of KV steps (see SpanArgs).
//  kSchedCluster: one item per cluster of cl_splits CTAs, each with an equal part of its KV steps; their results are merged
//  through L2 behind a cluster barrier.  For batches whose items, that many CTAs each, are on the device at once.
constexpr int kSchedList = 0, kSchedSpans = 1, kSchedCluster = 2;
constexpr int kMaxClusterSplits = 8;

struct TcArgs {
  PoolView pool;
  const __nv_bfloat16* q;
  const int* cu_q;
  const int* block_tables;
  int max_pages;
  const int* prefix_lens;
  const int* extend_lens;
  int batch, n_q_heads, group, lg_group;
  // mode 0: row t of sequence i sees the keys 0 .. P_i + t (extend).
  // mode 1: every row sees the keys [0, P_i) only.
  // mode 2 (fan-out): a "sequence" is a parent, its rows are the suffix tokens of its children stacked one
  //         after the other; a row sees the parent's keys [0, P) and then its own child's keys up to itself.
  //         The KV steps of an item are eight pages each of the parent's pages followed by those of every child that
  //         has a row in the item.
  int mode;
  FanArgs fan;
  float scale_log2;
  __nv_bfloat16* out;
  float* lse;
  const int4* items;   // two int4 per entry (see ItemRec), cost-sorted
  const int* n_items;  // number of valid entries in items
  int* next_item;      // work counter: the next item of the global list nobody has taken yet
  SpanArgs span;       // span scheduling and items per cluster (no plan, no counter)
  int cl_splits;
  int beside;          // a decode kernel is to run beside this one (attn_mixed)
};

// ------------------------------------------------------------------------------------------
// Plan: list the (sequence, tile pair) entries that have rows, heaviest first (counting sort on
// the number of KV tile steps).  Only the order of execution depends on it, never a result.
// ------------------------------------------------------------------------------------------
// One entry of the plan: everything a CTA needs to know about a (sequence, tile pair), so that the
// roles read one 32-byte record per item instead of chasing the length arrays.
struct ItemRec {
  int seq, tp, P, E;
  int row0, n_kv0, n_kv1, kv_end;  // first query row; KV tile steps of the two tiles; keys the item sees at most
                                   // (fan-out mode: kv_end holds the first child that has a row in the item, the upper
                                   // bits of tp the pages of its last step)
};

__device__ __forceinline__ ItemRec make_item(int seq, int tp, int P, int E, int row0, int lg, int max_pages, int mode,
                                             const FanArgs& fan) {
  ItemRec r{seq, tp, P, E, row0, 0, 0, 0};
  int tok_hi_t[2] = {-1, -1};
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int r_lo = tp * 256 + t * 128;
    const int tok_lo = r_lo >> lg;
    if (tok_lo >= E) break;
    const int tok_hi = min(E - 1, (r_lo + 127) >> lg);
    tok_hi_t[t] = tok_hi;
    const int sees = mode != 0 ? P : P + tok_hi + 1;
    (t ? r.n_kv1 : r.n_kv0) = (sees + 127) >> 7;
    r.kv_end = sees;
  }
  if ((mode != 0 ? P : P + E) > max_pages * kPageSize) r.n_kv0 = r.n_kv1 = 0;  // longer than its block-table row: skipped (reported by the plan)
  if (mode == 2 && tok_hi_t[0] >= 0) {
    // children with a row in this item: the first one whose last token lies at or after the item's first token,
    // then on until a child starts after the item's last token
    const int c0 = ptx::ld_plain(fan.cu_children + seq), c1 = ptx::ld_plain(fan.cu_children + seq + 1);
    const int tok_lo = (tp * 256) >> lg;
    int lo = c0, hi = c1;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (ptx::ld_plain(fan.cu_q + mid + 1) - row0 > tok_lo) hi = mid; else lo = mid + 1;
    }
    const int c_first = lo;
    const int tok_hi_item = max(tok_hi_t[0], tok_hi_t[1]);
    // The item's keys are a list of pages: the parent's, then those of every child with a row in the item (of the last
    // child only what the item's rows see).  A KV step is eight pages of that list, so that short children share a step
    // with each other and with the end of the parent.
    int pages0 = 0, pages = 0;  // of the children, for the first tile's rows and for both tiles'
    bool fits = P <= max_pages * kPageSize;
    for (int c = c_first; c < c1; ++c) {
      const int start = ptx::ld_plain(fan.cu_q + c) - row0, len = ptx::ld_plain(fan.cu_q + c + 1) - ptx::ld_plain(fan.cu_q + c);
      if (start > tok_hi_item) break;
      if (len > fan.max_pages * kPageSize) fits = false;
      if (start <= tok_hi_t[0]) pages0 = pages + ((min(len, tok_hi_t[0] - start + 1) + 15) >> 4);
      pages += (min(len, tok_hi_item - start + 1) + 15) >> 4;
    }
    const int own = (P + kPageSize - 1) / kPageSize, total = own + pages;
    r.n_kv0 = fits ? (own + pages0 + 7) >> 3 : 0;
    r.n_kv1 = fits && tok_hi_t[1] >= 0 ? (total + 7) >> 3 : 0;
    r.kv_end = c_first;
    r.tp |= ((total - 1) & 7) << 28;  // pages of the last step, less one
  }
  return r;
}

struct PlanArgs {
  const int* prefix_lens;
  const int* extend_lens;
  const int* cu_q;
  int batch, max_tp, lg, max_steps, capacity, max_pages, mode;
  FanArgs fan;
  int groups;
  int* status;
  int4* items;
  int* n_items;
  int* next_item;
  int first_free_item;
};

// Runs in one block of 1024 threads.
__device__ __forceinline__ void plan_body(const PlanArgs& pa) {
  const int* __restrict__ prefix_lens = pa.prefix_lens;
  const int* __restrict__ extend_lens = pa.extend_lens;
  const int* __restrict__ cu_q = pa.cu_q;
  const int batch = pa.batch, max_tp = pa.max_tp, lg = pa.lg, max_steps = pa.max_steps, capacity = pa.capacity;
  const int max_pages = pa.max_pages, mode = pa.mode, groups = pa.groups, first_free_item = pa.first_free_item;
  const FanArgs& fan = pa.fan;
  int* status = pa.status;
  int4* __restrict__ items = pa.items;
  int* __restrict__ n_items = pa.n_items;
  int* __restrict__ next_item = pa.next_item;
  if (threadIdx.x == 0) {
    next_item[0] = first_free_item;  // the CTAs start on items 0 .. grid-1 without asking
    next_item[1] = 0;                // CTAs of the attention kernel that have finished
  }
  __shared__ int hist[kPlanBuckets];
  for (int i = threadIdx.x; i < kPlanBuckets; i += blockDim.x) hist[i] = 0;
  __syncthreads();
  const int64_t n = (int64_t)batch * max_tp;
  // Fan-out mode: a sequence is a parent, its rows are those of its children, which follow one another in Q.
  auto row_of = [&](int seq) { return mode == 2 ? ptx::ld_plain(cu_q + ptx::ld_plain(fan.cu_children + seq)) : ptx::ld_plain(cu_q + seq); };
  auto rows_of = [&](int seq) { return mode == 2 ? row_of(seq + 1) - row_of(seq) : ptx::ld_plain(extend_lens + seq); };
  // A sequence with more suffix tokens than the host-side bound the grid was sized with would lose its last rows
  // without a trace: it is reported instead.
  for (int seq = threadIdx.x; seq < batch; seq += blockDim.x) {
    const int E = rows_of(seq);
    if (ptx::ld_plain(prefix_lens + seq) >= 0 && (int64_t)E > (((int64_t)max_tp * 256) >> lg)) report(status, KV_ERR_BOUNDS);
  }
  // The sequences are put into groups longest first, so that the last groups, which decide how evenly the CTAs
  // finish, hold the cheapest items: a counting sort of the sequences on their length (ties in arrival order: only
  // the order of execution depends on it).
  __shared__ int seq_hist[kPlanSeqBuckets];
  __shared__ unsigned short seq_rank[kPlanMaxRanked];
  const bool ranked = groups > 1 && batch <= kPlanMaxRanked;
  if (ranked) {
    __shared__ int seq_warp_tot[32];
    seq_hist[threadIdx.x] = 0;
    __syncthreads();
    const int64_t span = (int64_t)max(max_steps, 1) * 64 + 1;  // longer than any sequence the tables can hold
    auto bucket_of = [&](int P, int E) {
      return (int)min((int64_t)(kPlanSeqBuckets - 1), (int64_t)(P + E) * kPlanSeqBuckets / span);
    };
    for (int seq = threadIdx.x; seq < batch; seq += blockDim.x) {
      const int P = ptx::ld_plain(prefix_lens + seq), E = rows_of(seq);
      if (P >= 0 && E > 0) atomicAdd(&seq_hist[bucket_of(P, E)], 1);
    }
    __syncthreads();
    {  // exclusive prefix, longest bucket first: thread i owns bucket B-1-i
      const int b = kPlanSeqBuckets - 1 - (int)threadIdx.x;
      const int c = seq_hist[b];
      int incl = c;
      const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += v;
      }
      if (lane == 31) seq_warp_tot[w] = incl;
      __syncthreads();
      if (w == 0) {
        int t = seq_warp_tot[lane];
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, t, off);
          if (lane >= off) t += v;
        }
        seq_warp_tot[lane] = t;
      }
      __syncthreads();
      seq_hist[b] = (w > 0 ? seq_warp_tot[w - 1] : 0) + incl - c;
    }
    __syncthreads();
    for (int seq = threadIdx.x; seq < batch; seq += blockDim.x) {
      const int P = ptx::ld_plain(prefix_lens + seq), E = rows_of(seq);
      seq_rank[seq] = (P >= 0 && E > 0) ? (unsigned short)atomicAdd(&seq_hist[bucket_of(P, E)], 1) : 0;
    }
    __syncthreads();
  }
  // Sort key, larger = earlier: the sequences are taken group after group (a group's K/V stays in L2 while its items
  // run, and the tile pairs of a sequence read the same pages), heaviest item first inside a group.
  const int per_group = kPlanBuckets / groups;
  auto key_of = [&](int steps, int seq) {
    const int64_t k = (int64_t)steps * (per_group - 1) / max(max_steps, 1);
    const int cost = (int)min((int64_t)(per_group - 1), k);
    const int grp = (int)((int64_t)(ranked ? (int)seq_rank[seq] : seq) * groups / batch);
    return (groups - 1 - grp) * per_group + cost;
  };
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
    const int seq = (int)(e / max_tp), tp = (int)(e % max_tp);
    const int P = ptx::ld_plain(prefix_lens + seq), E = rows_of(seq);
    if (P < 0 || E <= 0) continue;
    if (((tp * 256) >> lg) >= E) continue;
    const ItemRec r = make_item(seq, tp, P, E, row_of(seq), lg, max_pages, mode, fan);
    const int steps = r.n_kv0 + r.n_kv1;
    if (steps > 0) atomicAdd(&hist[key_of(steps, seq)], 1);
  }
  __syncthreads();
  // exclusive prefix over the buckets, heaviest first: thread i owns buckets B-1-2i and B-2-2i
  {
    __shared__ int warp_tot[32];
    const int b0 = kPlanBuckets - 1 - 2 * (int)threadIdx.x, b1 = b0 - 1;
    const int c0 = hist[b0], c1 = hist[b1];
    int incl = c0 + c1;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += v;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    if (w == 0) {
      int t = warp_tot[lane];
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, t, off);
        if (lane >= off) t += v;
      }
      warp_tot[lane] = t;  // inclusive totals of the warps
    }
    __syncthreads();
    const int base = (w > 0 ? warp_tot[w - 1] : 0) + incl - (c0 + c1);
    hist[b0] = base;
    hist[b1] = base + c0;
    if (threadIdx.x == blockDim.x - 1) *n_items = min(base + c0 + c1, capacity);
  }
  __syncthreads();
  for (int64_t e = threadIdx.x; e < n; e += blockDim.x) {
    const int seq = (int)(e / max_tp), tp = (int)(e % max_tp);
    const int P = ptx::ld_plain(prefix_lens + seq), E = rows_of(seq);
    if (P < 0 || E <= 0) continue;
    if (((tp * 256) >> lg) >= E) continue;
    const ItemRec r = make_item(seq, tp, P, E, row_of(seq), lg, max_pages, mode, fan);
    const int steps = r.n_kv0 + r.n_kv1;
    if (steps == 0 && (mode == 0 || P > 0 || mode == 2)) report(status, KV_ERR_BOUNDS);  // rows exist but the lengths do not fit the tables
    if (steps > 0) {
      const int pos = atomicAdd(&hist[key_of(steps, seq)], 1);
      if (pos < capacity) {
        items[2 * pos] = make_int4(r.seq, r.tp, r.P, r.E);
        items[2 * pos + 1] = make_int4(r.row0, r.n_kv0, r.n_kv1, r.kv_end);
      } else {
        report(status, KV_ERR_BOUNDS);  // more rows on the device than the total the host gave: the entry is dropped
      }
    }
  }
}

__global__ void __launch_bounds__(1024) extend_tc_plan_kernel(const PlanArgs pa) {
  dependency_wait();
  // The attention kernel may set itself up meanwhile; it waits for this kernel before it reads the plan.  (Not before the
  // wait: a decode kernel that runs beside the attention kernel waits for nothing, and what precedes this kernel has to be
  // complete by then.)
  launch_dependents();
  plan_body(pa);
}

// Prologue of the fused append + extend call: block 0 builds the plan while the other blocks scatter the suffix K/V
// rows into their pages (one warp per token), so the step has one small kernel in front of the attention kernel
// instead of two in a row, and the attention kernel's launch and set-up overlap it.
__global__ void __launch_bounds__(1024) extend_prologue_kernel(const PlanArgs pa, const PoolView pool, const AppendArgs ap, int tokens_per_block) {
  dependency_wait();
  launch_dependents();
  if (blockIdx.x == 0) {
    plan_body(pa);
  } else {
    const int warp = threadIdx.x >> 5;
    if (warp < tokens_per_block) append_tokens<4>(pool, ap, (blockIdx.x - 1) * tokens_per_block + warp, (gridDim.x - 1) * tokens_per_block);
  }
}

__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// ------------------------------------------------------------------------------------------
template <int D>
struct TcCfg {
  static constexpr int kTileBytes = 128 * D * 2;   // a 128-row tile of Q, K or V
  static constexpr int kBlockBytes = 16 * D * 2;   // one (page, head) block
  static constexpr int kStages = D == 128 ? 5 : 8;
  static constexpr uint32_t kGroupStride = D * 16;  // bytes between 8-token groups inside the K/V tiles
  static constexpr int kHalves = D / 64;
  static constexpr int kQHalfStride = 128 * 128;    // Q tile: [half][row][128 B]
};

template <int D>
struct __align__(1024) TcSmem {
  unsigned char q[2][TcCfg<D>::kTileBytes];
  unsigned char kv[TcCfg<D>::kStages][TcCfg<D>::kTileBytes];
  unsigned long long kv_full[TcCfg<D>::kStages], kv_empty[TcCfg<D>::kStages];
  unsigned long long q_full[2], q_empty[2], s_full[2], p_full[2], o_full[2], o_empty[2], l_full[2];
  // Item queue of the CTA: the producer takes items off the global list (heaviest first, whoever is free
  // takes the next) and announces them here; every role walks the same sequence.
  unsigned long long sched_full[4], sched_empty[4];
  int sched_idx[4];
  int4 sched_rec[4][3];    // the whole record of an item (see SpanRec)
  int4 cl_unit;            // one item per cluster: its rows, first row in Q, tile pair, KV head
  float inv_l[2][2][128];  // [tile][item parity][row]: 1 / row sum, handed from the softmax to the epilogue warps
  uint32_t tmem_base;
  int abort_flag;
};

// Span scheduling: what the scheduler warp announces of a chunk of an item (P and kv_end count from the chunk's first key).
struct SpanRec {
  int seq, kvh, tp, P;
  int E, row0, n_kv0, n_kv1;
  int kv_end, first_tile, part;  // part: slot of the partial result, -1 for a whole item (fan-out mode: P counts from the
                                 // parent's first key, and the first child of the item follows)
};

struct Item {
  int seq, kvh, tp, P, E, row0;
  int n_kv[2];   // KV tile steps of the two query tiles (0 = tile has no rows)
  int ld_tiles;  // KV tiles the producer brings in
  int kv_end;    // keys the item can see at most (fan-out mode: slots of all its pages)
  int c_first;   // fan-out mode: first child with a row in the item
  int first_tile, part;  // span scheduling: first KV tile of the chunk, slot of its partial result (-1: none)
};

// Item k of the global list: entry k / Hkv of the plan, KV head k % Hkv.  Returns false past the end.
template <bool FAN>
__device__ __forceinline__ bool fetch_item(const TcArgs& a, int k, int n_total, Item& it) {
  if (k >= n_total) return false;
  const int Hkv = a.pool.n_kv_heads;
  const int e = k / Hkv;
  const int4 r0 = __ldcg(a.items + 2 * e), r1 = __ldcg(a.items + 2 * e + 1);  // written by the kernel before this one: read through L2
  it.seq = r0.x; it.tp = r0.y; it.P = r0.z; it.E = r0.w;
  it.row0 = r1.x; it.n_kv[0] = r1.y; it.n_kv[1] = r1.z; it.kv_end = r1.w;
  it.c_first = 0;
  it.kvh = k - e * Hkv;
  it.ld_tiles = max(it.n_kv[0], it.n_kv[1]);
  if (FAN) {
    it.c_first = r1.w;
    it.kv_end = ((it.ld_tiles - 1) * 8 + (int)((unsigned)r0.y >> 28) + 1) * kPageSize;  // slots of the item's pages
    it.tp = r0.y & 0x0fffffff;
  }
  return true;
}

// Span scheduling.  A sequence's items are ordered (KV head, tile pair); position x of the line of all steps is step
// `off` of the item (seq, kvh, tp) that starts at `at`.
struct SpanPos {
  int seq, kvh, tp, off, at;
};

// Rows of the sequence that count: none if the lengths do not fit the tables, no row past the host-side bounds.
__device__ __forceinline__ int span_rows(const TcArgs& a, int P, int E, int row0) {
  // (fan-out mode: the rows' own keys are not in the parent's table)
  if (P < 0 || E <= 0 || row0 < 0 || (a.mode != 0 ? P : P + E) > a.max_pages * kPageSize) return 0;
  return min(min(E, (int)min((int64_t)0x7fffffff, ((int64_t)a.span.max_tp * 256) >> a.lg_group)), max(0, a.span.total_q - row0));
}
// KV steps of tile pair tp of a sequence with E rows behind P keys
__device__ __forceinline__ int span_steps(int P, int E, int tp, int lg) { return (P + min(E, ((tp + 1) * 256) >> lg) + 127) >> 7; }
__device__ __forceinline__ int span_pairs(int E, int lg) { return (int)(((int64_t)E * (1 << lg) + 255) >> 8); }
// Steps of the first m tile pairs if all of them are full: sum over k = 1 .. m of ceil((P + k * 256 / G) / 128).  A pair's
// tokens are 256, 128, 64 or 32, so the terms grow by 2, by 1, or by 1 every 2 or 4 pairs.
__device__ __forceinline__ int span_full_steps(int P, int m, int lg) {
  const int cp = (P + 127) >> 7;
  if (lg < 2) return m * cp + (lg == 0 ? m * (m + 1) : (m * (m + 1)) >> 1);
  const int lq = lg - 1, tokens = 256 >> lg;
  int sum = 0;
  for (int r = 1; r <= (1 << lq); ++r) {
    const int cnt = m >= r ? ((m - r) >> lq) + 1 : 0;
    sum += cnt * ((P + tokens * r + 127) >> 7) + ((cnt * (cnt - 1)) >> 1);
  }
  return sum;
}
// Steps of all tile pairs of one KV head of a sequence
__device__ __forceinline__ int span_head_steps(int P, int E, int lg) {
  const int pairs = span_pairs(E, lg);
  return pairs == 0 ? 0 : span_full_steps(P, pairs - 1, lg) + span_steps(P, E, pairs - 1, lg);
}
__device__ __forceinline__ int span_count(const SpanArgs& a, int total) {
  return max(1, min(a.n_spans, (total + kSpanMinSteps - 1) / kSpanMinSteps));
}
// Where span s begins, among all steps
__device__ __forceinline__ int span_cut(int total, int n_spans, int s) {
  const int each = total / n_spans, rest = total - each * n_spans;
  return each * s + rest * s / n_spans;
}
// Where a cut at step `off` of an item of n steps goes: 0 or n (an edge), or it stays (unless items are not to be cut).
__device__ __forceinline__ int span_snap(const SpanArgs& a, int off, int n) {
  if (off <= kSpanSnap) return 0;
  if (n - off <= kSpanSnap) return n;
  return a.part_o != nullptr ? off : 2 * off < n ? 0 : n;
}

// The lengths of 32 sequences, one per lane.
struct SpanSeqs {
  int base, P, rows, row0;
};
__device__ __forceinline__ void span_load(const TcArgs& a, int base, SpanSeqs& q) {
  const int seq = base + (threadIdx.x & 31);
  q.base = base;
  q.P = q.rows = q.row0 = 0;
  if (seq < a.batch) {
    const int P = ptx::ld_plain(a.prefix_lens + seq), E = ptx::ld_plain(a.extend_lens + seq);
    q.row0 = ptx::ld_plain(a.cu_q + seq);
    q.P = P;
    q.rows = span_rows(a, P, E, q.row0);
    if (blockIdx.x == 0 && P >= 0 && q.rows < E) report(a.pool.status, KV_ERR_BOUNDS);
  }
}

// One warp: sums the steps of all sequences and finds the item and step at which span `first_span` begins (seq = batch:
// nothing to do).
__device__ __forceinline__ void span_locate(const TcArgs& a, int first_span, SpanPos& pos, int& total, SpanSeqs& q) {
  const int lane = threadIdx.x & 31, lg = a.lg_group, Hkv = a.pool.n_kv_heads;
  span_load(a, 0, q);
  int mine = span_head_steps(q.P, q.rows, lg);
  total = mine;
  for (int base = 32; base < a.batch; base += 32) {
    SpanSeqs t;
    span_load(a, base, t);
    total += span_head_steps(t.P, t.rows, lg);
  }
  total = __reduce_add_sync(0xffffffffu, total) * Hkv;
  pos = SpanPos{a.batch, 0, 0, 0, total};
  const int n_spans = span_count(a.span, total);
  if (first_span >= n_spans || total == 0) return;
  const int x = span_cut(total, n_spans, first_span);
  int before = 0;  // steps of the sequences in front
  while (true) {
    int incl = mine * Hkv;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += u;
    }
    const unsigned behind = __ballot_sync(0xffffffffu, before + incl > x);
    if (behind) {
      const int l = __ffs(behind) - 1;
      pos.seq = q.base + l;
      const int per_head = __shfl_sync(0xffffffffu, mine, l);
      int rem = x - before - (__shfl_sync(0xffffffffu, incl, l) - per_head * Hkv);
      const int P = __shfl_sync(0xffffffffu, q.P, l), rows = __shfl_sync(0xffffffffu, q.rows, l);
      pos.kvh = rem / per_head;
      rem -= pos.kvh * per_head;
      // tile pair: the last one with span_full_steps(pair) <= rem, 32 probes at a time
      int lo = 0, span = span_pairs(rows, lg);
      while (span > 1) {
        const int step = (span + 31) >> 5, idx = lo + lane * step, end = lo + span;
        const int k = __popc(__ballot_sync(0xffffffffu, idx < end && span_full_steps(P, idx, lg) <= rem)) - 1;
        lo += k * step;
        span = min(step, end - lo);
      }
      pos.tp = lo;
      pos.off = rem - span_full_steps(P, lo, lg);
      pos.at = x - pos.off;
      return;
    }
    before += __shfl_sync(0xffffffffu, incl, 31);
    span_load(a, q.base + 32, q);
    mine = span_head_steps(q.P, q.rows, lg);
  }
}

// Operand descriptors differ only in their low word (start address >> 4 plus the leading-dimension
// offset field); the high word is a constant.  Issuing an MMA then costs one add, so a single thread
// keeps the tensor pipe fed.
__device__ __forceinline__ uint64_t make_desc(uint32_t hi, uint32_t lo) { return ((uint64_t)hi << 32) | lo; }

// S[128 rows x 128 keys] = Q_t (K-major, shared) x K_stage (K-major, shared); q_lo / k_lo: low descriptor words
template <int D>
__device__ __forceinline__ void issue_s_mmas(uint32_t s_tmem, uint32_t q_lo, uint32_t k_lo) {
  constexpr uint32_t kHiQ = (1024u >> 4) | (1u << 14) | (2u << 29);        // SBO 1024, sm_100 descriptor, 128B swizzle
  constexpr uint32_t kHiK = ((uint32_t)(D * 16) >> 4) | (1u << 14) | (2u << 29);  // SBO = 8-token group stride
  constexpr uint32_t idesc = idesc_bf16(128, 128, 0, 0);
#pragma unroll
  for (int ks = 0; ks < D / 16; ++ks)
    mma_ss(s_tmem, make_desc(kHiQ, q_lo + (ks >> 2) * 1024 + (ks & 3) * 2), make_desc(kHiK, k_lo + (ks >> 2) * 64 + (ks & 3) * 2),
           idesc, ks > 0);
}

// O[128 rows x D] (+)= P (bf16 in tensor memory) x V_stage (MN-major, shared), one MMA per 16-token page
template <int D>
__device__ __forceinline__ void issue_pv_mmas(uint32_t o_tmem, uint32_t p_tmem, uint32_t v_lo, int np, bool first) {
  constexpr uint32_t kHiV = ((uint32_t)(D * 16) >> 4) | (1u << 14) | (2u << 29);
  constexpr uint32_t idesc = idesc_bf16(128, D, 0, 1);
  mma_ts(o_tmem, p_tmem, make_desc(kHiV, v_lo), idesc, first ? 0u : 1u);
#pragma unroll
  for (int p = 1; p < 8; ++p)
    if (p < np) mma_ts(o_tmem, p_tmem + p * 8, make_desc(kHiV, v_lo + p * (D * 2)), idesc, 1u);
}

// Partial results lie in pieces of eight dims: [slot][D / 8][rows][8].
// 32 dims of a row, scaled, from registers: four pieces (a warp's 32 rows are contiguous in each).
__device__ __forceinline__ void store_part8x4(float* dst, int rows, const uint32_t (&o)[32], float inv) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(dst + (int64_t)rows * 8 * i),
                 "f"(__uint_as_float(o[8 * i]) * inv), "f"(__uint_as_float(o[8 * i + 1]) * inv),
                 "f"(__uint_as_float(o[8 * i + 2]) * inv), "f"(__uint_as_float(o[8 * i + 3]) * inv),
                 "f"(__uint_as_float(o[8 * i + 4]) * inv), "f"(__uint_as_float(o[8 * i + 5]) * inv),
                 "f"(__uint_as_float(o[8 * i + 6]) * inv), "f"(__uint_as_float(o[8 * i + 7]) * inv)
                 : "memory");
}
__device__ __forceinline__ void store_part8x4(float* dst, int rows, const uint32_t (&o)[32]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(dst + (int64_t)rows * 8 * i), "r"(o[8 * i]), "r"(o[8 * i + 1]),
                 "r"(o[8 * i + 2]), "r"(o[8 * i + 3]), "r"(o[8 * i + 4]), "r"(o[8 * i + 5]), "r"(o[8 * i + 6]), "r"(o[8 * i + 7])
                 : "memory");
}
// A piece of a partial result: 32 bytes in one load (two of 16 bytes ask for every sector twice).
__device__ __forceinline__ void load_part8(const float* src, float (&x)[8]) {
  asm volatile("ld.global.L1::no_allocate.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(x[4]), "=f"(x[5]), "=f"(x[6]), "=f"(x[7])
               : "l"(src)
               : "memory");
}
// Merges piece g of row r over its chunks, in chunk order, U chunks' loads in flight: eight dims as bf16, and the
// log2-domain log-sum-exp.  slot(k): slot of chunk k; has(k): does chunk k hold a step of the row's tile (else its slot
// was not written; a chunk without a key the row sees has weight 0).
template <int D, int U, typename Slot, typename Has>
__device__ __forceinline__ uint4 merge_part8(const SpanArgs& a, int chunks, int r, int g, Slot slot, Has has, float& lse2) {
  float mx = -INFINITY, wsum = 0.f, o[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) o[e] = 0.f;
  for (int base = 0; base < chunks; base += U) {
    float l[U], x[U][8];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = base + u;
      l[u] = -INFINITY;
      if (k < chunks && has(k)) {
        const int sl = slot(k);
        l[u] = __ldcg(a.part_lse + sl * a.rows + r);
        load_part8(a.part_o + (((int64_t)sl * (D / 8) + g) * a.rows + r) * 8, x[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (l[u] == -INFINITY) continue;
      const float mn = fmaxf(mx, l[u]);
      const float keep = exp2f(mx - mn), w = exp2f(l[u] - mn);
      mx = mn;
      wsum = wsum * keep + w;
#pragma unroll
      for (int e = 0; e < 8; ++e) o[e] = o[e] * keep + w * x[u][e];
    }
  }
  const float inv = 1.f / wsum;
  uint32_t pk[4];
#pragma unroll
  for (int e = 0; e < 4; ++e)
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk[e]) : "f"(o[2 * e + 1] * inv), "f"(o[2 * e] * inv));
  lse2 = mx + log2f(wsum);
  return make_uint4(pk[0], pk[1], pk[2], pk[3]);
}

// OPT: the softmax warps skip the search for the row maximum after an item's first tile (see there); chosen by the
// host for batches whose sequences are long, where nearly every step is such a step.
// FAN: the fan-out mode (TcArgs::mode 2); the other modes are compiled without the walk over the children's tiles.
// SCHED: who takes which items (see kSchedList).
template <int D, bool OPT, bool FAN, int SCHED>
__global__ void __launch_bounds__(kTcThreads, 1) attn_extend_tc_kernel(const TcArgs a, const __grid_constant__ CUtensorMap q_map) {
  using Cfg = TcCfg<D>;
  constexpr bool SPAN = SCHED == kSchedSpans, CLUSTER = SCHED == kSchedCluster;
  constexpr bool REC = SPAN || CLUSTER;  // the scheduler warp announces whole records
  extern __shared__ unsigned char smem_raw[];
  // Dynamic shared memory starts on a 1024-byte boundary (this kernel has no static shared memory); the swizzled
  // operand tiles need that.  Checked instead of padded for: the tiles leave no room for padding.
  if ((smem_u32(smem_raw) & 1023u) != 0) {
    if (threadIdx.x == 0) report(a.pool.status, KV_ERR_CUDA);
    return;
  }
  // The mixed step's decode kernel, queued behind this one with the early-start attribute, may take the SMs this grid leaves free as
  // soon as every CTA of this grid is resident.  Any other kernel is let in at the end of the producer's work.
  if (a.beside) launch_dependents();
  TcSmem<D>& sm = *reinterpret_cast<TcSmem<D>*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  volatile int* abortp = &sm.abort_flag;

  if (tid == 0) {
    sm.abort_flag = 0;
    for (int s = 0; s < Cfg::kStages; ++s) {
      mbar_init(smem_u32(&sm.kv_full[s]), 1);
      mbar_init(smem_u32(&sm.kv_empty[s]), 1);
    }
    for (int s4 = 0; s4 < 4; ++s4) {
      mbar_init(smem_u32(&sm.sched_full[s4]), 1);    // the producer wrote the slot
      mbar_init(smem_u32(&sm.sched_empty[s4]), REC ? 15 : 14);  // MMA warp, Q loader, 8 softmax and 4 epilogue warps (and the producer) have read it
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(smem_u32(&sm.q_full[t]), 1);    // the Q tile's bytes have landed (transaction count)
      mbar_init(smem_u32(&sm.q_empty[t]), 1);   // tensor core finished the item's last S: the Q buffer may be refilled
      mbar_init(smem_u32(&sm.s_full[t]), 1);    // tensor core finished S (and everything issued before it)
      mbar_init(smem_u32(&sm.p_full[t]), 128);  // every softmax thread wrote its row of P
      mbar_init(smem_u32(&sm.o_full[t]), 1);    // tensor core finished the item's last PV
      mbar_init(smem_u32(&sm.o_empty[t]), 128); // every epilogue thread has read its row of O: the next item may overwrite it
      mbar_init(smem_u32(&sm.l_full[t]), 128);  // every softmax thread has published 1 / row sum
    }
    fence_mbar_init();
  }
  if (warp == kWarpProducer) {
    tmem_alloc(smem_u32(&sm.tmem_base), 512);
    tmem_relinquish();
  }
  int cl_P = 0, cl_E = 0, cl_row0 = 0;
  if (CLUSTER && warp == kWarpSched) {  // the item's lengths are asked for while the CTA is set up
    const int seq = (int)blockIdx.x / a.cl_splits / a.pool.n_kv_heads / a.span.max_tp;
    if (!a.span.plan_early) dependency_wait();
    cl_P = ptx::ld_plain(a.prefix_lens + seq);
    if (FAN) {  // a parent's rows are those of its children
      cl_row0 = ptx::ld_plain(a.fan.cu_q + ptx::ld_plain(a.fan.cu_children + seq));
      cl_E = ptx::ld_plain(a.fan.cu_q + ptx::ld_plain(a.fan.cu_children + seq + 1)) - cl_row0;
    } else {
      cl_E = ptx::ld_plain(a.extend_lens + seq);
      cl_row0 = ptx::ld_plain(a.cu_q + seq);
    }
    for (int b = lane * 32; b < a.max_pages; b += 1024) prefetch_l2(a.block_tables + (int64_t)seq * a.max_pages + b);
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = sm.tmem_base;
  // Everything up to here touched only this CTA's own shared and tensor memory and may have run while the kernel in
  // front of this one (the plan, or the plan and the suffix append) was still at work; its results are needed now.
  // (Behind this call's own append, which has waited for all that came before it: lengths, tables and Q may be read at
  // once, so the scheduler, the Q loader and the producer do not wait here; the producer does before its first K/V copy.)
  const bool reads_early = REC && a.span.plan_early;
  if (!reads_early || (warp != kWarpSched && warp != kWarpQ && warp != kWarpProducer)) dependency_wait();
  const int n_total = REC ? 0 : __ldcg(a.n_items) * a.pool.n_kv_heads;
  const int Hkv = a.pool.n_kv_heads;
  // Round r of this CTA works on item sched_get(r) of the global list (>= n_total: no more work).  A warp
  // calls sched_release(r) once it no longer needs the slot.
  auto sched_get = [&](int round) -> int {
    const bool got = mbar_wait(smem_u32(&sm.sched_full[round & 3]), (round >> 2) & 1, abortp);
    const int idx = *reinterpret_cast<volatile int*>(&sm.sched_idx[round & 3]);
    return got ? idx : 0x7fffffff;
  };
  auto sched_release = [&](int round) {
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&sm.sched_empty[round & 3]));
  };
  // The item of a round; false: no more work.
  auto fetch = [&](int round, Item& it) -> bool {
    if constexpr (REC) {
      if (!mbar_wait(smem_u32(&sm.sched_full[round & 3]), (round >> 2) & 1, abortp)) return false;
      const int4 r0 = sm.sched_rec[round & 3][0], r1 = sm.sched_rec[round & 3][1], r2 = sm.sched_rec[round & 3][2];
      it.seq = r0.x; it.kvh = r0.y; it.tp = r0.z; it.P = r0.w;
      it.E = r1.x; it.row0 = r1.y; it.n_kv[0] = r1.z; it.n_kv[1] = r1.w;
      it.kv_end = r2.x; it.first_tile = r2.y; it.part = r2.z;
      it.c_first = FAN ? r2.w : 0;
      it.ld_tiles = max(it.n_kv[0], it.n_kv[1]);
      return it.seq >= 0;
    } else {
      it.first_tile = 0;
      it.part = -1;
      return fetch_item<FAN>(a, sched_get(round), n_total, it);
    }
  };

  if (warp == kWarpProducer) {
    // =============================== producer =============================================
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    const char* kpool = reinterpret_cast<const char*>(a.pool.k);
    const char* vpool = reinterpret_cast<const char*>(a.pool.v);
    uint32_t loads = 0;  // stage loads issued so far (ring position)
    bool ok = true, wait_first = reads_early;
    // Announces item idx as round r (waits until every reader is done with the slot's previous round).
    auto announce = [&](int r, int idx) {
      if (lane == 0) {
        ok = mbar_wait(smem_u32(&sm.sched_empty[r & 3]), ((r >> 2) & 1) ^ 1, abortp);
        *reinterpret_cast<volatile int*>(&sm.sched_idx[r & 3]) = idx;
        mbar_arrive(smem_u32(&sm.sched_full[r & 3]));
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
    };
    int cur = blockIdx.x;
    if constexpr (!REC) announce(0, cur);
    for (int round = 0; ok && (REC || cur < n_total); ++round) {
      Item it;
      if constexpr (REC) {
        if (!fetch(round, it)) break;
        sched_release(round);
      } else {
        // The next item is taken and announced one item ahead, so that nobody waits for the counter.  (Taking it
        // two items ahead would hide the counter's latency from this warp too, but an item that is committed early
        // cannot go to a CTA that runs out of work: measured slower.)
        int nxt_idx = 0;
        if (lane == 0) nxt_idx = atomicAdd(a.next_item, 1);
        nxt_idx = __shfl_sync(0xffffffffu, nxt_idx, 0);
        announce(round + 1, nxt_idx);
        fetch_item<FAN>(a, cur, n_total, it);
        cur = nxt_idx;
      }
      if (!ok) break;
      const int* bt = a.block_tables + (int64_t)it.seq * a.max_pages + (REC ? it.first_tile * 8 : 0);
      const size_t head_off = (size_t)it.kvh * Cfg::kBlockBytes;
      const int n_own = FAN ? (it.P + kPageSize - 1) / kPageSize : 0;  // fan-out mode: the parent's pages
      int child = it.c_first, child_at = n_own;                        // this lane's child and its first page in the list
      for (int j = 0; j < it.ld_tiles && ok; ++j) {
        const int np = min(8, (it.kv_end - j * 128 + 15) >> 4);
        int page = 0;
        const int* src_bt = bt + j * 8;
        const int g = (j + (REC ? it.first_tile : 0)) * 8 + lane;
        if (FAN && lane < np && g >= n_own) {
          while (true) {
            const int pages = (ptx::ld_plain(a.fan.cu_q + child + 1) - ptx::ld_plain(a.fan.cu_q + child) + kPageSize - 1) / kPageSize;
            if (g < child_at + pages || child + 1 >= a.fan.n_children) break;
            child_at += pages;
            ++child;
          }
          src_bt = a.fan.tables + (int64_t)child * a.fan.max_pages + (g - child_at) - lane;
        }
        if (lane < np) {
          page = ptx::ld_plain(src_bt + lane);
          if ((unsigned)page >= (unsigned)a.pool.num_pages) {
            report(a.pool.status, KV_ERR_BOUNDS);
            page = 0;
          }
        }
        const size_t src_off = ((size_t)page * Hkv) * Cfg::kBlockBytes + head_off;
        if (REC && wait_first) {
          dependency_wait();
          wait_first = false;
        }
#pragma unroll
        for (int which = 0; which < 2; ++which) {  // 0: K tile, 1: V tile
          const uint32_t s = loads % Cfg::kStages, par = (loads / Cfg::kStages) & 1;
          const uint32_t full = smem_u32(&sm.kv_full[s]);
          if (lane == 0) {
            ok = mbar_wait(smem_u32(&sm.kv_empty[s]), par ^ 1, abortp);
            if (ok) mbar_arrive_expect_tx(full, (uint32_t)np * Cfg::kBlockBytes);
          }
          ok = __shfl_sync(0xffffffffu, ok, 0);
          if (!ok) break;
          if (lane < np)
            bulk_g2s(smem_u32(sm.kv[s]) + lane * Cfg::kBlockBytes, (which ? vpool : kpool) + src_off, Cfg::kBlockBytes,
                     full);
          ++loads;
        }
      }
    }
    // The kernel behind this one is let in when no CTA has copies left to ask for: its launch is hidden all the same, and its blocks
    // do not sit waiting on the SMs that are done while a CTA of another stream, which needs a whole SM, could run there.
    // Two streams of calls that append and extend, us for a call of each (it was let in at the start -> now): 20 sequences of 29
    // tokens behind 850, 16/4 heads, 39.0 -> 31.3; 14 of 58 behind 950, 32/8 heads, 47.4 -> 38.6.  Calls behind one another: 4 layers
    // of 9 sequences 158.8 -> 156.6, 1 sequence of 37 tokens 13.79 -> 13.66.  (At the last item of a list instead: 64 sequences of
    // 64-256 tokens 255.9 -> 259.5.)
    if (!a.beside) launch_dependents();
    if (!ok && lane == 0) {
      // give copies that were already issued time to land before the CTA's shared memory goes away
      const uint32_t first = loads > (uint32_t)Cfg::kStages ? loads - Cfg::kStages : 0;
      for (uint32_t i = first; i < loads; ++i) {
        const uint32_t s = i % Cfg::kStages, par = (i / Cfg::kStages) & 1;
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(smem_u32(&sm.kv_full[s]), par) && globaltimer_ns() - t0 < 100000000ull) {
        }
      }
    }
  } else if (warp == kWarpMma) {
    // =============================== MMA issuer ===========================================
    // One thread issues every MMA of the CTA.  Per KV tile j and query tile t:  O_t (+)= P_t V(j) as soon as
    // the softmax warps have written P_t, then S_t = Q_t K(j+1)^T into the columns P_t occupied (the tensor
    // core runs MMAs in issue order), so the other tile's MMAs fill the time this tile's softmax takes.
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    // Low descriptor words.  The address field takes 14 bits: in a cluster the upper bits of a shared address name the CTA.
    auto lo_word = [](const void* p, uint32_t lbo) { return ((smem_u32(p) >> 4) & 0x3FFFu) | ((lbo >> 4) << 16); };
    const uint32_t q_lo0 = lo_word(sm.q[0], 16), k_lo0 = lo_word(sm.kv[0], 16);
    const uint32_t v_lo0 = lo_word(sm.kv[0], 1024);  // V tiles: LBO = 64-dim half
    const uint32_t bar_s_full = smem_u32(&sm.s_full[0]), bar_p_full = smem_u32(&sm.p_full[0]);
    const uint32_t bar_q_full = smem_u32(&sm.q_full[0]), bar_o_full = smem_u32(&sm.o_full[0]);
    const uint32_t bar_q_empty = smem_u32(&sm.q_empty[0]), bar_o_empty = smem_u32(&sm.o_empty[0]);
    uint32_t o_uses[2] = {0, 0};        // items per tile whose PV has started (phase of o_empty)
    bool early0 = false;                // tile 0's first S of the coming item has been issued already
    uint32_t loads = 0;                 // ring position, mirrors the producer
    uint32_t steps[2] = {0, 0};         // softmax steps per tile so far (phase of p_full)
    uint32_t items_done[2] = {0, 0};    // items per tile so far (phase of q_full)
    bool ok = true;
    Item nxt;
    bool has_nxt = fetch(0, nxt);
    for (int round = 0; ok && has_nxt; ++round) {
      const Item it = nxt;
      has_nxt = fetch(round + 1, nxt);
      sched_release(round);
      if (it.ld_tiles == 0) continue;
      {
        // The whole warp runs this control flow (all values are warp-uniform); one elected lane issues.
        // first K tile: S(0) of each query tile as soon as its Q tile is in shared memory
        uint32_t stage = loads % Cfg::kStages;
        ok = mbar_wait(smem_u32(&sm.kv_full[stage]), (loads / Cfg::kStages) & 1, abortp);
        ++loads;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          if (!ok || it.n_kv[t] == 0) continue;
          if (t == 0 && early0) {
            early0 = false;
            continue;
          }
          ok = mbar_wait(bar_q_full + 8 * t, items_done[t] & 1, abortp);
          ++items_done[t];
          if (!ok) continue;
          if (elect_one_sync()) {
            issue_s_mmas<D>(tmem + t * 128, q_lo0 + t * (Cfg::kTileBytes >> 4), k_lo0 + stage * (Cfg::kTileBytes >> 4));
            mma_commit(bar_s_full + 8 * t);
            if (it.n_kv[t] == 1) mma_commit(bar_q_empty + 8 * t);
          }
          __syncwarp();
        }
        if (ok && elect_one_sync()) mma_commit(smem_u32(&sm.kv_empty[stage]));
        __syncwarp();
        for (int j = 0; j < it.ld_tiles && ok; ++j) {
          const int np = min(8, (it.kv_end - j * 128 + 15) >> 4);
          const uint32_t v_stage = loads % Cfg::kStages;
          ok = mbar_wait(smem_u32(&sm.kv_full[v_stage]), (loads / Cfg::kStages) & 1, abortp);
          ++loads;
          if (!ok) break;
          const bool more = j + 1 < it.ld_tiles;
          uint32_t k_stage = 0;
          if (more) {
            k_stage = loads % Cfg::kStages;
            ok = mbar_wait(smem_u32(&sm.kv_full[k_stage]), (loads / Cfg::kStages) & 1, abortp);
            ++loads;
            if (!ok) break;
          }
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            if (j >= it.n_kv[t]) continue;
            ok = mbar_wait(bar_p_full + 8 * t, steps[t] & 1, abortp);
            ++steps[t];
            if (ok && j == 0) {  // the first PV overwrites O: the previous item's rows must have been read out
              ok = mbar_wait(bar_o_empty + 8 * t, (o_uses[t] & 1) ^ 1, abortp);
              ++o_uses[t];
            }
            if (!ok) break;
            tc_fence_after_sync();
            if (elect_one_sync()) {
              issue_pv_mmas<D>(tmem + 256 + t * 128, tmem + t * 128, v_lo0 + v_stage * (Cfg::kTileBytes >> 4), np, j == 0);
              if (j + 1 < it.n_kv[t]) {
                issue_s_mmas<D>(tmem + t * 128, q_lo0 + t * (Cfg::kTileBytes >> 4), k_lo0 + k_stage * (Cfg::kTileBytes >> 4));
                mma_commit(bar_s_full + 8 * t);
                if (j + 2 == it.n_kv[t]) mma_commit(bar_q_empty + 8 * t);  // that was the item's last S of this tile
              } else {
                mma_commit(bar_o_full + 8 * t);
              }
            }
            __syncwarp();
            if (t == 0 && j + 1 == it.n_kv[0] && has_nxt && nxt.n_kv[0] > 0 && nxt.ld_tiles > 0) {
              // Tile 0 is done with this item while tile 1 still has a step or more to go: if the next item's Q
              // tile and first K tile are already there, its first S is issued now instead of after tile 1.
              const uint32_t k0 = loads + (more ? 0 : 0) + 2 * (uint32_t)(it.ld_tiles - 1 - j) - (more ? 1 : 0);
              const uint32_t st0 = k0 % Cfg::kStages;
              // (A stage's barrier may only be asked about load k0 once the stage's previous load, k0 - kStages, has
              // been waited for: otherwise the parity test would be answered by the phase before that one.  In the
              // fan-out mode tile 1 can have several steps more than tile 0, which puts k0 that far ahead.)
              if (k0 < loads + Cfg::kStages &&
                  __all_sync(0xffffffffu, mbar_test_wait(bar_q_full, items_done[0] & 1) &&
                                              mbar_test_wait(smem_u32(&sm.kv_full[st0]), (k0 / Cfg::kStages) & 1))) {
                ++items_done[0];
                early0 = true;
                if (elect_one_sync()) {
                  issue_s_mmas<D>(tmem, q_lo0, k_lo0 + st0 * (Cfg::kTileBytes >> 4));
                  mma_commit(bar_s_full);
                  if (nxt.n_kv[0] == 1) mma_commit(bar_q_empty);
                }
                __syncwarp();
              }
            }
          }
          if (!ok) break;
          if (elect_one_sync()) {
            mma_commit(smem_u32(&sm.kv_empty[v_stage]));
            if (more) mma_commit(smem_u32(&sm.kv_empty[k_stage]));
          }
          __syncwarp();
        }
      }
      ok = __all_sync(0xffffffffu, ok);
    }
  } else if (warp == kWarpQ) {
    // =============================== Q loader ============================================
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    uint32_t fills[2] = {0, 0};  // tiles loaded so far per buffer (phase of q_empty)
    bool ok = true;
    Item it;
    for (int round = 0; ok && fetch(round, it); ++round) {
      sched_release(round);
      if (it.ld_tiles == 0) continue;
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        if (it.n_kv[t] == 0 || !ok) continue;
        if (lane == 0) {
          // the buffer is free once the previous item's last S of this tile has been computed
          ok = mbar_wait(smem_u32(&sm.q_empty[t]), (fills[t] & 1) ^ 1, abortp);
          if (ok) {
            const uint32_t full = smem_u32(&sm.q_full[t]);
            mbar_arrive_expect_tx(full, Cfg::kTileBytes);
            const int tok0 = it.row0 + ((it.tp * 256 + t * 128) >> a.lg_group);
#pragma unroll
            for (int h = 0; h < Cfg::kHalves; ++h)
              tma_load_3d(smem_u32(sm.q[t]) + h * Cfg::kQHalfStride, &q_map, h * 64, it.kvh * a.group, tok0, full);
          }
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        ++fills[t];
      }
      // the next item's query tiles are asked into L2 now, a whole item ahead of their copy to shared memory
      Item nx;
      if (fetch(round + 1, nx) && nx.ld_tiles > 0 && lane == 0) {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          if (nx.n_kv[t] == 0) continue;
          const int tok0 = nx.row0 + ((nx.tp * 256 + t * 128) >> a.lg_group);
#pragma unroll
          for (int h = 0; h < Cfg::kHalves; ++h) tma_prefetch_3d(&q_map, h * 64, nx.kvh * a.group, tok0);
        }
      }
    }
  } else if (warp == kWarpSched) {
    if constexpr (!REC) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 24;");  // idle warp
    } else if constexpr (CLUSTER) {
      // =============================== scheduler (one item per cluster) =======================
      asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
      const int lg = a.lg_group, splits = a.cl_splits;
      const int unit = (int)blockIdx.x / splits, rank = (int)blockIdx.x - unit * splits;
      const int rest = unit / Hkv, kvh = unit - rest * Hkv, seq = rest / a.span.max_tp, tp = rest - seq * a.span.max_tp;
      const int P = cl_P, E = cl_E, row0 = cl_row0;
      const int rows = span_rows(a, P, E, row0), pairs = span_pairs(rows, lg);
      if (lane == 0) {
        if (tp == 0 && kvh == 0 && rank == 0 && P >= 0 && rows < E) report(a.pool.status, KV_ERR_BOUNDS);
        int n = 0, n0 = 0, n1 = 0, kv_end = 0, first_child = 0;
        if (tp < pairs) {
          const ItemRec r = make_item(seq, tp, P, rows, row0, lg, a.max_pages, a.mode, a.fan);
          n0 = r.n_kv0;
          n1 = r.n_kv1;
          n = max(n0, n1);
          first_child = r.kv_end;
          kv_end = FAN ? ((n - 1) * 8 + (int)((unsigned)r.tp >> 28) + 1) * kPageSize : r.kv_end;
          if (n == 0) report(a.pool.status, KV_ERR_BOUNDS);
        }
        const int off = n * rank / splits, end = n * (rank + 1) / splits;
        sm.cl_unit = make_int4(n > 0 ? min(256, (rows << lg) - tp * 256) : 0, row0, tp, kvh);
        int round = 0;
        if (end > off) {
          sm.sched_rec[0][0] = make_int4(seq, kvh, tp, FAN ? P : P - off * 128);
          sm.sched_rec[0][1] = make_int4(rows, row0, max(0, min(n0, end) - off), max(0, min(n1, end) - off));
          sm.sched_rec[0][2] = make_int4(kv_end - off * 128, off, -1, first_child);
          mbar_arrive(smem_u32(&sm.sched_full[0]));
          round = 1;
        }
        sm.sched_rec[round][0] = make_int4(-1, 0, 0, 0);
        sm.sched_rec[round][1] = sm.sched_rec[round][2] = make_int4(0, 0, 0, 0);
        mbar_arrive(smem_u32(&sm.sched_full[round]));
      }
    } else {
      // =============================== scheduler (span scheduling) ============================
      // Walks the items from the start of the CTA's first span to the end of its last and announces their chunks.
      // (Every lane walks; lane 0 writes.)
      asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
      const int lg = a.lg_group;
      SpanPos pos;
      int total, round = 0, span = (int)blockIdx.x * a.span.per_cta;
      SpanSeqs q;
      span_locate(a, span, pos, total, q);
      const int n_spans = span_count(a.span, total);
      const int span_end = min(span + a.span.per_cta, n_spans);
      bool ok = true;
      auto announce = [&](const SpanRec& r) {
        if (lane == 0) {
          ok = mbar_wait(smem_u32(&sm.sched_empty[round & 3]), ((round >> 2) & 1) ^ 1, abortp);
          sm.sched_rec[round & 3][0] = make_int4(r.seq, r.kvh, r.tp, r.P);
          sm.sched_rec[round & 3][1] = make_int4(r.E, r.row0, r.n_kv0, r.n_kv1);
          sm.sched_rec[round & 3][2] = make_int4(r.kv_end, r.first_tile, r.part, 0);
          mbar_arrive(smem_u32(&sm.sched_full[round & 3]));
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        ++round;
      };
      // spans that the batch has no work for leave no cut behind
      for (int s = max(span, span_end); s < min(((int)blockIdx.x + 1) * a.span.per_cta, a.span.n_spans); ++s)
        if (lane == 0) a.span.desc[3 * s] = make_int4(-1, 0, 0, 0);
      bool fresh = true;  // the start of the first span has not been moved to an item's edge yet
      if (span < span_end) {
        int off = pos.off;
        auto cut_at = [&](int s) { return s >= n_spans ? total : span_cut(total, n_spans, s); };
        for (int seq = pos.seq; seq < a.batch && span < span_end && ok; ++seq) {
          if (seq >= q.base + 32) span_load(a, seq, q);
          const int l = seq - q.base;
          const int P = __shfl_sync(0xffffffffu, q.P, l), row0 = __shfl_sync(0xffffffffu, q.row0, l);
          const int rows = __shfl_sync(0xffffffffu, q.rows, l), pairs = span_pairs(rows, lg);
          int kvh = seq == pos.seq ? pos.kvh : 0, tp = seq == pos.seq ? pos.tp : 0;
          for (; kvh < Hkv && pairs > 0 && span < span_end && ok; ++kvh, tp = 0) {
            for (; tp < pairs && span < span_end && ok; ++tp) {
              const int n = span_steps(P, rows, tp, lg);
              const int tok_1 = (tp * 256 + 128) >> lg;  // first token of the second tile
              const int hi0 = min(rows, tok_1), hi1 = tok_1 < rows ? min(rows, ((tp + 1) * 256) >> lg) : 0;
              const int n0 = (P + hi0 + 127) >> 7, n1 = hi1 > 0 ? (P + hi1 + 127) >> 7 : 0;
              auto put_cut = [&]() {
                if (lane == 0) {
                  a.span.desc[3 * span] = make_int4(off > 0 && off < n ? pos.at : -1, off, kvh, tp);
                  a.span.desc[3 * span + 1] = make_int4(rows, row0, n0, n1);
                }
              };
              if (fresh) {
                fresh = false;
                off = span_snap(a.span, off, n);
                put_cut();
              }
              // the chunks of this item, one per span
              while (off < n && span < span_end && ok) {
                const int raw = cut_at(span + 1) - pos.at;  // where the span ends, counted from the item's first step
                const int end = raw >= n ? n : raw <= 0 ? 0 : span_snap(a.span, raw, n);
                if (end > off) {
                  const int part = off > 0 ? 2 * span : end < n ? 2 * span + 1 : -1;
                  announce(SpanRec{seq, kvh, tp, P - off * 128, rows, row0, max(0, min(n0, end) - off), max(0, min(n1, end) - off),
                                   P + max(hi0, hi1) - off * 128, off, part});
                  off = end;
                }
                if (raw <= n && (raw < n || off == n)) {  // the span ends in (or with) this item
                  ++span;
                  if (span < span_end) put_cut();
                }
              }
              pos.at += n;
              off = 0;
            }
          }
        }
      }
      for (int s = span + (fresh ? 0 : 1); s < span_end; ++s)  // empty spans at the end of the line
        if (lane == 0) a.span.desc[3 * s] = make_int4(-1, 0, 0, 0);
      announce(SpanRec{-1, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0});
    }
  } else if (warp >= kWarpEpilogue) {
    // =============================== epilogue warpgroup ====================================
    // One thread per row (= TMEM lane), both tiles in turn: O / l -> bf16 -> global.
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    const int w4 = warp & 3;
    const int m = w4 * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(w4 * 32) << 16);
    const int G = a.group, lg = a.lg_group, Hq = a.n_q_heads;
    uint32_t done0 = 0, done1 = 0;  // items finished per tile (phase of o_full / l_full, parity of inv_l)
    bool ok = true;
    Item it;
    for (int round = 0; ok && fetch(round, it); ++round) {
      sched_release(round);
      if (CLUSTER && a.cl_splits > 1) {
        // The softmax warps hand the partial results over; the second half of the first tile's dims is left to these warps
        // (one sequence of 37 tokens, 128 of its 148 rows in that tile: 14.39 -> 14.16 us).
        if (it.n_kv[0] == 0) continue;
        ok = mbar_wait(smem_u32(&sm.o_full[0]), 0, abortp);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after_sync();
        float* dst = a.span.part_o + (((int64_t)blockIdx.x * (D / 8) + D / 16) * a.span.rows + m) * 8;
#pragma unroll 1
        for (int c = D / 64; c < D / 32; ++c, dst += (int64_t)a.span.rows * 32) {
          uint32_t orow[32];
          tmem_ld32(lane_base + 256 + c * 32, orow);
          tmem_wait_ld();
          if (m < sm.cl_unit.x) store_part8x4(dst, a.span.rows, orow);
        }
        continue;
      }
      if (it.ld_tiles == 0) continue;
#pragma unroll 1
      for (int t = 0; t < 2; ++t) {
        if ((t ? it.n_kv[1] : it.n_kv[0]) == 0 || !ok) continue;
        const int rg = it.tp * 256 + t * 128 + m;
        const int tok = rg >> lg;
        const bool valid = tok < it.E;
        const int64_t orow_idx = (int64_t)(it.row0 + tok) * Hq + it.kvh * G + (rg & (G - 1));
        const uint32_t par = (t ? done1 : done0) & 1;
        ok = mbar_wait(smem_u32(&sm.l_full[t]), par, abortp);
        if (ok) ok = mbar_wait(smem_u32(&sm.o_full[t]), par, abortp);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after_sync();
        const float inv = sm.inv_l[t][par][m];
        if (t) ++done1; else ++done0;
        const uint32_t o_addr = lane_base + 256 + t * 128;
        // A row is 2 * D contiguous bytes, but a warp holds 32 different rows: 16-byte stores from the thread
        // that owns the row touch 32 cache lines per instruction and half a sector each.  Instead two
        // neighbouring lanes exchange 32-byte pieces, so that every store instruction writes 64 contiguous
        // bytes per lane pair, in 32-byte (whole sector) pieces.
        const int q = lane & 1;
        char* row_ptr = reinterpret_cast<char*>(a.out + orow_idx * D);
        // the neighbour's row and whether it exists
        const uint32_t n_lo = __shfl_xor_sync(0xffffffffu, (uint32_t)reinterpret_cast<uintptr_t>(row_ptr), 1);
        const uint32_t n_hi = __shfl_xor_sync(0xffffffffu, (uint32_t)(reinterpret_cast<uintptr_t>(row_ptr) >> 32), 1);
        char* nb_ptr = reinterpret_cast<char*>(((uint64_t)n_hi << 32) | n_lo);
        const bool nb_valid = __shfl_xor_sync(0xffffffffu, (int)valid, 1) != 0;
#pragma unroll 1
        for (int c = 0; c < D / 32; ++c) {
          uint32_t orow[32];
          tmem_ld32(o_addr + c * 32, orow);
          tmem_wait_ld();
          if (c == D / 32 - 1) {  // all of the row has been read: the next item's PV may overwrite O
            tc_fence_before_sync();
            mbar_arrive(smem_u32(&sm.o_empty[t]));
          }
          if (SPAN && it.part >= 0) {  // a chunk of a cut item: its rows stay in fp32 until the chunks are merged
            if (valid) {
              store_part8x4(a.span.part_o + (((int64_t)it.part * (D / 8) + c * 4) * a.span.rows + t * 128 + m) * 8, a.span.rows, orow, inv);
            }
            continue;
          }
          uint32_t pk[16];  // columns [32c, 32c + 32) as bf16 pairs: two pieces of eight words
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float lo = __uint_as_float(orow[2 * i]) * inv, hi = __uint_as_float(orow[2 * i + 1]) * inv;
            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk[i]) : "f"(hi), "f"(lo));
          }
          // piece q of the own row is stored by this lane, piece 1-q by the neighbour, and vice versa
          uint32_t w[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint32_t give = q == 0 ? pk[8 + i] : pk[i];
            w[i] = __shfl_xor_sync(0xffffffffu, give, 1);
          }
          // first store: the even lane's row (its own piece 0, and piece 1 handed to the odd lane);
          // second store: the odd lane's row
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const bool own = (q == r);
            if (own ? valid : nb_valid) {
              char* dst = (own ? row_ptr : nb_ptr) + c * 64 + q * 32;
              uint32_t d[8];
#pragma unroll
              for (int i = 0; i < 8; ++i) d[i] = own ? (r == 0 ? pk[i] : pk[8 + i]) : w[i];
              asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(dst), "r"(d[0]), "r"(d[1]), "r"(d[2]), "r"(d[3]),
                           "r"(d[4]), "r"(d[5]), "r"(d[6]), "r"(d[7])
                           : "memory");
            }
          }
        }
      }
    }
  } else {
    // =============================== softmax warpgroups ======================================
    asm volatile("setmaxnreg.inc.sync.aligned.u32 192;");
    const int t = warp >> 2;                       // query tile of this warpgroup (warps 0-3: tile 0, 4-7: tile 1)
    const int w4 = warp & 3;                       // TMEM lane quarter this warp may access
    const int m = w4 * 32 + lane;                  // row inside the tile
    const uint32_t lane_base = tmem + ((uint32_t)(w4 * 32) << 16);
    const uint32_t s_addr = lane_base + t * 128, o_addr = lane_base + 256 + t * 128;
    const uint32_t bar_s_full = smem_u32(&sm.s_full[t]), bar_l_full = smem_u32(&sm.l_full[t]);
    const uint32_t bar_p_full = smem_u32(&sm.p_full[t]);
    const int G = a.group, lg = a.lg_group, Hq = a.n_q_heads;
    uint32_t steps = 0, items_done = 0;            // phase of s_full / p_full; items finished (parity of inv_l)
    bool ok = true;
    float cl_m = -INFINITY, cl_l = 0.f;            // cluster: the row's maximum and sum over this CTA's part

    // The item records are read where they are needed (they stay in L1) instead of being carried in registers
    // through the softmax loop, which needs the registers for the score row.
    for (int round = 0; ok; ++round) {
      int n_t, limit, part = -1;
      bool valid;
      int64_t orow_idx;
      int f_lo = 0, f_hi = 0;  // fan-out mode: this row's child's own keys that it sees, among the slots of the item's pages
      {
        Item it;
        const bool more_items = fetch(round, it);
        if (!more_items) break;
        sched_release(round);
        if (it.ld_tiles == 0) continue;
        n_t = it.n_kv[t];
        if (n_t == 0) continue;
        const int rg = it.tp * 256 + t * 128 + m;
        const int tok = rg >> lg;
        valid = tok < it.E;
        // keys this row sees (rows past the end: any); fan-out mode: the parent's
        limit = FAN ? it.P - it.first_tile * 128 : valid && a.mode == 0 ? it.P + tok + 1 : it.kv_end;
        orow_idx = (int64_t)(it.row0 + tok) * Hq + it.kvh * G + (rg & (G - 1));  // row of the LSE
        if (SPAN) part = it.part;
        if (FAN && valid) {
          int c = it.c_first, r0 = ptx::ld_plain(a.fan.cu_q + c) - it.row0, r1 = ptx::ld_plain(a.fan.cu_q + c + 1) - it.row0;
          f_lo = (it.P + kPageSize - 1) / kPageSize * kPageSize - it.first_tile * 128;
          while (tok >= r1 && c + 1 < a.fan.n_children) {
            f_lo += (r1 - r0 + kPageSize - 1) / kPageSize * kPageSize;
            ++c;
            r0 = r1;
            r1 = ptx::ld_plain(a.fan.cu_q + c + 1) - it.row0;
          }
          f_hi = f_lo + tok - r0 + 1;
        }
      }
      float m_run = -INFINITY, l_run = 0.f;

      for (int j = 0; j < n_t; ++j) {
        ok = mbar_wait(bar_s_full, steps & 1, abortp);
        ++steps;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after_sync();
        // One trip to tensor memory: the row's 128 scores are read into registers, reduced to the row
        // maximum, exponentiated in place and written back as bf16 P.
        // vis: how many of the tile's 128 key columns this row sees (diagonal / last tile: keys past the row's
        // limit are hidden); fan-out mode: also the columns lo .. hi - 1, its own child's keys up to its own token
        const int vis = limit - j * 128, lo = f_lo - j * 128, hi = f_hi - j * 128;
        const bool ragged = vis < 128;
        uint32_t sr[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(s_addr + c * 32, sr[c]);
        tmem_wait_ld();
        if (ragged) {
#pragma unroll
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (c * 32 + i >= vis && (!FAN || c * 32 + i < lo || c * 32 + i >= hi)) sr[c][i] = 0xff800000u;  // -inf by select: NaN-safe
        }
        if constexpr (OPT) {
          // The row maximum is needed only to keep the exponentials in range, and after the first tile it rarely
          // moves by much: the step first assumes that the maximum in use still serves (no search for the new one) and
          // looks at the row sum it gets.  A sum beyond kOptimisticSum (or not a number) in any row of the warp means
          // some score exceeds the maximum in use by up to 16 or more binades: the warp then takes the step again
          // with the exact maximum.  Both ways are a deterministic function of the inputs.
          // exponentials of the row against a given maximum: P (bf16) goes to tensor memory, the row sum comes back
          auto exp_pass = [&](float m_use) -> float {
            const float neg_m = (m_use == -INFINITY) ? 0.f : -m_use;
            const float2 sc2 = make_float2(a.scale_log2, a.scale_log2), nm2 = make_float2(neg_m, neg_m);
            float2 ls2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              uint32_t pk[16];
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const float2 x = __ffma2_rn(make_float2(__uint_as_float(sr[c][2 * i]), __uint_as_float(sr[c][2 * i + 1])), sc2, nm2);
                float2 pr;
                asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(pr.x) : "f"(x.x));
                asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(pr.y) : "f"(x.y));
                ls2[i & 1] = __fadd2_rn(ls2[i & 1], pr);
                asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk[i]) : "f"(pr.y), "f"(pr.x));
              }
              // P (bf16 pairs) goes over score columns [16c, 16c+16): all scores are in registers by now
              tmem_st16(s_addr + c * 16, pk);
            }
            return (ls2[0].x + ls2[0].y) + (ls2[1].x + ls2[1].y);
          };
          // the exact way: row maximum of the tile, and O and the row sum brought to it if it has grown by much
          auto exact_max = [&]() {
            float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
              for (int i = 0; i < 32; i += 2)
                mx4[c] = fmax3(mx4[c], __uint_as_float(sr[c][i]), __uint_as_float(sr[c][i + 1]));
            const float mx = fmax3(fmaxf(mx4[0], mx4[1]), mx4[2], mx4[3]) * a.scale_log2;
            const float m_new = fmaxf(m_run, mx);
            const bool grow = m_new > m_run + kRescaleThreshold;  // also true on the first tile (m_run = -inf)
            if (j > 0 && __any_sync(0xffffffffu, grow)) {
              // O holds sums scaled by 2^-m_run: bring them to the new maximum (the PV that produced them
              // has finished: the S this step waited for was committed after it)
              const float alpha = grow ? exp2f(m_run - m_new) : 1.f;
              l_run *= alpha;
#pragma unroll 1
              for (int c = 0; c < D / 16; ++c) {
                uint32_t orow[16];
                tmem_ld16(o_addr + c * 16, orow);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 16; ++i) orow[i] = __float_as_uint(__uint_as_float(orow[i]) * alpha);
                tmem_st16(o_addr + c * 16, orow);
              }
            }
            if (grow) m_run = m_new;
          };
          const bool first = j == 0 || __any_sync(0xffffffffu, m_run == -INFINITY);
          if (first) exact_max();
          float row_sum = exp_pass(m_run);
          if (!first && !__all_sync(0xffffffffu, row_sum <= kOptimisticSum)) {  // rare: the maximum has moved a long way
            exact_max();
            row_sum = exp_pass(m_run);
          }
          l_run += row_sum;
        } else {
          float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int i = 0; i < 32; i += 2)
              mx4[c] = fmax3(mx4[c], __uint_as_float(sr[c][i]), __uint_as_float(sr[c][i + 1]));
          const float mx = fmax3(fmaxf(mx4[0], mx4[1]), mx4[2], mx4[3]) * a.scale_log2;
          const float m_new = fmaxf(m_run, mx);
          const bool grow = m_new > m_run + kRescaleThreshold;  // also true on the first tile (m_run = -inf)
          const float m_use = grow ? m_new : m_run;
          if (j > 0 && __any_sync(0xffffffffu, grow)) {
            // O holds sums scaled by 2^-m_run: bring them to the new maximum (the PV that produced them
            // has finished: the S this step waited for was committed after it)
            const float alpha = grow ? exp2f(m_run - m_new) : 1.f;
            l_run *= alpha;
#pragma unroll 1
            for (int c = 0; c < D / 16; ++c) {
              uint32_t orow[16];
              tmem_ld16(o_addr + c * 16, orow);
              tmem_wait_ld();
#pragma unroll
              for (int i = 0; i < 16; ++i) orow[i] = __float_as_uint(__uint_as_float(orow[i]) * alpha);
              tmem_st16(o_addr + c * 16, orow);
            }
          }
          m_run = m_use;
          const float neg_m = (m_use == -INFINITY) ? 0.f : -m_use;
          const float2 sc2 = make_float2(a.scale_log2, a.scale_log2), nm2 = make_float2(neg_m, neg_m);
          float2 ls2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t pk[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float2 x = __ffma2_rn(make_float2(__uint_as_float(sr[c][2 * i]), __uint_as_float(sr[c][2 * i + 1])), sc2, nm2);
              float2 pr;
              asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(pr.x) : "f"(x.x));
              asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(pr.y) : "f"(x.y));
              ls2[i & 1] = __fadd2_rn(ls2[i & 1], pr);
              asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk[i]) : "f"(pr.y), "f"(pr.x));
            }
            // P (bf16 pairs) goes over score columns [16c, 16c+16): all scores are in registers by now
            tmem_st16(s_addr + c * 16, pk);
          }
          l_run += (ls2[0].x + ls2[0].y) + (ls2[1].x + ls2[1].y);
        }
        tmem_wait_st();
        tc_fence_before_sync();
        mbar_arrive(bar_p_full);
      }
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      if (CLUSTER && a.cl_splits > 1) {  // O is final once the last PV is done
        ok = mbar_wait(smem_u32(&sm.o_full[t]), 0, abortp);
        ok = __all_sync(0xffffffffu, ok);
        cl_m = m_run;
        cl_l = l_run;
        continue;
      }
      // ---- hand the row to the epilogue warps: 1 / row sum through shared memory; the LSE is written here.
      // The softmax of an item needs only S, so with one-step items it could finish two items before the
      // epilogue warps have looked at the first: a barrier must not get two phases ahead of its waiters, so
      // this hand-over waits until the previous item's rows of this tile have been read out.
      if (items_done > 0) {
        ok = mbar_wait(smem_u32(&sm.o_empty[t]), (items_done - 1) & 1, abortp);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
      }
      // (A row may see no key of its chunk of a cut item: its sum is exactly 0 and the chunk has weight 0.  A sum that is not a
      // number must reach the result: dropping the chunk would hide a broken key behind plausible values of the others.)
      const bool unseen = SPAN && part >= 0 && l_run == 0.f;
      sm.inv_l[t][items_done & 1][m] = unseen ? 0.f : 1.f / l_run;
      mbar_arrive(bar_l_full);
      ++items_done;
      if (SPAN && part >= 0) {
        if (valid) a.span.part_lse[part * a.span.rows + t * 128 + m] = unseen ? -INFINITY : m_run + log2f(l_run);
      } else if (valid) {
        a.lse[orow_idx] = (m_run + log2f(l_run)) * 0.6931471805599453f;
      }
    }
    if (CLUSTER && a.cl_splits > 1) {
      // The CTAs of the cluster hold partial results of the same rows.  Each writes its own out (the epilogue warps half of the first
      // tile's dims), then finishes an equal share of the rows from everybody's, through L2.  By the SM's clock, us, one sequence of 37
      // tokens behind 1483, 64 CTAs of 76 KB each: 4.3 from the end of the wait for the append to the last PV, 0.75 to write, 2.4 from
      // there to the end of the barrier (the stores, and the slowest CTA), 2.1 to merge; 9 of 64, two CTAs per item: 13.1, 0.7, 3.1 and
      // 3.7.  The merge took 3.6 with two loads of 16 bytes for a piece and the items one after the other where it took 2.4 without,
      // and 3.7 with the weights computed once per row in front (another wait for L2).
      const int splits = a.cl_splits, unit = (int)blockIdx.x / splits, rank = (int)blockIdx.x - unit * splits;
      const int4 u = sm.cl_unit;
      const int row = t * 128 + m;
      if (__any_sync(0xffffffffu, cl_l != 0.f)) {  // (a sum that is not a number is handed over like any other)
        tc_fence_after_sync();
        float* dst = a.span.part_o + ((int64_t)blockIdx.x * (D / 8) * a.span.rows + row) * 8;
#pragma unroll 1
        for (int c = 0; c < (t == 0 ? D / 64 : D / 32); ++c, dst += (int64_t)a.span.rows * 32) {
          uint32_t orow[32];
          tmem_ld32(o_addr + c * 32, orow);
          tmem_wait_ld();
          if (row < u.x) store_part8x4(dst, a.span.rows, orow);
        }
      }
      float2* part_ml = reinterpret_cast<float2*>(a.span.part_lse);  // [CTA][row]: maximum (log2 domain) and sum
      if (row < u.x) part_ml[blockIdx.x * a.span.rows + row] = make_float2(cl_m, cl_l);
      cluster_arrive();
      cluster_wait();
      const int r_begin = u.x * rank / splits, cnt = u.x * (rank + 1) / splits - r_begin;
      auto finish = [&](auto n) {
        // Item i: eight dims of a row; neighbouring lanes take neighbouring rows.  As many items of a thread at a time as make
        // sixteen loads: the wait for L2 is paid once.  From six chunks on one item: the code runs once per launch and is fetched as
        // it runs, so its length counts for as much.  One item / as many as make sixteen loads, us for a call, sequences x tokens behind
        // 1483: 8 chunks 13.80 / 13.76 (1 x 37) and 11.86 / 12.01 (the same, 64 dims), 6 chunks 17.44 / 17.56 (2 x 60), 4 chunks 18.68 /
        // 18.33 (3 x 64), 3 chunks 20.83 / 20.47 (5 x 50), 2 chunks 29.01 / 28.12 (9 x 64).
        constexpr int N = decltype(n)::value, ITEMS = N >= 6 ? 1 : 16 / N;
        const int items = cnt * (D / 8);
        for (int base = tid; base < items; base += 256 * ITEMS) {
          float2 ml[ITEMS][N];
          float x[ITEMS][N][8];
#pragma unroll
          for (int k = 0; k < ITEMS; ++k) {
            const int i = base + 256 * k;
            if (i >= items) break;
            const int g = i / cnt, r = r_begin + (i - g * cnt);
            const float2* src_ml = part_ml + unit * N * a.span.rows + r;
            const float* src = a.span.part_o + (((int64_t)unit * N * (D / 8) + g) * a.span.rows + r) * 8;
#pragma unroll
            for (int c = 0; c < N; ++c, src_ml += a.span.rows, src += (int64_t)a.span.rows * D) {
              ml[k][c] = __ldcg(src_ml);
              load_part8(src, x[k][c]);
            }
          }
#pragma unroll
          for (int k = 0; k < ITEMS; ++k) {
            const int i = base + 256 * k;
            if (i >= items) break;
            const int g = i / cnt, r = r_begin + (i - g * cnt);
            float mx = -INFINITY, sum = 0.f;
#pragma unroll
            for (int c = 0; c < N; ++c) mx = fmaxf(mx, ml[k][c].x);
            float2 o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) o[e] = make_float2(0.f, 0.f);
#pragma unroll
            for (int c = 0; c < N; ++c) {
              if (ml[k][c].y == 0.f) continue;  // (no step of the row's tile, or no key that the row sees: not written)
              // (Its bound for normal results is that of exp2f, whose longer code costs 0.2 to 0.6 us a call.  A weight below 2^-126 is
              // 0, as the probability of such a key is within a chunk.  merge_part8, in a kernel of its own, keeps exp2f.)
              float w;
              asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(w) : "f"(ml[k][c].x - mx));
              sum += w * ml[k][c].y;
#pragma unroll
              for (int e = 0; e < 4; ++e) o[e] = __ffma2_rn(make_float2(x[k][c][2 * e], x[k][c][2 * e + 1]), make_float2(w, w), o[e]);
            }
            const float inv = 1.f / sum;
            uint32_t pk[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk[e]) : "f"(o[e].y * inv), "f"(o[e].x * inv));
            const int rg = u.z * 256 + r;
            const int64_t orow = (int64_t)(u.y + (rg >> lg)) * Hq + u.w * G + (rg & (G - 1));
            reinterpret_cast<uint4*>(a.out + orow * D)[g] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            if (g == 0) a.lse[orow] = (mx + log2f(sum)) * 0.6931471805599453f;
          }
        }
      };
      switch (splits) {
        case 2: finish(std::integral_constant<int, 2>{}); break;
        case 3: finish(std::integral_constant<int, 3>{}); break;
        case 4: finish(std::integral_constant<int, 4>{}); break;
        case 6: finish(std::integral_constant<int, 6>{}); break;
        default: finish(std::integral_constant<int, 8>{});
      }
    }
  }
  if (CLUSTER && a.cl_splits > 1 && warp >= kWarpEpilogue) {  // the other warps' part in the cluster barrier
    cluster_arrive();
    cluster_wait();
  }

  tc_fence_before_sync();
  __syncthreads();
  if (tid == 0 && sm.abort_flag != 0) report(a.pool.status, KV_ERR_TIMEOUT);
  if (warp == kWarpProducer) tmem_dealloc(tmem, 512);
  // The last CTA to finish puts the work counter back where the plan left it, so that the same plan can serve
  // another launch (a model runs every layer of a step over the same lengths).  a.next_item + 1 counts the CTAs done.
  if (!REC && tid == 0) {
    __threadfence();
    if (atomicAdd(a.next_item + 1, 1) == (int)gridDim.x - 1) {
      a.next_item[0] = (int)gridDim.x;
      a.next_item[1] = 0;
      __threadfence();
    }
  }
}

// Merges the chunks of the items that the cuts between the spans went through.  Block (s - 1) * kCombineSlices + slice:
// the item of which cut s is the first, 256 / kCombineSlices of its rows in turns of 32; warp w takes the dims 8w .. 8w + 7,
// its lanes the rows.  Bound by latency and launch (a few MB through L2), so as many blocks as possible, most of which have
// nothing to do, are to be resident: three of 40 registers on an SM at 128 dims (588 blocks of 148 spans: a round and a third).
constexpr int kCombineSlices = 4;
template <int D>
__global__ void __launch_bounds__(D * 4, 384 / D) span_combine_kernel(const SpanArgs a, int n_q_heads, int group, int lg,
                                                                      __nv_bfloat16* out, float* lse) {
  launch_dependents();
  dependency_wait();
  constexpr int kRowWords = D / 2 + 4;  // a row of the result in shared memory, padded
  __shared__ int first_tile[256];
  __shared__ __align__(16) uint32_t rows[32 * kRowWords];
  const int s = 1 + (int)blockIdx.x / kCombineSlices, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // (all loads of the cuts in flight at once)
  const int mine = s + (int)threadIdx.x;
  int dk_at = -1, dk_off = 0;
  if (mine < a.n_spans && threadIdx.x < 255) {
    const int4 dk = __ldcg(a.desc + 3 * mine);
    dk_at = dk.x;
    dk_off = dk.y;
  }
  const int4 d0 = __ldcg(a.desc + 3 * s), d1 = __ldcg(a.desc + 3 * s + 1);
  const int before = __ldcg(a.desc + 3 * (s - 1)).x;
  if (d0.x < 0 || before == d0.x) return;  // no cut, or not the first one of its item
  // chunk 0 is the last of span s - 1, chunk k > 0 the first of span s + k - 1
  const bool same = dk_at == d0.x;
  if (same) first_tile[threadIdx.x + 1] = dk_off;
  if (threadIdx.x == 0) first_tile[0] = 0;
  const int chunks = 1 + __syncthreads_count(same);
  const int kvh = d0.z, tp = d0.w, E = d1.x, row0 = d1.y;
  auto row_of = [&](int mm) {  // row of the result
    const int rg = tp * 256 + mm;
    return (int64_t)(row0 + (rg >> lg)) * n_q_heads + kvh * group + (rg & (group - 1));
  };
  constexpr int kRows = 256 / kCombineSlices;
  for (int m_slice = (int)(blockIdx.x % kCombineSlices) * kRows, turn = 0; turn < kRows / 32; ++turn, m_slice += 32) {
    if (((tp * 256 + m_slice) >> lg) >= E) return;
    const int m = m_slice + lane;
    const int n_t = m < 128 ? d1.z : d1.w;
    const bool valid = ((tp * 256 + m) >> lg) < E;
    float lse2 = 0.f;
    uint4 o = make_uint4(0, 0, 0, 0);
    if (valid)
      o = merge_part8<D, 2>(a, chunks, m, warp, [&](int k) { return k == 0 ? 2 * s - 1 : 2 * (s + k - 1); },
                            [&](int k) { return first_tile[min(k, 255)] < n_t; }, lse2);
    *reinterpret_cast<uint4*>(&rows[lane * kRowWords + warp * 4]) = o;
    if (warp == 0 && valid) lse[row_of(m)] = lse2 * 0.6931471805599453f;
    __syncthreads();
    constexpr int kPieces = D / 8;  // 16-byte pieces of a row
    const int r = (int)threadIdx.x / kPieces, piece = (int)threadIdx.x % kPieces;  // (32 * kPieces threads)
    if (((tp * 256 + m_slice + r) >> lg) < E)
      reinterpret_cast<uint4*>(out + row_of(m_slice + r) * D)[piece] = *reinterpret_cast<const uint4*>(&rows[r * kRowWords + piece * 4]);
    __syncthreads();
  }
}

// The suffix append in front of a span-scheduled attention kernel (which is launched early and waits for it inside).
__global__ void __launch_bounds__(1024) append_prologue_kernel(const PoolView pool, const AppendArgs ap) {
  dependency_wait();
  launch_dependents();  // (the attention kernel reads the lengths before it waits for this one: not before the wait)
  const int warps_per_block = blockDim.x >> 5;
  append_tokens<4>(pool, ap, blockIdx.x * warps_per_block + (threadIdx.x >> 5), gridDim.x * warps_per_block);
}

// ------------------------------------------------------------------------------------------
static inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

static int64_t item_capacity(int n_q_heads, int n_kv_heads, int batch, int total_q) {
  const int G = n_q_heads / n_kv_heads;
  return (int64_t)total_q * G / 256 + batch + 1;
}

struct SpanLayout {
  int n_spans, slots, rows;
  bool cuts;              // may an item be cut?
  size_t lse, o, total;   // behind the cuts
};
static int64_t items_at_most(const kv_pool_t* p, int n_q_heads, int batch, int total_q) {
  return ((int64_t)total_q * (n_q_heads / p->n_kv_heads) / 256 + batch) * p->n_kv_heads;
}
static SpanLayout span_layout(const kv_pool_t* p, int n_q_heads, int batch, int total_q, int max_total_len) {
  const int64_t steps = ((int64_t)max_total_len + 127) / 128, sms = sm_count_of(p->device);
  const int64_t spans = (items_at_most(p, n_q_heads, batch, total_q) * steps + kSpanMinSteps - 1) / kSpanMinSteps;
  SpanLayout l;
  l.n_spans = (int)(spans < 1 ? 1 : spans < sms ? spans : sms);
  l.cuts = steps > 2 * kSpanSnap + 1;  // (an item of up to that many steps is never cut)
  const int64_t rows = (int64_t)total_q * (n_q_heads / p->n_kv_heads);
  l.slots = l.cuts ? 2 * l.n_spans : 0;
  l.rows = (int)(rows < 256 ? (rows + 7) / 8 * 8 : 256);
  l.lse = align256((size_t)l.n_spans * 3 * sizeof(int4));
  l.o = l.lse + align256((size_t)l.slots * l.rows * 2 * sizeof(float));
  l.total = l.o + (size_t)l.slots * l.rows * p->head_dim * sizeof(float);
  return l;
}
static size_t list_bytes(int batch, int total_q) {
  return 256 + align256(2 * sizeof(int4) * (size_t)((int64_t)total_q * 8 / 256 + batch + 1));
}

// The item list of the plan, or what span scheduling keeps, whichever is larger whatever the batch turns out to be (a
// workspace that is large enough for a batch is large enough for every smaller one); 256 bytes more to align the
// caller's pointer.
size_t extend_tc_workspace_bytes(const kv_pool_t* p, int n_q_heads, int batch, int total_q, int max_total_len) {
  if (batch <= 0 || total_q <= 0 || n_q_heads < p->n_kv_heads) return 0;
  const size_t list = list_bytes(batch, total_q), spans = span_layout(p, n_q_heads, batch, total_q, max_total_len).total;
  return 256 + (list > spans ? list : spans);
}
// The least the extend kernel runs with: the list, at any 16-byte boundary.
size_t extend_tc_min_workspace_bytes(int batch, int total_q) { return list_bytes(batch, total_q); }

bool extend_tc_supported(const kv_pool_t* p, int n_q_heads) {
  if (p->head_dim != 64 && p->head_dim != 128) return false;
  const int g = n_q_heads / p->n_kv_heads;
  return g == 1 || g == 2 || g == 4 || g == 8;
}

// Tensor map over Q [total_q][Hq][D] (bf16): a box is one 64-dim half of a query tile, that is 128/G tokens x the
// G heads of one KV head x 64 dims, written to shared memory with the 128-byte swizzle the MMA expects.  Rows past
// the end of Q read as zeros.
static kv_status_t make_q_map(CUtensorMap* map, const void* q, int total_q, int n_q_heads, int head_dim, int group) {
  typedef CUresult (*encode_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static encode_fn encode = nullptr;
  if (encode == nullptr) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    KV_CUDA_OK(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres));
    if (fn == nullptr || qres != cudaDriverEntryPointSuccess) return KV_ERR_CUDA;
    encode = reinterpret_cast<encode_fn>(fn);
  }
  const cuuint64_t dims[3] = {(cuuint64_t)head_dim, (cuuint64_t)n_q_heads, (cuuint64_t)total_q};
  const cuuint64_t strides[2] = {(cuuint64_t)head_dim * 2, (cuuint64_t)n_q_heads * head_dim * 2};
  const cuuint32_t box[3] = {64, (cuuint32_t)group, (cuuint32_t)(128 / group)};
  const cuuint32_t elem_strides[3] = {1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(q), dims, strides, box, elem_strides,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? KV_OK : KV_ERR_INVALID;
}

// One persistent CTA per SM, fewer if there are fewer items or the caller caps the kernel.
static kv_status_t tc_grid(const kv_pool_t* p, int n_items_bound, int cta_cap, int* grid_out) {
  const int sm_count = sm_count_of(p->device);
  int grid = n_items_bound < sm_count ? (n_items_bound < 1 ? 1 : n_items_bound) : sm_count;
  if (cta_cap > 0 && grid > cta_cap) grid = cta_cap;  // leave the other SMs to work that runs beside this kernel (< 0: no
                                                      // cap, and the kernel is launched without the early start)
  *grid_out = grid;
  return KV_OK;
}

template <int D, bool OPT, bool FAN, int SCHED>
static kv_status_t setup_tc(int device) {
  const size_t smem = sizeof(TcSmem<D>);
  static std::atomic<bool> configured[kMaxDevices];  // the attribute belongs to the function on one device
  if (device < 0 || device >= kMaxDevices) return KV_ERR_INVALID;
  if (!configured[device].load(std::memory_order_acquire)) {
    KV_CUDA_OK(cudaFuncSetAttribute(attn_extend_tc_kernel<D, OPT, FAN, SCHED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    if (SCHED == kSchedCluster)
      KV_CUDA_OK(cudaFuncSetAttribute(attn_extend_tc_kernel<D, OPT, FAN, SCHED>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    configured[device].store(true, std::memory_order_release);
  }
  return KV_OK;
}

template <int D, bool OPT, bool FAN, int SCHED>
static kv_status_t launch_tc(const TcArgs& a, const CUtensorMap& q_map, int grid, int device, bool early_start, cudaStream_t st) {
  const kv_status_t ss = setup_tc<D, OPT, FAN, SCHED>(device);
  if (ss != KV_OK) return ss;
  // early_start: launched so that it may start while the plan kernel in front of it still runs (it waits for it
  // inside).  Not wanted when another kernel is meant to take the SMs first (the mixed step's decode kernel): CTAs
  // that sit on an SM waiting for the plan keep that kernel's blocks away.
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kTcThreads);
  cfg.dynamicSmemBytes = sizeof(TcSmem<D>);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (early_start) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (SCHED == kSchedCluster && a.cl_splits > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)a.cl_splits;
    attr[n].val.clusterDim.y = attr[n].val.clusterDim.z = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  KV_CUDA_OK(cudaLaunchKernelEx(&cfg, attn_extend_tc_kernel<D, OPT, FAN, SCHED>, a, q_map));
  count_launch();
  return KV_OK;
}

static constexpr int kSplitChoices[] = {1, 2, 3, 4, 6, 8};

// How many clusters of c CTAs are on the device at a time (asked once per device and head size).
template <int D>
static kv_status_t resident_clusters(int device, int c, int* n) {
  static std::atomic<int> cached[kMaxDevices][kMaxClusterSplits + 1];  // value + 1
  const kv_status_t s = setup_tc<D, false, false, kSchedCluster>(device);
  if (s != KV_OK) return s;
  int v = cached[device][c].load(std::memory_order_relaxed);
  if (v == 0) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)c);
    cfg.blockDim = dim3(kTcThreads);
    cfg.dynamicSmemBytes = sizeof(TcSmem<D>);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)c;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, attn_extend_tc_kernel<D, false, false, kSchedCluster>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      clusters = 0;
    }
    v = clusters + 1;
    cached[device][c].store(v, std::memory_order_relaxed);
  }
  *n = v - 1;
  return KV_OK;
}

// Who takes which items, from the host-side bounds (and the workspace) alone; splits: CTAs per item for kSchedCluster.
//  - Items that are on the device at once go to a cluster each, as large as fits, one KV step per CTA at least: no plan
//    kernel, and the steps of an item run side by side.  Suffix append + extend of 1 / 4 / 8 / 16 sequences of 30-60 tokens
//    behind 1000-2000 (32/8 heads of 128): 32.1 / 38.2 / 42.2 / 43.7 us through the list, 15.7 / 24.4 / 31.8 / 41.0 this
//    way with 6 / 4 / 2 / 1 CTAs per item.
//  - Items that leave SMs idle: spans.  They cost a merge kernel behind the attention kernel and the partial results, 5 to
//    8 steps, and win what the other two leave idle, the SMs without a cluster or the last round of items.  8 / 16 sequences
//    of 9000-16000 keys 219 / 225 us through the list, 121 / 242 with clusters, 102 / 181 with spans; 160 items of 25 steps
//    (1.1 rounds) 93 and 70, 184 of 13 to 16 (1.2) 50 and 46, 68 and 61, but 160 of 10 40 and 40, 168 of 5 30 and 31.  The
//    number of items is known if a sequence has one; if it is estimated, the line lies higher: 320 of 22 (2.2) 122 and 106,
//    240 of 13 57 and 59.  More than four items per SM: the list (672 of 36 348 against 369).
static kv_status_t choose_schedule(const kv_pool_t* p, int n_q_heads, int batch, int total_q, int max_extend_len, int max_total_len,
                                   size_t workspace_bytes, int mode, int* sched, int* splits) {
  *sched = kSchedList;
  *splits = 1;
  const int G = n_q_heads / p->n_kv_heads, sms = sm_count_of(p->device);
  const int64_t pairs = ((int64_t)max_extend_len * G + 255) / 256, units = (int64_t)batch * pairs * p->n_kv_heads;
  const int64_t steps = ((int64_t)max_total_len + 127) / 128;
  const SpanLayout l = span_layout(p, n_q_heads, batch, total_q, max_total_len);
  const bool room = workspace_bytes >= 256 + l.total;  // (else: nothing that leaves partial results)
  const int64_t most = items_at_most(p, n_q_heads, batch, total_q);
  // (a sequence's last tile pair is half full on average, its keys somewhat fewer than the longest's; sequences of one pair
  // each are as many items as there are)
  const double rounds = (pairs == 1 ? (double)batch : (double)total_q * G / 256 + 0.5 * batch) * p->n_kv_heads / sms;
  const double even = 0.85 * steps * rounds;
  if (units <= sms || (most <= sms && units <= 2 * sms)) {
    *sched = kSchedCluster;
    if (!room || !l.cuts) return KV_OK;
    for (int c : kSplitChoices) {
      if (c > steps || units * c > l.slots) break;
      int resident = 0;
      const kv_status_t s = p->head_dim == 128 ? resident_clusters<128>(p->device, c, &resident) : resident_clusters<64>(p->device, c, &resident);
      if (s != KV_OK) return s;
      if (units <= resident) *splits = c;
    }
    if (mode == 0 && (double)steps / *splits - even > 12.0) *sched = kSchedSpans;
  } else if (mode == 0 && room && l.cuts && most <= 4ll * sms && 0.85 * steps * ceil(rounds) - even > (pairs == 1 ? 7.5 : 11.5)) {
    *sched = kSchedSpans;
  }
  return KV_OK;
}

static SpanArgs span_args(const SpanLayout& l, char* ws, int max_tp, int total_q, int cta_cap) {
  SpanArgs a{};
  a.n_spans = l.n_spans;  // (not the number of CTAs: the cuts, and with them the bits, are the same beside a decode kernel)
  // Two spans a CTA pay where the decode kernel, on the SMs that this leaves, takes longer than the extend kernel on all of
  // them; that is where the share is 0.6 of the SMs (three: 0.37).
  a.per_cta = cta_cap > 0 ? max(1, (int)((double)l.n_spans / cta_cap + 0.32)) : 1;
  a.max_tp = max_tp;
  a.total_q = total_q;
  a.rows = l.rows;
  a.desc = reinterpret_cast<int4*>(ws);
  a.part_lse = l.cuts ? reinterpret_cast<float*>(ws + l.lse) : nullptr;
  a.part_o = l.cuts ? reinterpret_cast<float*>(ws + l.o) : nullptr;
  return a;
}
// Where the workspace begins: on a 256-byte boundary, or, if that does not leave `need` bytes of it, where the caller says.
static char* align_workspace(void* ws, size_t bytes, size_t need) {
  char* at = reinterpret_cast<char*>((reinterpret_cast<uintptr_t>(ws) + 255) & ~(uintptr_t)255);
  const size_t skip = (size_t)(at - reinterpret_cast<char*>(ws));
  return skip + need <= bytes ? at : reinterpret_cast<char*>(ws);
}

// Merges the chunks of cut items behind a span-scheduled attention kernel; nothing to do for other batches.  early: that
// kernel is the one queued last.
kv_status_t launch_extend_combine(kv_pool_t* p, int n_q_heads, int batch, int total_q, int max_extend_len, int max_total_len, void* out, float* lse,
                                  void* workspace, size_t workspace_bytes, bool early, cudaStream_t st) {
  int sched, splits;
  const kv_status_t cs = choose_schedule(p, n_q_heads, batch, total_q, max_extend_len, max_total_len, workspace_bytes, 0, &sched, &splits);
  if (cs != KV_OK) return cs;
  if (sched != kSchedSpans) return KV_OK;
  const SpanLayout l = span_layout(p, n_q_heads, batch, total_q, max_total_len);
  if (!l.cuts || l.n_spans < 2) return KV_OK;
  const int G = n_q_heads / p->n_kv_heads;
  int lg = 0;
  while ((1 << lg) < G) ++lg;
  const SpanArgs a = span_args(l, align_workspace(workspace, workspace_bytes, l.total), 0, total_q, 0);
  const auto kernel = p->head_dim == 128 ? span_combine_kernel<128> : span_combine_kernel<64>;
  const unsigned blocks = (unsigned)((a.n_spans - 1) * kCombineSlices), threads = (unsigned)p->head_dim * 4;
  if (early) {
    KV_CUDA_OK(launch_early(kernel, blocks, threads, 0, st, a, n_q_heads, G, lg, (__nv_bfloat16*)out, lse));
  } else {
    kernel<<<blocks, threads, 0, st>>>(a, n_q_heads, G, lg, (__nv_bfloat16*)out, lse);
    KV_CUDA_OK(cudaGetLastError());
  }
  count_launch();
  return KV_OK;
}

kv_status_t launch_extend_tc(kv_pool_t* p, const void* q, int n_q_heads, const int* cu_q, const int* block_tables,
                             int max_pages, const int* prefix_lens, const int* extend_lens, int batch, int total_q,
                             int max_extend_len, int max_total_len, float scale, void* out, float* lse,
                             void* workspace, size_t workspace_bytes, int cta_cap, int mode, const FanArgs* fan,
                             const AppendArgs* app, int phase, cudaStream_t st) {
  // phase 0: plan (with the suffix append, if any) and attention; 1: the plan only; 2: attention over the plan that a
  // phase-1 call with the same arguments left in the workspace
  const size_t need = extend_tc_min_workspace_bytes(batch, total_q);
  if (workspace == nullptr || workspace_bytes < need) return KV_ERR_WORKSPACE;
  const int G = n_q_heads / p->n_kv_heads;
  // Q is read through a tensor map (16-byte base), O is written with 32-byte stores
  if ((reinterpret_cast<uintptr_t>(q) & 15) != 0 || (reinterpret_cast<uintptr_t>(out) & 31) != 0) return KV_ERR_INVALID;
  CUtensorMap q_map;
  if (phase != 1) {
    const kv_status_t ms = make_q_map(&q_map, q, total_q, n_q_heads, p->head_dim, G);
    if (ms != KV_OK) return ms;
  }
  int lg = 0;
  while ((1 << lg) < G) ++lg;
  char* ws = align_workspace(workspace, workspace_bytes, need);
  if ((reinterpret_cast<uintptr_t>(ws) & 15) != 0) return KV_ERR_WORKSPACE;  // (the list holds 16-byte records)
  int* n_items = reinterpret_cast<int*>(ws);
  int4* items = reinterpret_cast<int4*>(ws + 256);
  const int64_t capacity = item_capacity(n_q_heads, p->n_kv_heads, batch, total_q);
  const int max_tp = (int)(((int64_t)max_extend_len * G + 255) / 256);
  const int max_steps = 2 * ((max_total_len + 127) / 128);
  const int64_t bound = (int64_t)batch * max_tp * p->n_kv_heads;
  const int n_bound = bound > (1 << 30) ? (1 << 30) : (int)bound;
  int grid = 1;
  {
    const kv_status_t gs = tc_grid(p, n_bound, cta_cap, &grid);
    if (gs != KV_OK) return gs;
  }
  // about a hundred items per group (measured on the 8B extend, long-document and fan-out shapes: fewer and larger
  // groups lose the L2 reuse, one sequence per group loses balance when a sequence has few items)
  // (a batch with fewer than a dozen items per SM is left in pure cost order: there the balance matters more)
  int groups = n_bound >= 12 * sm_count_of(p->device) ? n_bound / 96 : 1;
  groups = groups < 1 ? 1 : groups;
  groups = groups > batch ? batch : groups;
  groups = groups > kPlanBuckets / 16 ? kPlanBuckets / 16 : groups;
  int sched = kSchedList, splits = 1;
  if (mode != 1) {
    const kv_status_t cs = choose_schedule(p, n_q_heads, batch, total_q, max_extend_len, max_total_len, workspace_bytes, mode, &sched, &splits);
    if (cs != KV_OK) return cs;
  }
  const PlanArgs pa{prefix_lens, extend_lens, cu_q, batch, max_tp, lg, max_steps, (int)capacity, max_pages, mode,
                    fan != nullptr ? *fan : FanArgs{}, groups, p->d_status, items, n_items, n_items + 1, grid};
  if (sched != kSchedList) {
    // no plan: the attention kernel's CTAs find their work themselves
    if (phase == 1) return KV_OK;
    if (app != nullptr && app->total_new > 0) {
      const int64_t want = ((int64_t)app->total_new + 31) / 32;
      const int64_t cap = 2 * (int64_t)sm_count_of(p->device);
      const AppendSpread sp = append_spread(app->total_new, p->n_kv_heads * (p->head_dim >> 3), sm_count_of(p->device));
      static std::atomic<bool> allowed[kMaxDevices];
      if (sp.blocks > 0 && allow_smem((const void*)append_prologue_kernel, spread_smem(1), allowed, p->device)) {
        KV_CUDA_OK(launch_early(append_prologue_kernel, (unsigned)sp.blocks, (unsigned)sp.warps * 32, (size_t)sp.smem_front, st, p->view(), *app));
      } else {
        KV_CUDA_OK(launch_early(append_prologue_kernel, (unsigned)(want < cap ? want : cap), 1024, 0, st, p->view(), *app));
      }
      count_launch();
    }
  } else if (phase == 2) {
    // the plan is in the workspace already
  } else if (app != nullptr && app->total_new > 0) {
    // Plan block + append blocks, one warp per token.  A block's 1024 threads take 64 registers each, so one block is on an SM at a
    // time: up to 32 tokens per SM the tokens are spread over as many blocks as there are SMs (28 sequences of 15-18 tokens behind
    // 64-95 18.0 -> 15.7 us, 33 of 29-31 behind 1100, 8/8 heads, 48.5 -> 46.3; on two streams 26.8 -> 24.8 and 72.4 -> 76.7, since the
    // blocks wait on whole SMs); a longer suffix runs in rounds of 32 and the attention kernel can start once the last block has.
    const int sms = sm_count_of(p->device), per_block = prologue_tokens(app->total_new, sms);
    const int64_t want = ((int64_t)app->total_new + per_block - 1) / per_block, cap = 2 * (int64_t)sms - 1;
    KV_CUDA_OK(launch_early(extend_prologue_kernel, (unsigned)(1 + (want < cap ? want : cap)), 1024, 0, st, pa, p->view(), *app, per_block));
    count_launch();
  } else {
    KV_CUDA_OK(launch_early(extend_tc_plan_kernel, 1, 1024, 0, st, pa));
    count_launch();
  }
  if (phase == 1) return KV_OK;

  TcArgs a{};
  a.pool = p->view();
  a.q = (const __nv_bfloat16*)q;
  a.cu_q = cu_q;
  a.block_tables = block_tables;
  a.max_pages = max_pages;
  a.prefix_lens = prefix_lens;
  a.extend_lens = extend_lens;
  a.batch = batch;
  a.n_q_heads = n_q_heads;
  a.group = G;
  a.lg_group = lg;
  a.mode = mode;
  a.fan = fan != nullptr ? *fan : FanArgs{};
  a.scale_log2 = scale * 1.4426950408889634f;
  a.out = (__nv_bfloat16*)out;
  a.lse = lse;
  a.items = items;
  a.n_items = n_items;
  a.next_item = n_items + 1;
  // Skipping the search for the row maximum pays where items have many KV steps (measured: +2 % on the
  // long-document shapes, -1 % on the 8B extend batch whose items have a dozen steps)
  const bool opt = max_total_len >= kOptimisticMinLen;
  a.beside = cta_cap != 0;
  bool early = cta_cap >= 0;
  if (sched != kSchedList) {
    const SpanLayout l = span_layout(p, n_q_heads, batch, total_q, max_total_len);
    a.span = span_args(l, align_workspace(workspace, workspace_bytes, l.total), max_tp, total_q, sched == kSchedSpans ? cta_cap : 0);
    a.span.plan_early = app != nullptr && app->total_new > 0;
    a.cl_splits = splits;
    grid = sched == kSchedSpans ? (a.span.n_spans + a.span.per_cta - 1) / a.span.per_cta : batch * max_tp * p->n_kv_heads * splits;
    // (beside a decode kernel that waits for nothing, this kernel has to start behind all that was queued before it)
    if (cta_cap > 0) early = false;
  }
  auto go = [&](auto d, auto o, auto f) {
    constexpr int DD = decltype(d)::value;
    constexpr bool OO = decltype(o)::value, FF = decltype(f)::value;
    if constexpr (!FF)
      if (sched == kSchedSpans) return launch_tc<DD, OO, false, kSchedSpans>(a, q_map, grid, p->device, early, st);
    if (sched == kSchedCluster) return launch_tc<DD, OO, FF, kSchedCluster>(a, q_map, grid, p->device, early, st);
    return launch_tc<DD, OO, FF, kSchedList>(a, q_map, grid, p->device, early, st);
  };
  using I128 = std::integral_constant<int, 128>;
  using I64 = std::integral_constant<int, 64>;
  const bool fan_mode = mode == 2;
  kv_status_t ls;
  if (p->head_dim == 128) {
    if (fan_mode) ls = opt ? go(I128{}, std::true_type{}, std::true_type{}) : go(I128{}, std::false_type{}, std::true_type{});
    else ls = opt ? go(I128{}, std::true_type{}, std::false_type{}) : go(I128{}, std::false_type{}, std::false_type{});
  } else if (fan_mode) {
    ls = opt ? go(I64{}, std::true_type{}, std::true_type{}) : go(I64{}, std::false_type{}, std::true_type{});
  } else {
    ls = opt ? go(I64{}, std::true_type{}, std::false_type{}) : go(I64{}, std::false_type{}, std::false_type{});
  }
  if (ls != KV_OK || sched != kSchedSpans || cta_cap > 0) return ls;
  return launch_extend_combine(p, n_q_heads, batch, total_q, max_extend_len, max_total_len, out, lse, workspace, workspace_bytes, true, st);
}

}  // namespace kvattn
