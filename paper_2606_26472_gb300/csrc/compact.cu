// In-place, order-preserving K/V compaction to the kept set (App. H).
//
// For every sequence that evicted in the last selection and every
// (layer, K|V, head group) stream: row i <- row kept[i] for i from the first
// evicted slot to the new cache length.  Rows are moved with 1-D TMA bulk
// copies global -> shared -> global (cp.async.bulk + mbarrier), no cluster
// multicast.  A persistent grid of one-warp CTAs walks its streams' batches
// through a ring of shared-memory stages: while batch k is stored, batches
// k+1 .. k+S-1 are loading.
//
// In-place safety without any inter-CTA wait: streams are disjoint bytes;
// inside a CTA's rows of a stream kept[i] >= i and rows are processed in
// increasing i, so a load (slot kept[i] >= i) never reads a slot that an
// earlier store has written, and a later store to a slot some earlier batch
// still had to read is issued only after that batch's loads completed.  With
// per-stream units one CTA owns each stream; the balanced split below cuts
// streams between CTAs and covers the reads across a cut with a stash.
//
// Under per-layer budgets (kLayers) each (sequence, layer) has its own kept
// list, first moved slot and length; the streams and the copy are unchanged.
// The balanced split then runs over (sequence, layer) pairs of two streams
// each.  Without it the streams differ in length (a layer's rows follow its
// budget), so the CTAs take units from a shared counter instead of a fixed
// stride, in layer-major order: with budgets that fall with depth, larger
// streams come first and the greedy assignment ends nearly level.
//
// Balanced split: the moved rows of all evicting streams,
// laid end to end, are cut into one equal chunk per CTA (long copies: and
// shorter ones for the CTAs that finish first, Chunks in plans.h), so one evicting
// sequence still covers the whole grid and no CTA carries a longer share.
// A chunk that ends inside a stream at slot a still reads, for its last rows,
// sources in [a, n_new) that later chunks overwrite.  compact_stash_kernel
// copies those rows aside before the compaction starts, and the chunk reads
// them there.  They are a suffix of the chunk's rows in that stream, no
// longer than the chunk nor than the eviction's largest shift
// kept[n-1] - (n-1).
//
// Head and tail split (token budgets, when both bounds exceed the stash): rows
// from the first one whose source lies at or past the new length, the tail,
// read slots that no row is written to.  compact_stash_kernel moves the rows
// before it, the head, in place, a CTA per (stream, head group) in increasing
// row order; the copy then moves every tail in chunks, with no row in any
// chunk's way.  Cutting n slots to K at random leaves about K * K /
// n rows in the head.  A batch of many streams whose heads are long keeps the
// per-stream units.  32 layers, 2 KiB rows, units (with their 512-byte to 1
// KiB pieces) / head + tail: 65,536, 38,940 and 12,345 slots to 4,096 (3.2 GB
// moved) 850 / 90 + 461 us (late chunks: 404); 9,000 to 3,000 461 / 52 + 97; 3 x 8,192 to 4,096
// 847 / 272 + 289 (half the rows are in the heads, at 6 TB/s); 4,396 to 4,096
// (nearly all in the head) 575 / 167 + 22.
//
// A selection's eviction is compacted once: compact_consumed_kernel, launched
// after the copy, sets each sequence's first moved slot to its length, so
// another compaction before the next selection moves nothing.
#include "common.cuh"
#include "kernels.h"

namespace epikv {

#ifndef EPIKV_COMPACT_STAGE_BYTES
#define EPIKV_COMPACT_STAGE_BYTES 16384
#endif
#ifndef EPIKV_COMPACT_CTAS_PER_SM
#define EPIKV_COMPACT_CTAS_PER_SM 2  // more CTAs per SM overload the memory system (measured)
#endif
#ifndef EPIKV_COMPACT_ORDER
#define EPIKV_COMPACT_ORDER 0  // 0: units sequence-major, 1: layer-major
#endif
#ifndef EPIKV_COMPACT_HEAD_SPLIT
#define EPIKV_COMPACT_HEAD_SPLIT 0  // 0: chosen on the device to fill the grid
#endif
constexpr int kStageBytes = EPIKV_COMPACT_STAGE_BYTES;
constexpr uint64_t kWaitNs = 2000000000ull;   // 2 s: far beyond any real copy
constexpr uint64_t kDrainNs = 100000000ull;   // 0.1 s per stage after a timeout

#ifndef EPIKV_COMPACT_BALANCED
#define EPIKV_COMPACT_BALANCED 1  // 0: per-stream units only
#endif
#ifndef EPIKV_COMPACT_STAGED_BLOCKS
#define EPIKV_COMPACT_STAGED_BLOCKS 1024  // block-table entries kept in shared memory (larger tables: global reads)
#endif
constexpr int kStagedBlocks = EPIKV_COMPACT_STAGED_BLOCKS;

constexpr int kStashThreads = 512;
constexpr int kStashUnroll = 4;
// Bytes moved (read and written) up to which the copy's CTAs are let in while
// the stash kernel runs, instead of as its CTAs end.  It hides the launch and
// the copy's own look-up of its rows, but CTAs placed early copy 1.3 % slower
// over a long copy: 0.13 GB 55.5 us per step early / 58.2 late (60.5 without
// programmatic launch), 1.2 GB 240.5 / 241.5 (246.5), 8.4 GB 1,359 / 1,342
// (1,342), 67 GB 10,400 / 10,250 (10,250).
constexpr int64_t kStashEarlyBytes = 1ll << 30;
constexpr int kHeadUnroll = 8;        // vectors per thread and batch of the head
constexpr int kMaxHeadRows = 512;     // rows per batch of the head
constexpr int64_t kUnitRounds = 4;    // streams per CTA from which per-stream units are even enough

// The balanced split's row space is made of pairs: under token budgets one
// per evicting entry, with its 2L streams; under per-layer budgets one per
// (evicting entry, layer), with that layer's K and V streams, at most
// kMaxLayerPairs of them (more: per-stream units).
// Per-layer budgets, 32 layers, 8,192-slot caches evicting 128 slots per
// step (compaction ms, balanced / per-stream units): 1 sequence 0.35 / 1.09,
// 2 sequences 0.68 / 1.24, 8 sequences 2.59 / 2.68, 32 sequences 10.18 /
// 9.95.  So the balanced split takes at most 256 (entry, layer) pairs.
#ifndef EPIKV_COMPACT_LAYER_PAIRS
#define EPIKV_COMPACT_LAYER_PAIRS 256
#endif
constexpr int kMaxLayerPairs = EPIKV_COMPACT_LAYER_PAIRS;
__host__ __device__ inline int list_ints(int n_seq) { return (n_seq + 31) / 32 * 32; }
__host__ __device__ inline int pairs_cap(int n_seq, int L, bool layers) {
  return layers ? (n_seq * L < kMaxLayerPairs ? n_seq * L : kMaxLayerPairs) : n_seq;
}
__host__ __device__ inline int pre_entries(int cap) { return (cap + 32) / 32 * 32; }

// The batch entries that evicted, in batch order, into list; with pre, the
// prefix sums of their moved rows per stream (pre[k] = rows of entries
// before the k-th).  One warp; every CTA of both kernels builds the same.
// Every entry's moved rows are loaded first (list holds them, list_ints(n_seq)
// >= n_seq words), all loads in flight together, then scanned in place.
__device__ int evicting_entries(const DevState& st, const Dims& dm, const int32_t* __restrict__ seq_ids,
                                int n_seq, int* list, int64_t* pre, int lane) {
#pragma unroll 4
  for (int b = lane; b < n_seq; b += 32) {
    const int seq = seq_ids[b];
    list[b] = (seq >= 0 && seq < dm.S) ? st.n_cache[seq] - st.first_changed[seq] : 0;
  }
  __syncwarp();
  int n_ev = 0;
  int64_t acc = 0;
  for (int base = 0; base < n_seq; base += 32) {
    const int b = base + lane;
    const int len = b < n_seq ? list[b] : 0;
    __syncwarp();  // the chunk's lengths are read before any of its entries is written
    const bool ev = len > 0;
    const unsigned m = __ballot_sync(0xffffffffu, ev);
    int incl = ev ? len : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (ev) {
      const int k = n_ev + __popc(m & ((1u << lane) - 1u));
      list[k] = b;   // k <= b: an entry already read
      if (pre) pre[k + 1] = acc + incl;
    }
    acc += __shfl_sync(0xffffffffu, incl, 31);
    n_ev += __popc(m);
    __syncwarp();
  }
  if (pre && lane == 0) pre[0] = 0;
  __syncwarp();
  return n_ev;
}

// Per-layer budgets: the prefix sums over the (entry, layer) pairs of their
// moved rows per stream (pre[k] = rows of the pairs before the k-th, pair k
// = entry k / L, layer k % L).  One warp; returns the pairs' total.
__device__ int64_t layer_pairs(const DevState& st, const Dims& dm, const int32_t* __restrict__ seq_ids,
                               const int* list, int n_ev, int64_t* pre, int lane) {
  const int np = n_ev * dm.L;
  // every pair's rows first (independent loads, several in flight), then the scan
#pragma unroll 4
  for (int k = lane; k < np; k += 32) {
    const int i = seq_ids[list[k / dm.L]] * dm.L + k % dm.L;
    pre[k + 1] = max(0, st.n_layer[i] - st.lfirst[i]);
  }
  __syncwarp();
  int64_t acc = 0;
  for (int base = 0; base < np; base += 32) {
    const int k = base + lane;
    const int len = k < np ? (int)pre[k + 1] : 0;
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (k < np) pre[k + 1] = acc + incl;
    acc += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) pre[0] = 0;
  __syncwarp();
  return acc;
}

// One pair's stream q (token budgets: layer * 2 + K|V; per-layer budgets:
// K|V): its entry, sequence, layer, first moved row, new length and kept list.
struct PairAt {
  int b, seq, layer, kvk, first, n_new;
  const int32_t* kl;
};
__device__ __forceinline__ PairAt pair_at(const DevState& st, const Dims& dm, const int32_t* __restrict__ seq_ids,
                                          const int* list, const int32_t* __restrict__ kept, int kept_stride,
                                          bool layers, int p, int q) {
  PairAt a;
  a.b = list[layers ? p / dm.L : p];
  a.seq = seq_ids[a.b];
  if (layers) {
    a.layer = p % dm.L;
    a.kvk = q;
    const int i = a.seq * dm.L + a.layer;
    a.first = st.lfirst[i];
    a.n_new = st.n_layer[i];
    a.kl = kept + ((size_t)a.b * dm.L + a.layer) * kept_stride;
  } else {
    a.layer = q >> 1;
    a.kvk = q & 1;
    a.first = st.first_changed[a.seq];
    a.n_new = st.n_cache[a.seq];
    a.kl = kept + (size_t)a.b * kept_stride;
  }
  return a;
}

// Whether the balanced split applies: a grid within the stash's CTAs, under
// per-layer budgets no more pairs than kMaxLayerPairs, and a bound on the
// rows of a chunk whose sources lie in later chunks' regions -- a suffix of
// the chunk's last stream segment, no longer than the segment (so than the
// chunk, ceil(total / grid) rows) nor than the largest shift
// kept[n-1] - (n-1) of any pair -- within one CTA's stash.  total = moved
// rows of all streams.  Returns the rows a stash needs, 0 if it does not apply.
__device__ int balanced_split(const DevState& st, const Dims& dm, const int32_t* __restrict__ seq_ids,
                               const int* list, int n_ev, const int32_t* __restrict__ kept, int kept_stride,
                               bool layers, int n_pairs, int64_t total, int lane) {
  if (!EPIKV_COMPACT_BALANCED || gridDim.x > kMaxStashCtas) return 0;
  if (layers && n_pairs > kMaxLayerPairs) return 0;
  if (chunks_fit_stash(total, gridDim.x, dm.stash_rows)) return dm.stash_rows;
  int shift = 1;
#pragma unroll 4
  for (int k = lane; k < n_pairs; k += 32) {
    const PairAt a = pair_at(st, dm, seq_ids, list, kept, kept_stride, layers, k, 0);
    if (a.n_new > a.first) shift = max(shift, __ldg(a.kl + a.n_new - 1) - (a.n_new - 1));
  }
  shift = __reduce_max_sync(0xffffffffu, shift);
  return shift_stride(shift, dm.stash_rows);
}

// Whether the head and tail split applies (not balanced_split): heads of at
// most a quarter of the moved rows, or too few streams to fill the grid
// evenly as units.  pre, which holds the prefix sums of the moved rows, then
// holds those of the tails.  One warp; every CTA of both kernels finds the
// same.
__device__ bool head_tail_split(const DevState& st, const Dims& dm, const int32_t* __restrict__ seq_ids,
                                const int* list, int n_ev, const int32_t* __restrict__ kept, int kept_stride,
                                int64_t* pre, int lane) {
  const int64_t total = pre[n_ev];
  __syncwarp();
  int64_t acc = 0;
  for (int base = 0; base < n_ev; base += 32) {
    const int k = base + lane;
    int incl = 0;
    if (k < n_ev) {
      const int b = list[k], seq = seq_ids[b], n_new = st.n_cache[seq];
      const int32_t* kl = kept + (size_t)b * kept_stride;
      incl = n_new - tail_start([kl](int i) { return __ldg(kl + i); }, st.first_changed[seq], n_new);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (k < n_ev) pre[k + 1] = acc + incl;
    acc += __shfl_sync(0xffffffffu, incl, 31);
  }
  __syncwarp();
  return (total - acc) * 4 <= total || (int64_t)n_ev * 2 * dm.L < kUnitRounds * (int64_t)gridDim.x;
}

// Entry e, stream q (layer * 2 + K|V) and row r (from the entry's first
// moved slot) of row o of the balanced row space.
__device__ __forceinline__ void locate_row(const int64_t* pre, int n_ev, int upe, int64_t o, int& e, int& q,
                                           int64_t& r) {
  int lo = 0, hi = n_ev - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] * upe <= o) lo = mid;
    else hi = mid - 1;
  }
  e = lo;
  const int64_t len = pre[e + 1] - pre[e];
  const int64_t rel = o - pre[e] * upe;
  q = (int)(rel / len);
  r = rel - (int64_t)q * len;
}

struct Cursor {
  int u;      // unit index (this CTA strides by gridDim.x); balanced: 0 while rows remain
  int i;      // next row of the unit
  int end;    // row past the last of the unit
  int b, seq, layer, kvk, hg;
  int stash_at;   // balanced: sources in [stash_at, n_new) are read from the next chunk's stash
  int n_new;      // balanced: the sequence's length after the eviction
  int row0;       // balanced: the row whose source is the stash's first row
  int64_t o_end;  // balanced: row `end` in the balanced row space
};

// kSplit: the balanced split is compiled in (token budgets always; per-layer
// budgets when the batch has at most kMaxLayerPairs (entry, layer) pairs --
// the instance for larger batches keeps the per-stream units' code alone,
// which measured 6 % faster there than with the split's code beside it).
template <bool kLayers, bool kSplit, bool kLong>
__global__ void __launch_bounds__(32) compact_kernel(DevState st, Dims dm, KvDev kv,
                                                     const int32_t* __restrict__ seq_ids, int n_seq,
                                                     const int32_t* __restrict__ kept, int kept_stride,
                                                     int after_stash) {
  // Launched programmatically after compact_stash_kernel (after_stash), the
  // CTAs start beside it: that kernel lets them in only after its own wait,
  // so the selection's results are complete, and it writes neither those nor
  // the cache.  What it writes, the stash, and what it still reads, the rows
  // this kernel overwrites, are first touched after the wait below.
  bool waited = !(kSplit && after_stash);
  if (waited) pdl_wait();
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[kStages];
  __shared__ char* dptr[kStages][kMaxRPB];
  __shared__ int stage_rows[kStages];
  int* list = reinterpret_cast<int*>(smem + kStages * kStageBytes);
  int64_t* pre = reinterpret_cast<int64_t*>(list + list_ints(n_seq));
  // the current sequence's block table
  int* bt_s = reinterpret_cast<int*>(pre + pre_entries(pairs_cap(n_seq, dm.L, kLayers)));
  const int lane = threadIdx.x;

  // ---- the batch entries that evicted (every CTA builds the same list)
  const int n_ev = evicting_entries(st, dm, seq_ids, n_seq, list, kLayers ? nullptr : pre, lane);
  if (n_ev == 0) {
    pdl_wait();   // this kernel ends after the stash kernel, for the kernels that wait for this one
    return;
  }
  // ---- the balanced split's pairs and their rows
  const int n_pairs = kLayers ? n_ev * dm.L : n_ev;
  const int sp = kLayers ? 2 : 2 * dm.L;  // streams per pair
  int64_t pair_rows = 0;
  int stride = 0;
  bool balanced = false, tails = false;   // tails: the balanced rows are the tails, no stash
  if constexpr (kSplit) {
    if (!kLayers) pair_rows = pre[n_ev];
    else if (n_pairs <= kMaxLayerPairs) pair_rows = layer_pairs(st, dm, seq_ids, list, n_ev, pre, lane);
    if (!kLayers || n_pairs <= kMaxLayerPairs)
      stride = balanced_split(st, dm, seq_ids, list, n_ev, kept, kept_stride, kLayers, n_pairs, pair_rows * sp, lane);
    balanced = stride > 0;
    if (!kLayers && !balanced && after_stash &&
        head_tail_split(st, dm, seq_ids, list, n_ev, kept, kept_stride, pre, lane)) {
      balanced = tails = true;
      pair_rows = pre[n_ev];
    }
  }

  // ---- per-stream units only: whole token rows unless too few streams
  // evict to give every CTA one (small TMA copies cost much more per byte
  // than a tail)
  const int G = gridDim.x;
  int hs = 1;
  if (!balanced) {
#if EPIKV_COMPACT_HEAD_SPLIT > 0
    if (dm.H % EPIKV_COMPACT_HEAD_SPLIT == 0) hs = EPIKV_COMPACT_HEAD_SPLIT;
#else
    while ((long)n_ev * 2 * dm.L * hs < G && dm.H % (2 * hs) == 0 && (dm.H / (2 * hs)) * dm.d * 2 >= 256) hs *= 2;
#endif
  }
  const int rb = (dm.H / hs) * dm.d * 2;               // bytes per row piece
  const int64_t piece_elems = (int64_t)(dm.H / hs) * dm.d;
  const int rpb = min(kStageBytes / rb, kMaxRPB);      // rows per batch
  const int upe = 2 * dm.L * hs;
  const int units = balanced ? 1 : n_ev * upe;
  // balanced: this CTA's current chunk [o_begin, o_stop) of the row space
  Chunks<kLong> ck{0, 0, G, G, 0};
  int chunk = blockIdx.x;
  int64_t o_begin = 0, o_stop = 0;
  if (balanced) {
    ck = make_chunks<kLong>(dm.stash_rows, pair_rows * sp, G, tails, stride, kv.layout == EPIKV_LAYOUT_PAGED);
    o_begin = ck.start(chunk);
    o_stop = ck.start(chunk + 1);
  }
  const bool paged = kv.layout == EPIKV_LAYOUT_PAGED;
  const bool bt_in_smem = paged && kv.max_blocks <= kStagedBlocks;

  if (lane == 0) {
    for (int s = 0; s < kStages; ++s) mbar_init(&full[s], 1);
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  __syncwarp();

  // the next unit of this CTA: a fixed stride, or the shared counter (kLayers)
  auto next_unit = [&](int u) -> int {
    if (!kLayers) return u + G;
    int v = 0;
    if (lane == 0) v = (int)atomicAdd(st.work, 1u);
    return __shfl_sync(0xffffffffu, v, 0);
  };
  auto load_unit = [&](Cursor& c) {
    while (c.u < units) {
      int e, rem;
      if (kLayers || EPIKV_COMPACT_ORDER == 1) {
        e = c.u % n_ev;
        rem = c.u / n_ev;
      } else {
        e = c.u / upe;
        rem = c.u % upe;
      }
      c.layer = rem / (2 * hs);
      c.kvk = (rem / hs) & 1;
      c.hg = rem % hs;
      c.b = list[e];
      c.seq = seq_ids[c.b];
      if (kLayers) {
        c.i = st.lfirst[c.seq * dm.L + c.layer];
        c.end = st.n_layer[c.seq * dm.L + c.layer];
      } else {
        c.i = st.first_changed[c.seq];
        c.end = st.n_cache[c.seq];
      }
      c.stash_at = INT_MAX;
      if (c.i < c.end) return;
      c.u = next_unit(c.u);
    }
  };
  // balanced: the stream segment holding row o of the chunk
  auto open_at = [&](Cursor& c, int64_t o) {
    int p, q;
    int64_t r;
    locate_row(pre, n_pairs, sp, o, p, q, r);
    const PairAt a = pair_at(st, dm, seq_ids, list, kept, kept_stride, kLayers, p, q);
    c.b = a.b;
    c.seq = a.seq;
    c.layer = a.layer;
    c.kvk = a.kvk;
    c.hg = 0;
    const int64_t rest = pre[p + 1] - pre[p] - r;       // rows of the stream from o on
    c.i = (tails ? a.n_new - (int)(pre[p + 1] - pre[p]) : a.first) + (int)r;
    if (!tails && o_stop - o < rest) {                   // the chunk ends inside this stream
      c.end = c.i + (int)(o_stop - o);
      c.stash_at = c.end;
      c.n_new = a.n_new;
      c.row0 = st.stash_row0[chunk + 1];                 // written by compact_stash_kernel (read again after the wait)
    } else {
      c.end = c.i + (int)min(rest, o_stop - o);
      c.stash_at = INT_MAX;
    }
    c.o_end = o + (c.end - c.i);
  };
  // balanced: the first row of the next late chunk that no CTA has taken
  // (-1: none is left)
  auto next_chunk = [&]() -> int64_t {
    while (kLong && ck.n > G) {
      int v = 0;
      if (lane == 0) v = G + (int)atomicAdd(st.work, 1u);
      chunk = __shfl_sync(0xffffffffu, v, 0);
      if (chunk >= ck.n) break;
      const int64_t o = ck.start(chunk);
      o_stop = ck.start(chunk + 1);
      if (o < o_stop) return o;
    }
    return -1;
  };
  auto advance = [&](Cursor& c) {
    c.i += rpb;
    if (c.i >= c.end) {
      if (balanced) {
        const int64_t o = c.o_end < o_stop ? c.o_end : next_chunk();
        if (o >= 0) open_at(c, o);
        else c.u = units;
      } else {
        c.u = next_unit(c.u);
        load_unit(c);
      }
    }
  };
  // kept slots of the batch at c, one load per row, issued early and used later
  auto prefetch = [&](const Cursor& c, int (&pk)[kMaxRowsPerLane]) {
    if (c.u >= units) return;
    const int nrows = min(rpb, c.end - c.i);
    const int32_t* kl = kept + (kLayers ? (size_t)c.b * dm.L + c.layer : (size_t)c.b) * kept_stride + c.i;
#pragma unroll
    for (int j = 0; j < kMaxRowsPerLane; ++j) {
      const int r = lane + 32 * j;
      pk[j] = r < nrows ? __ldg(kl + r) : 0;
    }
  };
  int staged_seq = -1, staged_layer = -1;
  // element offset of a slot of the current sequence, -1 outside the view
  auto slot_offset = [&](int layer, int seq, int slot) -> int64_t {
    if (!bt_in_smem) return kv_row_offset(kv, layer, seq, slot, dm.T);
    if (slot < 0) return -1;
    const int bi = slot / kv.block_size;
    if (bi >= kv.max_blocks) return -1;
    const int blk = bt_s[bi];
    if (blk < 0 || blk >= kv.num_blocks) return -1;
    return (int64_t)layer * kv.stride_layer + (int64_t)blk * kv.stride_block +
           (int64_t)(slot - bi * kv.block_size) * kv.stride_token;
  };

  // issue the loads of the batch at cursor c (kept slots pk) into stage s
  auto issue = [&](const Cursor& c, const int (&pk)[kMaxRowsPerLane], int s) {
    // the stream's block table (per layer when the layers have their own tables)
    if (bt_in_smem && (c.seq != staged_seq || (kv.table_stride_layer && c.layer != staged_layer))) {
      __syncwarp();
      const int32_t* tab = kv.block_table + (int64_t)c.layer * kv.table_stride_layer + (int64_t)c.seq * kv.max_blocks;
      for (int j = lane; j < kv.max_blocks; j += 32) bt_s[j] = __ldg(tab + j);
      __syncwarp();
      staged_seq = c.seq;
      staged_layer = c.layer;
    }
    const int nrows = min(rpb, c.end - c.i);
    char* kvb = c.kvk ? kv.base[1] : kv.base[0];
    unsigned char* stage = smem + s * kStageBytes;
    const char* src[kMaxRowsPerLane];
    uint32_t total = 0;
#pragma unroll
    for (int j = 0; j < kMaxRowsPerLane; ++j) {
      const int r = lane + 32 * j;
      src[j] = nullptr;
      bool ok = false;
      if (r < nrows) {
        const int i = c.i + r;
        const int from = pk[j];
        const int64_t dof = slot_offset(c.layer, c.seq, i);
        const char* from_ptr = nullptr;
        if (from >= c.stash_at && from < c.n_new) {  // saved before the copy: a later chunk overwrites it
          const int k = i - c.row0;
          if (k >= 0 && k < ck.stride)
            from_ptr = st.stash + ((size_t)(chunk + 1) * ck.stride + k) * rb;
        } else if (from >= i) {
          const int64_t so = slot_offset(c.layer, c.seq, from);
          if (so >= 0) from_ptr = kvb + (so + c.hg * piece_elems) * 2;
        }
        ok = from_ptr != nullptr && dof >= 0;
        if (ok) {
          src[j] = from_ptr;
          dptr[s][r] = kvb + (dof + c.hg * piece_elems) * 2;
        } else {
          dptr[s][r] = nullptr;
          set_error(st.err, from < i ? EPIKV_DEV_KEPT : EPIKV_DEV_SLOT);
        }
      }
      total += __popc(__ballot_sync(0xffffffffu, ok)) * (uint32_t)rb;
    }
    if (lane == 0) {
      stage_rows[s] = nrows;
      mbar_arrive_expect_tx(&full[s], total);
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < kMaxRowsPerLane; ++j)
      if (src[j]) tma_load_1d(stage + (lane + 32 * j) * rb, src[j], rb, &full[s]);
  };

  Cursor ld;
  if (balanced) {
    ld.u = o_begin < o_stop ? 0 : units;
    if (ld.u == 0) open_at(ld, o_begin);
  } else {
    ld.u = kLayers ? next_unit(0) : (int)blockIdx.x;
    load_unit(ld);
  }
  int pk[kMaxRowsPerLane];
  prefetch(ld, pk);
  int k_issue = 0, k_store = 0;
  bool timed_out = false;
  // the first loads go out before the wait, up to a batch with rows that
  // come from the stash
  auto wait_stash = [&] {
    pdl_wait();
    waited = true;
    if (ld.u < units && ld.stash_at != INT_MAX) ld.row0 = st.stash_row0[chunk + 1];
  };
  for (int p = 0; p < kStages - 1 && ld.u < units; ++p) {
    if (!waited) {
      bool stashed = false;
#pragma unroll
      for (int j = 0; j < kMaxRowsPerLane; ++j) stashed |= pk[j] >= ld.stash_at;
      if (__any_sync(0xffffffffu, stashed)) wait_stash();
    }
    issue(ld, pk, k_issue % kStages);
    ++k_issue;
    advance(ld);
    prefetch(ld, pk);
  }
  if (!waited) wait_stash();
  pdl_trigger();
  while (k_store < k_issue) {
    const int s = k_store % kStages;
    if (!mbar_wait_bounded(&full[s], (k_store / kStages) & 1, kWaitNs)) {
      timed_out = true;
      break;
    }
    __syncwarp();
    const int nrows = stage_rows[s];
    unsigned char* stage = smem + s * kStageBytes;
    for (int r = lane; r < nrows; r += 32)
      if (dptr[s][r]) tma_store_1d(dptr[s][r], stage + r * rb, rb);
    tma_commit();
    ++k_store;
    if (ld.u < units) {
      tma_wait_read<1>();  // the stage about to be refilled has been read out
      __syncwarp();
      issue(ld, pk, k_issue % kStages);
      ++k_issue;
      advance(ld);
      prefetch(ld, pk);    // its latency hides behind the next barrier wait
    }
  }
  if (timed_out) {
    if (lane == 0) set_error(st.err, EPIKV_DEV_TIMEOUT);
    // let the loads still in flight land before the CTA's shared memory goes away
    for (int k = k_store; k < k_issue; ++k)
      mbar_wait_bounded(&full[k % kStages], (k / kStages) & 1, kDrainNs);
  }
  tma_wait_all();
  if (kLayers && lane == 0) {
    // every CTA has fetched its last unit once all have counted in: the last resets
    __threadfence();
    if (atomicAdd(st.work + 1, 1u) == gridDim.x - 1) {
      st.work[0] = 0u;
      st.work[1] = 0u;
    }
  }
}

// The heads of the head and tail split, in place: a CTA per (entry, stream,
// head group) walks its rows in batches, all of a batch's loads before its
// stores (kept is increasing and kept[i] >= i, so a row's source is not
// written before its batch).  Rows are cut into pieces of 512 bytes or more
// until the units fill the grid twice.
__device__ void move_heads(const DevState& st, const Dims& dm, const KvDev& kv, const int32_t* __restrict__ seq_ids,
                           const int* list, const int64_t* pre, int n_ev, const int32_t* __restrict__ kept,
                           int kept_stride) {
  const int upe = 2 * dm.L, t = threadIdx.x;
  int hs = 1, vp = dm.H * dm.d / 8;   // pieces per row, 16-byte vectors per piece
  while ((int64_t)n_ev * upe * hs < 2 * (int64_t)gridDim.x && vp % 2 == 0 && vp / 2 >= 32) {
    hs *= 2;
    vp /= 2;
  }
  const int rows_max = min(kHeadUnroll * kStashThreads / vp, kMaxHeadRows);
  const int64_t units = (int64_t)n_ev * upe * hs;
  __shared__ const char* s_from[2][kMaxHeadRows];
  __shared__ char* s_to[2][kMaxHeadRows];
  int par = 0;
  for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
    const int k = (int)(u / (upe * hs)), b = list[k], seq = seq_ids[b];
    const int q = (int)(u / hs % upe), layer = q >> 1;
    char* base = (q & 1 ? kv.base[1] : kv.base[0]) + (int64_t)(u % hs) * vp * 16;
    const int32_t* kl = kept + (size_t)b * kept_stride;
    const int end = st.n_cache[seq] - (int)(pre[k + 1] - pre[k]);   // the tail's first row
    for (int i0 = st.first_changed[seq]; i0 < end; i0 += rows_max, par ^= 1) {
      const int rows = min(rows_max, end - i0);
      if (t < rows) {
        const int from = __ldg(kl + i0 + t);
        const int64_t so = from >= i0 + t ? kv_row_offset(kv, layer, seq, from, dm.T) : -1;
        const int64_t to = kv_row_offset(kv, layer, seq, i0 + t, dm.T);
        const bool ok = so >= 0 && to >= 0;
        if (!ok) set_error(st.err, from < i0 + t ? EPIKV_DEV_KEPT : EPIKV_DEV_SLOT);
        s_from[par][t] = ok ? base + so * 2 : nullptr;
        s_to[par][t] = ok ? base + to * 2 : nullptr;
      }
      __syncthreads();
      uint4 v[kHeadUnroll];
#pragma unroll
      for (int k = 0; k < kHeadUnroll; ++k) {
        const int e = t + k * kStashThreads, r = e / vp;
        if (r < rows && s_from[par][r]) v[k] = __ldcg(reinterpret_cast<const uint4*>(s_from[par][r]) + (e - r * vp));
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < kHeadUnroll; ++k) {
        const int e = t + k * kStashThreads, r = e / vp;
        if (r < rows && s_to[par][r]) *(reinterpret_cast<uint4*>(s_to[par][r]) + (e - r * vp)) = v[k];
      }
    }
  }
}

// Before a balanced compaction: where chunk g begins inside a stream (row a),
// CTA g saves into stash g the sources of the previous chunk's rows there
// that lie in [a, n_new) -- the region later chunks overwrite -- row by row
// from the first such row (stash_row0[g]).  Nothing of the cache is written,
// so every read sees the rows as the selection left them.
template <bool kLong>
__global__ void __launch_bounds__(kStashThreads, 2) compact_stash_kernel(DevState st, Dims dm, KvDev kv,
                                                                      const int32_t* __restrict__ seq_ids,
                                                                      int n_seq, const int32_t* __restrict__ kept,
                                                                      int kept_stride) {
  pdl_wait();
  // the counter of the copy's late chunks, which no CTA of the copy comes to
  // before its wait (kPrologueRows); under per-layer budgets the copy may take
  // units before that, and its last CTA leaves the counter at zero
  if (kLong && !dm.layer_budgets && blockIdx.x == 0 && threadIdx.x == 0) st.work[0] = 0u;
  extern __shared__ __align__(128) unsigned char smem[];
  int* list = reinterpret_cast<int*>(smem);
  int64_t* pre = reinterpret_cast<int64_t*>(list + list_ints(n_seq));
  const bool layers = dm.layer_budgets;
  const int sp = layers ? 2 : 2 * dm.L;  // streams per pair
  __shared__ int s_pairs, s_bal, s_heads;
  __shared__ int64_t s_rows;
  if (threadIdx.x < 32) {
    const int n_ev = evicting_entries(st, dm, seq_ids, n_seq, list, layers ? nullptr : pre, threadIdx.x);
    const int n_pairs = layers ? n_ev * dm.L : n_ev;
    int64_t rows = 0;
    if (!layers) rows = pre[n_ev];
    else if (n_pairs <= kMaxLayerPairs) rows = layer_pairs(st, dm, seq_ids, list, n_ev, pre, threadIdx.x);
    const int bal = n_ev > 0 && (!layers || n_pairs <= kMaxLayerPairs)
                        ? balanced_split(st, dm, seq_ids, list, n_ev, kept, kept_stride, layers, n_pairs, rows * sp,
                                         threadIdx.x)
                        : 0;
    const bool heads = n_ev > 0 && !layers && !bal &&
                       head_tail_split(st, dm, seq_ids, list, n_ev, kept, kept_stride, pre, threadIdx.x);
    if (threadIdx.x == 0) {
      s_heads = heads;
      s_pairs = n_pairs;
      s_rows = rows;
      s_bal = bal;
    }
  }
  __syncthreads();
  const int64_t total = s_rows * sp;
  if (s_heads) {
    move_heads(st, dm, kv, seq_ids, list, pre, s_pairs, kept, kept_stride);
    return;
  }
  // compact_kernel's CTAs are let in now, or as this kernel ends (kStashEarlyBytes)
  if (total * dm.H * dm.d * 4 <= kStashEarlyBytes) pdl_trigger();
  if (!s_bal) return;
  const int n_pairs = s_pairs;
  const Chunks<kLong> ck = make_chunks<kLong>(dm.stash_rows, total, gridDim.x, false, s_bal, kv.layout == EPIKV_LAYOUT_PAGED);
  __shared__ int s_src[kStashRows];  // the sources of rows lo .. a-1
  for (int g = blockIdx.x; g < ck.n; g += gridDim.x) {
    const int64_t o = ck.start(g);
    if (g == 0 || o >= total) continue;
    int p, q;
    int64_t r;
    locate_row(pre, n_pairs, sp, o, p, q, r);
    if (r == 0) continue;  // the chunk begins its stream: no other chunk reads its region
    const PairAt pa = pair_at(st, dm, seq_ids, list, kept, kept_stride, layers, p, q);
    const int seq = pa.seq, fe = pa.first, n_new = pa.n_new;
    const int a = fe + (int)r;
    const int32_t* kl = pa.kl;
    // the previous chunk's rows in this stream start at seg_start; those whose
    // sources lie in [a, n_new) are a suffix [i0, i1) of them, at most
    // stash_rows long (balanced_split), so inside [lo, a)
    const int64_t s0 = pre[p] * sp + (int64_t)q * (pre[p + 1] - pre[p]);
    const int64_t o_prev = ck.start(g - 1);
    const int seg_start = fe + (int)(o_prev > s0 ? o_prev - s0 : 0);
    const int lo = max(seg_start, a - ck.stride);
    const int t = threadIdx.x;
    if (kLong) __syncthreads();  // s_src is reused boundary after boundary
    const int src = t < a - lo ? __ldg(kl + lo + t) : INT_MAX;
    if (t < a - lo) s_src[t] = src;
    const int i0 = lo + __syncthreads_count(src < a);      // kept is increasing: counts of prefixes
    const int i1 = lo + __syncthreads_count(src < n_new);
    if (t == 0) st.stash_row0[g] = i0;
    const int x = i1 - i0;
    const int layer = pa.layer;
    const char* kvb = pa.kvk ? kv.base[1] : kv.base[0];
    const int v16 = dm.H * dm.d / 8;  // 16-byte vectors per row
    uint4* dst = reinterpret_cast<uint4*>(st.stash + (size_t)g * ck.stride * dm.H * dm.d * 2);
    // each warp copies two rows at a time, every lane's loads issued before its stores
    constexpr int kWarps = kStashThreads / 32;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    for (int r0 = warp; r0 < x; r0 += 2 * kWarps) {
      const int r1 = r0 + kWarps;
      const int64_t f0 = kv_row_offset(kv, layer, seq, s_src[i0 - lo + r0], dm.T);
      const int64_t f1 = r1 < x ? kv_row_offset(kv, layer, seq, s_src[i0 - lo + r1], dm.T) : -2;
      if ((f0 == -1 || f1 == -1) && lane == 0) set_error(st.err, EPIKV_DEV_SLOT);
      const uint4* p0 = reinterpret_cast<const uint4*>(kvb + f0 * 2);
      const uint4* p1 = reinterpret_cast<const uint4*>(kvb + f1 * 2);
      for (int k0 = lane; k0 < v16; k0 += kStashUnroll * 32) {
        uint4 v0[kStashUnroll], v1[kStashUnroll];
#pragma unroll
        for (int u = 0; u < kStashUnroll; ++u) {
          const int k = k0 + 32 * u;
          if (k < v16) {
            if (f0 >= 0) v0[u] = __ldg(p0 + k);
            if (f1 >= 0) v1[u] = __ldg(p1 + k);
          }
        }
#pragma unroll
        for (int u = 0; u < kStashUnroll; ++u) {
          const int k = k0 + 32 * u;
          if (k < v16) {
            if (f0 >= 0) dst[(size_t)r0 * v16 + k] = v0[u];
            if (f1 >= 0) dst[(size_t)r1 * v16 + k] = v1[u];
          }
        }
      }
    }
  }
}

// The batch entries' evictions have been applied: nothing is left pending.
__global__ void compact_consumed_kernel(DevState st, Dims dm, const int32_t* __restrict__ seq_ids, int n_seq) {
  // launched beside the copy, which does not write the lengths: they are
  // loaded before the wait
  const int per = dm.layer_budgets ? dm.L : 1;
  const int i = blockIdx.x * blockDim.x + threadIdx.x, b = i / per, l = i - b * per;
  const int seq = b < n_seq ? seq_ids[b] : -1;
  const bool ok = seq >= 0 && seq < dm.S;
  const int n = ok && l == 0 ? st.n_cache[seq] : 0;
  const int nl = ok && dm.layer_budgets ? st.n_layer[seq * dm.L + l] : 0;
  pdl_wait();
  pdl_trigger();
  if (!ok) return;
  if (l == 0) st.first_changed[seq] = n;
  if (dm.layer_budgets) st.lfirst[seq * dm.L + l] = nl;
}

static int g_ctas_per_sm = 0;

static size_t stash_smem(int n_seq, int L, bool layers) {
  return (size_t)list_ints(n_seq) * sizeof(int) + (size_t)pre_entries(pairs_cap(n_seq, L, layers)) * sizeof(int64_t);
}

static size_t compact_smem(int n_seq, int L, bool layers) {
  return (size_t)kStages * kStageBytes + stash_smem(n_seq, L, layers) + (size_t)kStagedBlocks * sizeof(int);
}

cudaError_t compact_prepare(int device, int* ctas_per_sm) {
  (void)device;
  // the largest batch's tables: token budgets take a prefix sum per sequence
  // (more than the kMaxLayerPairs of per-layer budgets)
  const int mx = (int)max(compact_smem(kMaxSeqs, 64, false), compact_smem(kMaxSeqs, 64, true));
  const int mx_stash = (int)max(stash_smem(kMaxSeqs, 64, false), stash_smem(kMaxSeqs, 64, true));
  cudaError_t e = cudaSuccess;
  auto allow = [&](auto kern) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, mx);
  };
  allow(compact_kernel<false, true, false>);
  allow(compact_kernel<false, true, true>);
  allow(compact_kernel<true, true, false>);
  allow(compact_kernel<true, true, true>);
  allow(compact_kernel<true, false, false>);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(compact_stash_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx_stash);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(compact_stash_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx_stash);
  if (e != cudaSuccess) return e;
  int n = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, compact_kernel<false, true, true>, 32, compact_smem(64, 32, false));
  if (e != cudaSuccess) return e;
  g_ctas_per_sm = n > 0 ? n : 1;
  if (EPIKV_COMPACT_CTAS_PER_SM > 0 && EPIKV_COMPACT_CTAS_PER_SM < g_ctas_per_sm)
    g_ctas_per_sm = EPIKV_COMPACT_CTAS_PER_SM;
  if (ctas_per_sm) *ctas_per_sm = g_ctas_per_sm;
  return cudaSuccess;
}

cudaError_t launch_compact(const DevState& st, const Dims& dm, int n_seq, const int32_t* seq_ids,
                           const int32_t* kept, int kept_stride, const KvDev& kv, int ctas,
                           cudaStream_t stream, int* launches) {
  if (n_seq == 0) return cudaSuccess;
  const bool layers = dm.layer_budgets;
  const bool split = !layers || n_seq * dm.L <= kMaxLayerPairs;  // the balanced split may apply
  const size_t smem = compact_smem(n_seq, dm.L, layers);
  const bool stash = split && ctas <= kMaxStashCtas;
  const bool longc = late_possible(n_seq, dm.T, dm.L, ctas);
  if (stash) {  // the balanced split's stash (the kernel checks whether it applies)
    auto go = [&](auto kern) {
      pdl_launch(kern, ctas, kStashThreads, stash_smem(n_seq, dm.L, layers), stream, st, dm, kv, seq_ids, n_seq, kept,
                 kept_stride);
    };
    if (longc) go(compact_stash_kernel<true>);
    else go(compact_stash_kernel<false>);
    ++*launches;
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  auto go = [&](auto kern) {
    if (stash)
      pdl_launch(kern, ctas, 32, smem, stream, st, dm, kv, seq_ids, n_seq, kept, kept_stride, 1);
    else
      plain_launch(kern, ctas, 32, smem, stream, st, dm, kv, seq_ids, n_seq, kept, kept_stride, 0);
  };
  if (!layers) longc ? go(compact_kernel<false, true, true>) : go(compact_kernel<false, true, false>);
  else if (split) longc ? go(compact_kernel<true, true, true>) : go(compact_kernel<true, true, false>);
  else go(compact_kernel<true, false, false>);
  ++*launches;
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int marks = n_seq * (layers ? dm.L : 1);
  pdl_launch(compact_consumed_kernel, (marks + 255) / 256, 256, 0, stream, st, dm, seq_ids, n_seq);
  ++*launches;
  return cudaGetLastError();
}

}  // namespace epikv
