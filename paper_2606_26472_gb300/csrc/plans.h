// The arithmetic of the compaction's chunks: how the copy kernel cuts its row
// space.  Plain C++ as well as device code, so that the plans that the
// kernels follow can be checked on the host as they stand here.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define EPIKV_PLAN __host__ __device__ __forceinline__
#else
#define EPIKV_PLAN inline
#endif

namespace epikv {

// The balanced compaction split: at most this many CTAs, each with a stash
// of at most kStashRows rows (the slots its left neighbour still reads).
constexpr int kMaxStashCtas = 512;
constexpr int kStashRows = 128;
constexpr int kMaxChunks = 1024;   // chunks of a split whose stashes need at most half those rows

#ifndef EPIKV_COMPACT_STAGES
#define EPIKV_COMPACT_STAGES 4
#endif
constexpr int kStages = EPIKV_COMPACT_STAGES;   // batches of rows that a CTA of the copy has in flight
constexpr int kMaxRowsPerLane = 4;
constexpr int kMaxRPB = 32 * kMaxRowsPerLane;   // rows per batch, at most

// Chunks of the balanced row space: one per CTA, and for long copies more,
// much shorter ones at its end, which the CTAs take as they finish: some SMs
// copy more slowly than others, always the same ones (8 x 4,160 contiguous
// slots in equal chunks: CTAs end between 1,131 and 1,328 us, median 1,195; a
// paged cache of 32 x 8,320: 9,643 to 9,986, median 9,796).  Each chunk that
// begins inside a stream needs a stash of `stride` rows, so a stashed split
// has at most as many chunks as the stash holds, and does this from kLateRows
// rows per CTA on, where the larger stash pays; the tails of the head and tail
// split need none.  Equal / late chunks, stash + copy in us:
//   contiguous (late chunks of 5 % of a CTA's share: 2 %, 3.5 %, 7 % 1,373,
//   1,298, 1,289): 8 x 4,160 slots 1,356 / 1,275, 20 x 8,100 6,418 / 6,135
//   paged (2 %, up to 768 chunks): 32 x 8,320 10,118 / 10,028, 8 x 4,160
//   1,316 / 1,299, 6 x 3,048 in chunks of 16 634 / 613, per-layer budgets
//   1,314 / 1,309
//   tails (2 %, eight per CTA): 65,536 + 38,940 + 12,345 to 4,096 slots 461 /
//   406 (copy), 9,000 to 3,000 97 / 106 (421 rows per CTA: not taken)
constexpr int kLateRows = 2048, kLateRowsTails = 768;
constexpr int kChunksPaged = 768;
constexpr int kLateContiguous = 50, kLatePaged = 20, kLateTails = 20;   // thousandths of a CTA's share
constexpr int kLatePerCta = 3, kLatePerCtaTails = 8;   // late chunks per CTA, at most (few CTAs: 15 % of the rows)

// Rows of the shortest chunk of a CTA's own (the first G chunks) in a split with
// late chunks: its share less what `per` late chunks per CTA of `part`
// thousandths take of it.  Whole divisions: never more than the kernels'.
constexpr int least_early_rows(int rows, int per, int part) { return rows - (rows * per * part + 999) / 1000 - 1; }

// Under token budgets the counter of the late chunks is zeroed by the stash
// kernel, which may still be running while the copy's CTAs load their first
// batches.  So no CTA may come to the end of its own chunk, and to that
// counter, within those kStages - 1 batches.
constexpr int kPrologueRows = (kStages - 1) * kMaxRPB;
static_assert(kPrologueRows < least_early_rows(kLateRowsTails, kLatePerCtaTails, kLateTails),
              "a tail's chunk could end before the copy has waited for the stash kernel");
static_assert(kPrologueRows < least_early_rows(kLateRows, kLatePerCta, kLateContiguous) &&
                  kPrologueRows < least_early_rows(kLateRows, kLatePerCta, kLatePaged),
              "a stashed chunk could end before the copy has waited for the stash kernel");

// kLong: the late chunks are compiled in.  The host takes the other instances
// for caches too small for them (late_possible): the code alone costs the
// smallest steps 1.6 us (512 slots 51.9 / 53.5 us, a 2,048-token trace 98.0 /
// 100.7).
template <bool kLong>
struct Chunks {
  int64_t total, early;   // rows, rows of the first G chunks
  int G, n;               // CTAs, chunks
  int stride;             // rows of a chunk's stash
  EPIKV_PLAN int64_t start(int c) const {
    if (!kLong) return total * c / G;
    return c <= G ? early * c / G : early + (total - early) * (c - G) / (n - G);
  }
};
template <bool kLong>
EPIKV_PLAN Chunks<kLong> make_chunks(int stash_rows, int64_t total, int G, bool tails, int stride, bool paged) {
  Chunks<kLong> k{total, total, G, G, stride};
  if (!kLong) return k;
  int late = 0;
  if (tails) {
    late = total >= (int64_t)kLateRowsTails * G ? kLatePerCtaTails * G : 0;
  } else if (total >= (int64_t)kLateRows * G) {
    const int cap = paged ? kChunksPaged : kMaxChunks, held = kMaxStashCtas * stash_rows / stride;
    late = (cap < held ? cap : held) - G;
    late = late < kLatePerCta * G ? late : kLatePerCta * G;
  }
  if (late > 0) {
    k.n = G + late;
    k.early = total - total * late / G * (tails ? kLateTails : paged ? kLatePaged : kLateContiguous) / 1000;
  }
  return k;
}

// Whether a batch of n_seq caches of `slots` slots and 2L streams can hold
// enough rows for late chunks.
inline bool late_possible(int n_seq, int slots, int L, int G) {
  return (int64_t)n_seq * slots * 2 * L >= (int64_t)(kLateRows < kLateRowsTails ? kLateRows : kLateRowsTails) * G;
}

}  // namespace epikv
