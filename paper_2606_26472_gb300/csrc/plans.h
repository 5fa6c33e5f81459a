// The arithmetic of the split kernels' plans: the chunks of the compaction's row
// space, the head and tail of a deep cut, the pieces of a long K/V score
// update.  Plain C++ as well as device code, so that the plans that the kernels
// follow can be checked on the host as they stand here.
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

// Rows of a chunk's stash, 0 if the balanced split does not apply: any chunk's
// own rows if none is longer than the stash, else the evictions' largest shift.
EPIKV_PLAN bool chunks_fit_stash(int64_t total, int G, int stash_rows) { return (total + G - 1) / G <= stash_rows; }
EPIKV_PLAN int shift_stride(int shift, int stash_rows) { return shift <= stash_rows ? shift : 0; }

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

// The first row in [first, n_new) of a kept list (at(i): its i-th slot) whose
// source is at or past n_new (n_new if none): an eight-way search, its probes
// loaded together.
template <typename At>
EPIKV_PLAN int tail_start(const At& at, int first, int n_new) {
  int lo = first, hi = n_new;
  while (lo < hi) {
    const int step = (hi - lo + 7) / 8;
    int below = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int i = lo + j * step < hi - 1 ? lo + j * step : hi - 1;
      below += at(i) < n_new;
    }
    if (below == 0) return lo;
    // the probes increase (and may repeat hi - 1): the answer lies after the
    // last one below n_new and not after the next one
    const int last = lo + (below - 1) * step < hi - 1 ? lo + (below - 1) * step : hi - 1;
    if (below < 8) hi = lo + below * step < hi - 1 ? lo + below * step : hi - 1;
    lo = last + 1;
  }
  return lo;
}

// Piece z of a K/V score update of n_new tokens starting at position p0, in
// pieces of `piece` tokens (a multiple of lag, at least 4 * lag; 0: one piece):
// the cuts lie at chunk boundaries, the first piece is two chunks shorter (it
// reads up to that much at the end of the call for the state), and the rows
// of the chunk before every cut belong to the call.
EPIKV_PLAN int lag_piece_start(int p0, int lag, int piece, int z) {
  return z == 0 ? 0 : (lag - p0 % lag) % lag + z * piece - 2 * lag;
}
// pieces that cover max_new tokens from any position
inline int lag_pieces(int max_new, int lag, int piece) {
  return piece ? (max_new + 2 * lag + piece - 1) / piece : 1;
}

#ifndef EPIKV_LAG_PIECE
#define EPIKV_LAG_PIECE 128  // shortest piece (tokens); never under 8 chunks, nor 4 in small calls
#endif
#ifndef EPIKV_LAG_CTAS
#define EPIKV_LAG_CTAS 56    // CTAs per SM wanted before pieces get longer: 8 rounds of 7 resident ones
#endif
// Tokens per piece of the K/V scoring kernel (lag_piece_start), 0 for one
// piece per stream.  One CTA per (layer, K|V, sequence) leaves a call of few
// sequences at one or two CTAs per SM, each a serial chain of loads: 4
// prompts of 4,099 to 517 tokens, 32 layers, took 695 us (1.7 TB/s), all six
// kinds of 2 prompts of 1,500 and 1,111 tokens 502 us.  Cut into pieces:
// 231 us (5.2 TB/s) and 125 us.  A piece re-reads the chunk before it (L2),
// so it has at least 8 chunks; 128 against 256 tokens 125 / 139 us on the
// second call, and 7, 14, 28, 100 CTAs per SM 274, 247, 234, 224 us on the
// first.  A call of less than two pieces stays whole (128 tokens of 32
// sequences fill the GPU as they are).
inline int lag_piece_tokens(int L, int lag_tokens, int n_seq, int max_new, int num_sms) {
  const int64_t lag = lag_tokens, streams = (int64_t)2 * L * n_seq;
  // half as long where whole pieces would not even fill one round of 7 CTAs
  // per SM: one prompt of 700 tokens 35 -> 29 us
  const bool few = streams * max_new < (int64_t)7 * num_sms * EPIKV_LAG_PIECE;
  const int64_t shortest = EPIKV_LAG_PIECE >> few, chunks = 8 >> few;
  const int64_t least = (shortest > chunks * lag ? (shortest + lag - 1) / lag * lag : chunks * lag);
  if (max_new < 2 * least) return 0;
  const int64_t want = (int64_t)EPIKV_LAG_CTAS * num_sms;
  const int64_t pieces = (want + streams - 1) / streams;
  int64_t piece = (max_new + pieces - 1) / pieces;
  piece = (piece + lag - 1) / lag * lag;
  if (piece < least) piece = least;
  return piece < max_new ? (int)piece : 0;
}

}  // namespace epikv
