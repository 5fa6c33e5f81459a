// Scoring kernels of the EpiKV hot path.
//
//   bandz_g_kernel         g_l(t) = ||h_l(t) - h_l(t-1)||_2 of every new token
//                          and band layer (Sec. 3.2, Eq. 1), streamed from the
//                          bf16 rows with 16-byte loads, fp32 accumulation.
//   lagkv_partial_kernel   Lag-KV (Sec. 3.3): each new token's K or V row of one
//                          layer, normalised by the previous chunk's per-channel
//                          range; population variance over the head dimension,
//                          summed over heads.  Keeps the running chunk ranges.
//   score_finalize_kernel  causal rolling z-score per band layer and the band
//                          combination (Eq. 3, Fig. 1); Lag-KV u(t) and its
//                          rolling mean; writes the frozen score and position of
//                          every new slot and commits the sequence's counters.
//
// Every result is independent of how a trace is split into calls: g values
// and u values are computed from the same bytes in the same order whether the
// previous row comes from the call or from the saved state, and the window
// reductions run over positions in a fixed lane order.
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace epikv {

#ifndef EPIKV_G_UNROLL
#define EPIKV_G_UNROLL 2  // tokens whose rows are loaded together (measured best: 2)
#endif
constexpr int kGThreads = 256;
constexpr int kGUnroll = EPIKV_G_UNROLL;
constexpr int kMaxTokPerCta = 32;  // tokens per run, between two block barriers: 116,822 tokens 2,011 us at 16, 1,996 at 32, 1,995 at 64

struct BandRows {
  const __nv_bfloat16* p[kMaxBand];
};

// Persistent grid; block: 256 threads.  The rows of the call, flattened as
// r = band * total_new + packed_row, are split into gridDim.x equal
// contiguous shares, so every CTA streams the same number of rows.  A CTA
// walks its share in runs that stay inside one (band layer, batch entry),
// kMaxTokPerCta tokens at most; the previous row of a run's first token is the last row
// of the run before it when they are consecutive, else it is loaded (from
// the saved h_prev for a sequence's first new token).
template <int VPT>
#ifndef EPIKV_G_MINB
#define EPIKV_G_MINB 0  // 0: by register need
#endif
__global__ void __launch_bounds__(kGThreads, (EPIKV_G_MINB > 0 ? EPIKV_G_MINB : VPT * kGUnroll >= 16 ? 2 : 4)) bandz_g_kernel(DevState st, Dims dm, BandRows rows,
                                                            int64_t row_stride,
                                                            const int32_t* __restrict__ seq_ids,
                                                            const int32_t* __restrict__ cu_new, int n_seq,
                                                            int max_new) {
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // the whole batch must be well formed, else nothing is read
  __shared__ int bad;
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int b = tid; b < n_seq; b += kGThreads) {
    const int seq = seq_ids[b], n = cu_new[b + 1] - cu_new[b];
    if (seq < 0 || seq >= dm.S || n < 0 || n > max_new || cu_new[0] != 0) bad = 1;
  }
  __syncthreads();
  if (bad) {
    if (tid == 0 && blockIdx.x == 0) set_error(st.err, EPIKV_DEV_BATCH);
    return;
  }
  const int nb = dm.nA + dm.nB;
  const int total = cu_new[n_seq];
  const int64_t R = (int64_t)nb * total;
  int64_t r = R * blockIdx.x / gridDim.x;
  const int64_t r_end = R * (blockIdx.x + 1) / gridDim.x;
  if (r >= r_end) return;
  const int VR = dm.D >> 3;  // 16-byte vectors per row
  __shared__ float red[kMaxTokPerCta][kGThreads / 32];  // per token of a run, per warp

  int band = (int)(r / total), row = (int)(r - (int64_t)band * total);
  int b = 0;  // batch entry holding `row` (largest b with cu_new[b] <= row and a token)
  {
    int lo = 0, hi = n_seq - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (cu_new[mid] <= row) lo = mid; else hi = mid - 1;
    }
    b = lo;
    while (cu_new[b + 1] <= row) ++b;  // skip empty entries
  }
  uint4 prev[VPT];
  int prev_band = -1, prev_row = -1;  // what `prev` holds
  while (r < r_end) {
    const int r0 = cu_new[b], n_new = cu_new[b + 1] - r0;
    const int seq = seq_ids[b];
    const int t0 = row - r0;
    const int len = (int)min((int64_t)min(kMaxTokPerCta, n_new - t0), r_end - r);
    const int t1 = t0 + len;
    const int p0 = st.n_seen[seq];
    const int par = st.hp_parity[seq];
    const __nv_bfloat16* base = rows.p[band];
    if (!(prev_band == band && prev_row == row - 1 && t0 > 0)) {
      const __nv_bfloat16* prow = t0 == 0 ? st.h_prev + ((size_t)(seq * 2 + par) * nb + band) * dm.D
                                          : base + (int64_t)(row - 1) * row_stride;
#pragma unroll
      for (int k = 0; k < VPT; ++k) {
        const int v = tid + k * kGThreads;
        prev[k] = v < VR ? ld_stream16(prow + v * 8) : make_uint4(0, 0, 0, 0);
      }
    }
    for (int t = t0; t < t1; t += kGUnroll) {
      uint4 cur[kGUnroll][VPT];
#pragma unroll
      for (int u = 0; u < kGUnroll; ++u) {
        const __nv_bfloat16* rp = base + (int64_t)(r0 + t + u) * row_stride;
#pragma unroll
        for (int k = 0; k < VPT; ++k) {
          const int v = tid + k * kGThreads;
          cur[u][k] = (t + u < t1 && v < VR) ? ld_stream16(rp + v * 8) : make_uint4(0, 0, 0, 0);
        }
      }
#pragma unroll
      for (int u = 0; u < kGUnroll; ++u) {
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < VPT; ++k) {
          float c[8], p[8];
          unpack8(cur[u][k], c);
          unpack8(u == 0 ? prev[k] : cur[u - 1][k], p);
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float dlt = c[e] - p[e];
            acc = fmaf(dlt, dlt, acc);
          }
        }
        acc = warp_sum(acc);
        if (lane == 0 && t + u < t1) red[t - t0 + u][warp] = acc;
      }
      // the last valid row of this group is the previous row of the next group
      const int last = min(kGUnroll, t1 - t) - 1;
#pragma unroll
      for (int u = 0; u < kGUnroll; ++u)
        if (u == last) {
#pragma unroll
          for (int k = 0; k < VPT; ++k) prev[k] = cur[u][k];
        }
    }
    __syncthreads();
    if (tid < len) {
      float sum = 0.f;
#pragma unroll
      for (int w = 0; w < kGThreads / 32; ++w) sum += red[tid][w];
      const int pos = p0 + t0 + tid;
      if (pos >= 1) st.g_ring[((size_t)seq * nb + band) * dm.G + (pos & (dm.G - 1))] = sqrtf(sum);
    }
    if (t1 == n_new) {  // the sequence's last new row of this band is the next call's previous row
      __nv_bfloat16* hp_wr = st.h_prev + ((size_t)(seq * 2 + (par ^ 1)) * nb + band) * dm.D;
#pragma unroll
      for (int k = 0; k < VPT; ++k) {
        const int v = tid + k * kGThreads;
        if (v < VR) *reinterpret_cast<uint4*>(hp_wr + v * 8) = prev[k];
      }
    }
    __syncthreads();  // red is reused by the next run
    prev_band = band;
    prev_row = row + len - 1;
    r += len;
    row += len;
    if (row == total) {
      row = 0;
      ++band;
      b = 0;
    }
    while (b < n_seq && cu_new[b + 1] <= row) ++b;
  }
}

#ifndef EPIKV_LAG_SEG
#define EPIKV_LAG_SEG 8
#endif
#ifndef EPIKV_LAG_MINB
#define EPIKV_LAG_MINB 3  // with EPIKV_LAG_MAXREG 0: registers capped at 80
#endif
#ifndef EPIKV_LAG_PF
#define EPIKV_LAG_PF 1  // measured: 1 segment ahead 110 us, none 115 us, 2 ahead 119 us
#endif
constexpr int kLagSeg = EPIKV_LAG_SEG;  // tokens per segment (never crosses a chunk boundary)
constexpr int kLagPf = EPIKV_LAG_PF;    // a row is prefetched into L2 this many segments ahead
constexpr int kLagOffs = 256;   // slot offsets looked up per group of tokens

// The previous chunk's range as a per-channel affine map y = x * a + c with
// a = 1 / (max - min + eps) and c = -min * a - 1/2, so that y = x~ - 1/2 for
// the range-normalised x~ (one fused multiply-add per channel).
__device__ __forceinline__ void prev_affine(const uint4& pmn, const uint4& pmx, float eps, f32x2 (&a)[4],
                                            f32x2 (&c)[4]) {
  float mn[8], mx[8], inv[8], bias[8];
  unpack8(pmn, mn);
  unpack8(pmx, mx);
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    inv[e] = __frcp_rn(mx[e] - mn[e] + eps);   // the correctly rounded reciprocal (as 1.f / x)
    bias[e] = fmaf(-mn[e], inv[e], -0.5f);
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    a[p] = f2_pack(inv[2 * p], inv[2 * p + 1]);
    c[p] = f2_pack(bias[2 * p], bias[2 * p + 1]);
  }
}

// Sums of y and y^2 over one thread's 8 channels of a token row.
__device__ __forceinline__ void lag_moments(const uint4& x, const f32x2 (&a)[4], const f32x2 (&c)[4], float& s1,
                                            float& s2) {
  const f32x2 y0 = f2_fma(bf16x2_to_f2(x.x), a[0], c[0]);
  const f32x2 y1 = f2_fma(bf16x2_to_f2(x.y), a[1], c[1]);
  const f32x2 y2 = f2_fma(bf16x2_to_f2(x.z), a[2], c[2]);
  const f32x2 y3 = f2_fma(bf16x2_to_f2(x.w), a[3], c[3]);
  const f32x2 t = f2_add(f2_add(y0, y1), f2_add(y2, y3));
  f32x2 u = f2_mul(y0, y0);
  u = f2_fma(y1, y1, u);
  u = f2_fma(y2, y2, u);
  u = f2_fma(y3, y3, u);
  s1 = f2_lo(t) + f2_hi(t);
  s2 = f2_lo(u) + f2_hi(u);
}

// grid: (2L (layer, K|V), batch entries); block: max(32, H*d/8) threads;
// LH = d/8 consecutive lanes own one head, 8 channels each.
//
// Tokens are taken in segments that stay inside one chunk: every token of a
// segment is normalised with the same previous-chunk range, so the segment's
// reductions are independent of one another.  Chunk ranges (min, max) are
// bf16 values and are kept packed (exact).  The variance of a token's head
// is taken from the moments of y = x~ - 1/2 (x~ in [0, 1] inside the range),
// computed two channels per instruction (f32x2); the segment's 2 x 8 moments
// are summed over the head's lanes by one transposed reduction into shared
// memory, where a thread per token forms each head's variance.
//
// The stream's work is lag_stream, which the one-token decode kernel
// (token_kernel) runs unchanged for its K/V CTAs.
// SEG is the longest segment: kLagSeg, or 1 for one-token calls (fewer
// registers; the reductions pair lanes in the same order either way, so the
// sums are the same bit for bit).  With HALF, each half of a 256-thread
// block runs its own stream (K in the first half, V in the second; H*d/8 <=
// 128), with its own shared memory.
// KINDS: 0 = whichever K/V kinds the context computes (runtime flags); 1 =
// the normalised kinds only; 2 = the raw kinds only (compile-time, so a
// kernel instance holds only the registers its kinds need).
#ifndef EPIKV_TOKEN_OWN_OFFSET
#define EPIKV_TOKEN_OWN_OFFSET 1  // 0: one-token calls also look the row up through shared memory
#endif
//
// The stream's tokens [t_lo, t_hi) of the call's n_new are taken: all of them,
// or (SPLIT) one piece of a long call, cut at chunk boundaries by
// lag_piece_start so that few sequences still fill the GPU.  A later piece forms
// its first chunk's previous range from that chunk's rows (bf16 minima and
// maxima, the same in any order) and leaves the saved state alone; the first
// piece, the only one that reads the state, also writes the state that the
// whole call leaves, from the call's last rows.
template <int LH, int SEG = kLagSeg, bool HALF = false, int KINDS = 0, bool SPLIT = false>
__device__ __forceinline__ void lag_stream(const DevState& st, const Dims& dm, const KvDev& kv, int seq,
                                           int t_lo, int t_hi, int n_new, int layer, int kvk, int nc0) {
  const int stream = layer * 2 + kvk;  // this stream's column of the per-token partials
  const int tid = HALF ? (int)(threadIdx.x & 127) : (int)threadIdx.x;
  const int nthr = HALF ? 128 : (int)blockDim.x;
  const int half = HALF ? kvk : 0;
  const int h = tid / LH, q = tid % LH;
  const bool active = h < dm.H;
  const int hd = dm.H * dm.d;
  const int p0 = st.n_seen[seq];
  const int ch = h * dm.d + q * 8;  // first channel of this thread within the token row
  const bool need_norm = KINDS ? (KINDS & 1) != 0 : (dm.kinds & kNormKinds) != 0;   // uniform across the grid
  const bool need_raw = KINDS ? (KINDS & 2) != 0 : (dm.kinds & kRawKinds) != 0;
  __nv_bfloat16* rng = need_norm ? st.lag_rng + ((((size_t)seq * dm.L + layer) * 2 + kvk) * 4) * hd : nullptr;

  // the previous chunk's range lives on only as its affine map; it is written
  // back as soon as a chunk completes, the running range at the end
  uint4 cmn = make_uint4(0, 0, 0, 0), cmx = cmn;
  f32x2 na[4], nc[4];
  {
    uint4 pmn = cmn, pmx = cmn;
    if (active && need_norm && !(SPLIT && t_lo > 0)) {
      pmn = *reinterpret_cast<const uint4*>(rng + 0 * hd + ch);
      pmx = *reinterpret_cast<const uint4*>(rng + 1 * hd + ch);
      cmn = *reinterpret_cast<const uint4*>(rng + 2 * hd + ch);
      cmx = *reinterpret_cast<const uint4*>(rng + 3 * hd + ch);
    }
    prev_affine(pmn, pmx, dm.lag_eps, na, nc);
  }

  const float inv_d = 1.f / (float)dm.d;
  const char* kvbase = kvk ? kv.base[1] : kv.base[0];  // a select: no local copy of the parameter struct
  const char* kvb_ch = kvbase + (int64_t)ch * 2;       // this thread's first channel in a row at offset 0
  __shared__ int64_t soff_s[HALF ? 2 : 1][kLagOffs];
  int64_t* soff = soff_s[half];
  const bool whole = !SPLIT || (t_lo == 0 && t_hi == n_new);   // the call's only piece of this stream

  // minimum and maximum of this thread's channels over the call's tokens [a, b), a < b
  auto range_of = [&](int a, int b, uint4& mn, uint4& mx) {
    bool first = true;
    for (int g0 = a; g0 < b; g0 += kLagOffs) {
      const int gn = min(kLagOffs, b - g0);
      __syncthreads();
      for (int t = tid; t < gn; t += nthr) soff[t] = kv_row_offset(kv, layer, seq, nc0 + g0 + t, dm.T);
      __syncthreads();
      for (int i = 0; i < gn; i += kLagSeg) {
        uint4 x[kLagSeg];
#pragma unroll
        for (int j = 0; j < kLagSeg; ++j) {   // past the end: the last row again
          const int64_t off = soff[min(i + j, gn - 1)];
          x[j] = ld_stream16_if(kvb_ch + off * 2, active && off >= 0);
        }
        if (first) mn = mx = x[0];
        first = false;
#pragma unroll
        for (int j = 0; j < kLagSeg; ++j) {
          mn = q_min(mn, x[j]);
          mx = q_max(mx, x[j]);
        }
      }
    }
  };

  if (SPLIT && t_lo > 0 && need_norm) {
    uint4 pmn, pmx;
    range_of(t_lo - dm.lag, t_lo, pmn, pmx);
    prev_affine(pmn, pmx, dm.lag_eps, na, nc);
  }
  constexpr int NV = 2 * SEG;      // moments of a segment: (sum y, sum y^2) per token
  __shared__ float red_s[HALF ? 2 : 1][2][32][NV];  // [half][segment parity][head][moment]; the host admits H <= 32
  __shared__ float hr_s[HALF ? 2 : 1][2][SEG][32];  // raw variances, same layout
  float (*red)[32][NV] = red_s[half];
  float (*hr)[SEG][32] = hr_s[half];
  float* part = need_norm ? st.lag_part + (size_t)seq * dm.max_new * (2 * dm.L) : nullptr;
  float* rpart = need_raw ? st.raw_part + (size_t)seq * dm.max_new * (2 * dm.L) : nullptr;
  // this stream's partials: [stream][token], so that neighbouring tokens'
  // lie together for score_finalize_kernel; a decode step's one token
  // [stream], for kv_token_scores
  const size_t part0 = SEG == 1 ? (size_t)stream : (size_t)stream * dm.max_new;
  int r = (p0 + t_lo) % dm.lag;          // position of the next token inside its chunk
  int parity = 0;

  for (int g0 = t_lo; g0 < t_hi; g0 += kLagOffs) {
    const int gn = min(kLagOffs, t_hi - g0);
    // one-token calls: every thread looks its row up itself (one broadcast
    // load per warp), so no shared table and none of its two barriers.  The
    // SEG == 1 instances run only in the decode-step kernel, whose calls
    // carry one token per sequence (it rejects n_new > 1), so the group holds
    // that one row.
    int64_t off1 = 0;
    if constexpr (SEG == 1 && EPIKV_TOKEN_OWN_OFFSET) {
      off1 = kv_row_offset(kv, layer, seq, nc0 + g0, dm.T);
    } else {
      __syncthreads();
      for (int t = tid; t < gn; t += nthr) soff[t] = kv_row_offset(kv, layer, seq, nc0 + g0 + t, dm.T);
      __syncthreads();
    }
    // rows are prefetched into L2 kLagPf segments ahead of their loads (whole
    // rows of H*d channels, one bulk prefetch each); the group's first ones here
    const uint32_t row_bytes = (uint32_t)hd * 2u;
    if constexpr (SEG > 1 && kLagPf > 0) {
      for (int t = tid; t < min(kLagPf * SEG, gn); t += nthr)
        if (soff[t] >= 0) prefetch_l2_bulk(kvbase + soff[t] * 2, row_bytes);
    }
    for (int i = 0; i < gn;) {
      const int seg = min(min(dm.lag - r, gn - i), SEG);
      const bool has_prev = p0 + g0 + i >= dm.lag;   // the segment's chunk is not chunk 0
      uint4 x[SEG];
      // FULL: every token of the segment is taken (the common case), so the
      // per-token conditions compile away; the arithmetic is the same
      auto body = [&](auto full_t, auto mom_t) {
        constexpr bool FULL = decltype(full_t)::value;
        constexpr bool MOM = decltype(mom_t)::value;  // has_prev && need_norm: the normalised moments
        int64_t offs[SEG];
        bool all_ok = active;
#pragma unroll
        for (int j = 0; j < SEG; ++j) {
          if constexpr (SEG == 1 && EPIKV_TOKEN_OWN_OFFSET) offs[j] = off1;
          else offs[j] = (FULL || j < seg) ? soff[i + j] : 0;
          all_ok &= offs[j] >= 0;
        }
        if (FULL && all_ok) {  // every row of the segment mapped: plain loads
#pragma unroll
          for (int j = 0; j < SEG; ++j) x[j] = ld_stream16(kvb_ch + offs[j] * 2);
        } else {
          bool bad = false;
#pragma unroll
          for (int j = 0; j < SEG; ++j) {
            const bool take = (FULL || j < seg) && active;
            bad |= take && offs[j] < 0;
            x[j] = ld_stream16_if(kvb_ch + offs[j] * 2, take && offs[j] >= 0);
          }
          if (bad) set_error(st.err, EPIKV_DEV_SLOT);
        }
        if constexpr (SEG > 1 && kLagPf > 0) {  // rows [i + kLagPf*SEG, + seg): every row once over the group
          const int t = i + kLagPf * SEG + tid;
          if (tid < seg && t < gn && soff[t] >= 0) prefetch_l2_bulk(kvbase + soff[t] * 2, row_bytes);
        }
        // the raw kinds, four tokens at a time (absent ones give unused
        // sums): population variances of the stored vectors over the head
        // dimension, two transposed reductions instead of eight butterflies
        if constexpr (SEG % 4 == 0) {
          if (need_raw) {
#pragma unroll
            for (int j0 = 0; j0 < SEG; j0 += 4) {
              float rv[4], tot[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                float xf[8], s1 = 0.f;
                unpack8(x[j0 + j], xf);
#pragma unroll
                for (int e = 0; e < 8; ++e) s1 += xf[e];
                rv[j] = s1;
              }
              group_totals<LH>(rv, tid & 31, tot);
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                float xf[8], s2 = 0.f;
                unpack8(x[j0 + j], xf);
                const float mean = tot[j] * inv_d;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                  const float dv = xf[e] - mean;
                  s2 = fmaf(dv, dv, s2);
                }
                rv[j] = s2;
              }
              transpose_sum<LH / 2, 4, 4>(rv, tid & 31);
              if (active) {
                if constexpr (LH <= 4) {
#pragma unroll
                  for (int k = 0; k < 4 / LH; ++k) hr[parity][j0 + k + (4 / LH) * q][h] = rv[k] * inv_d;
                } else {
                  if (q % (LH / 4) == 0) hr[parity][j0 + q / (LH / 4)][h] = rv[0] * inv_d;
                }
              }
            }
          }
        }
        // two tokens at a time, so that rows' registers are free once used:
        // their normalised moments, then the running range over both (the
        // same min/max sequence as token by token)
        float v[NV];
        if (r == 0) {
          cmn = x[0];
          cmx = x[0];
        }
#pragma unroll
        for (int j0 = 0; j0 < SEG; j0 += 2) {
#pragma unroll
          for (int j = j0; j < j0 + 2 && j < SEG; ++j) {
            if (FULL || j < seg) {
              if (SEG % 4 != 0 && need_raw) {  // population variance of the stored vector over the head dimension
                float xf[8], s1 = 0.f;
                unpack8(x[j], xf);
#pragma unroll
                for (int e = 0; e < 8; ++e) s1 += xf[e];
                const float mean = group_sum(s1, LH) * inv_d;
                float s2 = 0.f;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                  const float dv = xf[e] - mean;
                  s2 = fmaf(dv, dv, s2);
                }
                const float var_raw = group_sum(s2, LH) * inv_d;
                if (q == 0 && active) hr[parity][j][h] = var_raw;
              }
              if constexpr (MOM) lag_moments(x[j], na, nc, v[2 * j], v[2 * j + 1]);
            } else if constexpr (MOM) {
              v[2 * j] = v[2 * j + 1] = 0.f;
            }
          }
          if (j0 + 1 < SEG && (FULL || j0 + 1 < seg)) {
            cmn = q_min(q_min(cmn, x[j0]), x[j0 + 1]);
            cmx = q_max(q_max(cmx, x[j0]), x[j0 + 1]);
          } else if (FULL || j0 < seg) {
            cmn = q_min(cmn, x[j0]);
            cmx = q_max(cmx, x[j0]);
          }
        }
        if constexpr (MOM) {
          transpose_sum<LH / 2, NV, NV>(v, tid & 31);
          if (active) {
            if constexpr (LH <= NV) {
#pragma unroll
              for (int k = 0; k < NV / LH; ++k) red[parity][h][k + (NV / LH) * q] = v[k];
            } else {
              if (q % (LH / NV) == 0) red[parity][h][q / (LH / NV)] = v[0];
            }
          }
        }
      };
      if (has_prev && need_norm) {
        if (seg == SEG) body(std::true_type{}, std::true_type{});
        else body(std::false_type{}, std::true_type{});
      } else {
        if (seg == SEG) body(std::true_type{}, std::false_type{});
        else body(std::false_type{}, std::false_type{});
      }
      __syncthreads();
      if (tid < seg) {
        if (need_norm) {
          float sum = 0.f;
          if (has_prev)
            for (int hh = 0; hh < dm.H; ++hh) {
              const float mean = red[parity][hh][2 * tid] * inv_d;
              sum += fmaxf(fmaf(-mean, mean, red[parity][hh][2 * tid + 1] * inv_d), 0.f);
            }
          part[part0 + g0 + i + tid] = sum;
        }
        if (need_raw) {
          float sum = 0.f;
          for (int hh = 0; hh < dm.H; ++hh) sum += hr[parity][tid][hh];
          rpart[part0 + g0 + i + tid] = sum;
        }
      }
      parity ^= 1;
      r += seg;
      if (r == dm.lag) {  // chunk complete: it becomes the previous chunk
        prev_affine(cmn, cmx, dm.lag_eps, na, nc);
        if (active && need_norm && whole) {
          *reinterpret_cast<uint4*>(rng + 0 * hd + ch) = cmn;
          *reinterpret_cast<uint4*>(rng + 1 * hd + ch) = cmx;
        }
        r = 0;
      }
      i += seg;
    }
  }
  if (SPLIT && !whole) {
    if (t_lo > 0 || !need_norm) return;
    // the state after the call's last token: its last complete chunk's range
    // and the running one (all of these rows are the call's, lag_piece_start)
    const int tail = (p0 + n_new) % dm.lag, tc = n_new - tail;
    uint4 pmn, pmx;
    range_of(tc - dm.lag, tc, pmn, pmx);
    cmn = pmn;
    cmx = pmx;
    if (tail) range_of(tc, n_new, cmn, cmx);
    if (active) {
      *reinterpret_cast<uint4*>(rng + 0 * hd + ch) = pmn;
      *reinterpret_cast<uint4*>(rng + 1 * hd + ch) = pmx;
    }
  }
  if (active && need_norm) {
    *reinterpret_cast<uint4*>(rng + 2 * hd + ch) = cmn;
    *reinterpret_cast<uint4*>(rng + 3 * hd + ch) = cmx;
  }
}

#ifndef EPIKV_LAG_MAXREG
#define EPIKV_LAG_MAXREG 72  // 7 CTAs of 128 threads per SM: 2,048 CTAs in two rounds (measured best; 64 spills)
#endif
#ifndef EPIKV_LAG_RAWREG
// with the raw kinds: 96, five CTAs per SM.  Prompts of 1,500 and 1,111 tokens,
// 32 layers, at 72 / 80 / 96 / 128 registers: the raw kinds alone 67 / 66 / 62
// / 79 us (342 MB: 5.5 TB/s), all K/V kinds 135 / 126 / 109 / 119 us (72 and
// 80 spill); 125 us for all with a butterfly per sum instead of the
// transposed reductions
#define EPIKV_LAG_RAWREG 96
#endif
#if EPIKV_LAG_MAXREG > 0
#define EPIKV_LAG_BOUNDS __maxnreg__(KINDS == 1 ? EPIKV_LAG_MAXREG : EPIKV_LAG_RAWREG)
#else
#define EPIKV_LAG_BOUNDS __launch_bounds__(256, EPIKV_LAG_MINB)
#endif
// SPLIT: the instance that takes calls in pieces (the other keeps the
// registers of one piece).
template <int LH, int KINDS, bool SPLIT>
__global__ void EPIKV_LAG_BOUNDS lagkv_partial_kernel(DevState st, Dims dm, KvDev kv,
                                                             const int32_t* __restrict__ seq_ids,
                                                             const int32_t* __restrict__ cu_new,
                                                             int max_new, int piece, int beside_g) {
  // beside_g: launched programmatically after bandz_g_kernel, which lets this
  // kernel in after its own wait and writes nothing that is read here.  The
  // two run beside each other (one is bound by its loads, the other by its
  // instructions: all six kinds of 1,500 and 1,111 tokens 183.5 -> 181.6 us a
  // call), and every CTA waits before it ends, so that the finalize kernel,
  // which waits for this one, follows both.
  if (!beside_g) pdl_wait();
  pdl_trigger();
  struct WaitAtEnd {
    bool on;
    __device__ ~WaitAtEnd() {
      if (on) pdl_wait();
    }
  } at_end{beside_g != 0};
  const int b = blockIdx.y;
  const int seq = seq_ids[b];
  const int n_new = cu_new[b + 1] - cu_new[b];
  if (seq < 0 || seq >= dm.S || n_new < 0 || n_new > max_new) {
    if (threadIdx.x == 0) set_error(st.err, EPIKV_DEV_BATCH);
    return;
  }
  const int layer = blockIdx.x >> 1, kvk = blockIdx.x & 1;
  // the new rows' first slot: this layer's own length under per-layer budgets
  const int nc0 = dm.layer_budgets ? st.n_layer[seq * dm.L + layer] : st.n_cache[seq];
  if (nc0 + n_new > dm.T) {
    if (threadIdx.x == 0) set_error(st.err, EPIKV_DEV_CAPACITY);
    return;
  }
  int t_lo = 0, t_hi = n_new;
  if (SPLIT) {
    const int p0 = st.n_seen[seq], z = blockIdx.z;
    t_lo = lag_piece_start(p0, dm.lag, piece, z);
    t_hi = min(n_new, lag_piece_start(p0, dm.lag, piece, z + 1));
    if (t_lo >= n_new && z > 0) return;
  }
  lag_stream<LH, kLagSeg, false, KINDS, SPLIT>(st, dm, kv, seq, t_lo, t_hi, n_new, layer, kvk, nc0);
}

// A band's statistics over a window of n values of g, newest first (row[0],
// row[STEP], row[2 * STEP], ...), each a sum in that order by one thread: z of
// the newest value (Eq. 3; a shifted two-pass, so that a constant window gives
// exactly 0) and the window's mean (Eq. 2).  The values are taken from shared
// memory B at a time, so that the sums wait on their own additions and not on
// a load each (a decode step of 4 sequences 5.6 -> 5.3 us with the early row
// loads below; in token_kernel, at 48 registers, B = 1 measured best: 242.5
// us per 64-sequence call, 4 and 8 244 and 246).
template <int STEP, int B, typename F>
__device__ __forceinline__ void window_each(const float* row, int n, F&& f) {
  int k = 0;
  for (; k + B <= n; k += B) {
    float v[B];
#pragma unroll
    for (int j = 0; j < B; ++j) v[j] = row[(k + j) * STEP];
#pragma unroll
    for (int j = 0; j < B; ++j) f(v[j]);
  }
  for (; k < n; ++k) f(row[k * STEP]);
}

template <int STEP, int B = 16>
__device__ __forceinline__ float window_z(const float* row, int n, float eps) {
  const float gnew = row[0];
  float dsum = 0.f;
  window_each<STEP, B>(row, n, [&](float v) { dsum += v - gnew; });
  const float mean_d = dsum / (float)n;
  float dev = 0.f;
  window_each<STEP, B>(row, n, [&](float v) {
    const float e = (v - gnew) - mean_d;
    dev = fmaf(e, e, dev);
  });
  const float sigma = sqrtf(dev / (float)n);
  return -mean_d / (sigma + eps);  // g(t) - mu = -(mean of g - g(t))
}

template <int STEP, int B = 16>
__device__ __forceinline__ float window_mean(const float* row, int n) {
  float sum = 0.f;
  window_each<STEP, B>(row, n, [&](float v) { sum += v; });
  return sum / (float)n;
}

// Takes a ticket: what the CTA wrote before its last barrier is released to,
// and what the CTAs with earlier tickets released is acquired from, the whole
// GPU.  One thread; the others follow it through a barrier.  Two
// __threadfence around a relaxed atomic took 0.6 us longer (a decode step of
// 4 sequences 5.3 -> 4.7 us).
__device__ __forceinline__ uint32_t ticket_add(uint32_t* t) {
  uint32_t old;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(t) : "memory");
  return old;
}

#ifndef EPIKV_FIN_MINB
// CTAs per SM of the finalize kernel in calls of many tiles: registers capped
// at 40.  8 prompts of 4,000 tokens at no cap (74) / 4 / 5 / 6 / 8 CTAs 50 /
// 39 / 31 / 30 / 27 us, 4 prompts of 4,099 to 517 24 / 19 / 16 / 14 / 16.
// Calls whose tiles are all resident at three CTAs per SM take the instance
// with the registers for that: a step of 64 new tokens 53.0 -> 49.8 us, 2,048 100.0 -> 94.9.
#define EPIKV_FIN_MINB 6
#endif
constexpr int kFinFree = 3;   // CTAs per SM of the other instance
#ifndef EPIKV_FIN_TILE
#define EPIKV_FIN_TILE 16
#endif
constexpr int kFinTile = EPIKV_FIN_TILE;  // tokens per finalize CTA
constexpr int kFinThreads = 256;
constexpr int kMaxWindow = 1024;

// grid: (token tiles, batch entries, parts: the band kinds, then each K/V kind);
// block: 256 threads (a warp per token for the K/V kinds).
template <int WPL, bool kMany>
__global__ void __launch_bounds__(kFinThreads, kMany ? EPIKV_FIN_MINB : kFinFree) score_finalize_kernel(DevState st, Dims dm,
                                                                     const int32_t* __restrict__ seq_ids,
                                                                     const int32_t* __restrict__ cu_new,
                                                                     int max_new) {
  // the kernel before this one is the call's own g or K/V kernel, which was
  // let in after the caller's work and writes nothing of this: loaded before
  // the wait (with the selection's own a step of 64 tokens 50.6 ->
  // 48.1 us)
  const int b = blockIdx.y;
  const int seq = seq_ids[b];
  const int n_new = cu_new[b + 1] - cu_new[b];
  const bool good = seq >= 0 && seq < dm.S && n_new >= 0 && n_new <= max_new;
  const int nc0 = good ? st.n_cache[seq] : 0;
  const int p0 = good ? st.n_seen[seq] : 0;
  const int first = good ? st.first_changed[seq] : 0;
  pdl_wait();
  pdl_trigger();
  if (!good) {
    if (threadIdx.x == 0) set_error(st.err, EPIKV_DEV_BATCH);
    return;
  }
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool fits = nc0 + n_new <= dm.T;
  if (!fits && tid == 0 && blockIdx.x == 0) set_error(st.err, EPIKV_DEV_CAPACITY);
  const int i_lo = blockIdx.x * kFinTile;
  const int i_hi = min(i_lo + kFinTile, n_new);
  const int Gm = dm.G - 1;
  const int nb = dm.nA + dm.nB;
  // this CTA's part of the kinds: the band kinds first, then one K/V kind each
  const int part = blockIdx.z, kv_part = (dm.kinds & kBandKinds) ? part - 1 : part;

  extern __shared__ float sg[];  // band kinds: [nb][span] windows of g; a K/V kind: its u
  if (fits && i_lo < i_hi) {
    if (part == 0) for (int i = i_lo + warp; i < i_hi; i += kFinThreads / 32) {
      const int pos = p0 + i;
      if (lane == 0) st.pos[(size_t)seq * dm.T + nc0 + i] = pos;
      if (lane == 0 && dm.layer_budgets)  // a new token is in every layer
        st.lmask[(size_t)seq * dm.T + nc0 + i] = dm.L == 64 ? ~0ull : (1ull << dm.L) - 1ull;
    }
    if (kv_part < 0) {
      // every g value the tile's windows reach, all band layers, their loads in flight together
      const int span = kFinTile + dm.z_window - 1;
      const int pos_base = p0 + i_lo - (dm.z_window - 1);  // position held by sg[band][0]
      const int pos_end = p0 + i_hi;
      constexpr int U = 5;   // 15 layers x 79 values: one batch
      for (int idx0 = tid; idx0 < nb * span; idx0 += U * kFinThreads) {
        float v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int idx = idx0 + u * kFinThreads, band = idx / span;
          const int pos = pos_base + (idx - band * span);
          v[u] = idx < nb * span && pos >= 1 && pos < pos_end
                     ? __ldcg(st.g_ring + ((size_t)seq * nb + band) * dm.G + (pos & Gm)) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (idx0 + u * kFinThreads < nb * span) sg[idx0 + u * kFinThreads] = v[u];
      }
      __syncthreads();
      // a lane per (token, band layer): lpt lanes per token, 32/lpt tokens per warp
      const int lpt = nb <= 16 ? 16 : 32;
      const int sub = lane / lpt, band = lane % lpt;
      for (int i0 = i_lo + warp * (32 / lpt); i0 < i_hi; i0 += kFinThreads / lpt) {
        const int i = i0 + sub;
        const int pos = p0 + i;
        const bool live = i < i_hi && pos >= 1 && band < nb;
        float za = 0.f, zb = 0.f, ma = 0.f, mb = 0.f;
        if (live) {
          const int n = min(dm.z_window, pos);
          const float* row = sg + band * span + (pos - pos_base);   // row[-k] = g at position pos - k
          if (dm.kinds & EPIKV_SCORE_BANDZ) {
            const float z = window_z<-1>(row, n, dm.z_eps);
            if (band < dm.nA) za = z; else zb = z;
          }
          if (dm.kinds & EPIKV_SCORE_HSVAR) {
            const float gbar = window_mean<-1>(row, n);
            if (band < dm.nA) ma = gbar; else mb = gbar;
          }
        }
        for (int o = lpt >> 1; o > 0; o >>= 1) {  // stays inside each token's lane group
          za += __shfl_xor_sync(0xffffffffu, za, o);
          zb += __shfl_xor_sync(0xffffffffu, zb, o);
          ma += __shfl_xor_sync(0xffffffffu, ma, o);
          mb += __shfl_xor_sync(0xffffffffu, mb, o);
        }
        if (band == 0 && i < i_hi) {
          const size_t slot = (size_t)seq * dm.T + nc0 + i;
          if (dm.kinds & EPIKV_SCORE_BANDZ)
            st.score[0][slot] = pos >= 1 ? za / (float)dm.nA - zb / (float)dm.nB : 0.f;
          if (dm.kinds & EPIKV_SCORE_HSVAR)
            st.score[2][slot] = pos >= 1 ? ma / (float)dm.nA - mb / (float)dm.nB : 0.f;
        }
      }
    }
    if (kv_part >= 0) {
      // u of the tile's tokens and their windows' earlier ones in this call, a
      // thread per token, neighbouring threads' loads side by side (partials
      // [stream][token])
      int qk = 0;   // the kv_part-th K/V kind held
      for (int left = kv_part;; ++qk)
        if ((dm.kinds & kv_kind(qk)) && left-- == 0) break;
      const int kind = kv_kind(qk);
      float* su = sg;  // [lo .. i_hi)
      const int w = dm.lag_window;
      const int lo = max(0, i_lo - (w - 1));
      const float inv_lh = 1.f / (float)(dm.L * dm.H);
      // which partials: normalised or raw; all (layer, K|V) entries, keys only or values only
      const bool raw = kind & kRawKinds;
      const float* parts = (raw ? st.raw_part : st.lag_part) + (size_t)seq * dm.max_new * (2 * dm.L);
      const int q0 = kind == EPIKV_SCORE_KVVAL ? 1 : 0;
      const int qs = kind == EPIKV_SCORE_LAGKV ? 1 : 2;
      float* ring = st.u_ring[qk] + (size_t)seq * dm.G;
      float* out = st.score[kind_index(kind)] + (size_t)seq * dm.T + nc0;
      for (int i = lo + tid; i < i_hi; i += kFinThreads) {
        float u = 0.f;
        if (raw || p0 + i >= dm.lag) {  // the normalised kinds have no value in chunk 0
          const float* pp = parts + i;
          float s = 0.f;
#pragma unroll 16
          for (int q = q0; q < 2 * dm.L; q += qs) s += pp[(size_t)q * dm.max_new];
          u = s * inv_lh;
        }
        su[i - lo] = u;
      }
      __syncthreads();
      for (int i = i_lo + warp; i < i_hi; i += kFinThreads / 32) {
        const int pos = p0 + i;
        const int n = min(w, pos + 1);
        float acc = 0.f;
#pragma unroll
        for (int m = 0; m < WPL; ++m) {
          const int k = lane + 32 * m;
          if (k < n) acc += (i - k >= 0) ? su[i - k - lo] : ring[(pos - k) & Gm];
        }
        const float mean = warp_sum(acc) / (float)n;
        if (lane == 0) out[i] = mean;
      }
      for (int i = i_lo + tid; i < i_hi; i += kFinThreads) ring[(p0 + i) & Gm] = su[i - lo];
    }
  }

  // The last CTA of this sequence commits its counters (no CTA waits).
  __syncthreads();
  if (tid == 0) {
    if (ticket_add(&st.ticket[seq]) == gridDim.x * gridDim.z - 1) {
      if (fits) {
        // an eviction selected but not compacted before this update breaks the
        // call order; nothing is left pending for a later compaction either way
        if (first < nc0) set_error(st.err, EPIKV_DEV_KEPT);
        st.first_changed[seq] = nc0 + n_new;
        st.n_cache[seq] = nc0 + n_new;
        st.n_seen[seq] = p0 + n_new;
        if (dm.layer_budgets)
          for (int l = 0; l < dm.L; ++l) {
            st.n_layer[seq * dm.L + l] += n_new;
            st.lfirst[seq * dm.L + l] = st.n_layer[seq * dm.L + l];
          }
        if ((dm.kinds & kBandKinds) && n_new > 0) st.hp_parity[seq] ^= 1;
        atomicAdd(&st.stats[0], (unsigned long long)n_new);
      }
      st.ticket[seq] = 0u;
    }
  }
}

// ---- one new token per sequence (a decode step)
#ifndef EPIKV_TOKEN_MINB
// token_kernel CTAs resident per SM: 5 caps registers at 48 (64 ragged
// sequences' decode step: 45.7 / 41.1 / 38.5 / 38.5 us at 3 / 4 / 5 / 6)
#define EPIKV_TOKEN_MINB 5
#endif

// A thread's vectors of one band row of D channels, VR = D / 8.
template <int VPT>
__device__ __forceinline__ void band_row(const __nv_bfloat16* row, int VR, uint4 (&x)[VPT]) {
#pragma unroll
  for (int k = 0; k < VPT; ++k) {
    const int v = threadIdx.x + k * kGThreads;
    x[k] = v < VR ? ld_stream16(row + v * 8) : make_uint4(0, 0, 0, 0);
  }
}

// One new token's g for one band layer (Eq. 1), from its row and the saved
// previous row (h_prev), exactly as bandz_g_kernel forms it (same per-thread
// vectors, fused multiply-adds, warp sums and fixed-order cross-warp sum);
// the row is saved as the next call's previous row.  Then, for the band
// kinds' scores (Eq. 3), this band's z of the new g against its window and
// the window's mean, with score_finalize_kernel's arithmetic and order (window_z
// over g at positions pos, pos-1, ..., pos-n+1, one thread), stored per
// (sequence, band) for the last CTA to combine.  c and p are the thread's
// vectors of the row and the previous one (band_row); the window's earlier
// values are loaded into `win` (z_window floats of shared memory) while those
// loads are in flight.  Every thread of a kGThreads block calls it.
template <int VPT, int B>
__device__ __forceinline__ void band_token_g(const DevState& st, const Dims& dm, const uint4 (&c)[VPT],
                                             const uint4 (&p)[VPT], int band, int seq, int pos, int par, float* win) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nb = dm.nA + dm.nB;
  const int VR = dm.D >> 3;
  __shared__ float red[kGThreads / 32];
  __nv_bfloat16* hp_wr = st.h_prev + ((size_t)(seq * 2 + (par ^ 1)) * nb + band) * dm.D;
  float* ring = st.g_ring + ((size_t)seq * nb + band) * dm.G;
  const int n = pos >= 1 ? min(dm.z_window, pos) : 0;  // the new g's window, itself included
  for (int k = 1 + tid; k < n; k += kGThreads) win[k] = __ldcg(ring + ((pos - k) & (dm.G - 1)));
  float acc = 0.f;
#pragma unroll
  for (int k = 0; k < VPT; ++k) {
    float cf[8], pf[8];
    unpack8(c[k], cf);
    unpack8(p[k], pf);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float dlt = cf[e] - pf[e];
      acc = fmaf(dlt, dlt, acc);
    }
  }
  acc = warp_sum(acc);
  if (lane == 0) red[warp] = acc;
#pragma unroll
  for (int k = 0; k < VPT; ++k) {
    const int v = tid + k * kGThreads;
    if (v < VR) *reinterpret_cast<uint4*>(hp_wr + v * 8) = c[k];
  }
  __syncthreads();
  if (tid == 0) {
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < kGThreads / 32; ++w) sum += red[w];
    const float g = sqrtf(sum);
    if (pos >= 1) ring[pos & (dm.G - 1)] = g;
    if (n > 0) {
      win[0] = g;
      const float* row = win;  // row[k] = g at position pos - k
      float z = 0.f, gbar = 0.f;
      if (dm.kinds & EPIKV_SCORE_BANDZ) z = window_z<1, B>(row, n, dm.z_eps);
      if (dm.kinds & EPIKV_SCORE_HSVAR) gbar = window_mean<1, B>(row, n);
      st.ztok[(size_t)(seq * 2) * nb + band] = z;
      st.ztok[(size_t)(seq * 2 + 1) * nb + band] = gbar;
    }
  }
}

// The band kinds' scores of the new token at slot nc0: the per-band z and
// window means the band CTAs stored, combined exactly as
// score_finalize_kernel combines them (a lane per band, the same butterfly
// over the lanes).  One warp calls it.
__device__ __forceinline__ void band_token_combine(const DevState& st, const Dims& dm, int seq, int nc0, int pos) {
  const int lane = threadIdx.x & 31;
  const int nb = dm.nA + dm.nB;
  const int lpt = nb <= 16 ? 16 : 32;  // the lanes of one token, as in score_finalize_kernel
  const int bl = lane % lpt;
  const bool live = lane < lpt && pos >= 1 && bl < nb;
  float za = 0.f, zb = 0.f, ma = 0.f, mb = 0.f;
  if (live) {
    if (dm.kinds & EPIKV_SCORE_BANDZ) {
      const float z = __ldcg(st.ztok + (size_t)(seq * 2) * nb + bl);
      if (bl < dm.nA) za = z; else zb = z;
    }
    if (dm.kinds & EPIKV_SCORE_HSVAR) {
      const float gbar = __ldcg(st.ztok + (size_t)(seq * 2 + 1) * nb + bl);
      if (bl < dm.nA) ma = gbar; else mb = gbar;
    }
  }
  for (int o = lpt >> 1; o > 0; o >>= 1) {
    za += __shfl_xor_sync(0xffffffffu, za, o);
    zb += __shfl_xor_sync(0xffffffffu, zb, o);
    ma += __shfl_xor_sync(0xffffffffu, ma, o);
    mb += __shfl_xor_sync(0xffffffffu, mb, o);
  }
  if (lane == 0) {
    const size_t slot = (size_t)seq * dm.T + nc0;
    if (dm.kinds & EPIKV_SCORE_BANDZ) st.score[0][slot] = pos >= 1 ? za / (float)dm.nA - zb / (float)dm.nB : 0.f;
    if (dm.kinds & EPIKV_SCORE_HSVAR) st.score[2][slot] = pos >= 1 ? ma / (float)dm.nA - mb / (float)dm.nB : 0.f;
  }
}

// The K/V kinds' scores of the new token at slot nc0 (position pos), exactly
// as score_finalize_kernel forms them for a call's single token: u from the
// per-(layer, K|V) partials the stream CTAs wrote, summed in stream order by
// one thread (the warp first loads them into shared memory together, so the
// sum waits on one round of loads, not on 2L); its rolling mean over this u
// and the ring's earlier ones, a lane per window position in the same order,
// the same warp sum.  One warp calls it.
__device__ __forceinline__ void kv_token_scores(const DevState& st, const Dims& dm, int seq, int nc0, int pos) {
  const int lane = threadIdx.x & 31;
  __shared__ float pv[2 * 64];  // the host admits at most 64 layers
  const int Gm = dm.G - 1;
  const int w = dm.lag_window;
  const int n = min(w, pos + 1);
  const float inv_lh = 1.f / (float)(dm.L * dm.H);
  for (int qk = 0; qk < 4; ++qk) {
    const int kind = kv_kind(qk);
    if (!(dm.kinds & kind)) continue;
    const bool raw = kind & kRawKinds;
    const float* part = (raw ? st.raw_part : st.lag_part) + (size_t)seq * dm.max_new * (2 * dm.L);
    const int q0 = kind == EPIKV_SCORE_KVVAL ? 1 : 0;
    const int qs = kind == EPIKV_SCORE_LAGKV ? 1 : 2;
    float* ring = st.u_ring[qk] + (size_t)seq * dm.G;
    float u = 0.f;
    if (raw || pos >= dm.lag) {  // the normalised kinds have no value in chunk 0
      for (int q = lane; q < 2 * dm.L; q += 32) pv[q] = __ldcg(part + q);
      __syncwarp();
      if (lane == 0) {
        float s = 0.f;
        for (int q = q0; q < 2 * dm.L; q += qs) s += pv[q];
        u = s * inv_lh;
      }
      __syncwarp();  // pv is reused kind after kind
    }
    u = __shfl_sync(0xffffffffu, u, 0);
    float acc = 0.f;
    for (int k = lane; k < n; k += 32) acc += k == 0 ? u : __ldcg(ring + ((pos - k) & Gm));
    const float mean = warp_sum(acc) / (float)n;
    if (lane == 0) {
      st.score[kind_index(kind)][(size_t)seq * dm.T + nc0] = mean;
      ring[pos & Gm] = u;
    }
  }
}

// The decode step's commit of one sequence (as score_finalize_kernel's last
// CTA does it): the new slot's position, the counters, h_prev's parity.
// One thread.
__device__ __forceinline__ void token_commit(const DevState& st, const Dims& dm, int seq, int nc0, int pos) {
  const size_t slot = (size_t)seq * dm.T + nc0;
  st.pos[slot] = pos;
  if (dm.layer_budgets) {  // the new token is in every layer
    st.lmask[slot] = dm.L == 64 ? ~0ull : (1ull << dm.L) - 1ull;
    for (int l = 0; l < dm.L; ++l) {
      st.n_layer[seq * dm.L + l] += 1;
      st.lfirst[seq * dm.L + l] = st.n_layer[seq * dm.L + l];
    }
  }
  if (st.first_changed[seq] < nc0) set_error(st.err, EPIKV_DEV_KEPT);
  st.first_changed[seq] = nc0 + 1;
  st.n_cache[seq] = nc0 + 1;
  st.n_seen[seq] = pos + 1;
  if (dm.kinds & kBandKinds) st.hp_parity[seq] ^= 1;
  atomicAdd(&st.stats[0], 1ull);
  st.ticket[seq] = 0u;
}

// One new token per sequence with the band kinds only: g and the rolling
// z-score in one launch.  grid (band layers, batch entries), kGThreads
// threads: each CTA forms its band row's g and that band's z and window mean
// (band_token_g); the last CTA of a sequence (an acq_rel ticket; no
// CTA waits) combines them into the scores (band_token_combine) and commits
// the sequence.  Results equal the two-kernel path bit for bit.
template <int VPT>
__global__ void __launch_bounds__(kGThreads) bandz_token_kernel(DevState st, Dims dm, BandRows rows,
                                                                 int64_t row_stride,
                                                                 const int32_t* __restrict__ seq_ids,
                                                                 const int32_t* __restrict__ cu_new) {
  pdl_wait();
  pdl_trigger();
  const int band = blockIdx.x, b = blockIdx.y;
  const int tid = threadIdx.x;
  const int seq = seq_ids[b];
  const int r0 = cu_new[b], n_new = cu_new[b + 1] - r0;
  if (seq < 0 || seq >= dm.S || n_new < 0 || n_new > 1 || cu_new[0] != 0) {
    if (tid == 0 && band == 0) set_error(st.err, EPIKV_DEV_BATCH);
    return;
  }
  if (n_new == 0) return;
  const int nb = dm.nA + dm.nB;
  // both of the band's saved rows are loaded with the new one, before the
  // state says which of them is the previous row (one round trip less; the
  // step of 4 sequences reads 0.5 MB more from L2)
  uint4 c[VPT], p[VPT], p1[VPT];
  const __nv_bfloat16* saved = st.h_prev + ((size_t)(seq * 2) * nb + band) * dm.D;
  band_row(rows.p[band] + (int64_t)r0 * row_stride, dm.D >> 3, c);
  band_row(saved, dm.D >> 3, p);
  band_row(saved + (size_t)nb * dm.D, dm.D >> 3, p1);
  const int nc0 = st.n_cache[seq];
  const int pos = st.n_seen[seq];
  const int par = st.hp_parity[seq];
  if (nc0 + 1 > dm.T) {
    if (tid == 0 && band == 0) set_error(st.err, EPIKV_DEV_CAPACITY);
    return;
  }
  if (par) {
#pragma unroll
    for (int k = 0; k < VPT; ++k) p[k] = p1[k];
  }
  __shared__ int s_last;
  extern __shared__ float win[];  // [z_window]: this band's window of g
  band_token_g<VPT, 16>(st, dm, c, p, band, seq, pos, par, win);
  if (tid == 0) s_last = ticket_add(&st.ticket[seq]) == (unsigned)(nb - 1);
  __syncthreads();
  if (!s_last) return;
  if (tid < 32) band_token_combine(st, dm, seq, nc0, pos);
  if (tid == 32) token_commit(st, dm, seq, nc0, pos);  // meanwhile: they touch disjoint state
}

// One new token per sequence with a K/V kind (and any band kinds): the whole
// score update in one launch.  grid (band layers + L or 2L, batch entries),
// kGThreads threads: the first CTAs form the band rows' g, z and window means
// (band_token_g), the
// others the (layer, K|V) streams (lag_stream, the multi-token kernel's own
// code on a one-token call): a layer's K and V in the two halves of a CTA
// (`half`, when H*d/8 <= 128), else one stream per CTA; the last CTA of a
// sequence (ticket) forms every kind's score (band_token_combine,
// kv_token_scores) and commits.  Results equal the three-kernel path bit for
// bit.
template <int LH>
__global__ void __launch_bounds__(kGThreads, EPIKV_TOKEN_MINB) token_kernel(DevState st, Dims dm, BandRows rows, int64_t row_stride,
                                                           KvDev kv, const int32_t* __restrict__ seq_ids,
                                                           const int32_t* __restrict__ cu_new, int vpt, int half) {
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.y, tid = threadIdx.x;
  const int seq = seq_ids[b];
  const int r0 = cu_new[b], n_new = cu_new[b + 1] - r0;
  if (seq < 0 || seq >= dm.S || n_new < 0 || n_new > 1 || cu_new[0] != 0) {
    if (tid == 0 && blockIdx.x == 0) set_error(st.err, EPIKV_DEV_BATCH);
    return;
  }
  if (n_new == 0) return;
  const int nbc = (dm.kinds & kBandKinds) ? dm.nA + dm.nB : 0;  // band CTAs
  const int nc0 = st.n_cache[seq];
  const int pos = st.n_seen[seq];
  if (nc0 + 1 > dm.T) {
    if (tid == 0 && blockIdx.x == 0) set_error(st.err, EPIKV_DEV_CAPACITY);
    return;
  }
  __shared__ int s_last;
  extern __shared__ float win[];  // [z_window] (band CTAs): the band's window of g
  if ((int)blockIdx.x < nbc) {
    const int par = st.hp_parity[seq];
    const __nv_bfloat16* cur = rows.p[blockIdx.x] + (int64_t)r0 * row_stride;
    const __nv_bfloat16* prev = st.h_prev + ((size_t)(seq * 2 + par) * nbc + blockIdx.x) * dm.D;
    auto go = [&](auto vpt_t) {
      constexpr int VPT = decltype(vpt_t)::value;
      uint4 c[VPT], p[VPT];
      band_row(cur, dm.D >> 3, c);
      band_row(prev, dm.D >> 3, p);
      band_token_g<VPT, 1>(st, dm, c, p, blockIdx.x, seq, pos, par, win);
    };
    if (vpt == 1) go(std::integral_constant<int, 1>{});
    else if (vpt == 2) go(std::integral_constant<int, 2>{});
    else go(std::integral_constant<int, 4>{});
  } else {
    const int sidx = blockIdx.x - nbc;
    const int layer = half ? sidx : sidx >> 1;
    // the new row's slot: this layer's own length under per-layer budgets
    const int lnc0 = dm.layer_budgets ? st.n_layer[seq * dm.L + layer] : nc0;
    if (half) lag_stream<LH, 1, true>(st, dm, kv, seq, 0, 1, 1, layer, threadIdx.x >> 7, lnc0);
    else lag_stream<LH, 1>(st, dm, kv, seq, 0, 1, 1, layer, sidx & 1, lnc0);
  }
  __syncthreads();
  if (tid == 0) s_last = ticket_add(&st.ticket[seq]) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  // three warps at once, on disjoint state: the band scores (warp 0), the
  // K/V scores (warp 1) and the commit (warp 2)
  if (nbc && tid < 32) band_token_combine(st, dm, seq, nc0, pos);
  if (tid >= 32 && tid < 64) kv_token_scores(st, dm, seq, nc0, pos);
  if (tid == 64) token_commit(st, dm, seq, nc0, pos);
}

// ------------------------------------------------------------------ launchers
// dynamic shared memory of the finalize kernel: the band windows of a tile, or
// a K/V kind's u over it
static size_t finalize_smem(const Dims& dm) {
  const size_t band = (dm.kinds & kBandKinds) ? (size_t)(dm.nA + dm.nB) * (kFinTile + dm.z_window - 1) : 0;
  const size_t kv = (dm.kinds & kKvKinds) ? (size_t)(kFinTile + dm.lag_window - 1) : 0;
  return (band > kv ? band : kv) * sizeof(float);
}

cudaError_t finalize_prepare() {
  const int mx = (int)((size_t)kMaxBand * (kFinTile + kMaxWindow - 1) * sizeof(float));
  const int wmx = (int)((size_t)kMaxBand * kMaxWindow * sizeof(float));
  cudaError_t e = cudaSuccess;
  auto allow = [&](auto kern, int bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  allow(bandz_token_kernel<1>, wmx);
  allow(bandz_token_kernel<2>, wmx);
  allow(bandz_token_kernel<4>, wmx);
  allow(token_kernel<1>, wmx);
  allow(token_kernel<2>, wmx);
  allow(token_kernel<4>, wmx);
  allow(token_kernel<8>, wmx);
  allow(token_kernel<16>, wmx);
  allow(token_kernel<32>, wmx);
  allow(score_finalize_kernel<1, false>, mx);
  allow(score_finalize_kernel<2, false>, mx);
  allow(score_finalize_kernel<4, false>, mx);
  allow(score_finalize_kernel<8, false>, mx);
  allow(score_finalize_kernel<32, false>, mx);
  allow(score_finalize_kernel<1, true>, mx);
  allow(score_finalize_kernel<2, true>, mx);
  allow(score_finalize_kernel<4, true>, mx);
  allow(score_finalize_kernel<8, true>, mx);
  allow(score_finalize_kernel<32, true>, mx);
  return e;
}

cudaError_t launch_score_update(const DevState& st, const Dims& dm, int n_seq, const int32_t* seq_ids,
                                const int32_t* cu_new, int max_new, const epikv_hidden_view* hv,
                                const KvDev* kv, int num_sms, cudaStream_t stream, int* launches) {
  if (n_seq == 0 || max_new == 0) return cudaSuccess;
  const int nb = dm.nA + dm.nB;
  const bool band = dm.kinds & kBandKinds;
  BandRows rows;
  for (int i = 0; i < kMaxBand; ++i)
    rows.p[i] = band && i < nb ? static_cast<const __nv_bfloat16*>(hv->band_rows[i]) : nullptr;
  const int64_t rs = band ? hv->row_stride : 0;
  const int vr = dm.D / 8;
  const int vpt = vr <= kGThreads ? 1 : vr <= 2 * kGThreads ? 2 : 4;  // band row vectors per thread
  if (max_new == 1 && !(dm.kinds & kKvKinds)) {  // a decode step of the band kinds: one fused launch
    const dim3 grid(nb, n_seq);
    const size_t wsm = (size_t)dm.z_window * sizeof(float);  // a band CTA's window of g
    auto go = [&](auto kern) { pdl_launch(kern, grid, kGThreads, wsm, stream, st, dm, rows, rs, seq_ids, cu_new); };
    if (vpt == 1) go(bandz_token_kernel<1>);
    else if (vpt == 2) go(bandz_token_kernel<2>);
    else go(bandz_token_kernel<4>);
    ++*launches;
    return cudaGetLastError();
  }
  if (max_new == 1 && dm.L <= 64) {  // a decode step with a K/V kind: one fused launch
    const int half = dm.H * dm.d / 8 <= 128;  // a layer's K and V streams share a CTA
    const dim3 grid((band ? nb : 0) + (half ? dm.L : 2 * dm.L), n_seq);
    const size_t wsm = band ? (size_t)dm.z_window * sizeof(float) : 0;
    auto go = [&](auto kern) {
      pdl_launch(kern, grid, kGThreads, wsm, stream, st, dm, rows, rs, *kv, seq_ids, cu_new, vpt, half);
    };
    switch (dm.d / 8) {
      case 1: go(token_kernel<1>); break;
      case 2: go(token_kernel<2>); break;
      case 4: go(token_kernel<4>); break;
      case 8: go(token_kernel<8>); break;
      case 16: go(token_kernel<16>); break;
      default: go(token_kernel<32>); break;
    }
    ++*launches;
    return cudaGetLastError();
  }
  if (band) {
    // persistent: as many CTAs as are resident, never more than rows
    static int resident[3] = {0, 0, 0};
    const int vi = vpt == 1 ? 0 : vpt == 2 ? 1 : 2;
    if (!resident[vi]) {
      int per_sm = 1;
      if (vi == 0) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bandz_g_kernel<1>, kGThreads, 0);
      if (vi == 1) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bandz_g_kernel<2>, kGThreads, 0);
      if (vi == 2) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bandz_g_kernel<4>, kGThreads, 0);
      resident[vi] = (per_sm > 0 ? per_sm : 1) * num_sms;
    }
    const int64_t rows_bound = (int64_t)nb * n_seq * max_new;
    const int grid = (int)(rows_bound < resident[vi] ? rows_bound : resident[vi]);
    auto go = [&](auto kern) {
      pdl_launch(kern, grid, kGThreads, 0, stream, st, dm, rows, rs, seq_ids, cu_new, n_seq, max_new);
    };
    if (vi == 0) go(bandz_g_kernel<1>);
    else if (vi == 1) go(bandz_g_kernel<2>);
    else go(bandz_g_kernel<4>);
    ++*launches;
  }
  if (dm.kinds & kKvKinds) {
    const int piece = lag_piece_tokens(dm.L, dm.lag, n_seq, max_new, num_sms);
    const dim3 grid(2 * dm.L, n_seq, lag_pieces(max_new, dm.lag, piece));
    const int threads = max(32, (dm.H * dm.d / 8 + 31) / 32 * 32);
    auto go = [&](auto kern) {
      pdl_launch(kern, grid, threads, 0, stream, st, dm, *kv, seq_ids, cu_new, max_new, piece, band ? 1 : 0);
    };
    auto lanes = [&](auto kinds_t, auto split_t) {
      constexpr int KS = decltype(kinds_t)::value;
      constexpr bool SP = decltype(split_t)::value;
      switch (dm.d / 8) {
        case 1: go(lagkv_partial_kernel<1, KS, SP>); break;
        case 2: go(lagkv_partial_kernel<2, KS, SP>); break;
        case 4: go(lagkv_partial_kernel<4, KS, SP>); break;
        case 8: go(lagkv_partial_kernel<8, KS, SP>); break;
        case 16: go(lagkv_partial_kernel<16, KS, SP>); break;
        default: go(lagkv_partial_kernel<32, KS, SP>); break;
      }
    };
    auto kinds = [&](auto split_t) {
      const int ks = ((dm.kinds & kNormKinds) ? 1 : 0) | ((dm.kinds & kRawKinds) ? 2 : 0);
      if (ks == 1) lanes(std::integral_constant<int, 1>{}, split_t);
      else if (ks == 2) lanes(std::integral_constant<int, 2>{}, split_t);
      else lanes(std::integral_constant<int, 0>{}, split_t);   // both: the runtime flags (109 us, both fixed 168)
    };
    if (piece) kinds(std::true_type{});
    else kinds(std::false_type{});
    ++*launches;
  }
  {
    // the band kinds and every K/V kind in CTAs of their own: all six kinds of
    // 1,500 and 1,111 tokens 14 us, one CTA for all of a tile's kinds 24 us
    const dim3 grid((max_new + kFinTile - 1) / kFinTile, n_seq,
                    (band ? 1 : 0) + __builtin_popcount((unsigned)(dm.kinds & kKvKinds)));
    const int wmax = max(band ? dm.z_window : 1, (dm.kinds & kKvKinds) ? dm.lag_window : 1);
    const int wpl = (wmax + 31) / 32;
    const size_t smem = finalize_smem(dm);
    auto go = [&](auto kern) { pdl_launch(kern, grid, kFinThreads, smem, stream, st, dm, seq_ids, cu_new, max_new); };
    auto width = [&](auto many_t) {
      constexpr bool MANY = decltype(many_t)::value;
      if (wpl <= 1) go(score_finalize_kernel<1, MANY>);
      else if (wpl <= 2) go(score_finalize_kernel<2, MANY>);
      else if (wpl <= 4) go(score_finalize_kernel<4, MANY>);
      else if (wpl <= 8) go(score_finalize_kernel<8, MANY>);
      else go(score_finalize_kernel<32, MANY>);
    };
    if ((int64_t)grid.x * grid.y * grid.z > (int64_t)kFinFree * num_sms) width(std::true_type{});
    else width(std::false_type{});
    ++*launches;
  }
  return cudaGetLastError();
}

}  // namespace epikv
