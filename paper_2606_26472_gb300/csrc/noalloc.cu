// epikv_lagkv_score_noalloc: Lag-KV scores of a sequence's first n tokens in
// one call, for callers that cannot allocate device memory at all.
//
// Who needs it: a plugin running inside a host application whose own memory
// pool owns the whole device and refuses outside allocations, an embedded
// caller with no allocator bound to the GPU, or a latency-critical loop where
// a cudaMalloc (which can synchronise the device) is not acceptable.  Such a
// caller cannot create the workspace epikv_init needs, so this entry point
// keeps its working memory in a fixed array compiled into the library.
//
// The scratch is `g_noalloc_scratch`, a file-scope static device array of
// kNoallocScratchFloats floats (2 MiB).  Every GPU that loads the library
// holds it until the process exits.  In host code that name is only a host
// stand-in, not a device address: the first call in each CUDA context (with
// that context's device current) looks the real address up with
// cudaGetSymbolAddress and remembers it under the context's unique id, so a
// context that is torn down and created again (cudaDeviceReset) gets a fresh
// lookup instead of a stale address; that set-up is why the first call in a
// context should come before any stream capture.  The array is shared by
// every call and keeps the previous call's contents; every entry a call reads
// is written by the same call first, so nothing needs clearing, but two calls
// that overlap on the GPU (different streams, no ordering between them) race
// on it.
//
// Slots the view does not map (a negative or out-of-range block-table entry)
// are read as zero rows: this entry point has no error word, so such input
// is not reported.
//
// The kernels are variants of the Lag-KV partial and finalize kernels of the
// context path, for a sequence whose slots 0..n-1 hold positions 0..n-1.  They
// take each head's variance in two passes (mean, then squared deviations),
// where the context path uses shifted moments in one pass, so the scores agree
// with epikv_score_update's to fp32 rounding, not bit for bit.
#include <cuda.h>

#include <mutex>

#include "common.cuh"

namespace {

constexpr size_t kNoallocScratchFloats = size_t(1) << 19;  // 2 MiB: n * 2 * num_layers floats
constexpr int kMaxContexts = 64;  // contexts whose scratch address is remembered
constexpr int kSeg = 8;      // tokens per segment (never crosses a chunk boundary)
constexpr int kOffs = 256;   // row offsets looked up together
constexpr int kTile = 32;
constexpr int kThreads = 256;
constexpr int64_t kSms = 152;  // of a GB300, the only target (the length of pieces, never a result, depends on it)
#ifndef EPIKV_NOALLOC_CTAS
#define EPIKV_NOALLOC_CTAS 18   // CTAs per SM wanted before pieces get longer: three rounds of 6 resident ones
#endif
#ifndef EPIKV_NOALLOC_CHUNKS
#define EPIKV_NOALLOC_CHUNKS 2  // shortest piece
#endif
#ifndef EPIKV_NOALLOC_PF
#define EPIKV_NOALLOC_PF 1   // rows prefetched into L2 this many segments ahead (8,192 tokens: 0 237, 1 231, 2 234 us)
#endif
#ifndef EPIKV_NOALLOC_MAXREG
#define EPIKV_NOALLOC_MAXREG 80  // measured best with 72 (128, 80, 72: 171, 128, 127 us on 4,001 tokens; 72 is slower on 200)
#endif
#define EPIKV_NOALLOC_BOUNDS __maxnreg__(EPIKV_NOALLOC_MAXREG)

}  // namespace

static __device__ __align__(256) float g_noalloc_scratch[kNoallocScratchFloats];

namespace {

using epikv::KvDev;

// grid: (2L (layer, K|V), pieces of `piece` tokens, a multiple of lag);
// block: max(32, H*d/8) threads, d/8 lanes per head, 8 channels each.
//
// A piece first takes the minimum and maximum of the chunk before it (bf16
// values, kept packed; exact), so pieces are independent and one sequence
// fills the GPU.  A call on 4,001 tokens of a 32-layer cache (524 MB) takes
// 123 us (4.3 TB/s; bound by its instructions, two passes of arithmetic per
// row: 348 warp instructions a row, issue active 67 %), 200 tokens 19 us; one
// CTA per stream walking all tokens with a butterfly per sum took 2,150 and
// 116 us.  Tokens are taken in segments of up
// to 8 inside one chunk, their rows loaded together; the variance of a
// token's head is taken in two passes over the normalised values, four tokens
// at a time, their sums over the head's lanes by one transposed reduction.
// part[stream][token]: neighbouring tokens' sums are stored, and later read,
// together.
template <int LH>
__global__ void EPIKV_NOALLOC_BOUNDS noalloc_partial_kernel(KvDev kv, int seq, int n, int L, int H, int d, int lag,
                                                            float lag_eps, int piece, float* part) {
  using namespace epikv;
  const int layer = blockIdx.x >> 1, kvk = blockIdx.x & 1;
  const int tid = threadIdx.x, lane = tid & 31;
  const int h = tid / LH, q = tid % LH;
  const bool active = h < H;
  const int ch = h * d + q * 8;
  const float inv_d = 1.f / (float)d;
  const char* base = (kvk ? kv.base[1] : kv.base[0]) + (int64_t)ch * 2;
  const int t_lo = blockIdx.y * piece, t_hi = min(n, t_lo + piece);
  const int t_from = t_lo ? t_lo - lag : 0;   // the chunk before the piece: its range only
  __shared__ int64_t soff[kOffs];
  __shared__ float hv[2][kSeg][33];           // [parity][token][head]
  uint4 cmn = make_uint4(0, 0, 0, 0), cmx = cmn;
  f32x2 neg[4], inv[4];                       // -minimum and 1 / (maximum - minimum + eps) of the previous chunk
#pragma unroll
  for (int p = 0; p < 4; ++p) neg[p] = inv[p] = 0ull;
  int r = 0, parity = 0;                      // t_from is the first position of a chunk
  for (int g0 = t_from; g0 < t_hi; g0 += kOffs) {
    const int gn = min(kOffs, t_hi - g0);
    __syncthreads();
    for (int t = tid; t < gn; t += blockDim.x) soff[t] = kv_row_offset(kv, layer, seq, g0 + t, n);
    __syncthreads();
    for (int t = tid; t < min(EPIKV_NOALLOC_PF * kSeg, gn); t += blockDim.x)
      if (soff[t] >= 0)
        prefetch_l2_bulk((kvk ? kv.base[1] : kv.base[0]) + soff[t] * 2, (uint32_t)(H * d) * 2u);
    for (int i = 0; i < gn;) {
      const int seg = min(min(lag - r, gn - i), kSeg);
      const int t0 = g0 + i;
      const bool mine = t0 >= t_lo;           // a piece begins at a chunk, so never inside a segment
      const bool score = mine && t0 >= lag;   // chunk 0 has no previous range: u = 0
      uint4 x[kSeg];
#pragma unroll
      for (int j = 0; j < kSeg; ++j) {        // past the segment: its last row again, unused sums
        const int64_t off = soff[i + min(j, seg - 1)];
        x[j] = ld_stream16_if(base + off * 2, active && off >= 0);
      }
      {   // rows of later segments on their way to L2, each row once
        const int t = i + EPIKV_NOALLOC_PF * kSeg + tid;
        if (EPIKV_NOALLOC_PF > 0 && tid < seg && t < gn && soff[t] >= 0)
          prefetch_l2_bulk((kvk ? kv.base[1] : kv.base[0]) + soff[t] * 2, (uint32_t)(H * d) * 2u);
      }
      if (r == 0) cmn = cmx = x[0];
#pragma unroll
      for (int j = 0; j < kSeg; j += 2) {
        cmn = q_min(q_min(cmn, x[j]), x[j + 1]);
        cmx = q_max(q_max(cmx, x[j]), x[j + 1]);
      }
      if (score) {
#pragma unroll
        for (int j0 = 0; j0 < kSeg; j0 += 4) {
          f32x2 y[4][4];
          float v[4], tot[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint32_t w[4] = {x[j0 + j].x, x[j0 + j].y, x[j0 + j].z, x[j0 + j].w};
#pragma unroll
            for (int p = 0; p < 4; ++p) y[j][p] = f2_mul(f2_add(bf16x2_to_f2(w[p]), neg[p]), inv[p]);
            const f32x2 s = f2_add(f2_add(y[j][0], y[j][1]), f2_add(y[j][2], y[j][3]));
            v[j] = f2_lo(s) + f2_hi(s);
          }
          group_totals<LH>(v, lane, tot);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float m = -tot[j] * inv_d;
            const f32x2 nm = f2_pack(m, m);
            f32x2 ss = 0ull;
#pragma unroll
            for (int p = 0; p < 4; ++p) {
              const f32x2 dv = f2_add(y[j][p], nm);
              ss = f2_fma(dv, dv, ss);
            }
            v[j] = f2_lo(ss) + f2_hi(ss);
          }
          transpose_sum<LH / 2, 4, 4>(v, lane);
          if (active) {
            if constexpr (LH <= 4) {
#pragma unroll
              for (int k = 0; k < 4 / LH; ++k) hv[parity][j0 + k + (4 / LH) * q][h] = v[k];
            } else {
              if (q % (LH / 4) == 0) hv[parity][j0 + q / (LH / 4)][h] = v[0];
            }
          }
        }
      }
      if (mine) {
        __syncthreads();   // hv is double buffered: one barrier per segment
        if (tid < seg) {
          float s = 0.f;
          if (score)
            for (int hh = 0; hh < H; ++hh) s += hv[parity][tid][hh];
          part[(size_t)blockIdx.x * n + t0 + tid] = s * inv_d;
        }
        parity ^= 1;
      }
      r += seg;
      if (r == lag) {      // the chunk is complete: it becomes the previous one
        float mn[8], mx[8];
        unpack8(cmn, mn);
        unpack8(cmx, mx);
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          neg[p] = f2_pack(-mn[2 * p], -mn[2 * p + 1]);
          inv[p] = f2_pack(__frcp_rn(mx[2 * p] - mn[2 * p] + lag_eps), __frcp_rn(mx[2 * p + 1] - mn[2 * p + 1] + lag_eps));
        }
        r = 0;
      }
      i += seg;
    }
  }
}

// grid: token tiles of 32; block: 256 threads, a warp per token.
template <int WPL>
__global__ void __launch_bounds__(kThreads) noalloc_finalize_kernel(const float* part, int n, int L, int H, int lag,
                                                                    int w, float* out) {
  epikv::pdl_wait();
  __shared__ float su[kTile + 1024];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int i_lo = blockIdx.x * kTile, i_hi = min(i_lo + kTile, n);
  const int lo = max(0, i_lo - (w - 1));
  const float inv_lh = 1.f / (float)(L * H);
  for (int i = lo + tid; i < i_hi; i += kThreads) {
    float u = 0.f;
    if (i >= lag) {
      float s = 0.f;
#pragma unroll 16
      for (int q = 0; q < 2 * L; ++q) s += part[(size_t)q * n + i];
      u = s * inv_lh;
    }
    su[i - lo] = u;
  }
  __syncthreads();
  for (int i = i_lo + warp; i < i_hi; i += kThreads / 32) {
    const int cnt = min(w, i + 1);
    float acc = 0.f;
#pragma unroll
    for (int m = 0; m < WPL; ++m) {
      const int k = lane + 32 * m;
      if (k < cnt) acc += su[i - k - lo];
    }
    const float mean = epikv::warp_sum(acc) / (float)cnt;
    if (lane == 0) out[i] = mean;
  }
}

// Tokens per piece: as long as there are EPIKV_NOALLOC_CTAS CTAs per SM, since
// a piece re-reads (from L2) the chunk before it, and at least two chunks
// (8,192 / 4,001 / 1,000 tokens: 7 CTAs per SM 268 / 141 / 48 us, 12 225 / 123
// / 44, 14 232 / 127 / 46, 18 222 / 124 / 46, 28 237 / 130 / 46: whole rounds
// of 6; 200 tokens at least four chunks 24 us, two 19).
int piece_tokens(int n, int L, int lag) {
  const int64_t least = (int64_t)EPIKV_NOALLOC_CHUNKS * lag, streams = 2 * (int64_t)L;
  const int64_t pieces = (EPIKV_NOALLOC_CTAS * kSms + streams - 1) / streams;
  int64_t piece = ((n + pieces - 1) / pieces + lag - 1) / lag * lag;
  if (piece < least) piece = least;
  return piece < n ? (int)piece : n;
}

// The current context's unique id (driver entry points fetched through the
// runtime, so the library needs no link-time dependency on the driver).
typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);

std::mutex g_mu;
CtxGetCurrentFn g_ctx_current = nullptr;
CtxGetIdFn g_ctx_id = nullptr;
struct ScratchEntry {
  unsigned long long ctx_id;
  float* ptr;
};
ScratchEntry g_scratch[kMaxContexts] = {};
int g_scratch_next = 0;

cudaError_t current_context_id(unsigned long long* id) {
  if (!g_ctx_current || !g_ctx_id) {
    void* f1 = nullptr;
    void* f2 = nullptr;
    cudaDriverEntryPointQueryResult q1, q2;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1);
    if (e == cudaSuccess) e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2);
    if (e != cudaSuccess) return e;
    if (q1 != cudaDriverEntryPointSuccess || q2 != cudaDriverEntryPointSuccess || !f1 || !f2)
      return cudaErrorNotSupported;
    g_ctx_current = reinterpret_cast<CtxGetCurrentFn>(f1);
    g_ctx_id = reinterpret_cast<CtxGetIdFn>(f2);
  }
  CUcontext ctx = nullptr;
  if (g_ctx_current(&ctx) != CUDA_SUCCESS || !ctx) return cudaErrorDeviceUninitialized;
  return g_ctx_id(ctx, id) == CUDA_SUCCESS ? cudaSuccess : cudaErrorContextIsDestroyed;
}

// Device address of the scratch array in the current context: looked up once
// per context, then taken from the table.
cudaError_t scratch_address(float** out) {
  std::lock_guard<std::mutex> lock(g_mu);
  unsigned long long id = 0;
  if (current_context_id(&id) == cudaSuccess)
    for (const ScratchEntry& s : g_scratch)
      if (s.ptr && s.ctx_id == id) {
        *out = s.ptr;
        return cudaSuccess;
      }
  // first call in this context (this also makes the device's primary context
  // current if no context was yet)
  void* p = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  if (e != cudaSuccess) return e;
  e = current_context_id(&id);
  if (e != cudaSuccess) return e;
  g_scratch[g_scratch_next] = ScratchEntry{id, static_cast<float*>(p)};
  g_scratch_next = (g_scratch_next + 1) % kMaxContexts;
  *out = static_cast<float*>(p);
  return cudaSuccess;
}

bool view_ok(const epikv_kv_view* kv, int H, int d, KvDev* out) {
  if (!kv || !kv->k || !kv->v || ((uintptr_t)kv->k & 15u) || ((uintptr_t)kv->v & 15u)) return false;
  if (kv->stride_token < (int64_t)H * d || kv->stride_token % 8 || kv->stride_layer < 0 || kv->stride_layer % 8)
    return false;
  *out = KvDev{};
  out->base[0] = static_cast<char*>(kv->k);
  out->base[1] = static_cast<char*>(kv->v);
  out->layout = kv->layout;
  out->stride_layer = kv->stride_layer;
  out->stride_token = kv->stride_token;
  if (kv->layout == EPIKV_LAYOUT_CONTIGUOUS) {
    if (kv->stride_seq < 0 || kv->stride_seq % 8) return false;
    out->stride_seq = kv->stride_seq;
    return true;
  }
  if (kv->layout != EPIKV_LAYOUT_PAGED || !kv->block_table || kv->block_size < 1 || kv->max_blocks_per_seq < 1 ||
      kv->num_blocks < 1 || kv->stride_block < 0 || kv->stride_block % 8 || kv->stride_table_layer < 0)
    return false;
  out->stride_block = kv->stride_block;
  out->table_stride_layer = kv->stride_table_layer;
  out->block_table = kv->block_table;
  out->max_blocks = kv->max_blocks_per_seq;
  out->block_size = kv->block_size;
  out->num_blocks = kv->num_blocks;
  return true;
}

}  // namespace

extern "C" epikv_status epikv_lagkv_score_noalloc(const epikv_kv_view* kv, int32_t seq, int32_t n,
                                                  int32_t num_layers, int32_t num_kv_heads, int32_t head_dim,
                                                  int32_t lag, float lag_eps, int32_t window, float* d_scores,
                                                  cudaStream_t stream) {
  const int L = num_layers, H = num_kv_heads, d = head_dim;
  if (n < 1 || seq < 0 || L < 1 || H < 1 || H > 32 || d < 8 || d > 256 || (d & (d - 1)) || H * d / 8 > 256)
    return EPIKV_EINVAL;
  if (lag < 1 || window < 1 || window > 1024 || !(lag_eps >= 0.f) || !d_scores || ((uintptr_t)d_scores & 3u))
    return EPIKV_EINVAL;
  if ((size_t)n * 2 * (size_t)L > kNoallocScratchFloats) return EPIKV_EINVAL;  // beyond the fixed scratch
  KvDev kd;
  if (!view_ok(kv, H, d, &kd)) return EPIKV_EINVAL;
  // an error left by earlier, unrelated work stays with its owner: report it
  // without launching and without clearing it
  if (cudaPeekAtLastError() != cudaSuccess) return EPIKV_ECUDA;
  float* part = nullptr;
  if (scratch_address(&part) != cudaSuccess) return EPIKV_ECUDA;

  const int threads = (H * d / 8 + 31) / 32 * 32 < 32 ? 32 : (H * d / 8 + 31) / 32 * 32;
  const int piece = piece_tokens(n, L, lag);
  const dim3 g1(2 * L, (n + piece - 1) / piece);
  switch (d / 8) {
    case 1: noalloc_partial_kernel<1><<<g1, threads, 0, stream>>>(kd, seq, n, L, H, d, lag, lag_eps, piece, part); break;
    case 2: noalloc_partial_kernel<2><<<g1, threads, 0, stream>>>(kd, seq, n, L, H, d, lag, lag_eps, piece, part); break;
    case 4: noalloc_partial_kernel<4><<<g1, threads, 0, stream>>>(kd, seq, n, L, H, d, lag, lag_eps, piece, part); break;
    case 8: noalloc_partial_kernel<8><<<g1, threads, 0, stream>>>(kd, seq, n, L, H, d, lag, lag_eps, piece, part); break;
    case 16: noalloc_partial_kernel<16><<<g1, threads, 0, stream>>>(kd, seq, n, L, H, d, lag, lag_eps, piece, part); break;
    default: noalloc_partial_kernel<32><<<g1, threads, 0, stream>>>(kd, seq, n, L, H, d, lag, lag_eps, piece, part); break;
  }
  const dim3 g2((n + kTile - 1) / kTile);
  const int wpl = (window + 31) / 32;
  auto fin = [&](auto kern) {
    epikv::pdl_launch(kern, g2, dim3(kThreads), 0, stream, (const float*)part, n, L, H, lag, window, d_scores);
  };
  if (wpl <= 1) fin(noalloc_finalize_kernel<1>);
  else if (wpl <= 2) fin(noalloc_finalize_kernel<2>);
  else if (wpl <= 4) fin(noalloc_finalize_kernel<4>);
  else if (wpl <= 8) fin(noalloc_finalize_kernel<8>);
  else fin(noalloc_finalize_kernel<32>);
  // no error was pending before the launches, so any error now is theirs
  return cudaGetLastError() == cudaSuccess ? EPIKV_OK : EPIKV_ECUDA;
}
