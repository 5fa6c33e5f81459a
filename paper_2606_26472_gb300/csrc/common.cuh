// Device-side helpers shared by the EpiKV kernels: the context's device
// state, K/V row addressing for both layouts, the sticky error word, and
// inline-PTX wrappers for 1-D TMA bulk copies and mbarriers (sm_90+ ISA,
// compiled here for sm_103a only).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "epikv.h"
#include "plans.h"

namespace epikv {

constexpr int kMaxSeqs = 4096;  // sequences of a context, so entries of a batch
constexpr int kMaxBand = 32;
constexpr int kNumKinds = 6;  // score kind index k <-> mask bit (1 << k)
constexpr int kBandKinds = EPIKV_SCORE_BANDZ | EPIKV_SCORE_HSVAR;
constexpr int kNormKinds = EPIKV_SCORE_LAGKV | EPIKV_SCORE_LAGKEY;   // need the chunk ranges
constexpr int kRawKinds = EPIKV_SCORE_KVKEY | EPIKV_SCORE_KVVAL;
constexpr int kKvKinds = kNormKinds | kRawKinds;
// the K/V kinds in the order of their rolling-mean rings
__host__ __device__ __forceinline__ int kv_kind(int q) {
  return q == 0 ? EPIKV_SCORE_LAGKV : q == 1 ? EPIKV_SCORE_KVKEY : q == 2 ? EPIKV_SCORE_KVVAL : EPIKV_SCORE_LAGKEY;
}

__host__ __device__ __forceinline__ int kind_index(int bit) {
  int k = 0;
  while (bit > 1) {
    bit >>= 1;
    ++k;
  }
  return k;
}

// Device pointers carved out of the caller's workspace (one context).
struct DevState {
  int32_t* n_cache;        // [S] slots in use
  int32_t* n_seen;         // [S] next position
  int32_t* prefill;        // [S]
  int32_t* policy;         // [S] score kind driving selection (1 or 2)
  int32_t* hp_parity;      // [S] which h_prev buffer holds the last row
  int32_t* first_changed;  // [S] first slot moved by the last selection
  uint32_t* ticket;        // [S] last-CTA tickets of the finalize kernel
  int32_t* err;            // [1] sticky device error word
  unsigned long long* stats;  // [4] epikv_stats
  float* score[kNumKinds]; // [S][T] frozen scores per kind (null when the kind is off)
  int32_t* pos;            // [S][T] position of each slot
  __nv_bfloat16* h_prev;   // [S][2][n_band][D] last hidden row per band layer
  float* g_ring;           // [S][n_band][G] g by position (mod G)
  float* ztok;             // [S][2][n_band] a decode step's per-band z and window mean of g (band kinds)
  __nv_bfloat16* lag_rng;  // [S][L][2][4][H][d] prev min, prev max, cur min, cur max
  float* lag_part;         // [S][2L][max_new] per-(layer, K|V) head-summed normalised variances (a decode step: [S][2L] at the front)
  float* raw_part;         // the same of the raw variances
  float* u_ring[4];        // [S][G] per K/V kind (kv_kind order): u by position (mod G)
  int32_t* kept;           // [S][T] kept lists of epikv_step
  int32_t* n_kept;         // [S]
  uint32_t* ckey;          // [S][T] chunk-level selection: each candidate slot's chunk key (C > 1 only)
  // per-layer budgets only (null otherwise)
  int32_t* n_layer;        // [S][L] slots held by each layer
  int32_t* lfirst;         // [S][L] first slot of each layer moved by the last selection
  unsigned long long* lmask;      // [S][T] bit l: layer l holds the token of this slot
  unsigned long long* lmask_new;  // [S][T] the select kernel's new masks (scratch)
  uint32_t* lkeep;         // [S][L][ceil(T/32)] bit: layer l keeps the union slot (scratch)
  int32_t* mkept;          // [S][T] the select kernel's kept slots of the largest layer (scratch)
  uint32_t* work;          // [2] the compaction's next unit or late chunk and, under per-layer budgets, its finished CTAs
                           // (which leave both 0; under token budgets the stash kernel zeroes the first)
  char* stash;             // [kMaxStashCtas][stash_rows][H*d] bf16: compaction boundary rows, fewer per chunk for more chunks
  int32_t* stash_row0;     // [kMaxChunks] the row whose source is each stash's first row
};

struct Dims {
  int S, T, max_new, L, H, d, D, nA, nB, G;
  int stash_rows;  // min(kStashRows, T): rows of one CTA's compaction stash
  int z_window, lag, lag_window, recency_cap, kinds, select_chunk, layer_budgets;
  float z_eps, lag_eps;
};

struct KvDev {
  char* base[2];           // K, V
  int layout;
  int64_t stride_layer, stride_seq, stride_block, stride_token;  // elements
  const int32_t* block_table;
  int max_blocks, block_size, num_blocks;
  int64_t table_stride_layer;  // elements between layers' block tables (0: shared)
};

// Programmatic dependent launch.  The kernels of a step are launched with
// programmatic stream serialisation (pdl_launch): each may be scheduled once
// every CTA of the kernel before it on the stream has called pdl_trigger or
// ended, and pdl_wait returns when that kernel has completed and its writes are
// visible.  Launched without the attribute, both are no-ops.
//
// The order that this leaves.  Every kernel waits, so it completes after the
// one before it.  A kernel may read before its wait only what the one before
// it does not write, and only if that one triggers after its own wait: all
// that was launched earlier has then completed.  Those that do:
//   score_finalize_kernel  the batch and the sequences' counters (after the g
//                          or K/V kernel)
//   select_kernel          in a step: the batch, budgets, triggers, prefill
//                          lengths and policies (after the score update's last
//                          kernel)
//   compact_kernel         the selection's results and cache rows that the
//                          stash kernel does not move (per-layer budgets: it
//                          also counts units, which that kernel does not)
//   compact_consumed_kernel  the batch and the lengths (after the copy)
//   lagkv_partial_kernel   after the g kernel: all that it reads.  It also
//                          writes (partials and chunk ranges, of which the g
//                          kernel knows nothing), triggers at once and waits
//                          only before it ends.  The kernel after it is let in
//                          once its CTAs run, so after the g kernel's wait: the
//                          rule above holds for that one too, which then waits
//                          for both.
// Every other kernel waits first.  A trigger must not move ahead of a wait, nor
// a kernel come between two of these, without a look at this list.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

#ifndef EPIKV_PDL
#define EPIKV_PDL 1  // 0: plain stream order
#endif

template <typename... Params, typename... Args>
inline cudaError_t launch_kernel_now(bool programmatic, void (*kernel)(Params...), dim3 grid, dim3 block,
                                     size_t smem, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = programmatic && EPIKV_PDL ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Per-kernel timing (epikv_set_kernel_events): while an entry point of a
// context with kernel events runs, t_kernel_clock points at its record, and
// every kernel it launches is bracketed by two of the caller's events on the
// launch stream, its name (cudaFuncGetName) stored beside them.
struct KernelClock {
  cudaEvent_t* ev;      // [2 * cap]: before and after each kernel
  const char** names;   // [cap]
  int cap, used;
};
inline thread_local KernelClock* t_kernel_clock = nullptr;

template <typename... Params, typename... Args>
inline cudaError_t launch_kernel(bool programmatic, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem,
                                 cudaStream_t stream, Args... args) {
  KernelClock* kc = t_kernel_clock;
  if (kc && kc->used < kc->cap) {
    const cudaError_t e = cudaEventRecord(kc->ev[2 * kc->used], stream);
    if (e != cudaSuccess) return e;
  } else {
    kc = nullptr;
  }
  const cudaError_t e = launch_kernel_now(programmatic, kernel, grid, block, smem, stream, args...);
  if (e != cudaSuccess || !kc) return e;
  const char* name = nullptr;
  if (cudaFuncGetName(&name, reinterpret_cast<const void*>(kernel)) != cudaSuccess) name = nullptr;
  kc->names[kc->used] = name;
  return cudaEventRecord(kc->ev[2 * kc->used++ + 1], stream);
}


template <typename... Params, typename... Args>
inline cudaError_t pdl_launch(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                              Args... args) {
  return launch_kernel(true, kernel, grid, block, smem, stream, args...);
}

// Plain stream order: the copy kernel where no stash kernel runs before it.
template <typename... Params, typename... Args>
inline cudaError_t plain_launch(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                Args... args) {
  return launch_kernel(false, kernel, grid, block, smem, stream, args...);
}

__device__ __forceinline__ void set_error(int32_t* err, int code) {
  atomicCAS(err, 0, code);
}

// Element offset of (layer, seq, slot) or -1 if outside the view.
__device__ __forceinline__ int64_t kv_row_offset(const KvDev& v, int layer, int seq, int slot, int T) {
  if (slot < 0) return -1;
  if (v.layout == EPIKV_LAYOUT_CONTIGUOUS) {
    if (slot >= T) return -1;
    return (int64_t)layer * v.stride_layer + (int64_t)seq * v.stride_seq + (int64_t)slot * v.stride_token;
  }
  int bi = slot / v.block_size;
  if (bi >= v.max_blocks) return -1;
  int blk = __ldg(v.block_table + (int64_t)layer * v.table_stride_layer + (int64_t)seq * v.max_blocks + bi);
  if (blk < 0 || blk >= v.num_blocks) return -1;
  return (int64_t)layer * v.stride_layer + (int64_t)blk * v.stride_block +
         (int64_t)(slot - bi * v.block_size) * v.stride_token;
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

__device__ __forceinline__ void unpack8(const uint4& q, float* f) {
  f[0] = bf16_lo(q.x); f[1] = bf16_hi(q.x);
  f[2] = bf16_lo(q.y); f[3] = bf16_hi(q.y);
  f[4] = bf16_lo(q.z); f[5] = bf16_hi(q.z);
  f[6] = bf16_lo(q.w); f[7] = bf16_hi(q.w);
}

// Streaming 16-byte load that does not allocate in L1.
__device__ __forceinline__ uint4 ld_stream16(const void* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

// The same load when `take`, else zeros: a predicated instruction, no branch.
__device__ __forceinline__ uint4 ld_stream16_if(const void* p, bool take) {
  uint4 r = make_uint4(0, 0, 0, 0);
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n\t}"
      : "+r"(r.x), "+r"(r.y), "+r"(r.z), "+r"(r.w) : "l"(p), "r"((int)take));
  return r;
}

// ---------------------------------------------------------------- mbarrier
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;"
               :: "r"(smem_u32(bar)), "r"(bytes) : "memory");
}

#ifndef EPIKV_MBAR_SPIN
#define EPIKV_MBAR_SPIN 2
#endif

// One probe; true when the phase with `parity` has completed.  The default
// (2) may suspend the thread for a short, hardware-chosen time; 1 polls
// without suspending; 0 asks for a suspension of up to 1 us.
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
#if EPIKV_MBAR_SPIN == 1
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
#elif EPIKV_MBAR_SPIN == 2
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
#else
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, 1000;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
#endif
  return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Wait at most `limit_ns` of wall time; false if it gave up.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(bar, parity))
    if (global_ns() - t0 > limit_ns) return false;
  return true;
}

__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ------------------------------------------------------------ TMA bulk copies
// global -> shared, completion counted in bytes on `bar`.
__device__ __forceinline__ void tma_load_1d(void* smem_dst, const void* gmem_src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      :: "r"(smem_u32(smem_dst)), "l"(gmem_src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// shared -> global, tracked by this thread's bulk async-groups.
__device__ __forceinline__ void tma_store_1d(void* gmem_dst, const void* smem_src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
               :: "l"(gmem_dst), "r"(smem_u32(smem_src)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void tma_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }

// Wait until at most N of this thread's bulk groups still read shared memory.
template <int N>
__device__ __forceinline__ void tma_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" :: "n"(N) : "memory");
}

__device__ __forceinline__ void tma_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// ------------------------------------------------------------ warp helpers
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over aligned groups of `width` lanes (width a power of two <= 32).
__device__ __forceinline__ float group_sum(float v, int width) {
  for (int o = width >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ uint32_t bf16x2_min(uint32_t a, uint32_t b) {
  __nv_bfloat162 r = __hmin2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
  return *reinterpret_cast<uint32_t*>(&r);
}
__device__ __forceinline__ uint32_t bf16x2_max(uint32_t a, uint32_t b) {
  __nv_bfloat162 r = __hmax2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
  return *reinterpret_cast<uint32_t*>(&r);
}
__device__ __forceinline__ uint4 q_min(const uint4& a, const uint4& b) {
  return make_uint4(bf16x2_min(a.x, b.x), bf16x2_min(a.y, b.y), bf16x2_min(a.z, b.z), bf16x2_min(a.w, b.w));
}
__device__ __forceinline__ uint4 q_max(const uint4& a, const uint4& b) {
  return make_uint4(bf16x2_max(a.x, b.x), bf16x2_max(a.y, b.y), bf16x2_max(a.z, b.z), bf16x2_max(a.w, b.w));
}

// ---- packed fp32 pairs: Blackwell's f32x2 arithmetic, two channels per instruction
typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 f2_pack(float lo, float hi) {
  f32x2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ float f2_lo(f32x2 v) { return __uint_as_float((unsigned)(v & 0xffffffffull)); }
__device__ __forceinline__ float f2_hi(f32x2 v) { return __uint_as_float((unsigned)(v >> 32)); }
__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 f2_add(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 f2_mul(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// the two bf16 channels of a 32-bit word as an fp32 pair (exact)
__device__ __forceinline__ f32x2 bf16x2_to_f2(uint32_t w) { return f2_pack(bf16_lo(w), bf16_hi(w)); }

// Transposed sum over the O*2 lanes of a group: every level halves the values
// a lane keeps and sends the other half to its partner, so NV values cost
// NV - 1 shuffles in all instead of one butterfly of log2(lanes) shuffles per
// value.  With lanes <= NV, value k + (NV / lanes) * (lane % lanes) ends in
// v[k]; with more lanes than values, value (lane % lanes) / (lanes / NV) ends
// in v[0].
template <int O, int C, int NV>
__device__ __forceinline__ void transpose_sum(float (&v)[NV], int lane) {
  if constexpr (O >= 1) {
    if constexpr (C > 1) {
      const bool up = lane & O;
#pragma unroll
      for (int k = 0; k < C / 2; ++k) {
        const float send = up ? v[k] : v[k + C / 2];
        const float keep = up ? v[k + C / 2] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, O);
      }
      transpose_sum<O / 2, C / 2, NV>(v, lane);
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], O);
      transpose_sum<O / 2, 1, NV>(v, lane);
    }
  }
}

// Sums of NV values over the LH lanes of a group, every lane of which then
// holds total j in out[j]: the transposed sum and one shuffle per value (the
// same additions, in the same pairs, as NV butterflies).  NV = 4 or 8.
template <int LH, int NV>
__device__ __forceinline__ void group_totals(float (&v)[NV], int lane, float (&out)[NV]) {
  transpose_sum<LH / 2, NV, NV>(v, lane);
#pragma unroll
  for (int j = 0; j < NV; ++j) {
    if constexpr (LH == 1) out[j] = v[j];
    else if constexpr (LH <= NV) out[j] = __shfl_sync(0xffffffffu, v[j % (NV / LH)], j / (NV / LH), LH);
    else out[j] = __shfl_sync(0xffffffffu, v[0], j * (LH / NV), LH);
  }
}

// Fire-and-forget bulk prefetch of [p, p + bytes) into L2 (p 16-byte aligned,
// bytes a multiple of 16).
__device__ __forceinline__ void prefetch_l2_bulk(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(p), "r"(bytes) : "memory");
}

}  // namespace epikv
