// Internal declarations shared by the libdck translation units.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/dck.h"

namespace dck {

constexpr int kMaxKvHeads = 128;
constexpr int kMaxGroups = 128;
constexpr int kMaxQPerKv = 8;     // query heads per KV head handled by the kernels
constexpr int kMaxRankV = 2048;
constexpr int kMaxBatch = 4096;
constexpr int kMaxPrefillLen = 1 << 24;  // bound on a prefill call's q_max and max_seq_len
constexpr int kTile = 128;        // tokens per work tile (one UMMA M block)
constexpr int kSimtTile = 32;     // tokens per work tile of the CUDA-core path

// Device error word values (bit flags).
constexpr int kErrBadSeq = 1;     // a sequence's rows fall outside the cache
constexpr int kErrBadRow = 2;     // an append destination row is outside the cache
constexpr int kErrTimeout = 4;    // a bounded wait gave up

// Group table and shapes of one layer, passed by value to the kernels.
struct LayerTable {
  int32_t Hq, Hkv, d, G, Rk, rv, qpg;
  int32_t head_group[kMaxKvHeads];  // KV head -> group
  int32_t head_slot[kMaxKvHeads];   // KV head -> column-block slot in its group
  int32_t grp_rank[kMaxGroups];     // r_g
  int32_t grp_roff[kMaxGroups];     // first key-cache column of group g
  int32_t grp_nh[kMaxGroups];       // n_g
  int64_t grp_boff[kMaxGroups];     // element offset of B_g in the packed B_k
};

// Work decomposition of a decode call on the CUDA-core path: every sequence is
// cut into kSimtTile-token tiles; the flattened tile list is split into n_items
// contiguous ranges (item c: tiles [floor(c*NT/n), floor((c+1)*NT/n))).  Item c
// writes one partial per sequence b it touches, in slot c + b.  (Tensor-core
// path: the pair-tile plan of tc_common.cuh.)
struct DecodeArgs {
  const void* q;
  const void* kc;
  const void* vc;
  const void* Bk;
  const void* Bv;
  const int64_t* seq_start;
  const int32_t* seq_len;
  int64_t n_rows;
  int32_t B;
  int32_t n_items;
  int32_t fine_below;  // tensor-core path: the pair-tile plan of tc_common.cuh (n_items = 2 x CTA pairs), its fine
                       // split below this many tiles per pair (see main_tiles); 0: CUDA-core path
  float theta;
  float* part_u;   // [n_slots, Hq, rv]
  float* part_ml;  // [n_slots, Hq, 2]  (running max in log2 units, sum)
  void* out;       // [B, Hq, d]
  int* err;
  struct LaunchHook* hook;  // host-side launch count and optional timing events (never read by kernels)
  void* extra;     // workspace region of the tensor-core path (per-sequence folded factors)
};

// Host-side record of the kernels one entry-point call puts on its stream.
// When `n_ev` > 0, ev[0] (a cudaEvent_t) is recorded before the call's first
// kernel, ev[k] after its k-th kernel for k < n_ev - 1 and ev[n_ev - 1] after
// its last kernel, so that a caller can time the whole call (n_ev = 2, nothing
// recorded between the kernels) or every kernel of it (n_ev = kernels + 1).
struct LaunchHook {
  void* const* ev = nullptr;
  int n_ev = 0;
  int count = 0;
};
inline cudaError_t hook_begin(LaunchHook* h, cudaStream_t s);     // before the first kernel
inline cudaError_t hook_launched(LaunchHook* h, cudaStream_t s);  // after each kernel launch
inline cudaError_t hook_end(LaunchHook* h, cudaStream_t s);       // after the call's last kernel

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Host launchers (each defined in its own translation unit).
int simt_items(const LayerTable& lt, int dtype, int B, int64_t n_rows, int sms);
cudaError_t launch_decode_simt(const LayerTable& lt, const DecodeArgs& a, int dtype, bool after_append,
                               cudaStream_t s);
cudaError_t launch_combine(const LayerTable& lt, const DecodeArgs& a, int dtype, cudaStream_t s);
cudaError_t launch_append_simt(const void* x, int n_tok, int D, const void* A_k, const void* A_v, int Rk,
                               int rv, const int64_t* rows, void* kc, void* vc, int64_t n_rows, int dtype,
                               int* err, cudaStream_t s);
cudaError_t launch_synth_gaussian(void* dst, int64_t n, uint64_t key, int64_t start, float scale, int dtype,
                                  cudaStream_t s);
// Host-side argument checks shared by the decode entry points (no CUDA call).
dck_status decode_precheck(const dck_layer_desc* desc, const void* q, const void* kcache, const void* vcache,
                           int64_t n_rows, const void* B_k, const void* B_v, const int64_t* d_seq_start,
                           const int32_t* d_seq_len, int32_t batch, float rope_theta, const void* out);

// ---------------------------------------------------------------------------
// device helpers
// ---------------------------------------------------------------------------

template <typename T>
__device__ __forceinline__ float to_f32(T v);
template <>
__device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename T>
__device__ __forceinline__ T from_f32(float v);
template <>
__device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// Number of `tile`-token tiles of every sequence, as an exclusive prefix in
// shared memory prefix[0..B] (scratch: one int per warp).  Sequences whose rows
// fall outside the cache count as empty and raise kErrBadSeq.  Must be called
// by the whole block (full warps).  Returns the total tile count NT.
__device__ __forceinline__ int build_tile_prefix(const int32_t* __restrict__ seq_len,
                                                 const int64_t* __restrict__ seq_start, int B,
                                                 int64_t n_rows, int* prefix, int* scratch, int* err,
                                                 bool report, int tile) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  int base = 0;
  for (int c0 = 0; c0 < B; c0 += blockDim.x) {  // a sequence per thread
    const int b = c0 + (int)threadIdx.x;
    int n = 0;
    if (b < B) {
      int64_t L = seq_len[b];
      const int64_t st = seq_start[b];
      if (L < 0 || st < 0 || st + L > n_rows) {
        if (report) atomicOr(err, kErrBadSeq);
        L = 0;
      }
      n = (int)((L + tile - 1) / tile);
    }
    int v = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    if (lane == 31) scratch[warp] = v;
    __syncthreads();
    int before = base, all = base;
    for (int w = 0; w < nw; ++w) {
      if (w < warp) before += scratch[w];
      all += scratch[w];
    }
    if (b < B) prefix[b] = before + v - n;
    base = all;
    __syncthreads();
  }
  if (threadIdx.x == 0) prefix[B] = base;
  __syncthreads();
  return base;
}

// Length of sequence b as used by the kernels (0 when its rows are invalid).
__device__ __forceinline__ int valid_len(const int32_t* seq_len, const int64_t* seq_start, int b,
                                         int64_t n_rows) {
  int64_t L = seq_len[b];
  int64_t st = seq_start[b];
  if (L < 0 || st < 0 || st + L > n_rows) return 0;
  return (int)L;
}

__host__ __device__ __forceinline__ int item_begin(int c, int NT, int n_items) {
  return (int)(((int64_t)c * NT) / n_items);
}

// 16-byte global -> shared copies tracked per thread (cp.async groups).
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  cp_async16((uint32_t)__cvta_generic_to_shared(dst), src);
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the last N groups of this thread have landed
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Programmatic dependent launch: a kernel launched with launch_pdl may start
// while the previous kernel on the stream finishes; pdl_wait() returns once
// that kernel is complete and its memory visible (a no-op without PDL), and
// pdl_launch_dependents() lets the next kernel launch early in turn.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                              Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Args&&>(args)...);
}

// Tiles [0, main_tiles) are split in contiguous whole-tile ranges over the
// n_items work items: all of them, or only n_items * floor(NT / n_items), the rest
// ("extra tiles") being shared out more finely (see tc_common.cuh; fine_below 0, on
// the CUDA-core path: never).  A whole tile more on some CTAs costs the call a tile's
// time; an extra tile costs each of its CTAs a segment (a tile end, a partial), and
// there are more of those the more tiles are left over.  So fewer than kFineAlways
// tiles per item are always shared out, fewer than `fine_below` where no more than 3/8
// of a tile per item are left over.  Calls of the 32-head MHA layer, us, shared out /
// not, by tiles per CTA pair:
//   8.1 224 / 236    8.5 240 / 236    8.9 257 / 242    8.1, 9.9 (32 ragged sequences) 246 / 258, 298 / 284
//   16.1 401 / 410   16.5 415 / 413   16.9 433 / 417
//   31.1 731 / 736   31.5 748 / 741   31.9 765 / 742   48.1 1100 / 1107
// (from 32 tiles on a gain of 1% at most).  With several query heads per KV head a
// segment also rotates its queries again: 8.1 140 / 142, 8.5 150 / 143, 12.1 183 / 185
// and 16.1 228 / 229 on the 8-KV-head layer, so nothing is shared out from 8 tiles on.
// (Below 8 the share matters as much, 4.1 93 / 96 and 4.9 115 / 99 there: not used.)
constexpr int kFineAlways = 8;
__host__ __device__ __forceinline__ int main_tiles(int NT, int n_items, int fine_below) {
  const int q = NT / n_items, whole = q * n_items;
  const bool fine = q < fine_below && (q < kFineAlways || 8 * (NT - whole) <= 3 * n_items);
  return fine ? whole : NT;
}
inline int fine_split_below(int qpg) { return qpg == 1 ? 32 : kFineAlways; }

// The item whose tile range contains tile x (0 <= x < NT).
__device__ __forceinline__ int item_of_tile(int x, int NT, int n_items) {
  return (int)((((int64_t)(x + 1) * n_items) + NT - 1) / NT) - 1;
}

// Sequence owning flattened tile x: largest b with prefix[b] <= x and a
// non-empty tile range.
__device__ __forceinline__ int seq_of_tile(const int* prefix, int B, int x) {
  int lo = 0, hi = B - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

}  // namespace dck

namespace dck {
// Records a caller's timing event on `s`; inside stream capture it becomes an
// external event node, so that it can be timed after each graph replay.
inline cudaError_t record_timing_event(void* ev, cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess) return cudaErrorUnknown;
  if (st == cudaStreamCaptureStatusActive)
    return cudaEventRecordWithFlags(static_cast<cudaEvent_t>(ev), s, cudaEventRecordExternal);
  return cudaEventRecord(static_cast<cudaEvent_t>(ev), s);
}

inline cudaError_t hook_begin(LaunchHook* h, cudaStream_t s) {
  if (!h || h->n_ev <= 0) return cudaSuccess;
  return record_timing_event(h->ev[0], s);
}

// Events between kernels stop programmatic dependent launch from starting the
// next kernel early, so only the brackets a caller asked for are recorded:
// ev[k] after the k-th kernel for k < n_ev - 1, and ev[n_ev - 1] once, after
// the call's last kernel (hook_end).
inline cudaError_t hook_launched(LaunchHook* h, cudaStream_t s) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !h) return e;
  ++h->count;
  if (h->count >= h->n_ev - 1) return cudaSuccess;
  return record_timing_event(h->ev[h->count], s);
}

inline cudaError_t hook_end(LaunchHook* h, cudaStream_t s) {
  if (!h || h->n_ev <= 0) return cudaSuccess;
  return record_timing_event(h->ev[h->n_ev - 1], s);
}
}  // namespace dck
