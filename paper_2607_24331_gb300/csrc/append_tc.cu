// Tensor-core latent append (Sec. III-A z = x L, with the key factors of all
// Sec. III-C groups side by side and the Sec. III-D value factor):
//   kcache[rows[i]] = x_i A_k,   vcache[rows[i]] = x_i A_v
// as a tcgen05 GEMM, bf16 in, fp32 accumulate in TMEM, bf16 out.
//
// CTA tile 128 tokens x N_t (<= 256) columns of one of the two outputs; K in
// 64-wide stages staged by TMA (x: K-major, 128B swizzle; A: MN-major, 128B
// swizzle) through a 4-deep mbarrier ring.  Warp 0 issues TMA, warp 1 owns
// TMEM and issues tcgen05.mma, warps 2-5 drain the accumulator (one TMEM lane
// quadrant each).  Small batches (<= 256 tokens) split K over a cluster of four
// CTAs that add their partial sums through distributed shared memory
// (append_few_kernel below).  Longer appends (a prefill) with R_k and r_v
// multiples of 64 run on persistent CTA pairs (append_pair_kernel below).
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "sm100.cuh"
#include "tmap.h"

namespace dck {
namespace {

using namespace sm100;

constexpr int kBM = 128, kBK = 64, kMaxBN = 256, kStages = 4;
constexpr int kABytes = kBM * kBK * 2;          // 16 KB
constexpr int kBBytes = kBK * kMaxBN * 2;       // 32 KB
constexpr int kStageBytes = kABytes + kBBytes;
constexpr int kThreads = 192;
// Up to this many tokens K is split over clusters (append_few_kernel): the line of the
// split it replaced, at which its gain is largest, and not where the two kernels meet.
// Clusters / pairs, us, 32-head layer, 8-KV-head layer, 8-KV-head long-context layer:
// 256 tokens 16.8, 15.9, 8.9 / 23.6, 23.4, 23.4 (at 257); 300 22.4, 15.9, 14.4 / 24.0,
// 23.5, 23.4; 512 32.7, 24.2, 17.0 / 24.0, 23.7, 23.7; 1024 62.8, 40.4, 32.9 / 24.2,
// 24.3, 23.7 (the clusters' CTAs take two waves where they are level).
constexpr int kSplitMaxTok = 256;
// fp32 slices of a small batch's output that the workspace query asks for: no kernel
// uses them now, but a call without that space has always been refused.
constexpr int kMaxSplit = 32;

struct AppendParams {
  int n_tok, Rk, rv;
  int nt_k;      // N tiles over the key output
  int kblocks;   // ceil(D / 64)
  const int64_t* rows;  // cache row of each token
  __nv_bfloat16* kc;
  __nv_bfloat16* vc;
  int64_t n_rows;
  int* err;
  long long limit;  // kWithhold kernels: SM cycles after which the waits for operands give up
};

__device__ __forceinline__ void tile_of(const AppendParams& p, int t, bool& is_k, int& n0, int& nt) {
  is_k = t < p.nt_k;
  const int N = is_k ? p.Rk : p.rv;
  n0 = (is_k ? t : t - p.nt_k) * kMaxBN;
  nt = min(kMaxBN, N - n0);
}

// kWithhold: the self-test of the waits, whose last K block is never loaded.
template <bool kWithhold>
__global__ void __launch_bounds__(kThreads, 1)
    append_tc_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_ak,
                     const __grid_constant__ CUtensorMap tm_av, const AppendParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = align_1024(smem_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  uint64_t* empty = full + kStages;
  uint64_t* acc_bar = empty + kStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  bool is_k;
  int n0, nt;
  tile_of(p, blockIdx.x, is_k, n0, nt);
  const int m0 = blockIdx.y * kBM;
  const int nboxes = (nt + 63) / 64;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 256);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // programmatic dependent launch: the set-up above overlaps the previous
  // kernel's tail; every global access comes after that kernel is complete
  pdl_wait();
  pdl_launch_dependents();
  const uint32_t tmem = *tmem_slot;
  const CUtensorMap* tmb = is_k ? &tm_ak : &tm_av;

  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&tm_x);
    tma_prefetch_desc(tmb);
    for (int kb = 0; kb < p.kblocks - (kWithhold ? 1 : 0); ++kb) {
      const int s = kb % kStages;
      if (kb >= kStages && !mbar_wait(&empty[s], ((kb / kStages) - 1) & 1, abort_flag)) break;
      uint8_t* a = smem + s * kStageBytes;
      uint8_t* b = a + kABytes;
      mbar_expect_tx(&full[s], kABytes + nboxes * (kBK * 64 * 2));
      tma_load_2d(a, &tm_x, &full[s], kb * kBK, m0);
      for (int j = 0; j < nboxes; ++j) tma_load_2d(b + j * (kBK * 64 * 2), tmb, &full[s], n0 + 64 * j, kb * kBK);
    }
  } else if (warp == 1 && lane == 0) {
    const uint32_t idesc = idesc_bf16(kBM, nt, false, true);
    bool ok = true;
    for (int kb = 0; kb < p.kblocks; ++kb) {
      const int s = kb % kStages;
      if (!(ok = mbar_wait(&full[s], (kb / kStages) & 1, abort_flag, kWithhold ? p.limit : kWaitCycles))) break;
      tc_fence_after();
      const uint32_t a = smem_u32(smem + s * kStageBytes);
      const uint32_t b = a + kABytes;
#pragma unroll
      for (int k = 0; k < kBK / 16; ++k) {
        const uint64_t ad = sdesc(a + k * 32, 16, 1024, kSw128);
        const uint64_t bd = sdesc(b + k * 2048, kBK * 64 * 2, 1024, kSw128);
        umma_f16(tmem, ad, bd, idesc, (kb > 0 || k > 0) ? 1u : 0u);
      }
      umma_commit(&empty[s]);
    }
    if (ok) umma_commit(acc_bar);  // (a sum that is not whole is never announced)
  } else if (warp >= 2) {
    const int quad = warp & 3;
    const int m = m0 + quad * 32 + lane;
    const bool ok = __all_sync(0xffffffffu, mbar_wait(acc_bar, 0, abort_flag));
    tc_fence_after();
    int64_t row = -1;
    if (ok && m < p.n_tok) {
      row = p.rows[m];
      if (row < 0 || row >= p.n_rows) {
        atomicOr(p.err, kErrBadRow);
        row = -1;
      }
    }
    const int N = is_k ? p.Rk : p.rv;
    __nv_bfloat16* dst = is_k ? p.kc : p.vc;
    for (int c = 0; c < nt && ok; c += 16) {
      float v[16];
      tmem_ld16(tmem_addr(tmem, quad * 32, c), v);
      tmem_wait_ld();
      if (row >= 0) {
        uint4 pk[2];
        __nv_bfloat162* h2 = reinterpret_cast<__nv_bfloat162*>(pk);
#pragma unroll
        for (int i = 0; i < 8; ++i) h2[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
        uint4* o = reinterpret_cast<uint4*>(dst + row * N + n0 + c);
        o[0] = pk[0];
        o[1] = pk[1];
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    drain_in_flight();
    if (threadIdx.x == 0) atomicOr(p.err, kErrTimeout);
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
}

// ---------------------------------------------------------------------------
// Small batches (<= 256 tokens): a cluster of four CTAs per 128 tokens x 64
// output columns, CTA `rank` taking a quarter of K.  Bound by the latency of one
// pass over the factors (HBM, 2.5 us on the 32-head layer) and by each CTA's x
// stream from L2 (64 columns re-read it once per tile); seven 24 KB stages per
// CTA keep both in flight.  The CTAs push each 16-column slice of their partial
// sums into its owner rank's shared memory, meet at a cluster barrier, and every
// rank adds its slice's four partials and writes the rows.  (Partials through
// global memory, 19 slices written and read back by a second launch, took as long
// as the products: 19.4 us for 100 tokens on the 32-head layer.)
// ---------------------------------------------------------------------------

constexpr int kFN = 64;        // output columns of a cluster
constexpr int kFSplit = 4;     // K quarters = CTAs of a cluster; 16 columns of the sum each
constexpr int kFStages = 7;
constexpr int kFBBytes = kBK * kFN * 2;             // 8 KB
constexpr int kFStageBytes = kABytes + kFBBytes;
constexpr int kFRecvBytes = kFSplit * kBM * 16 * 4; // partial sums received: [source rank][token][16] fp32
static_assert(kFN == 16 * kFSplit, "a rank owns one 16-column slice");

// 16-byte chunk q of token row r in a slice: rotated over the rows, so that the
// pushes of a warp (one row per lane) spread over the banks.
__device__ __forceinline__ int few_chunk(int r, int q) { return (r * 4 + (q ^ ((r >> 1) & 3))) * 16; }

template <bool kWithhold>
__global__ void __launch_bounds__(kThreads, 1)
    append_few_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_ak,
                      const __grid_constant__ CUtensorMap tm_av, const AppendParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = align_1024(smem_raw);
  uint8_t* recv = smem + kFStages * kFStageBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(recv + kFRecvBytes);
  uint64_t* empty = full + kFStages;
  uint64_t* acc_bar = empty + kFStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int t = blockIdx.x / kFSplit;
  const bool is_k = t < p.nt_k;
  const int N = is_k ? p.Rk : p.rv, n0 = (is_k ? t : t - p.nt_k) * kFN;
  const int m0 = blockIdx.y * kBM;
  const int kb0 = rank * p.kblocks / kFSplit, kb1 = (rank + 1) * p.kblocks / kFSplit;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kFStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, kFN);
    tmem_relinquish();
  }
  tc_fence_before();
  cluster_sync();  // every CTA of the cluster runs: its shared memory may be written
  tc_fence_after();
  pdl_wait();
  pdl_launch_dependents();
  const uint32_t tmem = *tmem_slot;
  const CUtensorMap* tmb = is_k ? &tm_ak : &tm_av;
  // a wait that gave up stops the whole cluster: no rank adds sums that are not whole
  auto stop_cluster = [&]() {
    for (uint32_t c = 0; c < kFSplit; ++c) st_cluster_u32(mapa_shared(smem_u32((const void*)abort_flag), c), 1u);
  };

  if (warp == 0) {
    if (lane == 0) {
      const int kbe = kb1 - (kWithhold && rank == kFSplit - 1 ? 1 : 0);
      for (int kb = kb0; kb < kbe; ++kb) {
        const int i = kb - kb0, s = i % kFStages;
        if (i >= kFStages && !mbar_wait(&empty[s], ((i / kFStages) - 1) & 1, abort_flag)) {
          stop_cluster();
          break;
        }
        uint8_t* a = smem + s * kFStageBytes;
        mbar_expect_tx(&full[s], kFStageBytes);
        tma_load_2d(a + kABytes, tmb, &full[s], n0, kb * kBK);
        tma_load_2d(a, &tm_x, &full[s], kb * kBK, m0);
      }
    }
  } else if (warp == 1) {
    const bool el = elect_one();
    const uint32_t idesc = idesc_bf16(kBM, kFN, false, true), s0 = smem_u32(smem);
    const uint64_t da = sdesc(s0, 16, 1024, kSw128), db = sdesc(s0 + kABytes, kFBBytes, 1024, kSw128);
    bool ok = true;
    for (int i = 0; i < kb1 - kb0; ++i) {
      const int s = i % kFStages;
      ok = __all_sync(0xffffffffu, mbar_wait(&full[s], (i / kFStages) & 1, abort_flag,
                                             kWithhold ? p.limit : kWaitCycles));
      if (!ok) break;
      tc_fence_after();
      const uint64_t o = (uint64_t)(s * (kFStageBytes >> 4));
      if (el) {
#pragma unroll
        for (int k = 0; k < kBK / 16; ++k)
          umma_f16(tmem, da + o + 2 * k, db + o + 128 * k, idesc, (i > 0 || k > 0) ? 1u : 0u);
        umma_commit(&empty[s]);
      }
    }
    if (ok && el) umma_commit(acc_bar);
    if (!ok && lane == 0) stop_cluster();
  } else {
    const int quad = warp & 3, r = quad * 32 + lane;
    const bool ok = __all_sync(0xffffffffu, mbar_wait(acc_bar, 0, abort_flag));
    tc_fence_after();
    if (ok) {
#pragma unroll
      for (int c = 0; c < kFSplit; ++c) {
        float v[16];
        if (kb0 < kb1) {
          tmem_ld16(tmem_addr(tmem, quad * 32, 16 * c), v);
          tmem_wait_ld();
        } else {  // fewer K blocks than ranks
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = 0.f;
        }
        if (m0 + r < p.n_tok) {
          const uint32_t dst = mapa_shared(smem_u32(recv + rank * (kBM * 64)), (uint32_t)c);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst + few_chunk(r, q)),
                         "f"(v[4 * q]), "f"(v[4 * q + 1]), "f"(v[4 * q + 2]), "f"(v[4 * q + 3])
                         : "memory");
        }
      }
    } else if (lane == 0) {
      stop_cluster();
    }
  }
  tc_fence_before();
  __syncwarp();
  cluster_sync();  // every partial sum of this rank's slice has arrived, or the flag is set in every rank
  const bool stopped = *abort_flag != 0;
  if (stopped) {
    drain_in_flight();
    if (threadIdx.x == 0) atomicOr(p.err, kErrTimeout);
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kFN);
  }
  if (stopped) return;
  const int col = n0 + 16 * rank;
  __nv_bfloat16* dst = is_k ? p.kc : p.vc;
  for (int i = threadIdx.x; i < kBM * 4; i += kThreads) {
    const int r = i >> 2, q = i & 3;
    if (m0 + r >= p.n_tok) break;
    const int64_t row = p.rows[m0 + r];
    if (row < 0 || row >= p.n_rows) {
      atomicOr(p.err, kErrBadRow);
      continue;
    }
    if (col >= N) continue;  // the last tile of an output whose width is no multiple of 64
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int z = 0; z < kFSplit; ++z) {
      const float4 w = *reinterpret_cast<const float4*>(recv + z * (kBM * 64) + few_chunk(r, q));
      v = make_float4(v.x + w.x, v.y + w.y, v.z + w.z, v.w + w.w);
    }
    uint2 o;
    *reinterpret_cast<__nv_bfloat162*>(&o.x) = __floats2bfloat162_rn(v.x, v.y);
    *reinterpret_cast<__nv_bfloat162*>(&o.y) = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2*>(dst + row * N + col + 4 * q) = o;
  }
}

// ---------------------------------------------------------------------------
// Long appends (prefill): persistent CTA pairs.
//
// A pair tile covers 256 tokens (128 per CTA, its rows of the UMMA operand A:
// x) and w = 128 or 256 output columns of one of the two outputs (each CTA
// holding w/2 columns of operand B: A_k or A_v), the whole of K = D in 64-wide
// stages, one tcgen05 pair MMA (cta_group::2, M = 256) per 16 of K.  Per stage
// and CTA the operands are 16 KB of x and w/2 x 64 x 2 bytes of factor: at
// w = 256, 32 KB per 512 cycles of pair MMA, where the single-CTA tile of
// 128 x 256 above streams 48 KB per 512 cycles, more than an SM takes in from
// L2.  Tiles, flattened: for every 256-token block, the key output in
// 256-column tiles (the last one 128 wide when at most 128 columns remain;
// columns past R_k load as zeros and are not stored), then the value output
// likewise.  Pair p takes tiles p, p + P, p + 2P, ... of that list.  Two
// 256-column TMEM accumulators: the epilogue of one tile overlaps the next
// tile's MMAs.  The MMA schedule and the loads are run by whole warps with one
// lane issuing: 16384 tokens on the 8-KV-head long-context layer 116 -> 106 us
// (146 GFLOP; 76 us at the measured bf16 rate) against one-lane branches.  What
// bounds it now: the operands' 64 bytes per cycle and SM, and 4.75 tiles on the
// busiest pair for 3.8 on average.
// ---------------------------------------------------------------------------

constexpr int kPStages = 6;
constexpr int kPXBytes = kBM * kBK * 2;      // 16 KB: this CTA's 128 token rows x 64 of K
constexpr int kPBBytes = 2 * kBK * 64 * 2;   // 16 KB: up to 128 factor columns x 64 of K (64-column boxes)
constexpr int kPStageBytes = kPXBytes + kPBBytes;
constexpr int kPThreads = 192;
constexpr int kPRows = 2 * kBM;              // tokens of a pair tile
constexpr uint32_t kPTmemCols = 512;

// Pair tiles of one output of width N (a multiple of 64): 256-column tiles,
// the last one 128 wide when at most 128 columns remain.
__host__ __device__ inline int pt_count(int N) { return (N + 255) / 256; }
__host__ __device__ inline int pt_width(int N, int j) {
  return j + 1 < pt_count(N) || N - 256 * j > 128 ? 256 : 128;
}
struct PairTile {
  int m0;    // first token
  int out;   // 0: key output, 1: value output
  int n0;    // first output column
  int w;     // columns (128 or 256)
};

struct PairPlan {
  int tk, trow;  // key tiles, tiles of a 256-token block
  __device__ PairPlan(int Rk, int rv) : tk(pt_count(Rk)), trow(pt_count(Rk) + pt_count(rv)) {}
  __device__ PairTile tile(int64_t t, int Rk, int rv) const {
    const int64_t mt = t / trow;
    const int j = (int)(t - mt * trow);
    PairTile pt;
    pt.m0 = (int)(mt * kPRows);
    pt.out = j < tk ? 0 : 1;
    const int jj = pt.out ? j - tk : j;
    pt.n0 = 256 * jj;
    pt.w = pt_width(pt.out ? rv : Rk, jj);
    return pt;
  }
};

__global__ void __launch_bounds__(kPThreads, 1)
    append_pair_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_ak,
                       const __grid_constant__ CUtensorMap tm_av, const AppendParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = align_1024(smem_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kPStages * kPStageBytes);
  uint64_t* empty = full + kPStages;
  uint64_t* acc_full = empty + kPStages;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int hr = (int)cluster_ctarank();  // this CTA's half of every pair tile
  const bool leader = hr == 0;            // the even CTA issues the pair MMAs
  const int P = gridDim.x / 2, pair = blockIdx.x >> 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kPStages; ++s) {
      mbar_init(&full[s], 1);   // even CTA: its producer's expect_tx; both CTAs' copies complete on it
      mbar_init(&empty[s], 1);  // the pair MMAs' commit, in both CTAs
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 8);  // even CTA: the four epilogue warps of both CTAs
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, kPTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync();  // both CTAs' barriers initialised and TMEM allocated
  tc_fence_after();
  pdl_wait();
  pdl_launch_dependents();
  const uint32_t tmem = *tmem_slot;
  auto lead = [](const void* q) { return mapa_shared(smem_u32(q), 0); };
  auto stop_peer = [&]() { st_cluster_u32(mapa_shared(smem_u32((const void*)abort_flag), (uint32_t)(hr ^ 1)), 1u); };

  const PairPlan plan(p.Rk, p.rv);
  const int64_t n_mt = (p.n_tok + kPRows - 1) / kPRows;
  const int64_t n_tiles = n_mt * plan.trow;
  // pair p takes tiles p, p + P, p + 2P, ...: at any time the pairs work on P
  // consecutive tiles, the column tiles of a few token blocks, so a block's x
  // is read from HBM once and from L2 by the pairs of its other column tiles
  // (contiguous ranges per pair re-read x from HBM for every column tile:
  // 76 pairs' x blocks of 2 MB do not stay in L2 together)
  const int64_t t0 = pair, t1 = n_tiles, tstep = P;
  const int kb_n = p.kblocks;

  if (warp == 0) {
    // ---- TMA producer (both CTAs): this CTA's x rows and its half of the factor columns
    if (lane == 0) {
      tma_prefetch_desc(&tm_x);
      tma_prefetch_desc(&tm_ak);
      tma_prefetch_desc(&tm_av);
    }
    const bool el = elect_one();
    uint64_t pol_x;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol_x));
    const uint64_t pol_a = policy_evict_last();
    int s = 0, fills = 0;  // next stage, times round
    bool ok = true;
    for (int64_t t = t0; t < t1 && ok; t += tstep) {
      const PairTile pt = plan.tile(t, p.Rk, p.rv);
      const CUtensorMap* tb = pt.out ? &tm_av : &tm_ak;
      const int half = pt.w / 2;
      for (int kb = 0; kb < kb_n; ++kb) {
        if (fills && !(ok = __all_sync(0xffffffffu, mbar_wait(&empty[s], (uint32_t)((fills - 1) & 1), abort_flag))))
          break;
        if (el) {
          uint8_t* xs = smem + s * kPStageBytes;
          uint8_t* bs = xs + kPXBytes;
          const uint32_t bar = lead(&full[s]);
          if (leader) mbar_expect_tx(&full[s], 2u * (uint32_t)(kPXBytes + half * kBK * 2));
          tma_load_2d_pair(xs, &tm_x, bar, kb * kBK, pt.m0 + hr * kBM, pol_x);
          tma_load_2d_pair(bs, tb, bar, pt.n0 + hr * half, kb * kBK, pol_a);
          if (half > 64) tma_load_2d_pair(bs + kBK * 64 * 2, tb, bar, pt.n0 + hr * half + 64, kb * kBK, pol_a);
        }
        if (++s == kPStages) {
          s = 0;
          ++fills;
        }
      }
    }
    if (!ok && lane == 0) stop_peer();
  } else if (warp == 1) {
    // ---- pair MMAs (even CTA): the warp runs the schedule, one lane issues ----
    if (leader) {
      const bool el = elect_one();
      const uint32_t s0 = smem_u32(smem);
      const uint64_t dx = sdesc(s0, 16, 1024, kSw128), db = sdesc(s0 + kPXBytes, kBK * 64 * 2, 1024, kSw128);
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      int lt = 0;  // tiles of this pair so far
      for (int64_t t = t0; t < t1 && ok; t += tstep, ++lt) {
        const PairTile pt = plan.tile(t, p.Rk, p.rv);
        const int buf = lt & 1;
        if (lt >= 2 &&
            !(ok = __all_sync(0xffffffffu, mbar_wait(&acc_empty[buf], (uint32_t)(((lt >> 1) - 1) & 1), abort_flag))))
          break;
        const uint32_t idesc = pt.w == 256 ? idesc_bf16(kPRows, 256, false, true) : idesc_bf16(kPRows, 128, false, true);
        const uint32_t d = tmem + buf * 256;
        for (int kb = 0; kb < kb_n; ++kb) {
          if (!(ok = __all_sync(0xffffffffu, mbar_wait(&full[s], ph, abort_flag)))) break;
          tc_fence_after();
          const uint64_t o = (uint64_t)(s * (kPStageBytes >> 4));
          if (el) {
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k)
              umma_f16_pair(d, dx + o + 2 * k, db + o + 128 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
            umma_commit_pair(&empty[s]);  // the stage's slots in both CTAs, once these MMAs are done
          }
          if (++s == kPStages) {
            s = 0;
            ph ^= 1;
          }
        }
        if (ok && el) umma_commit_pair(&acc_full[buf]);
      }
      if (!ok && lane == 0) stop_peer();
    }
    __syncwarp();
  } else {
    // ---- epilogue (warps 2-5, both CTAs): this CTA's 128 rows of each tile -----
    const int quad = warp & 3;
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
    int lt = 0;
    bool ok = true;
    for (int64_t t = t0; t < t1 && ok; t += tstep, ++lt) {
      const PairTile pt = plan.tile(t, p.Rk, p.rv);
      const int buf = lt & 1;
      ok = mbar_wait(&acc_full[buf], (uint32_t)((lt >> 1) & 1), abort_flag);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after();
      const int m = pt.m0 + hr * kBM + quad * 32 + lane;
      int64_t row = -1;
      if (m < p.n_tok) {
        row = p.rows[m];
        if (row < 0 || row >= p.n_rows) {
          atomicOr(p.err, kErrBadRow);
          row = -1;
        }
      }
      const int N = pt.out ? p.rv : p.Rk;
      __nv_bfloat16* dst = pt.out ? p.vc : p.kc;
      for (int c = 0; c < pt.w; c += 32) {
        float v[32];
        tmem_ld32(tmem + lane_base + buf * 256 + c, v);
        tmem_wait_ld();
        if (row >= 0 && pt.n0 + c < N) {  // N and n0 are multiples of 64: a 32-column chunk is all in or all out
          uint4 pk[4];
          __nv_bfloat162* h2 = reinterpret_cast<__nv_bfloat162*>(pk);
#pragma unroll
          for (int i = 0; i < 16; ++i) h2[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
          uint4* o = reinterpret_cast<uint4*>(dst + row * N + pt.n0 + c);
#pragma unroll
          for (int i = 0; i < 4; ++i) o[i] = pk[i];
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (leader) mbar_arrive(&acc_empty[buf]);
        else mbar_arrive_cluster(lead(&acc_empty[buf]));
      }
    }
    if (!ok && lane == 0) stop_peer();
  }
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    drain_in_flight();
    if (threadIdx.x == 0) atomicOr(p.err, kErrTimeout);
  }
  cluster_sync();  // the peer no longer reads this CTA's operands or arrives on its barriers
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, kPTmemCols);
  }
}

// CTA pairs of the pair kernel that fit the device at once (one CTA per SM).
int append_pairs_of_device(size_t smem) {
  static int cache[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (cache[dev]) return cache[dev];
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (sms / 2));
  cfg.blockDim = dim3(kPThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, append_pair_kernel, &cfg) != cudaSuccess || n <= 0) {
    cudaGetLastError();
    return 0;
  }
  cache[dev] = std::min(n, sms / 2);
  return cache[dev];
}

}  // namespace

bool tc_append_supports(int D, int Rk, int rv, int dtype) {
  return dtype == DCK_BF16 && D % 8 == 0 && Rk % 16 == 0 && rv % 16 == 0;
}

size_t tc_append_workspace(int n_tok, int Rk, int rv) {
  return n_tok <= kSplitMaxTok ? align_up((size_t)kMaxSplit * n_tok * (Rk + rv) * sizeof(float), 256) : 0;
}

// withhold_limit > 0: the self-test of the waits (see kWithhold), with that limit.
cudaError_t launch_append_tc(const void* x, int n_tok, int D, const void* A_k, const void* A_v, int Rk, int rv,
                             const int64_t* rows, void* kc, void* vc, int64_t n_rows, int* err, cudaStream_t s,
                             int* n_launches, long long withhold_limit) {
  *n_launches = 1;
  const bool withhold = withhold_limit > 0;
  AppendParams p;
  p.n_tok = n_tok;
  p.Rk = Rk;
  p.rv = rv;
  p.nt_k = (Rk + kMaxBN - 1) / kMaxBN;
  p.kblocks = (D + kBK - 1) / kBK;
  p.rows = rows;
  p.kc = static_cast<__nv_bfloat16*>(kc);
  p.vc = static_cast<__nv_bfloat16*>(vc);
  p.n_rows = n_rows;
  p.err = err;
  p.limit = withhold_limit;
  CUtensorMap tx, tk, tv;
  if (!make_tmap_2d_bf16(&tx, x, D, n_tok, (uint64_t)D * 2, kBK, kBM, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !make_tmap_2d_bf16(&tk, A_k, Rk, D, (uint64_t)Rk * 2, 64, kBK, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !make_tmap_2d_bf16(&tv, A_v, rv, D, (uint64_t)rv * 2, 64, kBK, CU_TENSOR_MAP_SWIZZLE_128B))
    return cudaErrorInvalidValue;
  if (n_tok > kSplitMaxTok && Rk % 64 == 0 && rv % 64 == 0) {
    // long append: persistent CTA pairs over 256-token x 256-column tiles
    const size_t psmem = (size_t)kPStages * kPStageBytes + 1024 + 256;
    cudaError_t e = cudaFuncSetAttribute(append_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psmem);
    if (e != cudaSuccess) return e;
    const int pairs = append_pairs_of_device(psmem);
    if (withhold) return cudaErrorNotSupported;
    if (pairs > 0) {
      const int64_t n_mt = (n_tok + kPRows - 1) / kPRows;
      const int64_t tiles = n_mt * (pt_count(Rk) + pt_count(rv));
      const int P = (int)std::min<int64_t>(pairs, tiles);
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(2 * P);
      cfg.blockDim = dim3(kPThreads);
      cfg.dynamicSmemBytes = psmem;
      cfg.stream = s;
      cudaLaunchAttribute attr[2];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 2;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[1].val.programmaticStreamSerializationAllowed = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 2;
      return cudaLaunchKernelEx(&cfg, append_pair_kernel, tx, tk, tv, p);
    }
  }
  if (n_tok <= kSplitMaxTok) {
    p.nt_k = (Rk + kFN - 1) / kFN;
    const size_t fsmem = (size_t)kFStages * kFStageBytes + kFRecvBytes + 1024 + 256;
    auto k = withhold ? append_few_kernel<true> : append_few_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fsmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kFSplit * (p.nt_k + (rv + kFN - 1) / kFN), (n_tok + kBM - 1) / kBM);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = fsmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kFSplit;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, k, tx, tk, tv, p);
  }
  const int ntiles = p.nt_k + (rv + kMaxBN - 1) / kMaxBN;
  const size_t smem = (size_t)kStages * kStageBytes + 1024 + 256;
  auto k = withhold ? append_tc_kernel<true> : append_tc_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k, dim3(ntiles, (n_tok + kBM - 1) / kBM), dim3(kThreads), smem, s, tx, tk, tv, p);
}

}  // namespace dck
