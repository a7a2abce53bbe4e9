// Tensor-core (tcgen05) decode attention over DynaCalKV latent caches, bf16:
// the scores kernel (key reconstruction, RoPE, scores, online softmax).
//
// The kernel runs as persistent CTA pairs: a cluster of two CTAs on the two
// SMs of a TPC issues one tcgen05 pair MMA (cta_group::2) over a pair tile of
// 256 tokens, the even CTA holding the first 128 tokens' latents and the odd
// CTA the rest (the work plan is in tc_common.cuh).  For every pair tile and
// every key group g (Sec. III-C) the group's latent tile C_g [256 tokens x r_g]
// meets the factor columns of the group's KV heads, two heads per MMA where the
// group has them (M = 256 tokens, N = 256 or 128, K = r_g; each CTA holds the
// factor columns of one head, or one half of a lone head, and receives the
// fp32 accumulator rows of its own 128 tokens in its TMEM).  A pair MMA moves
// each SM's share of the factor operand once per 256 tokens instead of once
// per 128, and halves the MMA instructions per token.  Two 256-column
// accumulators (all of TMEM) let the epilogue read one unit while the tensor
// cores compute the next.  Per head:
//
//  * key mode (several query heads per KV head): the factor is B_g[:, slot(h)],
//    the product is the reconstructed key K^_h = C_g B_g[:, slot(h)]
//    (Sec. III-A x W ~ z R); the epilogue applies RoPE at the token's position
//    and scores every query head of h against its query rotated to L-1;
//
//  * query-folded mode (one query head per KV head): RoPE is a rotation of
//    each frequency pair, so <R_P q, R_t k> = sum_i cos(t w_i) (a_i x_i + b_i y_i)
//    + sin(t w_i) (b_i x_i - a_i y_i) with (a, b) the halves of q' = R_P q and
//    (x, y) those of k.  With k = c B_g[:, slot] both brackets are linear in the
//    latent c, so a per-sequence factor W (columns 2i and 2i+1:
//    a_i B[:, i] + b_i B[:, i+64] and b_i B[:, i] - a_i B[:, i+64]) gives
//    Y = C_g W on the tensor cores with the same flops, and the score is
//    sum_i cos(t w_i) Y[2i] + sin(t w_i) Y[2i+1]: two FMAs per frequency pair.
//
// Factor items (one latent piece's ranks x 128 columns of each head of a
// unit) are prepared once per call by factor_prep_kernel as the exact
// 128B-swizzled shared-memory image of the UMMA B operand (heads * ranks * 256
// bytes each, in consumption order); each CTA of a pair loads its half of an
// item (its head, or its half of a lone head) with one TMA copy.
//
// Scores are in log2 units; the online softmax keeps a per-head reference max
// that moves only when a tile's max exceeds it by 8 (probabilities <= 256).
// Each CTA runs the softmax of its own 128-token halves: their probabilities P
// (bf16, laid out as the B operand of the value absorption) and the reference
// maxima they were computed with go to the workspace per 128-token tile; at
// the end of each segment the reference max and the row sum (over the rounded
// P) are written as the segment's split partial.  The absorption kernel
// (absorb_tc.cu) forms U = C_v^T P from them.
//
// Warp roles (640 threads), in both CTAs unless noted; the copies of both CTAs
// complete on the even CTA's barriers, which its MMA warps wait on:
//   warp 0     latent pieces of C_g (ring A)
//   warp 2     factor items (ring W)
//   warp 1     TMEM owner; in the even CTA it issues pair MMAs (in query-folded
//              mode every other unit, warp 3 the others into the other
//              accumulator, so that one warp's waits and commits overlap the
//              other's MMAs); the MMA commits arrive on both CTAs' barriers
//   warps 4-19 epilogue: each TMEM lane quadrant (32 tokens) is served by four
//              warps, each with 16 of the 64 RoPE frequency pairs of every head;
//              their partial scores go to one shared-memory array per frequency
//              quarter, summed at the tile end.  Both CTAs' epilogues release an
//              accumulator on the even CTA's barrier.
// What bounds it: the chain of one accumulator (MMAs, commit, epilogue reads,
// release; all of TMEM is two 256-column accumulators) and the epilogue's work
// per unit, about 1.3 k cycles each against 1.1 k of MMAs on the 32-head MHA layer
// (clock64 timelines).  With eight epilogue warps of 32 frequencies each, whose
// loads, arithmetic and hand-offs ran in series, a unit took 2.2 k (query-folded)
// and 3.0 k (key mode); key mode's keys went through shared memory to reach the
// score MMA's operand layout, which the 16x256b TMEM load gives directly.  The
// rings hand out single pieces and items: with whole units, a second unit of
// three items did not fit and its load came after the first one's MMAs.
// Whole calls before / with these: 32-head MHA 16 x 4096 169.5 / 147.6 us, 32 ragged
// 367 / 321; GQA 8 x 32768 251 / 228, 2 x 131072 286 / 222 (with the changes of the
// other kernels and shared-space addressing since: 129, 251, 191, 189).
// Every wait is bounded (about 2 s); on expiry the CTA stops issuing work,
// tells its peer to stop, records kErrTimeout, waits for work in flight and
// still releases TMEM.
//
// Shared-memory operand layouts (128B swizzle unless noted), identical in both
// CTAs (a pair MMA reads the same offsets in each):
//   A slot  [128 tokens][w ranks] K-major, w in {64, 32, 16} with 128/64/32B
//           swizzle: this CTA's rows of the UMMA operand A;
//   W slot  [2 halves][w ranks][64 columns] MN-major (one head), or
//           [w ranks][64 columns] (half of a lone head): this CTA's columns of
//           operand B (the 64-column atoms w * 128 bytes apart);
// P ([2 token atoms][Hq_pad heads][64 tokens] bf16, K-major: the absorption's
// operand B) is written straight to the workspace by the tile-end owners.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>

#include "rope.cuh"
#include "tc_common.cuh"
#include "tc_host.h"
#include "tmap.h"

namespace dck {
namespace {

using namespace sm100;
using namespace tc;

constexpr int kD = 128;
constexpr int kSlot = 16384;     // latent slots: 128 tokens x 64 ranks
constexpr int kSlotW = 16384;    // factor slots: one head (2 x 64 ranks x 64 columns) of an item
constexpr int kMaxGroupsTc = 16;
constexpr int kMaxPieces = 5;
constexpr int kMaxHqTc = 32;
constexpr int kMaxItems = 256;
constexpr int kMaxUnits = 32;
constexpr int kCtlWarps = 4;      // producers and MMA issuers
constexpr int kEpiWarps = 16;
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kThreadsTc = 32 * kCtlWarps + kEpiThreads;
constexpr int kFreqW = kD / 2 / 4;  // RoPE pairs of a frequency quarter
constexpr float kRescaleThr = 8.f;  // log2 units: probabilities stay <= 256
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kKCols = 256;    // TMEM columns of one key accumulator
constexpr float kTurn32 = 1.4629180792671596e-9f;  // 2 pi / 2^32
constexpr float kLog2e = 1.4426950408889634f;

// Full barriers of the factor ring.  An MMA warp passes over the other's items
// without waiting for them, so it may wait for an item whose slot still awaits an
// earlier fill: with a barrier per slot it would take an older phase for that
// item's.  With 16, the item 16 earlier is complete whenever a warp waits: its own
// last item is at most 10 back (units of up to 5 items), and an item is loaded
// only once the one NW <= 5 before it has been read.
constexpr int kItemBars = 16;

template <bool kFold>
struct Ring {
  // latent-piece slots (16 KB each) and factor-item slots (half items, 16 KB
  // each): what the scores leave of shared memory.  The latent ring holds the
  // group in use while the next group's pieces arrive from HBM.
  static constexpr int NA = 5;
  static constexpr int NW = kFold ? 5 : 4;
  // MMA-issuing warps: two in query-folded mode; key mode's units carry up
  // to four items, which one warp streams better
  static constexpr int kMma = kFold ? 2 : 1;
};

// Latent-piece maps (box 64/32/16 ranks x 128 tokens, 128/64/32B swizzle) and
// factor-image maps (rows of 128 bytes, box 16/32/64/128 rows, no swizzle: the
// images are stored pre-swizzled).
struct Maps {
  CUtensorMap kc64, kc32, kc16;
  CUtensorMap im[4];
};

// Per-group facts the hot loops need; copied to shared memory at kernel start
// (indexing kernel-parameter tables at run time goes through the small constant
// cache, which several warps would share).  32 bytes each: at 24 the 32-head layer's
// steps took 2% longer (16 x 4096 tokens 128.7 -> 130.9 us).
struct alignas(32) GroupSm {
  int32_t roff;          // first key-cache column of the group
  int8_t np;             // latent pieces
  int8_t nh;             // heads
  int8_t nu;             // units (pairs of heads, the last one single when nh is odd)
  int8_t w[kMaxPieces];  // piece widths (ranks)
  int16_t u0;            // the group's first unit in the tile's unit order
  int16_t k[kMaxPieces]; // first rank of each piece
};

struct TcArgs {
  int hq_pad;
  int n_pairs;                   // P
  int64_t fimg_seq_bytes;        // factor image bytes per sequence (query-folded mode)
  uint8_t* pglob;                // per-tile P images (workspace)
  float* mglob;                  // per-tile reference maxima (workspace)
  int64_t max_tiles;
  RopeFreqs rf;                  // RoPE frequencies theta^(-2i/d) in turns
  GroupSm grp[kMaxGroupsTc];
  int n_units;                   // units per tile
  uint32_t uinfo[kMaxUnits];     // KV heads of each unit: first | second << 8 | count << 16
  int16_t uitem[kMaxUnits + 1];  // first factor item of each unit (and the item count)
  int8_t hunit[kMaxHqTc];        // unit of each query head
  uint32_t item[kMaxItems];      // factor item n: byte offset | (bytes / 4096) << 26
};

template <bool kFold>
struct Smem {
  uint8_t a[Ring<kFold>::NA][kSlot];
  uint8_t w[Ring<kFold>::NW][kSlotW];
  // scores [frequency quarter][query head][token]: each quarter's partial
  // scores by plain stores, summed at the tile end
  float x[4 * kMaxHqTc * 128];
  // key mode: rotated queries * log2(e)/sqrt(d), bf16 [query head][d] (the
  // B operand of the warps' score MMAs)
  __nv_bfloat16 qr[kFold ? 2 : kMaxHqTc * kD];
  uint2 freq[kD / 2];
  uint64_t a_full[Ring<kFold>::NA], a_empty[Ring<kFold>::NA];  // latent pieces
  uint64_t w_full[kItemBars], w_empty[Ring<kFold>::NW];        // factor items (full: item % kItemBars; empty: slot)
  uint64_t k_full[2], k_empty[2], epi_bar, x_free;
  GroupSm grp[kMaxGroupsTc];
  uint32_t uinfo[kMaxUnits];
  int8_t hunit[kMaxHqTc];
  uint32_t tmem_base;
  int abort_flag;
};

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
// d += a b for one 16 x 8 x 16 tile, bf16 inputs, fp32 accumulators.
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Rows (of 128 bytes) of a half item of `bytes` bytes -> factor-image map index.
__device__ __forceinline__ int im_map_of(uint32_t half_rows) {
  return half_rows == 16 ? 0 : (half_rows == 32 ? 1 : (half_rows == 64 ? 2 : 3));
}

// ---------------------------------------------------------------------------
// the scores kernel
// ---------------------------------------------------------------------------

template <bool kFold>
__global__ void __launch_bounds__(kThreadsTc, 1)
    decode_tc_kernel(const __grid_constant__ Maps maps, const LayerTable lt, const DecodeArgs a,
                     const __grid_constant__ TcArgs ta) {
  constexpr int kMma = Ring<kFold>::kMma, NW = Ring<kFold>::NW, kNA = Ring<kFold>::NA;
  extern __shared__ uint8_t smem_raw[];
  Smem<kFold>& sm = *reinterpret_cast<Smem<kFold>*>(align_1024(smem_raw));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  volatile int* abort_flag = &sm.abort_flag;
  const int hq_pad = ta.hq_pad;
  const int Hq = lt.Hq, qpg = lt.qpg;
  const int hr = (int)cluster_ctarank();  // the half of every pair tile this CTA holds
  const bool leader = hr == 0;            // the even CTA issues the pair MMAs
  const int P = ta.n_pairs, pair = blockIdx.x >> 1;

  // ---- setup -------------------------------------------------------------
  if (warp == 0) {  // a barrier per lane
    if (lane < kItemBars) mbar_init(&sm.w_full[lane], 1);
    if (lane < kNA) {
      mbar_init(&sm.a_full[lane], 1);      // even CTA: its producer's expect_tx; both CTAs' copies complete on it
      mbar_init(&sm.a_empty[lane], kMma);  // released by every MMA warp (arrivals reach both CTAs)
    }
    if (lane < NW) mbar_init(&sm.w_empty[lane], 1);
    if (lane < 2) {
      mbar_init(&sm.k_full[lane], 1);
      mbar_init(&sm.k_empty[lane], 2 * kEpiWarps);  // even CTA: both CTAs' epilogue warps
    }
    if (lane == 0) {
      mbar_init(&sm.epi_bar, kEpiWarps);
      mbar_init(&sm.x_free, kEpiWarps);
      sm.abort_flag = 0;
      tma_prefetch_desc(&maps.kc64);
      tma_prefetch_desc(&maps.im[3]);
    }
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(&sm.tmem_base, kTmemCols);
    tmem_relinquish_pair();
  }
  if (tid < lt.G) sm.grp[tid] = ta.grp[tid];
  if (tid < ta.n_units) sm.uinfo[tid] = ta.uinfo[tid];
  if (tid < Hq) sm.hunit[tid] = ta.hunit[tid];
  if (tid < kD / 2) sm.freq[tid] = ta.rf.f[tid];
  // Work of this pair: main pair tiles [X0, X1) (every unit), then units
  // [u_lo, u_hi) of the flattened (extra tile, unit) list, every extra tile a
  // segment of its own.
  const int U = ta.n_units;
  __shared__ PairScratch sc;
  const PairScan scan = pair_scan(a, sc);
  const int NP = scan.total256, NT128 = scan.total128;
  const PSplit sp(NP, P, a.fine_below);
  // the per-tile stores are sized for non-overlapping sequences; more tiles
  // than that is reported as invalid input and nothing is computed
  const bool fits = NT128 <= ta.max_tiles;
  if (!fits && tid == 0 && blockIdx.x == 0) atomicOr(a.err, kErrBadSeq);
  const int X0 = fits ? sp.main_begin(pair, P) : 0;
  const int X1 = fits ? sp.main_begin(pair + 1, P) : 0;
  const int xu = sp.R * U;
  const int u_lo = fits ? pair * xu / P : 0;  // (fewer than P extra tiles)
  const int u_hi = fits ? (pair + 1) * xu / P : 0;
  const int xe0 = sp.NPm + (u_lo < u_hi ? u_lo / U : 0), xe1 = sp.NPm + (u_lo < u_hi ? (u_hi - 1) / U + 1 : 0);
  pair_find(a, scan, X0, xe0, sc);
  const bool has_work = X0 < X1 || xe0 < xe1;  // the same in both CTAs of the pair
  // units [ua, ub) of flattened pair tile X in phase ph (0: main, 1: extra)
  auto units_of = [&](int ph, int X, int& ua, int& ub) {
    ua = 0;
    ub = U;
    if (ph) {
      const int e = X - sp.NPm;
      ua = max(u_lo - e * U, 0);
      ub = min(u_hi - e * U, U);
    }
  };
  tc_fence_before();
  cluster_sync();  // both CTAs' barriers initialised and TMEM allocated, the walkers' starts found
  tc_fence_after();
  auto walker = [&](int ph) {  // main or extra pair tiles of this pair
    return pair_walker(sc.at[ph], ph ? xe0 : X0, ph ? xe1 : X1, ph != 0);
  };
  const uint32_t tmem = sm.tmem_base;
  // shared::cluster addresses: a barrier of the even CTA, or a word of the peer
  auto lead = [](const void* p) { return mapa_shared(smem_u32(p), 0); };
  auto peer = [hr](const void* p) { return mapa_shared(smem_u32(p), (uint32_t)(hr ^ 1)); };
  // a wait that gave up stops the peer too
  auto stop_peer = [&]() { st_cluster_u32(peer(&sm.abort_flag), 1u); };
  PSegment seg;

  const int64_t img_seq_rows = ta.fimg_seq_bytes >> 7;
  // Programmatic dependent launch: every thread lets the absorption kernel
  // launch only after it has seen the preparation kernel complete, so that
  // the absorption's value loads ahead of its own grid-dependency wait find
  // the rows a decode step appends.
  griddep_wait();
  griddep_launch();

  if (warp == 0) {
    // ---- latent pieces (this CTA's 128 rows of each), issued as soon as their
    // slots are free.  No L2 prefetch runs ahead of them: two tiles ahead of every
    // CTA, it queued in HBM before the first tile's loads and cost 3 to 4 % of the
    // 32-head layer's steps ------------------------------------------------------
    if (has_work) {
      const uint64_t pol = policy_evict_first();
      const bool el = elect_one();
      int slot = 0, fills = 0;  // latent ring: next slot, times round
      bool ok = true;
      for (int ph = 0; ph < 2 && ok; ++ph)
        for (PairWalker walk = walker(ph); ok && walk.next(a, seg);) {
          for (int i = 0; i < seg.ntiles && ok; ++i) {
            const int64_t yrow = seg.row0 + seg.t0(i, hr);
            int ua, ub;
            units_of(ph, seg.X0 + i, ua, ub);
            for (int g = 0; g < lt.G && ok; ++g) {
              const GroupSm& gs = sm.grp[g];
              if (max(ua - gs.u0, 0) >= min(ub - gs.u0, (int)gs.nu)) continue;  // none of the group's units here
              for (int p = 0; p < gs.np; ++p) {
                if (fills && !(ok = wwait(&sm.a_empty[slot], (fills - 1) & 1, abort_flag))) break;
                if (el) {
                  const int w = gs.w[p];
                  if (leader) mbar_expect_tx(&sm.a_full[slot], 2 * kTile * 2 * w);
                  const CUtensorMap* m = w == 64 ? &maps.kc64 : (w == 32 ? &maps.kc32 : &maps.kc16);
                  tma_load_2d_pair(sm.a[slot], m, lead(&sm.a_full[slot]), gs.roff + gs.k[p], (int32_t)yrow, pol);
                }
                if (++slot == kNA) {
                  slot = 0;
                  ++fills;
                }
              }
            }
          }
        }
      if (!ok && lane == 0) stop_peer();
    }
  } else if (warp == 2) {
    // ---- factor items: this CTA's head of each (or its half of a lone head's),
    // one slot and one pair of barriers each, so that a unit's first MMAs start
    // when its first item is there and a slot refills as soon as it is read -----
    if (has_work) {
      const uint64_t pol = policy_evict_last();
      const bool el = elect_one();
      int slot = 0, fills = 0, pos = 0;  // factor ring: next slot, times round, items so far
      bool ok = true;
      for (int ph = 0; ph < 2 && ok; ++ph)
        for (PairWalker walk = walker(ph); ok && walk.next(a, seg);) {
          const int64_t img_row0 = kFold ? (int64_t)seg.b * img_seq_rows : 0;
          for (int i = 0; i < seg.ntiles && ok; ++i) {
            int ua, ub;
            units_of(ph, seg.X0 + i, ua, ub);
            const int n1 = ta.uitem[ub];
            for (int n = ta.uitem[ua]; n < n1; ++n) {
              if (fills && !(ok = wwait(&sm.w_empty[slot], (fills - 1) & 1, abort_flag))) break;
              if (el) {
                const uint32_t it = ta.item[n];
                const uint32_t hrows = ((it >> 26) << 12) / 256;
                uint64_t* full = &sm.w_full[pos % kItemBars];
                if (leader) mbar_expect_tx(full, (it >> 26) << 12);
                const int64_t y = img_row0 + ((it & 0x03FFFFFFu) >> 7) + hr * hrows;
                tma_load_2d_pair(sm.w[slot], &maps.im[im_map_of(hrows)], lead(full), 0, (int32_t)y, pol);
              }
              ++pos;
              if (++slot == NW) {
                slot = 0;
                ++fills;
              }
            }
          }
        }
      if (!ok && lane == 0) stop_peer();
    }
  } else if (warp == 1 || (kMma == 2 && warp == 3)) {
    // ---- MMA issuers (even CTA only): warp 1 (and warp 3 in query-folded mode)
    // runs the schedule of every kMma-th unit into its own accumulator, so one
    // warp's barrier waits and commits overlap the other's MMAs.  The whole warp
    // runs it and an elected lane issues (see elect_one), with descriptors as a
    // base per piece width plus a slot and a constant per k-step.  Per item: a
    // wait for it, its MMAs and the commit that frees its slot; per unit a wait
    // for the accumulator and its commit; per key group and warp a wait for each
    // latent piece and its release (commit, or arrivals in both CTAs when the warp
    // has no unit in the group, after the fill so that no barrier phase is passed
    // early). --------------------------------------------------------------------
    if (leader && has_work) {
      const bool el = elect_one();
      const int t = warp == 1 ? 0 : 1;
      const uint32_t sa0 = smem_u32(sm.a[0]), sw0 = smem_u32(sm.w[0]);
      const uint64_t da64 = sdesc(sa0, 16, 16 * 64, kSw128), dw64 = sdesc(sw0, 128 * 64, 1024, kSw128);
      const uint64_t da32 = sdesc(sa0, 16, 16 * 32, kSw64), dw32 = sdesc(sw0, 128 * 32, 1024, kSw128);
      const uint64_t da16 = sdesc(sa0, 16, 16 * 16, kSw32), dw16 = sdesc(sw0, 128 * 16, 1024, kSw128);
      int as = 0, aph = 0;  // latent ring: slot and phase of the next group's first piece
      int ws = 0, pos = 0;  // factor ring: slot and number of the next unit's first item
      int kc = 0, own = 0;  // units of the pair so far, units in this warp's accumulator
      bool ok = true;
      for (int ph = 0; ph < 2 && ok; ++ph)
        for (PairWalker walk = walker(ph); ok && walk.next(a, seg);) {
          for (int i = 0; i < seg.ntiles && ok; ++i) {
            int ua, ub;
            units_of(ph, seg.X0 + i, ua, ub);
            for (int g = 0; g < lt.G && ok; ++g) {
              const GroupSm& gs = sm.grp[g];
              const int np = gs.np;
              const int lo = max(ua - gs.u0, 0), hi = min(ub - gs.u0, (int)gs.nu);  // the group's units here
              if (lo >= hi) continue;
              const int uf = lo + (kMma == 2 ? (((kc & 1) == t) ? 0 : 1) : 0);  // this warp's first unit of the group
              if (uf >= hi) {  // no unit of this warp in the group: release its pieces in both CTAs
                for (int p = 0, sl = as, sp_ = aph; p < np; ++p) {
                  if (!(ok = wwait(&sm.a_full[sl], sp_, abort_flag))) break;
                  if (el) {
                    mbar_arrive(&sm.a_empty[sl]);
                    mbar_arrive_cluster(peer(&sm.a_empty[sl]));
                  }
                  if (++sl == kNA) {
                    sl = 0;
                    sp_ ^= 1;
                  }
                }
                if (!ok) break;
              }
              for (int u = lo; u < hi; ++u) {
                if (kMma == 2 && ((u - uf) & 1)) {  // the other warp's unit: skip its items
                  ws = ws + np >= NW ? ws + np - NW : ws + np;
                  pos += np;
                  continue;
                }
                const uint32_t idesc_k = 2 * u + 1 < gs.nh ? idesc_bf16(256, 2 * kD, false, true)
                                                           : idesc_bf16(256, kD, false, true);
                const int kg = kc + (u - lo);                 // unit index of the pair
                const int buf = kMma == 2 ? t : (kg & 1);
                const int use = kMma == 2 ? own : (kg >> 1);  // earlier units in this accumulator
                const uint32_t dcol = tmem + buf * kKCols;
                const bool first = u == uf, last = u + kMma >= hi;  // of this warp's units in the group
                for (int p = 0, sl = as, sp_ = aph; p < np; ++p) {
                  if (!(ok = wwait(&sm.w_full[pos % kItemBars], (pos / kItemBars) & 1, abort_flag))) break;
                  ++pos;
                  if (first && !(ok = wwait(&sm.a_full[sl], sp_, abort_flag))) break;
                  // both CTAs' epilogues have read this accumulator's previous unit
                  if (p == 0 && use >= 1 && !(ok = wwait(&sm.k_empty[buf], (use - 1) & 1, abort_flag))) break;
                  tc_fence_after();
                  const int w = gs.w[p];
                  const uint64_t ao = (uint64_t)(sl * (kSlot >> 4)), wo = (uint64_t)(ws * (kSlotW >> 4));
                  if (el) {
                    const uint32_t acc = p > 0 ? 1u : 0u;
                    if (w == 64) {
#pragma unroll
                      for (int k = 0; k < 4; ++k)
                        umma_f16_pair(dcol, da64 + ao + 2 * k, dw64 + wo + 128 * k, idesc_k, k ? 1u : acc);
                    } else if (w == 32) {
#pragma unroll
                      for (int k = 0; k < 2; ++k)
                        umma_f16_pair(dcol, da32 + ao + 2 * k, dw32 + wo + 128 * k, idesc_k, k ? 1u : acc);
                    } else {
                      umma_f16_pair(dcol, da16 + ao, dw16 + wo, idesc_k, acc);
                    }
                    umma_commit_pair(&sm.w_empty[ws]);
                    if (last) umma_commit_pair(&sm.a_empty[sl]);
                  }
                  ws = ws + 1 == NW ? 0 : ws + 1;
                  if (++sl == kNA) {
                    sl = 0;
                    sp_ ^= 1;
                  }
                }
                if (!ok) break;
                if (el) umma_commit_pair(&sm.k_full[buf]);
                ++own;
              }
              as += np;
              if (as >= kNA) {
                as -= kNA;
                aph ^= 1;
              }
              kc += hi - lo;
            }
          }
        }
      if (!ok && lane == 0) stop_peer();
    }
    __syncwarp();
  } else if (warp >= kCtlWarps) {
    // ---- epilogue: RoPE, scores, softmax, P of this CTA's 128-token halves ----
    const int e = tid - 32 * kCtlWarps;            // 0 .. 511
    const int quad = warp & 3;                     // TMEM lane quadrant
    const int fq = (warp - kCtlWarps) >> 2;        // frequency quarter: pairs [16 fq, 16 fq + 16)
    const int gid = lane >> 2, tig = lane & 3;     // key mode: rows and columns of the 16 x 256-bit fragments
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
    float* const xq = sm.x + fq * (kMaxHqTc * 128);  // this quarter's scores
    // tile and segment ends: thread e owns head jt and the 8 tokens [8 ct, 8 ct + 8)
    // of every half tile; the 16 owners of a head are adjacent lanes of one warp
    const int jt = e >> 4, ct = e & 15;
    int kc = 0, round = 0, tiles = 0;
    bool ok = true;
#define EPI_SYNC()                                  \
  do {                                              \
    __syncwarp();                                   \
    if (lane == 0) mbar_arrive(&sm.epi_bar);        \
    ok = wwait(&sm.epi_bar, round & 1, abort_flag); \
    ++round;                                        \
  } while (0)
    // an accumulator has been read by this warp: release it on the even CTA's barrier
    auto release_acc = [&](int buf) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (leader) mbar_arrive(&sm.k_empty[buf]);
        else mbar_arrive_cluster(lead(&sm.k_empty[buf]));
      }
    };
    for (int ph = 0; ph < 2 && ok; ++ph)
      for (PairWalker walk = walker(ph); ok && walk.next(a, seg);) {
        if (!kFold) {
          // rotated queries of this sequence at position L-1, scaled to log2 units
          // (its last tile's scores have been formed: that tile's EPI_SYNC)
          const float qscale = kLog2e * rsqrtf((float)kD);
          const __nv_bfloat16* qb = static_cast<const __nv_bfloat16*>(a.q) + (int64_t)seg.b * Hq * kD;
          const int pi = e & (kD / 2 - 1);
          float sn, cs;
          rope_sincos(sm.freq[pi], (uint32_t)(seg.L - 1), sn, cs);
          for (int j = e >> 6; j < Hq; j += kEpiThreads / (kD / 2)) {
            const float x1v = __bfloat162float(qb[j * kD + pi]), x2v = __bfloat162float(qb[j * kD + pi + kD / 2]);
            sm.qr[j * kD + pi] = __float2bfloat16_rn((x1v * cs - x2v * sn) * qscale);
            sm.qr[j * kD + pi + kD / 2] = __float2bfloat16_rn((x1v * sn + x2v * cs) * qscale);
          }
          EPI_SYNC();
          if (!ok) break;
        }
        // head jt's reference max (log2 units; the same in all 16 owners) and this
        // owner's share of its row sum, rescaled whenever the reference moves
        float m_run = -INFINITY, l_part = 0.f;
        int ua = 0, ub = 0;  // units of the current tile
        for (int i = 0; i < seg.ntiles && ok; ++i) {
          const int t0 = seg.t0(i, hr);
          const bool has = seg.has(i, hr);    // this half holds tokens of the sequence
          const int64_t x = seg.x128(i, hr);  // its flattened 128-token tile (when it has)
          units_of(ph, seg.X0 + i, ua, ub);
          // sines and cosines of this thread's accumulator elements: query-folded
          // mode, token `lane` of the quadrant at the quarter's 16 frequencies; key
          // mode, tokens gid + 8 k (k < 4) at frequencies 8 j + 2 tig + c (index 4 k + 2 j + c)
          float cs[kFreqW], sn[kFreqW];
#pragma unroll
          for (int ip = 0; ip < kFreqW; ++ip) {
            const int fi = kFreqW * fq + (kFold ? ip : 8 * ((ip >> 1) & 1) + 2 * tig + (ip & 1));
            const uint32_t pos = (uint32_t)(t0 + quad * 32 + (kFold ? lane : gid + 8 * (ip >> 2)));
            const uint2 f = sm.freq[fi];
            const float ang = (float)(int32_t)(__umulhi(pos, f.x) + pos * f.y) * kTurn32;
            __sincosf(ang, &sn[ip], &cs[ip]);
          }
          if (tiles >= 1 && !(ok = wwait(&sm.x_free, (tiles - 1) & 1, abort_flag))) break;  // the last tile's scores
          ++tiles;                                                                          // have been read
          // per unit (one or two KV heads), in MMA order: partial scores of this frequency quarter
          for (int u = ua; u < ub; ++u) {
            const uint32_t ui = sm.uinfo[u];
            const int h0 = ui & 0xFF, h1 = (ui >> 8) & 0xFF;
            const bool two = (ui >> 17) != 0;
            const int buf = kc & 1;
            if (!(ok = wwait(&sm.k_full[buf], (kc >> 1) & 1, abort_flag))) break;
            tc_fence_after();
            if (kFold) {
              // Y columns [32 fq, 32 fq + 32) of both heads: pairs (2i, 2i+1) of the 16 frequencies
              const uint32_t cb = tmem + lane_base + buf * kKCols + 2 * kFreqW * fq;
#pragma unroll
              for (int hh = 0; hh < 2; ++hh) {
                if (hh == 1 && !two) break;
                float y[32];
                tmem_ld32(cb + hh * kD, y);
                tmem_wait_ld();
                if (hh == 1 || !two) release_acc(buf);
                float pa[4] = {0.f, 0.f, 0.f, 0.f};  // independent chains
#pragma unroll
                for (int i2 = 0; i2 < kFreqW; ++i2)
                  pa[i2 & 3] = fmaf(cs[i2], y[2 * i2], fmaf(sn[i2], y[2 * i2 + 1], pa[i2 & 3]));
                xq[(hh ? h1 : h0) * 128 + quad * 32 + lane] = (pa[0] + pa[1]) + (pa[2] + pa[3]);
              }
            } else {
              // per head: the key's 16 frequency pairs of this quarter, read from TMEM
              // in the layout of the score MMA's A operand (m16n8k16: rows the warp's
              // 32 tokens in two m-tiles, k the 16 x-halves, then the 16 y-halves, n the
              // query heads padded to 8), rotated and rounded to bf16 in place
#pragma unroll
              for (int hh = 0; hh < 2; ++hh) {
                if (hh == 1 && !two) break;
                const int j0 = (hh ? h1 : h0) * qpg;
                const uint32_t cb = tmem + lane_base + buf * kKCols + hh * kD + kFreqW * fq;
                float xv[2][8], yv[2][8];
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                  tmem_ld_16x256b_x2(cb + ((uint32_t)(16 * mt) << 16), xv[mt]);
                  tmem_ld_16x256b_x2(cb + kD / 2 + ((uint32_t)(16 * mt) << 16), yv[mt]);
                }
                // B operand: query head n = gid (zero past qpg), k = 2 tig .. and 2 tig + 8 ..
                uint32_t bq[2][2] = {{0u, 0u}, {0u, 0u}};
                if (gid < qpg) {
                  const __nv_bfloat16* qrow = sm.qr + (j0 + gid) * kD + kFreqW * fq + 2 * tig;
#pragma unroll
                  for (int ks = 0; ks < 2; ++ks)
#pragma unroll
                    for (int j = 0; j < 2; ++j) bq[ks][j] = *reinterpret_cast<const uint32_t*>(qrow + 64 * ks + 8 * j);
                }
                tmem_wait_ld();
                if (hh == 1 || !two) release_acc(buf);
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                  uint32_t ax[4], ay[4];
#pragma unroll
                  for (int r = 0; r < 4; ++r) {  // rows gid + 8 (r & 1), frequencies 8 (r >> 1) + 2 tig, + 1
                    const int vi = 4 * (r >> 1) + 2 * (r & 1), ci = 4 * (2 * mt + (r & 1)) + 2 * (r >> 1);
                    const float x0 = xv[mt][vi], x1 = xv[mt][vi + 1], y0 = yv[mt][vi], y1 = yv[mt][vi + 1];
                    ax[r] = pack_bf16x2(fmaf(x0, cs[ci], -y0 * sn[ci]), fmaf(x1, cs[ci + 1], -y1 * sn[ci + 1]));
                    ay[r] = pack_bf16x2(fmaf(x0, sn[ci], y0 * cs[ci]), fmaf(x1, sn[ci + 1], y1 * cs[ci + 1]));
                  }
                  float acc[4] = {0.f, 0.f, 0.f, 0.f};
                  mma_bf16_16816(acc, ax, bq[0][0], bq[0][1]);
                  mma_bf16_16816(acc, ay, bq[1][0], bq[1][1]);
                  // scores: token (16 mt + gid [+ 8]) of this quadrant, query heads 2 tig, 2 tig + 1
#pragma unroll
                  for (int q = 0; q < 4; ++q) {
                    const int jj = 2 * tig + (q & 1), tt = quad * 32 + 16 * mt + gid + 8 * (q >> 1);
                    if (jj < qpg) xq[(j0 + jj) * 128 + tt] = acc[q];
                  }
                }
              }
            }
            ++kc;
          }
          if (!ok) break;
          // ---- tile end: reference max, P ------------------------------------
          EPI_SYNC();  // every partial score of the tile is in x
          if (!ok) break;
          {
            const bool own = jt < Hq && sm.hunit[jt] >= ua && sm.hunit[jt] < ub;  // head computed here
            const int tb = 8 * ct;  // first token of this owner
            float sc[8];
            const float4* xr = reinterpret_cast<const float4*>(&sm.x[jt * 128 + tb]);
#pragma unroll
            for (int q = 0; q < 2; ++q) {  // the sum of the four frequency quarters (every score is stored each tile)
              float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
              if (own) {
                const float4 w0 = xr[q], w1 = xr[kMaxHqTc * 32 + q], w2 = xr[2 * kMaxHqTc * 32 + q],
                             w3 = xr[3 * kMaxHqTc * 32 + q];
                v = make_float4((w0.x + w1.x) + (w2.x + w3.x), (w0.y + w1.y) + (w2.y + w3.y),
                                (w0.z + w1.z) + (w2.z + w3.z), (w0.w + w1.w) + (w2.w + w3.w));
              }
              sc[4 * q] = v.x;
              sc[4 * q + 1] = v.y;
              sc[4 * q + 2] = v.z;
              sc[4 * q + 3] = v.w;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.x_free);  // the next tile's scores may be stored
            const int nv = max(0, min(8, seg.L - (t0 + tb)));  // tokens inside the sequence
            float mx = -INFINITY;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              if (k >= nv || !own) sc[k] = -INFINITY;
              mx = fmaxf(mx, sc[k]);
            }
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            // the reference moves only when the tile's max exceeds it by the threshold
            if (own && (m_run == -INFINITY || mx > m_run + kRescaleThr)) {
              l_part *= exp2f(m_run - mx);
              m_run = mx;
            }
            if (has && own && ct == 0) ta.mglob[x * Hq + jt] = m_run;
            // probabilities (bf16, the absorption's operand) straight into this tile's
            // P image; the row sum uses the rounded values
            uint32_t pk[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const __nv_bfloat162 pv = __floats2bfloat162_rn(own ? ex2_approx(sc[2 * k] - m_run) : 0.f,
                                                              own ? ex2_approx(sc[2 * k + 1] - m_run) : 0.f);
              const float2 pf = __bfloat1622float2(pv);
              l_part += pf.x + pf.y;
              pk[k] = *reinterpret_cast<const uint32_t*>(&pv);
            }
            if (has && (own || (jt >= Hq && jt < hq_pad && ua == 0))) {  // padded heads get zero rows
              // image: [token atom (64)][head row][64 tokens], 128B rows, 16-byte chunks swizzled by row % 8
              uint8_t* img = ta.pglob + x * (hq_pad * 256) + (tb >> 6) * (hq_pad * 128) + (jt >> 3) * 1024 +
                             (jt & 7) * 128;
              *reinterpret_cast<uint4*>(img + (((ct & 7) ^ (jt & 7)) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
          }
        }
        if (!ok) break;
        // ---- segment end: reference max and row sum -> this half's partial slot ----
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) l_part += __shfl_xor_sync(0xffffffffu, l_part, o);
        if (jt < Hq && ct == 0 && sm.hunit[jt] >= ua && sm.hunit[jt] < ub) {
          const int64_t slot = ph ? pair_xslot(P, a.B, seg.X0 - sp.NPm, hr) : pair_slot(pair, seg.b, hr);
          a.part_ml[(slot * Hq + jt) * 2] = m_run;
          a.part_ml[(slot * Hq + jt) * 2 + 1] = l_part;
        }
      }
#undef EPI_SYNC
    if (!ok && lane == 0) stop_peer();
  }
  tc_fence_before();
  __syncthreads();
  if (sm.abort_flag) {
    drain_in_flight();
    if (tid == 0) atomicOr(a.err, kErrTimeout);
  }
  cluster_sync();  // the peer no longer reads this CTA's operands or arrives on its barriers
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, kTmemCols);
  }
}

// ---------------------------------------------------------------------------
// factor images
// ---------------------------------------------------------------------------

struct PrepItem {
  int32_t src;    // element of B_k at the item's first rank and head
  int32_t off;    // byte offset in a sequence's image
  int16_t ld;     // elements between ranks in B_k
  int8_t ws;      // ranks
  int8_t kv[2];   // KV head of each of the item's heads
};
// A warp's piece of the preparation: 8 ranks of one head (2 KB of image).
constexpr int kUnitBytes = 8 * kD * 2;
constexpr int kMaxPrepUnits = kMaxHqTc * 256 / 8;

// The decode step's latent append, done by the first blocks of the preparation
// launch: z_b = x_b [A_k | A_v] for the batch's new tokens, written to cache
// row rows[b] (Sec. III-A z = x L; Sec. III-C L_g side by side; Sec. III-D L_v).
struct StepAppend {
  const __nv_bfloat16* x;   // [B, D]
  const __nv_bfloat16* Ak;  // [D, Rk]
  const __nv_bfloat16* Av;  // [D, rv]
  const int64_t* rows;      // [B]
  int D;
  int n_blocks;             // GEMV blocks: one per 16 output columns
};

struct PrepArgs {
  int n_units;                  // pieces of one sequence's image
  int64_t seq_bytes;
  StepAppend app;
  RopeFreqs rf;
  PrepItem item[kMaxItems];
  uint8_t unit[kMaxPrepUnits];  // item of each piece
};

constexpr int kAppCols = 16;     // output columns of one GEMV block
constexpr int kAppMaxTok = 64;   // tokens of a fused append
constexpr int kAppWarps = 8;     // warps of a GEMV block, each a K range of D / 8

// Four 8x8 b16 matrices from shared memory, transposed.
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

// Four 8x8 b16 matrices from shared memory.
__device__ __forceinline__ void ldmatrix_x4_plain(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

constexpr int kAppStages = 6;    // k-steps of a warp in its ring, handled two at a time
// Dynamic shared memory of the append: per warp a ring of stages of a factor
// tile (512 B) and an x tile (16 tokens x 16 k per token m-tile); the warps'
// partial sums follow in the same place.  Every block of the launch carries it, and
// the factor pieces want three blocks per SM.
__host__ __device__ inline int app_stage_bytes(int batch) { return 512 + ((batch + 15) / 16) * 512; }
inline size_t app_smem_bytes(int batch) {
  return std::max((size_t)kAppWarps * kAppStages * app_stage_bytes(batch), (size_t)kAppWarps * batch * kAppCols * 4);
}

// One GEMV block: output columns [c0, c0 + 16) of [A_k | A_v] for B <= 64
// tokens.  Warp w accumulates K range [w D / 8, (w + 1) D / 8) with mma
// m16n8k16 (tokens x K) . (K x 16 columns).  Each k-step's factor tile
// [16 k][16 columns] and x tile [tokens][16 k] go through a per-warp ring of
// cp.async stages, kAppStages - 2 k-steps ahead, so the factor stream (read once)
// keeps enough bytes in flight; ldmatrix reads the operands (.trans for the
// column-major factor).  The eight warps' partial sums are added in shared
// memory, rounded to bf16 and written to the cache rows.
__device__ __forceinline__ void step_append_block(const LayerTable& lt, const DecodeArgs& a, const StepAppend& ap,
                                                  int blk) {
  extern __shared__ __align__(128) uint8_t app_dyn[];
  const int sb = app_stage_bytes(a.B);
  float* red = reinterpret_cast<float*>(app_dyn);  // [warp][B * 16], after the ring's last use
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gid = lane >> 2, tig = lane & 3;
  const int c0 = blk * kAppCols;
  const bool is_k = c0 < lt.Rk;
  const int N = is_k ? lt.Rk : lt.rv;
  const __nv_bfloat16* A = (is_k ? ap.Ak : ap.Av) + (is_k ? c0 : c0 - lt.Rk);
  const int B = a.B, D = ap.D;
  const int mt = (B + 15) / 16;  // token m-tiles
  const int kr = D / kAppWarps, kbeg = warp * kr, nks = kr / 16;
  float acc[kAppMaxTok / 16][2][4];
#pragma unroll
  for (int m = 0; m < kAppMaxTok / 16; ++m)
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[m][n][q] = 0.f;
  const uint32_t rbase = smem_u32(app_dyn + (size_t)warp * kAppStages * sb);
  // stage of a k-step: factor rows k (lane / 2), columns 8 (lane & 1) ..; x rows t,
  // 16-byte halves (two per row).  Rows past the batch are zeroed once.  The
  // pointers move along K, so a k-step is a copy or two and no address arithmetic
  // (formed anew, with the rows zeroed each time, it took 520 cycles: 9.5 us of a
  // step of one sequence on the 32-head layer, whose call this took from 40.3 to
  // 37.0 us, and 8 x 32768 on the 8-KV-head layer from 190 to 187).
  const int tr = lane >> 1, th = 8 * (lane & 1);
  const uint32_t so = (uint32_t)((tr * 16 + th) * 2);
  for (int sl = 0; sl < kAppStages; ++sl)
#pragma unroll
    for (int m = 0; m < kAppMaxTok / 16; ++m)
      if (m < mt && 16 * m + tr >= B)
        asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(rbase + (uint32_t)(sl * sb) + 512 + 512 * m + so),
                     "r"(0u)
                     : "memory");
  const __nv_bfloat16* pa = A + (int64_t)(kbeg + tr) * N + th;
  const __nv_bfloat16* px = ap.x + (int64_t)tr * D + kbeg + th;
  const int64_t astep = (int64_t)16 * N;
  int left = nks;  // k-steps not yet issued
  auto issue = [&](int slot) {
    if (left <= 0) return;
    --left;
    const uint32_t st = rbase + (uint32_t)(slot * sb) + so;
    cp_async16(st, pa);
#pragma unroll
    for (int m = 0; m < kAppMaxTok / 16; ++m)
      if (m < mt && 16 * m + tr < B) cp_async16(st + 512 + 512 * m, px + (int64_t)(16 * m) * D);
    pa += astep;
    px += 16;
  };
  constexpr int kPairs = kAppStages / 2;  // ring slots of two k-steps
#pragma unroll
  for (int q = 0; q < kPairs - 1; ++q) {
    issue(2 * q);
    issue(2 * q + 1);
    cp_async_commit();
  }
  int rd = 0, wr = kPairs - 1;  // slots read and refilled next
  const int m8 = lane >> 3, r8 = lane & 7;
  const uint32_t fo = (uint32_t)(((8 * (m8 & 1) + r8) * 16 + 8 * (m8 >> 1)) * 2);  // this lane's fragment row
  for (int kk = 0; kk < nks; kk += 2) {
    issue(2 * wr);
    issue(2 * wr + 1);
    cp_async_commit();
    wr = wr + 1 == kPairs ? 0 : wr + 1;
    cp_async_wait<kPairs - 1>();  // this slot has landed (this thread's copies)
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (kk + j >= nks) break;
      const uint32_t st = rbase + (uint32_t)((2 * rd + j) * sb) + fo;
      // B fragments: matrix m = lane / 8 covers k rows 8 (m & 1) .., n columns 8 (m >> 1) ..
      uint32_t bf[4];
      ldmatrix_x4_trans(bf, st);
#pragma unroll
      for (int m = 0; m < kAppMaxTok / 16; ++m) {
        if (m >= mt) break;
        // A fragments (tokens 16 m .., k 0..15): matrix q = lane / 8 covers rows 8 (q & 1) .., k 8 (q >> 1) ..
        uint32_t af[4];
        ldmatrix_x4_plain(af, st + 512 + 512 * m);
        mma_bf16_16816(acc[m][0], af, bf[0], bf[1]);
        mma_bf16_16816(acc[m][1], af, bf[2], bf[3]);
      }
    }
    rd = rd + 1 == kPairs ? 0 : rd + 1;
    __syncwarp();  // every lane is done with the slot before it is refilled
  }
  cp_async_wait<0>();
  __syncthreads();  // every warp is done with its ring
  // partial sums -> shared memory: token 16 m + gid (+8), column 8 n + 2 tig (+1)
#pragma unroll
  for (int m = 0; m < kAppMaxTok / 16; ++m)
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int t = 16 * m + gid + 8 * (q >> 1), c = 8 * n + 2 * tig + (q & 1);
        if (t < B) red[warp * B * kAppCols + t * kAppCols + c] = acc[m][n][q];
      }
  __syncthreads();
  __nv_bfloat16* cache = static_cast<__nv_bfloat16*>(const_cast<void*>(is_k ? a.kc : a.vc));
  for (int e = threadIdx.x; e < B * kAppCols; e += blockDim.x) {
    const int t = e / kAppCols, c = e % kAppCols;
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kAppWarps; ++w) v += red[w * B * kAppCols + e];
    const int64_t row = ap.rows[t];
    if (row < 0 || row >= a.n_rows) {
      if (c == 0) atomicOr(a.err, kErrBadRow);
      continue;
    }
    cache[row * N + (is_k ? c0 : c0 - lt.Rk) + c] = __float2bfloat16_rn(v);
  }
}

// Factor images: items of [nh heads][2 halves][ws rank rows][64 columns] bf16,
// 128B-swizzled (16-byte chunk c of row r stored at chunk c ^ (r % 8); every half
// starts on a 1024-byte swizzle atom).
// Key mode: columns of B_g[:, slot].  Query-folded mode: columns 2i and 2i+1 are
//   a_i B[:, i] + b_i B[:, i+64]  and  b_i B[:, i] - a_i B[:, i+64]
// with (a, b) the halves of RoPE(q_{b,h}, L_b - 1) * log2(e)/sqrt(d).
// The launch's first blocks do the fused append, if there is one (16 output
// columns each), the others write eight pieces each: 8 ranks of one head per
// warp, in query-folded mode for kPrepSeqs sequences.  A warp's loads (factors,
// queries) are all issued before the first is used, and a lane rotates the four
// frequency pairs that its columns need.  Bound by latency and the launch: with a
// whole item per block, fp64 angles and the loads in series it took 10.3 us for
// one sequence of the 32-head layer and 13 us for 16 (18 MB of images, written to
// L2).  Two sequences and three blocks per SM, so that 16 sequences' pieces start
// together with the append (four and two: 129.2 us for that step, now 128.3).
// Small blocks, not one per SM: SMs that have none left take the scores
// kernel's CTAs, whose set-up then overlaps (one 512-thread block per SM cost the
// step 4 to 10 us).
constexpr int kPrepSeqs = 2;
constexpr int kPrepThreads = 256;
template <bool kFold>
__global__ void __launch_bounds__(kPrepThreads, 3)
    factor_prep_kernel(const LayerTable lt, const DecodeArgs a, const __grid_constant__ PrepArgs pa,
                       uint8_t* __restrict__ img) {
  griddep_launch();
  if ((int)blockIdx.x < pa.app.n_blocks) {
    step_append_block(lt, a, pa.app, blockIdx.x);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int groups = kFold ? (a.B + kPrepSeqs - 1) / kPrepSeqs : 1;
  // lane: columns of pairs [4 ch, 4 ch + 4), i.e. 16-byte chunk c8 of a half, of ranks rl, rl + 2, ..
  const int ch = lane & 15, half = ch >> 3, c8 = ch & 7, rl = lane >> 4;
  const int w = (blockIdx.x - pa.app.n_blocks) * (kPrepThreads / 32) + warp;
  if (w < groups * pa.n_units) {
    const int u = w % pa.n_units, bs0 = w / pa.n_units * kPrepSeqs;
    const PrepItem it = pa.item[pa.unit[u]];
    const int ws = it.ws, r8 = (u * kUnitBytes - it.off) / kUnitBytes;  // eight-rank group of the item's heads
    const int hh = r8 / (ws / 8), r0 = r8 % (ws / 8) * 8;
    const __nv_bfloat16* __restrict__ Bs =
        static_cast<const __nv_bfloat16*>(a.Bk) + it.src + hh * kD + (int64_t)(r0 + rl) * it.ld;
    uint8_t* dst = img + it.off + (hh * 2 + half) * (ws * 128) + (r0 + rl) * 128;
    if (kFold) {
      // the x-halves B[:, i] and y-halves B[:, i+64] of four pairs in four ranks
      uint2 xr[4], yr[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        xr[k] = *reinterpret_cast<const uint2*>(Bs + (int64_t)(2 * k) * it.ld + 4 * ch);
        yr[k] = *reinterpret_cast<const uint2*>(Bs + (int64_t)(2 * k) * it.ld + kD / 2 + 4 * ch);
      }
      float q1[kPrepSeqs][4], q2[kPrepSeqs][4];
      int len[kPrepSeqs];
#pragma unroll
      for (int sb = 0; sb < kPrepSeqs; ++sb) {
        len[sb] = 0;  // no tile of an empty sequence is ever processed
        if (bs0 + sb >= a.B) continue;
        len[sb] = valid_len(a.seq_len, a.seq_start, bs0 + sb, a.n_rows);
        const __nv_bfloat16* q =
            static_cast<const __nv_bfloat16*>(a.q) + ((int64_t)(bs0 + sb) * lt.Hq + it.kv[hh]) * kD + 4 * ch;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          q1[sb][t] = __bfloat162float(q[t]);
          q2[sb][t] = __bfloat162float(q[kD / 2 + t]);
        }
      }
      const float sc = kLog2e * rsqrtf((float)kD);
#pragma unroll
      for (int sb = 0; sb < kPrepSeqs; ++sb) {
        if (len[sb] <= 0) continue;
        float qa[4], qb[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          float sn, cs;
          rope_sincos(pa.rf.f[4 * ch + t], (uint32_t)(len[sb] - 1), sn, cs);
          qa[t] = (q1[sb][t] * cs - q2[sb][t] * sn) * sc;
          qb[t] = (q1[sb][t] * sn + q2[sb][t] * cs) * sc;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 x01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&xr[k].x));
          const float2 x23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&xr[k].y));
          const float2 y01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&yr[k].x));
          const float2 y23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&yr[k].y));
          const uint4 out = make_uint4(
              pack_bf16x2(fmaf(qa[0], x01.x, qb[0] * y01.x), fmaf(qb[0], x01.x, -qa[0] * y01.x)),
              pack_bf16x2(fmaf(qa[1], x01.y, qb[1] * y01.y), fmaf(qb[1], x01.y, -qa[1] * y01.y)),
              pack_bf16x2(fmaf(qa[2], x23.x, qb[2] * y23.x), fmaf(qb[2], x23.x, -qa[2] * y23.x)),
              pack_bf16x2(fmaf(qa[3], x23.y, qb[3] * y23.y), fmaf(qb[3], x23.y, -qa[3] * y23.y)));
          *reinterpret_cast<uint4*>(dst + (int64_t)(bs0 + sb) * pa.seq_bytes + 256 * k +
                                    ((c8 ^ (rl + 2 * k)) << 4)) = out;  // rank row (rl + 2 k) mod 8 of its atom
        }
      }
    } else {
      uint4 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = *reinterpret_cast<const uint4*>(Bs + (int64_t)(2 * k) * it.ld + 8 * ch);
#pragma unroll
      for (int k = 0; k < 4; ++k) *reinterpret_cast<uint4*>(dst + 256 * k + ((c8 ^ (rl + 2 * k)) << 4)) = v[k];
    }
  }
}

// Split of a group rank into TMA/UMMA pieces of 64, 32 and 16 columns.
int make_pieces(int r, int8_t* w, int16_t* k) {
  int n = 0, off = 0;
  for (const int pw : {64, 32, 16})
    while (r - off >= pw) {
      if (n == kMaxPieces) return kMaxPieces + 1;
      w[n] = (int8_t)pw;
      k[n] = (int16_t)off;
      off += pw;
      ++n;
    }
  return off == r ? n : kMaxPieces + 1;
}

int hq_pad_of(int Hq) { return std::max(16, (Hq + 15) / 16 * 16); }

// Bytes of one copy of all factor images: sum over heads of r_g * 128 columns * 2.
size_t image_bytes_of(const LayerTable& lt) {
  size_t n = 0;
  for (int g = 0; g < lt.G; ++g) n += (size_t)lt.grp_nh[g] * lt.grp_rank[g] * 256;
  return n;
}

// Tensor maps depend only on the buffers and the layer: cache the last few.
struct MapsKey {
  const void* kc;
  int64_t n_rows;
  int Rk;
  const void* img;
  int64_t img_rows;
  bool operator==(const MapsKey& o) const {
    return kc == o.kc && n_rows == o.n_rows && Rk == o.Rk && img == o.img && img_rows == o.img_rows;
  }
};
constexpr int kMapsCache = 64;
std::mutex g_maps_mu;
MapsKey g_maps_key[kMapsCache];
Maps g_maps_val[kMapsCache];
int g_maps_n = 0, g_maps_next = 0;

bool build_maps(const LayerTable& lt, const DecodeArgs& a, const void* img, int64_t img_rows, Maps& maps) {
  std::memset(&maps, 0, sizeof(maps));
  const uint64_t rows = (uint64_t)std::max<int64_t>(1, a.n_rows);
  if (!(make_tmap_2d_bf16(&maps.kc64, a.kc, lt.Rk, rows, (uint64_t)lt.Rk * 2, 64, kTile, CU_TENSOR_MAP_SWIZZLE_128B) &&
        make_tmap_2d_bf16(&maps.kc32, a.kc, lt.Rk, rows, (uint64_t)lt.Rk * 2, 32, kTile, CU_TENSOR_MAP_SWIZZLE_64B) &&
        make_tmap_2d_bf16(&maps.kc16, a.kc, lt.Rk, rows, (uint64_t)lt.Rk * 2, 16, kTile, CU_TENSOR_MAP_SWIZZLE_32B)))
    return false;
  // the factor images as rows of 128 bytes (64 bf16), boxes of 16 .. 128 rows
  const uint32_t box_rows[4] = {16, 32, 64, 128};
  for (int i = 0; i < 4; ++i)
    if (!make_tmap_2d_bf16(&maps.im[i], img, 64, (uint64_t)std::max<int64_t>(img_rows, 128), 128, 64, box_rows[i],
                           CU_TENSOR_MAP_SWIZZLE_NONE))
      return false;
  return true;
}

static_assert(kMaxPieces <= Ring<true>::NW && Ring<true>::NW <= 5 && kMaxPieces <= 5, "see kItemBars");
static_assert(sizeof(Smem<true>) + 1024 + sizeof(PairScratch) <= 232448, "shared memory of the query-folded kernel");
static_assert(sizeof(Smem<false>) + 1024 + sizeof(PairScratch) <= 232448, "shared memory of the key-mode kernel");

template <bool kFold>
cudaError_t set_smem_attr() {
  static int attr_done[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  const bool dev_ok = dev >= 0 && dev < 64;
  if (dev_ok && attr_done[dev]) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(decode_tc_kernel<kFold>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(sizeof(Smem<kFold>) + 1024));
  if (e == cudaSuccess && dev_ok) attr_done[dev] = 1;
  return e;
}

// CTA pairs that can be resident at once (at most half the SMs): the scores
// kernel is persistent, so its grid is exactly that many pairs.
template <bool kFold>
int pairs_of_device() {
  static int pairs[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (pairs[dev]) return pairs[dev];
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (set_smem_attr<kFold>() != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (sms / 2));
  cfg.blockDim = dim3(kThreadsTc);
  cfg.dynamicSmemBytes = sizeof(Smem<kFold>) + 1024;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, decode_tc_kernel<kFold>, &cfg) != cudaSuccess || n <= 0) {
    cudaGetLastError();
    return 0;
  }
  pairs[dev] = std::min(n, sms / 2);
  return pairs[dev];
}

template <bool kFold>
cudaError_t launch_mode(const LayerTable& lt, const DecodeArgs& a, const Maps& maps, const TcArgs& ta,
                        const PrepArgs& pa, cudaStream_t s) {
  cudaError_t e = set_smem_attr<kFold>();
  if (e != cudaSuccess) return e;
  const size_t app_smem = pa.app.n_blocks ? app_smem_bytes(a.B) : 0;
  if (app_smem) {
    e = cudaFuncSetAttribute(factor_prep_kernel<kFold>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)app_smem);
    if (e != cudaSuccess) return e;
  }
  const int pieces = pa.n_units * (kFold ? (a.B + kPrepSeqs - 1) / kPrepSeqs : 1), per = kPrepThreads / 32;
  factor_prep_kernel<kFold><<<pa.app.n_blocks + (pieces + per - 1) / per, kPrepThreads, app_smem, s>>>(
      lt, a, pa, static_cast<uint8_t*>(a.extra));
  e = hook_launched(a.hook, s);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * ta.n_pairs);
  cfg.blockDim = dim3(kThreadsTc);
  cfg.dynamicSmemBytes = sizeof(Smem<kFold>) + 1024;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  e = cudaLaunchKernelEx(&cfg, decode_tc_kernel<kFold>, maps, lt, a, ta);
  return e != cudaSuccess ? e : hook_launched(a.hook, s);
}

// Order in which a tile's key groups are processed: the latent ring holds the
// pieces of the group in use while it fills with the next group's, so groups
// with many pieces are interleaved with groups with few (largest first, then
// smallest, ...), which keeps the piece counts of neighbours (cyclically: the
// last group is followed by the next tile's first) within the ring.
void group_order(const LayerTable& lt, int* order) {
  int idx[kMaxGroupsTc];
  int8_t w[kMaxPieces];
  int16_t k[kMaxPieces];
  int np[kMaxGroupsTc];
  for (int g = 0; g < lt.G; ++g) {
    idx[g] = g;
    np[g] = make_pieces(lt.grp_rank[g], w, k);
  }
  std::stable_sort(idx, idx + lt.G, [&](int x, int y) { return np[x] > np[y]; });
  for (int i = 0, lo = 0, hi = lt.G - 1; lo <= hi; ++i) order[i] = (i & 1) ? idx[hi--] : idx[lo++];
}

// Units, items and per-group tables of a layer (groups in processing order).
// Returns false when the layer does not fit the tables.
bool build_tables(const LayerTable& lt, TcArgs& ta, PrepArgs& pa) {
  std::memset(&ta, 0, sizeof(ta));
  std::memset(&pa, 0, sizeof(pa));
  ta.hq_pad = hq_pad_of(lt.Hq);
  if (lt.G > kMaxGroupsTc) return false;
  int gorder[kMaxGroupsTc];
  group_order(lt, gorder);
  int order[kMaxHqTc];  // KV head at each MMA position (group-major, slot order)
  int pos = 0, item = 0, off = 0, unit = 0;
  for (int gi = 0; gi < lt.G; ++gi) {
    const int g = gorder[gi];
    GroupSm& gs = ta.grp[gi];
    gs.roff = lt.grp_roff[g];
    int16_t kk[kMaxPieces];
    gs.np = (int8_t)make_pieces(lt.grp_rank[g], gs.w, kk);
    if (gs.np > kMaxPieces || gs.np > std::min(Ring<true>::NA, Ring<false>::NA)) return false;
    for (int p = 0; p < gs.np; ++p) gs.k[p] = kk[p];
    const int h0 = pos;  // MMA position of the group's first head
    gs.nh = (int8_t)lt.grp_nh[g];
    gs.nu = (int8_t)((lt.grp_nh[g] + 1) / 2);
    gs.u0 = (int16_t)unit;
    for (int sl = 0; sl < lt.grp_nh[g]; ++sl)
      for (int h = 0; h < lt.Hkv; ++h)
        if (lt.head_group[h] == g && lt.head_slot[h] == sl) {
          if (pos >= kMaxHqTc) return false;
          order[pos++] = h;
          for (int jj = 0; jj < lt.qpg; ++jj) ta.hunit[h * lt.qpg + jj] = (int8_t)(unit + sl / 2);
        }
    for (int s0 = 0; s0 < lt.grp_nh[g]; s0 += 2) {
      const int nh = std::min(2, lt.grp_nh[g] - s0);
      if (unit >= kMaxUnits) return false;
      ta.uitem[unit] = (int16_t)item;
      ta.uinfo[unit++] = (uint32_t)(order[h0 + s0] | (nh == 2 ? order[h0 + s0 + 1] << 8 : 0) | nh << 16);
      for (int p = 0; p < gs.np; ++p) {
        if (item >= kMaxItems) return false;
        const int w = gs.w[p], bytes = nh * w * 256;
        PrepItem& pi = pa.item[item];
        pi.src = (int32_t)(lt.grp_boff[g] + (int64_t)gs.k[p] * lt.grp_nh[g] * kD + s0 * kD);
        pi.ld = (int16_t)(lt.grp_nh[g] * kD);
        for (int hh = 0; hh < nh; ++hh)
          for (int h = 0; h < lt.Hkv; ++h)
            if (lt.head_group[h] == g && lt.head_slot[h] == s0 + hh) pi.kv[hh] = (int8_t)h;
        pi.ws = (int8_t)w;
        pi.off = off;
        if ((off + bytes) / kUnitBytes > kMaxPrepUnits) return false;
        for (int u = off / kUnitBytes; u < (off + bytes) / kUnitBytes; ++u) pa.unit[u] = (uint8_t)item;
        ta.item[item] = (uint32_t)off | ((uint32_t)(bytes >> 12) << 26);
        off += bytes;
        ++item;
      }
    }
  }
  ta.n_units = unit;
  ta.uitem[unit] = (int16_t)item;
  pa.n_units = off / kUnitBytes;
  pa.seq_bytes = off;
  ta.fimg_seq_bytes = off;
  return true;
}

// Workspace layout of the tensor-core path (after the split partials):
// factor images, then the per-tile P images, then the per-tile reference maxima.
struct ExtraLayout {
  size_t img, p, m, total;
};

ExtraLayout extra_layout(const LayerTable& lt, int batch, int64_t n_rows) {
  ExtraLayout x;
  const int64_t nt = max_tiles(n_rows, batch);
  x.img = align_up(lt.qpg == 1 ? image_bytes_of(lt) * std::max(batch, 1) : image_bytes_of(lt), 256);
  x.p = align_up((size_t)nt * hq_pad_of(lt.Hq) * 256, 256);
  x.m = align_up((size_t)nt * lt.Hq * sizeof(float), 256);
  x.total = x.img + x.p + x.m;
  return x;
}

}  // namespace

bool tc_decode_supports(const LayerTable& lt, int dtype) {
  if (dtype != DCK_BF16 || lt.d != kD) return false;
  if (lt.Hq > kMaxHqTc || lt.qpg > kMaxQPerKv || lt.G > kMaxGroupsTc) return false;
  if (lt.rv % 128 || (lt.rv / 128) * hq_pad_of(lt.Hq) > 512) return false;
  for (int g = 0; g < lt.G; ++g)
    if (lt.grp_rank[g] > 256 || lt.grp_rank[g] % 16) return false;
  static thread_local TcArgs ta;
  static thread_local PrepArgs pa;
  return build_tables(lt, ta, pa);
}

// Extra workspace of the tensor-core path.
size_t tc_decode_extra_ws(const LayerTable& lt, int batch, int64_t n_rows) {
  if (!tc_decode_supports(lt, DCK_BF16)) return 0;
  return extra_layout(lt, batch, n_rows).total;
}

// The fused decode-step append takes up to 64 tokens and widths D that split
// into eight warp ranges of 16-wide k-steps.
bool tc_step_append_supports(const LayerTable& lt, int D, int batch) {
  return batch >= 1 && batch <= kAppMaxTok && D % (kAppWarps * 16) == 0 && lt.Rk % kAppCols == 0 &&
         lt.rv % kAppCols == 0;
}

// CTA pairs of the tensor-core path on the current device (0 if it cannot run).
int tc_decode_pairs(const LayerTable& lt) { return lt.qpg == 1 ? pairs_of_device<true>() : pairs_of_device<false>(); }

cudaError_t launch_decode_tc(const LayerTable& lt, const DecodeArgs& a, const TcStepAppend* app, cudaStream_t s) {
  const bool fold = lt.qpg == 1;
  if (!a.extra || a.n_items < 2 || (a.n_items & 1)) return cudaErrorInvalidValue;
  static thread_local TcArgs ta;
  static thread_local PrepArgs pa;
  if (!build_tables(lt, ta, pa)) return cudaErrorInvalidValue;
  if (app) {
    if (!tc_step_append_supports(lt, app->D, a.B)) return cudaErrorInvalidValue;
    pa.app.x = static_cast<const __nv_bfloat16*>(app->x);
    pa.app.Ak = static_cast<const __nv_bfloat16*>(app->A_k);
    pa.app.Av = static_cast<const __nv_bfloat16*>(app->A_v);
    pa.app.rows = app->rows;
    pa.app.D = app->D;
    pa.app.n_blocks = (lt.Rk + lt.rv) / kAppCols;
  }
  ta.rf = pa.rf = rope_freqs_of(a.theta, kD);
  const ExtraLayout xl = extra_layout(lt, a.B, a.n_rows);
  uint8_t* base = static_cast<uint8_t*>(a.extra);
  ta.n_pairs = a.n_items / 2;
  ta.pglob = base + xl.img;
  ta.mglob = reinterpret_cast<float*>(base + xl.img + xl.p);
  ta.max_tiles = max_tiles(a.n_rows, a.B);
  const int64_t img_rows = (int64_t)(xl.img >> 7);
  const MapsKey key{a.kc, a.n_rows, lt.Rk, base, img_rows};
  Maps maps;
  bool have = false;
  {
    std::lock_guard<std::mutex> lk(g_maps_mu);
    for (int i = 0; i < g_maps_n && !have; ++i)
      if (g_maps_key[i] == key) {
        maps = g_maps_val[i];
        have = true;
      }
  }
  if (!have) {
    if (!build_maps(lt, a, base, img_rows, maps)) return cudaErrorInvalidValue;
    std::lock_guard<std::mutex> lk(g_maps_mu);
    g_maps_key[g_maps_next] = key;
    g_maps_val[g_maps_next] = maps;
    g_maps_next = (g_maps_next + 1) % kMapsCache;
    g_maps_n = std::min(g_maps_n + 1, kMapsCache);
  }
  cudaError_t e = hook_begin(a.hook, s);
  if (e != cudaSuccess) return e;
  e = fold ? launch_mode<true>(lt, a, maps, ta, pa, s) : launch_mode<false>(lt, a, maps, ta, pa, s);
  if (e != cudaSuccess) return e;
  TcRegions r;
  r.pglob = ta.pglob;
  r.mglob = ta.mglob;
  r.max_tiles = ta.max_tiles;
  r.hq_pad = ta.hq_pad;
  r.early_values = true;
  e = launch_absorb_tc(lt, a, r, s);
  return e != cudaSuccess ? e : hook_launched(a.hook, s);
}

}  // namespace dck
