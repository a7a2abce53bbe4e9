// Pieces shared by the tensor-core decode kernels (scores and absorption):
// bulk copies, bounded waits usable by one thread or a whole warp, ring-slot
// claims, the tile walk over sequence segments and the block-wide tile scan.
#pragma once

#include "common.cuh"
#include "sm100.cuh"

namespace dck {
namespace tc {

using namespace sm100;

__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Global -> shared bulk copy completing on `bar` (16-byte aligned, bytes % 16 == 0).
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
      : "memory");
}

// Bounded wait whose outcome is the same in every lane of the warp.
__device__ __forceinline__ bool wwait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  const bool r = mbar_wait(bar, parity, abort_flag);
  return __all_sync(0xffffffffu, r);
}

// Lane 0 waits for the `n` ring slots starting at ring position `cnt` (depth
// `depth`) to be released; the result is shared with the warp.
__device__ __forceinline__ bool wait_slots(uint64_t* empty, int depth, int cnt, int n, int lane,
                                           volatile int* abort_flag) {
  bool ok = true;
  if (lane == 0)
    for (int i = 0; i < n && ok; ++i) {
      const int c = cnt + i;
      if (c >= depth) ok = mbar_wait(&empty[c % depth], ((c / depth) - 1) & 1, abort_flag);
    }
  return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
}

// ---------------------------------------------------------------------------
// Work plan of the tensor-core decode path.
//
// The scores kernel runs as P CTA pairs (clusters of two CTAs, one tcgen05
// pair MMA of M = 256 tokens): every sequence is cut into pair tiles of 256
// tokens, whose first 128 tokens belong to the pair's even CTA (half 0) and
// the rest to its odd CTA (half 1).  The flattened pair-tile list (sequences in
// order) is split over the pairs: pair p takes the contiguous range
// [floor(p NPm / P), floor((p+1) NPm / P)) of the first NPm = main_tiles() tiles;
// the R = NP - NPm left over, where there are any, are shared out by units
// (groups of heads) instead, pair p taking units
// [floor(p R U / P), floor((p+1) R U / P)) of the flattened (extra tile, unit)
// list.  The absorption kernel's CTA c = 2p + h follows half h of pair p's
// tiles (its extra tiles it splits by r_v chunks instead).
//
// Softmax segments and their partial slots: half h of pair p over sequence b's
// tiles in p's main range writes slot 2 (p + b) + h; half h of extra tile e is
// a segment of its own, slot 2 (P + B - 1) + 2 e + h.  A slot is live when its
// half has at least one token (the odd half of a sequence's last pair tile can
// be empty); only live slots are read.
// ---------------------------------------------------------------------------

constexpr int kPTile = 256;  // tokens of a pair tile

__device__ __forceinline__ int n128_of(const DecodeArgs& a, int b) {
  return (valid_len(a.seq_len, a.seq_start, b, a.n_rows) + kTile - 1) / kTile;
}
__device__ __forceinline__ int n256_of(const DecodeArgs& a, int b) {
  return (valid_len(a.seq_len, a.seq_start, b, a.n_rows) + kPTile - 1) / kPTile;
}

__host__ __device__ inline int64_t pair_slot(int p, int b, int h) { return 2 * ((int64_t)p + b) + h; }
__host__ __device__ inline int64_t pair_xslot(int P, int B, int e, int h) {
  return 2 * ((int64_t)P + B - 1) + 2 * (int64_t)e + h;
}
// Partial slots of a call over caches of n_rows rows: main slots, then the
// extra tiles (fewer than P, and no more than the call's pair tiles,
// ceil(n_rows / 256) + B with non-overlapping sequences).
__host__ __device__ inline int64_t pair_slot_count(int P, int B, int64_t n_rows) {
  const int64_t tiles = (n_rows + kPTile - 1) / kPTile + B;
  const int64_t extra = P > 1 ? (P - 1 < tiles ? P - 1 : tiles) : 0;
  return 2 * ((int64_t)P + (B > 0 ? B - 1 : 0)) + 2 * extra;
}

// Split of NP pair tiles over P pairs (see above).
struct PSplit {
  int NP, NPm, R;
  __host__ __device__ PSplit(int np, int P, int fine_below)
      : NP(np), NPm(main_tiles(np, P, fine_below)), R(np - NPm) {}
  // floor(p NPm / P): the tiles of caches of fewer than 2^31 rows times the pairs of a GPU stay below 2^32
  __host__ __device__ int main_begin(int p, int P) const {
    return (int)((uint32_t)p * (uint32_t)NPm / (uint32_t)P);
  }
};

// A run of consecutive pair tiles of one sequence.
struct PSegment {
  int b, L;
  int i0;        // local index (within the sequence) of the run's first pair tile
  int ntiles;    // pair tiles in the run
  int X0;        // flattened index of the run's first pair tile
  int pre128;    // flattened index of the sequence's first 128-token tile
  int n128;      // 128-token tiles of the sequence
  int64_t row0;  // first cache row of the sequence
  // 128-token tile of local pair tile i0 + i, half h, and whether it exists
  __device__ int x128(int i, int h) const { return pre128 + 2 * (i0 + i) + h; }
  __device__ bool has(int i, int h) const { return 2 * (i0 + i) + h < n128; }
  __device__ int t0(int i, int h) const { return kPTile * (i0 + i) + kTile * h; }  // first token position
};

// Walks the sequences overlapping flattened pair tiles [X, X1) in order; with
// `single`, every pair tile is a run of its own.
struct PairWalker {
  int b, pre256, pre128, X, X1;
  bool single;
  __device__ bool next(const DecodeArgs& a, PSegment& sg) {
    while (X < X1 && b < a.B) {
      const int L = valid_len(a.seq_len, a.seq_start, b, a.n_rows);
      const int nt = (L + kPTile - 1) / kPTile;
      if (X >= pre256 + nt) {
        pre256 += nt;
        pre128 += (L + kTile - 1) / kTile;
        ++b;
        continue;
      }
      const int Xe = single ? X + 1 : min(X1, pre256 + nt);
      sg.b = b;
      sg.L = L;
      sg.i0 = X - pre256;
      sg.ntiles = Xe - X;
      sg.X0 = X;
      sg.pre128 = pre128;
      sg.n128 = (L + kTile - 1) / kTile;
      sg.row0 = a.seq_start[b];
      X = Xe;
      return true;
    }
    return false;
  }
};

// The batch's tile counts and where a thread's sequences lie in them: a block-wide
// scan (every thread of the block, of whole warps, takes part) whose results stay
// in registers.  Two barriers from the sequence lengths to the walkers: a CTA with
// one unit of work spends most of its time before its first load otherwise.
struct PairScan {
  int total256, total128;  // pair tiles and 128-token tiles of the batch
  int b0, per;             // this thread's sequences [b0, b0 + per)
  int r256, r128;          // tiles before them
  int n256, n128;          // tiles of them
};
struct PairFind {
  int b, p256, p128;  // sequence of a flattened pair tile, tiles before that sequence
};
struct PairScratch {
  int w256[32], w128[32];  // the warps' totals
  PairFind at[2];
};

// Block 0 of the grid reports sequences whose rows fall outside the cache.
__device__ __forceinline__ PairScan pair_scan(const DecodeArgs& a, PairScratch& sc) {
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  PairScan s;
  s.per = (a.B + nthr - 1) / nthr;
  s.b0 = tid * s.per;
  s.n256 = s.n128 = 0;
  for (int b = s.b0; b < s.b0 + s.per && b < a.B; ++b) {
    int64_t L = a.seq_len[b];
    const int64_t st = a.seq_start[b];
    if (L < 0 || st < 0 || st + L > a.n_rows) {
      if (blockIdx.x == 0) atomicOr(a.err, kErrBadSeq);
      L = 0;
    }
    s.n256 += (int)((L + kPTile - 1) / kPTile);
    s.n128 += (int)((L + kTile - 1) / kTile);
  }
  int i256 = s.n256, i128 = s.n128;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, i256, o), w = __shfl_up_sync(0xffffffffu, i128, o);
    if (lane >= o) {
      i256 += v;
      i128 += w;
    }
  }
  if (lane == 31) {
    sc.w256[warp] = i256;
    sc.w128[warp] = i128;
  }
  __syncthreads();
  int t256 = lane < (nthr >> 5) ? sc.w256[lane] : 0, t128 = lane < (nthr >> 5) ? sc.w128[lane] : 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, t256, o), w = __shfl_up_sync(0xffffffffu, t128, o);
    if (lane >= o) {
      t256 += v;
      t128 += w;
    }
  }
  s.total256 = __shfl_sync(0xffffffffu, t256, 31);
  s.total128 = __shfl_sync(0xffffffffu, t128, 31);
  const int b256 = __shfl_sync(0xffffffffu, t256, warp ? warp - 1 : 0);
  const int b128 = __shfl_sync(0xffffffffu, t128, warp ? warp - 1 : 0);
  s.r256 = i256 - s.n256 + (warp ? b256 : 0);
  s.r128 = i128 - s.n128 + (warp ? b128 : 0);
  return s;
}

// Looks up flattened pair tiles X0 and X1 (block-wide; a tile past the batch's
// last leaves its walker with nothing to walk, as its range is empty) and returns
// them in sc.at after a barrier that the caller passes next.
__device__ __forceinline__ void pair_find(const DecodeArgs& a, const PairScan& s, int X0, int X1, PairScratch& sc) {
  int r256 = s.r256, r128 = s.r128;
  for (int b = s.b0; b < s.b0 + s.per && b < a.B; ++b) {
    const int nt = s.per == 1 ? s.n256 : n256_of(a, b);
    if (X0 >= r256 && X0 < r256 + nt) sc.at[0] = PairFind{b, r256, r128};
    if (X1 >= r256 && X1 < r256 + nt) sc.at[1] = PairFind{b, r256, r128};
    r256 += nt;
    r128 += s.per == 1 ? s.n128 : n128_of(a, b);
  }
  if (threadIdx.x == 0) {
    if (X0 >= s.total256) sc.at[0] = PairFind{a.B, s.total256, s.total128};
    if (X1 >= s.total256) sc.at[1] = PairFind{a.B, s.total256, s.total128};
  }
}
__device__ __forceinline__ PairWalker pair_walker(const PairFind& f, int X, int X1, bool single) {
  return PairWalker{f.b, f.p256, f.p128, X, X1, single};
}

// Most 128-token tiles a call can have with non-overlapping sequences: the
// per-tile probability and reference-max stores of the tensor-core path are
// sized for this many.
__host__ __device__ inline int64_t max_tiles(int64_t n_rows, int batch) { return (n_rows + kTile - 1) / kTile + batch; }

}  // namespace tc
}  // namespace dck
