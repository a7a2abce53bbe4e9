// Value absorption in latent space on the tensor cores (Sec. III-D: the value
// up-projection x W^(v) ~ z_v R_v is applied once, after the attention sum):
//   U_seg[:, j] = sum over the 128-token tiles of a segment of C_v[tile]^T P_tile[:, j]
// with P_tile the bf16 probabilities the scores kernel wrote (already the
// 128B-swizzled image of the UMMA B operand) and C_v[tile] the tile's value
// latents [128 tokens x r_v].  The segments and their partial slots are those
// of the scores kernel (the pair-tile plan of tc_common.cuh): CTA c = 2p + h
// absorbs half h of CTA pair p's main pair tiles, one segment per sequence,
// and a share of the extra 128-token tiles by r_v chunks, each a segment of
// its own; the scores kernel has already written each segment's reference max
// and row sum.
//
// The scores kernel's reference max of a head can rise from one tile to the
// next (it moves only when a tile's max exceeds it by 8); before such a tile
// the epilogue warps rescale U by exp2(m_old - m_new) in TMEM, after the MMAs
// of the earlier tiles have completed.  The MMA threads and the epilogue all
// read from the stored maxima which tiles need this and hand off only there
// (drain, which both MMA threads commit, then tile_ok, which both wait for), so
// each hand-off phase follows the MMA threads' own commits.  U = [r_v / 128 chunks][Hq_pad heads] fp32 accumulators, one TMEM
// lane per r_v row of a chunk.
//
// Warps: 0 producer (P images by bulk copy, value chunks by TMA), 1 and 6 MMA
// issuers (M = 128 r_v rows, N = Hq_pad, K = 16 tokens; 8 per chunk and tile), each
// taking half of a tile's r_v chunks from its own ring of value slots (a single
// warp's issue, commits and barrier tests took longer than the values took to
// arrive); warp 1 owns TMEM.  2-5 epilogue (one TMEM lane quadrant each: rescales
// and the U readout).  Where a sequence ends inside a tile, the issuing warp clears
// the chunk's rows past it: by one lane, as the issuing once was, that was up to
// 2032 stores a chunk (steps of the 32-head layer, one lane / the warp: 32 ragged
// sequences 271 / 250 us, 8 x 777 tokens 54 / 46, 1 x 777 37 / 33).
// Every wait is bounded; on expiry the CTA records kErrTimeout and releases
// TMEM after the work in flight has landed.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "tc_common.cuh"
#include "tc_host.h"
#include "tmap.h"

namespace dck {
namespace {

using namespace sm100;
using namespace tc;

constexpr int kAThreads = 224;
constexpr int kVSlot = 32768;  // one r_v chunk: [2 halves][128 tokens][64 rv] bf16, 128B-swizzled
constexpr int kNVr = 3;        // value slots of each MMA thread's ring: six chunks in flight
constexpr int kPSlot = 8192;   // P image of one tile (Hq_pad <= 32)
constexpr int kNP = 2;
constexpr int kEpiWarpsA = 4;  // warps 2-5: one per TMEM lane quadrant
constexpr uint32_t kTmemCols = 512;

struct AMaps {
  CUtensorMap vc;
};

struct AbsArgs {
  int hq_pad;
  int n_chunks;        // r_v / 128
  const uint8_t* pglob;
  const float* mglob;
  int64_t max_tiles;
  int early_values;  // value loads may start before the scores kernel completes
};

struct ASmem {
  uint8_t v[2 * kNVr][kVSlot];  // ring of MMA thread t: slots [t kNVr, (t + 1) kNVr)
  uint8_t p[kNP][kPSlot];
  uint64_t v_full[2 * kNVr], v_empty[2 * kNVr], p_full[kNP], p_empty[kNP];
  uint64_t drain, tile_ok, u_ready[2], u_free[2];
  int pneed[kNP];  // P slot's tile raises some head's reference max (set by the producer before the slot fills)
  PairScratch sc;
  uint32_t tmem_base;
  int abort_flag;
};

// This CTA's share of the scores kernel's plan (see tc_common.cuh).
struct AbsPlan {
  int P, pr, hh, NPm, nc, c_lo, c_hi;
};

// One absorption segment: n 128-token tiles of one sequence, two tiles apart
// in the flattened tile list (one half of consecutive pair tiles), r_v chunks
// [ca, cb) of each, accumulated into partial slot `slot`.
struct ASeg {
  int L, n, ca, cb, t00;
  int64_t slot, x0, row0;
  __device__ int64_t x(int i) const { return x0 + 2 * (int64_t)i; }
  __device__ int64_t row(int i) const { return row0 + (int64_t)kPTile * i; }
  __device__ int nvalid(int i) const { return min(kTile, L - (t00 + kPTile * i)); }
};

// Segments of this CTA in order: half hh of each main run (the tiles that
// exist: the odd half of a sequence's last pair tile may hold none), then each
// extra 128-token tile (e, half) with chunks in [c_lo, c_hi).
struct AWalk {
  PairWalker wm, wx;
  int ph = 0, hx = 2;
  PSegment sx;
  __device__ bool next(const DecodeArgs& a, const AbsPlan& pl, ASeg& s) {
    PSegment sg;
    while (ph == 0) {
      if (!wm.next(a, sg)) {
        ph = 1;
        break;
      }
      const int n = min(sg.ntiles, max(0, (sg.n128 - pl.hh - 2 * sg.i0 + 1) / 2));
      if (n == 0) continue;
      s.L = sg.L;
      s.n = n;
      s.ca = 0;
      s.cb = pl.nc;
      s.t00 = sg.t0(0, pl.hh);
      s.slot = pair_slot(pl.pr, sg.b, pl.hh);
      s.x0 = sg.x128(0, pl.hh);
      s.row0 = sg.row0 + s.t00;
      return true;
    }
    while (true) {
      if (hx == 2) {
        if (!wx.next(a, sx)) return false;
        hx = 0;
      }
      const int h2 = hx++;
      const int e = sx.X0 - pl.NPm, q = 2 * e + h2;
      const int ca = max(pl.c_lo - q * pl.nc, 0), cb = min(pl.c_hi - q * pl.nc, pl.nc);
      if (ca >= cb || !sx.has(0, h2)) continue;
      s.L = sx.L;
      s.n = 1;
      s.ca = ca;
      s.cb = cb;
      s.t00 = sx.t0(0, h2);
      s.slot = pair_xslot(pl.P, a.B, e, h2);
      s.x0 = sx.x128(0, h2);
      s.row0 = sx.row0 + s.t00;
      return true;
    }
  }
};

__global__ void __launch_bounds__(kAThreads, 1)
    absorb_tc_kernel(const __grid_constant__ AMaps maps, const LayerTable lt, const DecodeArgs a, const AbsArgs aa) {
  extern __shared__ uint8_t smem_raw[];
  ASmem& sm = *reinterpret_cast<ASmem*>(align_1024(smem_raw));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  volatile int* abort_flag = &sm.abort_flag;
  const int Hq = lt.Hq, hq_pad = aa.hq_pad, n_chunks = aa.n_chunks;
  const uint32_t pbytes = (uint32_t)hq_pad * 256;
  griddep_launch();  // the combine kernel may stage its factors as CTAs finish

  if (warp == 0) {  // a barrier per lane
    if (lane < 2 * kNVr) {
      mbar_init(&sm.v_full[lane], 1);
      mbar_init(&sm.v_empty[lane], 1);
    }
    if (lane < kNP) {
      mbar_init(&sm.p_full[lane], 1);
      mbar_init(&sm.p_empty[lane], 2);  // released by both MMA threads
    }
    if (lane < 2) {
      mbar_init(&sm.u_ready[lane], 2);
      mbar_init(&sm.u_free[lane], kEpiWarpsA);
    }
    if (lane == 0) {
      mbar_init(&sm.drain, 2);
      mbar_init(&sm.tile_ok, kEpiWarpsA);
      sm.abort_flag = 0;
      tma_prefetch_desc(&maps.vc);
    }
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  // the work plan of the scores kernel: half hh of pair pr's main pair tiles
  // [X0, X1), one segment per sequence; then chunks [c_lo, c_hi) of the
  // flattened (extra 128-token tile (e, half), r_v chunk) list
  AbsPlan pl;
  pl.P = a.n_items / 2;
  pl.pr = blockIdx.x >> 1;
  pl.hh = blockIdx.x & 1;
  pl.nc = n_chunks;
  const PairScan scan = pair_scan(a, sm.sc);
  const int NP = scan.total256;
  const PSplit sp(NP, pl.P, a.fine_below);
  pl.NPm = sp.NPm;
  const bool fits = scan.total128 <= aa.max_tiles;  // else the scores kernel has reported the input
  const int X0 = fits ? sp.main_begin(pl.pr, pl.P) : 0;
  const int X1 = fits ? sp.main_begin(pl.pr + 1, pl.P) : 0;
  const int xc = 2 * sp.R * n_chunks;
  pl.c_lo = fits ? (int)blockIdx.x * xc / a.n_items : 0;  // (fewer than P extra pair tiles)
  pl.c_hi = fits ? (int)(blockIdx.x + 1) * xc / a.n_items : 0;
  const int q0 = pl.c_lo < pl.c_hi ? pl.c_lo / n_chunks : 0;
  const int q1 = pl.c_lo < pl.c_hi ? (pl.c_hi - 1) / n_chunks + 1 : 0;
  const int xx0 = sp.NPm + q0 / 2, xx1 = q0 < q1 ? sp.NPm + (q1 - 1) / 2 + 1 : sp.NPm;
  pair_find(a, scan, X0, xx0, sm.sc);
  const bool has_work = X0 < X1 || pl.c_lo < pl.c_hi;
  // the two MMA threads split a tile's chunks [ca, cb) at cm: thread 0 [ca, cm), thread 1 [cm, cb)
  auto chunk_mid = [](int ca, int cb) { return ca + (cb - ca + 1) / 2; };
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  AWalk walk0;
  walk0.wm = pair_walker(sm.sc.at[0], X0, X1, false);
  walk0.wx = pair_walker(sm.sc.at[1], xx0, xx1, true);
  const uint32_t tmem = sm.tmem_base;
  // U is double-buffered in TMEM where two copies fit: segment s accumulates in
  // buffer s % nub while the epilogue reads out segment s - 1
  const uint32_t ucols = (uint32_t)(n_chunks * hq_pad);
  const int nub = 2 * ucols <= kTmemCols ? 2 : 1;
  ASeg seg;

  if (warp == 0) {
    // ---- producer ------------------------------------------------------------
    // The value latents do not depend on the scores kernel, which may still be
    // running (programmatic dependent launch): the first tile's first chunks
    // are loaded before the wait for that kernel's probabilities and maxima.
    if (has_work) {
      const uint64_t pol = policy_evict_first();
      int v_cnt[2] = {0, 0}, p_cnt = 0;
      bool ok = true, first = true;
      // reference maxima (lane = head) of the previous tile and, loaded a tile
      // ahead (across segments) so that their latency hides behind the value
      // loads, of this one
      float m_prev = 0.f, m_pf = 0.f;
      bool have_pf = false;
      // No L2 prefetch ahead of the loads: the rings keep 192 KB in flight per
      // SM, which is enough for HBM's rate, and prefetches of later tiles issued
      // by every CTA at once only queued ahead of the first tile's loads
      // (clock64 timelines: the first MMAs started 8 us later with them).
      for (AWalk walk = walk0; ok && walk.next(a, pl, seg);) {
        for (int i = 0; i < seg.n && ok; ++i) {
          const int64_t x = seg.x(i);
          const int64_t yrow = seg.row(i);
          const int ca = seg.ca, cb = seg.cb;
          // chunks go to the two MMA threads' rings alternately (thread 0: [ca, cm),
          // thread 1: [cm, cb)), each chunk one slot filled by two boxes (lanes 0, 1)
          const int cm = chunk_mid(ca, cb), nch = cb - ca;
          int done = 0;
          // the j-th chunk issued for this tile, and its ring
          auto chunk_at = [&](int j, int& c, int& r) {
            const int n0 = cm - ca, n1 = cb - cm, m = min(n0, n1);
            if (j < 2 * m) {
              r = j & 1;
              c = (r ? cm : ca) + (j >> 1);
            } else {
              r = n0 > n1 ? 0 : 1;
              c = (r ? cm : ca) + m + (j - 2 * m);
            }
          };
          auto issue_chunk = [&](int c, int r) {
            const int sl = r * kNVr + v_cnt[r] % kNVr;
            if (lane == 0) mbar_expect_tx(&sm.v_full[sl], kVSlot);
            __syncwarp();
            if (lane < 2)
              tma_load_2d_hint(sm.v[sl] + lane * (kVSlot / 2), &maps.vc, &sm.v_full[sl], 128 * c + 64 * lane,
                               (int32_t)yrow, pol);
            __syncwarp();
            ++v_cnt[r];
          };
          if (first) {  // the chunks that fit the empty rings, ahead of the wait
            for (; done < nch && aa.early_values; ++done) {
              int c, r;
              chunk_at(done, c, r);
              if (v_cnt[r] >= kNVr) break;
              issue_chunk(c, r);
            }
            griddep_wait();
            first = false;
          }
          if (!(ok = wait_slots(sm.p_empty, kNP, p_cnt, 1, lane, abort_flag))) break;
          {
            // the P image first: the decision below needs the maxima, a round trip later
            // (the barrier completes only with the arrival that follows it)
            const int sl = p_cnt % kNP;
            if (lane == 0) bulk_load(sm.p[sl], aa.pglob + x * pbytes, pbytes, &sm.p_full[sl], pol);
            // does any head's reference max rise at this tile?  (decided here, once,
            // for the MMA thread; the epilogue warps take the same decision)
            bool need = false;
            const float m_now = have_pf ? m_pf : (lane < Hq ? aa.mglob[x * Hq + lane] : 0.f);
            if (i > 0) need = __any_sync(0xffffffffu, m_now > m_prev);
            if (lane == 0) {
              sm.pneed[sl] = need ? 1 : 0;
              mbar_expect_tx(&sm.p_full[sl], pbytes);
            }
            have_pf = true;
            if (i + 1 < seg.n) {
              m_pf = lane < Hq ? aa.mglob[seg.x(i + 1) * Hq + lane] : 0.f;
            } else {  // the next segment's first tile
              AWalk nw = walk;
              ASeg ns;
              if (nw.next(a, pl, ns)) m_pf = lane < Hq ? aa.mglob[ns.x(0) * Hq + lane] : 0.f;
              else have_pf = false;
            }
            m_prev = m_now;
          }
          __syncwarp();
          ++p_cnt;
          for (; done < nch && ok; ++done) {
            int c, r;
            chunk_at(done, c, r);
            if (!(ok = wait_slots(sm.v_empty + r * kNVr, kNVr, v_cnt[r], 1, lane, abort_flag))) break;
            issue_chunk(c, r);
          }
        }
      }
    }
  } else if (warp == 1 || warp == 6) {
    // ---- MMA issuers: warp 1 takes chunks [ca, cm) of every tile, warp 6 chunks
    // [cm, cb), each from its own value ring; both wait for every P slot and every
    // hand-off with the epilogue, and both release.  The whole warp runs the schedule
    // and an elected lane issues, with descriptors as a base plus a slot and a
    // constant per k-step ------------------------------------------------------
    if (has_work) {
      const bool el = elect_one();
      const int t = warp == 1 ? 0 : 1;
      const uint32_t idesc_v = idesc_bf16(128, hq_pad, true, false);
      const uint64_t dv = sdesc(smem_u32(sm.v[0]), kVSlot / 2, 1024, kSw128);
      const uint64_t dp = sdesc(smem_u32(sm.p[0]), 16, 1024, kSw128);
      const uint64_t patom = (uint64_t)(hq_pad * 128 >> 4);  // 64 tokens of P
      int vs = 0, vph = 0, p_cnt = 0, rc = 0, sgc = 0;
      bool ok = true;
      for (AWalk walk = walk0; ok && walk.next(a, pl, seg);) {
        const uint32_t ubuf = tmem + (sgc % nub) * ucols;
        for (int i = 0; i < seg.n && ok; ++i) {
          const int psl = p_cnt % kNP;
          if (!(ok = wwait(&sm.p_full[psl], (p_cnt / kNP) & 1, abort_flag))) break;
          if (i > 0) {
            // some head's reference max rises at this tile: the epilogue rescales U
            // once the earlier tiles' MMAs are done (drain) and releases this tile
            // (tile_ok)
            if (sm.pneed[psl]) {
              if (el) umma_commit(&sm.drain);
              if (!(ok = wwait(&sm.tile_ok, rc & 1, abort_flag))) break;
              tc_fence_after();
              ++rc;
            }
          } else if (sgc >= nub) {  // the epilogue has read out this buffer's previous segment
            if (!(ok = wwait(&sm.u_free[sgc % nub], (sgc / nub - 1) & 1, abort_flag))) break;
            tc_fence_after();
          }
          const int nvalid = seg.nvalid(i);
          const uint64_t pd = dp + (uint64_t)(psl * (kPSlot >> 4));
          // chunks in pairs: the K = 16 MMAs of one chunk form a dependent chain on
          // its accumulator (about 120 cycles each at N = Hq_pad), so two chunks'
          // chains are interleaved
          const int ca = seg.ca, cb = seg.cb;
          const int cm = chunk_mid(ca, cb);
          const int c0 = t ? cm : ca, c1 = t ? cb : cm;
          for (int c = c0; c < c1 && ok; c += 2) {
            const int nc = min(2, c1 - c);
            int sl[2] = {0, 0};
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              if (q == nc) break;
              sl[q] = t * kNVr + vs;
              if (!(ok = wwait(&sm.v_full[sl[q]], vph, abort_flag))) break;
              if (++vs == kNVr) {
                vs = 0;
                vph ^= 1;
              }
              if (nvalid < kTile) {  // rows past the sequence end: exact zeros
                uint8_t* v = sm.v[sl[q]];
                for (int e = lane; e < (kTile - nvalid) * 16; e += 32)
                  *reinterpret_cast<uint4*>(v + ((e >> 3) & 1) * (kVSlot / 2) + (nvalid + (e >> 4)) * 128 +
                                            (e & 7) * 16) = make_uint4(0, 0, 0, 0);
                fence_proxy_async_smem();
                __syncwarp();
              }
            }
            if (!ok) break;
            tc_fence_after();
            if (el) {
              const uint64_t v0 = dv + (uint64_t)(sl[0] * (kVSlot >> 4)), v1 = dv + (uint64_t)(sl[1] * (kVSlot >> 4));
              const uint32_t u0 = ubuf + c * hq_pad, u1 = u0 + hq_pad;
              if (nc == 2) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                  const uint64_t bd = pd + (k >> 2) * patom + 2 * (k & 3);
                  const uint32_t acc = i == 0 && k == 0 ? 0u : 1u;
                  umma_f16(u0, v0 + 128 * k, bd, idesc_v, acc);
                  umma_f16(u1, v1 + 128 * k, bd, idesc_v, acc);
                }
                umma_commit(&sm.v_empty[sl[0]]);
                umma_commit(&sm.v_empty[sl[1]]);
              } else {
#pragma unroll
                for (int k = 0; k < 8; ++k)
                  umma_f16(u0, v0 + 128 * k, pd + (k >> 2) * patom + 2 * (k & 3), idesc_v, i == 0 && k == 0 ? 0u : 1u);
                umma_commit(&sm.v_empty[sl[0]]);
              }
            }
          }
          if (!ok) break;
          if (el) umma_commit(&sm.p_empty[psl]);
          ++p_cnt;
        }
        if (!ok) break;
        if (el) umma_commit(&sm.u_ready[sgc % nub]);
        ++sgc;
      }
    }
    __syncwarp();
  } else {
    // ---- epilogue (warps 2-5): rescales between tiles, U readout -------------
    const int quad = warp & 3;
    const int tau = quad * 32 + lane;  // r_v row inside a chunk
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
    int rc = 0, sgc = 0;
    bool ok = true;
    griddep_wait();  // the maxima come from the scores kernel
    for (AWalk walk = walk0; ok && walk.next(a, pl, seg);) {
      for (int i = 1; i < seg.n && ok; ++i) {
        // reference maxima of this tile and the segment's previous one, head = lane
        const float mn = lane < Hq ? aa.mglob[seg.x(i) * Hq + lane] : 0.f;
        const float mo = lane < Hq ? aa.mglob[seg.x(i - 1) * Hq + lane] : 0.f;
        if (__any_sync(0xffffffffu, mn > mo)) {
          if (!(ok = wwait(&sm.drain, rc & 1, abort_flag))) break;
          tc_fence_after();
          const float al = lane < Hq ? exp2f(mo - mn) : 1.f;  // this lane's head
          for (int c = 0; c < n_chunks; ++c)
            for (int cb = 0; cb < hq_pad / 16; ++cb) {
              float v[16];
              const uint32_t tad = tmem + (sgc % nub) * ucols + lane_base + c * hq_pad + 16 * cb;
              tmem_ld16(tad, v);
              tmem_wait_ld();
#pragma unroll
              for (int i2 = 0; i2 < 16; ++i2) v[i2] *= __shfl_sync(0xffffffffu, al, 16 * cb + i2);
              tmem_st16(tad, v);
            }
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sm.tile_ok);
          ++rc;
        }
      }
      if (!ok) break;
      // segment end: U -> the segment's partial slot
      if (!(ok = wwait(&sm.u_ready[sgc % nub], (sgc / nub) & 1, abort_flag))) break;
      tc_fence_after();
      float* dst = a.part_u + seg.slot * Hq * lt.rv + tau;
      const int ca = seg.ca, cb = seg.cb;
      for (int c = ca; c < cb; ++c) {
        float v0[16], v1[16];
        const uint32_t ub = tmem + (sgc % nub) * ucols + lane_base + c * hq_pad;
        tmem_ld16(ub, v0);
        if (hq_pad > 16) tmem_ld16(ub + 16, v1);
        tmem_wait_ld();
#pragma unroll
        for (int i2 = 0; i2 < 16; ++i2) {
          if (i2 < Hq) dst[(int64_t)i2 * lt.rv + c * 128] = v0[i2];
          if (16 + i2 < Hq) dst[(int64_t)(16 + i2) * lt.rv + c * 128] = v1[i2];
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.u_free[sgc % nub]);
      ++sgc;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (sm.abort_flag) {
    drain_in_flight();
    if (tid == 0) atomicOr(a.err, kErrTimeout);
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

struct VKey {
  const void* vc;
  int64_t n_rows;
  int rv;
  bool operator==(const VKey& o) const { return vc == o.vc && n_rows == o.n_rows && rv == o.rv; }
};
constexpr int kVMaps = 64;
std::mutex g_vmaps_mu;
VKey g_vkey[kVMaps];
AMaps g_vval[kVMaps];
int g_vn = 0, g_vnext = 0;

}  // namespace

cudaError_t launch_absorb_tc(const LayerTable& lt, const DecodeArgs& a, const TcRegions& r, cudaStream_t s) {
  if (r.hq_pad * 256 > kPSlot || (lt.rv / 128) * r.hq_pad > (int)kTmemCols) return cudaErrorInvalidValue;
  const VKey key{a.vc, a.n_rows, lt.rv};
  AMaps maps;
  bool have = false;
  {
    std::lock_guard<std::mutex> lk(g_vmaps_mu);
    for (int i = 0; i < g_vn && !have; ++i)
      if (g_vkey[i] == key) {
        maps = g_vval[i];
        have = true;
      }
  }
  if (!have) {
    std::memset(&maps, 0, sizeof(maps));
    const uint64_t rows = (uint64_t)std::max<int64_t>(1, a.n_rows);
    if (!make_tmap_2d_bf16(&maps.vc, a.vc, lt.rv, rows, (uint64_t)lt.rv * 2, 64, kTile, CU_TENSOR_MAP_SWIZZLE_128B))
      return cudaErrorInvalidValue;
    std::lock_guard<std::mutex> lk(g_vmaps_mu);
    g_vkey[g_vnext] = key;
    g_vval[g_vnext] = maps;
    g_vnext = (g_vnext + 1) % kVMaps;
    g_vn = std::min(g_vn + 1, kVMaps);
  }
  AbsArgs aa;
  aa.hq_pad = r.hq_pad;
  aa.n_chunks = lt.rv / 128;
  aa.pglob = r.pglob;
  aa.mglob = r.mglob;
  aa.max_tiles = r.max_tiles;
  aa.early_values = r.early_values ? 1 : 0;
  const size_t smem = sizeof(ASmem) + 1024;
  static int attr_done[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  const bool dev_ok = dev >= 0 && dev < 64;
  if (!dev_ok || !attr_done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(absorb_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev_ok) attr_done[dev] = 1;
  }
  // programmatic dependent launch: CTAs start streaming value latents as the
  // scores kernel's CTAs finish; the kernel waits for that grid before reading
  // its outputs
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.n_items);
  cfg.blockDim = dim3(kAThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, absorb_tc_kernel, maps, lt, a, aa);
}

}  // namespace dck
