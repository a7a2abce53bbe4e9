// Prefill attention over DynaCalKV latent caches on the tensor cores (bf16).
//
// Prefill is decode with many queries per sequence: the Q_b new tokens of
// sequence b are the last Q_b rows of its cache and the i-th of them, at
// position p_i = L_b - Q_b + i, attends causally to the keys at positions
// 0 .. p_i.  Keys and values are rebuilt from the latents as in decode
// (Sec. III-A x W ~ z R; Sec. III-C one factorisation per head group;
// Sec. III-D one value factorisation for all heads), here once per cache row
// for all of a sequence's queries, as two dense GEMM chains:
//
//  1. recon_kernel: for every KV head h, K^_h = RoPE(C_g B_g[:, slot(h)]) at the
//     rows' positions and V^_h = C_v B_v[:, h d : (h+1) d] of every sequence's
//     rows (tcgen05 pair MMAs), written as bf16 to the workspace [n_rows][Hkv][d]
//     (keys) and [n_rows][Hkv][d] (values); the new tokens' queries, rotated
//     and scaled, go to `out`;
//  2. prefill_attn_kernel: causal flash attention over them, 128 query rows of
//     one KV head per tile (the qpg query heads of a KV head packed into the
//     rows: row r = query index r / qpg, head r % qpg), S = Q^ K^T and
//     O += P V^ on the tensor cores (M = 128 rows, N = 128, K = 128 / 128
//     keys), online softmax in log2 units with a lazy reference max (O in
//     TMEM is rescaled only when a tile's max exceeds it by 8).
//
// Every wait is bounded; on expiry the CTA records kErrTimeout, waits for
// work in flight and still releases TMEM.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "rope.cuh"
#include "tc_common.cuh"
#include "tmap.h"

namespace dck {

namespace {

using namespace sm100;
using namespace tc;

constexpr int kPD = 128;               // head dim of the tensor-core prefill
constexpr int kMaxGroupsP = 16;

// ---------------------------------------------------------------------------
// 1. reconstruction
//
// Keys and values of every sequence as dense GEMMs over its latent rows on
// persistent CTA pairs (tcgen05 pair MMAs, M = 256 rows): a tile is 256 rows of
// one sequence x the columns of one or two heads (w = 256 or 128), K = the
// group's rank or r_v in 64-wide stages, each CTA holding its 128 latent rows
// and half of the factor columns; two 256-column TMEM accumulators, so that the
// epilogue of one tile overlaps the next tile's MMAs.  Key tiles are rotated in
// the epilogue (a thread holds one row, both halves of every frequency pair).
// Pair p takes tiles p, p + P, ... of the list (values of every row tile, then
// keys: the costliest tiles first).  Six more warps of each CTA rotate and
// scale the queries into `out`, from where the attention kernel loads them by
// TMA before it overwrites them with the results: the tensor-bound GEMM hides
// that pass over q.
//
// One CTA per (row tile, head), as before, read a latent tile once per head and
// formed 64 sines and cosines per row and head (and the attention kernel 64 per
// query row).  Whole prefill calls, before and after: 32-head MHA prompt 2 x 4096
// 1193 -> 738 us, GQA prompt 8192 1228 -> 1041 us, four 300-512 token chunks in a
// pooled GQA cache 436 -> 268 us, eight MHA prompts of 44-214 tokens 139 -> 75 us.
// Then with deep loads for the queries, two epilogue warps per lane quadrant and
// MMAs issued by a uniform warp, the launches alone (cold): MHA prompt 101 + 40 ->
// 63 + 34 us, GQA prompt 81 + 21 -> 33 + 18 us.
//
// One launch for values and keys, whatever the size of the caller's cache: the row
// tiles are those of the sequences.  A launch for each, the second starting early,
// cost one set-up more and hid nothing: whole calls, us, two launches / one: one
// token 34 / 31, MHA prompt of 1000 57 / 52, eight GQA prompts of 512 74 / 69, MHA
// 2 x 4096 338 / 334, GQA 8192 451 / 442, 512 tokens after 32k 508 / 508 (GQA) and
// 706 / 705 (MHA); only past 64k tokens are they level or 0.8% apart the other way.
// ---------------------------------------------------------------------------

constexpr int kREpiWarps = 8;    // two per TMEM lane quadrant
constexpr int kRQWarps = 6;      // queries
constexpr int kRThreads = 32 * (2 + kREpiWarps + kRQWarps);  // warp 0 TMA, warp 1 MMA/TMEM, epilogue, queries
constexpr int kRStages = 6;
constexpr int kRBK = 64;
constexpr int kRABytes = kTile * kRBK * 2;   // 16 KB: this CTA's 128 latent rows x 64 of K
constexpr int kRBBytes = kRBK * 128 * 2;     // 16 KB: up to 128 factor columns x 64 of K (64-column boxes)
constexpr int kRStageBytes = kRABytes + kRBBytes;
constexpr int kRRows = 2 * kTile;            // rows of a pair tile
constexpr int kMaxColTiles = 160;            // key: <= 64 + 16, value: <= 64

struct RMaps {
  CUtensorMap ka[kMaxGroupsP];  // key latents of group g: [n_rows][r_g], box {64, 128 rows}, 128B swizzle
  CUtensorMap kb[kMaxGroupsP];  // B_g [r_g][n_g d]: box {64 columns, 64 ranks}, 128B swizzle
  CUtensorMap va, vb;           // value latents, B_v [r_v][Hkv d]
};

// Column tile of a row tile: factor columns [n0, n0 + w) of group g's B_g (g >= 0)
// or of B_v (g = -1), reduction length k, output heads h0 (and h1 when w = 256).
struct RCol {
  int16_t g, n0, w, h0, h1;
  int32_t k;
};

struct RArgs {
  const int64_t* seq_start;
  const int32_t* seq_len;
  const int32_t* q_len;
  int64_t n_rows;
  int B, Hq, Hkv, qmax, max_len;
  int n_val, n_key;               // value and key column tiles of a row tile
  RCol col[kMaxColTiles];         // value tiles, then key tiles
  RopeFreqs rf;
  float qscale;                   // log2(e) / sqrt(d)
  const __nv_bfloat16* q;
  __nv_bfloat16* qr;              // rotated, scaled queries (the out buffer)
  __nv_bfloat16* kw;              // [n_rows][Hkv][d]
  __nv_bfloat16* vw;              // [n_rows][Hkv][d]
  int* err;
};

// Cache rows of sequence b whose keys and values the attention kernel will read
// (0 for a sequence without new tokens or one that kernel rejects).
__device__ __forceinline__ int prefill_len(const int32_t* seq_len, const int64_t* seq_start, const int32_t* q_len,
                                           int b, int64_t n_rows, int qmax, int max_len) {
  const int L = valid_len(seq_len, seq_start, b, n_rows);
  const int Q = q_len[b];
  return Q <= 0 || Q > L || Q > qmax || L > max_len ? 0 : L;
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float2 unpack2(uint32_t v) {
  return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u));
}

__global__ void __launch_bounds__(kRThreads, 1)
    recon_kernel(const __grid_constant__ RMaps maps, const __grid_constant__ RArgs ra) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_1024(smem_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kRStages * kRStageBytes);
  uint64_t* empty = full + kRStages;
  uint64_t* acc_full = empty + kRStages;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* scan = reinterpret_cast<int*>(smem);            // [2][warps], before the first copy into the ring
  int* rpre = reinterpret_cast<int*>(tmem_slot + 2);   // [B + 1] row tiles before sequence b
  int* qpre = rpre + ra.B + 1;                         // [B + 1] queries before sequence b

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int hr = (int)cluster_ctarank();  // this CTA's half of every pair tile
  const bool leader = hr == 0;            // the even CTA issues the pair MMAs
  const int P = gridDim.x / 2, pair = blockIdx.x >> 1;
  if (tid == 0) {
    for (int s = 0; s < kRStages; ++s) {
      mbar_init(&full[s], 1);   // even CTA: its producer's expect_tx; both CTAs' copies complete on it
      mbar_init(&empty[s], 1);  // the pair MMAs' commit, in both CTAs
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 2 * kREpiWarps);  // even CTA: the epilogue warps of both CTAs
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  griddep_launch();
  if (warp == 1) {
    tmem_alloc_pair(tmem_slot, 512);
    tmem_relinquish_pair();
  }
  // exclusive prefixes of row tiles and of queries over the sequences
  {
    const int per = (ra.B + kRThreads - 1) / kRThreads, b0 = tid * per;
    int nr = 0, nq = 0;
    for (int b = b0; b < b0 + per && b < ra.B; ++b) {
      const int L = prefill_len(ra.seq_len, ra.seq_start, ra.q_len, b, ra.n_rows, ra.qmax, ra.max_len);
      nr += (L + kRRows - 1) / kRRows;
      nq += L ? ra.q_len[b] : 0;
    }
    int ir = nr, iq = nq;  // inclusive over the warp, then the totals of the warps before
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, ir, o), w = __shfl_up_sync(0xffffffffu, iq, o);
      if (lane >= o) {
        ir += v;
        iq += w;
      }
    }
    if (lane == 31) {
      scan[warp] = ir;
      scan[kRThreads / 32 + warp] = iq;
    }
    __syncthreads();
    int r = ir - nr, q = iq - nq, tr = 0, tq = 0;
    for (int w = 0; w < kRThreads / 32; ++w) {
      const int vr = scan[w], vq = scan[kRThreads / 32 + w];
      if (w < warp) {
        r += vr;
        q += vq;
      }
      tr += vr;
      tq += vq;
    }
    for (int b = b0; b < b0 + per && b < ra.B; ++b) {
      const int L = prefill_len(ra.seq_len, ra.seq_start, ra.q_len, b, ra.n_rows, ra.qmax, ra.max_len);
      rpre[b] = r;
      qpre[b] = q;
      r += (L + kRRows - 1) / kRRows;
      q += L ? ra.q_len[b] : 0;
    }
    if (tid == 0) {
      rpre[ra.B] = tr;
      qpre[ra.B] = tq;
    }
  }
  tc_fence_before();
  cluster_sync();  // both CTAs' barriers initialised and TMEM allocated (and the prefixes written)
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  auto lead = [](const void* q) { return mapa_shared(smem_u32(q), 0); };
  auto stop_peer = [&]() { st_cluster_u32(mapa_shared(smem_u32((const void*)abort_flag), (uint32_t)(hr ^ 1)), 1u); };

  const int64_t n_rt = rpre[ra.B];
  const int64_t n_vt = n_rt * ra.n_val, n_tiles = n_vt + n_rt * ra.n_key;
  // tile t: column tile, row tile of the flattened list
  auto tile_at = [&](int64_t t, int& rt) -> const RCol& {
    const bool v = t < n_vt;
    const int n = v ? ra.n_val : ra.n_key;
    const int64_t u = v ? t : t - n_vt;
    rt = (int)(u / n);
    return ra.col[(v ? 0 : ra.n_val) + (int)(u - (int64_t)rt * n)];
  };

  if (warp == 0) {
    // ---- TMA producer (both CTAs): this CTA's latent rows and its half of the factor columns
    const bool el = elect_one();
    const uint64_t pol = policy_evict_last();
    int st = 0, fills = 0;  // next stage, times round
    bool ok = true;
    for (int64_t t = pair; t < n_tiles && ok; t += P) {
      int rt;
      const RCol& c = tile_at(t, rt);
      const int b = seq_of_tile(rpre, ra.B, rt);
      const int32_t y = (int32_t)(ra.seq_start[b] + (int64_t)(rt - rpre[b]) * kRRows + hr * kTile);
      const CUtensorMap* am = c.g >= 0 ? &maps.ka[c.g] : &maps.va;
      const CUtensorMap* bm = c.g >= 0 ? &maps.kb[c.g] : &maps.vb;
      const int half = c.w / 2, ck = c.k, x0 = c.n0 + hr * half;
      for (int k0 = 0; k0 < ck; k0 += kRBK) {
        if (fills && !(ok = wwait(&empty[st], (uint32_t)((fills - 1) & 1), abort_flag))) break;
        if (el) {
          uint8_t* as = smem + st * kRStageBytes;
          uint8_t* bs = as + kRABytes;
          const uint32_t bar = lead(&full[st]);
          if (leader) mbar_expect_tx(&full[st], 2u * (uint32_t)(kRABytes + half * kRBK * 2));
          tma_load_2d_pair(as, am, bar, k0, y, pol);
          tma_load_2d_pair(bs, bm, bar, x0, k0, pol);
          if (half > 64) tma_load_2d_pair(bs + kRBK * 64 * 2, bm, bar, x0 + 64, k0, pol);
        }
        if (++st == kRStages) {
          st = 0;
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
      const uint64_t da = sdesc(s0, 16, 1024, kSw128), db = sdesc(s0 + kRABytes, kRBK * 64 * 2, 1024, kSw128);
      int st = 0;
      uint32_t sph = 0;
      bool ok = true;
      int lt = 0;  // tiles of this pair so far
      for (int64_t t = pair; t < n_tiles && ok; t += P, ++lt) {
        int rt;
        const RCol& c = tile_at(t, rt);
        const int buf = lt & 1, ck = c.k;
        if (lt >= 2 && !(ok = wwait(&acc_empty[buf], (uint32_t)(((lt >> 1) - 1) & 1), abort_flag))) break;
        const uint32_t idesc = c.w == 256 ? idesc_bf16(kRRows, 256, false, true) : idesc_bf16(kRRows, 128, false, true);
        const uint32_t d = tmem + buf * 256;
        for (int k0 = 0; k0 < ck; k0 += kRBK) {
          if (!(ok = wwait(&full[st], sph, abort_flag))) break;
          tc_fence_after();
          const uint64_t o = (uint64_t)(st * (kRStageBytes >> 4));
          if (el) {
#pragma unroll
            for (int k = 0; k < kRBK / 16; ++k)
              if (k0 + 16 * k < ck)
                umma_f16_pair(d, da + o + 2 * k, db + o + 128 * k, idesc, (k0 > 0 || k > 0) ? 1u : 0u);
            umma_commit_pair(&empty[st]);  // the stage's slots in both CTAs, once these MMAs are done
          }
          if (++st == kRStages) {
            st = 0;
            sph ^= 1;
          }
        }
        if (ok && el) umma_commit_pair(&acc_full[buf]);
      }
      if (!ok && lane == 0) stop_peer();
    }
    __syncwarp();
  } else if (warp < 2 + kREpiWarps) {
    // ---- epilogue (both CTAs): this CTA's 128 rows of each tile, half of the
    // frequency pairs per warp --------------------------------------------------
    const int quad = warp & 3, c_lo = (warp - 2) / 4 * (kPD / 4);
    const uint32_t lane_base = (uint32_t)(quad * 32) << 16;
    int lt = 0;
    bool ok = true;
    for (int64_t t = pair; t < n_tiles && ok; t += P, ++lt) {
      int rt;
      const RCol& c = tile_at(t, rt);
      const int b = seq_of_tile(rpre, ra.B, rt);
      const int pos = (rt - rpre[b]) * kRRows + hr * kTile + quad * 32 + lane;
      const bool in = pos < ra.seq_len[b];
      const int64_t row = ra.seq_start[b] + pos;
      const bool key = c.g >= 0;
      const int nh = c.w / kPD, buf = lt & 1;
      __nv_bfloat16* dst = (key ? ra.kw : ra.vw) + row * ra.Hkv * kPD;
      ok = wwait(&acc_full[buf], (uint32_t)((lt >> 1) & 1), abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t acc = tmem + lane_base + buf * 256;
      // frequency pairs (i, i + 64): columns [cc, cc + 16) with [64 + cc, 64 + cc + 16)
#pragma unroll 1
      for (int cc = c_lo; cc < c_lo + kPD / 4; cc += 16) {
        float sn[16], cs[16];
        if (key) {
#pragma unroll
          for (int i = 0; i < 16; ++i) rope_sincos(ra.rf.f[cc + i], (uint32_t)pos, sn[i], cs[i]);
        }
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          if (hh == nh) break;
          float x[16], y[16];
          tmem_ld16(acc + hh * kPD + cc, x);
          tmem_ld16(acc + hh * kPD + kPD / 2 + cc, y);
          tmem_wait_ld();
          if (key) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float xr = x[i] * cs[i] - y[i] * sn[i];
              y[i] = x[i] * sn[i] + y[i] * cs[i];
              x[i] = xr;
            }
          }
          if (in) {
            __nv_bfloat16* o = dst + (hh ? c.h1 : c.h0) * kPD + cc;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              reinterpret_cast<uint4*>(o)[q] =
                  make_uint4(pack2(x[8 * q], x[8 * q + 1]), pack2(x[8 * q + 2], x[8 * q + 3]),
                             pack2(x[8 * q + 4], x[8 * q + 5]), pack2(x[8 * q + 6], x[8 * q + 7]));
              reinterpret_cast<uint4*>(o + kPD / 2)[q] =
                  make_uint4(pack2(y[8 * q], y[8 * q + 1]), pack2(y[8 * q + 2], y[8 * q + 3]),
                             pack2(y[8 * q + 4], y[8 * q + 5]), pack2(y[8 * q + 6], y[8 * q + 7]));
            }
          }
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
  } else {
    // ---- queries: one warp per (sequence, new token); lane = (one of four heads
    // at a time, frequency pairs [8 c, 8 c + 8)).  Bound by the pass over q; the
    // loads of kQAhead rounds are issued before the first is used (with four
    // rounds on four warps the pass took longer than the products: 81 us of the
    // 8-KV-head prompt of 8192 for 134 MB) ---------------------------------------
    constexpr int kQAhead = 8;
    const int nw = kRQWarps * gridDim.x, nq = qpre[ra.B];
    const int c8 = lane & 7, hs = lane >> 3;
    for (int u = kRQWarps * blockIdx.x + warp - 2 - kREpiWarps; u < nq; u += nw) {
      const int b = seq_of_tile(qpre, ra.B, u), qi = u - qpre[b];
      const uint32_t pos = (uint32_t)(ra.seq_len[b] - ra.q_len[b] + qi);
      const int64_t off = ((int64_t)b * ra.qmax + qi) * ra.Hq * kPD + 8 * c8;
      float sn[8], cs[8];
      for (int h0 = hs; h0 < ra.Hq; h0 += 4 * kQAhead) {
        uint4 xv[kQAhead], yv[kQAhead];
#pragma unroll
        for (int r = 0; r < kQAhead; ++r)
          if (h0 + 4 * r < ra.Hq) {
            const __nv_bfloat16* src = ra.q + off + (h0 + 4 * r) * kPD;
            xv[r] = *reinterpret_cast<const uint4*>(src);
            yv[r] = *reinterpret_cast<const uint4*>(src + kPD / 2);
          }
        if (h0 == hs) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            rope_sincos(ra.rf.f[8 * c8 + i], pos, sn[i], cs[i]);
            sn[i] *= ra.qscale;
            cs[i] *= ra.qscale;
          }
        }
#pragma unroll
        for (int r = 0; r < kQAhead; ++r)
          if (h0 + 4 * r < ra.Hq) {
            const uint32_t xs[4] = {xv[r].x, xv[r].y, xv[r].z, xv[r].w}, ys[4] = {yv[r].x, yv[r].y, yv[r].z, yv[r].w};
            uint32_t xo[4], yo[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float2 x = unpack2(xs[i]), y = unpack2(ys[i]);
              xo[i] = pack2(x.x * cs[2 * i] - y.x * sn[2 * i], x.y * cs[2 * i + 1] - y.y * sn[2 * i + 1]);
              yo[i] = pack2(x.x * sn[2 * i] + y.x * cs[2 * i], x.y * sn[2 * i + 1] + y.y * cs[2 * i + 1]);
            }
            __nv_bfloat16* dst = ra.qr + off + (h0 + 4 * r) * kPD;
            *reinterpret_cast<uint4*>(dst) = make_uint4(xo[0], xo[1], xo[2], xo[3]);
            *reinterpret_cast<uint4*>(dst + kPD / 2) = make_uint4(yo[0], yo[1], yo[2], yo[3]);
          }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    drain_in_flight();
    if (tid == 0) atomicOr(ra.err, kErrTimeout);
  }
  cluster_sync();  // the peer no longer reads this CTA's operands or arrives on its barriers
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
}

size_t recon_smem(int B) {
  return 1024 + (size_t)kRStages * kRStageBytes + 256 + 2 * sizeof(int) * ((size_t)B + 1);
}

// CTA pairs of the reconstruction kernel that fit the device at once.
int recon_pairs_of_device() {
  static int cache[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  if (cache[dev]) return cache[dev];
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  const size_t smem = recon_smem(kMaxBatch);
  if (cudaFuncSetAttribute(recon_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (sms / 2));
  cfg.blockDim = dim3(kRThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, recon_kernel, &cfg) != cudaSuccess || n <= 0) {
    cudaGetLastError();
    return 0;
  }
  cache[dev] = std::min(n, sms / 2);
  return cache[dev];
}

cudaError_t launch_recon(const RMaps& rm, const RArgs& ra, int pairs, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(kRThreads);
  cfg.dynamicSmemBytes = recon_smem(ra.B);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, recon_kernel, rm, ra);
}

// ---------------------------------------------------------------------------
// 2. causal flash attention over the reconstructed keys and values
//
// Persistent CTAs, one per SM, over a list of items (ordered as PWalk says).  An item is
// two query tiles of 128 rows of one KV head (tile 1 the 128 / qpg positions
// after tile 0's; it may be missing), so that each K^ / V^ tile read from L2
// serves 256 rows (64 KB per 2048 cycles of MMA; a tile per CTA took 64 KB per
// 1024, the ~64 B/clk an SM takes in).  Per key tile the MMA warp issues
//   O0 += P0 V(j), S0 = Q0 K(j+1)^T, O1 += P1 V(j), S1 = Q1 K(j+1)^T
// so one tile's softmax runs under the other's MMAs.  P overwrites its scores in
// TMEM (the softmax has them in registers) and is the A operand of O += P V from
// there: shared memory holds two query tiles and five K^/V^ slots.  MMAs of one
// thread run in order, so S(j+1) may be issued right after the P V(j) that reads
// the same columns, and S(j+1) complete implies P V(j) complete (the softmax
// may then rescale O).  A softmax thread owns a row: no shuffles.  Four warps
// of their own write finished tiles out, while the next item's scores and
// probabilities are formed.
// TMEM: S0/P0 at column 0, S1/P1 at 128, O0 at 256, O1 at 384.
//
// A CTA per 128-row query tile, its softmax on four warps in series with its
// MMAs and P through shared memory, took 960 us on a 32-head MHA prompt of
// 2 x 4096 (275 GFLOP) and 1163 us on a GQA prompt of 8192 (550 GFLOP); this
// kernel 267 and 426 us (339 and 556 with its MMAs issued from a one-lane branch).
// ---------------------------------------------------------------------------

// warp 0 TMA, warp 1 MMA/TMEM, warp 2 schedule, warps 4-7 and 8-11 softmax of tile 0 and 1, warps 12-15 output
constexpr int kAThreadsP = 512;
constexpr int kAtom = 128 * 128;  // one 64-column swizzle atom of 128 rows (16 KB)
constexpr int kItems = 4;         // items in flight between the scheduler warp and the others
constexpr int kItemReaders = 14;  // producer, MMA warp, eight softmax warps, four output warps
constexpr int kKvSlots = 5;       // ring of K^ and V^ tiles (32 KB): K(0), V(0), K(1), V(1), ...
constexpr float kThr = 8.f;       // lazy reference max: probabilities stay <= 2^8
// registers: 512 threads x 128 at launch = 2 x 128 x 176 (softmax) + 2 x 128 x 80
constexpr int kRegsSoftmax = 176, kRegsOther = 80;

struct AMapsP {
  CUtensorMap kw, vw;  // [n_rows][Hkv d] bf16: box {64, 128 rows}, 128B swizzle
  CUtensorMap q;       // out as [B Qmax][Hq][d]: box {64, qpg, 128 / qpg}: 128 rows (position, head of the KV head)
};

struct AArgsP {
  const int32_t* q_len;    // [B]
  int qmax, max_len;
  const int64_t* seq_start;
  const int32_t* seq_len;
  int64_t n_rows;
  int B, Hq, Hkv, qpg;
  int ntp;                 // items (query tile pairs) of q_max queries
  int group;               // (sequence, KV head) streams whose items are interleaved
  __nv_bfloat16* out;      // [B, Qmax, Hq, d]: rotated queries in, results out
  int* err;
};

// One item: tiles 0 and 1 start at query indices i0 and i0 + 128 / qpg and
// attend to n[0] and n[1] key tiles (0: no such tile).
struct PItem {
  int b, h, i0, Q, L;
  int n[2];
  int bad;  // the sequence is rejected
  int64_t row0;
  __device__ int nk() const { return max(n[0], n[1]); }
};

struct ASmemP {
  uint8_t q[2][2][kAtom];          // Q^ [query tile][d atom][128 rows][128 B], K-major, 128B-swizzled
  uint8_t kv[kKvSlots][2][kAtom];  // K^ / V^ [slot][d atom][128 keys][128 B]
  float linv[2][128];              // [query tile][row] 1 / softmax denominator
  PItem item[kItems];              // items handed to the warps, in order; b < 0 ends the list
  uint64_t i_full[kItems], i_empty[kItems];
  uint64_t kv_full[kKvSlots], kv_empty[kKvSlots], q_full, q_empty;
  uint64_t s_full[2], p_full[2][2], l_full[2], o_full[2], o_free[2];  // [query tile] (P: [half of its keys])
  uint32_t tmem_base;
  int abort_flag;
};

// Walks the items of CTA blockIdx.x: rounds of gridDim.x items, every other one
// backwards.  The list takes `group` (sequence, KV head) streams at a time (their
// keys and values stay in L2 together), their last query tiles first: where the
// streams are alike, the ones that attend to the most keys.  Not so in a ragged
// batch: an index past a sequence's queries is dealt like any other and then passed
// over, and nothing weighs items by their keys (four chunks of 300 to 512 tokens on
// the 8-KV-head layer: 87 key tiles on the busiest CTA, 44 on average, 30 CTAs with
// none).
struct PWalk {
  int round = 0;
  __device__ bool next(const AArgsP& aa, PItem& it) {
    const int64_t streams = (int64_t)aa.B * aa.Hkv, total = streams * aa.ntp;
    const int G = gridDim.x, c = blockIdx.x;
    while (true) {
      const int64_t idx = (int64_t)round * G + ((round & 1) ? G - 1 - c : c);
      if (idx >= total) return false;
      ++round;
      const int64_t per = (int64_t)aa.group * aa.ntp;
      const int64_t g = idx / per, first = g * aa.group;
      const int gsz = (int)min((int64_t)aa.group, streams - first);
      const int64_t rem = idx - g * per;
      const int t = (int)(rem / gsz);
      const int64_t st = first + (rem - (int64_t)t * gsz);
      it.b = (int)(st / aa.Hkv);
      it.h = (int)(st - (int64_t)it.b * aa.Hkv);
      const int pp = 128 / aa.qpg;
      it.i0 = (aa.ntp - 1 - t) * 2 * pp;
      it.Q = aa.q_len[it.b];
      if (it.Q == 0) continue;  // no new tokens: nothing to write
      const int64_t L = aa.seq_len[it.b];
      it.row0 = aa.seq_start[it.b];
      it.L = (int)L;
      it.bad = it.Q < 0 || it.Q > L || it.Q > aa.qmax || L > aa.max_len || it.row0 < 0 || it.row0 + L > aa.n_rows;
      it.n[0] = it.n[1] = 0;
      if (it.bad) return true;
      if (it.i0 >= it.Q) continue;
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const int i = it.i0 + a * pp;
        if (i < it.Q) it.n[a] = (it.L - it.Q + min(it.Q, i + pp) - 1) / kTile + 1;
      }
      return true;
    }
  }
};

// A warp's copy of its CTA's item list (written by the scheduler warp).
struct PItems {
  int n = 0;
  __device__ bool next(ASmemP& sm, PItem& it, int lane, volatile int* abort_flag) {
    const int i = n % kItems;
    if (!wwait(&sm.i_full[i], (n / kItems) & 1, abort_flag)) return false;
    it = sm.item[i];
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm.i_empty[i]);
    ++n;
    return it.b >= 0;
  }
};

__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n add.rn.f32x2 z, x, y;\n"
      " mov.b64 {%0, %1}, z;\n}\n"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}

__global__ void __launch_bounds__(kAThreadsP, 1)
    prefill_attn_kernel(const __grid_constant__ AMapsP maps, const __grid_constant__ AArgsP aa) {
  extern __shared__ uint8_t smem_raw[];
  ASmemP& sm = *reinterpret_cast<ASmemP*>(align_1024(smem_raw));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  volatile int* abort_flag = &sm.abort_flag;
  const int qpg = aa.qpg, pp = 128 / qpg;
  if (tid == 0) {
    for (int i = 0; i < kKvSlots; ++i) {
      mbar_init(&sm.kv_full[i], 1);
      mbar_init(&sm.kv_empty[i], 1);
    }
    for (int i = 0; i < kItems; ++i) {
      mbar_init(&sm.i_full[i], 1);
      mbar_init(&sm.i_empty[i], kItemReaders);
    }
    mbar_init(&sm.q_full, 1);
    mbar_init(&sm.q_empty, 1);
    for (int a = 0; a < 2; ++a) {
      mbar_init(&sm.s_full[a], 1);
      mbar_init(&sm.p_full[a][0], 4);
      mbar_init(&sm.p_full[a][1], 4);
      mbar_init(&sm.l_full[a], 4);
      mbar_init(&sm.o_full[a], 1);
      mbar_init(&sm.o_free[a], 4);
    }
    sm.abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  griddep_wait();  // rotated queries, keys and values come from the launches before
  const uint32_t tmem = sm.tmem_base;
  PItems list;
  PItem it;

  if (warp < 4) {
    reg_dec<kRegsOther>();
    if (warp == 0) {
      const uint64_t pol = policy_evict_last();  // a K^ / V^ tile is read by several items
      int slot = 0;
      uint32_t sphase = 1, items = 0;  // a fresh barrier passes a wait for the phase before its first
      bool ok = true;
      while (ok && list.next(sm, it, lane, abort_flag)) {
        const int nk = it.nk();
        if (nk == 0) continue;
        auto load_kv = [&](const CUtensorMap* m, int kt) -> bool {
          if (!wwait(&sm.kv_empty[slot], sphase, abort_flag)) return false;
          if (lane == 0) mbar_expect_tx(&sm.kv_full[slot], 2 * kAtom);
          __syncwarp();
          const int32_t y = (int32_t)(it.row0 + (int64_t)kTile * kt);
          if (lane < 2) tma_load_2d_hint(sm.kv[slot][lane], m, &sm.kv_full[slot], it.h * kPD + 64 * lane, y, pol);
          if (++slot == kKvSlots) {
            slot = 0;
            sphase ^= 1;
          }
          return true;
        };
        if (!(ok = load_kv(&maps.kw, 0))) break;
        // the previous item's scores are all formed: its queries can go
        if (items >= 1 && !(ok = wwait(&sm.q_empty, (items - 1) & 1, abort_flag))) break;
        const int nq = it.n[1] ? 4 : 2;
        if (lane == 0) mbar_expect_tx(&sm.q_full, nq * kAtom);
        __syncwarp();
        if (lane < nq)
          tma_load_3d(sm.q[lane >> 1][lane & 1], &maps.q, &sm.q_full, 64 * (lane & 1), it.h * qpg,
                      it.b * aa.qmax + it.i0 + (lane >> 1) * pp);
        ++items;
        for (int kt = 0; kt < nk && ok; ++kt) {
          if (kt > 0) ok = load_kv(&maps.kw, kt);
          ok = ok && load_kv(&maps.vw, kt);
        }
      }
    } else if (warp == 1) {
      // ---- MMAs: the whole warp runs the schedule and one elected lane issues (see
      // elect_one).  One warp for both query tiles: with a warp for each, their MMAs
      // interleaved one by one, both tiles' scores were ready at the same time and
      // the tensor pipe idled under both softmaxes (GQA prompt 8192: 490 us against
      // 426). ----------------------------------------------------------------------
      const bool el = elect_one();
      const uint32_t id_s = idesc_bf16(128, 128, false, false);  // S = Q K^T: both K-major
      const uint32_t id_o = idesc_bf16(128, 128, false, true);   // O += P V: V MN-major
      const uint64_t dq = sdesc(smem_u32(sm.q[0][0]), 16, 1024, kSw128);
      const uint64_t dk = sdesc(smem_u32(sm.kv[0][0]), 16, 1024, kSw128);
      const uint64_t dv = sdesc(smem_u32(sm.kv[0][0]), kAtom, 1024, kSw128);
      int slot = 0;  // ring slot of the next K^/V^ tile and its phase
      uint32_t sphase = 0, items = 0;
      uint32_t pph[2] = {0, 0};  // P tiles so far
      uint32_t oph[2] = {0, 0};  // finished output tiles so far
      bool ok = true;
      // waits for the ring's next tile; its slot
      auto kv_next = [&](int& sl) {
        sl = slot;
        const bool r = wwait(&sm.kv_full[slot], sphase, abort_flag);
        if (++slot == kKvSlots) {
          slot = 0;
          sphase ^= 1;
        }
        return r;
      };
      while (ok && list.next(sm, it, lane, abort_flag)) {
        const int nk = it.nk();
        if (nk == 0) continue;
        const int n0 = it.n[0], n1 = it.n[1];
        // S_a = Q_a K^T
        auto scores = [&](int a, int sl) {
          const uint64_t qb = dq + (uint64_t)(a * (2 * kAtom >> 4)), kb = dk + (uint64_t)(sl * (2 * kAtom >> 4));
          if (el) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const uint64_t o = ((k >> 2) * kAtom + (k & 3) * 32) >> 4;
              umma_f16(tmem + 128 * a, qb + o, kb + o, id_s, k > 0 ? 1u : 0u);
            }
            umma_commit(&sm.s_full[a]);
          }
        };
        int ks, vs, kn = 0;
        if (!(ok = wwait(&sm.q_full, items & 1, abort_flag))) break;
        ++items;
        if (!(ok = kv_next(ks))) break;
        tc_fence_after();
        if (n0) scores(0, ks);
        if (n1) scores(1, ks);
        if (el) {
          umma_commit(&sm.kv_empty[ks]);
          if (nk == 1) umma_commit(&sm.q_empty);
        }
        for (int kt = 0; kt < nk && ok; ++kt) {
          const bool more = kt + 1 < nk;
          bool have_k = false;
          if (!(ok = kv_next(vs))) break;
          const uint64_t vb = dv + (uint64_t)(vs * (2 * kAtom >> 4));
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            const int n = a ? n1 : n0;
            if (kt < n) {
              if (kt == 0 && oph[a] >= 1 && !(ok = wwait(&sm.o_free[a], (oph[a] - 1) & 1, abort_flag))) break;
#pragma unroll
              for (int hf = 0; hf < 2; ++hf) {
                if (!(ok = wwait(&sm.p_full[a][hf], pph[a] & 1, abort_flag))) break;
                tc_fence_after();
                if (el) {
#pragma unroll
                  for (int k = 4 * hf; k < 4 * hf + 4; ++k)
                    umma_f16_ts(tmem + 256 + 128 * a, tmem + 128 * a + 8 * k, vb + (uint64_t)(k * 2048 >> 4), id_o,
                                (kt > 0 || k > 0) ? 1u : 0u);
                }
              }
              if (!ok) break;
              ++pph[a];
              if (kt + 1 == n) {
                if (el) umma_commit(&sm.o_full[a]);
                ++oph[a];
              }
            }
            if (kt + 1 < n) {
              if (!have_k && !(ok = kv_next(kn))) break;
              have_k = true;
              tc_fence_after();
              scores(a, kn);
            }
          }
          if (!ok) break;
          if (el) {
            umma_commit(&sm.kv_empty[vs]);
            if (more) umma_commit(&sm.kv_empty[kn]);
            if (kt + 2 == nk) umma_commit(&sm.q_empty);  // every score of the item has been issued
          }
        }
      }
    } else if (warp == 2) {
      // ---- schedule: the item list, a few items ahead ---------------------------
      PWalk walk;
      bool more = true;
      for (int n = 0; more; ++n) {
        const int i = n % kItems;
        if (n >= kItems && !wwait(&sm.i_empty[i], ((n / kItems) - 1) & 1, abort_flag)) break;
        more = walk.next(aa, it);
        if (!more) it.b = -1;
        if (lane == 0) {
          sm.item[i] = it;
          mbar_arrive(&sm.i_full[i]);
        }
      }
    }
  } else if (warp < 12) {
    // ---- softmax of query tile a: thread = row r ---------------------------------
    reg_inc<kRegsSoftmax>();
    const int a = (warp - 4) >> 2, quad = warp & 3, r = quad * 32 + lane;
    const uint32_t lb = (uint32_t)(quad * 32) << 16;
    const uint32_t sb = tmem + lb + 128 * a, ob = tmem + lb + 256 + 128 * a;
    int base = 0;
    uint32_t sph = 0, oph = 0;
    bool ok = true;
    while (ok && list.next(sm, it, lane, abort_flag)) {
      const int nk = it.nk(), n = it.n[a];
      if (n == 0) {
        base += 2 * nk;
        continue;
      }
      const int qi = it.i0 + a * pp + r / qpg;
      const bool valid = qi < it.Q;
      const int pos = it.L - it.Q + qi;
      float m = -INFINITY;
      float2 l = make_float2(0.f, 0.f);
      for (int kt = 0; kt < n; ++kt) {
        if (!(ok = wwait(&sm.s_full[a], sph & 1, abort_flag))) break;
        ++sph;
        tc_fence_after();
        float sv[128];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(sb + 32 * c, *reinterpret_cast<float(*)[32]>(&sv[32 * c]));
        tmem_wait_ld();
        const int kbase = kTile * kt;
        const int vis = valid ? pos - kbase + 1 : 0;  // visible keys of this tile: [0, vis)
        if (!__all_sync(0xffffffffu, vis >= kTile)) {
#pragma unroll
          for (int i = 0; i < 128; ++i) sv[i] = i < vis ? sv[i] : -INFINITY;
        }
        float mx[4] = {sv[0], sv[1], sv[2], sv[3]};
#pragma unroll
        for (int i = 4; i < 128; i += 8)
#pragma unroll
          for (int u = 0; u < 4; ++u) mx[u] = fmaxf(mx[u], i + 4 + u < 128 ? fmaxf(sv[i + u], sv[i + 4 + u]) : sv[i + u]);
        const float mt = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
        // a new reference max for this row when the tile's max passes the old one by
        // kThr; O and l are rescaled where a reference existed.  The TMEM loads and
        // stores are warp-collective, so the whole warp runs them when any row
        // rescales (factor 1 for the other rows).
        const bool upd = mt != -INFINITY && (m == -INFINITY || mt > m + kThr);
        const bool resc = upd && m != -INFINITY;
        if (__any_sync(0xffffffffu, resc)) {
          const float al = resc ? exp2f(m - mt) : 1.f;
#pragma unroll 1
          for (int c = 0; c < 8; ++c) {
            float v[16];
            tmem_ld16(ob + 16 * c, v);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] *= al;
            tmem_st16(ob + 16 * c, v);
          }
          l.x *= al;
          l.y *= al;
        }
        if (upd) m = mt;
        // keys past the sequence in its last tile: exact zeros in V^ (P is zero there),
        // written once by the first query tile that uses them
        if (kbase + kTile > it.L && a == (kt < it.n[0] ? 0 : 1)) {
          const int c = base + 2 * kt + 1;
          if (!(ok = wwait(&sm.kv_full[c % kKvSlots], (c / kKvSlots) & 1, abort_flag))) break;
          if (kbase + r >= it.L)
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              reinterpret_cast<uint4*>(sm.kv[c % kKvSlots][0] + r * 128)[q] = make_uint4(0, 0, 0, 0);
              reinterpret_cast<uint4*>(sm.kv[c % kKvSlots][1] + r * 128)[q] = make_uint4(0, 0, 0, 0);
            }
          fence_proxy_async_smem();
        }
        // P = 2^(s - m) (bf16, the row sum over the rounded values); no visible key yet: all zero
        const float mu = m == -INFINITY ? 0.f : m;
        const float2 nm = make_float2(-mu, -mu);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t pk[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float2 d = add2(make_float2(sv[64 * hf + 2 * i], sv[64 * hf + 2 * i + 1]), nm);
            pk[i] = pack2(ex2_approx(d.x), ex2_approx(d.y));
            l = add2(l, unpack2(pk[i]));
          }
          tmem_st32(sb + 32 * hf, pk);
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sm.p_full[a][hf]);
        }
      }
      if (!ok) break;
      base += 2 * nk;
      // the previous item's 1 / l has been read
      if (oph >= 1 && !(ok = wwait(&sm.o_free[a], (oph - 1) & 1, abort_flag))) break;
      ++oph;
      const float lt = l.x + l.y;
      sm.linv[a][r] = lt > 0.f ? 1.f / lt : 0.f;
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.l_full[a]);
    }
  } else {
    // ---- output: thread = row r of each tile --------------------------------------
    reg_dec<kRegsOther>();
    const int quad = warp & 3, r = quad * 32 + lane;
    const uint32_t lb = (uint32_t)(quad * 32) << 16;
    uint32_t oph[2] = {0, 0};
    bool ok = true;
    while (ok && list.next(sm, it, lane, abort_flag)) {
      if (it.bad) {
        // an invalid sequence: recorded, and its output rows of this item are zero
        if (tid == 12 * 32 && it.i0 == 0 && it.h == 0) atomicOr(aa.err, kErrBadSeq);
        for (int e = tid - 12 * 32; e < 256 * (kPD / 8); e += 128) {
          const int rr = e / (kPD / 8), qi = it.i0 + rr / qpg;
          if (qi < aa.qmax)
            *reinterpret_cast<uint4*>(aa.out + (((int64_t)it.b * aa.qmax + qi) * aa.Hq + it.h * qpg + rr % qpg) * kPD +
                                      8 * (e % (kPD / 8))) = make_uint4(0, 0, 0, 0);
        }
        continue;
      }
#pragma unroll 1
      for (int a = 0; a < 2 && ok; ++a) {
        if (it.n[a] == 0) continue;
        if (!(ok = wwait(&sm.o_full[a], oph[a] & 1, abort_flag))) break;
        if (!(ok = wwait(&sm.l_full[a], oph[a] & 1, abort_flag))) break;
        ++oph[a];
        tc_fence_after();
        const int qi = it.i0 + a * pp + r / qpg;
        const float inv = sm.linv[a][r];
        __nv_bfloat16* orow = aa.out + (((int64_t)it.b * aa.qmax + qi) * aa.Hq + it.h * qpg + r % qpg) * kPD;
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          float v[32];
          tmem_ld32(tmem + lb + 256 + 128 * a + 32 * c, v);
          tmem_wait_ld();
          if (qi < it.Q)
#pragma unroll
            for (int q = 0; q < 4; ++q)
              *reinterpret_cast<uint4*>(orow + 32 * c + 8 * q) =
                  make_uint4(pack2(v[8 * q] * inv, v[8 * q + 1] * inv), pack2(v[8 * q + 2] * inv, v[8 * q + 3] * inv),
                             pack2(v[8 * q + 4] * inv, v[8 * q + 5] * inv), pack2(v[8 * q + 6] * inv, v[8 * q + 7] * inv));
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.o_free[a]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (sm.abort_flag) {
    drain_in_flight();
    if (tid == 0) atomicOr(aa.err, kErrTimeout);
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace

static_assert(1024 + kRStages * kRStageBytes + 256 + 8 * (kMaxBatch + 1) <= 232448,
              "shared memory of the reconstruction kernel");
static_assert(sizeof(ASmemP) + 1024 <= 232448, "shared memory of the prefill attention kernel");

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------

bool tc_prefill_supports(const LayerTable& lt, int dtype) {
  if (dtype != DCK_BF16 || lt.d != kPD || lt.G > kMaxGroupsP || lt.Hkv > 128) return false;
  if (lt.qpg != 1 && lt.qpg != 2 && lt.qpg != 4 && lt.qpg != 8) return false;
  if (lt.rv % 16) return false;
  for (int g = 0; g < lt.G; ++g)
    if (lt.grp_rank[g] % 16) return false;
  return true;
}

size_t tc_prefill_workspace(const LayerTable& lt, int64_t n_rows) {
  return 2 * align_up((size_t)std::max<int64_t>(n_rows, 1) * lt.Hkv * kPD * 2, 256);
}

cudaError_t launch_prefill_tc(const LayerTable& lt, const void* q, const int32_t* q_len, int qmax, const void* kc,
                              const void* vc, int64_t n_rows, const void* Bk, const void* Bv,
                              const int64_t* seq_start, const int32_t* seq_len, int B, int max_len, float theta,
                              void* out, void* ws, int* err, LaunchHook* hook, cudaStream_t s) {
  const size_t half = tc_prefill_workspace(lt, n_rows) / 2;
  __nv_bfloat16* kw = static_cast<__nv_bfloat16*>(ws);
  __nv_bfloat16* vw = reinterpret_cast<__nv_bfloat16*>(static_cast<uint8_t*>(ws) + half);
  const uint64_t rows = (uint64_t)std::max<int64_t>(1, n_rows);
  RMaps rm;
  std::memset(&rm, 0, sizeof(rm));
  bool ok = make_tmap_2d_bf16(&rm.va, vc, lt.rv, rows, (uint64_t)lt.rv * 2, kRBK, kTile, CU_TENSOR_MAP_SWIZZLE_128B) &&
            make_tmap_2d_bf16(&rm.vb, Bv, (uint64_t)lt.Hkv * kPD, lt.rv, (uint64_t)lt.Hkv * kPD * 2, 64, kRBK,
                              CU_TENSOR_MAP_SWIZZLE_128B);
  // a group's own columns and ranks only: a 64-wide stage past them loads zeros
  for (int g = 0; g < lt.G && ok; ++g)
    ok = make_tmap_2d_bf16(&rm.ka[g], static_cast<const __nv_bfloat16*>(kc) + lt.grp_roff[g], lt.grp_rank[g], rows,
                           (uint64_t)lt.Rk * 2, kRBK, kTile, CU_TENSOR_MAP_SWIZZLE_128B) &&
         make_tmap_2d_bf16(&rm.kb[g], static_cast<const __nv_bfloat16*>(Bk) + lt.grp_boff[g],
                           (uint64_t)lt.grp_nh[g] * kPD, lt.grp_rank[g], (uint64_t)lt.grp_nh[g] * kPD * 2, 64, kRBK,
                           CU_TENSOR_MAP_SWIZZLE_128B);
  AMapsP am;
  ok = ok && make_tmap_2d_bf16(&am.kw, kw, (uint64_t)lt.Hkv * kPD, rows, (uint64_t)lt.Hkv * kPD * 2, 64, kTile,
                               CU_TENSOR_MAP_SWIZZLE_128B) &&
       make_tmap_2d_bf16(&am.vw, vw, (uint64_t)lt.Hkv * kPD, rows, (uint64_t)lt.Hkv * kPD * 2, 64, kTile,
                         CU_TENSOR_MAP_SWIZZLE_128B) &&
       make_tmap_3d_bf16(&am.q, out, kPD, lt.Hq, (uint64_t)B * qmax, kPD * 2, (uint64_t)lt.Hq * kPD * 2, 64, lt.qpg,
                         128 / lt.qpg, CU_TENSOR_MAP_SWIZZLE_128B);
  if (!ok) return cudaErrorInvalidValue;
  RArgs ra;
  std::memset(&ra, 0, sizeof(ra));
  ra.seq_start = seq_start;
  ra.seq_len = seq_len;
  ra.q_len = q_len;
  ra.n_rows = n_rows;
  ra.B = B;
  ra.Hq = lt.Hq;
  ra.Hkv = lt.Hkv;
  ra.qmax = qmax;
  ra.max_len = max_len;
  for (int h = 0; h < lt.Hkv; h += 2) {
    const int nh = std::min(2, lt.Hkv - h);
    ra.col[ra.n_val++] = RCol{-1, (int16_t)(h * kPD), (int16_t)(nh * kPD), (int16_t)h, (int16_t)(h + 1), lt.rv};
  }
  int head_at[kMaxGroupsP][kMaxKvHeads];
  for (int h = 0; h < lt.Hkv; ++h) head_at[lt.head_group[h]][lt.head_slot[h]] = h;
  for (int g = 0; g < lt.G; ++g)
    for (int sl = 0; sl < lt.grp_nh[g]; sl += 2) {
      const int nh = std::min(2, lt.grp_nh[g] - sl);
      ra.col[ra.n_val + ra.n_key++] = RCol{(int16_t)g, (int16_t)(sl * kPD), (int16_t)(nh * kPD),
                                           (int16_t)head_at[g][sl],
                                           (int16_t)(nh == 2 ? head_at[g][sl + 1] : 0), lt.grp_rank[g]};
    }
  ra.rf = rope_freqs_of(theta, kPD);
  ra.qscale = 1.4426950408889634f / std::sqrt((float)kPD);
  ra.q = static_cast<const __nv_bfloat16*>(q);
  ra.kw = kw;
  ra.vw = vw;
  ra.qr = static_cast<__nv_bfloat16*>(out);
  ra.err = err;
  cudaError_t e = hook_begin(hook, s);
  if (e != cudaSuccess) return e;
  const size_t asmem = sizeof(ASmemP) + 1024;
  const int pairs = recon_pairs_of_device();
  if (pairs <= 0) return cudaErrorInvalidConfiguration;
  e = cudaFuncSetAttribute(prefill_attn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)asmem);
  if (e != cudaSuccess) return e;
  if ((e = launch_recon(rm, ra, pairs, s)) != cudaSuccess) return e;
  if ((e = hook_launched(hook, s)) != cudaSuccess) return e;
  AArgsP aa;
  std::memset(&aa, 0, sizeof(aa));
  aa.q_len = q_len;
  aa.qmax = qmax;
  aa.max_len = max_len;
  aa.seq_start = seq_start;
  aa.seq_len = seq_len;
  aa.n_rows = n_rows;
  aa.B = B;
  aa.Hq = lt.Hq;
  aa.Hkv = lt.Hkv;
  aa.qpg = lt.qpg;
  aa.out = static_cast<__nv_bfloat16*>(out);
  aa.err = err;
  const int pp2 = 2 * (128 / lt.qpg);
  aa.ntp = (qmax + pp2 - 1) / pp2;
  // streams whose keys and values (at most) share L2: about half of it
  const int64_t streams = (int64_t)B * lt.Hkv;
  aa.group = (int)std::max<int64_t>(1, std::min<int64_t>(streams, (int64_t(64) << 20) / ((int64_t)max_len * kPD * 4)));
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int64_t items = streams * aa.ntp;
  // its set-up overlaps the reconstruction's end
  e = launch_pdl(prefill_attn_kernel, dim3((unsigned)std::min<int64_t>(items, sms)), dim3(kAThreadsP), asmem, s, am, aa);
  return e != cudaSuccess ? e : hook_launched(hook, s);
}

}  // namespace dck
