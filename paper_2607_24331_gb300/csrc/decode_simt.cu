// CUDA-core decode attention over the DynaCalKV latent caches.
//
// The general kernel: any head_dim in {64, 128}, fp32 or bf16 storage, fp32
// arithmetic, RoPE angles exact in integers.  It is the kernel for fp32 layers
// (whose 1e-5 tolerance tensor-core bf16/tf32 products cannot meet) and for
// shapes the tensor-core kernel does not take.
//
// Block (item c, KV head h): for every sequence segment in item c's range of
// 32-token tiles, tile by tile
//   k_t = c_t^g B_g[:, slot(h)]        (Sec. III-A/III-C reconstruction)
//   RoPE(k_t, t); scores against RoPE(q_j, L-1) / sqrt(d) for the query heads
//   of h; online softmax in log2 units;
//   u_j += p_t v_t                      (value latent, Sec. III-D; B_v is
//                                        applied once after the split merge)
// and the segment's (u_j, m_j, l_j) is written to partial slot c + b.
//
// What bounds it: latency.  The fp32 layer's call of 512 tokens is 0.04 GFLOP
// over 1 MB; a block's time is its chain of dependent memory round trips and
// barriers.  So the head's factor slice sits in shared memory for the whole
// item, copied together with the first latent tile (one round trip instead of
// one per rank), the next latent and value tiles are in flight under the
// current one, a thread's keys are held as RoPE pairs in registers from the
// reconstruction to the scores, and angles use integers: fp64 sine and cosine,
// at a couple of fp64 operations per cycle and SM, took most of the kernel
// before.  Tiles of 32 tokens, so that a short sequence still fills the SMs.
// Step of the fp32 layer (append, this kernel, merge), L2 flushed, before / now:
// 1 x 512 tokens 246 / 20 us, 3 x 777 255 / 30, 8 x 4096 1004 / 178 (35 us of
// multiply-adds).
#include <algorithm>

#include "common.cuh"
#include "rope.cuh"

namespace dck {
namespace {

constexpr int kThreads = 256;
constexpr int kTok = kSimtTile;   // tokens of a tile
constexpr int kMaxRankK = 256;  // per-group rank handled by this kernel
// Blocks of one query head per KV head resident on an SM (three: 172 us at 8 x
// 4096, but 34 against 30 at 3 x 777, and spills at d = 128).
constexpr int kBlocksPerSm = 2;
constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ float2 pair_of(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 pair_of(const __nv_bfloat16* p) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
}
__device__ __forceinline__ float4 quad_of(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 quad_of(const __nv_bfloat16* p) {
  const float2 a = pair_of(p), b = pair_of(p + 2);
  return make_float4(a.x, a.y, b.x, b.y);
}

// Row stride of the staged latent tile: padded by 16 bytes, so that the token
// rows one warp reads lie in different banks.
template <typename T>
__host__ __device__ constexpr int ldc_of(int r) {
  return r + 16 / (int)sizeof(T);
}

// Shared memory of a block, for the layer's widest group.
template <typename T, int D>
__host__ __device__ constexpr size_t simt_smem(int rmax, int B) {
  return sizeof(T) * ((size_t)rmax * D + 2 * (size_t)kTok * ldc_of<T>(rmax)) +
         sizeof(float) * (kMaxQPerKv * D + kMaxQPerKv * kTok + kMaxQPerKv) + sizeof(int) * (B + 1 + kThreads / 32);
}

// QP: query heads per KV head the thread's accumulators are sized for.
template <typename T, int D, int QP>
__global__ void __launch_bounds__(kThreads, QP == 1 ? kBlocksPerSm : 1)
    decode_simt_kernel(const LayerTable lt, const DecodeArgs a, const RopeFreqs rf, int rmax) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  const int c = blockIdx.x;
  const int h = blockIdx.y;
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int B = a.B;

  T* sB = reinterpret_cast<T*>(smem_raw);                            // [r][D] the head's factor slice
  T* sC = sB + (size_t)rmax * D;                                     // 2 x [kTok][ldc] latent tiles
  float* sq = reinterpret_cast<float*>(sC + 2 * (size_t)kTok * ldc_of<T>(rmax));  // [qpg][D] rotated queries
  float* sP = sq + kMaxQPerKv * D;                                   // [qpg][kTok]
  float* sAlpha = sP + kMaxQPerKv * kTok;                            // [qpg]
  int* prefix = reinterpret_cast<int*>(sAlpha + kMaxQPerKv);         // [B + 1]
  int* scan = prefix + B + 1;                                        // [warps]

  pdl_launch_dependents();
  const int g = lt.head_group[h];
  const int slot = lt.head_slot[h];
  const int r = lt.grp_rank[g];
  const int roff = lt.grp_roff[g];
  const int qpg = QP == 1 ? 1 : lt.qpg;
  const int rv = lt.rv;
  const int Rk = lt.Rk;
  const int ldc = ldc_of<T>(r);
  const T* __restrict__ kc = static_cast<const T*>(a.kc);
  const T* __restrict__ vc = static_cast<const T*>(a.vc);

  const int NT = build_tile_prefix(a.seq_len, a.seq_start, B, a.n_rows, prefix, scan, a.err,
                                   c == 0 && h == 0, kTok);
  const int x0 = item_begin(c, NT, a.n_items);
  const int x1 = item_begin(c + 1, NT, a.n_items);
  if (x0 >= x1) {
    pdl_wait();  // this grid is not complete before the one it was launched after
    return;
  }
  {  // the head's factor slice, with the first latent tile's copy group
    const T* Bg = static_cast<const T*>(a.Bk) + lt.grp_boff[g] + (int64_t)slot * D;
    const int64_t ld = (int64_t)lt.grp_nh[g] * D;
    constexpr int kSeg = D * (int)sizeof(T) / 16;
    for (int i = tid; i < r * kSeg; i += kThreads)
      cp_async16(reinterpret_cast<uint8_t*>(sB + (size_t)(i / kSeg) * D) + (i % kSeg) * 16,
                 reinterpret_cast<const uint8_t*>(Bg + (int64_t)(i / kSeg) * ld) + (i % kSeg) * 16);
  }
  pdl_wait();  // the kernel before may append the step's own latents

  // Thread: 4 columns of the key as two RoPE pairs (e0, e0 + D/2), (e0 + 1, ..),
  // and every kTG-th token of a tile.
  constexpr int kDG = D / 4;            // column groups
  constexpr int kTG = kThreads / kDG;   // token groups
  constexpr int TPT = kTok / kTG;       // tokens per thread: 2 (D = 64) or 4
  const int dg = tid % kDG, tg = tid / kDG;
  const int e0 = 2 * dg;
  constexpr int kRvPerThread = kMaxRankV / kThreads;

  int buf = 0;
  for (int x = x0; x < x1;) {
    const int b = seq_of_tile(prefix, B, x);
    const int seg_end_tile = min(x1, prefix[b + 1]);
    const int L = valid_len(a.seq_len, a.seq_start, b, a.n_rows);
    const int64_t row0 = a.seq_start[b];
    const int t_begin = (x - prefix[b]) * kTok;
    const int t_end = min(L, (seg_end_tile - prefix[b]) * kTok);
    x = seg_end_tile;

    // latent tile at t0 into buffer bf (rows past the segment repeat its last)
    auto load_c = [&](int t0, int bf) {
      const int segs = r * (int)sizeof(T) / 16;
      T* dst = sC + (size_t)bf * kTok * ldc_of<T>(rmax);
      for (int i = tid; i < kTok * segs; i += kThreads) {
        const int t = i / segs, s = i % segs;
        cp_async16(reinterpret_cast<uint8_t*>(dst + t * ldc) + s * 16,
                   reinterpret_cast<const uint8_t*>(kc + (row0 + min(t0 + t, t_end - 1)) * Rk + roff) + s * 16);
      }
      cp_async_commit();
    };
    // value latents of tile t0, column tid (the first kThreads of r_v)
    float vs[kTok];
    auto load_v = [&](int t0, int rr) {
#pragma unroll
      for (int t = 0; t < kTok; ++t) vs[t] = to_f32(vc[(row0 + min(t0 + t, t_end - 1)) * rv + rr]);
    };
    load_c(t_begin, buf);
    if (tid < rv) load_v(t_begin, tid);
    // rotated, scaled query heads of this KV head (position L-1)
    const float qscale = rsqrtf((float)D) * kLog2e;
    for (int i = tid; i < qpg * (D / 2); i += kThreads) {
      const int jj = i / (D / 2), p = i % (D / 2);
      const T* qp = static_cast<const T*>(a.q) + ((int64_t)b * lt.Hq + h * qpg + jj) * D;
      float sn, cs;
      rope_sincos(rf.f[p], (uint32_t)(L - 1), sn, cs);
      const float x1v = to_f32(qp[p]), x2v = to_f32(qp[p + D / 2]);
      sq[jj * D + p] = fmaf(x1v, cs, -x2v * sn) * qscale;
      sq[jj * D + p + D / 2] = fmaf(x1v, sn, x2v * cs) * qscale;
    }
    float acc[QP][kRvPerThread];
#pragma unroll
    for (int jj = 0; jj < QP; ++jj)
#pragma unroll
      for (int k = 0; k < kRvPerThread; ++k) acc[jj][k] = 0.f;
    float m_run = -INFINITY, l_run = 0.f;  // meaningful in warp jj for jj < qpg

    for (int t0 = t_begin; t0 < t_end; t0 += kTok) {
      const int nt = min(kTok, t_end - t0);
      cp_async_wait<0>();
      __syncthreads();  // the tile (and the factor slice, the queries) are there; the other buffer is free
      const T* cb = sC + (size_t)buf * kTok * ldc_of<T>(rmax);
      buf ^= 1;
      if (t0 + kTok < t_end) load_c(t0 + kTok, buf);
      // reconstruction: k_t[e] = sum_k c_t[k] B_g[k][slot*D + e], four ranks at a
      // time; every kChains-th rank is summed apart (shorter rounding chains)
      constexpr int kChains = TPT == 2 ? 4 : 2;
      float kc_[kChains][TPT][4];
#pragma unroll
      for (int q = 0; q < kChains; ++q)
#pragma unroll
        for (int u = 0; u < TPT; ++u)
#pragma unroll
          for (int j = 0; j < 4; ++j) kc_[q][u][j] = 0.f;
#pragma unroll 2
      for (int k = 0; k < r; k += 4) {
        float4 cv[TPT];
#pragma unroll
        for (int u = 0; u < TPT; ++u) cv[u] = quad_of(cb + (tg + u * kTG) * ldc + k);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 lo = pair_of(sB + (size_t)(k + q) * D + e0);
          const float2 hi = pair_of(sB + (size_t)(k + q) * D + D / 2 + e0);
#pragma unroll
          for (int u = 0; u < TPT; ++u) {
            const float w = q == 0 ? cv[u].x : (q == 1 ? cv[u].y : (q == 2 ? cv[u].z : cv[u].w));
            float(&kk)[4] = kc_[q % kChains][u];
            kk[0] = fmaf(w, lo.x, kk[0]);
            kk[1] = fmaf(w, lo.y, kk[1]);
            kk[2] = fmaf(w, hi.x, kk[2]);
            kk[3] = fmaf(w, hi.y, kk[3]);
          }
        }
      }
      float ka[TPT][4];
#pragma unroll
      for (int u = 0; u < TPT; ++u)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          ka[u][j] = kChains == 4 ? (kc_[0][u][j] + kc_[1][u][j]) + (kc_[2 % kChains][u][j] + kc_[3 % kChains][u][j])
                                  : kc_[0][u][j] + kc_[1][u][j];
      // RoPE at the token's position, then the scores (log2 units): this thread's
      // four columns, summed over the column groups
#pragma unroll
      for (int u = 0; u < TPT; ++u) {
        const uint32_t pos = (uint32_t)(t0 + tg + u * kTG);
        float sn, cs;
        rope_sincos(rf.f[e0], pos, sn, cs);
        const float a0 = fmaf(ka[u][0], cs, -ka[u][2] * sn), b0 = fmaf(ka[u][0], sn, ka[u][2] * cs);
        rope_sincos(rf.f[e0 + 1], pos, sn, cs);
        const float a1 = fmaf(ka[u][1], cs, -ka[u][3] * sn), b1 = fmaf(ka[u][1], sn, ka[u][3] * cs);
        for (int jj = 0; jj < qpg; ++jj) {
          const float2 ql = pair_of(sq + jj * D + e0), qh = pair_of(sq + jj * D + D / 2 + e0);
          float s = fmaf(ql.x, a0, ql.y * a1) + fmaf(qh.x, b0, qh.y * b1);
#pragma unroll
          for (int o = kDG / 2; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (dg == 0) sP[jj * kTok + tg + u * kTG] = tg + u * kTG < nt ? s : -INFINITY;
        }
      }
      __syncthreads();
      // online softmax: warp jj owns query head jj
      if (warp < qpg) {
        const float s = sP[warp * kTok + lane];
        float mx = s;
#pragma unroll
        for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float m_new = fmaxf(m_run, mx);
        const float alpha = exp2f(m_run - m_new);  // 0 on the first tile
        const float p = exp2f(s - m_new);
        float ps = p;
#pragma unroll
        for (int o = 16; o; o >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, o);
        l_run = l_run * alpha + ps;
        m_run = m_new;
        sP[warp * kTok + lane] = p;
        if (lane == 0) sAlpha[warp] = alpha;
      }
      __syncthreads();
      // u_j = alpha u_j + sum_t p_t v_t
#pragma unroll
      for (int k = 0; k < kRvPerThread; ++k) {
        const int rr = tid + k * kThreads;
        if (rr < rv) {
          if (k > 0) load_v(t0, rr);
#pragma unroll
          for (int jj = 0; jj < QP; ++jj) {
            if (jj < qpg) {
              float s[4] = {acc[jj][k] * sAlpha[jj], 0.f, 0.f, 0.f};
#pragma unroll
              for (int t = 0; t < kTok; t += 4) {
                const float4 p4 = quad_of(sP + jj * kTok + t);
                s[0] = fmaf(p4.x, vs[t], s[0]);
                s[1] = fmaf(p4.y, vs[t + 1], s[1]);
                s[2] = fmaf(p4.z, vs[t + 2], s[2]);
                s[3] = fmaf(p4.w, vs[t + 3], s[3]);
              }
              acc[jj][k] = (s[0] + s[1]) + (s[2] + s[3]);
            }
          }
        }
      }
      if (t0 + kTok < t_end && tid < rv) load_v(t0 + kTok, tid);
    }
    // partial of (item c, sequence b) -> slot c + b
    const int64_t slot_id = (int64_t)c + b;
#pragma unroll
    for (int jj = 0; jj < QP; ++jj) {
      if (jj < qpg) {
        const int j = h * qpg + jj;
        float* pu = a.part_u + (slot_id * lt.Hq + j) * (int64_t)rv;
#pragma unroll
        for (int k = 0; k < kRvPerThread; ++k) {
          const int rr = tid + k * kThreads;
          if (rr < rv) pu[rr] = acc[jj][k];
        }
      }
    }
    if (warp < qpg && lane == 0) {
      const int j = h * qpg + warp;
      float* pm = a.part_ml + (slot_id * lt.Hq + j) * 2;
      pm[0] = t_end > t_begin ? m_run : -INFINITY;
      pm[1] = l_run;
    }
    __syncthreads();  // the segment's queries and latent tiles have been read
  }
}

int max_rank(const LayerTable& lt) {
  int r = 0;
  for (int g = 0; g < lt.G; ++g) r = std::max(r, lt.grp_rank[g]);
  return r;
}

size_t smem_of(const LayerTable& lt, int dtype, int B) {
  const int r = max_rank(lt);
  if (dtype == DCK_F32) return lt.d == 64 ? simt_smem<float, 64>(r, B) : simt_smem<float, 128>(r, B);
  return lt.d == 64 ? simt_smem<__nv_bfloat16, 64>(r, B) : simt_smem<__nv_bfloat16, 128>(r, B);
}

template <typename T, int D, int QP>
cudaError_t launch_qp(const LayerTable& lt, const DecodeArgs& a, bool after_append, size_t smem, cudaStream_t s) {
  auto k = decode_simt_kernel<T, D, QP>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const dim3 grid(a.n_items, lt.Hkv);
  if ((e = hook_begin(a.hook, s)) != cudaSuccess) return e;
  const RopeFreqs rf = rope_freqs_of(a.theta, D);
  const int rmax = max_rank(lt);
  // Only after this library's own append may the kernel start early: what it
  // reads before its wait is then known to be complete.
  if (after_append) {
    if ((e = launch_pdl(k, grid, dim3(kThreads), smem, s, lt, a, rf, rmax)) != cudaSuccess) return e;
  } else {
    k<<<grid, kThreads, smem, s>>>(lt, a, rf, rmax);
  }
  return hook_launched(a.hook, s);
}

template <typename T, int D>
cudaError_t launch_t(const LayerTable& lt, const DecodeArgs& a, bool after_append, size_t smem, cudaStream_t s) {
  return lt.qpg == 1 ? launch_qp<T, D, 1>(lt, a, after_append, smem, s)
                     : launch_qp<T, D, kMaxQPerKv>(lt, a, after_append, smem, s);
}

}  // namespace

bool simt_supports(const LayerTable& lt) {
  if (lt.d != 64 && lt.d != 128) return false;
  if (lt.qpg > kMaxQPerKv || lt.rv > kMaxRankV) return false;
  return max_rank(lt) <= kMaxRankK;
}

// Work items of a call: enough blocks (items x KV heads) for one wave of
// resident blocks, no more items than tiles or SMs (the partial slots are
// sized for one item per SM).
int simt_items(const LayerTable& lt, int dtype, int B, int64_t n_rows, int sms) {
  const size_t smem = smem_of(lt, dtype, B) + 1024;
  const int per_sm = std::max(1, std::min<int>(lt.qpg == 1 ? kBlocksPerSm : 1, (int)(233472 / smem)));
  const int64_t tiles = (n_rows + kSimtTile - 1) / kSimtTile + B;
  const int64_t n = std::min<int64_t>(tiles, std::max(1, sms * per_sm / lt.Hkv));
  return (int)std::max<int64_t>(1, std::min<int64_t>(n, sms));
}

cudaError_t launch_decode_simt(const LayerTable& lt, const DecodeArgs& a, int dtype, bool after_append,
                               cudaStream_t s) {
  const size_t smem = smem_of(lt, dtype, a.B);
  if (dtype == DCK_F32)
    return lt.d == 64 ? launch_t<float, 64>(lt, a, after_append, smem, s)
                      : launch_t<float, 128>(lt, a, after_append, smem, s);
  return lt.d == 64 ? launch_t<__nv_bfloat16, 64>(lt, a, after_append, smem, s)
                    : launch_t<__nv_bfloat16, 128>(lt, a, after_append, smem, s);
}

}  // namespace dck
