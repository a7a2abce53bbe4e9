// CUDA-core latent append: key and value latents of new tokens,
//   kcache[rows[i]] = x_i A_k,  vcache[rows[i]] = x_i A_v     (Sec. III-A z = x L)
// with fp32 accumulation.  Used for fp32 layers and as the general kernel; bf16
// layers take the tensor-core kernel.  A few tokens (a decode step's) are a
// matrix-vector product that wants every factor byte in flight at once; many
// are a plain 64x64-tiled GEMM.
#include "common.cuh"

namespace dck {
namespace {

constexpr int kBM = 64, kBN = 64, kBK = 16;

template <typename T>
__global__ void __launch_bounds__(256) append_simt_kernel(const T* __restrict__ x, int n_tok, int D,
                                                          const T* __restrict__ Ak, const T* __restrict__ Av,
                                                          int Rk, int rv, const int64_t* __restrict__ rows,
                                                          T* kc, T* vc, int64_t n_rows, int* err) {
  __shared__ float sx[kBK][kBM + 1];
  __shared__ float sa[kBK][kBN];
  const int n0 = blockIdx.x * kBN;  // column over [0, Rk + rv)
  const int m0 = blockIdx.y * kBM;
  const int N = Rk + rv;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < D; k0 += kBK) {
    for (int i = threadIdx.x; i < kBK * kBM; i += 256) {
      const int mm = i / kBK, kk = i % kBK;
      const int m = m0 + mm, k = k0 + kk;
      sx[kk][mm] = (m < n_tok && k < D) ? to_f32(x[(int64_t)m * D + k]) : 0.f;
    }
    for (int i = threadIdx.x; i < kBK * kBN; i += 256) {
      const int kk = i / kBN, nn = i % kBN;
      const int n = n0 + nn, k = k0 + kk;
      float v = 0.f;
      if (k < D && n < N) v = n < Rk ? to_f32(Ak[(int64_t)k * Rk + n]) : to_f32(Av[(int64_t)k * rv + (n - Rk)]);
      sa[kk][nn] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kBK; ++kk) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(sx[kk][ty * 4 + i], sa[kk][tx * 4 + j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty * 4 + i;
    if (m >= n_tok) continue;
    const int64_t row = rows[m];
    if (row < 0 || row >= n_rows) {
      atomicOr(err, kErrBadRow);
      continue;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx * 4 + j;
      if (n < Rk) kc[row * Rk + n] = from_f32<T>(acc[i][j]);
      else if (n < N) vc[row * rv + (n - Rk)] = from_f32<T>(acc[i][j]);
    }
  }
}

// Few tokens: block (8 output columns, 8 tokens).  Bound by latency (the fp32
// layer's factors are 0.6 MB): the 128 row lanes of a block each take every
// 128th row of D, four rows' loads in flight together, and the sums of the
// lanes meet in shuffles and shared memory once.
constexpr int kVCols = 8, kVTok = 8;
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xFFFF0000u));
}

template <typename T>
__global__ void __launch_bounds__(256) append_few_kernel(const T* __restrict__ x, int n_tok, int D,
                                                         const T* __restrict__ Ak, const T* __restrict__ Av, int Rk,
                                                         int rv, const int64_t* __restrict__ rows, T* kc, T* vc,
                                                         int64_t n_rows, int* err) {
  __shared__ float red[8][kVTok][kVCols];
  pdl_launch_dependents();
  const int c0 = blockIdx.x * kVCols;  // R_k and r_v are multiples of 16: a block has columns of one factor
  const bool is_k = c0 < Rk;
  const int N = is_k ? Rk : rv, col = is_k ? c0 : c0 - Rk;
  const int m0 = blockIdx.y * kVTok, nm = min(kVTok, n_tok - m0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kl = threadIdx.x >> 1;     // row lane
  const T* __restrict__ A = (is_k ? Ak : Av) + col + 4 * (threadIdx.x & 1);
  const T* __restrict__ xm = x + (int64_t)m0 * D;
  float acc[kVTok][4] = {};
  for (int k0 = kl; k0 < D; k0 += 4 * 128) {
    float4 w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      w[q] = k0 + 128 * q < D ? load4(A + (int64_t)(k0 + 128 * q) * N) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int m = 0; m < kVTok; ++m) {
      if (m >= nm) break;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float xv = k0 + 128 * q < D ? to_f32(xm[(int64_t)m * D + k0 + 128 * q]) : 0.f;
        acc[m][0] = fmaf(xv, w[q].x, acc[m][0]);
        acc[m][1] = fmaf(xv, w[q].y, acc[m][1]);
        acc[m][2] = fmaf(xv, w[q].z, acc[m][2]);
        acc[m][3] = fmaf(xv, w[q].w, acc[m][3]);
      }
    }
  }
#pragma unroll
  for (int m = 0; m < kVTok; ++m) {
    if (m >= nm) break;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int o = 16; o > 1; o >>= 1) acc[m][j] += __shfl_xor_sync(0xffffffffu, acc[m][j], o);
      if (lane < 2) red[warp][m][4 * lane + j] = acc[m][j];
    }
  }
  __syncthreads();
  const int m = threadIdx.x / kVCols, c = threadIdx.x % kVCols;
  if (m >= nm) return;
  float v = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) v += red[w][m][c];
  const int64_t row = rows[m0 + m];
  if (row < 0 || row >= n_rows) {
    atomicOr(err, kErrBadRow);
    return;
  }
  (is_k ? kc : vc)[row * N + col + c] = from_f32<T>(v);
}

// Whether a call is one of few tokens.  The tile kernel's time is set by its D / 16
// steps in series (about 8 + 0.22 D us while its tiles fit the SMs); this one's by its
// multiply-adds, for every eight tokens of which the factors are read again from L2, and
// by its blocks (about 9 + 0.49 n_tok (R_k + r_v) (D + 225) / 10^6 us): equal where
// n_tok (R_k + r_v) (D + 225) = 4.5 10^5 D.  fp32, us, tile kernel / this one, by
// n_tok (R_k + r_v) in thousands, ! where the rule takes the tile kernel:
//   D = 64:   66 19 / 19    78 21 / 21    131 21 / 27!   262 22 / 46!   2097 27 / 314!
//   D = 512:  66 105 / 33   156 113 / 70  262 124 / 103  393 122 / 148! 2097 138 / 758!
//   D = 2048: 66 398 / 99   156 461 / 232 262 476 / 324  393 474 / 482! 2097 523 / 2443!
// (Not beyond 512 tokens, where neither was measured on narrow layers.)
constexpr int kFewTokens = 512;
inline bool few_tokens(int n_tok, int D, int width) {
  return n_tok <= kFewTokens && (int64_t)n_tok * width * (D + 256) <= (int64_t)400000 * D;
}

template <typename T>
cudaError_t launch_t(const void* x, int n_tok, int D, const void* A_k, const void* A_v, int Rk, int rv,
                     const int64_t* rows, void* kc, void* vc, int64_t n_rows, int* err, cudaStream_t s) {
  if (few_tokens(n_tok, D, Rk + rv))
    append_few_kernel<T><<<dim3((Rk + rv) / kVCols, (n_tok + kVTok - 1) / kVTok), 256, 0, s>>>(
        (const T*)x, n_tok, D, (const T*)A_k, (const T*)A_v, Rk, rv, rows, (T*)kc, (T*)vc, n_rows, err);
  else
    append_simt_kernel<T><<<dim3((Rk + rv + kBN - 1) / kBN, (n_tok + kBM - 1) / kBM), 256, 0, s>>>(
        (const T*)x, n_tok, D, (const T*)A_k, (const T*)A_v, Rk, rv, rows, (T*)kc, (T*)vc, n_rows, err);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_append_simt(const void* x, int n_tok, int D, const void* A_k, const void* A_v, int Rk, int rv,
                               const int64_t* rows, void* kc, void* vc, int64_t n_rows, int dtype, int* err,
                               cudaStream_t s) {
  return dtype == DCK_F32
             ? launch_t<float>(x, n_tok, D, A_k, A_v, Rk, rv, rows, kc, vc, n_rows, err, s)
             : launch_t<__nv_bfloat16>(x, n_tok, D, A_k, A_v, Rk, rv, rows, kc, vc, n_rows, err, s);
}

}  // namespace dck
