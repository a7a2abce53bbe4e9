// RoPE angles as exact fractions of a turn, shared by the kernels that rotate
// keys and queries at given positions.
#pragma once

#include <cmath>

#include "common.cuh"

namespace dck {

constexpr int kMaxHeadDim = 128;

// Frequency w_i / (2 pi) as a 64-bit binary fraction: position t turns pair i
// by the fraction t * f (mod 2^64), exactly, so an angle needs two integer
// multiplies and no fp64, and its reduction mod 2 pi is the wrap-around.
struct RopeFreqs {
  uint2 f[kMaxHeadDim / 2];  // {low, high} words
};

// sin and cos of 2 pi u / 2^32.  The nearest quarter turn is taken off exactly
// in integers; the remainder, within +-pi/4, goes through the Taylor series of
// sine (to x^9) and cosine (to x^10), whose truncation errors there (1.8e-9
// and 1.2e-10) are below fp32 rounding.
__device__ __forceinline__ void turn_sincos(uint32_t u, float& sn, float& cs) {
  const uint32_t q = (u + 0x20000000u) >> 30;
  const float x = (float)(int32_t)(u - (q << 30)) * 1.4629180792671596e-9f;  // 2 pi / 2^32
  const float x2 = x * x;
  float s = fmaf(x2, 2.7557319e-6f, -1.9841270e-4f);
  s = fmaf(x2, s, 8.3333333e-3f);
  s = fmaf(x2, s, -1.6666667e-1f);
  s = fmaf(x * x2, s, x);
  float c = fmaf(x2, -2.7557319e-7f, 2.4801587e-5f);
  c = fmaf(x2, c, -1.3888889e-3f);
  c = fmaf(x2, c, 4.1666667e-2f);
  c = fmaf(x2, c, -0.5f);
  c = fmaf(x2, c, 1.f);
  const float a = (q & 1) ? c : s, b = (q & 1) ? s : c;
  sn = __uint_as_float(__float_as_uint(a) ^ ((q & 2) << 30));
  cs = __uint_as_float(__float_as_uint(b) ^ (((q + 1) & 2) << 30));
}
__device__ __forceinline__ void rope_sincos(uint2 f, uint32_t pos, float& sn, float& cs) {
  turn_sincos(__umulhi(pos, f.x) + pos * f.y, sn, cs);
}

// The frequencies theta^(-2i/d) of head dim d.
inline RopeFreqs rope_freqs_of(float theta, int d) {
  RopeFreqs r = {};
  for (int i = 0; i < d / 2; ++i) {
    const double turns = std::exp2(-2.0 * i / d * std::log2((double)theta)) * 0.15915494309189533577;
    const double fr = turns - std::floor(turns);  // a whole number of turns per position is none
    const uint64_t f = (uint64_t)std::ldexp(fr, 64);
    r.f[i] = make_uint2((uint32_t)f, (uint32_t)(f >> 32));
  }
  return r;
}

}  // namespace dck
