// graph_device.cuh -- device code shared by the +-1 graph kernels: fp32 bounds on the
// heat-bath threshold and the decision of one lane that the top bytes leave open.
#pragma once

#include <cstdint>

#include "shaken_internal.cuh"

namespace shk {

// 2^x (PTX ex2.approx: relative error below 2^-22 over the range used here).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Bounds lo <= T <= hi on T = floor(2^32 / (1 + 2^x)), x = kb h, kb = -2 beta log2(e),
// from the fp32 field hf.  hf carries at most four roundings of magnitude <= B
// (B = d + |q| + |lambda| + 1), so kb hf is within |kb| B 2^-22 of kb h; with the
// rounding of kb hf, ex2.approx (2^-22), 1 + e, the reciprocal and the product, T~ is
// within min(T~, 2^32 - T~) eps + 2^8 of 2^32 p, eps = 2^-21 (2 + |x| + |kb| B)
// bounding twice the relative error; the margin 1024 also covers the floor.
__device__ __forceinline__ void t_bounds(float hf, float kb, float kbB, float& lo, float& hi) {
  const float x = kb * hf;
  const float e = ex2_approx(x);
  const float T = 4294967296.0f * rcp_approx(1.0f + e);
  const float m = fminf(T, 4294967296.0f - T);
  const float eps = 4.76837158203125e-07f * (2.0f + fabsf(x) + kbB);
  const float D = fmaf(m, eps, 1024.0f);
  lo = fmaxf(T - D, 0.0f);
  hi = fminf(T + D, 4294967296.0f);
}

// A field of exactly 0 gives T = 2^31 exactly (p = 1/2), on a byte boundary where the
// fp32 bounds cannot fix the top byte: with integer couplings and lambda = 0 (or q
// canceling lambda) it is a whole class of lanes.  When the fp32 field is 0, the fp64
// field (the rounding order of the threshold's definition) decides whether T is
// exactly 2^31.
static __device__ __noinline__ bool field_is_zero(int s, int sig, double q, float lam) {
  return field_h(1.0, s, q, sig ? 1 : -1, (double)lam) == 0.0;
}

// Top byte of a value in [0, 2^32] (2^32, i.e. T that always accepts, maps to 255: a
// lane whose draw has top byte 255 is then left to the per-lane decision).
__device__ __forceinline__ uint32_t top_byte(float v) {
  const uint32_t b = __float2uint_rz(v * 5.9604644775390625e-08f);
  return b > 255u ? 255u : b;
}

// Bits k of eight plane words, most significant first.
__device__ __forceinline__ uint32_t lane_byte(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3,
                                              uint32_t w4, uint32_t w5, uint32_t w6, uint32_t w7,
                                              int k) {
  return (((w0 >> k) & 1u) << 7) | (((w1 >> k) & 1u) << 6) | (((w2 >> k) & 1u) << 5) |
         (((w3 >> k) & 1u) << 4) | (((w4 >> k) & 1u) << 3) | (((w5 >> k) & 1u) << 2) |
         (((w6 >> k) & 1u) << 1) | ((w7 >> k) & 1u);
}

// Decision of one lane left undecided by the head (its draw's top byte u8 equals the
// threshold's, or its class's top byte was not certain): planes 8..15 and then 16..31
// against the fp32 bounds on T, and T in fp64 where the bounds do not decide
// (force_exact: straight to fp64).  Out of line: reached by about 2^-8 of the lanes.
static __device__ __noinline__ bool decide_lane(uint32_t key0, uint32_t key1, uint32_t x, uint32_t g,
                                         uint32_t t, uint32_t typ, int k, uint32_t u8, int a,
                                         int d, int sig, float bp, float bm, double q, float lam,
                                         float kb, float kbB, double beta, bool force_exact) {
  float lo = 0.0f, hi = 4294967296.0f;
  if (!force_exact) {
    const float hf = fmaf(2.0f, (float)a, sig ? bp : bm);
    t_bounds(hf, kb, kbB, lo, hi);
    if (hf == 0.0f && field_is_zero(2 * a - d, sig, q, lam)) lo = hi = 2147483648.0f;  // T = 2^31
    if ((float)(u8 + 1u) * 16777216.0f <= lo) return true;  // u < (u8 + 1) 2^24 <= T
    if ((float)u8 * 16777216.0f >= hi) return false;        // u >= u8 2^24 >= T
  }
  const PhKey K = ph_key(key0, key1);
  const uint4 c2 = ph_call(K, x, g, t, typ + 4u), c3 = ph_call(K, x, g, t, typ + 6u);
  const uint32_t u16 = (u8 << 8) | lane_byte(c2.x, c2.y, c2.z, c2.w, c3.x, c3.y, c3.z, c3.w, k);
  if (!force_exact) {
    if ((float)(u16 + 1u) * 65536.0f <= lo) return true;
    if ((float)u16 * 65536.0f >= hi) return false;
  }
  const uint4 c4 = ph_call(K, x, g, t, typ + 8u), c5 = ph_call(K, x, g, t, typ + 10u);
  const uint4 c6 = ph_call(K, x, g, t, typ + 12u), c7 = ph_call(K, x, g, t, typ + 14u);
  const uint32_t u = (u16 << 16) |
                     (lane_byte(c4.x, c4.y, c4.z, c4.w, c5.x, c5.y, c5.z, c5.w, k) << 8) |
                     lane_byte(c6.x, c6.y, c6.z, c6.w, c7.x, c7.y, c7.z, c7.w, k);
  if (!force_exact) {
    if ((double)u < (double)lo) return true;
    if ((double)u >= (double)hi) return false;
  }
  const double h = field_h(1.0, 2 * a - d, q, sig ? 1 : -1, (double)lam);
  return (unsigned long long)u < threshold_T(h, beta);
}

// Per-replica partial values v[0..31] of the 32 lanes of a warp -> lane k holds the
// sum over the warp of v[k] in v[0] (each level halves the values a lane keeps).
template <typename V>
__device__ __forceinline__ V warp_transpose_sum(V (&v)[32], int lane) {
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const bool up = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const V send = up ? v[i] : v[i + s];
      const V keep = up ? v[i + s] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
    }
  }
  return v[0];
}

// Lane k's column of the warp's 32 words (bit i = bit k of lane i's word): five butterfly
// exchanges, as in warp_column_count.
__device__ __forceinline__ uint32_t warp_column(uint32_t x, int lane) {
  const uint32_t Hm[5] = {0xFFFF0000u, 0xFF00FF00u, 0xF0F0F0F0u, 0xCCCCCCCCu, 0xAAAAAAAAu};
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const int j = 16 >> i;
    const uint32_t p = __shfl_xor_sync(0xffffffffu, x, j);
    const bool hi = (lane & j) != 0;
    const uint32_t t = hi ? (p >> j) : (p << j);
    const uint32_t M = hi ? ~Hm[i] : Hm[i];
    x = (x & ~M) | (t & M);
  }
  return x;
}

__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) {
  return (a & b) | (a & c) | (b & c);
}

}  // namespace shk
