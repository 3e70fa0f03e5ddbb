// graph_planes.cuh -- the bit-sliced comparison of the +-1 graph kernels: threshold planes by
// trees of selects over the class index, against the planes of the draws.
#pragma once

#include <cstdint>

#include "graph_device.cuh"
#include "shaken_internal.cuh"

namespace shk {

// 0 or ~0: the sign bit of byte B of t, replicated over the word.
template <int B>
__device__ __forceinline__ uint32_t byte_sign(uint32_t t) {
  uint32_t r;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(t), "n"(0x8888 + 0x1111 * B));
  return r;
}

// Selects leaf idx of 2^NB leaves given by the sign bits of the bytes of tb[0 .. 2^NB / 4),
// for each of W words with idx planes I[b][.].
template <int NB, int W>
__device__ __forceinline__ void mux_tree(const uint32_t* tb, const uint32_t (*I)[W],
                                         uint32_t (&q)[W]) {
  if constexpr (NB == 2) {
    const uint32_t m0 = byte_sign<0>(tb[0]), m1 = byte_sign<1>(tb[0]), m2 = byte_sign<2>(tb[0]),
                   m3 = byte_sign<3>(tb[0]);
#pragma unroll
    for (int j = 0; j < W; ++j) {
      const uint32_t lo = (I[0][j] & m1) | (~I[0][j] & m0);
      const uint32_t hi = (I[0][j] & m3) | (~I[0][j] & m2);
      q[j] = (I[1][j] & hi) | (~I[1][j] & lo);
    }
  } else {
    uint32_t lo[W], hi[W];
    mux_tree<NB - 1, W>(tb, I, lo);
    mux_tree<NB - 1, W>(tb + (1 << NB) / 8, I, hi);
#pragma unroll
    for (int j = 0; j < W; ++j) q[j] = (I[NB - 1][j] & hi[j]) | (~I[NB - 1][j] & lo[j]);
  }
}

constexpr int kIdx = 5;  // planes of a class index (at most 32 classes)

// Planes 4 call + 3 .. 4 call (least significant first) of the draws o against the
// thresholds of vertices with at most 2^NB classes.  The call's class bits are the upper
// (call 1: planes 7..4) or lower four of the bit-reversed bytes.
template <int NB, int W>
__device__ __forceinline__ void sliced_planes(const uint8_t* tbv, int call,
                                              const uint32_t (&I)[kIdx][W], uint32_t (&o)[4][W],
                                              uint32_t (&lt)[W], uint32_t (&eq)[W]) {
  constexpr int NW = (1 << NB) / 4;
  uint32_t tb[NW];
#pragma unroll
  for (int k = 0; k < NW; ++k)
    tb[k] = reinterpret_cast<const uint32_t*>(tbv)[k] << (call != 0 ? 0 : 4);
  auto plane = [&]() {
    uint32_t Q[W];
    mux_tree<NB, W>(tb, I, Q);
#pragma unroll
    for (int k = 0; k < NW; ++k) tb[k] <<= 1;
#pragma unroll
    for (int j = 0; j < W; ++j) {
      lt[j] = maj3(~o[3][j], Q[j], lt[j]);
      eq[j] &= ~(o[3][j] ^ Q[j]);
      o[3][j] = o[2][j];
      o[2][j] = o[1][j];
      o[1][j] = o[0][j];
    }
  };
#pragma unroll 1
  for (int i = 0; i < 4; ++i) plane();  // a loop, for the instruction cache
}

// What a thread knows about its vertex and words.
template <int W>
struct SlicedWord {
  uint32_t x, go, d, slot;  // vertex, first group of the thread within the job, degree, slot
  uint32_t last;            // words of the thread beyond the first
  int p0;
  bool valid, collapse;
  uint32_t F;        // frozen mask
  uint32_t vamb;     // classes of uncertain top byte
  uint32_t h01[W], l01[W];  // Philox: halves of M0 * u0 of the thread's groups
  uint32_t c3base;   // update type
  uint32_t u1;
};

// The Philox call of planes 4 call .. 4 call + 3 for the thread's W groups (counter words
// (x, g, t, typ + 2 call)): x, t and the call are common to the words, so round 0 and
// half of rounds 1 and 2 are computed once (ph_call_shared shares over x instead).
template <int W>
__device__ __forceinline__ void sliced_call(const uint2* key, const SlicedWord<W>& w,
                                            uint32_t c3, uint32_t (&o)[4][W]) {
  const unsigned long long p0 = (unsigned long long)kPhM0 * w.x;
  const unsigned long long p1 =
      (unsigned long long)kPhM1 * ((uint32_t)(p0 >> 32) ^ c3 ^ key[0].y);
  const uint32_t a0 = (uint32_t)(p1 >> 32) ^ w.u1 ^ key[1].x;
  const uint32_t a1 = (uint32_t)p1;
  const unsigned long long q0 = (unsigned long long)kPhM0 * a0;
#pragma unroll
  for (int j = 0; j < W; ++j) {
    const uint32_t c2 = w.h01[j] ^ (uint32_t)p0 ^ key[1].y;
    const unsigned long long q1 = (unsigned long long)kPhM1 * c2;
    o[0][j] = (uint32_t)(q1 >> 32) ^ a1 ^ key[2].x;
    o[1][j] = (uint32_t)q1;
    o[2][j] = (uint32_t)(q0 >> 32) ^ w.l01[j] ^ key[2].y;
    o[3][j] = (uint32_t)q0;
  }
#pragma unroll
  for (int r = 3; r < 10; ++r) {
    const uint2 k = key[r];
#pragma unroll
    for (int j = 0; j < W; ++j) {
      const unsigned long long s0 = (unsigned long long)kPhM0 * o[0][j];
      const unsigned long long s1 = (unsigned long long)kPhM1 * o[2][j];
      o[0][j] = (uint32_t)(s1 >> 32) ^ o[1][j] ^ k.x;
      o[2][j] = (uint32_t)(s0 >> 32) ^ o[3][j] ^ k.y;
      o[1][j] = (uint32_t)s1;
      o[3][j] = (uint32_t)s0;
    }
  }
}

// Class i of a vertex of degree d and field lam (collapsed, q = 1: i = a + [sigma = +1], else
// 2 a + [sigma = +1]) at kb = -2 beta log2(e): its top byte into tbv[i] (bit-reversed);
// 1 if the bounds do not fix it.  qint: q is an integer.
__device__ __forceinline__ uint32_t sliced_class(double q, bool collapse, bool qint, float kb,
                                                 uint32_t i, uint32_t d, float lam, uint8_t* tbv) {
  const uint32_t a = collapse ? i : i >> 1;
  const bool up = !collapse && (i & 1u) != 0u;
  const float qf = (float)q, fd = (float)d;
  const float h0 = __fadd_rn(__fadd_rn(lam, -fd), up ? qf : -qf);  // h = 2a + (lambda - d +- q)
  const float hf = fmaf(2.0f, (float)a, h0);
  float lo, hi;
  t_bounds(hf, kb, fabsf(kb) * (fd + fabsf(qf) + fabsf(lam) + 1.0f), lo, hi);
  uint32_t bl = top_byte(lo), bh = top_byte(hi);
  // a field of exactly 0 has T = 2^31; with lambda = 0 and an integer q the fp32 field is
  // exact
  if (hf == 0.0f && (lam == 0.0f ? qint : field_is_zero(2 * (int)a - (int)d, up, q, lam)))
    bl = bh = 0x80u;
  tbv[i] = (uint8_t)(__brev(bh) >> 24);
  return bl != bh ? 1u : 0u;
}

// The lane of a queue entry (word (x, g), lane k, class idx of a vertex of degree d and field
// lam; byte: its draw's top byte, or amb: not known yet) decided: +1?
__device__ __forceinline__ bool sliced_lane(uint32_t key0, uint32_t key1, uint32_t x, uint32_t g,
                                            uint32_t t, uint32_t typ, double q, bool collapse,
                                            float kb, double beta, int d, float lam, int k,
                                            uint32_t idx, uint32_t byte, bool amb) {
  const int a = (int)(collapse ? idx : idx >> 1), sig = collapse ? 0 : (int)(idx & 1u);
  const float qf = (float)q, lmd = __fadd_rn(lam, -(float)d);
  const float bp = __fadd_rn(lmd, qf), bm = __fadd_rn(lmd, -qf);
  const float B = (float)d + fabsf(qf) + fabsf(lam) + 1.0f;
  uint32_t u8 = byte;
  if (amb) {  // class of uncertain top byte: the draw's own
    const PhKey K = ph_key(key0, key1);
    const uint4 c0 = ph_call(K, x, g, t, typ), c1 = ph_call(K, x, g, t, typ + 2u);
    u8 = lane_byte(c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w, k);
  }
  return decide_lane(key0, key1, x, g, t, typ, k, u8, a, d, sig, bp, bm, q, lam, kb,
                     fabsf(kb) * B, beta, false);
}

}  // namespace shk
