// lattice_device.cuh -- device code shared by the lattice kernels: the bit-plane decision of a
// lane word, the byte / bit conversions and the neighbour loads.
#pragma once

#include <cstdint>

#include "shaken_internal.cuh"

namespace shk {

// --------------------------------------------------------------------------- decision core
// Field classes of a lane word.  S = sigma_x bits, V / H = the two in-neighbour
// bits (vertical / horizontal); x = V ^ H marks one +1 neighbour (n = 1), and
// where V == H the class is n = 0 (V = 0) or n = 2 (V = 1).
struct LaneWord {
  uint32_t S, V, X, U, res;  // U = lanes still undecided
};

// One plane of a threshold table, read from shared memory once and applied to
// every lane word of the thread.
struct PlaneRow {
  uint4 lo;  // classes 0..3 (collapsed: c = 0..3)
  uint2 hi;  // classes 4, 5 (unused when collapsed)
};

template <bool COLL>
__device__ __forceinline__ PlaneRow plane_row(const LatTable& tab, int j) {
  PlaneRow r;
  if (COLL) {
    r.lo = *reinterpret_cast<const uint4*>(&tab.tmc[j][0]);
    r.hi = make_uint2(0u, 0u);
  } else {
    r.lo = *reinterpret_cast<const uint4*>(&tab.tm[j][0]);
    r.hi = *reinterpret_cast<const uint2*>(&tab.tm[j][4]);
  }
  return r;
}

// Threshold bit of plane j for every lane: first select by sigma within each
// n-class, then by n: 5 three-input selects.
// Collapsed tables (thresholds by c = n + s): with c0 = parity and c1 =
// majority of (V, H, S), c = c0 + 2 c1 and the plane bit is 3 selects; there
// L.V holds c1 and L.X holds c0.
template <bool COLL>
__device__ __forceinline__ uint32_t plane_bits(const LaneWord& L, const PlaneRow& r) {
  if (COLL) {
    const uint32_t lo = (L.X & r.lo.y) | (~L.X & r.lo.x);  // c1 = 0
    const uint32_t hi = (L.X & r.lo.w) | (~L.X & r.lo.z);  // c1 = 1
    return (L.V & hi) | (~L.V & lo);
  }
  const uint32_t b0 = (L.S & r.lo.y) | (~L.S & r.lo.x);  // n = 0
  const uint32_t b1 = (L.S & r.lo.w) | (~L.S & r.lo.z);  // n = 1
  const uint32_t b2 = (L.S & r.hi.y) | (~L.S & r.hi.x);  // n = 2
  const uint32_t m = (L.V & b2) | (~L.V & b0);           // V == H
  return (L.X & b1) | (~L.X & m);
}

// MSB-first comparison of u_k with T_k over the four planes of one Philox call.
template <bool COLL>
__device__ __forceinline__ void apply_call(LaneWord& L, const uint4 w, const LatTable& tab,
                                           uint32_t call) {
  const uint32_t Wj[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t P = plane_bits<COLL>(L, plane_row<COLL>(tab, 4 * call + i));
    const uint32_t diff = (Wj[i] ^ P) & L.U;  // first plane where u and T differ
    L.res |= diff & P;                        // T has the 1 there: u < T
    L.U &= ~diff;
  }
}

// Initial classification: frozen lanes and saturated thresholds (T = 0 or 2^32)
// are decided before any draw.  For collapsed tables V and X are replaced by
// the majority and the parity of (V, H, S).
template <bool COLL>
__device__ __forceinline__ LaneWord classify(uint32_t S, uint32_t V, uint32_t H, uint32_t F,
                                             const LatTable& tab) {
  LaneWord L;
  L.S = S;
  L.V = V;
  L.X = V ^ H;
  uint32_t dec = F, res = F;
  if (tab.anysat) {
    const uint32_t n2 = V & H, n0 = ~(V | H), n1 = L.X;
    const uint32_t M[6] = {n0 & ~S, n0 & S, n1 & ~S, n1 & S, n2 & ~S, n2 & S};
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      dec |= M[c] & (tab.satp[c] | tab.satm[c]);
      res |= M[c] & tab.satp[c];
    }
  }
  if (COLL) {
    L.V = (V & H) | (S & (V | H));  // majority
    L.X = V ^ H ^ S;                // parity
  }
  L.U = ~dec;
  L.res = res;
  return L;
}

// Calls 0, 1 and 2 (planes 31..20) of a lane word, made unconditionally (the
// resident small-lattice kernel, where a half step is a dependent chain and the
// warp needs call 2 for some word about 98% of the time anyway): the three
// Philox calls are independent and overlap.  A lane is decided by its first
// differing plane, as call by call; after the twelve planes a lane is undecided
// with probability 2^-12.
template <bool COLL>
__device__ __forceinline__ void decide_head3(LaneWord& L, const LatTable& tab, const PhKey& K,
                                             const PhShared& P, uint32_t a, uint32_t half,
                                             uint32_t& calls) {
  const uint4 w0 = ph_call_shared(K, P, a, half);
  const uint4 w1 = ph_call_shared(K, P, a, half + 2u);
  const uint4 w2 = ph_call_shared(K, P, a, half + 4u);
  calls += 3;
  // the top twelve bits of u and T compared as a subtraction, least significant
  // plane first (borrow lt, equality eq): two short independent chains
  uint32_t lt = 0u, eq = 0xffffffffu;
#pragma unroll
  for (int j = 11; j >= 0; --j) {
    const uint4 Wc = j >= 8 ? w2 : j >= 4 ? w1 : w0;
    const int i = j & 3;
    const uint32_t w = i == 0 ? Wc.x : i == 1 ? Wc.y : i == 2 ? Wc.z : Wc.w;
    const uint32_t Pj = plane_bits<COLL>(L, plane_row<COLL>(tab, j));
    lt = (~w & Pj) | (~w & lt) | (Pj & lt);
    eq &= ~(w ^ Pj);
  }
  L.res |= L.U & ~eq & lt;
  L.U &= eq;
}

// The same comparison from calls made before (lattice_cluster_kernel).  Not the body of
// decide_head3: with the calls in an array the whole-run kernel took 8 % longer.
template <bool COLL>
__device__ __forceinline__ void decide_planes3(LaneWord& L, const LatTable& tab,
                                               const uint4 (&W)[3]) {
  // the top twelve bits of u and T compared as a subtraction, least significant
  // plane first (borrow lt, equality eq): two short independent chains
  uint32_t lt = 0u, eq = 0xffffffffu;
#pragma unroll
  for (int j = 11; j >= 0; --j) {
    const uint4 Wc = W[j >> 2];
    const int i = j & 3;
    const uint32_t w = i == 0 ? Wc.x : i == 1 ? Wc.y : i == 2 ? Wc.z : Wc.w;
    const uint32_t Pj = plane_bits<COLL>(L, plane_row<COLL>(tab, j));
    lt = (~w & Pj) | (~w & lt) | (Pj & lt);
    eq &= ~(w ^ Pj);
  }
  L.res |= L.U & ~eq & lt;
  L.U &= eq;
}

// Planes 31..24 (calls 0 and 1) of the thread's WPT lane words, plane-major:
// every table row is read once for all the words, and the WPT Philox calls of
// a group are independent of one another.  The top eight bits of u_k and T_k
// are compared as an eight-bit subtraction, least significant plane first:
// the borrow lt <- maj(~w, P, lt) ends as [u_top < T_top] and eq as
// [u_top == T_top].  Lanes with equal top bits stay undecided for planes 23..0
// (the warp queue of the tiled kernel, or decide_tail); the others are decided
// exactly as by the first differing plane.
// Four planes of one call (planes 4c+3 .. 4c, least significant first) for
// the WPT words: one step of the borrow chain per plane.
template <bool COLL, int WPT>
__device__ __forceinline__ void head_planes(const LaneWord (&Lw)[WPT], const LatTable& tab,
                                            int call, const uint4 (&W)[WPT], uint32_t (&lt)[WPT],
                                            uint32_t (&eq)[WPT]) {
#pragma unroll
  for (int i = 3; i >= 0; --i) {
    const PlaneRow r = plane_row<COLL>(tab, 4 * call + i);
#pragma unroll
    for (int k = 0; k < WPT; ++k) {
      const uint32_t w = i == 0 ? W[k].x : i == 1 ? W[k].y : i == 2 ? W[k].z : W[k].w;
      const uint32_t P = plane_bits<COLL>(Lw[k], r);
      lt[k] = (~w & P) | (~w & lt[k]) | (P & lt[k]);
      eq[k] &= ~(w ^ P);
    }
  }
}

// The same four planes for mirror tables: with c1 = majority (L.V) and c0 =
// parity (L.X), the class c = c0 + 2 c1 has field h > 0 exactly when c1 = 1, and
// |h| is the larger value when c0 == c1.  The plane is the T(|h|) plane picked by
// sel = ~(c0 ^ c1) from the rows of c = 2 and c = 3, complemented on the lanes
// with h < 0: two logic operations instead of three selects.
template <int WPT>
__device__ __forceinline__ void head_planes_mirror(const LaneWord (&Lw)[WPT],
                                                   const uint32_t (&sel)[WPT],
                                                   const LatTable& tab, int call,
                                                   const uint4 (&W)[WPT], uint32_t (&lt)[WPT],
                                                   uint32_t (&eq)[WPT]) {
#pragma unroll
  for (int i = 3; i >= 0; --i) {
    const uint2 r = *reinterpret_cast<const uint2*>(&tab.tmc[4 * call + i][2]);
#pragma unroll
    for (int k = 0; k < WPT; ++k) {
      const uint32_t w = i == 0 ? W[k].x : i == 1 ? W[k].y : i == 2 ? W[k].z : W[k].w;
      const uint32_t Q = (sel[k] & r.y) | (~sel[k] & r.x);
      const uint32_t P = ~(Q ^ Lw[k].V);
      lt[k] = (~w & P) | (~w & lt[k]) | (P & lt[k]);
      eq[k] &= ~(w ^ P);
    }
  }
}

template <int WPT>
__device__ __forceinline__ void head_finish(LaneWord (&Lw)[WPT], const uint32_t (&lt)[WPT],
                                            const uint32_t (&eq)[WPT]) {
#pragma unroll
  for (int k = 0; k < WPT; ++k) {
    Lw[k].res |= Lw[k].U & ~eq[k] & lt[k];
    Lw[k].U &= eq[k];
  }
}

// MIR: the table is a mirror table (collapsed, `mirror` set).
template <bool COLL, int WPT, bool MIR = false>
__device__ __forceinline__ void decide_head_words(LaneWord (&Lw)[WPT], const LatTable& tab,
                                                  const PhKey& K, const PhShared& P,
                                                  const uint32_t (&a)[WPT], uint32_t half) {
  uint32_t lt[WPT], eq[WPT], sel[WPT];
#pragma unroll
  for (int k = 0; k < WPT; ++k) {
    lt[k] = 0u;
    eq[k] = 0xffffffffu;
    sel[k] = MIR ? ~(Lw[k].X ^ Lw[k].V) : 0u;
  }
#pragma unroll
  for (int call = 1; call >= 0; --call) {
    uint4 W[WPT];
#pragma unroll
    for (int k = 0; k < WPT; ++k) W[k] = ph_call_shared(K, P, a[k], half + 2u * (uint32_t)call);
    if (MIR)
      head_planes_mirror<WPT>(Lw, sel, tab, call, W, lt, eq);
    else
      head_planes<COLL, WPT>(Lw, tab, call, W, lt, eq);
  }
  head_finish<WPT>(Lw, lt, eq);
}

// Calls first..7 while some lane is undecided (one word at a time: the resident
// small-lattice kernel).
template <bool COLL>
__device__ __forceinline__ void decide_tail(LaneWord& L, const LatTable& tab, const PhKey& K,
                                            const PhShared& P, uint32_t a, uint32_t half,
                                            uint32_t first) {
#pragma unroll 1
  for (uint32_t call = first; call < 8 && L.U != 0u; ++call) {
    const uint4 w = ph_call_shared(K, P, a, half + 2u * call);
    apply_call<COLL>(L, w, tab, call);
  }
}

// --------------------------------------------------------------------------- int8 <-> bits
// +1 = 0x01, -1 = 0xFF: the sign bit of a byte is clear for +1.
// Eight bytes (w0: sites 0..3, w1: sites 4..7, memory order) -> bits 24..31 of the
// result (bit 24 + j = site j is +1): the clear sign bits go to bits 0, 8, 16, 24
// (w0) and 4, 12, 20, 28 (w1), and one multiply by 2^24 + 2^17 + 2^10 + 2^3 moves
// byte k of w0 to bit 24 + k and byte k of w1 to bit 28 + k; every other partial
// product lands below bit 24 at a distinct position or above bit 31, so nothing
// carries into the top byte.
__device__ __forceinline__ uint32_t bits8_top(uint32_t w0, uint32_t w1) {
  const uint32_t m = ((~w0 >> 7) & 0x01010101u) | ((~w1 >> 3) & 0x10101010u);
  return m * 0x01020408u;
}
// 32 bytes (sites 0..15 in a, 16..31 in b) -> 32 bits, bit j = site j is +1.
__device__ __forceinline__ uint32_t bits32(uint4 a, uint4 b) {
  const uint32_t lo = __byte_perm(bits8_top(a.x, a.y), bits8_top(a.z, a.w), 0x0073u);
  const uint32_t hi = __byte_perm(bits8_top(b.x, b.y), bits8_top(b.z, b.w), 0x0073u);
  return __byte_perm(lo, hi, 0x5410u);
}
// 4 bits -> 4 bytes of +1/-1: bit k -> byte k (0 or 1), then 0xFF - 0xFE t per byte
// (no byte borrows from its neighbour)
__device__ __forceinline__ uint32_t bytes4(uint32_t b) {
  const uint32_t t = ((b & 0xFu) * 0x00204081u) & 0x01010101u;
  return 0xFFFFFFFFu - 0xFEu * t;
}
__device__ __forceinline__ uint4 bytes16(uint32_t b) {
  return make_uint4(bytes4(b), bytes4(b >> 4), bytes4(b >> 8), bytes4(b >> 12));
}

enum { kEncInt8 = 0, kEncPacked = 1, kEncMultispin = 2 };

// Lane-word coordinates: row i and word column c of lane word w.
__device__ __forceinline__ void word_rc(const LatJob& J, uint32_t w, uint32_t& i, uint32_t& c) {
  if (J.wpr_shift != 0xffffffffu) {
    i = w >> J.wpr_shift;
    c = w & (J.wpr - 1u);
  } else {
    i = w / J.wpr;
    c = w - i * J.wpr;
  }
}

// Loads the three lane words a decision needs from buffer src: S (own), V (the
// vertical in-neighbour row: i-1 for half 0, i+1 for half 1) and H (the
// horizontal in-neighbour: j-1 for half 0, j+1 for half 1).
// NC: buf is a global buffer not written during the launch (read through the
// non-coherent cache); otherwise a plain load (shared memory).
template <bool NC, typename T>
__device__ __forceinline__ T ld_ro(const T* p) {
  if (NC) return __ldg(p);
  return *p;
}

template <int ENC, bool NC = true>
__device__ __forceinline__ void load_lane_words(const LatJob& J, const void* buf, uint32_t w,
                                                uint32_t half, uint32_t& S, uint32_t& V,
                                                uint32_t& H) {
  const uint32_t L = J.L, wpr = J.wpr;
  if (ENC != kEncInt8 && J.wpr_shift != 0xffffffffu) {
    // power-of-two rows (then L * wpr is one too): the neighbour words by masks --
    // the vertical one wpr words away modulo the lattice, the horizontal one the
    // next word of the same row, cyclically
    const uint32_t* A = static_cast<const uint32_t*>(buf);
    const uint32_t rowmask = wpr - 1u, allmask = J.nwords - 1u;
    const uint32_t dv = half == 0u ? 0u - wpr : wpr;
    const uint32_t dh = half == 0u ? 0xffffffffu : 1u;
    S = ld_ro<NC>(A + w);
    V = ld_ro<NC>(A + ((w + dv) & allmask));
    const uint32_t hn = ld_ro<NC>(A + ((w & ~rowmask) | ((w + dh) & rowmask)));
    if (ENC == kEncPacked)
      H = half == 0u ? ((S << 1) | (hn >> 31)) : ((S >> 1) | (hn << 31));
    else
      H = hn;
    return;
  }
  uint32_t i, c;
  word_rc(J, w, i, c);
  const uint32_t iv = half == 0u ? (i == 0u ? L - 1u : i - 1u) : (i + 1u == L ? 0u : i + 1u);
  if (ENC == kEncInt8) {
    const uint8_t* A = static_cast<const uint8_t*>(buf);
    const uint4* own = reinterpret_cast<const uint4*>(A + (size_t)i * L + 32u * c);
    const uint4* ver = reinterpret_cast<const uint4*>(A + (size_t)iv * L + 32u * c);
    const uint4 o0 = ld_ro<NC>(own), o1 = ld_ro<NC>(own + 1), v0 = ld_ro<NC>(ver),
                v1 = ld_ro<NC>(ver + 1);
    const uint32_t jn = half == 0u ? (c == 0u ? L - 1u : 32u * c - 1u)
                                   : (32u * c + 32u == L ? 0u : 32u * c + 32u);
    const uint32_t nb = (ld_ro<NC>(A + (size_t)i * L + jn) >> 7) ^ 1u;  // 1 if +1
    S = bits32(o0, o1);
    V = bits32(v0, v1);
    H = half == 0u ? ((S << 1) | nb) : ((S >> 1) | (nb << 31));
  } else if (ENC == kEncPacked) {
    const uint32_t* A = static_cast<const uint32_t*>(buf);
    S = ld_ro<NC>(A + (size_t)i * wpr + c);
    V = ld_ro<NC>(A + (size_t)iv * wpr + c);
    if (half == 0u) {
      const uint32_t cl = c == 0u ? wpr - 1u : c - 1u;
      H = (S << 1) | (ld_ro<NC>(A + (size_t)i * wpr + cl) >> 31);
    } else {
      const uint32_t cr = c + 1u == wpr ? 0u : c + 1u;
      H = (S >> 1) | (ld_ro<NC>(A + (size_t)i * wpr + cr) << 31);
    }
  } else {
    const uint32_t* A = static_cast<const uint32_t*>(buf);
    const uint32_t jn = half == 0u ? (c == 0u ? L - 1u : c - 1u) : (c + 1u == L ? 0u : c + 1u);
    S = ld_ro<NC>(A + w);
    V = ld_ro<NC>(A + (size_t)iv * L + c);
    H = ld_ro<NC>(A + (size_t)i * L + jn);
  }
}

template <int ENC>
__device__ __forceinline__ uint32_t resident_load(const LatJob& J, uint32_t w) {
  if (ENC == kEncInt8) {
    uint32_t i, c;
    word_rc(J, w, i, c);
    const uint4* p = reinterpret_cast<const uint4*>(static_cast<const uint8_t*>(J.A) +
                                                    (size_t)i * J.L + 32u * c);
    return bits32(p[0], p[1]);
  }
  return static_cast<const uint32_t*>(J.A)[w];
}

template <int ENC>
__device__ __forceinline__ void resident_store(const LatJob& J, void* buf, uint32_t w,
                                               uint32_t bits) {
  if (ENC == kEncInt8) {
    uint32_t i, c;
    word_rc(J, w, i, c);
    uint4* p = reinterpret_cast<uint4*>(static_cast<uint8_t*>(buf) + (size_t)i * J.L + 32u * c);
    p[0] = bytes16(bits);
    p[1] = bytes16(bits >> 16);
  } else {
    static_cast<uint32_t*>(buf)[w] = bits;
  }
}

}  // namespace shk
