// graph_sliced.cu -- half steps of +-1 graphs at one inverse temperature (anneals, uniform
// beta), bit-sliced: the 32 replicas of a word are never taken apart.
//
// A vertex x of degree d has at most 32 classes of lanes: with a = number of
// neighbours with J_xy s_y = +1, the threshold T depends on the lane only through
// idx = a + [sigma = +1] (q = 1, where h(a, +1) = h(a + 1, -1) exactly) or idx = 2 a +
// [sigma = +1].  One thread owns W group words of a vertex (adjacent in memory).  It
//   * counts a in bit planes (full adders over the neighbour words, four edges at a
//     time): 3-4 logic operations per edge and word;
//   * for each of the top eight threshold planes, selects the class's bit with a tree of
//     three-input selects over the planes of idx, whose leaves are 0 / ~0 masks taken
//     from the vertex's class bytes (PRMT with sign replication, shared by the W words);
//   * compares with the draw's planes least significant first: e = ~(w ^ Q),
//     lt = e ? lt : Q, eq &= e.
// Lanes whose top byte equals the threshold's (2^-8), or whose class byte the fp32 bounds
// do not fix, go one by one to a per-warp queue decided 32 at a time (decide_lane).
//
// What bounds it: integer issue.  A LOP3, a PRMT and a wide product each hold the SM
// quarter's common issue port for two cycles (a product and k logic operations take
// max(4, 2 + 2k) cycles), so a word of the Erdos-Renyi graph (mean degree 8, n = 10^6,
// 256 replicas) with its ~300 such operations needs 600 cycles: a bound of 120 us a half
// step, measured 178 us (ALU pipe 56 %, issue 51 %, 1720 warp instructions per
// 4-word thread, next: gathers).  The general kernel's byte counters, byte lookups and
// bit transposes take 907 instructions a word and 370 us; with tracking 238 against
// 412 us.  Four words a thread (16 warps an SM at 128 registers) against two (20 warps):
// 10.1 against 11.7 ms for 20 tracked steps; against four at 20 warps: 10.6 ms.
#include <atomic>
#include <cstdint>

#include "graph_planes.cuh"
#include "shaken_internal.cuh"

namespace shk {

static_assert(kSlicedTile == 128, "four threads per degree 0 .. 31 build the class bytes");
constexpr int kSlicedQueue = 96;  // queue entries per warp (31 waiting and two per lane)
constexpr int kSlicedCnt = 10;     // planes of the tracking counters (flushed before 1023)
constexpr int kSlicedTot = 64;     // groups of a job whose totals a block keeps

struct SlicedShared {
  // top bytes of T by class, bit-reversed: with one lambda for all vertices by degree, else
  // by [warp][vertex] of the current tile
  __align__(16) uint8_t tb[kSlicedTile / 32][32][32];
  uint32_t amb[32];  // classes of uncertain top byte by degree (one lambda)
  uint2 key[10];     // Philox round keys
  uint4 col[kSlicedTile];  // the first four columns of each thread's vertex in the next tile
  GraphJob J;
  const uint32_t* src;
  uint32_t* dst;
  uint32_t t, typ, skip, fuse, qint, collapse, by_degree;
  float kb;
  double beta;
  unsigned long long dsum;  // degrees of the block's vertices of this job (tracking)
  uint2 q[kSlicedTile / 32][kSlicedQueue];
};

template <int W>
struct SlicedTrack {
  uint32_t cnt[kSlicedCnt][kSlicedTile][W];       // bit planes of each thread's agreeing-edge counts
  unsigned int tot[kSlicedTot][32];         // block totals [group of the job][replica lane]
};

template <int W>
struct alignas(W == 3 ? 4 : 4 * W) Words {
  uint32_t v[W];
};

// The W words from p on: one vector load where rows are a multiple of W words, else words
// p[min(j, last)] (a row's last thread may have fewer words: the last one again).
template <int W, bool VEC>
__device__ __forceinline__ Words<W> ld_words(const uint32_t* p, uint32_t last) {
  Words<W> r;
  if constexpr (VEC && W == 4) {
    const uint4 u = __ldg(reinterpret_cast<const uint4*>(p));
    r.v[0] = u.x; r.v[1] = u.y; r.v[2] = u.z; r.v[3] = u.w;
  } else if constexpr (VEC && W == 2) {
    const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
    r.v[0] = u.x; r.v[1] = u.y;
  } else if constexpr (W == 1) {
    r.v[0] = __ldg(p);
  } else {
#pragma unroll
    for (uint32_t j = 0; j < W; ++j) r.v[j] = __ldg(p + min(j, last));
  }
  return r;
}

template <int W, bool VEC>
__device__ __forceinline__ void st_words(uint32_t* p, uint32_t last, const uint32_t (&v)[W]) {
  if constexpr (VEC && W == 4) {
    *reinterpret_cast<uint4*>(p) = make_uint4(v[0], v[1], v[2], v[3]);
  } else if constexpr (VEC && W == 2) {
    *reinterpret_cast<uint2*>(p) = make_uint2(v[0], v[1]);
  } else {
#pragma unroll
    for (uint32_t j = 0; j < W; ++j)
      if (j <= last) p[j] = v[j];
  }
}

// Up to 32 entries of the warp's queue: lane i decides entry i (i < cnt) and sets its bit in
// the stored word if it is +1.  Entry: (slot, k | idx << 5 | go << 10 | byte << 18 | amb << 26).
__device__ __noinline__ void sliced_round(const SlicedShared& sh, const uint2* q, int cnt,
                                             int lane) {
  __syncwarp();
  if (lane < cnt) {
    const uint2 e = q[lane];
    const GraphJob& J = sh.J;
    const uint4 vi = __ldg((sh.typ == 0u ? J.in_visit : J.out_visit) + e.x);
    const int k = (int)(e.y & 31u);
    const uint32_t idx = (e.y >> 5) & 31u, g = J.g0 + ((e.y >> 10) & 255u);
    if (sliced_lane(J.key0, J.key1, vi.x, g, sh.t, sh.typ, J.q, sh.collapse != 0u, sh.kb, sh.beta,
                    (int)vi.z, __uint_as_float(vi.w), k, idx, (e.y >> 18) & 0xFFu,
                    ((e.y >> 26) & 1u) != 0u))
      atomicOr(sh.dst + (size_t)vi.x * J.G + g, 1u << k);
  }
  __syncwarp();
}

// Decisions of the warp's vertices (one tile row); ncls: the most classes among them.
// Only the plane comparison is compiled once per class width, the rest of the body is
// common: four whole bodies (119 KB) missed the instruction cache for a third of the stalls.
template <int W, bool VEC, bool TRACK>
__device__ __forceinline__ void sliced_decide(SlicedShared& sh, SlicedTrack<W>* tr,
                                              const SlicedWord<W>& w, const uint8_t* tbv,
                                              uint32_t ncls, bool have, const uint4* next,
                                              uint2* q, int& qn, int lane) {
  const GraphJob& J = sh.J;
  const uint32_t G = J.G;
  const uint32_t* src = sh.src + J.g0 + w.go;
  const uint32_t* col = w.c3base == 0u ? J.in_col : J.out_col;
  uint32_t I[kIdx][W], S[W];
#pragma unroll
  for (int j = 0; j < W; ++j) {
    S[j] = 0u;
#pragma unroll
    for (int b = 0; b < kIdx; ++b) I[b][j] = 0u;
  }
  if (w.valid) {
    const Words<W> own = ld_words<W, VEC>(src + (size_t)w.x * G, w.last);
#pragma unroll
    for (int j = 0; j < W; ++j) S[j] = own.v[j];
    uint32_t cv[4];  // four edges at a time; beyond the degree the last edge again, masked out
    if (have) {      // copied during the previous tile
      asm volatile("cp.async.wait_all;" ::: "memory");
      const uint4 c = sh.col[threadIdx.x];
      cv[0] = c.x; cv[1] = c.y; cv[2] = c.z; cv[3] = c.w;
    } else if (w.d != 0u) {
#pragma unroll
      for (uint32_t i = 0; i < 4; ++i) cv[i] = __ldg(col + w.p0 + min(i, w.d - 1u));
    }
#pragma unroll 1
    for (uint32_t e = 0; e < w.d; e += 4) {
      uint32_t x[4][W];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const Words<W> nb = ld_words<W, VEC>(src + (size_t)(cv[i] & 0x7fffffffu) * G, w.last);
        const uint32_t s = (uint32_t)((int32_t)cv[i] >> 31);  // J < 0
        const uint32_t m = e + i < w.d ? 0xffffffffu : 0u;
#pragma unroll
        for (int j = 0; j < W; ++j) x[i][j] = (nb.v[j] ^ s) & m;
      }
      if (e + 4u < w.d) {
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i) cv[i] = __ldg(col + w.p0 + min(e + 4u + i, w.d - 1u));
      }
      uint32_t c[W];
#pragma unroll
      for (int j = 0; j < W; ++j) {
        const uint32_t s0 = I[0][j] ^ x[0][j] ^ x[1][j], ca = maj3(I[0][j], x[0][j], x[1][j]);
        const uint32_t cb = maj3(s0, x[2][j], x[3][j]);
        I[0][j] = s0 ^ x[2][j] ^ x[3][j];
        const uint32_t cc = maj3(I[1][j], ca, cb);
        I[1][j] ^= ca ^ cb;
        c[j] = I[2][j] & cc;
        I[2][j] ^= cc;
      }
      if (ncls > 8u) {  // counts beyond three planes
#pragma unroll
        for (int j = 0; j < W; ++j) {
          I[4][j] ^= I[3][j] & c[j];
          I[3][j] ^= c[j];
        }
      }
    }
  }
  if (next != nullptr && next->z != 0u) {  // the next tile's columns, on their way during the rest
    const uint32_t at = (uint32_t)__cvta_generic_to_shared(&sh.col[threadIdx.x]);
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(at + 4u * i),
                   "l"(col + next->y + min(i, next->z - 1u))
                   : "memory");
  }
  if (TRACK && sh.fuse) {
    // agreeing edges (J_xy s_x s_y = +1) per lane: a where sigma = +1, d - a otherwise,
    // added to the thread's counter planes
    const uint32_t dd = w.valid ? w.d : 0u;
    uint32_t br[W], carry[W];
#pragma unroll
    for (int j = 0; j < W; ++j) br[j] = carry[j] = 0u;
#pragma unroll
    for (int b = 0; b < kIdx; ++b) {
      const uint32_t D = 0u - ((dd >> b) & 1u);
      Words<W>& cw = *reinterpret_cast<Words<W>*>(tr->cnt[b][threadIdx.x]);
      Words<W> c = cw;
#pragma unroll
      for (int j = 0; j < W; ++j) {
        const uint32_t A = I[b][j], df = D ^ A ^ br[j], old = c.v[j];
        br[j] = (~D & A) | (~D & br[j]) | (A & br[j]);
        const uint32_t ag = (S[j] & A) | (~S[j] & df);
        c.v[j] = old ^ ag ^ carry[j];
        carry[j] = maj3(old, ag, carry[j]);
      }
      cw = c;
    }
#pragma unroll 1
    for (int b = kIdx; b < kSlicedCnt; ++b) {
      Words<W>& cw = *reinterpret_cast<Words<W>*>(tr->cnt[b][threadIdx.x]);
      Words<W> c = cw;
      uint32_t any = 0u;
#pragma unroll
      for (int j = 0; j < W; ++j) {
        const uint32_t old = c.v[j];
        c.v[j] = old ^ carry[j];
        carry[j] &= old;
        any |= carry[j];
      }
      cw = c;
      if (any == 0u) break;
    }
  }
  if (w.collapse) {  // idx = a + sigma
#pragma unroll
    for (int j = 0; j < W; ++j) {
      uint32_t c = S[j];
#pragma unroll
      for (int b = 0; b < kIdx; ++b) {
        const uint32_t t = I[b][j] & c;
        I[b][j] ^= c;
        c = t;
      }
    }
  } else {  // idx = 2 a + sigma
#pragma unroll
    for (int j = 0; j < W; ++j) {
#pragma unroll
      for (int b = kIdx - 1; b > 0; --b) I[b][j] = I[b - 1][j];
      I[0][j] = S[j];
    }
  }
  uint32_t lt[W], eq[W];
#pragma unroll
  for (int j = 0; j < W; ++j) {
    lt[j] = 0u;
    eq[j] = ~w.F;
  }
#pragma unroll 1
  for (int call = 1; call >= 0; --call) {
    uint32_t o[4][W];
    sliced_call<W>(sh.key, w, w.c3base + 2u * (uint32_t)call, o);
    if (ncls <= 4u)
      sliced_planes<2, W>(tbv, call, I, o, lt, eq);
    else if (ncls <= 8u)
      sliced_planes<3, W>(tbv, call, I, o, lt, eq);
    else if (ncls <= 16u)
      sliced_planes<4, W>(tbv, call, I, o, lt, eq);
    else
      sliced_planes<5, W>(tbv, call, I, o, lt, eq);
  }
  uint32_t cu = 0u;  // lanes left to the queue
#pragma unroll
  for (int j = 0; j < W; ++j) {
    uint32_t amb = 0u;
#pragma unroll 1
    for (uint32_t m = w.vamb; m != 0u; m &= m - 1u) {  // rare: lanes of uncertain classes
      const uint32_t c = (uint32_t)__ffs(m) - 1u;
      uint32_t is = 0xffffffffu;
#pragma unroll
      for (int b = 0; b < kIdx; ++b) is &= ~(I[b][j] ^ (0u - ((c >> b) & 1u)));
      amb |= is;
    }
    eq[j] = w.valid && (VEC || (uint32_t)j <= w.last) ? (eq[j] | amb) & ~w.F : 0u;  // undecided
    lt[j] = (lt[j] & ~eq[j]) | w.F;
    cu += (uint32_t)__popc(eq[j]);
  }
  if (w.valid) st_words<W, VEC>(sh.dst + J.g0 + w.go + (size_t)w.x * G, w.last, lt);
  if (!__any_sync(0xffffffffu, cu != 0u)) return;
  // queue entries of the undecided lanes
  const uint32_t below = (1u << lane) - 1u;
  auto entry = [&](int j, int k) {
    uint32_t idx = 0u;
#pragma unroll
    for (int b = 0; b < kIdx; ++b) idx |= ((I[b][j] >> k) & 1u) << b;
    return make_uint2(w.slot, (uint32_t)k | (idx << 5) | ((w.go + (uint32_t)j) << 10) |
                                  ((__brev((uint32_t)tbv[idx]) >> 24) << 18) |
                                  (((w.vamb >> idx) & 1u) << 26));
  };
  // places by a prefix sum over the lanes' counts: all of them when they fit, else at most
  // two of each lane at a time; a round whenever 32 wait
#pragma unroll 1
  do {
    uint32_t c = min(cu, 7u), pos, total;
    auto places = [&]() {
      pos = (uint32_t)qn;
      total = 0u;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const uint32_t m = __ballot_sync(0xffffffffu, (c >> b) & 1u);
        pos += (uint32_t)__popc(m & below) << b;
        total += (uint32_t)__popc(m) << b;
      }
    };
    places();
    if (qn + (int)total > kSlicedQueue) {  // uniform
      c = min(cu, 2u);
      places();
    }
    cu -= c;
#pragma unroll
    for (int j = 0; j < W; ++j)
      while (c != 0u && eq[j] != 0u) {
        q[pos++] = entry(j, __ffs(eq[j]) - 1);
        eq[j] &= eq[j] - 1u;
        --c;
      }
    qn += (int)total;
    while (qn >= 32) {
      qn -= 32;
      sliced_round(sh, q + qn, 32, lane);
    }
  } while (__any_sync(0xffffffffu, cu != 0u));
}

// The warp's counter planes into the block's totals (or, for jobs of more groups than the
// block keeps, into the sums), and cleared.
template <int W>
__device__ __noinline__ void sliced_flush(SlicedShared& sh, SlicedTrack<W>* tr, int lane) {
  const GraphJob& J = sh.J;
  const uint32_t sw = J.sGp < 32u ? J.sGp : 32u;
  const uint32_t base = ((uint32_t)threadIdx.x & ~31u) & (J.sGp - 1u);
#pragma unroll 1
  for (int j = 0; j < W; ++j) {
    uint32_t col[kSlicedCnt];
#pragma unroll
    for (int b = 0; b < kSlicedCnt; ++b) {
      col[b] = warp_column(tr->cnt[b][threadIdx.x][j], lane);
      tr->cnt[b][threadIdx.x][j] = 0u;
    }
    uint32_t mask = 0u;
#pragma unroll 1
    for (uint32_t i = 0; i < 32u; i += sw) mask |= 1u << i;
#pragma unroll 1
    for (uint32_t s = 0; s < sw; ++s, mask <<= 1) {
      uint32_t c = 0u;
#pragma unroll
      for (int b = 0; b < kSlicedCnt; ++b) c += (uint32_t)__popc(col[b] & mask) << b;
      const uint32_t go = (base + s) * W + (uint32_t)j;
      if (go < J.Gj && c != 0u) {
        if (J.Gj <= (uint32_t)kSlicedTot)
          atomicAdd(&tr->tot[go][lane], c);
        else
          atomicAdd(J.sums + (size_t)(32u * (J.g0 + go) + (uint32_t)lane) * kNumSums + kSumE,
                    2.0 * (double)c);
      }
    }
  }
}

template <int W, bool VEC, bool TRACK>
__global__ void __launch_bounds__(kSlicedTile, 4) graph_sliced_kernel(
    const GraphJob* __restrict__ jobs, const Tile* __restrict__ tiles, int n_tiles,
    uint32_t half) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SlicedShared& sh = *reinterpret_cast<SlicedShared*>(smem_raw);
  SlicedTrack<W>* tr = reinterpret_cast<SlicedTrack<W>*>(smem_raw + (sizeof(SlicedShared) + 15) / 16 * 16);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tb = (int)(((long long)blockIdx.x * n_tiles) / gridDim.x);
  const int te = (int)(((long long)(blockIdx.x + 1) * n_tiles) / gridDim.x);
  const GraphJob& J = sh.J;
  int cur_job = -1, qn = 0;
  uint32_t bound = 0u;  // no counter of the warp exceeds this (warp-uniform)
  uint2* q = sh.q[warp];
  SlicedWord<W> w;
  const uint4* visit = nullptr;
  bool have = false;  // this thread's columns were copied during the previous tile
  if (TRACK) {
#pragma unroll 1
    for (int i = tid; i < kSlicedTot * 32; i += kSlicedTile) (&tr->tot[0][0])[i] = 0u;
#pragma unroll
    for (int b = 0; b < kSlicedCnt; ++b)
#pragma unroll
      for (int j = 0; j < W; ++j) tr->cnt[b][tid][j] = 0u;
  }
  // the job's queued lanes and tracking sums, before another job is staged
  auto leave = [&]() {
    if (qn > 0) sliced_round(sh, q, qn, lane);
    qn = 0;
    if (TRACK && sh.fuse) {
      sliced_flush<W>(sh, tr, lane);
      bound = 0u;
      __syncthreads();
      const double ds = (double)sh.dsum;
#pragma unroll 1
      for (uint32_t o = (uint32_t)tid; o < 32u * J.Gj; o += kSlicedTile) {
        double v = -ds;
        if (J.Gj <= (uint32_t)kSlicedTot) {
          v += 2.0 * (double)(&tr->tot[0][0])[o];
          (&tr->tot[0][0])[o] = 0u;
        }
        if (v != 0.0) atomicAdd(J.sums + (size_t)(32u * J.g0 + o) * kNumSums + kSumE, v);
      }
    }
  };
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  Tile tl = tiles[tb], tn;
  uint4 vi = make_uint4(0u, 0u, 0u, 0u), vn;  // visit entries of this tile and the next
  for (int ti = tb; ti < te; ++ti, tl = tn, vi = vn) {
    if (ti + 1 < te) tn = tiles[ti + 1];
    if ((int)tl.job != cur_job) {
      if (cur_job >= 0) leave();
      __syncthreads();  // shared per-job values are about to change
      if (tid < (int)(sizeof(GraphJob) / 4))
        reinterpret_cast<uint32_t*>(&sh.J)[tid] =
            reinterpret_cast<const uint32_t*>(jobs + tl.job)[tid];
      __syncthreads();
      // tiles, jobs and visit entries are the plan's; the step and the spins the kernel's before
      asm volatile("griddepcontrol.wait;" ::: "memory");
      if (tid == 0) {
        const CtxDev* cd = J.cd;
        const uint32_t t = cd->step;
        double b0;
        if (J.beta_sched != nullptr && cd->anneal_len != 0u) {
          uint32_t k = t - cd->anneal_t0;
          if (k >= cd->anneal_len) k = cd->anneal_len - 1u;
          b0 = J.beta_sched[k];
        } else {
          b0 = J.beta_lane[32u * J.g0];
        }
        const bool skip = t >= cd->t_end;
        sh.skip = skip ? 1u : 0u;
        sh.fuse = (TRACK && !skip && half == 0u && cd->tracking && !cd->record &&
                   J.sums != nullptr) ? 1u : 0u;
        sh.src = half == 0u ? J.A : J.B;
        sh.dst = half == 0u ? J.B : J.A;
        sh.t = t;
        sh.typ = half ^ cd->order;
        sh.beta = b0;
        sh.kb = (float)(-2.0 * b0 * 1.4426950408889634);
        sh.collapse = J.q == 1.0 ? 1u : 0u;
        sh.by_degree = J.lambda == nullptr ? 1u : 0u;
        sh.qint = J.q == rint(J.q) ? 1u : 0u;
        sh.dsum = 0ull;
      }
      __syncthreads();
      cur_job = (int)tl.job;
      have = false;
      visit = sh.typ == 0u ? J.in_visit : J.out_visit;
      if (tl.w0 + (uint32_t)tid / J.sGp < J.n) vi = __ldg(visit + tl.w0 + (uint32_t)tid / J.sGp);
      if (tid < 10) sh.key[tid] = make_uint2(J.key0 + (uint32_t)tid * kPhW0, J.key1 + (uint32_t)tid * kPhW1);
      if (sh.by_degree && !sh.skip) {  // four lanes of a degree's classes each
        const uint32_t d = (uint32_t)tid >> 2;
        const uint32_t ncls = sh.collapse ? d + 2u : 2u * d + 2u;
        uint32_t mine = 0u;
        for (uint32_t i = (uint32_t)tid & 3u; i < ncls && i < 32u; i += 4u)
          mine |= sliced_class(J.q, sh.collapse != 0u, sh.qint != 0u, sh.kb, i, d, J.lambda_c,
                               &sh.tb[0][0][0] + 32u * d) << i;
        mine |= __shfl_xor_sync(0xffffffffu, mine, 1);
        mine |= __shfl_xor_sync(0xffffffffu, mine, 2);
        if ((tid & 3) == 0) sh.amb[d] = mine;
      }
      __syncthreads();
      w.collapse = sh.collapse != 0u;
      w.go = ((uint32_t)tid & (J.sGp - 1u)) * W;
      w.last = w.go < J.Gj ? min((uint32_t)W - 1u, J.Gj - 1u - w.go) : 0u;
      w.c3base = sh.typ;
      const unsigned long long p1 = (unsigned long long)kPhM1 * sh.t;
      w.u1 = (uint32_t)p1;
#pragma unroll
      for (int j = 0; j < W; ++j) {
        const uint32_t u0 = (uint32_t)(p1 >> 32) ^ (J.g0 + w.go + (uint32_t)j) ^ J.key0;
        const unsigned long long m = (unsigned long long)kPhM0 * u0;
        w.h01[j] = (uint32_t)(m >> 32);
        w.l01[j] = (uint32_t)m;
      }
    }
    if (sh.skip) continue;
    const uint32_t Gp = J.sGp, sw = Gp < 32u ? Gp : 32u, gs = (uint32_t)lane & (sw - 1u);
    const uint32_t slot = tl.w0 + (uint32_t)tid / Gp;
    const bool in = slot < J.n;
    w.slot = slot;
    w.valid = in && w.go < J.Gj;
    w.x = in ? vi.x : 0u;
    w.p0 = in ? (int)vi.y : 0;
    w.d = in ? vi.z : 0u;
    const float lam = in ? __uint_as_float(vi.w) : 0.0f;
    // the next tile's entry, in flight during this one (another job's: read when staged)
    bool more = false;
    if (ti + 1 < te && (int)tn.job == cur_job) {
      const uint32_t ns = tn.w0 + (uint32_t)tid / Gp;
      more = ns < J.n && w.go < J.Gj;
      if (ns < J.n) vn = __ldg(visit + ns);
    }
    w.F = (in && J.frozen != nullptr) ? __ldg(J.frozen + w.x) : 0u;
    const uint32_t ncls = !in ? 0u : w.collapse ? w.d + 2u : 2u * w.d + 2u;
    const uint8_t* tbv;
    if (sh.by_degree) {
      const uint32_t d = min(w.d, 31u);
      tbv = &sh.tb[0][0][0] + 32u * d;
      w.vamb = sh.amb[d];
    } else {  // the vertex's threads take turns
      uint8_t* own = sh.tb[warp][(uint32_t)lane / sw];
      uint32_t mine = 0u;
      for (uint32_t i = gs; i < ncls; i += sw)
        mine |= sliced_class(J.q, w.collapse, sh.qint != 0u, sh.kb, i, w.d, lam, own) << i;
      for (uint32_t s = 1u; s < sw; s <<= 1) mine |= __shfl_xor_sync(0xffffffffu, mine, s);
      w.vamb = mine;
      tbv = own;
    }
    const uint32_t nm = __reduce_max_sync(0xffffffffu, ncls);
    __syncwarp();
    if (TRACK && sh.fuse) {
      const uint32_t dm = __reduce_max_sync(0xffffffffu, w.d);
      if (bound + dm > (1u << kSlicedCnt) - 1u) {
        sliced_flush<W>(sh, tr, lane);
        bound = 0u;
      }
      bound += dm;
      const uint32_t ds = __reduce_add_sync(0xffffffffu, w.valid && w.go == 0u ? w.d : 0u);
      if (lane == 0 && ds != 0u) atomicAdd(&sh.dsum, (unsigned long long)ds);
    }
    sliced_decide<W, VEC, TRACK>(sh, tr, w, tbv, nm, have, more ? &vn : nullptr, q, qn, lane);
    have = more && vn.z != 0u;
    __syncwarp();  // the class bytes are read before the next vertices' are written
  }
  if (cur_job >= 0 && !sh.skip) leave();
}

// Dynamic shared memory and resident blocks of a variant on the current device.
template <int W, bool TRACK>
static size_t sliced_bytes() {
  return (sizeof(SlicedShared) + 15) / 16 * 16 + (TRACK ? sizeof(SlicedTrack<W>) : 0);
}

template <int W, bool VEC, bool TRACK>
static int sliced_blocks_t() {
  cudaFuncSetAttribute(graph_sliced_kernel<W, VEC, TRACK>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sliced_bytes<W, TRACK>());
  static std::atomic<int> occ{0};
  int o = occ.load(), dev = 0, sms = 152;
  if (o == 0) {
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, graph_sliced_kernel<W, VEC, TRACK>,
                                                  kSlicedTile, sliced_bytes<W, TRACK>());
    occ = o > 0 ? o : 1;
  }
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return (o > 0 ? o : 1) * sms;
}

template <int W, bool VEC, bool TRACK>
static cudaError_t launch_sliced_t(const GraphJob* jobs, const Tile* tiles, int n_tiles,
                                   uint32_t half, cudaStream_t st) {
  const int blocks = sliced_blocks_t<W, VEC, TRACK>();
  const dim3 grid(n_tiles < blocks ? n_tiles : blocks);
  // A launch of few tiles is mostly its start, which then overlaps the end of the kernel before
  // (100 annealed steps of a 256^2 torus 5.22 -> 4.98 ms, n = 16000, one group, 23.3 -> 20.8 us a
  // step); with long tile ranges nothing is gained.
  if (n_tiles < 4 * blocks)
    return launch_dependent(graph_sliced_kernel<W, VEC, TRACK>, grid, dim3(kSlicedTile),
                            sliced_bytes<W, TRACK>(), st, jobs, tiles, n_tiles, half);
  graph_sliced_kernel<W, VEC, TRACK>
      <<<grid, kSlicedTile, sliced_bytes<W, TRACK>(), st>>>(jobs, tiles, n_tiles, half);
  return cudaGetLastError();
}

// shape: index in kSlicedShapes (words per thread, whole aligned rows)
int graph_sliced_blocks(int shape, bool track) {
  switch (shape) {
    case 0: return track ? sliced_blocks_t<1, true, true>() : sliced_blocks_t<1, true, false>();
    case 1: return track ? sliced_blocks_t<2, true, true>() : sliced_blocks_t<2, true, false>();
    case 2: return track ? sliced_blocks_t<3, false, true>() : sliced_blocks_t<3, false, false>();
    case 3: return track ? sliced_blocks_t<4, true, true>() : sliced_blocks_t<4, true, false>();
    default: return track ? sliced_blocks_t<4, false, true>() : sliced_blocks_t<4, false, false>();
  }
}

cudaError_t launch_graph_sliced(int shape, bool track, const GraphJob* jobs, const Tile* tiles,
                                int n_tiles, uint32_t half, cudaStream_t st) {
  if (n_tiles <= 0) return cudaSuccess;
  switch (shape) {
    case 0:
      return track ? launch_sliced_t<1, true, true>(jobs, tiles, n_tiles, half, st)
                   : launch_sliced_t<1, true, false>(jobs, tiles, n_tiles, half, st);
    case 1:
      return track ? launch_sliced_t<2, true, true>(jobs, tiles, n_tiles, half, st)
                   : launch_sliced_t<2, true, false>(jobs, tiles, n_tiles, half, st);
    case 2:
      return track ? launch_sliced_t<3, false, true>(jobs, tiles, n_tiles, half, st)
                   : launch_sliced_t<3, false, false>(jobs, tiles, n_tiles, half, st);
    case 3:
      return track ? launch_sliced_t<4, true, true>(jobs, tiles, n_tiles, half, st)
                   : launch_sliced_t<4, true, false>(jobs, tiles, n_tiles, half, st);
    default:
      return track ? launch_sliced_t<4, false, true>(jobs, tiles, n_tiles, half, st)
                   : launch_sliced_t<4, false, false>(jobs, tiles, n_tiles, half, st);
  }
}

}  // namespace shk
