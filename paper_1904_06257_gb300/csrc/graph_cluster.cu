// graph_cluster.cu -- whole runs of small +-1 graphs: one thread-block cluster owns one group of
// 32 replicas of a graph for n steps, its words in the blocks' shared memory.
//
// Vertex x's word lives in block x mod C (C a power of two), so neighbours are gathered
// from distributed shared memory; 32 consecutive slots of the degree order make a warp's
// pass, dealt round the blocks.  A block keeps its slots' entries and columns of both
// directions in shared memory, too (lane-major per pass): read from global memory they
// came from L2 in every half step, since the cluster barrier empties L1.  The first pass's
// two Philox calls of the next half step are made between arriving at the barrier and
// waiting for it.  A half step ends at the cluster barrier.  Draws, classes and
// decisions are those of graph_sliced_kernel, so the trajectory is the same.  One lambda on
// all vertices: the class bytes of the next step (by degree) are made during the second
// half step.  With tracking the agreeing edges of sigma_t are counted in the first
// half, gathered by the cluster's first block during the second and turned into best
// energies and series behind the next barrier (lambda = 0).
//
// Bound by a half step's chain: barrier, entry and column loads, gathers, two Philox calls,
// the plane comparison, a round of queued lanes -- about 1250 instructions of the warps that have
// vertices, one of them at a time on a scheduler (7 cycles each).  n = 2000, mean degree 6,
// 32 replicas, tracked anneal: 11 us a step in clusters of 16 (14 us in clusters of 4),
// against 19 us of the half-step kernels and 37 us of the general kernel.
#include <cooperative_groups.h>

#include <cstdint>

#include "graph_planes.cuh"
#include "shaken_internal.cuh"

namespace shk {

namespace cg = cooperative_groups;

constexpr int kGclThreads = 256;  // 255 registers a thread: local memory is as far as L2 here
constexpr int kGclWarps = kGclThreads / 32;
constexpr int kGclPlanes = 10;  // counter planes: at most kGclPasses passes of degree <= 31
constexpr int kGclPasses = 32;
constexpr uint32_t kGclColSlack = 3 * 32 * 31;  // see gcl_col_words

struct GclShared {
  __align__(16) uint8_t by_deg[2][32][32];  // [step parity][degree][class] top bytes, bit-reversed
  GraphJob J;
  uint32_t amb[2][32];       // classes of uncertain top byte, by degree
  uint2 q[kGclWarps][64];
  uint2 key[10];
  double beta[2];            // by step parity
  float kb[2];
  uint32_t base[2][kGclPasses * kGclWarps];  // first padded column word of a pass, per direction
  unsigned int block[2][32];  // up spins and agreeing edges of this block's vertices, per replica
  unsigned int all[2][32];    // of the cluster (used in block 0)
};

__device__ __forceinline__ uint32_t dsm_addr(uint32_t local, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
  return a;
}
__device__ __forceinline__ uint32_t dsm_ld(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void dsm_st(uint32_t a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dsm_or(uint32_t a, uint32_t v) {
  asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dsm_add(uint32_t a, uint32_t v) {
  asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// Up to 32 queued lanes (entries as in graph_sliced_kernel, without the group).
__device__ __noinline__ void gcl_round(const GclShared& sh, const uint4* entry, const uint2* q,
                                       int cnt, uint32_t dst, uint32_t t, uint32_t typ,
                                       uint32_t C, uint32_t lc, int lane) {
  __syncwarp();
  if (lane < cnt) {
    const uint2 e = q[lane];
    const GraphJob& J = sh.J;
    const uint4 vi = entry[e.x];
    const int k = (int)(e.y & 31u);
    if (sliced_lane(J.key0, J.key1, vi.x, J.g0, t, typ, J.q, J.q == 1.0, sh.kb[t & 1u],
                    sh.beta[t & 1u], (int)vi.z, __uint_as_float(vi.w), k, (e.y >> 5) & 31u,
                    (e.y >> 18) & 0xFFu, ((e.y >> 26) & 1u) != 0u))
      dsm_or(dsm_addr(dst + 4u * (vi.x >> lc), vi.x & (C - 1u)), 1u << k);
  }
  __syncwarp();
}

// jobs: one per group (g0); n_steps: at most, a context stops at its t_end; col_words: the
// padded column words of a direction that the shared memory holds.
__global__ void __launch_bounds__(kGclThreads, 1) graph_cluster_kernel(
    const GraphJob* __restrict__ jobs, uint32_t n_steps, uint32_t col_words) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  GclShared& sh = *reinterpret_cast<GclShared*>(smem_raw);
  uint32_t* words = reinterpret_cast<uint32_t*>(smem_raw + (sizeof(GclShared) + 15) / 16 * 16);
  cg::cluster_group cl = cg::this_cluster();
  const uint32_t C = cl.num_blocks(), r = cl.block_rank(), lc = 31u - (uint32_t)__clz((int)C);
  const int tid = (int)threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const GraphJob& J = sh.J;
  if (tid < (int)(sizeof(GraphJob) / 4))
    reinterpret_cast<uint32_t*>(&sh.J)[tid] =
        reinterpret_cast<const uint32_t*>(jobs + blockIdx.x / C)[tid];
  if (tid < 64) (&sh.block[0][0])[tid] = (&sh.all[0][0])[tid] = 0u;
  __syncthreads();
  const CtxDev* cd = J.cd;
  const uint32_t t0 = cd->step, t_end = cd->t_end, order = cd->order;
  if (t0 >= t_end) return;  // every block of the cluster
  const uint32_t steps = min(n_steps, t_end - t0);
  const uint32_t n = J.n, nper = (n + C - 1u) >> lc, g = J.g0, G = J.G;
  const uint32_t anneal_t0 = cd->anneal_t0, anneal_len = cd->anneal_len;
  const bool anneal = J.beta_sched != nullptr && anneal_len != 0u;
  const bool track = cd->tracking && J.sums != nullptr, record = track && cd->record;
  const bool collapse = J.q == 1.0, qint = J.q == rint(J.q);
  const uint32_t buf0 = (uint32_t)__cvta_generic_to_shared(words);
  if (tid < 10)
    sh.key[tid] = make_uint2(J.key0 + (uint32_t)tid * kPhW0, J.key1 + (uint32_t)tid * kPhW1);
  for (uint32_t i = (uint32_t)tid; i < nper; i += kGclThreads) {
    const uint32_t x = (i << lc) + r;
    words[i] = x < n ? J.A[(size_t)x * G + g] : 0u;
  }
  // beta, and the class bytes by degree (eight threads a degree), of step t
  // the block's slots of both directions: entries (vertex, -, degree, lambda), columns
  const uint32_t chunks = (n + 31u) / 32u;                    // passes of the whole graph
  const uint32_t mine_n = chunks > r ? (chunks - r + C - 1u) >> lc : 0u;  // of this block: j = i C + r
  const uint32_t slots = ((chunks + C - 1u) >> lc) * 32u;
  uint4* const entries = reinterpret_cast<uint4*>(words + ((2u * nper + 3u) & ~3u));
  uint32_t* const columns = reinterpret_cast<uint32_t*>(entries + 2u * slots);
  for (uint32_t dir = 0; dir < 2u; ++dir) {
    const uint4* visit = dir == 0u ? J.in_visit : J.out_visit;
    for (uint32_t o = (uint32_t)tid; o < mine_n * 32u; o += kGclThreads) {
      const uint32_t s = ((o >> 5) * C + r) * 32u + (o & 31u);
      entries[dir * slots + o] = s < n ? visit[s] : make_uint4(0u, 0u, 0u, 0u);
    }
  }
  __syncthreads();
  if (warp < 2) {  // prefix sums of 32 x the largest degree of each pass (its last slot)
    uint32_t run = 0u;
    for (uint32_t i0 = 0; i0 < mine_n; i0 += 32u) {
      const uint32_t i = i0 + (uint32_t)lane;
      uint32_t v = 0u;
      if (i < mine_n) {
        const uint32_t last = min(31u, n - 1u - (i * C + r) * 32u);
        v = 32u * entries[(uint32_t)warp * slots + i * 32u + last].z;
      }
      uint32_t sum = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, sum, o);
        if (lane >= o) sum += u;
      }
      if (i < mine_n) sh.base[warp][i] = run + sum - v;
      run += __shfl_sync(0xffffffffu, sum, 31);
    }
  }
  __syncthreads();
  for (uint32_t dir = 0; dir < 2u; ++dir) {
    const uint32_t* col = dir == 0u ? J.in_col : J.out_col;
    for (uint32_t o = (uint32_t)tid; o < mine_n * 32u; o += kGclThreads) {
      const uint4 vi = entries[dir * slots + o];
      uint32_t* c = columns + dir * col_words + sh.base[dir][o >> 5] + (o & 31u);
      for (uint32_t e = 0; e < vi.z; ++e) c[32u * e] = __ldg(col + vi.y + e);
    }
  }
  auto beta_of = [&](uint32_t t) {
    uint32_t k = t - anneal_t0;
    if (k >= anneal_len) k = anneal_len - 1u;
    return anneal ? __ldg(J.beta_sched + k) : __ldg(J.beta_lane + 32u * g);
  };
  auto stage = [&](uint32_t t, double b) {
    const float kb = (float)(-2.0 * b * 1.4426950408889634);
    if (tid == 0) {
      sh.beta[t & 1u] = b;
      sh.kb[t & 1u] = kb;
    }
    {
      const uint32_t d = (uint32_t)tid >> 3, ncls = collapse ? d + 2u : 2u * d + 2u;
      uint32_t mine = 0u;
      for (uint32_t i = (uint32_t)tid & 7u; i < min(ncls, 32u); i += 8u)
        mine |= sliced_class(J.q, collapse, qint, kb, i, d, J.lambda_c, sh.by_deg[t & 1u][d]) << i;
#pragma unroll
      for (int s = 1; s < 8; s <<= 1) mine |= __shfl_xor_sync(0xffffffffu, mine, s);
      if ((tid & 7) == 0) sh.amb[t & 1u][d] = mine;
    }
  };
  double b_next = beta_of(t0 + 1u);  // read a step ahead
  stage(t0, beta_of(t0));
  if (!anneal) stage(t0 + 1u, b_next);
  const bool keeper = track && r == 0u && tid >= kGclThreads - 32;
  const uint32_t fwd = (uint32_t)tid - (kGclThreads - 96u);  // < 64: forwards the block's sums
  const uint32_t rep = 32u * g + (uint32_t)lane;
  double best = keeper ? cd->best[rep] : 0.0;
  const double inv_n = cd->inv_n;
  const uint32_t series_t0 = cd->series_t0, series_cap = cd->series_cap, Rn = cd->R;
  double* const series_m = record ? cd->series_m : nullptr;
  double* const series_H = record ? cd->series_H : nullptr;
  double* const best_p = cd->best;
  long long* const best_step_p = cd->best_step;
  const double m_edges = (double)J.in_ptr[n];
  auto close = [&](uint32_t t) {  // the sums of sigma_t, gathered, into best and series
    const double M = 2.0 * (double)sh.all[0][lane] - (double)n;
    const double H = -(2.0 * (double)sh.all[1][lane] - m_edges);
    sh.all[0][lane] = sh.all[1][lane] = 0u;
    if (H < best) {
      best = H;
      best_p[rep] = H;
      best_step_p[rep] = (long long)t;
    }
    if (record && t - series_t0 < series_cap) {
      const size_t k = (size_t)(t - series_t0) * Rn + rep;
      if (series_m) series_m[k] = M * inv_n;
      if (series_H) series_H[k] = H;
    }
  };
  cl.sync();
  SlicedWord<1> w;
  uint2* q = sh.q[warp];
  const uint32_t below = (1u << lane) - 1u;
  // the parts of a step's Philox calls that all vertices share
  auto philox_step = [&](uint32_t t) {
    const unsigned long long p1 = (unsigned long long)kPhM1 * t;
    w.u1 = (uint32_t)p1;
    const unsigned long long pm = (unsigned long long)kPhM0 * ((uint32_t)(p1 >> 32) ^ g ^ J.key0);
    w.h01[0] = (uint32_t)(pm >> 32);
    w.l01[0] = (uint32_t)pm;
  };
  uint32_t ahead[2][4][1];  // the first pass's calls
  auto call_ahead = [&](uint32_t typ) {
    if ((uint32_t)warp >= mine_n) return;
    w.x = entries[typ * slots + (uint32_t)tid].x;
    sliced_call<1>(sh.key, w, typ, ahead[0]);
    sliced_call<1>(sh.key, w, typ + 2u, ahead[1]);
  };
  philox_step(t0);
  call_ahead(order);
#pragma unroll 1
  for (uint32_t st = 0; st < steps; ++st) {
    const uint32_t t = t0 + st;
#pragma unroll 1
    for (uint32_t pos = 0; pos < 2u; ++pos) {
      const uint32_t typ = pos ^ order;
      const uint32_t src = buf0 + 4u * nper * pos, dst = buf0 + 4u * nper * (pos ^ 1u);
      const bool sums = track && pos == 0u;
      if (keeper && pos == 0u && st != 0u) close(t - 1u);
      if (track && pos == 1u && fwd < 64u) {  // this block's sums to block 0
        unsigned int* s = &sh.block[0][0] + fwd;
        const uint32_t v = *s;
        *s = 0u;
        if (v != 0u)
          dsm_add(dsm_addr((uint32_t)__cvta_generic_to_shared(&sh.all[0][0] + fwd), 0u), v);
      }
      int qn = 0;
      uint32_t cnt[kGclPlanes], bound = 0u, ups[6] = {0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
      for (int b = 0; b < kGclPlanes; ++b) cnt[b] = 0u;
#pragma unroll 1
      for (uint32_t i = (uint32_t)warp; i < mine_n; i += (uint32_t)kGclWarps) {
        const uint32_t local = 32u * i + (uint32_t)lane;
        const bool in = (i * C + r) * 32u + (uint32_t)lane < n;
        const uint4 vi = entries[typ * slots + local];
        const uint32_t* col = columns + typ * col_words + sh.base[typ][i] + lane;
        w.x = vi.x;
        const uint32_t d = vi.z;
        const uint32_t S = in ? dsm_ld(dsm_addr(src + 4u * (w.x >> lc), w.x & (C - 1u))) : 0u;
        uint32_t I[kIdx][1];
#pragma unroll
        for (int b = 0; b < kIdx; ++b) I[b][0] = 0u;
#pragma unroll 1
        for (uint32_t e = 0; e < d; e += 4) {  // four edges at a time, the last again beyond d
          uint32_t cv[4], x[4];
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k) cv[k] = col[32u * min(e + k, d - 1u)];
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t y = cv[k] & 0x7fffffffu;
            x[k] = dsm_ld(dsm_addr(src + 4u * (y >> lc), y & (C - 1u)));
          }
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k)
            x[k] = e + k < d ? x[k] ^ (uint32_t)((int32_t)cv[k] >> 31) : 0u;
          const uint32_t s0 = I[0][0] ^ x[0] ^ x[1], ca = maj3(I[0][0], x[0], x[1]);
          const uint32_t cb = maj3(s0, x[2], x[3]);
          I[0][0] = s0 ^ x[2] ^ x[3];
          uint32_t c = maj3(I[1][0], ca, cb);
          I[1][0] ^= ca ^ cb;
#pragma unroll
          for (int b = 2; b < kIdx; ++b) {
            const uint32_t u = I[b][0] & c;
            I[b][0] ^= c;
            c = u;
          }
        }
        if (sums) {  // agreeing edges: a where sigma = +1, d - a otherwise
          uint32_t br = 0u, carry = 0u;
#pragma unroll
          for (int b = 0; b < kGclPlanes; ++b) {
            uint32_t ag = 0u;
            if (b < kIdx) {
              const uint32_t D = 0u - ((d >> b) & 1u), A = I[b][0];
              ag = (S & A) | (~S & (D ^ A ^ br));
              br = (~D & A) | (~D & br) | (A & br);
            }
            const uint32_t old = cnt[b];
            cnt[b] = old ^ ag ^ carry;
            carry = maj3(old, ag, carry);
          }
          bound += 31u;
          uint32_t c = S;
#pragma unroll
          for (int b = 0; b < 6; ++b) {
            const uint32_t u = ups[b] & c;
            ups[b] ^= c;
            c = u;
          }
        }
        uint32_t ncls = 0u;
        if (collapse) {  // idx = a + sigma
          uint32_t c = S;
#pragma unroll
          for (int b = 0; b < kIdx; ++b) {
            const uint32_t u = I[b][0] & c;
            I[b][0] ^= c;
            c = u;
          }
          ncls = d + 2u;
        } else {  // idx = 2 a + sigma
#pragma unroll
          for (int b = kIdx - 1; b > 0; --b) I[b][0] = I[b - 1][0];
          I[0][0] = S;
          ncls = 2u * d + 2u;
        }
        const uint8_t* tbv = sh.by_deg[t & 1u][d];
        w.vamb = sh.amb[t & 1u][d];
        w.F = in ? (J.frozen != nullptr ? __ldg(J.frozen + w.x) : 0u) : 0xffffffffu;
        const uint32_t nm = __reduce_max_sync(0xffffffffu, ncls);
        uint32_t lt[1] = {0u}, eq[1] = {~w.F};
#pragma unroll 1
        for (int call = 1; call >= 0; --call) {
          uint32_t o[4][1];
          if (i < (uint32_t)kGclWarps) {
#pragma unroll
            for (int k = 0; k < 4; ++k) o[k][0] = call != 0 ? ahead[1][k][0] : ahead[0][k][0];
          } else {
            sliced_call<1>(sh.key, w, typ + 2u * (uint32_t)call, o);
          }
          if (nm <= 4u)
            sliced_planes<2, 1>(tbv, call, I, o, lt, eq);
          else if (nm <= 8u)
            sliced_planes<3, 1>(tbv, call, I, o, lt, eq);
          else if (nm <= 16u)
            sliced_planes<4, 1>(tbv, call, I, o, lt, eq);
          else
            sliced_planes<5, 1>(tbv, call, I, o, lt, eq);
        }
        uint32_t amb = 0u;
#pragma unroll 1
        for (uint32_t m = w.vamb; m != 0u; m &= m - 1u) {  // rare: lanes of uncertain classes
          const uint32_t c = (uint32_t)__ffs(m) - 1u;
          uint32_t is = 0xffffffffu;
#pragma unroll
          for (int b = 0; b < kIdx; ++b) is &= ~(I[b][0] ^ (0u - ((c >> b) & 1u)));
          amb |= is;
        }
        uint32_t und = (eq[0] | amb) & ~w.F;
        if (in)
          dsm_st(dsm_addr(dst + 4u * (w.x >> lc), w.x & (C - 1u)), (lt[0] & ~und) | w.F);
#pragma unroll 1
        while (true) {  // one undecided lane of each thread at a time
          const uint32_t ball = __ballot_sync(0xffffffffu, und != 0u);
          if (ball == 0u) break;
          if (und != 0u) {
            const int k = __ffs(und) - 1;
            und &= und - 1u;
            uint32_t idx = 0u;
#pragma unroll
            for (int b = 0; b < kIdx; ++b) idx |= ((I[b][0] >> k) & 1u) << b;
            q[qn + __popc(ball & below)] =
                make_uint2(local, (uint32_t)k | (idx << 5) |
                                     ((__brev((uint32_t)tbv[idx]) >> 24) << 18) |
                                     (((w.vamb >> idx) & 1u) << 26));
          }
          qn += __popc(ball);
          if (qn >= 32) {
            qn -= 32;
            gcl_round(sh, entries + typ * slots, q + qn, 32, dst, t, typ, C, lc, lane);
          }
        }
      }
      if (qn > 0) gcl_round(sh, entries + typ * slots, q, qn, dst, t, typ, C, lc, lane);
      if (sums && bound != 0u) {  // the warp's threads: per-replica counts of its planes
        uint32_t cm = 0u, ce = 0u;
#pragma unroll
        for (int b = 0; b < kGclPlanes; ++b)
          if ((bound >> b) != 0u) ce += (uint32_t)__popc(warp_column(cnt[b], lane)) << b;
        if (record) {
#pragma unroll
          for (int b = 0; b < 6; ++b) cm += (uint32_t)__popc(warp_column(ups[b], lane)) << b;
          if (cm) atomicAdd(&sh.block[0][lane], cm);
        }
        if (ce) atomicAdd(&sh.block[1][lane], ce);
      }
      if (anneal && pos == 1u) {  // the next step's thresholds
        stage(t + 1u, b_next);
        b_next = beta_of(t + 2u);
      }
      cl.barrier_arrive();
      if (pos == 1u) philox_step(t + 1u);
      call_ahead(typ ^ 1u);  // the next half step's (the next step begins with the other type)
      cl.barrier_wait();
    }
  }
  if (keeper) close(t0 + steps - 1u);
  for (uint32_t i = (uint32_t)tid; i < nper; i += kGclThreads) {
    const uint32_t x = (i << lc) + r;
    if (x < n) {
      J.A[(size_t)x * G + g] = words[i];
      J.B[(size_t)x * G + g] = words[nper + i];
    }
  }
}

// The step counters of contexts whose whole run went through graph_cluster_kernel.
__global__ void advance_kernel(CtxDev* const* __restrict__ ctxs, int n, uint32_t steps) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= n) return;
  CtxDev* cd = ctxs[i];
  if (cd->step < cd->t_end) cd->step += min(steps, cd->t_end - cd->step);
}

// Padded column words of a block and direction.  Passes ascend by degree, so 32 x the largest
// degree of a pass is at most the edges of the next one (if that is whole), and the edges of
// every C-th pass are at most m / C and one pass; the last two passes have no whole next
// one: m / C + 3 x 32 x 31.
static uint32_t gcl_col_words(uint64_t m, uint32_t C) {
  return (uint32_t)(m / C) + kGclColSlack;
}

static size_t gcl_bytes(uint32_t n, uint64_t m, uint32_t C) {
  const size_t nper = (n + C - 1u) / C, slots = ((n + 31u) / 32u + C - 1u) / C * 32u;
  return (sizeof(GclShared) + 15) / 16 * 16 + (2 * nper + 3) / 4 * 16 + 2 * slots * sizeof(uint4) +
         2 * (size_t)gcl_col_words(m, C) * sizeof(uint32_t);
}

static cudaError_t gcl_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, uint32_t n,
                              uint64_t m, uint32_t C, int clusters, cudaStream_t st) {
  const size_t bytes = gcl_bytes(n, m, C);
  cudaError_t e = cudaFuncSetAttribute(graph_cluster_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(graph_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed,
                             1);
  if (e != cudaSuccess) return e;
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3((unsigned)clusters * C);
  cfg.blockDim = dim3(kGclThreads);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaSuccess;
}

// Blocks per cluster for `clusters` groups of graphs of at most n vertices, and the microseconds
// of a step: the size of least time, a half step taking 2.5 us and 11.5 ns per vertex of a
// block, times the waves of clusters (as in lattice_cluster_shape); 0: too large.
int graph_cluster_shape(uint32_t n, uint64_t m, int clusters, double* us) {
  int dev = 0, max_smem = 0, best = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  for (uint32_t C = 1; C <= 16u; C *= 2) {
    const uint32_t passes = (n + C * kGclThreads - 1u) / (C * kGclThreads);
    if (gcl_bytes(n, m, C) + 1024 > (size_t)max_smem || passes > (uint32_t)kGclPasses) continue;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    int fit = 0;
    if (gcl_config(cfg, attr, n, m, C, clusters, nullptr) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&fit, graph_cluster_kernel, &cfg) != cudaSuccess ||
        fit < 1) {
      cudaGetLastError();
      continue;
    }
    const int wave = C == 1u || fit < 4 ? fit : fit * 3 / 4;
    const double t = 2.0 * (2.5 + 1.15e-2 * n / C) * ((clusters + wave - 1) / wave);
    if (best == 0 || t < *us) {
      best = (int)C;
      *us = t;
    }
  }
  return best;
}

cudaError_t launch_graph_cluster(const GraphJob* jobs, int clusters, uint32_t n, uint64_t m, int C,
                                 CtxDev* const* ctxs, int n_ctx, uint32_t steps, cudaStream_t st) {
  if (clusters <= 0 || steps == 0) return cudaSuccess;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cudaError_t e = gcl_config(cfg, attr, n, m, (uint32_t)C, clusters, st);
  if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, graph_cluster_kernel, jobs, steps, gcl_col_words(m, (uint32_t)C));
  if (e != cudaSuccess) return e;
  advance_kernel<<<(n_ctx + 127) / 128, 128, 0, st>>>(ctxs, n_ctx, steps);
  return cudaGetLastError();
}

}  // namespace shk
