// graph_cluster.cu -- whole runs of small +-1 graphs: one thread-block cluster owns one group of
// 32 replicas of a graph for a chunk of steps, its words in the blocks' shared memory, the draws
// compared ahead of the run.
//
// A draw depends on (seed, vertex, group, step, half) alone and a threshold on the class (agreeing
// neighbours, own spin) alone, so the outcome of every class is known before the configuration is.
// graph_thresholds_kernel makes the thresholds of a chunk of steps (fp64, by degree and class),
// graph_ahead_kernel the outcome words of every vertex and class on the whole GPU, and
// graph_cluster_kernel only counts neighbours and selects.  The outcomes are those of all 32
// planes, so the trajectory is that of the half-step kernels.
//
// Every block holds all of the group's words, so neighbours are gathers from its own shared
// memory.  32 consecutive slots of a direction's degree order make a warp's pass, dealt
// round the blocks; the buffer a half step writes is in the order of its own direction, so a
// pass's results are one line to each block (distributed shared memory).  A block keeps
// the entries and columns of its slots in both directions in shared memory, too, as places in
// the buffer that the half step reads (lane-major per pass).  The outcome words of a
// warp's next pass are on their way (cp.async) during a pass.  A half step ends at the
// cluster barrier.  With tracking the agreeing edges of sigma_t are counted in the first
// half, gathered by the cluster's first block during the second and turned into best
// energies and series behind the next barrier (lambda = 0).
//
// Bound by a half step's chain (barrier, gathers, selects, stores to the other blocks).  n = 2000,
// mean degree 6, 32 replicas, 200 annealed steps: 4.5 us a step; 6.3 with each word in one block,
// gathered from distributed shared memory (5 ns a vertex of a block against 1.4); 10.6 with the draws
// made in the run; 19 in the half-step kernels.  n = 8000: 7.0 against 20.6 us.
#include <cooperative_groups.h>
#include <cuda_pipeline_primitives.h>

#include <cstdint>

#include "graph_planes.cuh"
#include "shaken_internal.cuh"

namespace shk {

namespace cg = cooperative_groups;

cudaError_t launch_advance(CtxDev* const*, int, uint32_t, cudaStream_t);

constexpr int kGclThreads = 512;
constexpr int kGclWarps = kGclThreads / 32;
constexpr int kAheadThreads = 256;  // of graph_ahead_kernel
constexpr int kGclPlanes = 10;  // counter planes: at most kGclPasses passes of degree <= 31
constexpr int kGclPasses = 32;
constexpr uint32_t kGclColSlack = 3 * 32 * 31;  // see gcl_col_words
constexpr int kGclDegs = 32, kGclClasses = 32;  // degrees 0..31, classes of a vertex at most

struct GclShared {
  GraphJob J;
  uint32_t base[2][kGclPasses * kGclWarps];  // first padded column word of a pass, per direction
  uint8_t ncls[2][kGclPasses * kGclWarps];   // most classes of a pass's vertices
  unsigned int block[2][32];  // up spins and agreeing edges of this block's vertices, per replica
  unsigned int all[2][32];    // of the cluster (used in block 0)
};

// Classes of a vertex of degree d: i = a + [sigma = +1] at q = 1 (a agreeing in-neighbours;
// the field of (a, +1) is that of (a + 1, -1) exactly), else 2 a + [sigma = +1].
__device__ __forceinline__ uint32_t gcl_classes(bool collapse, uint32_t d) {
  return collapse ? d + 2u : 2u * d + 2u;
}

// T of every degree and class for step cd->step + k of a context (the block of its first group):
// tab[((job n_steps + k) 32 + d) 32 + i] = (low word, ~0 where T = 2^32); without an anneal
// all steps share step 0's.
__global__ void __launch_bounds__(128) graph_thresholds_kernel(const GraphJob* __restrict__ jobs,
                                                               uint32_t n_steps,
                                                               uint2* __restrict__ tab) {
  const uint32_t job = blockIdx.x / n_steps, k = blockIdx.x % n_steps;
  const GraphJob& J = jobs[job];
  if (J.g0 != 0u) return;
  const CtxDev* cd = J.cd;
  const uint32_t t = cd->step + k, anneal_len = cd->anneal_len;
  const bool anneal = J.beta_sched != nullptr && anneal_len != 0u;
  if (t >= cd->t_end || (k != 0u && !anneal)) return;
  const double beta =
      anneal ? J.beta_sched[min(t - cd->anneal_t0, anneal_len - 1u)] : J.beta_lane[0];
  const uint32_t dmax = max(J.in_visit[J.n - 1u].z, J.out_visit[J.n - 1u].z);
  const bool collapse = J.q == 1.0;
  uint2* out = tab + (size_t)blockIdx.x * (kGclDegs * kGclClasses);
  for (uint32_t o = threadIdx.x; o < (dmax + 1u) * kGclClasses; o += blockDim.x) {
    const uint32_t d = o / kGclClasses, i = o % kGclClasses;
    if (d >= (uint32_t)kGclDegs || i >= gcl_classes(collapse, d)) continue;
    const int a = (int)(collapse ? i : i >> 1), up = collapse ? 0 : (int)(i & 1u);
    const double h = field_h(1.0, 2 * a - (int)d, J.q, 2 * up - 1, (double)J.lambda_c);
    const unsigned long long T = threshold_T(h, beta);
    out[o] = make_uint2((uint32_t)T, T >> 32 != 0ull ? 0xffffffffu : 0u);
  }
}

// Outcomes u < T of every class, one warp per pass of 32 slots of a half step's degree order:
// out[((k 2 + pos) ptot + off[job] + pass) stride + 32 i + lane] for class i.
// Bound by integer issue: three Philox calls and, a class, four operations a plane.
// (8000 vertices, 4 groups, mean degree 8: 180 ns per 1000 words and step.)
__global__ void __launch_bounds__(kAheadThreads) graph_ahead_kernel(
    const GraphJob* __restrict__ jobs, const uint32_t* __restrict__ off, uint32_t n_steps,
    uint32_t per, uint32_t ptot, uint32_t stride, const uint2* __restrict__ tab,
    uint32_t* __restrict__ out) {
  uint32_t item = blockIdx.x / per;
  const uint32_t pass = (blockIdx.x % per) * (kAheadThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31u;
  const uint32_t pos = item & 1u, k = (item >> 1) % n_steps, job = (item >> 1) / n_steps;
  const GraphJob& J = jobs[job];
  const CtxDev* cd = J.cd;
  const uint32_t t = cd->step + k, n = J.n, s = pass * 32u + lane;
  if (t >= cd->t_end || pass * 32u >= n) return;
  const uint32_t typ = pos ^ cd->order;
  const bool anneal = J.beta_sched != nullptr && cd->anneal_len != 0u;
  const bool in = s < n;
  const uint4 vi = in ? (typ == 0u ? J.in_visit : J.out_visit)[s] : make_uint4(0u, 0u, 0u, 0u);
  const uint32_t x = vi.x, ncls = in ? gcl_classes(J.q == 1.0, vi.z) : 0u;
  const uint32_t F = in && J.frozen != nullptr ? __ldg(J.frozen + x) : 0u;
  const PhKey K = ph_key(J.key0, J.key1);
  const PhShared P = ph_shared(K, J.g0, t);
  const uint4 W[3] = {ph_call_shared(K, P, x, typ), ph_call_shared(K, P, x, typ + 2u),
                      ph_call_shared(K, P, x, typ + 4u)};
  const uint2* T = tab + ((size_t)(job - J.g0) * n_steps + (anneal ? k : 0u)) *
                             (kGclDegs * kGclClasses) + vi.z * kGclClasses;
  uint32_t* o = out + ((size_t)(2u * k + pos) * ptot + off[job] + pass) * stride + lane;
  const uint32_t most = __reduce_max_sync(0xffffffffu, ncls);
#pragma unroll 1
  for (uint32_t i = 0; i < most; ++i) {
    const uint2 th = i < ncls ? __ldg(T + i) : make_uint2(0u, 0xffffffffu);
    uint32_t lt = 0u, eq = 0xffffffffu;
#pragma unroll
    for (int j = 11; j >= 0; --j) {  // twelve planes as a subtraction: borrow and equality
      const uint4& q = W[j >> 2];
      const uint32_t w = (j & 3) == 0 ? q.x : (j & 3) == 1 ? q.y : (j & 3) == 2 ? q.z : q.w;
      const uint32_t m = (uint32_t)((int32_t)(th.x << j) >> 31);
      lt = maj3(~w, m, lt);
      eq &= ~(w ^ m);
    }
    const uint32_t sure = F | th.y;
    lt &= ~eq;
    eq &= ~sure;
#pragma unroll 1
    for (uint32_t call = 3; call < 8u && eq != 0u; ++call) {
      const uint4 q = ph_call_shared(K, P, x, typ + 2u * call);
#pragma unroll
      for (uint32_t b = 0; b < 4u; ++b) {
        const uint32_t w = b == 0u ? q.x : b == 1u ? q.y : b == 2u ? q.z : q.w;
        const uint32_t m = (uint32_t)((int32_t)(th.x << (4u * call + b)) >> 31);
        const uint32_t diff = (w ^ m) & eq;
        lt |= diff & m;
        eq &= ~diff;
      }
    }
    if (i < ncls) o[32u * i] = lt | sure;
  }
}

// Class idx (planes I) of the 2^NB outcome words p[32 i].
template <int NB>
__device__ __forceinline__ uint32_t gcl_select(const uint32_t* p, const uint32_t (&I)[kIdx]) {
  if constexpr (NB == 0) {
    return *p;
  } else {
    const uint32_t lo = gcl_select<NB - 1>(p, I), hi = gcl_select<NB - 1>(p + (32 << (NB - 1)), I);
    return (I[NB - 1] & hi) | (~I[NB - 1] & lo);
  }
}

__device__ __forceinline__ uint32_t dsm_addr(uint32_t local, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local), "r"(rank));
  return a;
}
__device__ __forceinline__ void dsm_st(uint32_t a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dsm_add(uint32_t a, uint32_t v) {
  asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// jobs: one per group (g0); n_steps: at most, a context stops at its t_end; col_words: the
// padded column words of a direction that the shared memory holds; off, ptot, stride, ahead: the
// outcome words (graph_ahead_kernel).
__global__ void __launch_bounds__(kGclThreads, 1) graph_cluster_kernel(
    const GraphJob* __restrict__ jobs, const uint32_t* __restrict__ off, uint32_t n_steps,
    uint32_t col_words, uint32_t ptot, uint32_t stride, const uint32_t* __restrict__ ahead) {
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
  const uint32_t n = J.n, g = J.g0, G = J.G;
  const bool track = cd->tracking && J.sums != nullptr, record = track && cd->record;
  const bool collapse = J.q == 1.0;
  const uint32_t* const mine = ahead + (size_t)off[blockIdx.x / C] * stride;
  const uint32_t chunks = (n + 31u) / 32u;                    // passes of the whole graph
  const uint32_t mine_n = chunks > r ? (chunks - r + C - 1u) >> lc : 0u;  // of this block: j = i C + r
  const uint32_t slots = ((chunks + C - 1u) >> lc) * 32u, nw = 32u * chunks;
  uint32_t* const entries = words + 2u * nw;
  uint32_t* const stages = entries + 2u * slots;  // two a warp
  uint32_t* const columns = stages + 2u * kGclWarps * stride + 32u * kGclClasses;
  const uint32_t words_at = (uint32_t)__cvta_generic_to_shared(words);
  auto visits = [&](uint32_t dir) { return dir == 0u ? J.in_visit : J.out_visit; };
  // each vertex's slot in both orders, where the words will be
  for (uint32_t dir = 0; dir < 2u; ++dir)
    for (uint32_t s = (uint32_t)tid; s < n; s += kGclThreads)
      words[dir * nw + visits(dir)[s].x] = s;
  __syncthreads();
  // the block's slots of both directions: entries (own word in the buffer read | degree << 24),
  // columns (neighbour's word | sign of J)
  for (uint32_t dir = 0; dir < 2u; ++dir) {
    const uint32_t* at = words + (dir ^ 1u) * nw;
    for (uint32_t o = (uint32_t)tid; o < mine_n * 32u; o += kGclThreads) {
      const uint32_t s = ((o >> 5) * C + r) * 32u + (o & 31u);
      const uint4 vi = s < n ? visits(dir)[s] : make_uint4(0u, 0u, 0u, 0u);
      entries[dir * slots + o] = at[vi.x] | vi.z << 24;
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
        const uint32_t d = entries[(uint32_t)warp * slots + i * 32u + last] >> 24;
        v = 32u * d;
        sh.ncls[warp][i] = (uint8_t)gcl_classes(collapse, d);
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
    const uint32_t* at = words + (dir ^ 1u) * nw;
    const uint32_t* col = dir == 0u ? J.in_col : J.out_col;
    for (uint32_t o = (uint32_t)tid; o < mine_n * 32u; o += kGclThreads) {
      const uint32_t s = ((o >> 5) * C + r) * 32u + (o & 31u);
      if (s >= n) continue;
      const uint4 vi = visits(dir)[s];
      uint32_t* c = columns + dir * col_words + sh.base[dir][o >> 5] + (o & 31u);
      for (uint32_t e = 0; e < vi.z; ++e) {
        const uint32_t v = __ldg(col + vi.y + e);
        c[32u * e] = at[v & 0x7fffffffu] | (v & 0x80000000u);
      }
    }
  }
  __syncthreads();
  // buffer 0 (sigma) is written by the step's second half, buffer 1 (sigma') by its first
  for (uint32_t s = (uint32_t)tid; s < n; s += kGclThreads)
    words[s] = J.A[(size_t)visits(order ^ 1u)[s].x * G + g];
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
  // the outcome words of pass i of a half step into one of the warp's stages
  uint32_t* const stage = stages + 2u * (uint32_t)warp * stride;
  uint32_t flip = 0u;
  auto fetch = [&](uint32_t st, uint32_t pos, uint32_t i) {
    if (i < mine_n && st < steps) {
      const uint32_t* src = mine + ((size_t)(2u * st + pos) * ptot + i * C + r) * stride;
      uint32_t* dst = stage + flip * stride;
      const uint32_t chunks16 = 8u * sh.ncls[pos ^ order][i];
      for (uint32_t c = (uint32_t)lane; c < chunks16; c += 32u)
        __pipeline_memcpy_async(dst + 4u * c, src + 4u * c, 16);
    }
    __pipeline_commit();
    flip ^= 1u;
  };
  if ((uint32_t)warp < mine_n) fetch(0u, 0u, (uint32_t)warp);
#pragma unroll 1
  for (uint32_t st = 0; st < steps; ++st) {
    const uint32_t t = t0 + st;
#pragma unroll 1
    for (uint32_t pos = 0; pos < 2u; ++pos) {
      const uint32_t typ = pos ^ order;
      const uint32_t* src = words + nw * pos;
      const uint32_t dst = words_at + 4u * nw * (pos ^ 1u);
      const bool sums = track && pos == 0u;
      if (keeper && pos == 0u && st != 0u) close(t - 1u);
      if (track && pos == 1u && fwd < 64u) {  // this block's sums to block 0
        unsigned int* s = &sh.block[0][0] + fwd;
        const uint32_t v = *s;
        *s = 0u;
        if (v != 0u)
          dsm_add(dsm_addr((uint32_t)__cvta_generic_to_shared(&sh.all[0][0] + fwd), 0u), v);
      }
      uint32_t cnt[kGclPlanes], bound = 0u, ups[6] = {0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
      for (int b = 0; b < kGclPlanes; ++b) cnt[b] = 0u;
#pragma unroll 1
      for (uint32_t i = (uint32_t)warp; i < mine_n; i += (uint32_t)kGclWarps) {
        const uint32_t local = 32u * i + (uint32_t)lane;
        const bool more = i + (uint32_t)kGclWarps < mine_n;
        fetch(more || pos == 0u ? st : st + 1u, more ? pos : pos ^ 1u,
              more ? i + (uint32_t)kGclWarps : (uint32_t)warp);
        const bool in = (i * C + r) * 32u + (uint32_t)lane < n;
        const uint32_t entry = entries[typ * slots + local];
        const uint32_t* col = columns + typ * col_words + sh.base[typ][i] + lane;
        const uint32_t d = entry >> 24;
        const uint32_t S = in ? src[entry & 0xffffffu] : 0u;
        uint32_t I[kIdx];
#pragma unroll
        for (int b = 0; b < kIdx; ++b) I[b] = 0u;
#pragma unroll 1
        for (uint32_t e = 0; e < d; e += 4) {  // four edges at a time, the last again beyond d
          uint32_t cv[4], x[4];
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k) cv[k] = col[32u * min(e + k, d - 1u)];
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k) x[k] = src[cv[k] & 0x7fffffffu];
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k)
            x[k] = e + k < d ? x[k] ^ (uint32_t)((int32_t)cv[k] >> 31) : 0u;
          const uint32_t s0 = I[0] ^ x[0] ^ x[1], ca = maj3(I[0], x[0], x[1]);
          const uint32_t cb = maj3(s0, x[2], x[3]);
          I[0] = s0 ^ x[2] ^ x[3];
          uint32_t c = maj3(I[1], ca, cb);
          I[1] ^= ca ^ cb;
#pragma unroll
          for (int b = 2; b < kIdx; ++b) {
            const uint32_t u = I[b] & c;
            I[b] ^= c;
            c = u;
          }
        }
        if (sums) {  // agreeing edges: a where sigma = +1, d - a otherwise
          uint32_t br = 0u, carry = 0u;
#pragma unroll
          for (int b = 0; b < kGclPlanes; ++b) {
            uint32_t ag = 0u;
            if (b < kIdx) {
              const uint32_t D = 0u - ((d >> b) & 1u), A = I[b];
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
        if (collapse) {  // idx = a + sigma
          uint32_t c = S;
#pragma unroll
          for (int b = 0; b < kIdx; ++b) {
            const uint32_t u = I[b] & c;
            I[b] ^= c;
            c = u;
          }
        } else {  // idx = 2 a + sigma
#pragma unroll
          for (int b = kIdx - 1; b > 0; --b) I[b] = I[b - 1];
          I[0] = S;
        }
        __pipeline_wait_prior(1);
        __syncwarp();
        const uint32_t* o = stage + flip * stride + lane;  // the stage before the one in flight
        const uint32_t nm = sh.ncls[typ][i];
        const uint32_t res = nm <= 4u    ? gcl_select<2>(o, I)
                             : nm <= 8u  ? gcl_select<3>(o, I)
                             : nm <= 16u ? gcl_select<4>(o, I)
                                         : gcl_select<5>(o, I);
        if (in) {  // to every block
          const uint32_t to = dst + 4u * ((i * C + r) * 32u + (uint32_t)lane);
#pragma unroll 4
          for (uint32_t c = 0; c < C; ++c) dsm_st(dsm_addr(to, (r + c) & (C - 1u)), res);
        }
        __syncwarp();  // before the stage is filled again
      }
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
      cl.sync();
    }
  }
  if (keeper) close(t0 + steps - 1u);
  for (uint32_t o = (uint32_t)tid; o < mine_n * 32u; o += kGclThreads) {
    const uint32_t s = ((o >> 5) * C + r) * 32u + (o & 31u);
    if (s >= n) continue;
    J.A[(size_t)visits(order ^ 1u)[s].x * G + g] = words[s];
    J.B[(size_t)visits(order)[s].x * G + g] = words[nw + s];
  }
}

// Padded column words of a block and direction.  Passes ascend by degree, so 32 x the largest
// degree of a pass is at most the edges of the next one (if that is whole), and the edges of
// every C-th pass are at most m / C and one pass; the last two passes have no whole next
// one: m / C + 3 x 32 x 31.
static uint32_t gcl_col_words(uint64_t m, uint32_t C) {
  return (uint32_t)(m / C) + kGclColSlack;
}

// Words of a pass's outcomes.
static uint32_t gcl_stride(int classes) { return 32u * (uint32_t)classes; }

static size_t gcl_bytes(uint32_t n, uint64_t m, uint32_t C, int classes) {
  const size_t chunks = (n + 31u) / 32u, slots = (chunks + C - 1u) / C * 32u;
  return (sizeof(GclShared) + 15) / 16 * 16 + 2 * 32 * chunks * sizeof(uint32_t) + 2 * slots * sizeof(uint32_t) +
         (2 * kGclWarps * gcl_stride(classes) + 32 * kGclClasses) * sizeof(uint32_t) +
         2 * (size_t)gcl_col_words(m, C) * sizeof(uint32_t);
}

static cudaError_t gcl_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, uint32_t n,
                              uint64_t m, uint32_t C, int classes, int clusters, cudaStream_t st) {
  cudaError_t e = allow_block_smem<graph_cluster_kernel>();
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(graph_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3((unsigned)clusters * C);
  cfg.blockDim = dim3(kGclThreads);
  cfg.dynamicSmemBytes = gcl_bytes(n, m, C, classes);
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaSuccess;
}

// Blocks per cluster for `clusters` groups of graphs of at most n vertices, and the microseconds
// of a step: the size of least time, a half step taking 0.8 us, 1.45 ns per vertex of a block
// and, in clusters, 0.1 ns per vertex of the graph (results stored to every block), times the
// waves of clusters (as in lattice_cluster_shape); 0: too large.  Fitted to 100 steps of n = 500 ..
// 10000; one group of n = 2000 with 1, 2, 4, 8, 16 blocks: 7.8, 5.3, 3.8, 3.5, 3.7 us a step.
int graph_cluster_shape(uint32_t n, uint64_t m, int classes, int clusters, double* us) {
  int dev = 0, max_smem = 0, best = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  for (uint32_t C = 1; C <= 16u; C *= 2) {
    const uint32_t passes = (n + C * kGclThreads - 1u) / (C * kGclThreads);
    if (gcl_bytes(n, m, C, classes) + 1024 > (size_t)max_smem || passes > (uint32_t)kGclPasses) continue;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    int fit = 0;
    if (gcl_config(cfg, attr, n, m, C, classes, clusters, nullptr) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&fit, graph_cluster_kernel, &cfg) != cudaSuccess ||
        fit < 1) {
      cudaGetLastError();
      continue;
    }
    const int wave = C == 1u || fit < 4 ? fit : fit * 3 / 4;
    const double t = 2.0 * (0.8 + 1.45e-3 * n / C + (C > 1u ? 1e-4 * n : 0.0)) *
                     ((clusters + wave - 1) / wave);
    if (best == 0 || t < *us) {
      best = (int)C;
      *us = t;
    }
  }
  return best;
}

// Bytes of the outcome words and thresholds of a step.
size_t graph_cluster_step_bytes(int classes, int clusters, uint32_t ptot) {
  return (size_t)2 * ptot * gcl_stride(classes) * sizeof(uint32_t) +
         (size_t)clusters * kGclDegs * kGclClasses * sizeof(uint2);
}

// `steps` steps (the work buffer holds that many: graph_cluster_step_bytes each) of `clusters`
// groups; off: first pass of each group among ptot.
cudaError_t launch_graph_cluster(const GraphJob* jobs, const uint32_t* off, int clusters, uint32_t n,
                                 uint64_t m, int classes, uint32_t ptot, int C, CtxDev* const* ctxs,
                                 int n_ctx, uint32_t steps, void* work, cudaStream_t st) {
  if (clusters <= 0 || steps == 0) return cudaSuccess;
  const uint32_t stride = gcl_stride(classes);
  uint32_t* const out = static_cast<uint32_t*>(work);
  uint2* const tab = reinterpret_cast<uint2*>(out + (size_t)2 * steps * ptot * stride);
  graph_thresholds_kernel<<<(unsigned)clusters * steps, 128, 0, st>>>(jobs, steps, tab);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const uint32_t per = ((n + 31u) / 32u + kAheadThreads / 32 - 1u) / (kAheadThreads / 32);
  graph_ahead_kernel<<<(unsigned)clusters * steps * 2u * per, kAheadThreads, 0, st>>>(
      jobs, off, steps, per, ptot, stride, tab, out);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  e = gcl_config(cfg, attr, n, m, (uint32_t)C, classes, clusters, st);
  if (e == cudaSuccess)
    e = cudaLaunchKernelEx(&cfg, graph_cluster_kernel, jobs, off, steps,
                           gcl_col_words(m, (uint32_t)C), ptot, stride, (const uint32_t*)out);
  if (e != cudaSuccess) return e;
  return launch_advance(ctxs, n_ctx, steps, st);
}

}  // namespace shk
