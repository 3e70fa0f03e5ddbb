// graph_obs.cu -- observables of graph contexts (energy, pair energy, magnetisation, cut) as
// per-replica sums.
//
// Integer couplings (graph_obs_kernel): every sum is a count of lanes -- edges with
// J s_x s_y = +1, edges with s_x = s_y, vertices with s = +1, ... -- so each thread, which
// owns one group word of a run of vertices, adds its words to bit-sliced counters (ten
// planes per sum, four edges at a time through full adders); a warp turns its planes into
// per-replica counts once per job (or before a counter could overflow) by 32 x 32 bit
// transposes and popcounts, the block adds its warps, and one atomic per block, replica and
// sum goes out.  Vertices of degree above kHubDeg are left to graph_obs_hub_kernel, one
// warp per (chunk of 2048 edges, group): a thread walking a hub's 10^5 edges took 20 ms.
// The group words of a vertex are read by adjacent threads (whole sectors).
// Real couplings (graph_obs_real_kernel): fp32 sums, one vertex per thread and group.
#include <atomic>
#include <cstdint>

#include "graph_device.cuh"
#include "shaken_internal.cuh"

namespace shk {

constexpr int kObsPlanes = 10;
constexpr uint32_t kObsMax = (1u << kObsPlanes) - 1u;
constexpr uint32_t kObsGroups = 64;  // groups of a job whose totals a block keeps

// A bit-sliced counter: bit k of plane b is bit b of lane k's count.
struct Counter {
  uint32_t p[kObsPlanes];
};

__device__ __forceinline__ void add_from(Counter& c, uint32_t x, int b0) {
#pragma unroll
  for (int b = 0; b < kObsPlanes; ++b) {
    if (b < b0) continue;
    const uint32_t t = c.p[b] & x;
    c.p[b] ^= x;
    x = t;
  }
}

__device__ __forceinline__ void add4(Counter& c, uint32_t x0, uint32_t x1, uint32_t x2,
                                     uint32_t x3) {
  const uint32_t s = c.p[0] ^ x0 ^ x1, ca = maj3(c.p[0], x0, x1);
  const uint32_t cb = maj3(s, x2, x3);
  c.p[0] = s ^ x2 ^ x3;
  const uint32_t cc = maj3(c.p[1], ca, cb);
  c.p[1] ^= ca ^ cb;
  add_from(c, cc, 2);
}

// Edges of one direction of vertex x against the words Y: agree (and, with the sign of J,
// agreej) count the edges with s_x = s_y (J s_x s_y = +1).
template <bool CUT>
__device__ __forceinline__ void count_edges(const uint32_t* __restrict__ col,
                                            const uint32_t* __restrict__ Y, uint32_t d, uint32_t S,
                                            uint32_t G, Counter& agreej, Counter& agree) {
#pragma unroll 1
  for (uint32_t e = 0; e < d; e += 4) {
    uint32_t cv[4], a[4], aj[4];
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i) cv[i] = __ldg(col + min(e + i, d - 1u));
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i) {
      const uint32_t w = __ldg(Y + (size_t)(cv[i] & 0x7fffffffu) * G);
      const uint32_t m = e + i < d ? 0xffffffffu : 0u;
      a[i] = ~(S ^ w) & m;
      aj[i] = (~(S ^ w) ^ (uint32_t)((int32_t)cv[i] >> 31)) & m;
    }
    add4(agreej, aj[0], aj[1], aj[2], aj[3]);
    if (CUT) add4(agree, a[0], a[1], a[2], a[3]);
  }
}

struct ObsShared {
  GraphJob J;
  unsigned int tot[5][kObsGroups][32];  // block totals by sum, group and replica lane
  unsigned int nv, din, dout;           // vertices and counted edges of the block's job range
};

// The warp's counter of sum s into the block's totals (or, for jobs of more groups than the
// block keeps, scale x the count into the sums).
__device__ __noinline__ void flush_counter(ObsShared& sh, int s, const Counter c, double* sums,
                                           int slot, double scale, int lane) {
  const GraphJob& J = sh.J;
  const uint32_t sw = J.Gp < 32u ? J.Gp : 32u;
  const uint32_t base = ((uint32_t)threadIdx.x & ~31u) & (J.Gp - 1u);
  uint32_t col[kObsPlanes];
#pragma unroll
  for (int b = 0; b < kObsPlanes; ++b) col[b] = warp_column(c.p[b], lane);
  uint32_t mask = 0u;
#pragma unroll 1
  for (uint32_t i = 0; i < 32u; i += sw) mask |= 1u << i;
#pragma unroll 1
  for (uint32_t i = 0; i < sw; ++i, mask <<= 1) {
    uint32_t v = 0u;
#pragma unroll
    for (int b = 0; b < kObsPlanes; ++b) v += (uint32_t)__popc(col[b] & mask) << b;
    const uint32_t go = base + i;
    if (go < J.Gj && v != 0u) {
      if (J.Gj <= kObsGroups)
        atomicAdd(&sh.tot[s][go][lane], v);
      else
        atomicAdd(sums + (size_t)(32u * (J.g0 + go) + (uint32_t)lane) * kNumSums + slot,
                  scale * (double)v);
    }
  }
}

// which: 0 into the step sums, 1 into the on-demand sums; full: also the pair sums.
// Counts to sums: E = 2 agreej - edges, cut = edges - agree, P1 = 2 agreej' - edges',
// P2 = 2 agree'' - n, M = 2 up - n.
__global__ void __launch_bounds__(kTile, 2) graph_obs_kernel(const GraphJob* __restrict__ jobs,
                                                             const Tile* __restrict__ tiles,
                                                             int n_tiles, int which, int full) {
  __shared__ ObsShared sh;
  pdl_enter();
  const int tid = threadIdx.x, lane = tid & 31;
  const int tb = (int)(((long long)blockIdx.x * n_tiles) / gridDim.x);
  const int te = (int)(((long long)(blockIdx.x + 1) * n_tiles) / gridDim.x);
  const GraphJob& J = sh.J;
  Counter cE, cC, cP, cM, cQ;  // agreej, agree, agreej', up, agree''
  auto clear = [](Counter& c) {
#pragma unroll
    for (int b = 0; b < kObsPlanes; ++b) c.p[b] = 0u;
  };
  auto clear_all = [&]() {
    clear(cE);
    clear(cC);
    clear(cP);
    clear(cM);
    clear(cQ);
  };
  clear_all();
  for (int i = tid; i < 5 * (int)kObsGroups * 32; i += kTile) (&sh.tot[0][0][0])[i] = 0u;
  uint32_t bound = 0u;
  int cur_job = -1;
  double* sums = nullptr;
  auto flush = [&]() {
    flush_counter(sh, 0, cE, sums, kSumE, 2.0, lane);
    flush_counter(sh, 1, cC, sums, kSumCut, -1.0, lane);
    flush_counter(sh, 3, cM, sums, kSumM, 2.0, lane);
    if (full) {
      flush_counter(sh, 2, cP, sums, kSumP1, 2.0, lane);
      flush_counter(sh, 4, cQ, sums, kSumP2, 2.0, lane);
    }
    clear_all();
    bound = 0u;
  };
  // the block's totals of the job out: sums = scale x count + offset (per block)
  auto leave = [&]() {
    flush();
    __syncthreads();
    const double nv = (double)sh.nv, di = (double)sh.din, dn = (double)sh.dout;
    const bool kept = J.Gj <= kObsGroups;
#pragma unroll 1
    for (uint32_t o = (uint32_t)tid; o < 32u * J.Gj; o += kTile) {
      double* d = sums + (size_t)(32u * J.g0 + o) * kNumSums;
      double c[5];
#pragma unroll
      for (int s = 0; s < 5; ++s) {
        c[s] = kept ? (double)(&sh.tot[s][0][0])[o] : 0.0;
        if (kept) (&sh.tot[s][0][0])[o] = 0u;
      }
      atomicAdd(d + kSumE, 2.0 * c[0] - di);
      atomicAdd(d + kSumCut, di - c[1]);
      atomicAdd(d + kSumM, 2.0 * c[3] - nv);
      if (full) {
        atomicAdd(d + kSumP1, 2.0 * c[2] - dn);
        atomicAdd(d + kSumP2, 2.0 * c[4] - nv);
      }
    }
  };
  for (int ti = tb; ti < te; ++ti) {
    const Tile tl = tiles[ti];
    if ((int)tl.job != cur_job) {
      if (cur_job >= 0) leave();
      __syncthreads();
      if (tid < (int)(sizeof(GraphJob) / 4))
        reinterpret_cast<uint32_t*>(&sh.J)[tid] =
            reinterpret_cast<const uint32_t*>(jobs + tl.job)[tid];
      if (tid == 0) sh.nv = sh.din = sh.dout = 0u;
      __syncthreads();
      cur_job = (int)tl.job;
      sums = which ? J.obs : J.sums;
    }
    const uint32_t Gp = J.Gp, G = J.G, go = (uint32_t)tid & (Gp - 1u);
    const uint32_t x = tl.w0 + (uint32_t)tid / Gp;
    const bool act = x < J.n && go < J.Gj;
    uint32_t e0 = 0u, d = 0u, o0 = 0u, od = 0u;
    if (act) {
      e0 = (uint32_t)__ldg(J.in_ptr + x);
      d = (uint32_t)__ldg(J.in_ptr + x + 1) - e0;
      if (d > kHubDeg) d = 0u;
      if (full) {
        o0 = (uint32_t)__ldg(J.out_ptr + x);
        od = (uint32_t)__ldg(J.out_ptr + x + 1) - o0;
        if (od > kHubDeg) od = 0u;
      }
    }
    const uint32_t most = __reduce_max_sync(0xffffffffu, max(max(d, od), 1u));
    if (bound + most > kObsMax) flush();
    bound += most;
    const bool one = act && go == 0u;  // a vertex's edges count once
    const uint32_t sd = __reduce_add_sync(0xffffffffu, one ? d : 0u);
    const uint32_t so = __reduce_add_sync(0xffffffffu, one ? od : 0u);
    const uint32_t nv = (uint32_t)__popc(__ballot_sync(0xffffffffu, one));
    if (lane == 0) {
      if (nv) atomicAdd(&sh.nv, nv);
      if (sd) atomicAdd(&sh.din, sd);
      if (so) atomicAdd(&sh.dout, so);
    }
    if (act) {
      const uint32_t g = J.g0 + go;
      const uint32_t S = J.A[(size_t)x * G + g];
      add_from(cM, S, 0);
      count_edges<true>(J.in_col + e0, J.A + g, d, S, G, cE, cC);
      if (full) {
        add_from(cQ, ~(S ^ J.B[(size_t)x * G + g]), 0);
        count_edges<false>(J.out_col + o0, J.B + g, od, S, G, cP, cC);
      }
    }
  }
  if (cur_job >= 0) leave();
}

// Edge sums of the vertices of degree above kHubDeg, one warp per (chunk of kHubChunk edges,
// group): lane l takes edges e0 + l, e0 + l + 32, ... into byte counters (at most 64
// each), a transposing butterfly gives lane k replica k's counts.
__global__ void __launch_bounds__(kTile) graph_obs_hub_kernel(
    const GraphJob* __restrict__ jobs, const HubItem* __restrict__ items,
    const uint32_t* __restrict__ unit_item, int n_units, int which, int full) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int u = blockIdx.x * (kTile / 32) + (threadIdx.x >> 5);
  if (u >= n_units) return;  // the whole warp
  const HubItem it = items[unit_item[u]];
  if (it.dir != 0u && !full) return;
  const GraphJob& J = jobs[it.job];
  const uint32_t g = J.g0 + (uint32_t)u - it.ubase, G = J.G;
  const uint32_t* col = it.dir == 0u ? J.in_col : J.out_col;
  const uint32_t* Y = it.dir == 0u ? J.A : J.B;  // in-edges: sigma, out-edges: sigma'
  const uint32_t S = J.A[(size_t)it.x * G + g];
  uint32_t Cj[8], Ca[8];
#pragma unroll
  for (int m = 0; m < 8; ++m) Cj[m] = Ca[m] = 0u;
  for (uint32_t e = it.e0 + (uint32_t)lane; e < it.e1; e += 32u) {
    const uint32_t cv = __ldg(col + e);
    const uint32_t a = ~(S ^ __ldg(Y + (size_t)(cv & 0x7fffffffu) * G + g));
    const uint32_t aj = a ^ (uint32_t)((int32_t)cv >> 31);
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      Cj[m] += (aj >> m) & 0x01010101u;
      Ca[m] += (a >> m) & 0x01010101u;
    }
  }
  uint32_t v[32];
#pragma unroll
  for (int k = 0; k < 32; ++k)  // both counts in one word (at most 2048 each)
    v[k] = ((Cj[k & 7] >> (8 * (k >> 3))) & 0xFFu) | (((Ca[k & 7] >> (8 * (k >> 3))) & 0xFFu) << 16);
  const uint32_t t = warp_transpose_sum(v, lane);
  const double ne = (double)(it.e1 - it.e0);
  double* d = (which ? J.obs : J.sums) + (size_t)(32u * g + (uint32_t)lane) * kNumSums;
  atomicAdd(d + (it.dir == 0u ? kSumE : kSumP1), 2.0 * (double)(t & 0xFFFFu) - ne);
  if (it.dir == 0u) atomicAdd(d + kSumCut, ne - (double)(t >> 16));
}

// ------------------------------------------------------------------ real couplings, fields
// Jobs of one group each (Gj = 1); tiles of kTile vertices in index order, one vertex per
// thread.  Sums of the fields lambda_x sigma_x: fp32 over the warp's 32 vertices by a
// transposing butterfly, fp64 beyond.
__device__ __forceinline__ double field_sum(uint32_t S, float lam, int lane) {
  float v[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) v[k] = ((S >> k) & 1u) ? lam : -lam;
  return (double)warp_transpose_sum(v, lane);
}

// Block totals of the listed sums, one atomic per replica and sum.
template <int N>
__device__ __forceinline__ void block_out(double (&red)[kTile / 32][32][N], const double (&acc)[N],
                                          const int (&slot)[N], double* dst) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < N; ++q) red[warp][lane][q] = acc[q];
  __syncthreads();
  if (threadIdx.x < 32) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
      if (slot[q] < 0) continue;
      double s = 0.0;
      for (int wv = 0; wv < kTile / 32; ++wv) s += red[wv][threadIdx.x][q];
      if (s != 0.0) atomicAdd(dst + (size_t)threadIdx.x * kNumSums + slot[q], s);
    }
  }
  __syncthreads();
}

// LS and LS2 of integer-coupling graphs with fields.
__global__ void __launch_bounds__(kTile) graph_obs_field_kernel(const GraphJob* __restrict__ jobs,
                                                                const Tile* __restrict__ tiles,
                                                                int n_tiles, int which, int full) {
  __shared__ double red[kTile / 32][32][2];
  pdl_enter();
  const int lane = threadIdx.x & 31;
  for (int ti = blockIdx.x; ti < n_tiles; ti += gridDim.x) {
    const Tile tl = tiles[ti];
    const GraphJob& J = jobs[tl.job];
    if (J.lambda == nullptr && J.lambda_c == 0.0f) continue;  // the whole block
    const uint32_t x = tl.w0 + (uint32_t)threadIdx.x;
    const bool act = x < J.n;
    const size_t at = (size_t)x * J.G + J.g0;
    const float lam = act ? (J.lambda != nullptr ? J.lambda[x] : J.lambda_c) : 0.0f;
    const double acc[2] = {field_sum(act ? J.A[at] : 0u, lam, lane),
                           full ? field_sum(act ? J.B[at] : 0u, lam, lane) : 0.0};
    const int slot[2] = {kSumLS, full ? (int)kSumLS2 : -1};
    block_out<2>(red, acc, slot, (which ? J.obs : J.sums) + (size_t)32 * J.g0 * kNumSums);
  }
}

// Sum over the CSR edges (x -> y) of the warp's 32 vertices (thread t: vertex x of lane t) of
// J_xy s_x s_y, s_y from Y, for lane k's replica, and (if want_cut) the number of those
// edges with s_x != s_y.  A thread's edges are read four at a time, the loads of the four
// independent of one another.
__device__ __forceinline__ void obs_edges_real(const int32_t* ptr, const uint32_t* col,
                                               const float* Jr, const uint32_t* Y, uint32_t x,
                                               bool act, uint32_t S, uint32_t G, uint32_t g,
                                               bool want_cut, int lane, double& esum,
                                               double& cut) {
  const int e0 = act ? ptr[x] : 0;
  const int d = act ? ptr[x + 1] - e0 : 0;
  const int dmax = __reduce_max_sync(0xffffffffu, d);
  const int dsum = __reduce_add_sync(0xffffffffu, d);
  long long ca = 0;
  float fv[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) fv[k] = 0.0f;
  for (int base = 0; base < dmax; base += 1020) {
    Counter pa;
#pragma unroll
    for (int b = 0; b < kObsPlanes; ++b) pa.p[b] = 0u;
    const int hi = min(d, base + 1020);
    for (int e = base; e < hi; e += 4) {
      uint32_t cv[4], w[4], a[4];
      float Jv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) cv[i] = e + i < hi ? __ldg(col + e0 + e + i) : 0u;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        w[i] = e + i < hi ? __ldg(Y + (size_t)(cv[i] & 0x7fffffffu) * G + g) : 0u;
        Jv[i] = e + i < hi ? __ldg(Jr + e0 + e + i) : 0.0f;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i] = 0u;
        if (e + i < hi) {
          a[i] = ~(S ^ w[i]);
#pragma unroll
          for (int k = 0; k < 32; ++k) fv[k] += ((a[i] >> k) & 1u) ? Jv[i] : -Jv[i];
        }
      }
      if (want_cut) add4(pa, a[0], a[1], a[2], a[3]);
    }
    if (want_cut) {
#pragma unroll
      for (int b = 0; b < kObsPlanes; ++b) ca += (long long)warp_column_count(pa.p[b], lane) << b;
    }
  }
  esum = (double)warp_transpose_sum(fv, lane);
  cut = want_cut ? (double)(dsum - ca) : 0.0;
}

__global__ void __launch_bounds__(kTile) graph_obs_real_kernel(const GraphJob* __restrict__ jobs,
                                                               const Tile* __restrict__ tiles,
                                                               int n_tiles, int which, int full) {
  __shared__ double red[kTile / 32][32][7];
  pdl_enter();
  const int lane = threadIdx.x & 31;
  for (int ti = blockIdx.x; ti < n_tiles; ti += gridDim.x) {
    const Tile tl = tiles[ti];
    const GraphJob& J = jobs[tl.job];
    const uint32_t G = J.G, g = J.g0;
    const uint32_t x = tl.w0 + (uint32_t)threadIdx.x;
    const bool act = x < J.n;
    const uint32_t am = act ? 0xffffffffu : 0u;
    const uint32_t S = act ? J.A[(size_t)x * G + g] : 0u;
    const uint32_t S2 = (act && full) ? J.B[(size_t)x * G + g] : 0u;
    const float lam = act ? (J.lambda != nullptr ? J.lambda[x] : J.lambda_c) : 0.0f;
    const int nact = __popc(__ballot_sync(0xffffffffu, act));
    double acc[7] = {0, 0, 0, 0, 0, 0, 0};  // M, LS, E, cut, P2, LS2, P1
    acc[0] = (double)(2 * warp_column_count(S & am, lane) - nact);
    acc[1] = field_sum(S, lam, lane);
    obs_edges_real(J.in_ptr, J.in_col, J.in_J, J.A, x, act, S, G, g, true, lane, acc[2], acc[3]);
    if (full) {
      acc[4] = (double)(2 * warp_column_count(~(S ^ S2) & am, lane) - nact);
      acc[5] = field_sum(S2, lam, lane);
      double unused;
      obs_edges_real(J.out_ptr, J.out_col, J.out_J, J.B, x, act, S, G, g, false, lane, acc[6],
                     unused);
    }
    const int f = full ? 0 : -8;  // negative: not written
    const int slot[7] = {kSumM, kSumLS, kSumE, kSumCut, kSumP2 + f, kSumLS2 + f, kSumP1 + f};
    block_out<7>(red, acc, slot, (which ? J.obs : J.sums) + (size_t)32 * g * kNumSums);
  }
}

// ------------------------------------------------------------------ launchers
static int sm_count() {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Integer couplings: edge and spin counts over the half-step jobs, then the hubs' edges.
cudaError_t launch_graph_obs(const GraphJob* jobs, const Tile* tiles, int n_tiles,
                             const HubItem* hub_items, const uint32_t* hub_units, int n_hub_units,
                             int which, int full, cudaStream_t st) {
  if (n_tiles <= 0) return cudaSuccess;
  static std::atomic<int> occ{0};
  int o = occ.load();
  if (o == 0) {
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, graph_obs_kernel, kTile, 0);
    occ = o = o > 0 ? o : 1;
  }
  const int grid = n_tiles < o * sm_count() ? n_tiles : o * sm_count();
  cudaError_t e = launch_dependent(graph_obs_kernel, dim3(grid), dim3(kTile), 0, st, jobs, tiles,
                                   n_tiles, which, full);
  if (e != cudaSuccess || n_hub_units <= 0) return e;
  constexpr int per = kTile / 32;
  return launch_dependent(graph_obs_hub_kernel, dim3((n_hub_units + per - 1) / per), dim3(kTile),
                          0, st, jobs, hub_items, hub_units, n_hub_units, which, full);
}

// Per-group jobs: everything for real couplings, the field sums for integer ones.
cudaError_t launch_graph_obs_group(bool integer, const GraphJob* jobs, const Tile* tiles,
                                   int n_tiles, int which, int full, cudaStream_t st) {
  if (n_tiles <= 0) return cudaSuccess;
  const int most = 4 * sm_count();
  const dim3 grid(n_tiles < most ? n_tiles : most);
  return launch_dependent(integer ? graph_obs_field_kernel : graph_obs_real_kernel, grid,
                          dim3(kTile), 0, st, jobs, tiles, n_tiles, which, full);
}

}  // namespace shk
