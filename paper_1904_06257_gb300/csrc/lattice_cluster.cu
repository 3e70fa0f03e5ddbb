// lattice_cluster.cu -- whole runs of small MULTISPIN lattices: one thread-block cluster owns one
// group of 32 replicas for n steps, the lattice in its blocks' shared memory.
//
// Block r of a cluster of C holds rows [r L / C, (r + 1) L / C) of sigma and sigma' and one
// halo row.  A dl half step reads the row above each row, an ur half step the row below, so
// between two half steps one row crosses each block boundary in one direction: the block
// that decides it also stores it into its neighbour's halo row (distributed shared
// memory), and the cluster barrier that ends the half step makes it visible.  The draws,
// thresholds and decisions are those of lattice_half_kernel, so the trajectory is the same.
// With tracking the sums of sigma_t are taken in the step's first half (bit-sliced per thread,
// 32 x 32 bit transposes per warp), gathered by the cluster's first block during the
// second, and turned into best energies and series behind the next barrier.
//
// Bound by the chain of a half step -- neighbour loads, three Philox calls, twelve planes,
// the cluster barrier: 0.5 us, and 1.9 ns a word of a block (integer issue of one SM).  A
// step at L = 64, 128 replicas takes 2.0 us in clusters of 16, 3.5 us with m and H recorded
// (the metastability curves), against 16 us of four launches (observables, two half
// steps, epilogue), and 17 us of the former one-block-per-group run without sums.
#include <cooperative_groups.h>

#include <cstdint>

#include "graph_device.cuh"  // warp_column
#include "lattice_device.cuh"
#include "shaken_internal.cuh"

namespace shk {

namespace cg = cooperative_groups;

constexpr int kClusterThreads = 512;
constexpr int kClusterMax = 16;   // blocks per cluster (above 8: non-portable size)
constexpr int kTrackPlanes = 6;   // counter planes per thread: at most 16 words, two bonds each

template <int N>
__device__ __forceinline__ void add_plane(uint32_t (&p)[N], uint32_t x, int b0) {
#pragma unroll
  for (int b = 0; b < N; ++b) {
    if (b < b0) continue;
    const uint32_t t = p[b] & x;
    p[b] ^= x;
    x = t;
  }
}

struct ClusterTotals {
  int block[2][32];   // M count and agreeing bonds of this block's rows, per replica lane
  int all[2][32];     // of the cluster (used in block 0)
};

__global__ void __launch_bounds__(kClusterThreads, 1) lattice_cluster_kernel(
    const LatJob* __restrict__ jobs, uint32_t t0, uint32_t n_steps) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ LatTable stab[2];  // by step parity (annealing: one table per step)
  __shared__ ClusterTotals tot;
  cg::cluster_group cl = cg::this_cluster();
  const uint32_t C = cl.num_blocks(), r = cl.block_rank();
  const LatJob J = jobs[blockIdx.x / C];  // by value: the fields stay in registers
  const uint32_t L = J.L, rows = L / C, own = rows * L, tid = threadIdx.x;
  const int lane = (int)(tid & 31u);
  uint32_t* buf[2] = {smem, smem + own};                        // sigma, sigma'
  uint32_t* halo[2] = {smem + 2u * own, smem + 2u * own + L};   // by position of the reading half
  const uint32_t prev = r == 0u ? C - 1u : r - 1u, next = r + 1u == C ? 0u : r + 1u;
  const CtxDev* cd = J.cd;
  const uint32_t order = cd->order, anneal_t0 = cd->anneal_t0, anneal_len = cd->anneal_len;
  const bool track = cd->tracking && J.sums != nullptr;
  const bool record = track && cd->record;
  const bool anneal = J.anneal_tables != nullptr && anneal_len != 0u;
  const uint32_t w_first = r * own;  // first lane word of the block: row r rows, column 0
  const bool pow2 = J.wpr_shift != 0xffffffffu;
  const PhKey K = ph_key(J.key0, J.key1);
  auto table_of = [&](uint32_t t) {
    if (!anneal) return J.table;
    uint32_t k = t - anneal_t0;
    if (k >= anneal_len) k = anneal_len - 1u;
    return J.anneal_tables + k;
  };
  auto stage = [&](uint32_t t) {
    const uint32_t* g = reinterpret_cast<const uint32_t*>(table_of(t));
    uint32_t* d = reinterpret_cast<uint32_t*>(&stab[t & 1u]);
    for (uint32_t k = tid; k < sizeof(LatTable) / 4; k += kClusterThreads) d[k] = __ldg(g + k);
  };
  stage(t0);
  if (!anneal) stage(t0 + 1u);
  if (tid < 64u) (&tot.block[0][0])[tid] = (&tot.all[0][0])[tid] = 0;
  const uint32_t* A = static_cast<const uint32_t*>(J.A);
  for (uint32_t o = tid; o < own; o += kClusterThreads) buf[0][o] = A[w_first + o];
  {  // the halo row of the first half step
    const uint32_t g = order == 0u ? (r * rows + L - 1u) % L : (r * rows + rows) % L;
    for (uint32_t c = tid; c < L; c += kClusterThreads) halo[0][c] = A[g * L + c];
  }
  // block 0, last warp: lane k keeps replica k's best energy (the last warps have the fewest
  // words, often none)
  const bool keeper = track && r == 0u && tid >= kClusterThreads - 32u;
  const uint32_t fwd = tid - (kClusterThreads - 96u);  // < 64: forwards the block's sums
  const double Jc = cd->Jc, lam2 = 2.0 * cd->lamc, inv_n = cd->inv_n;
  const uint32_t series_t0 = cd->series_t0, series_cap = cd->series_cap, Rn = cd->R;
  double* const series_m = record ? cd->series_m : nullptr;
  double* const series_H = record ? cd->series_H : nullptr;
  double* const best_p = cd->best;
  long long* const best_step_p = cd->best_step;
  double best = keeper ? cd->best[J.rep0 + (uint32_t)lane] : 0.0;
  cl.sync();
  auto close = [&](uint32_t t) {  // the sums of sigma_t, gathered, into best and series
    const double N = (double)L * (double)L;
    const double M = 2.0 * (double)tot.all[0][lane] - N;
    const double E = 2.0 * (double)tot.all[1][lane] - 2.0 * N;
    tot.all[0][lane] = tot.all[1][lane] = 0;
    const double H = -(Jc * E) - lam2 * M;
    const uint32_t rep = J.rep0 + (uint32_t)lane;
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
  uint32_t calls = 0;
  for (uint32_t st = 0; st < n_steps; ++st) {
    const uint32_t t = t0 + st;
    const LatTable& tab = stab[t & 1u];
    const PhShared P = ph_shared(K, J.b, t);
#pragma unroll 1
    for (uint32_t pos = 0; pos < 2u; ++pos) {
      const uint32_t typ = pos ^ order, nxt = typ ^ 1u;
      const uint32_t* in = buf[pos];
      uint32_t* out = buf[pos ^ 1u];
      const bool sums = track && pos == 0u;
      if (keeper && pos == 0u && st != 0u) close(t - 1u);
      if (track && pos == 1u && fwd < 64u) {  // this block's sums to block 0
        int* src = &tot.block[0][0] + fwd;
        const int v = *src;
        *src = 0;
        if (v != 0) atomicAdd(cl.map_shared_rank(&tot.all[0][0] + fwd, 0), v);
      }
      if (anneal && pos == 1u && st + 1u < n_steps) stage(t + 1u);
      // the row the neighbour needs next: dl (0) reads above, so the last row goes down
      uint32_t* give = cl.map_shared_rank(halo[pos ^ 1u], nxt == 0u ? next : prev);
      const uint32_t give_row = nxt == 0u ? own - L : 0u;
      uint32_t pm[kTrackPlanes - 1], pe[kTrackPlanes];
      if (sums) {
#pragma unroll
        for (int b = 0; b < kTrackPlanes; ++b) pe[b] = 0u;
#pragma unroll
        for (int b = 0; b < kTrackPlanes - 1; ++b) pm[b] = 0u;
      }
#pragma unroll 1
      for (uint32_t o = tid; o < own; o += kClusterThreads) {
        const uint32_t c = pow2 ? (o & (L - 1u)) : o % L;
        const uint32_t S = in[o];
        uint32_t V, H;
        if (typ == 0u) {
          V = o < L ? halo[pos][c] : in[o - L];
          H = in[o - c + (c == 0u ? L - 1u : c - 1u)];
        } else {
          V = o + L >= own ? halo[pos][c] : in[o + L];
          H = in[o - c + (c + 1u == L ? 0u : c + 1u)];
        }
        const uint32_t w = w_first + o;
        const uint32_t F = J.frozen != nullptr ? __ldg(J.frozen + w) : 0u;
        LaneWord Lw;
        if (tab.collapsed) {
          Lw = classify<true>(S, V, H, F, tab);
          decide_head3<true>(Lw, tab, K, P, w, typ, calls);
          decide_tail<true>(Lw, tab, K, P, w, typ, 3u, calls);
        } else {
          Lw = classify<false>(S, V, H, F, tab);
          decide_head3<false>(Lw, tab, K, P, w, typ, calls);
          decide_tail<false>(Lw, tab, K, P, w, typ, 3u, calls);
        }
        out[o] = Lw.res;
        if (o - give_row < L) give[c] = Lw.res;
        if (sums) {
          const uint32_t a = ~(S ^ V), b = ~(S ^ H);
          add_plane(pm, S, 0);
          // two bonds: sum bit and carry
          const uint32_t s = pe[0] ^ a ^ b, cy = maj3(pe[0], a, b);
          pe[0] = s;
          add_plane(pe, cy, 1);
        }
      }
      if (sums) {  // a warp's threads: per-replica counts of its planes
        __syncwarp();
        const uint32_t words = (own + kClusterThreads - 1u) / kClusterThreads;  // most per thread
        int cm = 0, ce = 0;
#pragma unroll
        for (int b = 0; b < kTrackPlanes; ++b) {
          if (b < kTrackPlanes - 1 && (words >> b) != 0u)
            cm += __popc(warp_column(pm[b], lane)) << b;
          if (((2u * words) >> b) != 0u) ce += __popc(warp_column(pe[b], lane)) << b;
        }
        if (cm) atomicAdd(&tot.block[0][lane], cm);
        if (ce) atomicAdd(&tot.block[1][lane], ce);
      }
      cl.sync();
    }
  }
  if (keeper && n_steps != 0u) close(t0 + n_steps - 1u);
  for (uint32_t o = tid; o < own; o += kClusterThreads) {
    static_cast<uint32_t*>(J.A)[w_first + o] = buf[0][o];
    static_cast<uint32_t*>(J.B)[w_first + o] = buf[1][o];
  }
  (void)calls;
}

static size_t cluster_bytes(uint32_t L, uint32_t C) {
  return ((size_t)2 * (L / C) * L + 2 * L) * sizeof(uint32_t);
}

static cudaError_t cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, uint32_t L,
                                  uint32_t C, int n_jobs, cudaStream_t st) {
  const size_t bytes = cluster_bytes(L, C);
  cudaError_t e = cudaFuncSetAttribute(lattice_cluster_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(lattice_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed,
                             1);
  if (e != cudaSuccess) return e;
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3((unsigned)n_jobs * C);
  cfg.blockDim = dim3(kClusterThreads);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaSuccess;
}

// Blocks per cluster for n_jobs groups of an L x L lattice and the microseconds of a step: the
// size of least time, a half step taking 0.5 us and 1.9 ns per word of a block, times the
// waves of clusters; 0: the lattice does not fit (shared memory, counter planes).  A wave
// is taken as three quarters of the clusters that the occupancy query allows: 16 clusters of
// 8 ran in two waves (L = 128: 17 us a step against 6 us for 4 clusters of 16).
int lattice_cluster_shape(uint32_t L, int n_jobs, double* us) {
  int dev = 0, max_smem = 0, best = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  for (uint32_t C = 1; C <= (uint32_t)kClusterMax; C *= 2) {
    const uint32_t own = L / C * L;
    if (cluster_bytes(L, C) + sizeof(LatTable) * 2 + 2048 > (size_t)max_smem) continue;
    if ((own + kClusterThreads - 1u) / kClusterThreads > 16u) continue;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    int fit = 0;
    if (cluster_config(cfg, attr, L, C, n_jobs, nullptr) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&fit, lattice_cluster_kernel, &cfg) != cudaSuccess ||
        fit < 1) {
      cudaGetLastError();
      continue;
    }
    const int wave = C == 1u || fit < 4 ? fit : fit * 3 / 4;
    const double t = 2.0 * (0.5 + 1.9e-3 * own) * ((n_jobs + wave - 1) / wave);
    if (best == 0 || t < *us) {
      best = (int)C;
      *us = t;
    }
  }
  return best;
}

cudaError_t launch_lattice_cluster(const LatJob* jobs, int n_jobs, uint32_t L, int C, uint32_t t0,
                                   uint32_t n_steps, cudaStream_t st) {
  if (n_jobs <= 0 || n_steps == 0) return cudaSuccess;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  cudaError_t e = cluster_config(cfg, attr, L, (uint32_t)C, n_jobs, st);
  if (e != cudaSuccess) return e;
  return cudaLaunchKernelEx(&cfg, lattice_cluster_kernel, jobs, t0, n_steps);
}

}  // namespace shk
