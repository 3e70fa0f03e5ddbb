// lattice_cluster.cu -- whole runs of small MULTISPIN lattices: one thread-block cluster owns one
// group of 32 replicas for a chunk of steps, the lattice in its blocks' shared memory.
//
// Block r of a cluster of C holds rows [r L / C, (r + 1) L / C) of sigma and sigma' and one
// halo row.  A dl half step reads the row above each row, an ur half step the row below, so
// between two half steps one row crosses each block boundary in one direction: the block
// that decides it also stores it into its neighbour's halo row (distributed shared
// memory), and the cluster barrier that ends the half step makes it visible.  The draws,
// thresholds and decisions are those of lattice_half_kernel, so the trajectory is the same; the three
// Philox calls of a thread's first word of the next half step are made between arriving at the
// barrier and waiting for it.  With tracking the sums of sigma_t are taken in the step's first
// half, by the warps that have the fewest words to decide (bit-sliced per thread, 32 x 32 bit
// transposes per warp), added up in the cluster's first block during the second, and turned into
// best energies and series after the last step.
//
// Bound by the chain of a half step -- neighbour loads, twelve planes, the cluster barrier with the
// next draws -- and 1.9 ns a word of a block (integer issue of one SM).  100 steps at L = 64, 128
// replicas (clusters of 16): 2.3 us a step, 3.2 with m and H recorded; 2.7 and 4.2 us with the
// draws behind the barrier and the energies evaluated on the way, 16 us as four launches
// (observables, two half steps, epilogue).  Outcome words made ahead by the whole GPU, as for the
// small INT8 lattices, pay for one group only (L = 128: 2.8 against 4.8 us; 16 groups at
// L = 64: 4.9 against 4.7 us): a step of many groups is that kernel's time.
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

__global__ void __launch_bounds__(kClusterThreads, 1) lattice_cluster_kernel(
    const LatJob* __restrict__ jobs, uint32_t t0, uint32_t n_steps) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ LatTable stab[2];  // by step parity (annealing: one table per step)
  __shared__ int part[2][32];  // +1 sites and agreeing bonds of this block's rows, per replica lane
  __shared__ double red_H[kClusterThreads / 32][32];
  __shared__ uint32_t red_k[kClusterThreads / 32][32];
  cg::cluster_group cl = cg::this_cluster();
  const uint32_t C = cl.num_blocks(), r = cl.block_rank();
  const LatJob J = jobs[blockIdx.x / C];  // by value: the fields stay in registers
  const uint32_t L = J.L, rows = L / C, own = rows * L, tid = threadIdx.x;
  const int lane = (int)(tid & 31u);
  // smem: sigma, sigma', two halo rows (by position of the reading half step), sums
  int* const all = reinterpret_cast<int*>(smem + 2u * own + 2u * L);  // [step][2][32], in block 0
  const uint32_t prev = r == 0u ? C - 1u : r - 1u, next = r + 1u == C ? 0u : r + 1u;
  const CtxDev* cd = J.cd;
  const uint32_t order = cd->order, anneal_t0 = cd->anneal_t0, anneal_len = cd->anneal_len;
  const bool track = cd->tracking && J.sums != nullptr;
  const bool anneal = J.anneal_tables != nullptr && anneal_len != 0u;
  const uint32_t w_first = r * own;  // first lane word of the block: row r rows, column 0
  const bool pow2 = J.wpr_shift != 0xffffffffu;
  const PhKey K = ph_key(J.key0, J.key1);
  auto stage = [&](uint32_t t) {
    const uint32_t k = min(t - anneal_t0, anneal_len - 1u);
    const uint32_t* g = reinterpret_cast<const uint32_t*>(anneal ? J.anneal_tables + k : J.table);
    uint32_t* d = reinterpret_cast<uint32_t*>(&stab[t & 1u]);
    for (uint32_t i = tid; i < sizeof(LatTable) / 4; i += kClusterThreads) d[i] = __ldg(g + i);
  };
  stage(t0);
  if (!anneal) stage(t0 + 1u);
  if (tid < 64u) (&part[0][0])[tid] = 0;
  if (track && r == 0u)
    for (uint32_t k = tid; k < 64u * n_steps; k += kClusterThreads) all[k] = 0;
  const uint32_t* A = static_cast<const uint32_t*>(J.A);
  for (uint32_t o = tid; o < own; o += kClusterThreads) smem[o] = A[w_first + o];
  {  // the halo row of the first half step
    const uint32_t g = order == 0u ? (r * rows + L - 1u) % L : (r * rows + rows) % L;
    for (uint32_t c = tid; c < L; c += kClusterThreads) smem[2u * own + c] = A[g * L + c];
  }
  cl.sync();
  const uint32_t most = (own + kClusterThreads - 1u) / kClusterThreads;  // words per thread
  const uint32_t fwd = tid - (kClusterThreads - 64u);  // the last warps: the fewest words
  PhShared P = ph_shared(K, J.b, t0);
  uint4 W[3];  // the calls of the thread's first word
  auto call_ahead = [&](uint32_t typ) {
    if (tid >= own) return;
#pragma unroll
    for (uint32_t k = 0; k < 3u; ++k) W[k] = ph_call_shared(K, P, w_first + tid, typ + 2u * k);
  };
  call_ahead(order);
#pragma unroll 1
  for (uint32_t hs = 0; hs < 2u * n_steps; ++hs) {
    const uint32_t pos = hs & 1u, typ = pos ^ order, nxt = typ ^ 1u, t = t0 + (hs >> 1);
    const LatTable& tab = stab[t & 1u];
    const uint32_t* in = smem + pos * own;
    uint32_t* out = smem + (pos ^ 1u) * own;
    const uint32_t* halo = smem + 2u * own + pos * L;
    if (track && pos == 1u && fwd < 64u) {  // this block's sums to block 0
      int* src = &part[0][0] + fwd;
      const int v = *src;
      *src = 0;
      if (v != 0) atomicAdd(cl.map_shared_rank(all + 64u * (hs >> 1) + fwd, 0), v);
    }
    if (anneal && pos == 1u) stage(t + 1u);
    // the row the neighbour needs next: dl (0) reads above, so the last row goes down
    uint32_t* give = cl.map_shared_rank(smem + 2u * own + (pos ^ 1u) * L, nxt == 0u ? next : prev);
    const uint32_t give_row = nxt == 0u ? own - L : 0u;
    auto words = [&](uint32_t o, uint32_t& c, uint32_t& S, uint32_t& V, uint32_t& H) {
      c = pow2 ? (o & (L - 1u)) : o % L;
      S = in[o];
      if (typ == 0u) {
        V = o < L ? halo[c] : in[o - L];
        H = in[o - c + (c == 0u ? L - 1u : c - 1u)];
      } else {
        V = o + L >= own ? halo[c] : in[o + L];
        H = in[o - c + (c + 1u == L ? 0u : c + 1u)];
      }
    };
#pragma unroll 1
    for (uint32_t o = tid; o < own; o += kClusterThreads) {
      uint32_t c, S, V, H;
      words(o, c, S, V, H);
      const uint32_t w = w_first + o;
      const uint32_t F = J.frozen != nullptr ? __ldg(J.frozen + w) : 0u;
      if (o != tid) {
#pragma unroll
        for (uint32_t k = 0; k < 3u; ++k) W[k] = ph_call_shared(K, P, w, typ + 2u * k);
      }
      LaneWord Lw;
      if (tab.collapsed) {
        Lw = classify<true>(S, V, H, F, tab);
        decide_planes3<true>(Lw, tab, W);
        decide_tail<true>(Lw, tab, K, P, w, typ, 3u);
      } else {
        Lw = classify<false>(S, V, H, F, tab);
        decide_planes3<false>(Lw, tab, W);
        decide_tail<false>(Lw, tab, K, P, w, typ, 3u);
      }
      const uint32_t res = Lw.res;
      out[o] = res;
      if (o - give_row < L) give[c] = res;
    }
    if (track && pos == 0u && kClusterThreads - 32u - (tid & ~31u) < own) {
      // sums of sigma_t, the last warps first; a warp's threads: per-replica counts of planes
      uint32_t pm[kTrackPlanes - 1], pe[kTrackPlanes];
#pragma unroll
      for (int b = 0; b < kTrackPlanes; ++b) pe[b] = 0u;
#pragma unroll
      for (int b = 0; b < kTrackPlanes - 1; ++b) pm[b] = 0u;
#pragma unroll 1
      for (uint32_t o = kClusterThreads - 1u - tid; o < own; o += kClusterThreads) {
        uint32_t c, S, V, H;
        words(o, c, S, V, H);
        const uint32_t a = ~(S ^ V), b = ~(S ^ H);
        add_plane(pm, S, 0);
        // two bonds: sum bit and carry
        const uint32_t x = pe[0] ^ a ^ b, cy = maj3(pe[0], a, b);
        pe[0] = x;
        add_plane(pe, cy, 1);
      }
      __syncwarp();
      int cm = 0, ce = 0;
#pragma unroll
      for (int b = 0; b < kTrackPlanes; ++b) {
        if (b < kTrackPlanes - 1 && (most >> b) != 0u)
          cm += __popc(warp_column(pm[b], lane)) << b;
        if (((2u * most) >> b) != 0u) ce += __popc(warp_column(pe[b], lane)) << b;
      }
      if (cm) atomicAdd(&part[0][lane], cm);
      if (ce) atomicAdd(&part[1][lane], ce);
    }
    cl.barrier_arrive();
    if (pos == 1u) P = ph_shared(K, J.b, t + 1u);
    call_ahead(nxt);  // of the next half step (the next step begins with the other type)
    cl.barrier_wait();
  }
  for (uint32_t o = tid; o < own; o += kClusterThreads) {
    static_cast<uint32_t*>(J.A)[w_first + o] = smem[o];
    static_cast<uint32_t*>(J.B)[w_first + o] = smem[own + o];
  }
  if (!track || r != 0u) return;
  // block 0: m and H of every step of the chunk, lane k replica k; the first of the least H
  const double Jc = cd->Jc, lam2 = 2.0 * cd->lamc, inv_n = cd->inv_n;
  const uint32_t series_t0 = cd->series_t0, series_cap = cd->series_cap, Rn = cd->R;
  double* const series_m = cd->record ? cd->series_m : nullptr;
  double* const series_H = cd->record ? cd->series_H : nullptr;
  const uint32_t rep = J.rep0 + (uint32_t)lane, warp = tid >> 5;
  double best = cd->best[rep];
  uint32_t at = 0xffffffffu;
  for (uint32_t k = warp; k < n_steps; k += kClusterThreads / 32) {
    const double N = (double)L * (double)L;
    const double M = 2.0 * (double)all[64u * k + (uint32_t)lane] - N;
    const double E = 2.0 * (double)all[64u * k + 32u + (uint32_t)lane] - 2.0 * N;
    const double H = -(Jc * E) - lam2 * M;
    if (H < best) best = H, at = k;
    const uint32_t t = t0 + k;
    if (t - series_t0 < series_cap) {
      const size_t o = (size_t)(t - series_t0) * Rn + rep;
      if (series_m) series_m[o] = M * inv_n;
      if (series_H) series_H[o] = H;
    }
  }
  red_H[warp][lane] = best;
  red_k[warp][lane] = at;
  __syncthreads();
  if (warp != 0u) return;
  for (uint32_t w = 1; w < kClusterThreads / 32; ++w) {
    const double h = red_H[w][lane];
    const uint32_t k = red_k[w][lane];
    if (h < best || (h == best && k < at)) best = h, at = k;
  }
  if (at != 0xffffffffu) {
    cd->best[rep] = best;
    cd->best_step[rep] = (long long)(t0 + at);
  }
}

static size_t cluster_bytes(uint32_t L, uint32_t C) {
  return ((size_t)2 * (L / C) * L + 2 * L + (size_t)kClusterSteps * 64) * sizeof(uint32_t);
}

static cudaError_t cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, uint32_t L,
                                  uint32_t C, int n_jobs, cudaStream_t st) {
  cudaError_t e = allow_block_smem<lattice_cluster_kernel>();
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(lattice_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed,
                             1);
  if (e != cudaSuccess) return e;
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3((unsigned)n_jobs * C);
  cfg.blockDim = dim3(kClusterThreads);
  cfg.dynamicSmemBytes = cluster_bytes(L, C);
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
    if (cluster_bytes(L, C) + sizeof(LatTable) * 2 + 8192 > (size_t)max_smem) continue;
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

// n_steps of every group, at most kClusterSteps.
cudaError_t launch_lattice_cluster(const LatJob* jobs, int n_jobs, uint32_t L, int C, uint32_t t0,
                                   uint32_t n_steps, cudaStream_t st) {
  if (n_jobs <= 0 || n_steps == 0) return cudaSuccess;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[1];
  const cudaError_t e = cluster_config(cfg, attr, L, (uint32_t)C, n_jobs, st);
  return e != cudaSuccess ? e
                          : cudaLaunchKernelEx(&cfg, lattice_cluster_kernel, jobs, t0, n_steps);
}

}  // namespace shk
