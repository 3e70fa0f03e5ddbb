// lattice_ahead.cu -- runs of small INT8 / PACKED lattices with the draws compared ahead of the run.
//
// A draw u of the heat bath depends on (seed, word, replica, step, half) alone and a threshold T on
// the field class alone, so the outcome u < T of every class is known before the configuration
// is.  lattice_ahead_kernel makes these words for a chunk of steps on the whole GPU;
// lattice_follow_kernel, one block per replica with the lattice in shared memory, only selects:
// three neighbour words, two or five three-input selects, a store and a barrier a half step, the
// words of the half steps ahead on their way through a cp.async ring.  The outcomes are those of
// all 32 planes, so the trajectory is that of the half-step kernels.
//
// A run that makes its own draws is a chain of three Philox calls and twelve planes a half step
// on one SM: 1.35 us a step at L = 64, 18.5 us at L = 352.  With the draws ahead 0.36 and 3.5 us;
// 500 recorded steps at L = 64 with state and observables read back 860 -> 288 us.
#include <cuda_pipeline_primitives.h>

#include <cstdint>

#include "lattice_device.cuh"
#include "shaken_internal.cuh"

namespace shk {

constexpr int kAheadWords = 1024;  // lane words per block of lattice_ahead_kernel
constexpr int kAheadSteps = 256;   // steps per chunk, at most
// outcome words per chunk: at most 24 MB (an allocation at the first call; at 8 MB 64 replicas of L = 64
// took 1.10 instead of 0.87 us a step), or 16 steps, and at most what stays in L2
constexpr size_t kAheadBytes = 24u << 20, kAheadMost = 48u << 20;

// Outcomes of NC field classes (6: 2 n + s; 4: n + s, thresholds equal within each) of every
// lane word of a job, for step t0 + k and position p of it: out4[((job n_steps + k) 2 + p) nw + w]
// holds classes 0..3, out2 classes 4, 5.
// Bound by integer issue: three Philox calls and 2 NC operations a plane; 29 lane words a
// nanosecond with four classes, 20 with six.
template <int NC>
__global__ void __launch_bounds__(kTile) lattice_ahead_kernel(const LatJob* __restrict__ jobs,
                                                              uint32_t t0, uint32_t n_steps,
                                                              uint32_t per, uint4* __restrict__ out4,
                                                              uint2* __restrict__ out2) {
  __shared__ LatTable tab;
  const uint32_t part = blockIdx.x % per, item = blockIdx.x / per;  // item = (job, step, position)
  const uint32_t pos = item & 1u, k = (item >> 1) % n_steps;
  const LatJob& J = jobs[(item >> 1) / n_steps];
  const CtxDev* cd = J.cd;
  const uint32_t nw = J.nwords, t = t0 + k, half = pos ^ cd->order;
  const LatTable* src = J.table;
  if (J.anneal_tables != nullptr && cd->anneal_len != 0u) {
    const uint32_t a = t - cd->anneal_t0;
    src = J.anneal_tables + min(a, cd->anneal_len - 1u);
  }
  for (uint32_t i = threadIdx.x; i < sizeof(LatTable) / 4; i += blockDim.x)
    reinterpret_cast<uint32_t*>(&tab)[i] = __ldg(reinterpret_cast<const uint32_t*>(src) + i);
  __syncthreads();
  const PhKey K = ph_key(J.key0, J.key1);
  const PhShared P = ph_shared(K, J.b, t);
  const uint32_t* frozen = J.frozen;
  auto row = [&](uint32_t j, uint32_t (&p)[NC]) {  // plane j (31 - j) of the classes
    const uint4 lo = NC == 4 ? *reinterpret_cast<const uint4*>(&tab.tmc[j][0])
                             : *reinterpret_cast<const uint4*>(&tab.tm[j][0]);
    p[0] = lo.x, p[1] = lo.y, p[2] = lo.z, p[3] = lo.w;
    if (NC == 6) {
      const uint2 hi = *reinterpret_cast<const uint2*>(&tab.tm[j][4]);
      p[NC - 2] = hi.x, p[NC - 1] = hi.y;
    }
  };
  const uint32_t end = min(nw, (part + 1u) * (uint32_t)kAheadWords);
#pragma unroll 1
  for (uint32_t w = part * kAheadWords + threadIdx.x; w < end; w += blockDim.x) {
    const uint4 W[3] = {ph_call_shared(K, P, w, half), ph_call_shared(K, P, w, half + 2u),
                        ph_call_shared(K, P, w, half + 4u)};
    uint32_t res[NC], U[NC], p[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) res[c] = 0u, U[c] = 0xffffffffu;
#pragma unroll
    for (int j = 11; j >= 0; --j) {  // twelve planes as a subtraction: borrow and equality
      const uint4& q = W[j >> 2];
      const uint32_t x = (j & 3) == 0 ? q.x : (j & 3) == 1 ? q.y : (j & 3) == 2 ? q.z : q.w;
      row((uint32_t)j, p);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        res[c] = (~x & p[c]) | (~x & res[c]) | (p[c] & res[c]);
        U[c] &= ~(x ^ p[c]);
      }
    }
    const uint32_t F = frozen != nullptr ? __ldg(frozen + w) : 0u;
    uint32_t any = 0u;
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int cls = NC == 6 || c == 0 ? c : 2 * c - 1;  // 0, 1, 3, 5: classes of c = n + s
      res[c] &= ~U[c];
      const uint32_t plus = tab.satp[cls] | F;
      res[c] = (res[c] & ~tab.satm[cls]) | plus;
      U[c] &= ~(tab.satm[cls] | plus);
      any |= U[c];
    }
#pragma unroll 1
    for (uint32_t call = 3; call < 8 && any != 0u; ++call) {
      const uint4 q = ph_call_shared(K, P, w, half + 2u * call);
      any = 0u;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t x = i == 0 ? q.x : i == 1 ? q.y : i == 2 ? q.z : q.w;
        row(4u * call + (uint32_t)i, p);
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const uint32_t diff = (x ^ p[c]) & U[c];
          res[c] |= diff & p[c];
          U[c] &= ~diff;
          if (i == 3) any |= U[c];
        }
      }
    }
    const size_t o = (size_t)item * nw + w;
    out4[o] = make_uint4(res[0], res[1], res[2], res[3]);
    if (NC == 6) out2[o] = make_uint2(res[NC - 2], res[NC - 1]);
  }
}

// n_steps steps of every job, one block each, from the outcomes in out4 / out2.  DEPTH: stages
// of the ring, one half step each; a thread loads the words it will use itself, so a stage needs
// no barrier, and takes its first word's outcomes before the barrier that ends the half step (the
// others' wait and loads are then off the chain).  With tracking the sums of sigma_t are added per step in shared memory and
// turned into best energies and series after the last step.
// Bound by the chain of a half step: barrier, neighbour loads, selects, store.
template <int ENC, int NC, int DEPTH>
__global__ void __launch_bounds__(1024, 1) lattice_follow_kernel(
    const LatJob* __restrict__ jobs, uint32_t t0, uint32_t n_steps,
    const uint4* __restrict__ out4, const uint2* __restrict__ out2) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t tot[kAheadSteps][2];  // +1 sites and disagreeing bonds of sigma_t
  __shared__ double red_H[32];
  __shared__ uint32_t red_k[32];
  const LatJob J = jobs[blockIdx.x];  // by value: the fields stay in registers
  const uint32_t nw = J.nwords, T = blockDim.x, tid = threadIdx.x;
  uint4* const ring4 = reinterpret_cast<uint4*>(smem_raw);
  uint2* const ring2 = reinterpret_cast<uint2*>(ring4 + (size_t)DEPTH * nw);
  uint32_t* const sA = reinterpret_cast<uint32_t*>(ring2 + (NC == 6 ? (size_t)DEPTH * nw : 0u));
  uint32_t* const sB = sA + nw;
  const CtxDev* cd = J.cd;
  const bool track = cd->tracking && J.sums != nullptr;
  const uint32_t order = cd->order;
  const size_t base = (size_t)blockIdx.x * n_steps * 2u * nw;
  const uint32_t halves = 2u * n_steps;
  auto fetch = [&](uint32_t hs, uint32_t s) {
    if (hs < halves) {
      for (uint32_t w = tid; w < nw; w += T) {
        const size_t o = base + (size_t)hs * nw + w;
        __pipeline_memcpy_async(ring4 + s * nw + w, out4 + o, 16);
        if (NC == 6) __pipeline_memcpy_async(ring2 + s * nw + w, out2 + o, 8);
      }
    }
    __pipeline_commit();
  };
#pragma unroll 1
  for (uint32_t hs = 0; hs + 1u < (uint32_t)DEPTH; ++hs) fetch(hs, hs);
  for (uint32_t w = tid; w < nw; w += T) sA[w] = resident_load<ENC>(J, w);
  for (uint32_t k = tid; k < 2u * n_steps; k += T) (&tot[0][0])[k] = 0u;
  __syncthreads();
  const uint32_t wpr = J.wpr;
  const bool pow2 = J.wpr_shift != 0xffffffffu;
  // words of the vertical and the horizontal neighbours of lane word w (typ 0: above and left)
  auto near = [&](uint32_t w, uint32_t typ, uint32_t& v, uint32_t& h) {
    const uint32_t c = pow2 ? (w & (wpr - 1u)) : w % wpr;
    if (typ == 0u) {
      v = w >= wpr ? w - wpr : w + nw - wpr;
      h = c == 0u ? w + wpr - 1u : w - 1u;
    } else {
      v = w + wpr < nw ? w + wpr : w + wpr - nw;
      h = c + 1u == wpr ? w - c : w + 1u;
    }
  };
  auto decide = [&](uint32_t S, uint32_t V, uint32_t H, const uint4& d, const uint2& e) {
    if (NC == 4) {
      const uint32_t c0 = V ^ H ^ S, c1 = (V & H) | (S & (V | H));
      const uint32_t lo = (c0 & d.y) | (~c0 & d.x), hi = (c0 & d.w) | (~c0 & d.z);
      return (c1 & hi) | (~c1 & lo);
    }
    const uint32_t b0 = (S & d.y) | (~S & d.x), b1 = (S & d.w) | (~S & d.z);
    const uint32_t b2 = (S & e.y) | (~S & e.x), X = V ^ H;
    const uint32_t m = (V & b2) | (~V & b0);
    return (X & b1) | (~X & m);
  };
  uint32_t s = 0;  // stage of this half step
  // the thread's first word: its neighbours' places, its spins, its outcomes of the coming half step
  uint32_t v0, h0, v1, h1, S0 = sA[tid];
  near(tid, order, v0, h0);
  near(tid, order ^ 1u, v1, h1);
  uint4 d = make_uint4(0u, 0u, 0u, 0u);
  uint2 e = make_uint2(0u, 0u);
  auto take_next = [&](uint32_t stage) {
    __pipeline_wait_prior(DEPTH - 2);
    d = ring4[stage * nw + tid];
    if (NC == 6) e = ring2[stage * nw + tid];
  };
  take_next(0u);
  auto half = [&](uint32_t hs, uint32_t pos, const uint32_t* in, uint32_t* out, uint32_t v,
                  uint32_t h) {
    const uint32_t typ = pos ^ order;
    const bool sums = track && pos == 0u;
    uint32_t acc = 0u;  // +1 sites | disagreeing bonds << 16 (at most four words a thread)
    auto one = [&](uint32_t w, uint32_t S, uint32_t V, uint32_t N, const uint4& dw,
                   const uint2& ew) {
      const uint32_t H = typ == 0u ? __funnelshift_l(N, S, 1) : __funnelshift_r(S, N, 1);
      const uint32_t r = decide(S, V, H, dw, ew);
      out[w] = r;
      if (sums)
        acc += (uint32_t)__popc(S) + ((uint32_t)(__popc(S ^ V) + __popc(S ^ H)) << 16);
      return r;
    };
    S0 = one(tid, S0, in[v], in[h], d, e);
    for (uint32_t w = tid + T; w < nw; w += T) {
      uint32_t vw, hw;
      near(w, typ, vw, hw);
      one(w, in[w], in[vw], in[hw], ring4[s * nw + w],
          NC == 6 ? ring2[s * nw + w] : make_uint2(0u, 0u));
    }
    fetch(hs + (uint32_t)DEPTH - 1u, s == 0u ? (uint32_t)DEPTH - 1u : s - 1u);
    s = s + 1u == (uint32_t)DEPTH ? 0u : s + 1u;
    take_next(s);
    if (sums) {
      acc = __reduce_add_sync(0xffffffffu, acc);
      if ((tid & 31u) == 0u) {
        atomicAdd(&tot[hs >> 1][0], acc & 0xffffu);
        atomicAdd(&tot[hs >> 1][1], acc >> 16);
      }
    }
    __syncthreads();
  };
#pragma unroll 1
  for (uint32_t hs = 0; hs < halves; hs += 2u) {
    half(hs, 0u, sA, sB, v0, h0);
    half(hs + 1u, 1u, sB, sA, v1, h1);
  }
  for (uint32_t w = tid; w < nw; w += T) {
    resident_store<ENC>(J, J.A, w, sA[w]);
    resident_store<ENC>(J, J.B, w, sB[w]);
  }
  if (!track) return;
  // H(sigma_t) of every step of the chunk (Eq. (HGibbs)); the first of the least ones
  const uint32_t r = J.rep0, series_t0 = cd->series_t0, series_cap = cd->series_cap, Rn = cd->R;
  const double Jc = cd->Jc, lamc = cd->lamc, inv_n = cd->inv_n;
  double* const series_m = cd->record ? cd->series_m : nullptr;
  double* const series_H = cd->record ? cd->series_H : nullptr;
  double best = cd->best[r];
  uint32_t at = 0xffffffffu;
  for (uint32_t k = tid; k < n_steps; k += T) {
    const double M = (double)(2 * (int)tot[k][0] - 32 * (int)nw);
    const double E = (double)(64 * (int)nw - 2 * (int)tot[k][1]);
    const double Hs = -(Jc * E) - 2.0 * lamc * M;
    if (Hs < best) best = Hs, at = k;
    const uint32_t t = t0 + k;
    if (t - series_t0 < series_cap) {
      const size_t o = (size_t)(t - series_t0) * Rn + r;
      if (series_m) series_m[o] = M * inv_n;
      if (series_H) series_H[o] = Hs;
    }
  }
  auto take = [&](double h, uint32_t k) {
    if (h < best || (h == best && k < at)) best = h, at = k;
  };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double h = __shfl_xor_sync(0xffffffffu, best, o);
    const uint32_t k = __shfl_xor_sync(0xffffffffu, at, o);
    take(h, k);
  }
  if ((tid & 31u) == 0u) red_H[tid >> 5] = best, red_k[tid >> 5] = at;
  __syncthreads();
  if (tid == 0u) {
    for (uint32_t w = 1; w < T / 32u; ++w) take(red_H[w], red_k[w]);
    if (at != 0xffffffffu) {
      cd->best[r] = best;
      cd->best_step[r] = (long long)(t0 + at);
    }
  }
}

static size_t follow_bytes(int nc, uint32_t nw, int depth) {
  return (size_t)nw * ((size_t)depth * nc * 4 + 8);
}

// Stages of the ring for lattices of nw words: 12 half steps cover the L2 latency of the smallest
// ones; the largest (L = 352: 217 KB) have room for two.  0: more than a block holds.
static int follow_depth(int nc, uint32_t nw) {
  int dev = 0, max_smem = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const size_t room = (size_t)max_smem - sizeof(uint32_t) * 2 * kAheadSteps - 1024;
  for (int depth : {12, 4, 2})
    if (follow_bytes(nc, nw, depth) <= (depth == 12 ? room / 4 : room)) return depth;
  return 0;
}

// Whether a step of n_jobs INT8 / PACKED lattices of nw words takes less time this way (both kernels)
// than with the draws made by the block itself (lattice_resident_kernel, one wave of blocks).
// Fitted to 200 steps of sides 32 .. 352 and 1 .. 2048 replicas; both sides, L = 64: 1 replica 0.36
// (ahead) against 1.35 us a step, 64 replicas 0.87 against 1.37, 256 replicas 2.6 against 1.7; L = 352: 1
// replica 3.5 against 18.5, 32 replicas 9.5 against 18.6 (six classes 13.7 against 21), 152
// replicas 35 against 18.7.
bool lattice_ahead_faster(int nc, int n_jobs, uint32_t nw) {
  if (follow_depth(nc, nw) == 0) return false;
  const double ahead = 0.45 + 8.5e-4 * nw + (nc == 4 ? 7.0e-5 : 1.0e-4) * nw * n_jobs;
  const double own = 1.2 + 1.2e-3 * nw > 4.4e-3 * nw ? 1.2 + 1.2e-3 * nw : 4.4e-3 * nw;
  return ahead < own;
}

// Steps of a chunk and bytes of its outcome words for n_jobs lattices of nw words and a run of
// n_steps; 0: a step is more than a chunk holds.
uint32_t lattice_ahead_chunk(int nc, int n_jobs, uint32_t nw, uint64_t n_steps, size_t* bytes) {
  const size_t step = (size_t)n_jobs * 2 * nw * nc * 4;
  uint64_t chunk = kAheadBytes / step;
  if (chunk < 16) chunk = kAheadMost / step < 16 ? kAheadMost / step : 16;
  if (chunk > (uint64_t)kAheadSteps) chunk = kAheadSteps;
  if (chunk > n_steps) chunk = n_steps;
  *bytes = chunk * step;
  return (uint32_t)chunk;
}

template <int ENC, int NC, int DEPTH>
static cudaError_t follow(const LatJob* jobs, int n_jobs, uint32_t nw, uint32_t t0,
                          uint32_t n_steps, const uint4* out4, const uint2* out2,
                          cudaStream_t st) {
  const size_t bytes = follow_bytes(NC, nw, DEPTH);
  const cudaError_t e = allow_block_smem<lattice_follow_kernel<ENC, NC, DEPTH>>();
  if (e != cudaSuccess) return e;
  lattice_follow_kernel<ENC, NC, DEPTH><<<n_jobs, nw < 1024u ? nw : 1024u, bytes, st>>>(jobs, t0, n_steps, out4, out2);
  return cudaGetLastError();
}

template <int NC>
static cudaError_t follow_enc(int enc, const LatJob* jobs, int n_jobs, uint32_t nw, uint32_t t0,
                              uint32_t n_steps, const uint4* out4, const uint2* out2,
                              cudaStream_t st) {
  const int depth = follow_depth(NC, nw);
  if (enc == kEncInt8) {
    if (depth == 12) return follow<kEncInt8, NC, 12>(jobs, n_jobs, nw, t0, n_steps, out4, out2, st);
    if (depth == 4) return follow<kEncInt8, NC, 4>(jobs, n_jobs, nw, t0, n_steps, out4, out2, st);
    return follow<kEncInt8, NC, 2>(jobs, n_jobs, nw, t0, n_steps, out4, out2, st);
  }
  if (depth == 12) return follow<kEncPacked, NC, 12>(jobs, n_jobs, nw, t0, n_steps, out4, out2, st);
  if (depth == 4) return follow<kEncPacked, NC, 4>(jobs, n_jobs, nw, t0, n_steps, out4, out2, st);
  return follow<kEncPacked, NC, 2>(jobs, n_jobs, nw, t0, n_steps, out4, out2, st);
}

// The outcome words of n_steps (at most a chunk) of every job.  nc: 4 where q = J (equal
// thresholds by n + s), else 6.
cudaError_t launch_lattice_ahead(int nc, const LatJob* jobs, int n_jobs, uint32_t nw, uint32_t t0,
                                 uint32_t n_steps, void* out, cudaStream_t st) {
  if (n_jobs <= 0 || n_steps == 0) return cudaSuccess;
  uint4* const out4 = static_cast<uint4*>(out);
  uint2* const out2 = reinterpret_cast<uint2*>(out4 + (size_t)n_jobs * n_steps * 2 * nw);
  const uint32_t per = (nw + kAheadWords - 1) / kAheadWords;
  const uint32_t blocks = (uint32_t)n_jobs * n_steps * 2u * per, threads = nw < kTile ? nw : kTile;
  if (nc == 4)
    lattice_ahead_kernel<4><<<blocks, threads, 0, st>>>(jobs, t0, n_steps, per, out4, out2);
  else
    lattice_ahead_kernel<6><<<blocks, threads, 0, st>>>(jobs, t0, n_steps, per, out4, out2);
  return cudaGetLastError();
}

// The same steps of INT8 / PACKED jobs from those words.
cudaError_t launch_lattice_follow(int enc, int nc, const LatJob* jobs, int n_jobs, uint32_t nw,
                                  uint32_t t0, uint32_t n_steps, const void* out,
                                  cudaStream_t st) {
  if (n_jobs <= 0 || n_steps == 0) return cudaSuccess;
  const uint4* out4 = static_cast<const uint4*>(out);
  const uint2* out2 = reinterpret_cast<const uint2*>(out4 + (size_t)n_jobs * n_steps * 2 * nw);
  return nc == 4 ? follow_enc<4>(enc, jobs, n_jobs, nw, t0, n_steps, out4, out2, st)
                 : follow_enc<6>(enc, jobs, n_jobs, nw, t0, n_steps, out4, out2, st);
}

}  // namespace shk
