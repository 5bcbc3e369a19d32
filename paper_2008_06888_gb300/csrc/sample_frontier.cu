// sample_frontier.cu -- ground states drawn from one sweep of exact counts.
//
// Fixing the spins one at a time needs, at every step, the numbers of ground states
// that extend the fixed spins with +1 and with -1.  Those depend on the fixed spins only
// through the ones that still have neighbours to come, so one sweep from the last spin
// to the first tabulates them for every state of that frontier: value and number of the
// best completions.  A draw then reads two entries per spin.  The tables hold 12 bytes
// per state; a 12 x 12 lattice in row order has 144 of 2^12 states, 7 MB.  Counting every
// prefix of every sample as a contraction of its own instead (n + 1 dependent batches)
// took 89 ms for 16 samples of that lattice; the sweep and the draws take 0.43 ms.
//
// The counts are the same integers as those of the contractions and the random numbers
// are keyed by (seed, sample, step) as in sampler.cpp, so the samples are the same.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"
#include "modarith.cuh"
#include "sampler.h"

namespace tn {

namespace {

constexpr int kSweepThreads = 1024;
constexpr int kDrawThreads = 32;
constexpr int kChunkSteps = 128;   // steps whose records a block stages at a time
constexpr int kChunkNbs = 512;     // and neighbour entries staged with them
// Tables of up to 2^13 states are swept by one block that keeps the last table in
// shared memory (2 x 12 bytes per state) and separates the steps with a barrier (well
// under a microsecond each); wider ones get a launch per step, about 2.5 us, whose
// grid then has at least 16 blocks to spread.
constexpr int kBlockStates = 1 << 13;

struct Entry {
  int32_t x;
  uint64_t n;
};

__device__ __forceinline__ int32_t local_field(const FrontierStep &st, const FrontierNb *nb,
                                               uint32_t i) {
  int32_t z = st.h;
  for (int k = 0; k < st.nnb; ++k) z += (i >> nb[k].slot) & 1 ? -nb[k].J : nb[k].J;
  return z;
}

// (value, count) of state i: the better of the new spin's two values, counts added on a
// tie; X, N: the table behind the step
__device__ __forceinline__ Entry step_entry(const FrontierStep &st, const FrontierNb *nb,
                                            uint32_t i, const int32_t *X, const uint64_t *N) {
  const int32_t z = local_field(st, nb, i);
  const uint32_t up = i & st.keep, dn = st.slot >= 0 ? up | (1u << st.slot) : up;
  const int32_t a = X[up] + z, b = X[dn] - z;
  const uint64_t na = N[up], nb_ = N[dn];
  Entry e;
  e.x = max(a, b);
  e.n = a > b ? na : (a < b ? nb_ : addsat64(na, nb_));
  return e;
}

__global__ void k_sweep_end(int32_t *X, uint64_t *N) {
  *X = 0;
  *N = 1;
}

// one step over a grid
__global__ void __launch_bounds__(256) k_sweep_step(const FrontierStep *__restrict__ steps,
                                                    const FrontierNb *__restrict__ nbs, int t,
                                                    int32_t *__restrict__ X,
                                                    uint64_t *__restrict__ N) {
  const FrontierStep st = steps[t];
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint64_t i = blockIdx.x * blockDim.x + threadIdx.x; i < st.size; i += stride) {
    const Entry e = step_entry(st, nbs + st.nb, (uint32_t)i, X + st.next, N + st.next);
    X[st.off + i] = e.x;
    N[st.off + i] = e.n;
  }
}

// steps t1 - 1 down to t0 in one block (every table at most kBlockStates states)
__global__ void __launch_bounds__(kSweepThreads) k_sweep_block(
    const FrontierStep *__restrict__ steps, const FrontierNb *__restrict__ nbs, int t0, int t1,
    uint32_t next_size, int cap, int32_t *X, uint64_t *N) {
  extern __shared__ __align__(16) char raw[];
  uint64_t *sN = reinterpret_cast<uint64_t *>(raw);               // 2 tables of cap
  int32_t *sX = reinterpret_cast<int32_t *>(sN + 2 * (size_t)cap);
  __shared__ FrontierStep sS[kChunkSteps];
  __shared__ FrontierNb sB[kChunkNbs];
  const int64_t behind = steps[t1 - 1].next;
  for (uint32_t i = threadIdx.x; i < next_size; i += blockDim.x) {
    sX[i] = X[behind + i];
    sN[i] = N[behind + i];
  }
  int cur = 0;
  for (int hi = t1; hi > t0; hi -= kChunkSteps) {
    const int lo = max(t0, hi - kChunkSteps);
    __syncthreads();   // the steps before are done with the staged records
    for (int k = threadIdx.x; k < hi - lo; k += blockDim.x) sS[k] = steps[lo + k];
    const int b0 = steps[lo].nb, b1 = steps[hi - 1].nb + steps[hi - 1].nnb;
    const bool staged = b1 - b0 <= kChunkNbs;
    if (staged)
      for (int k = threadIdx.x; k < b1 - b0; k += blockDim.x) sB[k] = nbs[b0 + k];
    __syncthreads();
    for (int t = hi - 1; t >= lo; --t) {
      const FrontierStep &st = sS[t - lo];
      const FrontierNb *nb = staged ? sB + (st.nb - b0) : nbs + st.nb;
      const int32_t *cx = sX + cur * cap;
      const uint64_t *cn = sN + cur * cap;
      cur ^= 1;
      for (uint32_t i = threadIdx.x; i < st.size; i += blockDim.x) {
        const Entry e = step_entry(st, nb, i, cx, cn);
        sX[cur * cap + i] = e.x;
        sN[cur * cap + i] = e.n;
        X[st.off + i] = e.x;
        N[st.off + i] = e.n;
      }
      __syncthreads();
    }
  }
}

__device__ __forceinline__ uint64_t mix(uint64_t x) {   // as mix64 of sampler.cpp
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}

// One sample per thread.  Its chain is serial: the state picks two entries (loads in
// flight together), the draw picks the next state.  The first attempt's random word
// does not depend on the state and is computed while the entries load.  *err: the
// counts were inconsistent or the rejection did not end (the caller counts prefix by
// prefix then).
__global__ void __launch_bounds__(kDrawThreads) k_draw(const FrontierStep *__restrict__ steps,
                                                       const FrontierNb *__restrict__ nbs, int n,
                                                       const int32_t *__restrict__ X,
                                                       const uint64_t *__restrict__ N, int S,
                                                       uint64_t seed, int8_t *__restrict__ sigma,
                                                       int *err) {
  __shared__ FrontierStep sS[kChunkSteps];
  __shared__ FrontierNb sB[kChunkNbs];
  const int s = blockIdx.x * kDrawThreads + threadIdx.x;
  const bool live = s < S;
  const uint64_t ks = mix(mix(seed) ^ (uint64_t)s);
  const uint64_t first = mix(0);
  uint32_t state = 0;
  bool bad = false;
  for (int lo = 0; lo < n; lo += kChunkSteps) {
    const int hi = min(n, lo + kChunkSteps);
    __syncthreads();
    for (int k = threadIdx.x; k < hi - lo; k += kDrawThreads) sS[k] = steps[lo + k];
    const int b0 = steps[lo].nb, b1 = steps[hi - 1].nb + steps[hi - 1].nnb;
    const bool staged = b1 - b0 <= kChunkNbs;
    if (staged)
      for (int k = threadIdx.x; k < b1 - b0; k += kDrawThreads) sB[k] = nbs[b0 + k];
    __syncthreads();
    for (int t = lo; t < hi; ++t) {
      const FrontierStep &st = sS[t - lo];
      const FrontierNb *nb = staged ? sB + (st.nb - b0) : nbs + st.nb;
      const uint32_t up = state & st.keep, dn = st.slot >= 0 ? up | (1u << st.slot) : up;
      const int32_t xa = X[st.next + up], xb = X[st.next + dn];
      const uint64_t na = N[st.next + up], nb_ = N[st.next + dn];
      const uint64_t key = mix(ks ^ (uint64_t)t);
      uint64_t r = mix(key ^ first);
      const int32_t z = local_field(st, nb, state);
      const int32_t a = xa + z, b = xb - z;
      const uint64_t wp = a >= b ? na : 0, wm = b >= a ? nb_ : 0, tot = wp + wm;
      if (tot == 0) {
        bad = true;
        break;
      }
      const uint64_t mask = ~0ull >> __clzll((long long)tot);
      uint64_t attempt = 0;
      while ((r & mask) >= tot && attempt < 4096) {
        ++attempt;
        r = mix(key ^ mix(attempt << 16));
      }
      bad |= attempt >= 4096;
      const bool plus = (r & mask) < wp;
      state = plus ? up : dn;
      if (live) sigma[(int64_t)s * n + st.spin] = plus ? 1 : -1;
    }
  }
  if (live && bad) *err = 1;
}

}  // namespace

cudaError_t launch_frontier_sample(const FrontierPlan &p, const FrontierStep *steps,
                                   const FrontierNb *nbs, int32_t *X, uint64_t *N, int S,
                                   uint64_t seed, int8_t *sigma, int *err, int *launches,
                                   cudaStream_t st) {
  const int n = (int)p.steps.size();
  k_sweep_end<<<1, 1, 0, st>>>(X + p.elements - 1, N + p.elements - 1);
  ++*launches;
  cudaError_t e = cudaSuccess;
  for (int t = n; t > 0;) {
    const uint32_t behind = t < n ? p.steps[t].size : 1;
    int lo = t;
    if (behind <= kBlockStates)
      while (lo > 0 && p.steps[lo - 1].size <= kBlockStates) --lo;
    if (lo < t) {
      uint32_t cap = std::max<uint32_t>(behind, 2);
      for (int k = lo; k < t; ++k) cap = std::max(cap, p.steps[k].size);
      const size_t smem = (size_t)cap * 24;
      e = cudaFuncSetAttribute(k_sweep_block, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               kBlockStates * 24);
      if (e != cudaSuccess) return e;
      k_sweep_block<<<1, kSweepThreads, smem, st>>>(steps, nbs, lo, t, behind, (int)cap, X, N);
      t = lo;
    } else {
      --t;
      const int64_t need = ((int64_t)p.steps[t].size + 255) / 256;
      k_sweep_step<<<(unsigned)std::min<int64_t>(need, 8 * (int64_t)num_sms()), 256, 0, st>>>(
          steps, nbs, t, X, N);
    }
    ++*launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  k_draw<<<(S + kDrawThreads - 1) / kDrawThreads, kDrawThreads, 0, st>>>(steps, nbs, n, X, N, S,
                                                                         seed, sigma, err);
  ++*launches;
  return cudaGetLastError();
}

}  // namespace tn
