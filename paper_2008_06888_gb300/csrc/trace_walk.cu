// trace_walk.cu -- the argmax traceback of q = 2 plans (Sec. III).
//
// A traceback is a serial walk: every record needs the spins that the records before it
// fixed, so its time is its chain of dependent latencies, about 1-2 us a record.  What
// does not depend on the spins is kept out of that chain: the gate tables of all chain
// records are built first, by one block per record (k_walk_tables), and while warp 0
// walks a record the other warps copy the next record and its tables to shared memory.
// A chain's replay keeps its 2^t states in the registers of warp 0 (state e in lane
// e mod 32), exchanges the replaced leg's partner with a shuffle and leaves one choice
// bit per state and gate (a ballot), so the way back through its gates is a few bit
// operations per gate.  Steps that contract many states at once (the two halves of the
// network into the root scalar) are searched by a grid (k_walk_big) between two walks.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"
#include "chain_dev.cuh"

namespace tn {

namespace {

constexpr int kWalkThreads = 128;

__device__ __forceinline__ int64_t pair64(const int32_t *w) {
  return (int64_t)((uint64_t)(uint32_t)w[0] | ((uint64_t)(uint32_t)w[1] << 32));
}

// unsigned order of values, -0 and +0 alike
__device__ __forceinline__ uint32_t value_key(float x) {
  const uint32_t u = __float_as_uint(x + 0.0f);
  return u & 0x80000000u ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ uint32_t value_key(int32_t x) { return (uint32_t)x ^ 0x80000000u; }

// A search compares each value with the best before it, so NaN (from couplings that
// overflow) is never taken but as the first state, which it stays.  nan: the key of NaN,
// chosen ahead of the load by the state's number.
__device__ __forceinline__ uint32_t state_key(float x, uint32_t nan) {
  const uint32_t key = value_key(x);
  return x != x ? nan : key;
}
__device__ __forceinline__ uint32_t state_key(int32_t x, uint32_t) { return value_key(x); }

// OR over the warp of a 64-bit word per lane (offsets are sums of distinct powers of two)
__device__ __forceinline__ int64_t or64(int64_t x) {
  const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)x);
  const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)((uint64_t)x >> 32));
  return (int64_t)((uint64_t)lo | ((uint64_t)hi << 32));
}

// Digit of a spin that an earlier record must have fixed.
__device__ __forceinline__ int digit(const int8_t *st, int spin, int *err) {
  const int d = st[spin];
  if (d == 0 || d == 1) return d;
  *err = 1;
  return 0;
}

// element offset of the fixed legs of one operand: n (spin, log2 stride) pairs
__device__ __forceinline__ int64_t fixed_offset(const int32_t *legs, int n, int lane,
                                                const int8_t *st, int *err) {
  int64_t o = 0;
  for (int i = lane; i < n; i += 32) o |= (int64_t)digit(st, legs[2 * i], err) << legs[2 * i + 1];
  return or64(o);
}

// Record layouts (32-bit words); see encode_walk.
enum { P_NFA = 1, P_NFB = 2, P_NK = 3, P_A = 4, P_B = 6, P_LEGS = 8 };
enum { C_NOUT = 1, C_T = 2, C_NTG = 3, C_IN = 4, C_LOC = 8, C_SH = 14, C_LEGS = 20 };

// offsets of contracted state k: nk (spin, shift in A, shift in B) triples, the first the
// slowest digit
__device__ __forceinline__ void k_offsets(const int32_t *kl, int nk, int64_t k, int64_t *oa,
                                          int64_t *ob) {
  int64_t a = 0, b = 0;
  for (int j = nk - 1; j >= 0; --j) {
    const int64_t d = k & 1;
    k >>= 1;
    a |= d << kl[3 * j + 1];
    b |= d << kl[3 * j + 2];
  }
  *oa = a;
  *ob = b;
}

template <typename T>
__device__ __forceinline__ void walk_plain(const int32_t *r, const T *X, int8_t *st, int *err) {
  const int lane = threadIdx.x & 31;
  const int nfa = r[P_NFA], nfb = r[P_NFB], nk = r[P_NK];
  const int32_t *la = r + P_LEGS, *lb = la + 2 * nfa, *kl = lb + 2 * nfb;
  const int64_t offB = pair64(r + P_B);
  const T *A = X + pair64(r + P_A) + fixed_offset(la, nfa, lane, st, err);
  const T *B = X + (offB >= 0 ? offB : 0) + fixed_offset(lb, nfb, lane, st, err);
  const int Ks = 1 << nk;
  uint32_t key = 0, bk = 0xffffffffu;
  for (int k = lane; k < Ks; k += 32) {
    int64_t oa, ob;
    const uint32_t nan = k == 0 ? 0xffffffffu : 0u;
    k_offsets(kl, nk, k, &oa, &ob);
    T v = A[oa];
    if (offB >= 0) v = v + B[ob];
    const uint32_t kv = state_key(v, nan);
    if (kv > key || (kv == key && (uint32_t)k < bk)) {   // the first k of the largest value
      key = kv;
      bk = (uint32_t)k;
    }
  }
  const uint32_t top = __reduce_max_sync(0xffffffffu, key);
  const uint32_t k = __reduce_min_sync(0xffffffffu, key == top ? bk : 0xffffffffu);
  if (lane < nk) st[kl[3 * lane]] = (int8_t)((k >> (nk - 1 - lane)) & 1);
  __syncwarp();
}

// The states of the chain selected by the outer spins are recomputed through the table
// gates (the sums of the forward kernels), then each replaced spin is chosen backwards.
template <typename T>
__device__ __forceinline__ void walk_chain(const int32_t *r, const T *tab, const T *X, int8_t *st,
                                           int *err, uint64_t *choice) {
  const int lane = threadIdx.x & 31;
  const int nout = r[C_NOUT], t = r[C_T], ntg = r[C_NTG];
  const int32_t *legs = r + C_LEGS, *gates = legs + 3 * nout;
  int64_t base = 0, tau = 0;
  for (int i = lane; i < nout; i += 32) {
    const int64_t d = digit(st, legs[3 * i], err);
    base |= d << legs[3 * i + 1];
    tau |= d << legs[3 * i + 2];
  }
  base = or64(base);
  tau = or64(tau);
  const int E = 1 << t;
  const T *src = X + pair64(r + C_IN) + base;
  T v[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int e = (lane + 32 * h) & (E - 1);
    int64_t o = 0;
    for (int j = 0; j < t; ++j)   // shift 63: the leg the chain adds (not in its input)
      if (((e >> j) & 1) && r[C_SH + j] < 63) o |= int64_t(1) << r[C_SH + j];
    v[h] = src[o];
  }
  for (int gi = 0; gi < ntg; ++gi) {
    const int32_t *g = gates + 4 * gi;
    const int kind = g[0] & 0xff, J = ((g[0] >> 8) & 0xff) - 1, K = ((g[0] >> 16) & 0xff) - 1;
    int f = 0;
#pragma unroll
    for (int i = 0; i < TN_TG_MAXF; ++i) f |= (int)((tau >> ((g[1] >> (8 * i)) & 0xff)) & 1) << i;
    const T *ts = tab + g[2] + 8 * f;
    if (kind == 1) {   // diagonal
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int e = lane + 32 * h;
        const int x0 = J >= 0 ? (e >> J) & 1 : 0, x1 = K >= 0 ? (e >> K) & 1 : 0;
        v[h] = v[h] + ts[x0 | (x1 << 1)];
      }
      continue;
    }
    T o[2];
    if (J < 5) {
      o[0] = __shfl_xor_sync(0xffffffffu, v[0], 1 << J);
      o[1] = __shfl_xor_sync(0xffffffffu, v[1], 1 << J);
    } else {
      o[0] = v[1];
      o[1] = v[0];
    }
    uint32_t bits[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = lane + 32 * h;
      const int x = (e >> J) & 1, k = K >= 0 ? (e >> K) & 1 : 0;
      // a contraction's outputs have digit 0; the others' values are not used
      const int xn = kind == 2 ? 0 : x;
      const T a = (x ? o[h] : v[h]) + ts[k * 4 + xn * 2], b = (x ? v[h] : o[h]) + ts[k * 4 + xn * 2 + 1];
      bits[h] = __ballot_sync(0xffffffffu, b > a);
      v[h] = max(a, b);
    }
    if (lane == 0) choice[gi] = (uint64_t)bits[0] | ((uint64_t)bits[1] << 32);
  }
  __syncwarp();
  if (lane == 0) {
    const int32_t *last = gates + 4 * (ntg - 1);
    const int cj = (last[0] & 0xff) == 2 ? ((last[0] >> 8) & 0xff) - 1 : -1;
    int x = 0;
    for (int j = 0; j < t; ++j)
      if (j != cj) x |= digit(st, r[C_LOC + j], err) << j;
    for (int gi = ntg - 1; gi >= 0; --gi) {
      const int32_t *g = gates + 4 * gi;
      if ((g[0] & 0xff) == 1) continue;
      const int J = ((g[0] >> 8) & 0xff) - 1;
      const int u = (int)((choice[gi] >> x) & 1);
      st[g[3]] = (int8_t)u;
      x = (x & ~(1 << J)) | (u << J);
    }
  }
  __syncwarp();
}

// tables of chain record blockIdx.x of this trace (instance blockIdx.y)
template <typename T>
__global__ void __launch_bounds__(128) k_walk_tables(const ChainTrace *chains, const WalkIdx *idx,
                                                     const int32_t *list, char *arena, int64_t ib) {
  T *X = reinterpret_cast<T *>(arena + blockIdx.y * ib);
  const int s = list[2 * blockIdx.x], ch = list[2 * blockIdx.x + 1];
  build_tables<T>(chains[ch].p, X, X + idx[s].tab);
}

// Walk records [0, n) of idx after assigning the spins of a pending wide record (pend,
// null if none) from the search result in `best`; `best` is cleared for the next one.
template <typename T>
__global__ void __launch_bounds__(kWalkThreads) k_walk(const int32_t *__restrict__ recs,
                                                       const WalkIdx *__restrict__ idx, int n,
                                                       const int32_t *pend, int64_t best,
                                                       char *arena, int8_t *state, int nspins,
                                                       int *err, int64_t ib) {
  arena += blockIdx.x * ib;
  state += (int64_t)blockIdx.x * nspins;
  const T *X = reinterpret_cast<const T *>(arena);
  extern __shared__ __align__(16) char wsm[];
  T *stab = reinterpret_cast<T *>(wsm);                                   // [2][tables]
  int32_t *srec = reinterpret_cast<int32_t *>(stab + 2 * kWalkTable);     // [2][record]
  uint64_t *choice = reinterpret_cast<uint64_t *>(srec + 2 * kWalkRec);
  int8_t *st = reinterpret_cast<int8_t *>(choice + TN_CHAIN_MAX_G);
  __shared__ int serr;
  if (threadIdx.x == 0) serr = 0;
  for (int i = threadIdx.x; i < nspins; i += kWalkThreads) st[i] = state[i];
  __syncthreads();
  unsigned long long *bp = best >= 0 ? reinterpret_cast<unsigned long long *>(arena + best) : nullptr;
  if (pend != nullptr && threadIdx.x < 32) {
    const uint32_t k = 0xffffffffu - (uint32_t)*bp;
    const int nk = pend[P_NK];
    const int32_t *kl = pend + P_LEGS + 2 * pend[P_NFA] + 2 * pend[P_NFB];
    if (threadIdx.x < nk) st[kl[3 * threadIdx.x]] = (int8_t)((k >> (nk - 1 - threadIdx.x)) & 1);
  }
  // copies of a record and its tables, by threads [first, kWalkThreads)
  auto fetch = [&](int s, int first) {
    const WalkIdx w = idx[s];
    int32_t *dr = srec + (s & 1) * kWalkRec;
    T *dt = stab + (s & 1) * kWalkTable;
    for (int i = threadIdx.x - first; i < w.len / 4; i += kWalkThreads - first)
      cp_async16(dr + 4 * i, recs + w.rec + 4 * i);
    for (int i = threadIdx.x - first; i < w.ntab / 4; i += kWalkThreads - first)
      cp_async16(dt + 4 * i, X + w.tab + 4 * i);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  };
  if (n > 0) fetch(0, 0);
  __syncthreads();
  for (int s = 0; s < n; ++s) {
    if (threadIdx.x < 32) {
      const int32_t *r = srec + (s & 1) * kWalkRec;
      if (r[0] == 0) walk_plain<T>(r, X, st, &serr);
      else walk_chain<T>(r, stab + (s & 1) * kWalkTable, X, st, &serr, choice);
    } else if (s + 1 < n) {
      fetch(s + 1, 32);
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < nspins; i += kWalkThreads) state[i] = st[i];
  if (threadIdx.x == 0) {
    if (serr) *err = 1;
    if (bp != nullptr) *bp = 0;
  }
}

// The first k of the largest A + B of a wide record: blocks take strided k, their
// (value, first k) keys meet in an atomicMax.
template <typename T>
__global__ void __launch_bounds__(256) k_walk_big(const int32_t *__restrict__ rec, int64_t best,
                                                  char *arena, const int8_t *state, int nspins,
                                                  int *err, int64_t ib) {
  arena += blockIdx.y * ib;
  state += (int64_t)blockIdx.y * nspins;
  const T *X = reinterpret_cast<const T *>(arena);
  const int lane = threadIdx.x & 31;
  const int nfa = rec[P_NFA], nfb = rec[P_NFB], nk = rec[P_NK];
  const int32_t *la = rec + P_LEGS, *lb = la + 2 * nfa, *kl = lb + 2 * nfb;
  __shared__ int32_t skl[3 * TN_MAX_TRACE_LEGS];
  for (int i = threadIdx.x; i < 3 * nk; i += blockDim.x) skl[i] = kl[i];
  __syncthreads();
  int bad = 0;
  const int64_t offB = pair64(rec + P_B);
  const T *A = X + pair64(rec + P_A) + fixed_offset(la, nfa, lane, state, &bad);
  const T *B = X + (offB >= 0 ? offB : 0) + fixed_offset(lb, nfb, lane, state, &bad);
  if (bad) *err = 1;
  const int64_t Ks = int64_t(1) << nk;
  unsigned long long top = 0;
#pragma unroll 4
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < Ks;
       k += (int64_t)gridDim.x * blockDim.x) {
    int64_t oa, ob;
    k_offsets(skl, nk, k, &oa, &ob);
    T v = A[oa];
    if (offB >= 0) v = v + B[ob];
    const unsigned long long key =
        ((unsigned long long)state_key(v, k == 0 ? 0xffffffffu : 0u) << 32) | (0xffffffffu - (uint32_t)k);
    top = max(top, key);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
  if (lane == 0 && top) atomicMax(reinterpret_cast<unsigned long long *>(arena + best), top);
}

template <typename T>
cudaError_t run(const WalkArgs &w, char *arena, int8_t *state, int nspins, int *err,
                const Batch &bt, cudaStream_t st) {
  if (w.nlist > 0)
    k_walk_tables<T><<<dim3((unsigned)w.nlist, bt.B), 128, 0, st>>>(w.chains, w.idx, w.list, arena,
                                                                     bt.ib);
  const size_t smem = 2 * kWalkTable * sizeof(T) + 2 * kWalkRec * 4 + TN_CHAIN_MAX_G * 8 +
                      ((size_t)nspins + 15) / 16 * 16;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_walk<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
  }
  const int32_t *pend = nullptr;
  int at = 0;
  for (int i = 0; i <= w.nbig; ++i) {
    const int end = i < w.nbig ? w.big[i] : w.n;
    k_walk<T><<<bt.B, kWalkThreads, smem, st>>>(w.recs, w.idx + at, end - at, pend, w.best, arena,
                                                state, nspins, err, bt.ib);
    if (i == w.nbig) break;
    pend = w.recs + w.big_rec[i];
    const int64_t want = std::max<int64_t>(1, w.big_k[i] / (256 * 4));
    const int64_t blocks = std::min<int64_t>(want, std::max<int64_t>(1, num_sms() * 8 / bt.B));
    k_walk_big<T><<<dim3((unsigned)blocks, bt.B), 256, 0, st>>>(pend, w.best, arena, state, nspins,
                                                                err, bt.ib);
    at = end + 1;
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_walk(Dtype dt, const WalkArgs &w, char *arena, int8_t *state, int nspins,
                        int *err, const Batch &bt, cudaStream_t st) {
  return dt == DT_F32 ? run<float>(w, arena, state, nspins, err, bt, st)
                      : run<int32_t>(w, arena, state, nspins, err, bt, st);
}

}  // namespace tn
