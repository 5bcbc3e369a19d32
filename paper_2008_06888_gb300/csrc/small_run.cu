// small_run.cu -- runs of small contraction steps in one launch.
//
// A contraction plan starts (and ends) with many steps on tensors of a few elements:
// merging the bond tensors around a spin, growing the state from nothing.  Each takes
// about 2 us as a kernel of its own, all of it launch and drain.  Here one block per
// instance runs a whole list of them: steps are sorted by dependency level, the
// elements of a level's outputs are spread over the block's threads, and a barrier
// separates the levels (an output written before it is read after it by the same
// block).  A level costs its chain of dependent loads, so the leaves and the outputs that
// later levels read stay in shared memory (as far as kSmallScratch elements go; the others
// are read back through L2) and a level's items are decoded while the one before runs.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "modarith.cuh"

namespace tn {

namespace {

constexpr int kSmallThreads = 512;
// words of a body before its digit and offset tables
enum { W_A = 0, W_B = 2, W_C = 4, W_NA = 6, W_NB = 8, W_NC = 10, W_SEG = 12, W_K = 13, W_N = 14,
       W_FLAGS = 15, W_SA = 16, W_SB = 17, W_SC = 18, W_TAB = 19 };
enum { F_UNIT = 1, F_KEEP = 2, F_LOW = 4 };

__device__ __forceinline__ int64_t word64(const int32_t *w) {
  return (int64_t)((uint64_t)(uint32_t)w[0] | ((uint64_t)(uint32_t)w[1] << 32));
}

// What a thread does for one output: its operands, terms and destinations.
template <typename T>
struct Item {
  const T *A, *B;                // B: nullptr when there is none
  const uint64_t *nA, *nB;       // nB: nullptr when B's counts are all 1
  const int32_t *kt;             // (kA, kB) of each k
  int Ks;
  int flags;
  T *C, *sC;                     // global and staged copy (either may be nullptr)
  uint64_t *nC, *snC;
};

template <typename T, bool CNT>
__global__ void __launch_bounds__(kSmallThreads) k_small(const int32_t *__restrict__ desc,
                                                         int words, int scratch, char *arena,
                                                         int64_t ib) {
  extern __shared__ __align__(16) int32_t sd[];
  uint64_t *sN = reinterpret_cast<uint64_t *>(sd + words);            // CNT: [scratch]
  T *sX = reinterpret_cast<T *>(sN + (CNT ? scratch : 0));            // [scratch]
  arena += blockIdx.x * ib;
  T *X = reinterpret_cast<T *>(arena);
  uint64_t *N = reinterpret_cast<uint64_t *>(arena);
#pragma unroll 4
  for (int i = threadIdx.x; i < words / 4; i += kSmallThreads)
    reinterpret_cast<int4 *>(sd)[i] = reinterpret_cast<const int4 *>(desc)[i];
  __syncthreads();
  const int nops = sd[0], nlev = sd[1];
  const int32_t *lev = sd + 2, *tot = lev + nlev + 1, *first = tot + nlev, *body = first + nops;
  auto decode = [&](int l, int i) {
    int lo = lev[l], hi = lev[l + 1] - 1;   // the op whose outputs hold i
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (first[mid] <= i) lo = mid; else hi = mid - 1;
    }
    const int32_t *b = sd + body[lo];
    const int out = i - first[lo];
    const int nseg = b[W_SEG], Ks = b[W_K], Ns = b[W_N];
    const int32_t *seg = b + W_TAB;              // (size, sA, sB) of each digit
    Item<T> w;
    w.kt = seg + 3 * nseg;
    w.Ks = Ks;
    const int32_t *nt = w.kt + 2 * Ks;           // nB of each n
    int r = out, oa = 0, ob = 0;
    if (Ns > 1) {
      ob = nt[r % Ns];
      r /= Ns;
    }
    for (int s = nseg - 1; s >= 0; --s) {
      const int sz = seg[3 * s];
      int d;
      if ((sz & (sz - 1)) == 0) {
        d = r & (sz - 1);
        r >>= 31 - __clz(sz);
      } else {
        d = r % sz;
        r /= sz;
      }
      oa += d * seg[3 * s + 1];
      ob += d * seg[3 * s + 2];
    }
    const int64_t offB = word64(b + W_B), offC = word64(b + W_C);
    const int sa = b[W_SA], sb = b[W_SB], sc = b[W_SC];
    const bool mul = CNT && offB >= 0 && !(b[W_FLAGS] & F_UNIT);
    w.flags = b[W_FLAGS];
    w.A = (sa >= 0 ? sX + sa : X + word64(b + W_A)) + oa;
    w.B = offB < 0 ? nullptr : (sb >= 0 ? sX + sb : X + offB) + ob;
    w.nA = !CNT ? nullptr : (sa >= 0 ? sN + sa : N + word64(b + W_NA)) + oa;
    w.nB = !mul ? nullptr : (sb >= 0 ? sN + sb : N + word64(b + W_NB)) + ob;
    w.C = offC < 0 ? nullptr : X + offC + out;
    w.sC = sc < 0 ? nullptr : sX + sc + out;
    w.nC = !CNT || offC < 0 ? nullptr : N + word64(b + W_NC) + out;
    w.snC = !CNT || sc < 0 ? nullptr : sN + sc + out;
    return w;
  };
  auto run = [&](const Item<T> &w) {
    const T first = w.B != nullptr ? w.A[w.kt[0]] + w.B[w.kt[1]] : w.A[w.kt[0]];
    T best = first;
    uint64_t cnt = 0;
    if (CNT) {
      cnt = w.nA[w.kt[0]];
      if (w.nB != nullptr) cnt = mulsat64(cnt, w.nB[w.kt[1]]);
    }
#pragma unroll 4
    for (int k = 1; k < w.Ks; ++k) {
      T v = w.A[w.kt[2 * k]];
      if (w.B != nullptr) v = v + w.B[w.kt[2 * k + 1]];
      if (CNT) {
        uint64_t c = w.nA[w.kt[2 * k]];
        if (w.nB != nullptr) c = mulsat64(c, w.nB[w.kt[2 * k + 1]]);
        cnt = v > best ? c : (v == best ? addsat64(cnt, c) : cnt);
        if (v > best) best = v;
      } else {
        best = max(best, v);
      }
    }
    // Couplings near the type's largest value overflow to infinities, whose differences are
    // NaN.  Values keep the rules of the steps' own kernels: a maximum passes NaN over, in
    // the generic gate's steps only behind the first term, and a GEMM's starts at -inf.
    // (Counting runs have no rule for it: it costs 11% of an FP32 count.)
    if constexpr (!CNT && std::is_floating_point<T>::value) {
      if ((w.flags & F_KEEP) && first != first) best = first;
      if (w.flags & F_LOW) best = max(best, (T)-INFINITY);
    }
    if (w.C != nullptr) *w.C = best;
    if (w.sC != nullptr) *w.sC = best;
    if (CNT) {
      if (w.nC != nullptr) *w.nC = cnt;
      if (w.snC != nullptr) *w.snC = cnt;
    }
  };
  // Odd levels start at the other half of the block, so that (with at most half a block of
  // outputs, the usual case) one half decodes the next level while the other runs this one.
  auto start = [&](int l) {
    return (int)(threadIdx.x + (l & 1) * (kSmallThreads / 2)) & (kSmallThreads - 1);
  };
  int total = tot[0];
  Item<T> w;
  if (start(0) < total) w = decode(0, start(0));
  for (int l = 0; l < nlev; ++l) {
    const int next = l + 1 < nlev ? tot[l + 1] : 0;
    int i = start(l);
    if (i < total) run(w);
    for (i += kSmallThreads; i < total; i += kSmallThreads) run(decode(l, i));
    if (start(l + 1) < next) w = decode(l + 1, start(l + 1));
    total = next;
    __syncthreads();
  }
}

template <typename T, bool CNT>
cudaError_t run(const int32_t *d, int words, int scratch, char *arena, const Batch &bt,
                cudaStream_t st) {
  const size_t smem = (size_t)words * 4 + (size_t)scratch * (CNT ? 12 : 4);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_small<T, CNT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kSmallMaxWords * 4 + kSmallScratch * 12);
    if (e != cudaSuccess) return e;
  }
  k_small<T, CNT><<<bt.B, kSmallThreads, smem, st>>>(d, words, scratch, arena, bt.ib);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_small(Dtype dt, bool sat, const int32_t *d_desc, int words, int scratch,
                         char *arena, const Batch &bt, cudaStream_t st) {
  if (dt == DT_F32)
    return sat ? run<float, true>(d_desc, words, scratch, arena, bt, st)
               : run<float, false>(d_desc, words, scratch, arena, bt, st);
  return sat ? run<int32_t, true>(d_desc, words, scratch, arena, bt, st)
             : run<int32_t, false>(d_desc, words, scratch, arena, bt, st);
}

}  // namespace tn
