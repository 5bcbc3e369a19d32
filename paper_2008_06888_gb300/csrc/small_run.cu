// small_run.cu -- runs of small contraction steps in one launch.
//
// A contraction plan starts (and ends) with many steps on tensors of a few elements:
// merging the bond tensors around a spin, growing the state from nothing.  Each takes
// about 2 us as a kernel of its own, all of it launch and drain.  Here one block per
// instance runs a whole list of them: steps are sorted by dependency level, the
// elements of a level's outputs are spread over the block's threads, and a barrier
// separates the levels (an output written before it is read after it by the same
// block).  A level costs a few hundred ns: its chain of dependent loads.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"
#include "modarith.cuh"

namespace tn {

namespace {

constexpr int kSmallThreads = 512;
// words of a body before its digit and offset tables
enum { W_A = 0, W_B = 2, W_C = 4, W_NA = 6, W_NB = 8, W_NC = 10, W_SEG = 12, W_K = 13, W_N = 14,
       W_UNIT = 15, W_TAB = 16 };

__device__ __forceinline__ int64_t word64(const int32_t *w) {
  return (int64_t)((uint64_t)(uint32_t)w[0] | ((uint64_t)(uint32_t)w[1] << 32));
}

template <typename T, bool CNT>
__global__ void __launch_bounds__(kSmallThreads) k_small(const int32_t *__restrict__ desc,
                                                         int words, char *arena, int64_t ib) {
  extern __shared__ __align__(16) int32_t sd[];
  arena += blockIdx.x * ib;
  T *X = reinterpret_cast<T *>(arena);
  uint64_t *N = reinterpret_cast<uint64_t *>(arena);
  for (int i = threadIdx.x; i < words; i += kSmallThreads) sd[i] = desc[i];
  __syncthreads();
  const int nops = sd[0], nlev = sd[1];
  const int32_t *lev = sd + 2, *first = lev + nlev + 1, *body = first + nops;
  for (int l = 0; l < nlev; ++l) {
    const int o0 = lev[l], o1 = lev[l + 1];
    // outputs of the level: those of its last op end it (word after the last body)
    const int32_t *lb = sd + body[o1 - 1];
    const int total = first[o1 - 1] + lb[W_TAB];
    for (int i = threadIdx.x; i < total; i += kSmallThreads) {
      int lo = o0, hi = o1 - 1;   // the op whose outputs hold i
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (first[mid] <= i) lo = mid; else hi = mid - 1;
      }
      const int32_t *b = sd + body[lo];
      const int out = i - first[lo];
      const int nseg = b[W_SEG], Ks = b[W_K], Ns = b[W_N];
      const int32_t *seg = b + W_TAB + 1;          // (size, sA, sB) of each digit
      const int32_t *kt = seg + 3 * nseg;          // (kA, kB) of each k
      const int32_t *nt = kt + 2 * Ks;             // nB of each n
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
      const int64_t offB = word64(b + W_B);
      const T *A = X + word64(b + W_A) + oa;
      const T *B = offB >= 0 ? X + offB + ob : nullptr;
      const bool mul = CNT && B != nullptr && !b[W_UNIT];
      const uint64_t *nA = CNT ? N + word64(b + W_NA) + oa : nullptr;
      const uint64_t *nB = mul ? N + word64(b + W_NB) + ob : nullptr;
      T best = A[kt[0]];
      if (B != nullptr) best = best + B[kt[1]];
      uint64_t cnt = 0;
      if (CNT) {
        cnt = nA[kt[0]];
        if (mul) cnt = mulsat64(cnt, nB[kt[1]]);
      }
#pragma unroll 4
      for (int k = 1; k < Ks; ++k) {
        T v = A[kt[2 * k]];
        if (B != nullptr) v = v + B[kt[2 * k + 1]];
        if (CNT) {
          uint64_t c = nA[kt[2 * k]];
          if (mul) c = mulsat64(c, nB[kt[2 * k + 1]]);
          cnt = v > best ? c : (v == best ? addsat64(cnt, c) : cnt);
        }
        if (v > best) best = v;
      }
      X[word64(b + W_C) + out] = best;
      if (CNT) N[word64(b + W_NC) + out] = cnt;
    }
    __syncthreads();
  }
}

template <typename T, bool CNT>
cudaError_t run(const int32_t *d, int words, char *arena, const Batch &bt, cudaStream_t st) {
  const size_t smem = (size_t)words * 4;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_small<T, CNT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kSmallMaxWords * 4);
    if (e != cudaSuccess) return e;
  }
  k_small<T, CNT><<<bt.B, kSmallThreads, smem, st>>>(d, words, arena, bt.ib);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_small(Dtype dt, bool sat, const int32_t *d_desc, int words, char *arena,
                         const Batch &bt, cudaStream_t st) {
  if (dt == DT_F32)
    return sat ? run<float, true>(d_desc, words, arena, bt, st)
               : run<float, false>(d_desc, words, arena, bt, st);
  return sat ? run<int32_t, true>(d_desc, words, arena, bt, st)
             : run<int32_t, false>(d_desc, words, arena, bt, st);
}

}  // namespace tn
