// gate_sum.cu -- Hadamard products of gate contractions in one pass.
//
// Cell rows of hardware graphs build their tensor as a product of two to four gate
// contractions over the same legs: C[o, n] = sum_g max_k (A_g[o, k] + B_g[k, n]) (counts
// multiply).  As steps of their own, each contraction writes a tensor eight times its
// input, and each product reads two of them and writes a third: with 2^24 elements and
// 64-bit counts, four contractions and three products are 4 x 78 + 3 x 115 us.  Here
// they are one kernel that reads the small operands and writes C once: 135 us with counts
// (ALU: four tie selections and three products of counts per element; 30 us for its bytes),
// 36 us for values alone.
//
// A thread owns four consecutive n of an outer index (one 16-byte store per word of the
// element, lanes side by side) and keeps its slice of the B tables, 2 x 4 values per
// gate, in registers.  Terms and sums are those of the separate steps, in their order.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "chain_dev.cuh"
#include "gate_dev.cuh"
#include "modarith.cuh"

namespace tn {

namespace {

constexpr int kThreads = 256;

struct SumPtrs {
  const void *A[TN_SUM_MAX_G], *B[TN_SUM_MAX_G];
  const uint64_t *nA[TN_SUM_MAX_G];
};

// resident blocks per SM: one wave of them, so that the B tables are loaded once per block
constexpr int blocks_per_sm(int NG, bool CNT) { return NG == 4 ? (CNT ? 2 : 3) : (CNT ? 4 : 6); }

// saturating product: counts below 2^32, the usual case, need one 32-bit multiplication
// where the general form takes a 128-bit product
__device__ __forceinline__ uint64_t mulcount(uint64_t a, uint64_t b) {
  if (((a | b) >> 32) == 0) return (uint64_t)(uint32_t)a * (uint32_t)b;
  return mulsat64(a, b);
}

template <typename T, int NG, bool CNT>
__global__ void __launch_bounds__(kThreads, blocks_per_sm(NG, CNT)) k_gate_sum(const __grid_constant__ GateSum p,
                                                       const __grid_constant__ SumPtrs ptr, T *C,
                                                       uint64_t *nC, int64_t ib) {
  C = inst_ptr(C, ib);
  if (CNT) nC = inst_ptr(nC, ib);
  const int per = p.Ns / 4;                       // threads per outer index (a power of two)
  const int n0 = 4 * (threadIdx.x & (per - 1));   // kThreads and the stride are multiples of it
  T b[NG][2][4];
  const T *A[NG];
  const uint64_t *nA[NG];
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    const T *B = inst_ptr(static_cast<const T *>(ptr.B[g]), ib);
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int j = 0; j < 4; ++j) b[g][k][j] = B[p.kB[g][k] + p.nB[g][n0 + j]];
    A[g] = inst_ptr(static_cast<const T *>(ptr.A[g]), ib);
    nA[g] = CNT ? inst_ptr(ptr.nA[g], ib) : nullptr;
  }
  const int step = (int)(gridDim.x * kThreads) / per;
  for (int o = (int)(blockIdx.x * kThreads + threadIdx.x) / per; o < p.outer; o += step) {
    int r = o, oc = 0, oa[NG];
#pragma unroll
    for (int g = 0; g < NG; ++g) oa[g] = 0;
    for (int s = p.nseg - 1; s >= 0; --s) {
      const int i = r & (p.seg_size[s] - 1);
      r >>= p.seg_sh[s];
      oc += i * p.seg_sC[s];
#pragma unroll
      for (int g = 0; g < NG; ++g) oa[g] += i * p.seg_sA[g][s];
    }
    T a[NG][2];
    uint64_t na[NG][2];
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int e = oa[g] + p.kA[g][k];
        a[g][k] = A[g][e];
        if (CNT) na[g][k] = nA[g][e];
      }
    T out[4];
    uint64_t cnt[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      T v[NG];
      uint64_t c[NG];
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        const T x = a[g][0] + b[g][0][j], y = a[g][1] + b[g][1][j];
        // NaN terms (couplings that overflow) as in the separate steps: values keep a first
        // one, counting steps take maxima and count the terms that equal them
        if constexpr (!CNT) {
          v[g] = y > x ? y : x;
        } else {
          v[g] = max(x, y);
          if constexpr (std::is_floating_point<T>::value)
            c[g] = addsat64(x == v[g] ? na[g][0] : 0, y == v[g] ? na[g][1] : 0);
          else
            c[g] = x > y ? na[g][0] : (x < y ? na[g][1] : addsat64(na[g][0], na[g][1]));
        }
      }
      if constexpr (NG == 2) {
        out[j] = v[0] + v[1];
        if (CNT) cnt[j] = mulcount(c[0], c[1]);
      } else {
        out[j] = (v[0] + v[1]) + (v[2] + v[3]);
        if (CNT) cnt[j] = mulcount(mulcount(c[0], c[1]), mulcount(c[2], c[3]));
      }
    }
    typename Vec4<T>::t w;
    w.x = out[0];
    w.y = out[1];
    w.z = out[2];
    w.w = out[3];
    *reinterpret_cast<typename Vec4<T>::t *>(C + oc + n0) = w;
    if (CNT) {
      ulonglong2 *d = reinterpret_cast<ulonglong2 *>(nC + oc + n0);
      d[0] = make_ulonglong2(cnt[0], cnt[1]);
      d[1] = make_ulonglong2(cnt[2], cnt[3]);
    }
  }
}

template <typename T, int NG, bool CNT>
cudaError_t run(const GateSum &p, const SumPtrs &ptr, void *C, uint64_t *nC, const Batch &bt,
                cudaStream_t st) {
  const int64_t need = (p.outer * (p.Ns / 4) + kThreads - 1) / kThreads;
  const int64_t cap = std::max<int64_t>(1, (int64_t)num_sms() * blocks_per_sm(NG, CNT) / bt.B);
  k_gate_sum<T, NG, CNT><<<dim3((unsigned)std::min(need, cap), bt.B), kThreads, 0, st>>>(
      p, ptr, static_cast<T *>(C), nC, bt.ib);
  return cudaGetLastError();
}

template <typename T>
cudaError_t run_t(bool cnt, const GateSum &p, const SumPtrs &ptr, void *C, uint64_t *nC,
                  const Batch &bt, cudaStream_t st) {
  if (p.n == 2)
    return cnt ? run<T, 2, true>(p, ptr, C, nC, bt, st) : run<T, 2, false>(p, ptr, C, nC, bt, st);
  if (p.n == 4)
    return cnt ? run<T, 4, true>(p, ptr, C, nC, bt, st) : run<T, 4, false>(p, ptr, C, nC, bt, st);
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_gate_sum(Dtype dt, bool cnt, const GateSum &p, const void *const *A,
                            const void *const *B, const uint64_t *const *nA, void *C,
                            uint64_t *nC, const Batch &bt, cudaStream_t st) {
  SumPtrs ptr{};
  for (int g = 0; g < p.n; ++g) {
    ptr.A[g] = A[g];
    ptr.B[g] = B[g];
    ptr.nA[g] = nA[g];
  }
  if (dt == DT_F32) return run_t<float>(cnt, p, ptr, C, nC, bt, st);
  return run_t<int32_t>(cnt, p, ptr, C, nC, bt, st);
}

}  // namespace tn
