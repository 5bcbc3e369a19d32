// chain3.cu -- fused gate chains of q = 3 states (values).
//
// A chain's tile (3^t elements: the fastest legs, for runs of consecutive elements, and
// the legs its gates touch) is staged in shared memory.  One gate at a time over the
// staged tile costs a shared-memory pass with integer divisions per gate: 65 chains of
// 108 us for a 15 x 15 lattice (7.0 ms), where moving the 3^15 elements takes 17 us.  Here the gates are cut into groups
// of at most three replaced legs: a thread holds the 27 elements that differ in a group's
// legs in registers, applies all of its gates there and writes them back, so a chain
// makes two or three passes over its tile (46 chains of 52 us, 2.4 ms).  Gates on other legs of the tile read the
// thread's fixed digits.  Blocks are persistent and copy the next tile (cp.async) while
// they work on this one.
// Every element sees the same sums and maxima in the same order as one gate at a time.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"
#include "chain_dev.cuh"

namespace tn {

namespace {

constexpr int kThreads = 256;   // 3^5 of them own 27 elements each of a 3^8 tile
constexpr int kBlocksPerSm = 4; // 2 x 26 KB of tiles each
constexpr int kMaxT = 8;
constexpr int kRun = 81;        // elements of a run: the four fastest legs
// copies: 3 runs at a time, so a thread keeps its place in the run
constexpr int kCopyRuns = kThreads / kRun, kCopyThreads = kCopyRuns * kRun;
constexpr int kB = 27;          // values of a gate's operand at most

struct Gate3 {
  int32_t code;          // replace: 4 J + K + 1; diagonal: 12 + 4 (a + 1) + b + 1, a < b
  int32_t bk, bn;        // operand strides: contracted, new digit
  int32_t b0, b1;        // of the register legs K (replace) or a, b (diagonal)
  int32_t nfix;
  int32_t fr[2], fb[2];  // legs fixed per thread: their place among the rest, operand stride
};
struct Group3 {
  int32_t g0, g1;        // gates [g0, g1)
  int32_t s[3];          // local strides of the register legs
  int32_t rest[kMaxT - 3];
};
struct Plan3 {
  int32_t ngrp, nrest;
  Gate3 gate[TN_CHAIN_MAX_G];
  Group3 grp[TN_CHAIN_MAX_G];
};

__host__ __device__ constexpr int pow3(int e) { return e == 0 ? 1 : 3 * pow3(e - 1); }

__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ int32_t max3(int32_t a, int32_t b, int32_t c) {
  return max(max(a, b), c);
}

// Replace leg J: v'[n] = max_u v[u] + B[u, n], for each digit of register leg K (-1: none).
template <int J, int K, typename T>
__device__ __forceinline__ void rep3(T (&v)[27], const T *B, const Gate3 &g) {
  constexpr int sj = pow3(J), sk = K < 0 ? 1 : pow3(K);
#pragma unroll
  for (int k = 0; k < (K < 0 ? 1 : 3); ++k) {
    T m[3][3];
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
      for (int n = 0; n < 3; ++n) m[u][n] = B[k * g.b0 + u * g.bk + n * g.bn];
#pragma unroll
    for (int e = 0; e < 27; ++e) {
      if ((e / sj) % 3 != 0) continue;
      if (K >= 0 && (e / sk) % 3 != k) continue;
      const T a = v[e], b = v[e + sj], c = v[e + 2 * sj];
#pragma unroll
      for (int n = 0; n < 3; ++n)
        v[e + n * sj] = max3(a + m[0][n], b + m[1][n], c + m[2][n]);
    }
  }
}

// Add B over register legs a (-1: none) and b (-1: none).
template <int A, int Bb, typename T>
__device__ __forceinline__ void diag3(T (&v)[27], const T *B, const Gate3 &g) {
  constexpr int sa = A < 0 ? 1 : pow3(A), sb = Bb < 0 ? 1 : pow3(Bb);
#pragma unroll
  for (int x = 0; x < (A < 0 ? 1 : 3); ++x)
#pragma unroll
    for (int y = 0; y < (Bb < 0 ? 1 : 3); ++y) {
      const T add = B[x * g.b0 + y * g.b1];
#pragma unroll
      for (int e = 0; e < 27; ++e)
        if ((A < 0 || (e / sa) % 3 == x) && (Bb < 0 || (e / sb) % 3 == y)) v[e] = v[e] + add;
    }
}

template <typename T>
__device__ __forceinline__ void apply3(const Gate3 &g, const T *B, T (&v)[27]) {
#define TN_R3(J, K) case 4 * (J) + (K) + 1: rep3<J, K>(v, B, g); break;
#define TN_D3(A, Bb) case 12 + 4 * ((A) + 1) + (Bb) + 1: diag3<A, Bb>(v, B, g); break;
  switch (g.code) {
    TN_R3(0, -1) TN_R3(0, 1) TN_R3(0, 2)
    TN_R3(1, -1) TN_R3(1, 0) TN_R3(1, 2)
    TN_R3(2, -1) TN_R3(2, 0) TN_R3(2, 1)
    TN_D3(-1, -1) TN_D3(-1, 0) TN_D3(-1, 1) TN_D3(-1, 2)
    TN_D3(0, 1) TN_D3(0, 2) TN_D3(1, 2)
  }
#undef TN_R3
#undef TN_D3
}

template <typename T>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm)
    k_chain3(const ChainParams p, const __grid_constant__ Plan3 pl, const T *__restrict__ X,
             const T *__restrict__ A, T *__restrict__ C, int64_t ib) {
  X = inst_ptr(X, ib);
  A = inst_ptr(A, ib);
  C = inst_ptr(C, ib);
  extern __shared__ __align__(16) char raw3[];
  T *tiles = reinterpret_cast<T *>(raw3);
  __shared__ T sB[TN_CHAIN_MAX_G * kB];
  __shared__ Gate3 sG[TN_CHAIN_MAX_G];
  __shared__ int64_t sHi[TN_CHAIN_MAX_HI];
  for (int i = threadIdx.x; i < p.ngates * kB; i += kThreads) {
    const ChainGate &g = p.g[i / kB];
    if (i % kB < g.nBel) sB[i] = X[g.offB + i % kB];
  }
  for (int i = threadIdx.x; i < p.ngates; i += kThreads) sG[i] = pl.gate[i];
  for (int i = threadIdx.x; i < p.nhi; i += kThreads) sHi[i] = p.hi_off[i];
  __syncthreads();
  const int run0 = threadIdx.x / kRun, col = threadIdx.x % kRun;
  auto base_of = [&](int64_t o) {
    int64_t b = 0;
    for (int sg = p.nseg - 1; sg >= 0; --sg) {
      const int64_t sz = p.seg_size[sg], q = o / sz;
      b += (o - q * sz) * p.seg_s[sg];
      o = q;
    }
    return b;
  };
  auto fetch = [&](int64_t o, T *dst) {
    if (o < p.outer) {
      const T *src = A + base_of(o);
      if (threadIdx.x < kCopyThreads)
#pragma unroll 9
        for (int h = run0; h < p.nhi; h += kCopyRuns)
          cp_async4(dst + h * kRun + col, src + sHi[h] + col);
    }
    cp_async_commit();
  };
  const int owners = p.tile / 27;
  fetch(blockIdx.x, tiles);
  int cur = 0;
  for (int64_t o = blockIdx.x; o < p.outer; o += gridDim.x, cur ^= 1) {
    T *s = tiles + cur * p.tile;
    fetch(o + gridDim.x, tiles + (cur ^ 1) * p.tile);
    cp_async_wait_prev();
    __syncthreads();
    for (int gr = 0; gr < pl.ngrp; ++gr) {
      const Group3 &G = pl.grp[gr];
      for (int j = threadIdx.x; j < owners; j += kThreads) {
        int r = j, base = 0, dig = 0;
#pragma unroll
        for (int k = 0; k < kMaxT - 3; ++k) {
          if (k < pl.nrest) {
            const int d = r % 3;
            r /= 3;
            base += d * G.rest[k];
            dig |= d << (2 * k);
          }
        }
        T v[27];
        const int s0 = G.s[0], s1 = G.s[1], s2 = G.s[2];
#pragma unroll
        for (int e = 0; e < 27; ++e)
          v[e] = s[base + (e % 3) * s0 + (e / 3 % 3) * s1 + (e / 9) * s2];
        for (int gi = G.g0; gi < G.g1; ++gi) {
          const Gate3 &g = sG[gi];
          const T *B = sB + gi * kB;
          if (g.nfix > 0) B += ((dig >> (2 * g.fr[0])) & 3) * g.fb[0];
          if (g.nfix > 1) B += ((dig >> (2 * g.fr[1])) & 3) * g.fb[1];
          apply3(g, B, v);
        }
#pragma unroll
        for (int e = 0; e < 27; ++e)
          s[base + (e % 3) * s0 + (e / 3 % 3) * s1 + (e / 9) * s2] = v[e];
      }
      __syncthreads();
    }
    T *dst = C + base_of(o);
    if (threadIdx.x < kCopyThreads)
#pragma unroll 9
      for (int h = run0; h < p.nhi; h += kCopyRuns) dst[sHi[h] + col] = s[h * kRun + col];
    __syncthreads();   // the next fetch but one overwrites this tile
  }
}

// Groups of gates with at most three replaced legs, and each gate's legs as register legs
// or fixed digits of its group.  false: an operand the kernel has no form for.
bool plan3(const ChainParams &p, Plan3 *pl) {
  *pl = Plan3{};
  if (p.t < 3 || p.t > kMaxT) return false;
  pl->nrest = p.t - 3;
  int strides[kMaxT];
  for (int i = 0, s = 1; i < p.t; ++i, s *= 3) strides[i] = s;
  for (int g0 = 0; g0 < p.ngates;) {
    Group3 &G = pl->grp[pl->ngrp++];
    int n = 0, g1 = g0;
    for (; g1 < p.ngates; ++g1) {
      const ChainGate &g = p.g[g1];
      if (g.kind > 1 || g.nb > 2 || (g.kind == 0 && g.nb > 1) || g.nBel > kB) return false;
      if (g.kind != 0) continue;
      if (std::find(G.s, G.s + n, g.ls) != G.s + n) continue;
      if (n == 3) break;
      G.s[n++] = g.ls;
    }
    // free register legs go to legs that the group's gates read, then to the slowest
    for (int gi = g0; gi < g1; ++gi)
      for (int j = 0; j < p.g[gi].nb; ++j)
        if (n < 3 && std::find(G.s, G.s + n, p.g[gi].lsb[j]) == G.s + n) G.s[n++] = p.g[gi].lsb[j];
    for (int i = p.t - 1; n < 3; --i)
      if (std::find(G.s, G.s + n, strides[i]) == G.s + n) G.s[n++] = strides[i];
    int nr = 0;
    for (int i = 0; i < p.t; ++i)
      if (std::find(G.s, G.s + 3, strides[i]) == G.s + 3) G.rest[nr++] = strides[i];
    auto reg = [&](int s) {
      const int *at = std::find(G.s, G.s + 3, s);
      return at == G.s + 3 ? -1 : (int)(at - G.s);
    };
    for (int gi = g0; gi < g1; ++gi) {
      const ChainGate &g = p.g[gi];
      Gate3 &o = pl->gate[gi];
      o.bk = (int32_t)g.sBk;
      o.bn = (int32_t)g.sBn;
      int a = -1, b = -1;   // register legs of the operand
      for (int j = 0; j < g.nb; ++j) {
        const int r = reg(g.lsb[j]);
        if (r < 0) {
          o.fr[o.nfix] = (int32_t)(std::find(G.rest, G.rest + nr, g.lsb[j]) - G.rest);
          o.fb[o.nfix++] = (int32_t)g.sBb[j];
        } else if (b < 0) {
          b = r;
          o.b1 = (int32_t)g.sBb[j];
        } else {
          a = r;
          o.b0 = (int32_t)g.sBb[j];
        }
      }
      if (g.kind == 0) {
        o.b0 = o.b1;
        o.code = 4 * reg(g.ls) + b + 1;
      } else {
        if (a > b) {
          std::swap(a, b);
          std::swap(o.b0, o.b1);
        }
        o.code = 12 + 4 * (a + 1) + b + 1;
      }
    }
    G.g0 = g0;
    G.g1 = g1;
    g0 = g1;
  }
  return true;
}

template <typename T>
cudaError_t run(const ChainParams &p, const Plan3 &pl, const char *arena, const void *A, void *C,
                const Batch &bt, cudaStream_t st) {
  const size_t smem = (size_t)2 * p.tile * sizeof(T);
  cudaError_t e = cudaFuncSetAttribute(k_chain3<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       2 * pow3(kMaxT) * (int)sizeof(T));
  if (e != cudaSuccess) return e;
  // one wave of resident blocks that walk equal numbers of tiles
  const int64_t slots = std::max<int64_t>(1, (int64_t)kBlocksPerSm * num_sms() / bt.B);
  const int64_t trips = (p.outer + slots - 1) / slots;
  const int64_t blocks = (p.outer + trips - 1) / trips;
  k_chain3<T><<<dim3((unsigned)blocks, bt.B), kThreads, smem, st>>>(
      p, pl, reinterpret_cast<const T *>(arena), static_cast<const T *>(A), static_cast<T *>(C),
      bt.ib);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_chain3(Dtype dt, const ChainParams &p, const char *arena, const void *A,
                          void *C, const Batch &bt, cudaStream_t st) {
  Plan3 pl;
  if (!plan3(p, &pl)) return cudaErrorInvalidValue;
  if (p.lo != kRun) return cudaErrorInvalidValue;
  if (dt == DT_F32) return run<float>(p, pl, arena, A, C, bt, st);
  return run<int32_t>(p, pl, arena, A, C, bt, st);
}

}  // namespace tn
