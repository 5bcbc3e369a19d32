// chain_sat.cu -- register chains of the exact 64-bit counting programs: INT32
// values and one plane of saturating 64-bit counts (q = 2), folded table gates.
//
// A thread owns the 2^RB states of the chain's register legs for one outer index:
// RB = 4 legs and 12 bytes per state are 48 registers, against 3 legs with the seven
// 4-byte residue planes of the modular counts.  One pass then moves (4 + 8) bytes per
// element each way for up to four replaced legs, where the residue form moves (4 + 28)
// for three.  A replace gate costs about 10 instructions per state (two sums, a
// maximum, two comparisons, the selection of the 64-bit count, half of its sum).  Five
// blocks of 128 threads per SM leave 96 registers a thread: every form spills 8 to 64 bytes.
//
// Gate counts: a leaf operand counts 1 everywhere, so a table gate made of leaves
// only selects and adds the states' counts; otherwise its count table (the product
// of its components' counts) multiplies in, which a diagonal term may do in the
// replace gate it was folded into: products of counts commute with the (max, +)
// selection exactly as the sums of the values do.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>

#include "kernels.h"
#include "chain_dev.cuh"
#include "modarith.cuh"

namespace tn {

namespace {

// 2^LW consecutive elements of a value or count array (aligned to the vector)
template <int LW>
__device__ __forceinline__ void sload(const int32_t *src, int32_t *dst) {
  if constexpr (LW == 0) {
    dst[0] = *src;
  } else if constexpr (LW == 1) {
    const int2 x = *reinterpret_cast<const int2 *>(src);
    dst[0] = x.x;
    dst[1] = x.y;
  } else {
    const int4 x = *reinterpret_cast<const int4 *>(src);
    dst[0] = x.x;
    dst[1] = x.y;
    dst[2] = x.z;
    dst[3] = x.w;
  }
}
template <int LW>
__device__ __forceinline__ void sload(const uint64_t *src, uint64_t *dst) {
  if constexpr (LW == 0) {
    dst[0] = *src;
  } else {
#pragma unroll
    for (int i = 0; i < (1 << LW); i += 2) {
      const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(src + i);
      dst[i] = x.x;
      dst[i + 1] = x.y;
    }
  }
}
template <int LW>
__device__ __forceinline__ void sstore(int32_t *dst, const int32_t *src) {
  if constexpr (LW == 0)
    *dst = src[0];
  else if constexpr (LW == 1)
    *reinterpret_cast<int2 *>(dst) = make_int2(src[0], src[1]);
  else
    *reinterpret_cast<int4 *>(dst) = make_int4(src[0], src[1], src[2], src[3]);
}
template <int LW>
__device__ __forceinline__ void sstore(uint64_t *dst, const uint64_t *src) {
  if constexpr (LW == 0) {
    *dst = src[0];
  } else {
#pragma unroll
    for (int i = 0; i < (1 << LW); i += 2)
      *reinterpret_cast<ulonglong2 *>(dst + i) = make_ulonglong2(src[i], src[i + 1]);
  }
}

// Saturation inside a chain: the upper words of the counts are clamped when they are
// loaded (to kCap + 2^32 at most) and after every fourth gate, and a gate at most
// doubles a count, so sums never wrap.  Counts below kCap are exact; a sum or product
// with a term of kCap or more is itself at least kCap.  (One instruction per clamp,
// against five per saturating 64-bit sum.)
constexpr uint32_t kCapHi = 1u << 27;   // kCap = 2^59
__device__ __forceinline__ uint64_t clamp_count(uint64_t n) {
  const uint32_t hi = min((uint32_t)(n >> 32), kCapHi);
  return ((uint64_t)hi << 32) | (uint32_t)n;
}
__device__ __forceinline__ uint64_t mulcap(uint64_t a, uint64_t b) {
  return clamp_count(mulsat64(a, b));
}

// (x, n) of the larger of two terms, counts added on a tie (both: their sum)
__device__ __forceinline__ uint64_t tie(int32_t x, int32_t y, uint64_t nx, uint64_t ny,
                                        uint64_t both) {
  return x > y ? nx : (x < y ? ny : both);
}

// Replace (CON: final contraction, no new digit) on register bit J with the extra
// register leg K (-1: none), whose digit chooses between the table halves lo and hi,
// each (x, x') = (0,0), (1,0), (0,1), (1,1).
template <int RB, int J, int K, bool CON>
__device__ __forceinline__ void srep(int32_t (&v)[1 << RB], uint64_t (&n)[1 << RB], const int4 &lo,
                                     const int4 &hi) {
#pragma unroll
  for (int e = 0; e < (1 << RB); ++e) {
    if (e & (1 << J)) continue;
    const int e1 = e | (1 << J);
    const bool k = K >= 0 && ((e >> (K < 0 ? 0 : K)) & 1);
    const int32_t a = v[e], b = v[e1];
    const uint64_t na = n[e], nb = n[e1], both = na + nb;
    const int32_t s00 = a + (k ? hi.x : lo.x), s10 = b + (k ? hi.y : lo.y);
    v[e] = max(s00, s10);
    n[e] = tie(s00, s10, na, nb, both);
    if (!CON) {
      const int32_t s01 = a + (k ? hi.z : lo.z), s11 = b + (k ? hi.w : lo.w);
      v[e1] = max(s01, s11);
      n[e1] = tie(s01, s11, na, nb, both);
    }
  }
}

// The same with gate counts: cn is the count table in the order of lo, hi.
template <int RB, int J, bool CON>
__device__ __forceinline__ void srep_n(int32_t (&v)[1 << RB], uint64_t (&n)[1 << RB],
                                       const int4 &lo, const int4 &hi, int km,
                                       const uint64_t *cn) {
#pragma unroll
  for (int e = 0; e < (1 << RB); ++e) {
    if (e & (1 << J)) continue;
    const int e1 = e | (1 << J);
    const bool k = (e & km) != 0;
    const uint64_t *c = cn + (k ? 4 : 0);
    const int32_t a = v[e], b = v[e1];
    const uint64_t na = n[e], nb = n[e1];
    const int32_t s00 = a + (k ? hi.x : lo.x), s10 = b + (k ? hi.y : lo.y);
    const uint64_t p00 = mulcap(na, c[0]), p10 = mulcap(nb, c[1]);
    v[e] = max(s00, s10);
    n[e] = tie(s00, s10, p00, p10, p00 + p10);
    if (!CON) {
      const int32_t s01 = a + (k ? hi.z : lo.z), s11 = b + (k ? hi.w : lo.w);
      const uint64_t p01 = mulcap(na, c[2]), p11 = mulcap(nb, c[3]);
      v[e1] = max(s01, s11);
      n[e1] = tie(s01, s11, p01, p11, p01 + p11);
    }
  }
}

// diagonal gate on register bits J (table index bit 0) and K (bit 1), -1: none
template <int RB>
__device__ __forceinline__ void sdiag(int32_t (&v)[1 << RB], uint64_t (&n)[1 << RB], int J, int K,
                                      const int4 &lo, const uint64_t *cn) {
  const int mj = J >= 0 ? 1 << J : 0, mk = K >= 0 ? 1 << K : 0;
#pragma unroll
  for (int e = 0; e < (1 << RB); ++e) {
    const bool x0 = (e & mj) != 0, x1 = (e & mk) != 0;
    v[e] = v[e] + (x1 ? (x0 ? lo.w : lo.z) : (x0 ? lo.y : lo.x));
    if (cn != nullptr) n[e] = mulcap(n[e], cn[(x0 ? 1 : 0) | (x1 ? 2 : 0)]);
  }
}

// dispatch: replace on J with extra leg K is code J * 7 + K + 1, a contraction 100
// above it; diagonal gates are 42 + (J + 1) * 7 + K + 1
template <int RB>
__device__ __forceinline__ void sapply(int code, int32_t (&v)[1 << RB], uint64_t (&n)[1 << RB],
                                       const int4 &lo, const int4 &hi, const uint64_t *cn) {
  static_assert(RB == 4, "the cases below are those of four register legs");
  if (cn == nullptr) {
#define TN_S(J, K)                                                     \
  case (J) * 7 + (K) + 1: srep<RB, J, K, false>(v, n, lo, hi); break;    \
  case 100 + (J) * 7 + (K) + 1: srep<RB, J, K, true>(v, n, lo, hi); break;
    switch (code) {
      TN_S(0, -1) TN_S(0, 1) TN_S(0, 2) TN_S(0, 3)
      TN_S(1, -1) TN_S(1, 0) TN_S(1, 2) TN_S(1, 3)
      TN_S(2, -1) TN_S(2, 0) TN_S(2, 1) TN_S(2, 3)
      TN_S(3, -1) TN_S(3, 0) TN_S(3, 1) TN_S(3, 2)
      default: sdiag<RB>(v, n, (code - 42) / 7 - 1, (code - 42) % 7 - 1, lo, cn); break;
    }
#undef TN_S
    return;
  }
  const bool con = code >= 100;
  const int r = con ? code - 100 : code, J = r / 7, K = r % 7 - 1, km = K >= 0 ? 1 << K : 0;
  if (!con && code >= 42) {
    sdiag<RB>(v, n, (code - 42) / 7 - 1, (code - 42) % 7 - 1, lo, cn);
    return;
  }
  switch (con ? J + 4 : J) {
    case 0: srep_n<RB, 0, false>(v, n, lo, hi, km, cn); break;
    case 1: srep_n<RB, 1, false>(v, n, lo, hi, km, cn); break;
    case 2: srep_n<RB, 2, false>(v, n, lo, hi, km, cn); break;
    case 3: srep_n<RB, 3, false>(v, n, lo, hi, km, cn); break;
    case 4: srep_n<RB, 0, true>(v, n, lo, hi, km, cn); break;
    case 5: srep_n<RB, 1, true>(v, n, lo, hi, km, cn); break;
    case 6: srep_n<RB, 2, true>(v, n, lo, hi, km, cn); break;
    default: srep_n<RB, 3, true>(v, n, lo, hi, km, cn); break;
  }
}

// LWI / LWO: the register legs 0..LW-1 sit at memory positions 0..LW-1 of the
// input / output, so the 2^LW states that differ in them move with one access per
// array.  I: element offsets (32 bits when the tensors have fewer than 2^31).
template <int RB, int LWI, int LWO, typename I, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_schain(const ChainParams p,
                                                     const int32_t *__restrict__ X,
                                                     const uint64_t *__restrict__ Xn,
                                                     const int32_t *__restrict__ A,
                                                     const uint64_t *__restrict__ An,
                                                     int32_t *__restrict__ C,
                                                     uint64_t *__restrict__ Cn, int64_t ib) {
  X = inst_ptr(X, ib);
  Xn = inst_ptr(Xn, ib);
  A = inst_ptr(A, ib);
  An = inst_ptr(An, ib);
  C = inst_ptr(C, ib);
  Cn = inst_ptr(Cn, ib);
  __shared__ __align__(16) int32_t sT[TN_CHAIN_MAX_G * TN_TG_TABLE];
  __shared__ uint64_t sN[TN_CHAIN_MAX_G * TN_TG_TABLE];
  __shared__ int4 sD[TN_CHAIN_MAX_G];
  build_tables<int32_t>(p, X, sT);
  // count tables: the product of the components' counts (leaves count 1)
  for (int i = threadIdx.x; i < p.ttotal; i += blockDim.x) {
    int k = 0;
    while (k + 1 < p.ntg && p.tg[k + 1].toff <= i) ++k;
    const TGate &t = p.tg[k];
    const int li = i - t.toff;
    uint64_t prod = 1;
    for (int c = 0; c < t.ncomp; ++c) {
      const ChainGate &g = p.g[t.cg[c]];
      if (g.unitB) continue;
      const int64_t st[4] = {g.sBk, g.sBn, g.sBb[0], g.sBb[1]};
      int64_t o = 0;
      for (int l = 0; l < 4; ++l)
        if (t.cbit[c][l] >= 0) o += (int64_t)((li >> t.cbit[c][l]) & 1) * st[l];
      prod = mulsat64(prod, Xn[g.offBn + o]);
    }
    sN[i] = prod;
  }
  if (threadIdx.x < p.ntg) {
    const TGate &t = p.tg[threadIdx.x];
    int sh[TN_TG_MAXF], unit = 1;
    for (int i = 0; i < TN_TG_MAXF; ++i) sh[i] = i < t.nf ? t.fsh[i] : 62;   // 0 bit
    for (int c = 0; c < t.ncomp; ++c) unit &= p.g[t.cg[c]].unitB;
    sD[threadIdx.x] = make_int4(t.code, t.toff, sh[0] | (sh[1] << 8) | (sh[2] << 16), unit);
  }
  __syncthreads();
  I sS[RB], sO[RB];   // register-leg strides in the input and in the output
#pragma unroll
  for (int j = 0; j < RB; ++j) {
    sS[j] = (I)p.hi_in[1 << j];
    sO[j] = (I)p.hi_out[1 << j];
  }
  const int cmask = p.tg[p.ntg - 1].kind == 2 ? 1 << p.tg[p.ntg - 1].J : 0;
  const int64_t step = (int64_t)gridDim.x * NT;
  for (int64_t tau = blockIdx.x * (int64_t)NT + threadIdx.x; tau < p.outer; tau += step) {
    int32_t v[1 << RB];
    uint64_t n[1 << RB];
    {
      const I bi = rc_base_l<I>(p, tau, p.ssh_in);
      const int32_t *src = A + bi;
      const uint64_t *srn = An + bi;
      I o[1 << RB];
      o[0] = 0;
#pragma unroll
      for (int e = 1; e < (1 << RB); ++e) {
        const int hb = 31 - __clz(e);
        o[e] = o[e ^ (1 << hb)] + sS[hb];
      }
#pragma unroll
      for (int e = 0; e < (1 << RB); e += 1 << LWI) {
        sload<LWI>(src + o[e], &v[e]);
        sload<LWI>(srn + o[e], &n[e]);
      }
#pragma unroll
      for (int e = 0; e < (1 << RB); ++e) n[e] = clamp_count(n[e]);
    }
    for (int gi = 0; gi < p.ntg; ++gi) {
      const int4 d = sD[gi];
      const int a = tc_slice(d, tau);
      const int4 lo = *reinterpret_cast<const int4 *>(sT + a);
      const int4 hi = *reinterpret_cast<const int4 *>(sT + a + 4);
      sapply<RB>(d.x, v, n, lo, hi, d.w ? nullptr : sN + a);
      if ((gi & 3) == 3) {
#pragma unroll
        for (int e = 0; e < (1 << RB); ++e) n[e] = clamp_count(n[e]);
      }
    }
    const I bo = rc_base_l<I>(p, tau, p.ssh_out);
    int32_t *dst = C + bo;
    uint64_t *dsn = Cn + bo;
    I o[1 << RB];
    o[0] = 0;
#pragma unroll
    for (int e = 1; e < (1 << RB); ++e) {
      const int hb = 31 - __clz(e);
      o[e] = o[e ^ (1 << hb)] + sO[hb];
    }
#pragma unroll
    for (int e = 0; e < (1 << RB); e += 1 << LWO) {
      if (!(e & cmask)) {
        sstore<LWO>(dst + o[e], &v[e]);
        sstore<LWO>(dsn + o[e], &n[e]);
      }
    }
  }
}

// Renumber the register legs so that those at memory positions 0 and 1 of the
// input lead (state bits 0 and 1); returns how many do (0..2).  *out: how many of
// them sit at the same positions of the output and are stored there.
int lead_low_legs(const ChainParams &p, ChainParams *q, int *out) {
  const int RB = p.t;
  int l[2] = {-1, -1};
  for (int b = 0; b < RB; ++b)
    for (int j = 0; j < 2; ++j)
      if (p.hi_in[1 << b] == (1 << j)) l[j] = b;
  const int lw = l[0] < 0 ? 0 : l[1] < 0 ? 1 : 2;
  *out = 0;
  *q = p;
  if (lw == 0) return 0;
  const TGate &last = p.tg[p.ntg - 1];
  const int con = last.kind == 2 ? last.J : -1;
  for (int j = 0; j < lw && l[j] != con && p.hi_out[1 << l[j]] == (1 << j); ++j) ++*out;
  if (*out < lw) *out = 0;   // the kernel's forms: all of them or none
  int perm[8], next = lw;    // old leg -> new leg
  for (int b = 0; b < RB; ++b) perm[b] = b == l[0] ? 0 : (lw == 2 && b == l[1]) ? 1 : next++;
  for (int e = 0; e < (1 << RB); ++e) {
    int f = 0;
    for (int b = 0; b < RB; ++b)
      if ((e >> b) & 1) f |= 1 << perm[b];
    q->hi_in[f] = p.hi_in[e];
    q->hi_out[f] = p.hi_out[e];
  }
  for (int i = 0; i < p.ntg; ++i) {
    TGate &t = q->tg[i];
    const int J = t.J >= 0 ? perm[t.J] : -1, K = t.K >= 0 ? perm[t.K] : -1;
    t.J = (int8_t)J;
    t.K = (int8_t)K;
    t.code = (int16_t)(t.kind == 0   ? J * 7 + K + 1
                       : t.kind == 2 ? 100 + J * 7 + K + 1
                                     : 42 + (J + 1) * 7 + K + 1);
  }
  return lw;
}

template <int RB, int LWI, int LWO, typename I>
cudaError_t run(const ChainParams &p, const char *arena, const void *Ax, const uint64_t *An,
                void *Cx, uint64_t *Cn, const Batch &bt, cudaStream_t st) {
  constexpr int NT = 128, MINB = 5;
  // one wave of resident blocks that walk equal numbers of outer indices: every block
  // builds the gate tables first (a few dependent loads)
  const int64_t need = (p.outer + NT - 1) / NT;
  const int64_t slots = (int64_t)MINB * num_sms();
  const int64_t trips = (need * bt.B + slots - 1) / slots;
  const int64_t blocks = (need + trips - 1) / trips;
  k_schain<RB, LWI, LWO, I, NT, MINB><<<dim3((unsigned)blocks, bt.B), NT, 0, st>>>(
      p, reinterpret_cast<const int32_t *>(arena), reinterpret_cast<const uint64_t *>(arena),
      static_cast<const int32_t *>(Ax), An, static_cast<int32_t *>(Cx), Cn, bt.ib);
  return cudaGetLastError();
}

template <int RB>
cudaError_t run_rb(const ChainParams &p, const char *arena, const void *Ax, const uint64_t *An,
                   void *Cx, uint64_t *Cn, const Batch &bt, cudaStream_t st) {
  if (p.outer << RB >= (int64_t(1) << 31))
    return run<RB, 0, 0, int64_t>(p, arena, Ax, An, Cx, Cn, bt, st);
  ChainParams q;
  int lwo = 0;
  int lw = lead_low_legs(p, &q, &lwo);
  // vector accesses: every array start and the instance stride are multiples of 16
  // bytes (tensors start on 256-byte boundaries)
  if ((reinterpret_cast<uintptr_t>(Ax) | reinterpret_cast<uintptr_t>(Cx) |
       reinterpret_cast<uintptr_t>(An) | reinterpret_cast<uintptr_t>(Cn) | (uintptr_t)bt.ib) % 16)
    lw = 0;
  if (lw == 0) return run<RB, 0, 0, int32_t>(p, arena, Ax, An, Cx, Cn, bt, st);
  if (lw == 1)
    return lwo ? run<RB, 1, 1, int32_t>(q, arena, Ax, An, Cx, Cn, bt, st)
               : run<RB, 1, 0, int32_t>(q, arena, Ax, An, Cx, Cn, bt, st);
  return lwo ? run<RB, 2, 2, int32_t>(q, arena, Ax, An, Cx, Cn, bt, st)
             : run<RB, 2, 0, int32_t>(q, arena, Ax, An, Cx, Cn, bt, st);
}

}  // namespace

cudaError_t launch_schain(const ChainParams &p, const char *arena, const void *Ax,
                          const uint64_t *An, void *Cx, uint64_t *Cn, const Batch &bt,
                          cudaStream_t st) {
  if (p.outer == 0) return cudaSuccess;
  if (p.ntg < 1 || p.P != 1) return cudaErrorInvalidValue;
  if (p.t == 4) return run_rb<4>(p, arena, Ax, An, Cx, Cn, bt, st);
  return cudaErrorInvalidValue;
}

}  // namespace tn
