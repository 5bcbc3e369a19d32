// gate_dev.cuh -- outer-index decoding of the gate kernels.
#pragma once
#include <stdint.h>

#include <algorithm>

#include "tn_internal.h"

namespace tn {

// Offsets of outer index r in A, B and C.  I = int32_t where gate_fits32: a 64-bit
// digit costs about 20 instructions (three 64-bit products), a 32-bit one five, and a
// small step does little else (6 x 6 chimera, 2^24 elements: adding two tensors 75 -> 45 us,
// the counting form 115 -> 89 us; contractions of 2 states to 16 new ones 70 -> 22 us,
// with the compile-time form and 16-byte stores).
template <typename I>
__device__ __forceinline__ void gate_decode(const GateParams &p, I r, I &oa, I &ob, I &oc) {
  oa = ob = oc = 0;
  for (int s = p.nseg - 1; s >= 0; --s) {
    I i;
    if (p.seg_sh[s] >= 0) {
      i = r & (I)(p.seg_size[s] - 1);
      r >>= p.seg_sh[s];
    } else if constexpr (sizeof(I) == 4) {
      const uint32_t q = (uint32_t)r / (uint32_t)p.seg_size[s];
      i = r - (I)(q * (uint32_t)p.seg_size[s]);
      r = (I)q;
    } else {
      i = r % p.seg_size[s];
      r /= p.seg_size[s];
    }
    oa += i * (I)p.seg_sA[s];
    ob += i * (I)p.seg_sB[s];
    oc += i * (I)p.seg_sC[s];
  }
}

// whether every outer index (and a grid stride past it) and every element offset of the
// step fits 32 bits
inline bool gate_fits32(const GateParams &p) {
  int64_t a = 0, b = 0, c = 0, ka = 0, kb = 0, nb = 0, nc = 0;
  for (int s = 0; s < p.nseg; ++s) {
    a += (p.seg_size[s] - 1) * p.seg_sA[s];
    b += (p.seg_size[s] - 1) * p.seg_sB[s];
    c += (p.seg_size[s] - 1) * p.seg_sC[s];
  }
  for (int k = 0; k < p.Ks; ++k) {
    ka = std::max(ka, p.kA[k]);
    kb = std::max(kb, p.kB[k]);
  }
  for (int n = 0; n < p.Ns; ++n) {
    nb = std::max(nb, p.nB[n]);
    nc = std::max(nc, p.nC[n]);
  }
  const int64_t lim = int64_t(1) << 31;
  return p.outer < lim / 2 && a + ka < lim && b + kb + nb < lim && c + nc < lim;
}

}  // namespace tn
