// gate_dev.cuh -- outer-index decoding of the gate kernels.
#pragma once
#include <stdint.h>

#include "kernels.h"

namespace tn {

// Offsets of outer index r in A, B and C.  I = int32_t where gate_fits32 (kernels.h): a 64-bit
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

}  // namespace tn
