// Device side of a batched launch (BatchParams, kernels.h).
#pragma once

#include "kernels.h"

namespace tn {

__device__ __forceinline__ int64_t batch_offset(const BatchParams& p, const BatchOperand& o, int b) {
  if (o.n_bits == 0) return b * o.stride;
  const int64_t q = p.q0 + b;
  const int64_t id = (q >> p.ni) | ((q & ((1LL << p.ni) - 1)) << p.k);
  int64_t v = 0;
  for (int t = 0; t < o.n_bits; ++t) v |= ((id >> o.bits[t]) & 1) << t;
  return v * o.var_size;
}

}  // namespace tn
