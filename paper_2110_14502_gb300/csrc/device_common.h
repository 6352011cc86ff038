// Device helpers shared by the kernels.
#pragma once

#include <cuda_runtime.h>

#include "kernels.h"

namespace tn {

// Slice selection: offset in the leaf store of unit u's sub-tensor of a leaf
// (its fixed indices set to the unit's slice id and bitstring bits), and of the
// sub-tensor's element e.
__device__ __forceinline__ int64_t leaf_fixed_offset(const LeafGather& L, const GroupInfo& g, int u) {
  const int64_t s = g.slice0 + u % g.nslice;
  const int64_t b = g.b0 + u / g.nslice;
  int64_t o = L.store_off;
  for (int f = 0; f < L.nfixed; ++f) {
    const int src = L.fixed_src[f];
    int v;
    if (src >= 0) v = (int)((s >> src) & 1);
    else {
      const int q = -src - 2;
      v = (int)((g.bits[b * g.words + (q >> 6)] >> (q & 63)) & 1);
    }
    if (v) o += L.fixed_stride[f];
  }
  return o;
}
__device__ __forceinline__ int64_t leaf_kept_offset(const LeafGather& L, int64_t fixed_off, int e) {
  int64_t o = fixed_off;
  for (int p = 0; p < L.nkept; ++p)
    if ((e >> (L.nkept - 1 - p)) & 1) o += L.kept_stride[p];
  return o;
}

// Multiplication by 2^e for the exponent shifts of the scaled formats.  A
// power of two in the normal range multiplies exactly, so one multiply gives
// the correctly rounded x 2^e (the value ldexpf returns); shifts outside
// [-126, 127] go through ldexpf.
struct Pow2 {
  int e;
  float f;
  bool direct;
  __device__ explicit Pow2(int e_) {
    e = e_;
    direct = e_ >= -126 && e_ <= 127;
    f = __int_as_float((min(max(e_, -126), 127) + 127) << 23);
  }
  __device__ float operator()(float x) const { return direct ? x * f : ldexpf(x, e); }
};

}  // namespace tn
