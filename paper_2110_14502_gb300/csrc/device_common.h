// Device helpers shared by the kernels.
#pragma once

#include <cuda_runtime.h>

namespace tn {

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
