// FP64 operations of the 2D and 3D diagnostics done by integer instructions:
// GB300 issues an FP64 instruction every 17 cycles per SM.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

// max(m, |v|) for m >= 0; NaN in v is ignored, as fmax does.  FP64 by the bits
// (non-negative doubles order like their bits), off the FP64 pipe.
__device__ __forceinline__ float abs_max(float m, float v) { return fmax(m, fabs(v)); }
__device__ __forceinline__ double abs_max(double m, double v) {
  const long long b = __double_as_longlong(v) & 0x7fffffffffffffffll, a = __double_as_longlong(m);
  return b > a && b <= 0x7ff0000000000000ll ? __longlong_as_double(b) : m;
}

// 64-bit integer to double, to nearest (ties away from zero), by integer
// instructions: the conversion instruction runs on the narrow FP64 pipe.
__device__ __forceinline__ double i64_to_f64(long long v) {
  const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int n = __clzll((long long)a);
  unsigned long long x = a << (n & 63);
  const unsigned long long r = x + 0x400ull;
  const unsigned carry = r < x;  // all ones rounded up: the next power of two
  const unsigned e = n == 64 ? 0u : (unsigned)(1023 + 63 - 1 - n) << 20;
  const unsigned hi = (unsigned)(r >> 43) + e + (carry << 21);
  return __hiloint2double((int)(hi | (v < 0 ? 0x80000000u : 0u)), (int)(unsigned)(r >> 11));
}

}  // namespace lbm
