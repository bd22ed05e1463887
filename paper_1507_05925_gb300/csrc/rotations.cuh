// Givens rotations of the GMRES steps, by one thread in FP64.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace bie {

// The rotation that takes (x, y) to (r, 0).
__device__ __forceinline__ void givens(double x, double y, double& c, double& s, double& r) {
  const double q = fma(x, x, y * y);
  if (q > 1e-280 && q < 1e280) {
    const double i = rsqrt(q);
    r = q * i;
    c = x * i;
    s = y * i;
    return;
  }
  r = hypot(x, y);
  c = r > 0.0 ? x / r : 1.0;
  s = r > 0.0 ? y / r : 0.0;
}

// The previous rotations (css, sns) on column h[0..j], the running entry in a register: one
// FP64 multiply-add a rotation is the chain (through shared memory it was 450 clocks).
// Returns the last entry.
__device__ __forceinline__ double rotate_column(const double* css, const double* sns, double* h, int j) {
  double x = h[0];
#pragma unroll 4
  for (int i = 0; i < j; ++i) {
    const double c = css[i], s = sns[i], y = h[i + 1];
    h[i] = fma(c, x, s * y);
    x = fma(-s, x, c * y);
  }
  return x;
}

}  // namespace bie
