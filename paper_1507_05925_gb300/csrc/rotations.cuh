// Scalar steps of GMRES: Givens rotations, by one thread in FP64, and the scale of the new
// basis vector.
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

// ||w - V h||^2 = ||w||^2 - ||h||^2 stands in for the sum over the new vector while h is that
// small a part: the rounding of ||h||^2 then is below a tenth of ||w||^2's own.
constexpr double kNormBySubtraction = 0x1p-10;

// 1/sqrt(h + l), h > 0 and l its low part, in FP32 to within (1/2 + 2^-15) ulp, as the
// rounded quotient of the FP64 root is: one Newton step on the quotient of the rounded root (1
// ulp off), whose residual 1 - (h + l) y^2 comes out of error-free products.  (FP64 by
// every thread costs the narrow pipe thousands of clocks.)
__host__ __device__ __forceinline__ float rsqrt_rounded(float h, float l) {
  const float y = 1.f / sqrtf(h);
  const float p = y * y, d = fmaf(y, y, -p);
  const float e = fmaf(-l, p, fmaf(-h, d, fmaf(-h, p, 1.f)));
  return fabsf(e) < 1e-3f ? fmaf(0.5f * y, e, y) : y;  // (y^2 outside FP32's range: no step)
}

}  // namespace bie
