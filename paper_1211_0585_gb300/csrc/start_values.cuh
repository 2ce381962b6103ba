// Shared parts of the kernels that find each (m, ring pair)'s first Legendre
// term (FP64 and double-float cuts): lambda_mm as a scaled value with an
// explicit binary exponent.
#pragma once

#include <cuda_runtime.h>

namespace wfk {

// floor(log2 |v|) of v != 0 (ilogb), from the exponent bits
__device__ __forceinline__ int exponent_of(double v) {
  const int b = (__double2hiint(v) >> 20) & 0x7ff;
  return b ? b - 1023 : ilogb(v);
}

// croot[i] = sqrt((2i + 1) / 2i), i = 1 .. mmax, by the whole CTA (barrier at the end)
__device__ __forceinline__ void lambda_mm_factors(double *croot, int mmax) {
  for (int i = 1 + threadIdx.x; i <= mmax; i += blockDim.x) croot[i] = sqrt((2.0 * i + 1.0) / (2.0 * i));
  __syncthreads();
}

// lambda_mm = (-1)^m sqrt((2m + 1) / 4 pi prod_{i <= m} (2i - 1) / 2i) sin^m(theta) = returned value 2^e (e starts
// at 0). The value is brought back up by 2^400 whenever it falls below 2^-400; powers of two, so that no digit
// depends on when.
__device__ __forceinline__ double lambda_mm_scaled(const double *croot, int m, double st, int &e) {
  double v = 0.28209479177387814347;  // 1 / sqrt(4 pi)
  for (int i = 1; i <= m; ++i) {
    v *= -croot[i] * st;
    if (exponent_of(v) < -400) { v *= 0x1p400; e -= 400; }
  }
  return v;
}

}  // namespace wfk
