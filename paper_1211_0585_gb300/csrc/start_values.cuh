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

// threads a CTA for n columns: 256, or 64 where that would leave SMs without a CTA (FP64 work: 16 cycles a warp
// instruction and SM)
inline int start_value_threads(long long n) { return n < 256 * 300 ? 64 : 256; }

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

// The first l >= m at which the scaled recurrence from lambda_mm = v 2^e reaches 2^cut, and the values there and at
// l + 1 (0 past lmax); returns none if it never does. rec: the column's coefficients (a_l, b_l) from l = m. The
// coefficients are loaded kRecAhead steps before their use: one at a time, a load's latency was the loop's.
constexpr int kRecAhead = 8;
__device__ __forceinline__ int walk_to_cut(const double2 *rec, double x, double v, int e, int m, int lmax, int cut,
                                           int none, double &v0, double &v1) {
  double p2 = v, p1 = x * sqrt(2.0 * m + 3.0) * v;   // lambda_l, lambda_{l+1} (scaled)
  double2 ab[kRecAhead];                             // of l + 2, l + 3, ..
#pragma unroll
  for (int j = 0; j < kRecAhead; ++j) ab[j] = rec[min(2 + j, lmax - m)];
  for (int l0 = m; l0 <= lmax; l0 += kRecAhead) {
#pragma unroll
    for (int j = 0; j < kRecAhead; ++j) {            // compile-time buffer indices
      const int l = l0 + j;
      if (l > lmax) return none;
      if (p2 != 0.0 && exponent_of(p2) + e >= cut) {
        v0 = ldexp(p2, e);
        v1 = (l + 1 <= lmax) ? ldexp(p1, e) : 0.0;
        return l;
      }
      if (l + 2 <= lmax) {
        const double nx = ab[j].x * x * p1 - ab[j].y * p2;
        ab[j] = rec[min(l + 2 + kRecAhead, lmax) - m];
        p2 = p1;
        p1 = nx;
        if (exponent_of(p2) >= 400 || exponent_of(p1) >= 400) { p1 *= 0x1p-400; p2 *= 0x1p-400; e += 400; }
      } else {
        p2 = p1;
        p1 = 0.0;
      }
    }
  }
  return none;
}

}  // namespace wfk
