// FP32 quotients a / c by one divisor, from its FP64 reciprocal (host and
// device code without other headers).
#pragma once

#include <cmath>
#include <cstring>

#if defined(__CUDACC__)
#define LD_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define LD_HOST_DEVICE inline
#endif

namespace ld {

// The reciprocal of c for scaled_quotient, or 0 where it has to divide.
inline double quotient_reciprocal(double c) {
  return std::fabs(c) > 1e-100 && std::fabs(c) < 1e100 ? 1.0 / c : 0.0;
}

// a / c rounded to FP64 and then to FP32; y from quotient_reciprocal.  q = a y
// is within two units of the quotient, and q + y (a - q c), the residual exact,
// is the quotient rounded to FP64 (Markstein, IBM J. Res. Dev. 34, 1990; where
// the significand of c is all ones it may be the neighbour): three operations
// instead of a division.  Zero and exponents where the residual could leave the
// range are divided.
LD_HOST_DEVICE float scaled_quotient(double a, double c, double y) {
#if defined(__CUDA_ARCH__)
  const int e = (__double2hiint(a) >> 20) & 0x7ff;
#else
  unsigned long long b;
  std::memcpy(&b, &a, sizeof b);
  const int e = (int)(b >> 52) & 0x7ff;
#endif
  if (y != 0.0 && e > 1023 - 400 && e < 1023 + 400) {
    const double q = a * y;
    return (float)std::fma(std::fma(-q, c, a), y, q);
  }
  return (float)(a / c);
}

}  // namespace ld
