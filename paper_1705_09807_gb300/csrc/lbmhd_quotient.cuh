// Binary64 quotients that share a divisor: one correctly rounded reciprocal and three instructions
// each, where a division takes about ten on units that set the time.
#pragma once

#include <cuda_runtime.h>

namespace lbmhd_gpu {
namespace {

// a / b from y = 1 / b rounded to nearest: Markstein's correction (IBM J. Res. Dev. 34 (1990) 111)
// of a y by its exact residual, the correctly rounded quotient but for ties that 2^-100 decides.
__device__ __forceinline__ double quotient(double a, double b, double y) {
  const double q = a * y;
  return fma(fma(-q, b, a), y, q);
}

// Exponents for which nothing over- or underflows on the way (a may be zero), by integer tests.
__device__ __forceinline__ bool in_range(double v) {
  return ((unsigned)__double2hiint(v) & 0x7fffffffu) - 0x30000000u < 0x20000000u;  // 2^-255 .. 2^257
}
__device__ __forceinline__ bool is_zero(double v) {
  return (((unsigned)__double2hiint(v) & 0x7fffffffu) | (unsigned)__double2loint(v)) == 0u;
}
__device__ __forceinline__ bool quotient_in_range(double a, double b) {
  return in_range(b) && (in_range(a) || is_zero(a));
}

}  // namespace
}  // namespace lbmhd_gpu
