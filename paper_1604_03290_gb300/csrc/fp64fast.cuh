// FP64 reciprocal and reciprocal square root for the FP64 kernels.
//
// On GB300 the FP64 unit takes a warp instruction every 16 cycles or so per
// SM, and a correctly rounded FP64 division or square root is a sequence of
// eight to ten of them: in the pair loops those sequences were half of all
// FP64 instructions (126 per pair in each neighbour pass).  The hardware's
// approximate reciprocals (rcp/rsqrt.approx.ftz.f64) run on another unit and
// give about 20 bits; one third-order step of Householder's method then
// leaves a relative error of the order of the rounding of its last operation:
//   1/x:        e = 1 - x y,    y (1 + e + e^2)             error e^3
//   1/sqrt(x):  e = 1 - x y^2,  y (1 + e/2 + 3 e^2 / 8)     error (5/16) e^3
// in three and five FP64 instructions.  The errors are at most 0.51 and 1.02
// units in the last place (0.5 and 1.5 for the correctly rounded division and
// for a division by a correctly rounded root), which
// tests/test_gpu_fp64_reciprocals.py derives and holds them to.  Operands outside 2^-959..2^961 (where
// the seed could flush or overflow), zero, negatives, infinities and NaN take
// the correctly rounded operations, out of line.  Divisions outside the pair
// loops keep the language's operator.
#pragma once

#include <stdint.h>

namespace sph {

// exponent field of x in [64, 1984): a positive normal number far from both ends
__device__ __forceinline__ bool mid_range(double x) {
  return (uint32_t)__double2hiint(x) - 0x04000000u < 0x78000000u;
}

static __device__ __noinline__ double rcp64_slow(double x) { return 1.0 / x; }
static __device__ __noinline__ double rsqrt64_slow(double x) { return x > 0.0 ? 1.0 / sqrt(x) : 0.0; }

__device__ __forceinline__ double rcp64(double x) {
  if (!mid_range(x)) return rcp64_slow(x);
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// 1 / sqrt(x), and 0 for x = 0 (a pair of coincident particles has no direction)
__device__ __forceinline__ double rsqrt64(double x) {
  if (!mid_range(x)) return rsqrt64_slow(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

}  // namespace sph
