// FP64 scalars of a Jacobi rotation with few instructions of the FP64 pipe, which takes a warp
// instruction for 64 cycles of its quarter of an SM whatever its lanes do (measured; a division is 23
// of them, a square root 13): seeds in FP32, one or two corrections in FP64, tests on the bits.
#pragma once
#include <cuda_runtime.h>

namespace mrd {

__device__ __forceinline__ bool bits_less_equal(double a, double b) {   // of non-negative numbers
  return __double_as_longlong(a) <= __double_as_longlong(b);
}

// x 2^k for a normal result; numbers that would leave the normal range downwards, and denormal ones, give zero.
__device__ __forceinline__ double scale2(double x, int k) {
  const int hi = __double2hiint(x), f = (hi >> 20) & 0x7ff;
  return f == 0 || f + k <= 0 ? 0.0 : __hiloint2double(hi + (k << 20), __double2loint(x));
}

// A float close to |x| (truncated mantissa; |x| within the FP32 exponent range), and a double from a normal
// float, without the FP64 pipe.
__device__ __forceinline__ float mag_f32(double x) {
  const int hi = __double2hiint(x) & 0x7fffffff;
  return __int_as_float(((hi >> 20) - 1023 + 127) << 23 | (hi & 0xfffff) << 3 | (int)((unsigned)__double2loint(x) >> 29));
}
__device__ __forceinline__ double from_f32(float x) {
  const int i = __float_as_int(x);
  return __hiloint2double((i & 0x80000000) | (((i >> 3) & 0x0fffffff) + ((1023 - 127) << 20)), i << 29);
}

// 1 / sqrt(x), x > 0 normal, to 2 ulp: an FP32 seed y with e = 1 - x y^2 (|e| below 2^-20), and the binomial
// series of y (1 - e)^(-1/2) to second order, y (1 + e / 2 + 3 e^2 / 8); the next term, 5 e^3 / 16, is below
// 2^-61.
__device__ __forceinline__ double rsqrt_fp64(double x) {
  const int hi = __double2hiint(x);
  const int k = ((hi >> 20) - 1023) & ~1;                                    // x = m 2^k, m in [1, 4)
  const double m = __hiloint2double(hi - (k << 20), __double2loint(x));
  const double y = from_f32(rsqrtf(mag_f32(m)));
  const double e = fma(-(m * y), y, 1.0);
  const double r = fma(y * e, fma(0.375, e, 0.5), y);
  return __hiloint2double(__double2hiint(r) - ((k / 2) << 20), __double2loint(r));
}

// t = sign(zeta) / (|zeta| + sqrt(1 + zeta^2)), |zeta| below 2^120, to rounding: in FP32, then two Newton
// steps for t^2 + 2 zeta t = 1 with the FP32 slope (one step leaves 2^-44, from the slope's rounding).
__device__ __forceinline__ double jacobi_tangent(double zeta) {
  const int ex = ((__double2hiint(zeta) >> 20) & 0x7ff) - 1023;
  const bool neg = __double2hiint(zeta) < 0;
  const float z = ex < -60 ? 0.f : mag_f32(zeta);
  const float t0 = z > 1e9f ? 0.5f / z : 1.f / (z + sqrtf(1.f + z * z));
  const double r0 = from_f32(0.5f / (t0 + z));             // 1 / f'
  const double zz = neg ? -zeta : zeta;
  double t = from_f32(t0);
  t = fma(-fma(t, fma(2.0, zz, t), -1.0), r0, t);
  t = fma(-fma(t, fma(2.0, zz, t), -1.0), r0, t);
  return neg ? -t : t;
}

}  // namespace mrd
