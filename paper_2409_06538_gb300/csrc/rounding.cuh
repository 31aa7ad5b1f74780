// Short forms of operations whose special cases cost more than the operation, each with the range it
// holds in; tests/test_gpu_rounding.py compares them with the full forms over every float of the range.
// Below them the roots and rotations of the environment build (tests/test_gpu_rotations.py).
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace tnmc {

// 1 / x, correctly rounded for x in [1e-37, 8e37]: the hardware's approximation and one Newton step with a
// fused residual (Markstein 1990).  The division's branch for its special cases keeps it from overlapping
// with the operations around it.  Above 2^126, where 1 / x is subnormal, the approximation flushes to zero.
__device__ __forceinline__ float inverse(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return fmaf(r, fmaf(-x, r, 1.0f), r);
}

__device__ __forceinline__ float tf32_rna(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}
// The same rounding of a finite x below the largest binade, in two integer operations: half of the 11-bit
// significand's last place is added to the magnitude and the rest cut off.  cvt.rna takes four issue slots.
__device__ __forceinline__ float tf32_rna_finite(float x) {
  return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u);
}

// Square root of a column's squared norm.  In FP64 from the reciprocal root and one step of Newton's
// iteration, s + (ss - s^2) / (2 s): half the instructions of the pipe that the factorisation waits for.
__device__ __forceinline__ float norm_of(float ss) { return sqrtf(ss); }
__device__ __forceinline__ double norm_of(double ss) {
  if (!(ss > 0.0 && ss < INFINITY)) return ss;
  const double r = rsqrt(ss), s = ss * r;
  return fma(0.5 * r, fma(-s, s, ss), s);
}

// Jacobi rotation (c, s) that makes columns p, q orthogonal, from a = |y_p|^2, b = |y_q|^2,
// g = y_p . y_q (y_p' = c y_p - s y_q, y_q' = s y_p + c y_q).  The angle solves
// tan 2theta = 2g / (b - a) with |theta| <= pi/4:
//   r = sqrt((b-a)^2 + 4 g^2), cos 2theta = |b-a| / r, c = sqrt((1 + cos 2theta) / 2),
//   s = sgn(b-a) g / (r c)   (sgn(0) = +1),
// two reciprocal square roots in sequence instead of the divide/sqrt chain of the tangent
// form.  FP32 uses the hardware rsqrt with one Newton step each, so c^2 + s^2 = 1 to
// working precision; FP64 calls the library's, which leaves out a root and a division each.
__device__ __forceinline__ float rsqrt_nr(float x) {
  const float r = rsqrtf(x);
  return r * fmaf(-0.5f * x * r, r, 1.5f);
}
__device__ __forceinline__ void rotation_from_gram(double a, double b, double g, double& c, double& s) {
  const double d = b - a;
  const double rinv = rsqrt(fma(d, d, 4.0 * g * g));
  const double h = fma(0.5 * fabs(d), rinv, 0.5);
  const double ic = rsqrt(h);
  c = h * ic;
  s = (d < 0.0 ? -g : g) * rinv * ic;
}
__device__ __forceinline__ void rotation_from_gram(float a, float b, float g, float& c, float& s) {
  const float d = b - a;
  const float rinv = rsqrt_nr(fmaf(d, d, 4.0f * g * g));
  const float h = fmaf(0.5f * fabsf(d), rinv, 0.5f);
  const float ic = rsqrt_nr(h);
  c = h * ic;
  s = (d < 0.0f ? -g : g) * rinv * ic;
}

}  // namespace tnmc
