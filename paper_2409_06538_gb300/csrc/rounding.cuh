// Short forms of operations whose special cases cost more than the operation, each with the range it
// holds in; tests/test_gpu_rounding.py compares them with the full forms over every float of the range.
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

}  // namespace tnmc
