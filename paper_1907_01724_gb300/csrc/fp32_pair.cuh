// Device helpers of the pair sums (pair, field, move and allocation-free kernels): the MUFU
// reciprocal square root (FP32, and refined to FP64), cp.async staging, and the (hi, lo) FP32 split of an FP64 value.
#pragma once
#include <cuda_runtime.h>

#include "df64.cuh"

namespace hsma {

// 1/sqrt(x) by one MUFU instruction (rsqrt.approx, ~2^-22.9 relative; flushes subnormals).
__device__ __forceinline__ float rsqrt_mufu(float x)
{
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 1/sqrt(x): the approximate reciprocal root y, then, with e = 1 - x y^2, the binomial series of
// (1 - e)^(-1/2): y + y e (1/2 + 3/8 e).  y has 21 significant bits (the instruction leaves the low
// word zero), so y^2 is exact and e, |e| <= 2^-19.04, has one rounding of 2^-72; the next term of the
// series, 5/16 e^3, is below 2^-58.  So the error is the last operation's rounding: over
// 2^28 arguments at most 1.016 x 2^-53, rms 0.433, as CUDA's rsqrt(); the root and the division that
// it replaces 1.499 and 0.601, and the same step with e = 1 - (x y) y 1.257 and 0.481.
// Arguments whose exponent leaves no room for the step (zero, subnormal, near overflow, not finite)
// take the square root and the division.
__device__ __forceinline__ double rsqrt_f64(double x)
{
  const unsigned int top = (unsigned int)__double2hiint(x) >> 20;  // sign and exponent
  if (top - 0x040u > 0x780u - 0x040u) return 1.0 / sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y * y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// 1/s for the power of two s above x > 0: s = 2^(e + 1) for x in [2^e, 2^(e + 1)) (a unit of length
// whose scalings are exact)
__device__ __forceinline__ float inv_unit(float x)
{
  return __int_as_float(0x7e800000 - (__float_as_int(x) & 0x7f800000));
}

// 16-byte asynchronous global -> shared copy (both addresses 16-byte aligned), its commit group
// and the wait for all but the N most recent groups.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem)
{
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// x = hi + lo to ~2^-48 relative: hi = fl32(x), lo = fl32(x - hi) (split_double, df64.cuh).
__device__ __forceinline__ void split_hilo(double x, float& hi, float& lo) { split_double(x, hi, lo); }
__device__ __forceinline__ float2 split_pair(double x)
{
  float2 r;
  split_hilo(x, r.x, r.y);
  return r;
}

// 1/|a - b| of two hi/lo-split points: with dh the FP32 difference of the high parts (exact for
// nearby points) and dl that of the low parts, dh + dl is the coordinate difference to FP32
// relative accuracy at any distance.
__device__ __forceinline__ float inv_hilo(float ax, float ay, float az, float alx, float aly, float alz, float bx,
                                          float by, float bz, float blx, float bly, float blz)
{
  const float dx = ax - bx, dy = ay - by, dz = az - bz;
  const float ex = (alx - blx) + dx, ey = (aly - bly) + dy, ez = (alz - blz) + dz;
  float r2 = ex * ex;
  r2 = fmaf(ey, ey, r2);
  r2 = fmaf(ez, ez, r2);
  return rsqrt_mufu(r2);
}

}  // namespace hsma
