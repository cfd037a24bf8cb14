// Reciprocals for the elimination chains: the hardware's approximation and Newton-Raphson steps.
#pragma once

namespace bte {

// 1 / p to FP32 rounding: the hardware's approximation and one Newton-Raphson step (the IEEE division
// is a call with special cases, about 250 cycles in the panel's chain)
__device__ __forceinline__ float recip(float p) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(p));
  return fmaf(r, fmaf(-p, r, 1.f), r);
}

// The same in FP64, with two steps (the approximation has about 20 bits).
__device__ __forceinline__ double recip(double p) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(p));
  r = fma(r, fma(-p, r, 1.0), r);
  return fma(r, fma(-p, r, 1.0), r);
}

}  // namespace bte
