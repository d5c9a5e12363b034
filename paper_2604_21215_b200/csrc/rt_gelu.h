// x Phi(x) and its derivative for the loops of wide batches (rt_wide_loop.cu, rt_wide_backward.cu): erfc by Abramowitz and Stegun 7.1.26, a third
// of the instructions of erff, which a step that applies it to 128 x 128 accumulators per CTA notices (4 us of a position before).
//
// In fp32 with a correctly rounded reciprocal and exponential (tests/test_gelu.py) the largest error of x Phi(x) over [-10, 10] is 4.3e-7, at x = 3.1, where
// a result is rounded by 2.4e-7 at most; 0.5 x (1 + erf) has 4.5e-7.  Relative to the result: 7e-7 for |x| < 1 (2e-7), 5e-5 for x in (-3, -2) (1e-5), 5e-4 in (-4, -3)
// (5e-4), 4e-3 in (-6, -5), where 1 + erf has lost everything.  The derivative is within 3.1e-7 (1.4e-7).  The values go on as bf16 (2e-3 of them), the
// derivative as an fp32 factor.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define RT_GELU_FN __host__ __device__ __forceinline__
#else
#define RT_GELU_FN inline
#endif

namespace rt {

constexpr float kErfcSlope = 0.3275911f * 0.70710678f;

// Phi(-|x|) from t = 1 / (1 + kErfcSlope |x|) and e = exp(-x^2 / 2)
RT_GELU_FN float phi_tail(float t, float e) {
  const float poly = t * fmaf(t, fmaf(t, fmaf(t, fmaf(t, 0.5f * 1.061405429f, -0.5f * 1.453152027f), 0.5f * 1.421413741f), -0.5f * 0.284496736f), 0.5f * 0.254829592f);
  return poly * e;
}
RT_GELU_FN float gelu_of(float x, float t, float e) {
  const float q = phi_tail(t, e);
  return x * (x < 0.f ? q : 1.0f - q);
}
RT_GELU_FN float gelu_grad_of(float x, float t, float e) {      // Phi(x) + x phi(x)
  const float q = phi_tail(t, e);
  return (x < 0.f ? q : 1.0f - q) + x * 0.3989422804014327f * e;
}

}  // namespace rt
