// GELU in its erf form and its derivative, FP32, for the surrogate's dense
// layers (the tiled and the tcgen05 GEMM epilogues share them, so both
// paths train the same function), and the optimiser's update.
#pragma once

namespace cem {

// GELU(z) = z Phi(z) = z (1 + erf(z / sqrt 2)) / 2
__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }

// GELU'(z) = Phi(z) + z phi(z)
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// both at once (they share the erf)
__device__ __forceinline__ void gelu_both(float z, float& act, float& grad) {
  act = gelu(z);
  grad = gelu_grad(z);
}

// one AdamW update (decoupled decay) of a parameter x and its moments by the
// gradient g; c1, c2: the bias corrections 1 - b^t.  The roundings are written
// out: training follows every last bit of its first steps.
__device__ __forceinline__ void adamw_value(float& x, float& m1, float& m2, float g, int decay, float lr, float b1, float b2,
                                            float eps, float wd, float c1, float c2) {
  const float a = __fmaf_rn(1.0f - b1, g, __fmul_rn(b1, m1));
  const float v = __fmaf_rn(__fmul_rn(1.0f - b2, g), g, __fmul_rn(b2, m2));
  m1 = a;
  m2 = v;
  const float kept = __fmaf_rn(-__fmul_rn(lr, decay ? wd : 0.0f), x, x);
  x = __fsub_rn(kept, __fmul_rn(lr, a / c1) / (sqrtf(v / c2) + eps));
}

// the same on parameter i in memory; returns the new parameter
__device__ __forceinline__ float adamw(float* __restrict__ p, float* __restrict__ m1, float* __restrict__ m2, int i, float g,
                                       int decay, float lr, float b1, float b2, float eps, float wd, float c1, float c2) {
  float x = p[i], a = m1[i], v = m2[i];
  adamw_value(x, a, v, g, decay, lr, b1, b2, eps, wd, c1, c2);
  m1[i] = a;
  m2[i] = v;
  p[i] = x;
  return x;
}

}  // namespace cem
