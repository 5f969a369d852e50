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

// one AdamW update of parameter i (decoupled decay), moments included; c1, c2
// the bias corrections 1 - b^t.  Returns the new parameter.
__device__ __forceinline__ float adamw(float* __restrict__ p, float* __restrict__ m1, float* __restrict__ m2, int i, float g,
                                       int decay, float lr, float b1, float b2, float eps, float wd, float c1, float c2) {
  const float a = b1 * m1[i] + (1.0f - b1) * g;
  const float v = b2 * m2[i] + (1.0f - b2) * g * g;
  m1[i] = a;
  m2[i] = v;
  float x = p[i];
  x = x - lr * (decay ? wd : 0.0f) * x - lr * (a / c1) / (sqrtf(v / c2) + eps);
  p[i] = x;
  return x;
}

}  // namespace cem
