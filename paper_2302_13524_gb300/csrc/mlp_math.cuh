// mlp_math.cuh -- the elementwise functions of the learned initialiser's
// network, shared by its kernels (mlp.cu) and the GEMM's epilogues (gemm_tc.cu).
#pragma once

namespace tmr {

__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float x)
{
    return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * expf(-0.5f * x * x) * 0.39894228040143268f;
}

// One Adam update (beta1 0.9, beta2 0.999, eps 1e-8) of weight w with gradient
// g; c1, c2: the bias corrections 1 - beta^step.
__device__ __forceinline__ void adam_update(float &w, float g, float &m, float &v, float lr, float c1, float c2)
{
    m = 0.9f * m + 0.1f * g;
    v = 0.999f * v + 0.001f * g * g;
    w = w - lr * (m / c1) / (sqrtf(v / c2) + 1e-8f);
}

}  // namespace tmr
