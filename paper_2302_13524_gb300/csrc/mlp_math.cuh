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
//
// IEEE division and square root leave their fast path for denormal operands,
// and a weight whose gradient has vanished holds a denormal m for good (0.9 m
// rounds back to m): in a long training run that made the weight updates, which
// are bound by memory otherwise, twice as slow (a step of batch 256, 8192 x 1024 x
// 1024 x 4096, after a thousand steps with its weights read back: 424 us against
// 284 at the start of the run; 260 now throughout, with the tiles of gemm_tc.cu).
// So the operands are kept out of that range without moving the result: below 1e-31, sqrt(v / c2) is less than
// half an ulp of eps, and a small m is scaled by a power of two around the
// divisions.
__device__ __forceinline__ void adam_update(float &w, float g, float &m, float &v, float lr, float c1, float c2)
{
    m = 0.9f * m + 0.1f * g;
    v = 0.999f * v + 0.001f * g * g;
    const bool small = fabsf(m) < 1e-20f;
    const float ms = m * (small ? 0x1p64f : 1.f);
    const float step = lr * (ms / c1) / (sqrtf(fmaxf(v, 1e-31f * c2) / c2) + 1e-8f);
    w = w - step * (small ? 0x1p-64f : 1.f);
}

}  // namespace tmr
