// lp_mlp.cuh -- constants and the device-side evaluation of the learned state
// estimator (8 -> 32 ReLU -> 1 sigmoid, BF16 weights, FP32 accumulation), and
// the eight stencil features it reads.
#pragma once

#include <cuda_bf16.h>

#include "lp_internal.cuh"

namespace lp {

constexpr int MLP_IN = 8;
constexpr int MLP_H = 32;
constexpr int OFF_B1 = MLP_H * MLP_IN;
constexpr int OFF_W2 = OFF_B1 + MLP_H;
constexpr int OFF_B2 = OFF_W2 + MLP_H;
constexpr int MLP_NPARAM = OFF_B2 + 1;
constexpr unsigned MLP_POLLS = 1u << 22;                         // seconds: the blocks of a cooperative launch all run
constexpr int MLP_EPOCHS = 1024;                                 // epochs of one training launch
constexpr int MLP_WORK = 2 + MLP_EPOCHS + 3 * (MLP_NPARAM + 1);        // floats: a flag, epoch losses, gradients, barrier

// logit of the network for features x
__device__ inline float mlp_logit(const float (&x)[MLP_IN], const __nv_bfloat16* __restrict__ w)
{
    float z = __bfloat162float(w[OFF_B2]);
#pragma unroll 4
    for (int j = 0; j < MLP_H; ++j) {
        float a = __bfloat162float(w[OFF_B1 + j]);
#pragma unroll
        for (int k = 0; k < MLP_IN; ++k) a = fmaf(__bfloat162float(w[j * MLP_IN + k]), x[k], a);
        z = fmaf(__bfloat162float(w[OFF_W2 + j]), a > 0.0f ? a : 0.0f, z);
    }
    return z;
}

__device__ inline float mlp_prob(const float (&x)[MLP_IN], const __nv_bfloat16* __restrict__ w)
{
    return 1.0f / (1.0f + __expf(-mlp_logit(x, w)));
}

// mlp_prob by a warp whose lanes hold the same x: a lane per hidden unit, their
// terms added in mlp_logit's order
__device__ inline float mlp_prob_warp(const float (&x)[MLP_IN], const __nv_bfloat16* __restrict__ w)
{
    const int j = (int)(threadIdx.x & 31u);
    float a = __bfloat162float(w[OFF_B1 + j]);
#pragma unroll
    for (int k = 0; k < MLP_IN; ++k) a = fmaf(__bfloat162float(w[j * MLP_IN + k]), x[k], a);
    const float h = a > 0.0f ? a : 0.0f, w2 = __bfloat162float(w[OFF_W2 + j]);
    float z = __bfloat162float(w[OFF_B2]);
#pragma unroll 4
    for (int q = 0; q < MLP_H; ++q)
        z = fmaf(__shfl_sync(0xffffffffu, w2, q), __shfl_sync(0xffffffffu, h, q), z);
    return 1.0f / (1.0f + __expf(-z));
}

// feature transform: log(1 + 10 |f|), with the sign kept for the divergence term
__device__ inline float feat_t(float f) { return log1pf(10.0f * fabsf(f)); }
__device__ inline float feat_ts(float f) { return copysignf(log1pf(10.0f * fabsf(f)), f); }

}  // namespace lp
