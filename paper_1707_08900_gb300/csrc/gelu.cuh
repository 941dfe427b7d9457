// The network's activation, exact GELU h Phi(h), and its derivative
// Phi(h) + h phi(h), by CUDA's erff and expf: at most 1.5e-7 off.  A degree-7 polynomial
// times exp2f in packed FP32x2 arithmetic takes 13 instead of 45 instructions per
// value, but was 3.4e-7 off as the derivative (refitted, 1.5e-7 at the least); an
// Adam step at 8 x 64^3 took 970 us with it and 1042 us like this.  In the forward pass
// it moves activations across a BF16 rounding now and then, which corrected runs
// amplify to 1e-4 of the state within eight steps.
#pragma once

#include <cuda_runtime.h>

namespace gbfd {
namespace cnn {

__device__ __forceinline__ float gelu(float h)
{
    return 0.5f * h * (1.0f + erff(h * 0.70710678118654752f));
}

__device__ __forceinline__ float gelu_grad(float h)
{
    return 0.5f * (1.0f + erff(h * 0.70710678118654752f)) +
           h * expf(-0.5f * h * h) * 0.39894228040143268f;
}

}  // namespace cnn
}  // namespace gbfd
