// pair_ops.cuh -- arithmetic on two lattice cells at once. The two cells are the lanes of a packed
// f32x2 register pair, so one instruction does both; each lane is rounded exactly as the scalar
// operation, so results do not depend on which cells share a pair.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b: the product with -1 is exact, so this rounds once
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, dup2(-1.0f), a); }

}  // namespace lbm
