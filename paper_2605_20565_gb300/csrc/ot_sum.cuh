// ot_sum.cuh -- running sums in three floats, for kernels that FP64 additions would bound: an SM's FP64
// pipe does 1.6 additions (1.9 fused multiply-adds) per clock, measured with eight independent chains
// per thread and 64 warps; its FP32 pipes 128.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace ot {

// Sum of floats that carries 72 bits: the rounding error of each addition (Knuth's two-sum, exact) goes
// to the next float.
struct Sum3 {
    float a = 0.0f, b = 0.0f, c = 0.0f;
    __device__ __forceinline__ static float two_sum(float& s, float v) {
        const float t = __fadd_rn(s, v), u = __fsub_rn(t, s);
        const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, u)), __fsub_rn(v, u));
        s = t;
        return e;
    }
    __device__ __forceinline__ void add(float v) { c = __fadd_rn(c, two_sum(b, two_sum(a, v))); }
    // terms some 2^-20 (low) and 2^-40 (last) below the others
    __device__ __forceinline__ void low(float v) { c = __fadd_rn(c, two_sum(b, v)); }
    __device__ __forceinline__ void last(float v) { c = __fadd_rn(c, v); }
    __device__ __forceinline__ void add(const Sum3& v) { add(v.a), low(v.b), last(v.c); }
    __device__ __forceinline__ double value() const { return ((double)c + (double)b) + (double)a; }
};
// v is zero or 2^-40 <= |v| < 2^74: its products with multiples of 2^-62 below 1, and their rounding
// errors, are then floats, and no sum of them overflows.
__device__ __forceinline__ bool plain(float v) { return v == 0.0f || ((__float_as_uint(v) >> 23) & 0xFFu) - 87u < 114u; }

} // namespace ot
