// Pairs of FP32 numbers: unevaluated sums h + l that carry about 48 bits (Knuth's TwoSum, FMA TwoProd).
// Sums and products that need more than FP32 use them up to the point where FP64 takes over: this chip
// does 64 FP32 operations for one in FP64, a conversion between the two included.
#pragma once

#include <cuda_runtime.h>

namespace pic {

// a + b = s + e exactly
__device__ __forceinline__ void add2(float a, float b, float& s, float& e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

struct PairSum {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void add(float h2, float l2) {
        float s, e;
        add2(h, h2, s, e);
        h = s;
        l += e + l2;
    }
    // += x (dh + dl)
    __device__ __forceinline__ void fma(float x, float dh, float dl) {
        const float p = x * dh;
        add(p, fmaf(x, dl, fmaf(x, dh, -p)));
    }
    // *= ch + cl
    __device__ __forceinline__ void scale(float ch, float cl) {
        const float p = h * ch;
        l = fmaf(h, ch, -p) + fmaf(h, cl, l * ch);
        h = p;
    }
    // the sum over a warp, in every lane
    __device__ __forceinline__ void warp_sum() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float h2 = __shfl_xor_sync(0xffffffffu, h, o), l2 = __shfl_xor_sync(0xffffffffu, l, o);
            add(h2, l2);
        }
    }
    __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};

}  // namespace pic
