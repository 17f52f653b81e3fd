// Sums and products that need FP64 or more, out of FP32 and integer operations: this chip does 64 FP32
// operations for one in FP64, a conversion between the two included.  Plain C++ (compiled without contraction)
// as well as device code.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define PIC_HD __host__ __device__ __forceinline__
#else
#define PIC_HD inline
#endif

namespace pic {

// One rounding each: the compiler may fuse a plain product into the sum that uses it, and the error terms
// below would then belong to another sum.
#ifdef __CUDA_ARCH__
PIC_HD float add_rn(float a, float b) { return __fadd_rn(a, b); }
PIC_HD float sub_rn(float a, float b) { return __fsub_rn(a, b); }
PIC_HD float mul_rn(float a, float b) { return __fmul_rn(a, b); }
#else
PIC_HD float add_rn(float a, float b) { return a + b; }
PIC_HD float sub_rn(float a, float b) { return a - b; }
PIC_HD float mul_rn(float a, float b) { return a * b; }
#endif

// a + b = s + e exactly (Knuth's TwoSum)
PIC_HD void two_sum(float a, float b, float& s, float& e) {
    const float t = add_rn(a, b), bb = sub_rn(t, a);
    e = add_rn(sub_rn(a, sub_rn(t, bb)), sub_rn(b, bb));
    s = t;
}
// a b = p + e exactly (FMA TwoProd; |a b| from 2^-100 up)
PIC_HD void two_prod(float a, float b, float& p, float& e) {
    p = mul_rn(a, b);
    e = fmaf(a, b, -p);
}

// A sum kept as h + m + l, unevaluated: an addition loses about 2^-72 of |h|, where FP64 loses 2^-53.
struct WideSum {
    float h = 0.f, m = 0.f, l = 0.f;
    PIC_HD void add(float a, float b, float c) {           // += a + b + c, |a| >> |b| >> |c|
        float e, f, g;
        two_sum(h, a, h, e);
        two_sum(m, b, m, f);
        two_sum(m, e, m, g);
        l += (f + g) + c;
    }
    PIC_HD void add(float a) {
        float e, g;
        two_sum(h, a, h, e);
        two_sum(m, e, m, g);
        l += g;
    }
    // += x (dh + dm + dl); returns the largest part of the product
    PIC_HD float fma(float x, float dh, float dm, float dl = 0.f) {
        float p, r, q, t, e;
        two_prod(x, dh, p, r);
        two_prod(x, dm, q, t);
        two_sum(r, q, r, e);
        add(p, r, fmaf(x, dl, e + t));
        return p;
    }
#ifdef __CUDACC__
    __device__ __forceinline__ void add_lane(const WideSum& s, int o) {       // += the s of the lane at distance o
        add(__shfl_xor_sync(0xffffffffu, s.h, o), __shfl_xor_sync(0xffffffffu, s.m, o), __shfl_xor_sync(0xffffffffu, s.l, o));
    }
#endif
    PIC_HD double value() const { return (double)h + ((double)m + (double)l); }
};

}  // namespace pic
