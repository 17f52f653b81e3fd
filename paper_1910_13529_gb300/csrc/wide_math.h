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
    // *= ch + cm + cl
    PIC_HD void scale(float ch, float cm, float cl) {
        float p, e, q, t, r, u, f, g;
        two_prod(h, ch, p, e);
        two_prod(h, cm, q, t);
        two_prod(m, ch, r, u);
        two_sum(q, r, q, f);
        two_sum(e, q, e, g);
        l = ((f + g) + (t + u)) + fmaf(h, cl, fmaf(m, cm, l * ch));
        h = p;
        m = e;
    }
    PIC_HD void normalise() {                              // h the nearest FP32 of the sum, m of the rest
        float e;
        two_sum(h, m, h, m);
        two_sum(m, l, m, l);
        two_sum(h, m, h, e);
        m = e;
    }
#ifdef __CUDACC__
    __device__ __forceinline__ void add_lane(const WideSum& s, int o) {       // += the s of the lane at distance o
        add(__shfl_xor_sync(0xffffffffu, s.h, o), __shfl_xor_sync(0xffffffffu, s.m, o), __shfl_xor_sync(0xffffffffu, s.l, o));
    }
#endif
    PIC_HD double value() const { return (double)h + ((double)m + (double)l); }
};

// gamma - 1 of a momentum u as a WideSum, for |u|^2 below 1e30: u^2 / (gamma + 1), which cancels nothing for
// slow particles.  The root and the quotient start from FP32 and take two corrections from exact
// residuals each (2^-22, 2^-46, 2^-70).
PIC_HD WideSum gamma_minus_one(float u0, float u1, float u2) {
    WideSum s;                                     // |u|^2
    float p, e, r, f, q, t, v, w;
    two_prod(u0, u0, s.h, s.m);
    two_prod(u1, u1, p, e);
    s.add(p, e, 0.f);
    two_prod(u2, u2, p, e);
    s.add(p, e, 0.f);
    s.normalise();
    WideSum g2 = s;                                // gamma^2
    g2.add(1.f);
    g2.normalise();
    // gamma = a + b + c: g2 - a^2 and then g2 - (a + b)^2, each sum ordered so that its large parts cancel
    const float a = sqrtf(g2.h), ra = 0.5f / a;
    two_prod(a, a, p, e);
    two_sum(g2.h - p, -e, r, f);                   // (the difference is exact)
    two_sum(r, g2.m, r, v);
    const float b = r * ra;
    two_prod(2.f * a, b, q, t);
    const float c = ((r - q) + ((f + v) + g2.l) - (t + b * b)) * ra;
    // d = gamma + 1 and s / d
    WideSum d{a, b, c};
    d.add(1.f);
    d.normalise();
    const float q0 = s.h / d.h;
    two_prod(q0, d.h, p, e);
    two_prod(q0, d.m, q, t);
    two_sum(s.h - p, s.m, r, f);                   // (s.h - q0 d.h is exact with e)
    two_sum(r, -e, r, v);
    two_sum(r, -q, r, w);
    const float rest = ((f + v) + w) + (s.l - t - q0 * d.l);
    const float q1 = r / d.h;
    const float q2 = (fmaf(-q1, d.h, r) + (rest - q1 * d.m)) / d.h;
    return WideSum{q0, q1, q2};
}

}  // namespace pic
