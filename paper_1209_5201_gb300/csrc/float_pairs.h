// Sums and products of FP32 values to about FP64 precision in FP32
// instructions (error-free transformations: Knuth's TwoSum, and a product with
// its FMA remainder), for device code, where an FP64 instruction takes a warp 64
// cycles, and for the host.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif

namespace lbm {

// Rounded operations that no compiler contracts or reorders (the host side is
// built without contraction).
LBM_HD float add32(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);
#else
    return a + b;
#endif
}
LBM_HD float sub32(float a, float b) { return add32(a, -b); }
LBM_HD float mul32(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}
LBM_HD float fma32(float a, float b, float c) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(a, b, c);
#else
    return std::fma(a, b, c);
#endif
}

LBM_HD void two_sum(float a, float b, float &s, float &e) {
    s = add32(a, b);
    const float bb = sub32(s, a);
    e = add32(sub32(a, sub32(s, bb)), sub32(b, bb));
}

struct Sum3 {                                // a running sum h + m + l
    float h = 0.0f, m = 0.0f, l = 0.0f;
    LBM_HD void add(float x) {
        float e, e2;
        two_sum(h, x, h, e);
        two_sum(m, e, m, e2);
        l = add32(l, e2);
    }
    LBM_HD void add(const float &xh, const float &xm, const float &xl) {   // another sum
        add(xh);
        add(xm);
        l = add32(l, xl);
    }
};

// c0 + d c with c0 = W c - w, both constants as three floats.
struct Emit3 { float c0h, c0m, c0l, ch, cm, cl; };

inline Emit3 emit3_of(double c, double W, double w) {
    Emit3 e;
    // W c - w as a sum of two doubles: the product and its remainder, TwoSum
    const double p = W * c, pe = std::fma(W, c, -p);
    const double s = p - w, b = s - p, se = (p - (s - b)) - (w + b);
    const double lo = se + pe;
    e.c0h = (float)s;
    e.c0m = (float)(s - (double)e.c0h);
    e.c0l = (float)((s - (double)e.c0h) - (double)e.c0m + lo);
    e.ch = (float)c;
    e.cm = (float)(c - (double)e.ch);
    e.cl = (float)((c - (double)e.ch) - (double)e.cm);
    return e;
}

// c0 + d c as hi + lo, lo the FP32 remainder of hi.  What is lost is below what
// FP64 loses on (W + d) c - w, whose cancellation against w this form avoids.
LBM_HD void emit3(const Emit3 &c, const Sum3 &d, float &hi, float &lo) {
    const float dh = add32(d.h, d.m), dl = add32(sub32(d.m, sub32(dh, d.h)), d.l);
    // dh ch = p + e, dh cm = q + qe, dl ch = g + ge
    const float p = mul32(dh, c.ch), e = fma32(dh, c.ch, -p);
    const float q = mul32(dh, c.cm), qe = fma32(dh, c.cm, -q);
    const float g = mul32(dl, c.ch), ge = fma32(dl, c.ch, -g);
    float v, r, t, te, u, ue, y, ye, z, ze;
    two_sum(c.c0h, p, v, r);                 // leading part, the rest 2^-24 of it
    two_sum(g, e, t, te);
    two_sum(q, t, u, ue);
    two_sum(c.c0m, u, y, ye);
    two_sum(r, y, z, ze);
    // ... and 2^-48 of it
    const float f = add32(add32(fma32(dh, c.cl, c.c0l), add32(qe, ge)), add32(add32(te, ue), add32(ye, ze)));
    hi = add32(v, z);
    lo = add32(sub32(z, sub32(hi, v)), f);
}

}  // namespace lbm
