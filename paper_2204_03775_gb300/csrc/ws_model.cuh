// The stored model (V dt / h)^2 from a velocity or a squared slowness.
#pragma once

#include "ws_internal.h"

namespace ws {

// (V dt / h)^2 from V, and (dt / h)^2 / m from m = 1/V^2, each the double
// result rounded to float. GB300 runs FP64 at a small fraction of FP32, so
// the value is formed as a sum q + q2 of two floats (error below 2^-44 of it:
// the scale as two floats, products and remainders exact through fma), whose
// nearest float is that of the double result unless both lie within 2^-42 of
// a tie between two floats; then, and outside the range in which no term
// underflows, the double expression itself is evaluated (about one cell in
// 2^18). The stored floats are the same bits either way.
struct ModelScale {
    double c;       // dt / h, or (dt / h)^2
    float hi, lo;   // c as two floats
    bool fast;      // hi in [2^-60, 2^60]
};

inline ModelScale model_scale(double c) {
    ModelScale s{c, (float)c, 0.0f, false};
    s.lo = (float)(c - (double)s.hi);
    s.fast = s.hi >= 0x1p-60f && s.hi <= 0x1p60f;
    return s;
}

// The nearest float of q + q2 if the sum moved by +-2^-42 q rounds alike.
static __device__ __forceinline__ bool round_sum(float q, float q2, float *w) {
    const float a = q + fmaf(q, 0x1p-42f, q2), b = q + fmaf(q, -0x1p-42f, q2);
    *w = a;
    return a == b && q >= 0x1p-60f && q <= 0x1p60f;
}

struct FromVelocity {
    // (a call: inlined, its two products were issued for every cell)
    static __device__ __noinline__ float slow(float v, double c) {
        const double r = __dmul_rn((double)v, c);   // as ws_energy_noalloc forms it
        return (float)__dmul_rn(r, r);
    }
    static __device__ __forceinline__ bool fast(float v, const ModelScale &k, float *w) {
        const float p = __fmul_rn(v, k.hi);
        const float l = fmaf(v, k.lo, fmaf(v, k.hi, -p));
        const float s = __fadd_rn(p, l), t = __fsub_rn(l, __fsub_rn(s, p));   // V dt / h = s + t
        const float q = __fmul_rn(s, s);
        return round_sum(q, fmaf(2.0f * s, t, fmaf(s, s, -q)), w) && k.fast;
    }
};

struct FromSlowness2 {
    static __device__ __noinline__ float slow(float m, double c) {
        return (float)(c / (double)m);
    }
    static __device__ __forceinline__ bool fast(float m, const ModelScale &k, float *w) {
        const float q = __fdiv_rn(k.hi, m);
        const float r = __fadd_rn(fmaf(-q, m, k.hi), k.lo);   // c - q m
        return round_sum(q, __fdividef(r, m), w) && k.fast && m >= 0x1p-100f && m <= 0x1p100f;
    }
};

template <class Conv>
__device__ __forceinline__ float to_model(float x, const ModelScale &k) {
    float w;
    return Conv::fast(x, k, &w) ? w : Conv::slow(x, k.c);
}

}  // namespace ws
