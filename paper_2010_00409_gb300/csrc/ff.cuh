// Double-float arithmetic on the float32 pipe: a value is the unevaluated sum
// h + l of two float32 numbers (|l| <= ulp(h) / 2), about 48 significant bits.
// Products are exact through fmaf (two_prod), sums through the two-sum of Knuth
// (two_sum); no float64 instruction is issued.  GB300 runs float64 at 1/64 of
// the float32 rate, so the float32-storage kernels that need more than float32
// accuracy (the pulse geometry, the focal-plane sums) use these instead.
//
// The compiler keeps IEEE semantics here (no reassociation without fast-math;
// the only contractions are the explicit fmaf calls).
#pragma once

#include <cuda_runtime.h>

namespace psatd {

struct FF {
    float h, l;
};

__host__ __device__ __forceinline__ FF ff_from(double v) {
    FF f;
    f.h = (float)v;
    f.l = (float)(v - (double)f.h);
    return f;
}
__device__ __forceinline__ FF two_sum(float a, float b) {
    const float s = a + b, bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ FF quick_two_sum(float a, float b) {   // |a| >= |b|
    const float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ FF two_prod(float a, float b) {
    const float p = a * b;
    return {p, fmaf(a, b, -p)};
}
__device__ __forceinline__ FF ff_add(FF a, FF b) {
    const FF s = two_sum(a.h, b.h);
    return quick_two_sum(s.h, s.l + (a.l + b.l));
}
__device__ __forceinline__ FF ff_sub(FF a, FF b) { return ff_add(a, {-b.h, -b.l}); }
__device__ __forceinline__ FF ff_neg(FF a) { return {-a.h, -a.l}; }
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
    const FF p = two_prod(a.h, b.h);
    return quick_two_sum(p.h, fmaf(a.h, b.l, fmaf(a.l, b.h, p.l)));
}
__device__ __forceinline__ FF ff_mul_f(FF a, float b) {
    const FF p = two_prod(a.h, b);
    return quick_two_sum(p.h, fmaf(a.l, b, p.l));
}
__device__ __forceinline__ FF ff_sqr(FF a) {
    const FF p = two_prod(a.h, a.h);
    return quick_two_sum(p.h, fmaf(2.f * a.h, a.l, p.l));
}
__device__ __forceinline__ float ff_float(FF a) { return a.h + a.l; }

// complex double-float, stored as float4 {re.h, re.l, im.h, im.l}
struct CFF {
    FF re, im;
};
__device__ __forceinline__ CFF cff_load(const float4& v) { return {{v.x, v.y}, {v.z, v.w}}; }
__device__ __forceinline__ float4 cff_store(const CFF& c) { return make_float4(c.re.h, c.re.l, c.im.h, c.im.l); }
__host__ __device__ __forceinline__ float4 cff_from(double re, double im) {
    const FF r = ff_from(re), i = ff_from(im);
    return make_float4(r.h, r.l, i.h, i.l);
}
__device__ __forceinline__ CFF cff_add(const CFF& a, const CFF& b) { return {ff_add(a.re, b.re), ff_add(a.im, b.im)}; }

// Compensated dot products (Dot2 of Ogita, Rump and Oishi, "Accurate sum and dot
// product", 2005): the sum s takes every exact product by a two-sum, the rounding
// errors and the low-order product terms are summed in c, and s + c is the sum as
// if formed with twice the float32 precision.  One real term costs 11 (12 for a
// double-float v) float32 instructions; adding each product to a renormalised
// pair costs about 17.
struct Dot2 {
    float s, c;
};
struct Dot2C {
    Dot2 re, im;
};
// d += (wh + wl) v
__device__ __forceinline__ void dot2_term(Dot2& d, float wh, float wl, float v) {
    const FF p = two_prod(wh, v), t = two_sum(d.s, p.h);
    d.s = t.h;
    d.c += t.l + fmaf(wl, v, p.l);
}
// d += (wh + wl) (vh + vl)
__device__ __forceinline__ void dot2_term(Dot2& d, float wh, float wl, float vh, float vl) {
    const FF p = two_prod(wh, vh), t = two_sum(d.s, p.h);
    d.s = t.h;
    d.c += t.l + fmaf(wh, vl, fmaf(wl, vh, p.l));
}
// acc += w v, w a double-float complex value {re.h, re.l, im.h, im.l}
__device__ __forceinline__ void dot2_mac(Dot2C& acc, const float4& w, float2 v) {
    dot2_term(acc.re, w.x, w.y, v.x);
    dot2_term(acc.re, -w.z, -w.w, v.y);
    dot2_term(acc.im, w.x, w.y, v.y);
    dot2_term(acc.im, w.z, w.w, v.x);
}
__device__ __forceinline__ void dot2_mac_real(Dot2C& acc, const float4& w, float v) {
    dot2_term(acc.re, w.x, w.y, v);
    dot2_term(acc.im, w.z, w.w, v);
}
__device__ __forceinline__ void dot2_mac_cff(Dot2C& acc, const float4& w, const float4& v) {
    dot2_term(acc.re, w.x, w.y, v.x, v.y);
    dot2_term(acc.re, -w.z, -w.w, v.z, v.w);
    dot2_term(acc.im, w.x, w.y, v.z, v.w);
    dot2_term(acc.im, w.z, w.w, v.x, v.y);
}
__device__ __forceinline__ CFF dot2_value(const Dot2C& a) {
    return {two_sum(a.re.s, a.re.c), two_sum(a.im.s, a.im.c)};
}

}  // namespace psatd
