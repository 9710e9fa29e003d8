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

// Compensated dot products (after Dot2 of Ogita, Rump and Oishi, "Accurate sum and
// dot product", 2005): the sum s takes the exact products by two-sums, the rounding
// errors and the low-order product terms go to c, and s + c is the sum as if formed
// with twice the float32 precision.  The two real products of a part are added to each
// other first, and the callers renormalise the pair (dot2_norm) after every second
// complex product: c is plain float32, so if it grew over a long sum its own roundings
// would count (an error in proportion to the square of the length).  A part of a complex
// product costs 23.5 (25.5 for a double-float v) float32 instructions with that;
// products and sums each rounded to a renormalised pair, about 36.  (Renormalised after
// each product, with its chain of ten dependent additions, a plane of 64 x 64 points on
// 128^3 took 22 % longer.)
// Error of y or z sums of n products of one sign against 64 bits, rms over the sum of
// the magnitudes, with every product and sum renormalised and with these (four chains):
// n = 64 5.4e-15 and 1.9e-15, n = 256 10.7e-15 and 3.2e-15, n = 512 15.4e-15 and
// 4.4e-15.
struct Dot2 {
    float s, c;
};
struct Dot2C {
    Dot2 re, im;
};
// (wh + wl) v: the leading product and everything below it
__device__ __forceinline__ FF dot2_prod(float wh, float wl, float v) {
    const FF p = two_prod(wh, v);
    return {p.h, fmaf(wl, v, p.l)};
}
// (wh + wl) (vh + vl)
__device__ __forceinline__ FF dot2_prod(float wh, float wl, float vh, float vl) {
    const FF p = two_prod(wh, vh);
    return {p.h, fmaf(wh, vl, fmaf(wl, vh, p.l))};
}
// d += p + q
__device__ __forceinline__ void dot2_add(Dot2& d, const FF& p, const FF& q) {
    const FF h = two_sum(p.h, q.h), t = two_sum(d.s, h.h);
    d.s = t.h;
    d.c += t.l + (h.l + (p.l + q.l));
}
__device__ __forceinline__ void dot2_norm(Dot2C& d) {
    const FF re = quick_two_sum(d.re.s, d.re.c), im = quick_two_sum(d.im.s, d.im.c);
    d = {{re.h, re.l}, {im.h, im.l}};
}
// acc += w v, w a double-float complex value {re.h, re.l, im.h, im.l}
__device__ __forceinline__ void dot2_mac(Dot2C& acc, const float4& w, float2 v) {
    dot2_add(acc.re, dot2_prod(w.x, w.y, v.x), dot2_prod(-w.z, -w.w, v.y));
    dot2_add(acc.im, dot2_prod(w.x, w.y, v.y), dot2_prod(w.z, w.w, v.x));
}
// acc += w0 v.x + w1 v.y for two real values
__device__ __forceinline__ void dot2_mac_real(Dot2C& acc, const float4& w0, const float4& w1, float2 v) {
    dot2_add(acc.re, dot2_prod(w0.x, w0.y, v.x), dot2_prod(w1.x, w1.y, v.y));
    dot2_add(acc.im, dot2_prod(w0.z, w0.w, v.x), dot2_prod(w1.z, w1.w, v.y));
}
__device__ __forceinline__ void dot2_mac_cff(Dot2C& acc, const float4& w, const float4& v) {
    dot2_add(acc.re, dot2_prod(w.x, w.y, v.x, v.y), dot2_prod(-w.z, -w.w, v.z, v.w));
    dot2_add(acc.im, dot2_prod(w.x, w.y, v.z, v.w), dot2_prod(w.z, w.w, v.x, v.y));
}
__device__ __forceinline__ CFF dot2_value(const Dot2C& a) {
    return {quick_two_sum(a.re.s, a.re.c), quick_two_sum(a.im.s, a.im.c)};
}

}  // namespace psatd
