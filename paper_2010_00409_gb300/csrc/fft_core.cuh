// Device FFT building blocks: radix-2/3/4/5/8 butterflies.
//
// Sign convention: S = -1 is the forward transform (kernel exp(-2 pi i nk/N)),
// S = +1 the inverse; neither is normalised.
#pragma once

#include "common.cuh"

namespace psatd {

// Complex sum and difference of butterfly operands.  float32 pairs on the GPU
// use the packed two-lane adds of sm_100-class SMs (add/sub.rn.f32x2: one
// instruction per complex add, the same round-to-nearest result as two scalar
// adds); double pairs and host code use cadd / csub.
template <typename V> __host__ __device__ __forceinline__ V badd(V a, V b) { return cadd(a, b); }
template <typename V> __host__ __device__ __forceinline__ V bsub(V a, V b) { return csub(a, b); }
__host__ __device__ __forceinline__ float2 badd(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    float2 r;
    asm("{.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\t"
        "mov.b64 rb, {%4, %5};\n\t"
        "add.rn.f32x2 rd, ra, rb;\n\t"
        "mov.b64 {%0, %1}, rd;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
#else
    return cadd(a, b);
#endif
}
__host__ __device__ __forceinline__ float2 bsub(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    float2 r;
    asm("{.reg .b64 ra, rb, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\t"
        "mov.b64 rb, {%4, %5};\n\t"
        "sub.rn.f32x2 rd, ra, rb;\n\t"
        "mov.b64 {%0, %1}, rd;}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
#else
    return csub(a, b);
#endif
}

// t + S i u and t - S i u in scalar form: the lane swap of i u does not pack.
template <typename V, int S>
__host__ __device__ __forceinline__ void add_sub_si(const V& t, const V& u, V& plus, V& minus) {
    if constexpr (S > 0) {
        plus.x = t.x - u.y; plus.y = t.y + u.x;
        minus.x = t.x + u.y; minus.y = t.y - u.x;
    } else {
        plus.x = t.x + u.y; plus.y = t.y - u.x;
        minus.x = t.x - u.y; minus.y = t.y + u.x;
    }
}

template <typename V, int S>
__host__ __device__ __forceinline__ void bfly2(V& a0, V& a1) {
    V t = a0; a0 = badd(t, a1); a1 = bsub(t, a1);
}

template <typename V, int S>
__host__ __device__ __forceinline__ void bfly4(V& a0, V& a1, V& a2, V& a3) {
    V t0 = badd(a0, a2), t1 = bsub(a0, a2), t2 = badd(a1, a3), u = bsub(a1, a3);
    a0 = badd(t0, t2); a2 = bsub(t0, t2);
    add_sub_si<V, S>(t1, u, a1, a3);                 // t1 +- S i (a1 - a3)
}

// x / sqrt 2.  In float32 the rounded 1/sqrt 2 makes |(1 + i)/sqrt 2|^2 =
// 1 - 3.4e-8, an energy loss that every 45-degree rotation of every transform
// would repeat each step; the product is therefore formed with the rounding
// residue of 1/sqrt 2 added in (one more multiply), which leaves only the
// unbiased rounding of the result.
template <typename T> __host__ __device__ __forceinline__ T mul_rsqrt2(T x) {
    if constexpr (sizeof(T) == 4) {
        constexpr float hi = (float)0.70710678118654752440;
        constexpr float lo = (float)(0.70710678118654752440 - (double)hi);
        return fmaf(x, hi, x * lo);
    } else {
        return x * (T)0.70710678118654752440;
    }
}

template <typename T, int S>
__host__ __device__ __forceinline__ void bfly8(cplx<T>* v) {
    // even / odd 4-point DFTs, then combine with exp(S 2 pi i k / 8)
    bfly4<cplx<T>, S>(v[0], v[2], v[4], v[6]);
    bfly4<cplx<T>, S>(v[1], v[3], v[5], v[7]);
    cplx<T> o1 = v[3], o2 = v[5], o3 = v[7];
    // W^1 = (1 + S i)/sqrt2
    cplx<T> w1 = mk<T>(mul_rsqrt2<T>(o1.x - S * o1.y), mul_rsqrt2<T>(o1.y + S * o1.x));
    // W^3 = (-1 + S i)/sqrt2
    cplx<T> w3 = mk<T>(-mul_rsqrt2<T>(o3.x + S * o3.y), mul_rsqrt2<T>(S * o3.x - o3.y));
    cplx<T> e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
    v[0] = badd(e0, o0); v[4] = bsub(e0, o0);
    v[1] = badd(e1, w1); v[5] = bsub(e1, w1);
    add_sub_si<cplx<T>, S>(e2, o2, v[2], v[6]);     // W^2 = S i
    v[3] = badd(e3, w3); v[7] = bsub(e3, w3);
}

// x * C for a constant C.  In float32 the rounding residue of C is added by one more
// multiply (as in mul_rsqrt2), so the constant's rounding does not scale the
// field's energy by the same factor every step.
template <typename T> __host__ __device__ __forceinline__ T mul_const(T x, double C) {
    if constexpr (sizeof(T) == 4) {
        const float hi = (float)C, lo = (float)(C - (double)hi);
        return fmaf(x, hi, x * lo);
    } else {
        return x * (T)C;
    }
}

template <typename T, int S>
__host__ __device__ __forceinline__ void bfly3(cplx<T>& a0, cplx<T>& a1, cplx<T>& a2) {
    constexpr double h = 0.86602540378443864676;   // sin(2 pi / 3)
    cplx<T> t = badd(a1, a2), u = bsub(a1, a2);
    cplx<T> m = mk<T>(a0.x - (T)0.5 * t.x, a0.y - (T)0.5 * t.y);
    u = mk<T>(mul_const<T>(u.x, h), mul_const<T>(u.y, h));
    a0 = badd(a0, t);
    add_sub_si<cplx<T>, S>(m, u, a1, a2);
}

// x * A + y * B for constants A, B, with their rounding residues in float32
template <typename T> __host__ __device__ __forceinline__ T dot_const(T x, double A, T y, double B) {
    if constexpr (sizeof(T) == 4) {
        const float ah = (float)A, al = (float)(A - (double)ah), bh = (float)B, bl = (float)(B - (double)bh);
        return fmaf(x, ah, fmaf(y, bh, fmaf(x, al, y * bl)));
    } else {
        return x * (T)A + y * (T)B;
    }
}

// 5-point DFT: the even part as a0 - t/4 +- (sqrt 5 / 4)(t1 - t2), t = t1 + t2 (one
// constant instead of cos(2 pi / 5) and cos(4 pi / 5)).
template <typename T, int S>
__host__ __device__ __forceinline__ void bfly5(cplx<T>* a) {
    constexpr double q5 = 0.55901699437494742410;   // sqrt(5) / 4
    constexpr double s1 = 0.95105651629515357212;    // sin(2 pi / 5)
    constexpr double s2 = 0.58778525229247312917;    // sin(4 pi / 5)
    cplx<T> t1 = badd(a[1], a[4]), t2 = badd(a[2], a[3]);
    cplx<T> u1 = bsub(a[1], a[4]), u2 = bsub(a[2], a[3]);
    cplx<T> t = badd(t1, t2), d = bsub(t1, t2);
    cplx<T> m = mk<T>(a[0].x - (T)0.25 * t.x, a[0].y - (T)0.25 * t.y);
    cplx<T> e = mk<T>(mul_const<T>(d.x, q5), mul_const<T>(d.y, q5));
    cplx<T> p1 = badd(m, e), p2 = bsub(m, e);
    cplx<T> q1 = mk<T>(dot_const<T>(u1.x, s1, u2.x, s2), dot_const<T>(u1.y, s1, u2.y, s2));
    cplx<T> q2 = mk<T>(dot_const<T>(u1.x, s2, u2.x, -s1), dot_const<T>(u1.y, s2, u2.y, -s1));
    a[0] = badd(a[0], t);
    add_sub_si<cplx<T>, S>(p1, q1, a[1], a[4]);
    add_sub_si<cplx<T>, S>(p2, q2, a[2], a[3]);
}

template <typename T, int R, int S>
__host__ __device__ __forceinline__ void dft_r(cplx<T>* v) {
    if constexpr (R == 2) bfly2<cplx<T>, S>(v[0], v[1]);
    else if constexpr (R == 3) bfly3<T, S>(v[0], v[1], v[2]);
    else if constexpr (R == 4) bfly4<cplx<T>, S>(v[0], v[1], v[2], v[3]);
    else if constexpr (R == 5) bfly5<T, S>(v);
    else if constexpr (R == 8) bfly8<T, S>(v);
}

}  // namespace psatd
