// One value (float) or the values of two lattice points (float2) in the same
// code: every helper is one operation with one rounding, on float2 one packed
// FP32x2 instruction whose halves round as the scalar one, so that code
// written with them gives a point the same bits alone and in a pair.  One
// thing to keep to: the compiler may fuse a packed product that is used once
// into a packed sum that takes it (the scalar intrinsics stay apart), so
// every product that goes into a sum here is written as a vfma, and 2 x as
// vtwice.  Also the real roots of the monic cubics and quartics that the moment bounds
// meet, whose roots are all real.
#pragma once
#include "mboit_device.cuh"

namespace mb {

template <class T> struct Vec;
template <> struct Vec<float> {
#if defined(__CUDACC__)
    static __host__ __device__ __forceinline__ float splat(float a) { return a; }
#else
    static inline float splat(float a) { return a; }
#endif
};
MB_HD float vadd(float a, float b) { return fadd(a, b); }
MB_HD float vsub(float a, float b) { return fadd(a, -b); }
MB_HD float vmul(float a, float b) { return fmul(a, b); }
MB_HD float vfma(float a, float b, float c) { return ffma(a, b, c); }
MB_HD float vneg(float a) { return -a; }
MB_HD float vtwice(float a) { return fmul(a, 2.0f); }
MB_HD float vmax(float a, float b) { return fmax_(a, b); }
MB_HD float vmin(float a, float b) { return fmin_(a, b); }
MB_HD float vrcp(float a) { return frcp(a); }
MB_HD float vsqrt(float a) { return fsqrt_fast(a); }
MB_HD float vnonzero(float a, float b) { return a != 0.0f ? b : 0.0f; }     // b where a is not 0, else 0

#if defined(__CUDACC__)
template <> struct Vec<float2> {
    static __device__ __forceinline__ float2 splat(float a) { return make_float2(a, a); }
};
#define MB_V2 __device__ __forceinline__ float2
MB_V2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
MB_V2 vsub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
MB_V2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
MB_V2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
MB_V2 vneg(float2 a) { return make_float2(-a.x, -a.y); }
MB_V2 vtwice(float2 a) { return __fmul2_rn(a, make_float2(2.0f, 2.0f)); }
MB_V2 vmax(float2 a, float2 b) { return make_float2(fmax_(a.x, b.x), fmax_(a.y, b.y)); }
MB_V2 vmin(float2 a, float2 b) { return make_float2(fmin_(a.x, b.x), fmin_(a.y, b.y)); }
MB_V2 vrcp(float2 a) { return make_float2(frcp(a.x), frcp(a.y)); }
MB_V2 vsqrt(float2 a) { return make_float2(fsqrt_fast(a.x), fsqrt_fast(a.y)); }
MB_V2 vnonzero(float2 a, float2 b) { return make_float2(vnonzero(a.x, b.x), vnonzero(a.y, b.y)); }
#undef MB_V2
#endif

// Per-point truth values and counts that go with T.
template <class T> struct Lanes;
template <> struct Lanes<float> {
    int a;
};
#if defined(__CUDACC__)
template <> struct Lanes<float2> {
    int a, b;
};
#endif
MB_HD Lanes<float> below(float x, float y) { return {x < y ? 1 : 0}; }
MB_HD Lanes<float> operator+(Lanes<float> p, Lanes<float> q) { return {p.a + q.a}; }
MB_HD float pick_eq(Lanes<float> n, int v, float x, float y) { return n.a == v ? x : y; }
MB_HD float pick_gt(Lanes<float> n, int v, float x, float y) { return n.a > v ? x : y; }
MB_HD bool any_eq(Lanes<float> n, int v) { return n.a == v; }
#if defined(__CUDACC__)
#define MB_L2 __device__ __forceinline__
MB_L2 Lanes<float2> below(float2 x, float2 y) { return {x.x < y.x ? 1 : 0, x.y < y.y ? 1 : 0}; }
MB_L2 Lanes<float2> operator+(Lanes<float2> p, Lanes<float2> q) { return {p.a + q.a, p.b + q.b}; }
MB_L2 float2 pick_eq(Lanes<float2> n, int v, float2 x, float2 y) {
    return make_float2(n.a == v ? x.x : y.x, n.b == v ? x.y : y.y);
}
MB_L2 float2 pick_gt(Lanes<float2> n, int v, float2 x, float2 y) {
    return make_float2(n.a > v ? x.x : y.x, n.b > v ? x.y : y.y);
}
MB_L2 bool any_eq(Lanes<float2> n, int v) { return n.a == v || n.b == v; }
#undef MB_L2
#endif

// cos(acos(u) / 3) for u in [-1, 1].  With v = cos(acos(u) / 2) = sqrt((1 + u) /
// 2) it is cos(2/3 acos v), analytic on [0, 1] (also at v = 1, where the
// cosine is even in acos v): the polynomial of degree 7 through its values at
// the eight Chebyshev points of [0, 1], within 2.6e-8 of it (1.2e-7 evaluated
// in float32).  acos and cos themselves cost about three times as much.
template <class T>
MB_HD T cos_third(T u) {
    const T h = Vec<T>::splat(0.5f);
    const T v = vsqrt(vfma(h, u, h));
    T p = Vec<T>::splat(0.00112763629f);
    p = vfma(p, v, Vec<T>::splat(-0.00608934555f));
    p = vfma(p, v, Vec<T>::splat(0.0160472803f));
    p = vfma(p, v, Vec<T>::splat(-0.0302353967f));
    p = vfma(p, v, Vec<T>::splat(0.05284141f));
    p = vfma(p, v, Vec<T>::splat(-0.111038513f));
    p = vfma(p, v, Vec<T>::splat(0.577346921f));
    return vfma(p, v, Vec<T>::splat(0.5f));
}

// One Newton step of the monic cubic s^3 + a s^2 + b s + c at s (none where the
// derivative is 0).
template <class T>
MB_HD T newton3(T a, T b, T c, T s) {
    const T f = vfma(vfma(vadd(s, a), s, b), s, c);
    const T df = vfma(vfma(Vec<T>::splat(3.0f), s, vtwice(a)), s, b);
    return vsub(s, vnonzero(df, vmul(f, vrcp(df))));
}

// Viete's form of a cubic whose roots are all real: the amplitude m, the
// centre a / 3 and the largest cosine.
template <class T>
MB_HD void viete(T a, T b, T c, T& a3, T& m, T& cs) {
    a3 = vmul(a, Vec<T>::splat(1.0f / 3.0f));
    const T p = vfma(vneg(a), a3, b);
    const T q = vfma(vfma(vtwice(a3), a3, vneg(b)), a3, c);   // 2 a3^3 - b a3 + c
    const T pm = vmin(p, Vec<T>::splat(-1e-30f));
    const T h = vsqrt(vmul(pm, Vec<T>::splat(-1.0f / 3.0f)));
    m = vtwice(h);
    const T arg = vmul(vmul(Vec<T>::splat(3.0f), q), vrcp(vmul(pm, m)));
    cs = cos_third(vmax(vmin(arg, Vec<T>::splat(1.0f)), Vec<T>::splat(-1.0f)));
}

// The roots in ascending order: Viete's three cosines (those of th - 2 pi / 3 and
// th + 2 pi / 3 from the cosine and sine of th in [0, pi / 3]), one Newton step
// each.
template <class T>
MB_HD void cubic3(T a, T b, T c, T r[3]) {
    T a3, m, cs;
    viete(a, b, c, a3, m, cs);
    const T sn = vsqrt(vfma(vneg(cs), cs, Vec<T>::splat(1.0f)));
    const T h = vmul(cs, Vec<T>::splat(-0.5f));
    const T k = Vec<T>::splat(0.8660254037844386f);
    const T na3 = vneg(a3);
    r[2] = vfma(m, cs, na3);
    r[1] = vfma(m, vfma(k, sn, h), na3);
    r[0] = vfma(m, vfma(vneg(k), sn, h), na3);
#pragma unroll
    for (int i = 0; i < 3; ++i) r[i] = newton3(a, b, c, r[i]);
}

// Real roots of the monic quartic s^4 + a s^3 + b s^2 + c s + d whose roots are all
// real, ascending: Ferrari's two quadratics from the resolvent cubic's largest
// root, which pairs the two largest roots and the two smallest, then one
// Newton step each.
template <class T>
MB_HD void quartic4(T a, T b, T c, T d, T r[4]) {
    const T a4 = vmul(Vec<T>::splat(0.25f), a);
    const T a42 = vmul(a4, a4);
    const T p = vfma(Vec<T>::splat(-6.0f), a42, b);
    const T q = vfma(vfma(Vec<T>::splat(8.0f), a42, vmul(Vec<T>::splat(-2.0f), b)), a4, c);   // c - 2 b a4 + 8 a4^3
    const T w = vfma(vfma(vfma(Vec<T>::splat(-3.0f), a42, b), a4, vneg(c)), a4, d);          // d - c a4 + b a4^2 - 3 a4^4
    // m^3 + p m^2 + (p^2 / 4 - w) m - q^2 / 8 = 0, the largest root (positive)
    const T rb = vfma(vmul(Vec<T>::splat(0.25f), p), p, vneg(w)), rc = vmul(vmul(Vec<T>::splat(-0.125f), q), q);
    T a3, am, cs;
    viete(p, rb, rc, a3, am, cs);
    const T m = vmax(newton3(p, rb, rc, vfma(am, cs, vneg(a3))), Vec<T>::splat(1e-30f));
    const T m2 = vtwice(m);
    const T sq = vsqrt(m2);
    const T h = vfma(Vec<T>::splat(0.5f), p, m), g = vmul(q, vrcp(vtwice(sq)));
    // y^2 - sq y + (h + g) = 0 and y^2 + sq y + (h - g) = 0
    const T zero = Vec<T>::splat(0.0f), half = Vec<T>::splat(0.5f), four = Vec<T>::splat(-4.0f);
    const T d1 = vsqrt(vmax(vfma(four, vadd(h, g), m2), zero));
    const T d2 = vsqrt(vmax(vfma(four, vsub(h, g), m2), zero));
    r[0] = vmul(half, vneg(vadd(sq, d2)));
    r[1] = vmul(half, vsub(d2, sq));
    r[2] = vmul(half, vsub(sq, d1));
    r[3] = vmul(half, vadd(sq, d1));
    const T b2 = vtwice(b), a3x = vmul(Vec<T>::splat(3.0f), a);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const T s = vsub(r[i], a4);
        const T f = vfma(vfma(vfma(vadd(s, a), s, b), s, c), s, d);
        const T df = vfma(vfma(vfma(Vec<T>::splat(4.0f), s, a3x), s, b2), s, c);
        r[i] = vsub(s, vnonzero(df, vmul(f, vrcp(df))));
    }
}

}  // namespace mb
