// drt_ff.cuh -- "two-float" numbers: a value held as the unevaluated sum h + l of two FP32 numbers, |l| <= ulp(h) / 2,
// about 47 bits.  FP64 runs at 1/64 of the FP32 rate on GB300 (65 cycles per warp instruction and sub-partition, measured);
// an addition here is 11 and a product 7 FP32 instructions, so work whose result is FP32 (the synthesis records of H) gains
// 4 to 8 times by it and keeps its FP64-like error: relative 2^-46 per operation, 1e-12 m on a 100 m path, 1e-9 rad at 60 GHz.
//
// The error-free transformations are Knuth's two-sum and Dekker's fast two-sum and the FMA product (T. J. Dekker, "A
// floating-point technique for extending the available precision", Numer. Math. 18, 1971; Knuth, TAOCP 2, 4.2.2); the dot product
// accumulates its errors in a second sum (Ogita, Rump, Oishi, "Accurate sum and dot product", 2005).  They need every rounding
// as written: all FP32 operations go through the _rn intrinsics, which the compiler neither contracts nor reorders.
#pragma once
#include "drt_math.cuh"
#include "drt_fftrig.h"

namespace drt {

struct alignas(8) ff {
    float h, l;
    ff() = default;
    DRT_HD constexpr ff(float hh, float ll) : h(hh), l(ll) {}
    DRT_HD constexpr ff(double d) : h((float)d), l((float)(d - (double)(float)d)) {}   // compile-time constants
    DRT_HD constexpr ff(float f) : h(f), l(0.f) {}
    DRT_HD constexpr ff(int i) : h((float)i), l(0.f) {}                               // |i| < 2^24
};
// a double split on the host (infinite values keep l = 0)
inline ff ff_host(double d) {
    const float h = (float)d;
    return ff(h, h - h == 0.f ? (float)(d - (double)h) : 0.f);
}

#define FF_D DRT_HD
#ifdef __CUDA_ARCH__
FF_D float fadd(float a, float b) { return __fadd_rn(a, b); }
FF_D float fmul(float a, float b) { return __fmul_rn(a, b); }
FF_D float ffma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
FF_D float frcp(float a) { return __fdividef(1.f, a); }
#else   // compiled, never called
FF_D float fadd(float a, float b) { return a + b; }
FF_D float fmul(float a, float b) { return a * b; }
FF_D float ffma(float a, float b, float c) { return fmaf(a, b, c); }
FF_D float frcp(float a) { return 1.f / a; }
#endif
FF_D float fsub(float a, float b) { return fadd(a, -b); }
FF_D ff quick(float a, float b) {   // |a| >= |b|
    const float s = fadd(a, b);
    return ff(s, fsub(b, fsub(s, a)));
}
FF_D void two_sum(float a, float b, float &s, float &e) {
    s = fadd(a, b);
    const float bb = fsub(s, a);
    e = fadd(fsub(a, fsub(s, bb)), fsub(b, bb));
}
FF_D ff operator-(ff a) { return ff(-a.h, -a.l); }
FF_D ff operator+(ff a, ff b) {
    float s, e;
    two_sum(a.h, b.h, s, e);
    return quick(s, fadd(e, fadd(a.l, b.l)));
}
FF_D ff operator-(ff a, ff b) { return a + (-b); }
FF_D ff operator*(ff a, ff b) {
    const float p = fmul(a.h, b.h);
    return quick(p, ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p))));
}
FF_D ff operator*(ff a, float b) {
    const float p = fmul(a.h, b);
    return quick(p, ffma(a.l, b, ffma(a.h, b, -p)));
}
FF_D ff fma(ff a, ff b, ff c) {
    const float p = fmul(a.h, b.h), pe = ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p)));
    float s, e;
    two_sum(p, c.h, s, e);
    return quick(s, fadd(e, fadd(pe, c.l)));
}
FF_D ff &operator+=(ff &a, ff b) { return a = a + b; }
FF_D ff &operator*=(ff &a, ff b) { return a = a * b; }
FF_D ff halve(ff a) { return ff(0.5f * a.h, 0.5f * a.l); }
FF_D ff twice(ff a) { return ff(2.f * a.h, 2.f * a.l); }
// quotient: FP32 quotient and the exact remainder's
FF_D ff operator/(ff a, ff b) {
    const float y = frcp(b.h), q = fmul(a.h, y);
    const float p = fmul(q, b.h);
    const float r = ffma(-q, b.l, fadd(fsub(fsub(a.h, p), ffma(q, b.h, -p)), a.l));
    return quick(q, fmul(r, y));
}
// x^(-1/2): the hardware's estimate y and one third-order step in r = 1 - x y^2 (0 gives a NaN)
FF_D ff rsqrt(ff a) {
    const float y = rsqrtf(a.h);
    const float p = fmul(y, y), e = ffma(y, y, -p);
    const float q = fmul(a.h, p), qe = ffma(a.h, p, -q);
    const float r = fsub(fsub(fsub(1.f, q), qe), ffma(a.h, e, fmul(a.l, p)));
    return quick(y, fmul(fmul(y, r), ffma(0.375f, r, 0.5f)));
}
FF_D ff sqrt(ff a) {   // 0 gives a NaN
    const float y = rsqrtf(a.h), s = fmul(a.h, y), p = fmul(s, s);
    const float d = fadd(fsub(fsub(a.h, p), ffma(s, s, -p)), a.l);
    return quick(s, fmul(d, 0.5f * y));
}
FF_D ff fabs(ff a) { return a.h < 0.f ? -a : a; }
FF_D bool operator<(ff a, ff b) { return a.h < b.h || (a.h == b.h && a.l < b.l); }
FF_D bool operator>(ff a, ff b) { return b < a; }
FF_D bool operator<=(ff a, ff b) { return a.h < b.h || (a.h == b.h && a.l <= b.l); }
FF_D bool operator>=(ff a, ff b) { return a.h > b.h || (a.h == b.h && a.l >= b.l); }
FF_D bool operator==(ff a, ff b) { return a.h == b.h && a.l == b.l; }
FF_D ff fmax(ff a, ff b) { return a < b ? b : a; }
FF_D ff copysign(ff a, ff b) { return (a.h < 0.f) == (b.h < 0.f) ? a : -a; }
FF_D ff ldexp(ff a, int e) { return ff(::ldexpf(a.h, e), ::ldexpf(a.l, e)); }
FF_D double to_double(ff a) { return (double)a.h + (double)a.l; }
FF_D ff from_double(double d) {
    const float h = (float)d;
    return ff(h, (float)(d - (double)h));
}

using ::copysign;
using ::fabs;
using ::fma;
using ::fmax;
using ::ldexp;
using ::rsqrt;
using ::sqrt;

template <> struct ST<ff> {   // values only, as for double
    typedef ff R;
    static DRT_HD ff val(ff x) { return x; }
    static DRT_HD ff rate(ff) { return ff(0.f, 0.f); }
    static DRT_HD ff cst(ff x) { return x; }
};

FF_D ff dsqrt(ff x) { return sqrt(x); }
// three products with one renormalisation: 31 instructions instead of 43
FF_D ff dot(v3<ff> a, v3<ff> b) {
    const float p0 = fmul(a.x.h, b.x.h), p1 = fmul(a.y.h, b.y.h), p2 = fmul(a.z.h, b.z.h);
    float e0 = ffma(a.x.h, b.x.h, -p0), e1 = ffma(a.y.h, b.y.h, -p1), e2 = ffma(a.z.h, b.z.h, -p2);
    e0 = ffma(a.x.l, b.x.h, ffma(a.x.h, b.x.l, e0));
    e1 = ffma(a.y.l, b.y.h, ffma(a.y.h, b.y.l, e1));
    e2 = ffma(a.z.l, b.z.h, ffma(a.z.h, b.z.l, e2));
    float s, t, u, v;
    two_sum(p0, p1, s, t);
    two_sum(s, p2, u, v);
    return quick(u, fadd(fadd(t, v), fadd(fadd(e0, e1), e2)));
}
// a b - c d
FF_D ff det2(ff a, ff b, ff c, ff d) {
    const float p = fmul(a.h, b.h), q = fmul(c.h, d.h);
    const float e = ffma(a.l, b.h, ffma(a.h, b.l, ffma(a.h, b.h, -p)));
    const float f = ffma(c.l, d.h, ffma(c.h, d.l, ffma(c.h, d.h, -q)));
    float s, t;
    two_sum(p, -q, s, t);
    return quick(s, fadd(t, fsub(e, f)));
}
// X + n s
FF_D v3<ff> axpy(v3<ff> X, v3<ff> n, ff s) { return {fma(n.x, s, X.x), fma(n.y, s, X.y), fma(n.z, s, X.z)}; }
FF_D v3<ff> cross(v3<ff> a, v3<ff> b) {
    return {det2(a.y, b.z, a.z, b.y), det2(a.z, b.x, a.x, b.z), det2(a.x, b.y, a.y, b.x)};
}
FF_D ff norm(v3<ff> a) { return sqrt(dot(a, a)); }
FF_D v3<ff> unit(v3<ff> a) { return a * rsqrt(dot(a, a)); }
FF_D cx<ff> cdot(c3<ff> E, v3<ff> e) {
    return {dot(V3<ff>(E.x.re, E.y.re, E.z.re), e), dot(V3<ff>(E.x.im, E.y.im, E.z.im), e)};
}
// a s + b t
FF_D cx<ff> mix(ff a, cx<ff> s, ff b, cx<ff> t) { return {det2(a, s.re, -b, t.re), det2(a, s.im, -b, t.im)}; }
FF_D c3<ff> mix(v3<ff> a, cx<ff> s, v3<ff> b, cx<ff> t) {
    return {mix(a.x, s, b.x, t), mix(a.y, s, b.y, t), mix(a.z, s, b.z, t)};
}
FF_D ff cabs2(cx<ff> a) { return det2(a.re, a.re, -a.im, a.im); }
FF_D cx<ff> operator*(cx<ff> a, cx<ff> b) {
    return {det2(a.re, b.re, a.im, b.im), det2(a.re, b.im, -a.im, b.re)};
}

// sine and cosine of x (|x| < 6.4; beyond, or not a number: no angle's, but no read past the table): the nearest multiple
// of 1/32 from a table, the remainder |d| <= 1/64 by its Taylor terms (what is below 2^-24 of the result in FP32), joined
// by angle addition
struct FFSinCos { ff s, c; };
inline __host__ __device__ __noinline__ FFSinCos sincos_ff(ff x) {
    const float i = rintf(32.f * x.h);
#ifdef __CUDA_ARCH__
    const float4 t = __ldg(&kFFTrig[(int)::fminf(::fabsf(i), 205.f)]);   // (sin h, sin l, cos h, cos l)
#else
    const float4 t = make_float4(0.f, 0.f, 1.f, 0.f);
#endif
    const ff S = i < 0.f ? ff(-t.x, -t.y) : ff(t.x, t.y), C(t.z, t.w);
    const ff d = quick(fsub(x.h, i * 0.03125f), x.l);            // exact: i / 32 has x's exponent or less
    const float z = fmul(d.h, d.h);
    // sin d = d - d^3 / 6 (1 - d^2 / 20), cos d - 1 = -d^2 / 2 + d^4 / 24 (1 - d^2 / 30)
    const ff sd = quick(d.h, ffma(fmul(d.h, z), ffma(z, 1.f / 120.f, -1.f / 6.f), d.l));
    const ff d2 = d * d;
    const ff cd = quick(-0.5f * d2.h, ffma(fmul(z, z), ffma(z, -1.f / 720.f, 1.f / 24.f), -0.5f * d2.l));
    return FFSinCos{S + fma(S, cd, C * sd), C + fma(C, cd, -(S * sd))};
}
DRT_HD void sincos_ff(ff x, ff &s, ff &c) {
    const FFSinCos r = sincos_ff(x);
    s = r.s;
    c = r.c;
}
// the angle of (x, y) in [0, 2 pi): an FP32 angle t and the angle from it, (y cos t - x sin t) / |(x, y)|
inline __host__ __device__ __noinline__ ff angle2pi(ff y, ff x) {
    float t = atan2f(y.h, x.h);
    if (t < 0.f) t += 6.28318530717958648f;
    ff s, c;
    sincos_ff(ff(t, 0.f), s, c);
    const ff num = det2(y, c, x, s);
    return quick(t, fmul(num.h, rsqrtf(ffma(x.h, x.h, fmul(y.h, y.h)))));
}

// the angle of (x, y) as atan2f gives it, to its FP32 rounding: the FP32 angle and the angle from it
inline __host__ __device__ __noinline__ float atan2_ff(ff y, ff x) {
    const float t = atan2f(y.h, x.h), q = ffma(x.h, x.h, fmul(y.h, y.h));
    if (!(q > 0.f)) return t;
    ff s, c;
    sincos_ff(ff(t, 0.f), s, c);
    return fadd(t, fmul(det2(y, c, x, s).h, rsqrtf(q)));
}

}  // namespace drt
