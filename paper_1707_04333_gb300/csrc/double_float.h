// Double-float arithmetic and the relativistic push in it, for particles above
// gamma = 10, where FP32 loses 1 - v/c and the cancellation in sigma.
//
// A value is held as an unevaluated sum h + l of two floats, |l| of a few ulp(h)
// at most: some 47 significand bits from FP32 additions and fused multiply-adds
// (Dekker 1971; Knuth's two-sum).  GB300 issues FP64 at 2 lanes per SM and clock
// and FP32 at 60 times that, so the operations of one double-float operation
// take a fraction of one FP64 instruction's time.
//
// What fewer bits than FP64's 53 leave of the result is decided by the order of
// the operations.  The former FP64 push took its roots from a single-precision
// seed and one Newton step, which left 3e-15 in 1/gamma.  Here that step has one
// more term, and u^{n+1/2} is u^{n-1/2} + 2 eps, exact in two floats, plus the
// rotation, a small share of u, in three.  rms (largest) error of |u| and of
// 1/gamma against extended precision before the rounding to FP32, a million
// particles each on the device, FP64 push / here:
//   gamma 10 to 1000, kick and |beta| up to gamma / 50 (a beam)
//     Higuera-Cary  u 7.1e-17 (1.0e-15) / 4.4e-17 (8.1e-16)   1/gamma 3.4e-15 (3.3e-14) / 2.3e-15 (1.9e-14)
//     Vay           u 1.7e-15 (8.3e-15) / 4.0e-17 (8.1e-16)   1/gamma 3.1e-15 (3.2e-14) / 2.6e-15 (2.2e-14)
//     Boris         u 7.4e-17 (1.1e-15) / 4.1e-17 (6.9e-16)   1/gamma 3.4e-15 (3.3e-14) / 2.3e-15 (2.2e-14)
//     Boris-tan     u 7.4e-17 (1.2e-15) / 4.3e-17 (6.7e-16)   1/gamma 3.4e-15 (3.4e-14) / 2.3e-15 (2.3e-14)
//   gamma 10 to 1000, kick and |beta| between gamma / 33 and gamma / 8
//     Higuera-Cary  u 6.1e-16 (7.0e-15) / 5.0e-16 (5.3e-15)   Vay        2.2e-15 (8.3e-15) / 4.5e-16 (5.2e-15)
//     Boris         u 6.6e-16 (8.1e-15) / 4.5e-16 (4.1e-15)   Boris-tan  1.8e-16 (2.0e-15) / 1.2e-16 (1.3e-15)
// and below the FP64 push's likewise over gamma 10 to 3e8 and kicks down to
// 1e-9 gamma.  The stored FP32 momenta and the FP32 velocities, rounded at 6e-8,
// agree but for one in a million.
//
// Host code runs the same functions (tests/double_float_host.cpp measures them).
#pragma once

#include <cmath>

#include "fetdpic.h"

#ifdef __CUDACC__
#define DF_FN __device__ __forceinline__
#else
#define DF_FN inline
#endif

namespace fetdpic {

// Operations rounded one by one: the error terms must not be contracted.  V2 is
// a vector's two components in one register pair: the packed FP32 instructions
// round each half as the scalar ones do and take one issue slot for two
// operations (the rate in lanes is the same: 120 per SM and clock either way),
// and it is issue slots that a kernel full of pushes is bound by.
#ifdef __CUDACC__
DF_FN float add_f(float a, float b) { return __fadd_rn(a, b); }
DF_FN float sub_f(float a, float b) { return __fsub_rn(a, b); }
DF_FN float mul_f(float a, float b) { return __fmul_rn(a, b); }
DF_FN float fma_f(float a, float b, float c) { return __fmaf_rn(a, b, c); }
DF_FN float rsqrt_seed(float a) { return rsqrtf(a); }
DF_FN float rcp_seed(float a) { return __fdividef(1.f, a); }
struct V2 { unsigned long long v; };
DF_FN V2 vec(float x, float y)
{
    V2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
DF_FN void parts(V2 a, float &x, float &y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v)); }
DF_FN V2 operator+(V2 a, V2 b)
{
    V2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
DF_FN V2 operator-(V2 a, V2 b)
{
    V2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
DF_FN V2 operator*(V2 a, V2 b)
{
    V2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
DF_FN V2 fma(V2 a, V2 b, V2 c)
{
    V2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
#else
DF_FN float add_f(float a, float b) { return a + b; }
DF_FN float sub_f(float a, float b) { return a - b; }
DF_FN float mul_f(float a, float b) { return a * b; }
DF_FN float fma_f(float a, float b, float c) { return std::fma(a, b, c); }
float rsqrt_seed(float a);                    // the test supplies seeds with errors
float rcp_seed(float a);
struct V2 { float x, y; };
DF_FN V2 vec(float x, float y) { return V2{x, y}; }
DF_FN void parts(V2 a, float &x, float &y) { x = a.x; y = a.y; }
DF_FN V2 operator+(V2 a, V2 b) { return V2{a.x + b.x, a.y + b.y}; }
DF_FN V2 operator-(V2 a, V2 b) { return V2{a.x - b.x, a.y - b.y}; }
DF_FN V2 operator*(V2 a, V2 b) { return V2{a.x * b.x, a.y * b.y}; }
DF_FN V2 fma(V2 a, V2 b, V2 c) { return V2{std::fma(a.x, b.x, c.x), std::fma(a.y, b.y, c.y)}; }
#endif

// A result is renormalised only where its low part's size shows: products and sums take a low part of a
// few ulp as well as one of half an ulp.
struct F2 {
    float h, l;
    DF_FN F2() {}
    DF_FN F2(float a, float b) : h(a), l(b) {}
};
DF_FN F2 quick_two_sum(float a, float b)          // |a| >= |b|
{
    const float s = add_f(a, b);
    return F2(s, sub_f(b, sub_f(s, a)));
}
DF_FN F2 two_sum(float a, float b)
{
    const float s = add_f(a, b), t = sub_f(s, a);
    return F2(s, add_f(sub_f(a, sub_f(s, t)), sub_f(b, t)));
}
DF_FN F2 two_prod(float a, float b)
{
    const float p = mul_f(a, b);
    return F2(p, fma_f(a, b, -p));
}
DF_FN F2 add_small(const F2 &a, float b)          // |a| >= |b|
{
    const F2 s = quick_two_sum(a.h, b);
    return F2(s.h, add_f(s.l, a.l));
}
DF_FN F2 add_small(const F2 &a, const F2 &b)
{
    const F2 s = quick_two_sum(a.h, b.h);
    return F2(s.h, add_f(s.l, add_f(a.l, b.l)));
}
DF_FN F2 operator*(const F2 &a, const F2 &b)
{
    const F2 p = two_prod(a.h, b.h);
    return F2(p.h, fma_f(a.l, b.h, fma_f(a.h, b.l, p.l)));
}
DF_FN F2 operator*(const F2 &a, float b)
{
    const F2 p = two_prod(a.h, b);
    return F2(p.h, fma_f(a.l, b, p.l));
}
DF_FN F2 sqr(const F2 &a)
{
    const F2 p = two_prod(a.h, a.h);
    return F2(p.h, fma_f(add_f(a.h, a.h), a.l, p.l));
}
DF_FN F2 normal(const F2 &a) { return quick_two_sum(a.h, a.l); }
DF_FN F2 scale(const F2 &a, float p2) { return F2(a.h * p2, a.l * p2); }   // p2: a power of two
// 1/sqrt(x), sqrt(x), 1/x from a single-precision seed y: with the residual e = 1 - x y^2
// (1 - x y), formed without rounding its leading part, y (1 + e/2 + 3 e^2 / 8) and y (1 + e + e^2).
// A seed within 2 ulp leaves the roundings, some 2^-48.
DF_FN float rsqrt_residual(const F2 &x, float y, F2 &xy)
{
    xy = two_prod(x.h, y);
    xy.l = fma_f(x.l, y, xy.l);
    return fma_f(-xy.l, y, fma_f(-xy.h, y, 1.f));
}
DF_FN F2 rsqrt_f2(const F2 &x)
{
    const float y = rsqrt_seed(x.h);
    F2 xy;
    const float e = rsqrt_residual(x, y, xy);
    return F2(y, fma_f(0.5f * y, e, 0.375f * (y * e) * e));
}
DF_FN F2 sqrt_f2(const F2 &x)
{
    const float y = rsqrt_seed(x.h);
    F2 xy;
    const float e = rsqrt_residual(x, y, xy);
    return F2(xy.h, fma_f(0.5f * xy.h, e, fma_f(0.375f * (xy.h * e), e, xy.l)));
}
DF_FN F2 rcp_f2(const F2 &x)
{
    const float y = rcp_seed(x.h);
    const float e = fma_f(-x.l, y, fma_f(-x.h, y, 1.f));
    return F2(y, y * fma_f(e, e, e));
}

DF_FN V2 neg(V2 a)
{
    float x, y;
    parts(a, x, y);
    return vec(-x, -y);
}
DF_FN V2 swap(V2 a)
{
    float x, y;
    parts(a, x, y);
    return vec(y, x);
}
struct D2 { V2 h, l; };                                                // a vector of two double-floats
DF_FN D2 two_sum(V2 a, V2 b)
{
    const V2 s = a + b, t = s - a;
    return D2{s, (a - (s - t)) + (b - t)};
}
DF_FN D2 normal(const D2 &a)
{
    const V2 s = a.h + a.l;
    return D2{s, a.l - (s - a.h)};
}
DF_FN D2 operator*(const D2 &a, const D2 &b)
{
    const V2 p = a.h * b.h;
    return D2{p, fma(a.l, b.h, fma(a.h, b.l, fma(a.h, b.h, neg(p))))};
}
DF_FN D2 operator+(const D2 &a, const D2 &b)
{
    const D2 s = two_sum(a.h, b.h);
    return D2{s.h, s.l + (a.l + b.l)};
}
// (a_y, a_x) (s, -s)
DF_FN D2 cross(V2 a, const F2 &s)
{
    const V2 b = swap(a), h = vec(s.h, -s.h), p = b * h;
    return D2{p, fma(b, vec(s.l, -s.l), fma(b, h, neg(p)))};
}
DF_FN D2 operator*(const D2 &a, const F2 &s) { return a * D2{vec(s.h, s.h), vec(s.l, s.l)}; }
// 1 + a_x^2 + a_y^2, where |a| > 1
DF_FN F2 one_plus_norm2(const D2 &a)
{
    const V2 p = a.h * a.h, l = fma(a.h + a.h, a.l, fma(a.h, a.h, neg(p)));
    float px, py, lx, ly;
    parts(p, px, py);
    parts(l, lx, ly);
    const F2 s = two_sum(px, py);
    return add_small(F2(s.h, add_f(s.l, add_f(lx, ly))), 1.f);
}

DF_FN F2 one_plus_norm2(V2 a)
{
    const V2 p = a * a, l = fma(a, a, neg(p));
    float px, py, lx, ly;
    parts(p, px, py);
    parts(l, lx, ly);
    const F2 s = two_sum(px, py);
    return add_small(F2(s.h, add_f(s.l, add_f(lx, ly))), 1.f);
}

DF_FN D2 perp(const D2 &a)                                         // a x z = (a_y, -a_x)
{
    float hx, hy, lx, ly;
    parts(a.h, hx, hy);
    parts(a.l, lx, ly);
    return D2{vec(hy, -hx), vec(ly, -lx)};
}
// Three floats a component, (x.h, x.l) normalised: where a sum's low parts are rounded to one float, that
// rounding shows beside the error of a small addend.
struct T2 { D2 x; V2 l; };
DF_FN T2 add_exact(const D2 &a, const D2 &b)
{
    const D2 s = two_sum(a.h, b.h), p = two_sum(a.l, s.l), m = two_sum(p.h, b.l);
    return T2{normal(D2{s.h, m.h}), p.l + m.l};
}

// u^{n+1/2} and 1/gamma^{n+1/2}.
struct HighPush { T2 u; F2 ig; };

template <int PUSHER>
DF_FN HighPush high_gamma_push(float ux, float uy, float ex, float ey, float bz)
{
    // gamma > 10, |kick| < gamma / 8 and |beta| < gamma / 8, so |u^-|^2, |u'|^2 and |u^{n+1}|^2 exceed
    // both 1 and |beta|^2, and t^2 < 1: those sums need no two-sum.  u^{n+1/2} is formed as u^{n-1/2} + 2 eps,
    // exact in two floats, plus the rotation, whose error is a small share of u
    const V2 u = vec(ux, uy), eps = vec(ex, ey);
    HighPush o;
    if (PUSHER == FETDPIC_VAY) {
        const F2 w = rsqrt_f2(one_plus_norm2(u)) * bz;
        const T2 up = add_exact(two_sum(u, eps + eps), cross(u, w));
        const F2 bb = two_prod(bz, bz);
        const F2 sigma = normal(add_small(one_plus_norm2(up.x), F2(-bb.h, -bb.l)));
        const F2 root = sqrt_f2(add_small(sqr(sigma), scale(bb, 4.f)));
        o.ig = rsqrt_f2(scale(add_small(root, sigma), 0.5f));
        const F2 tz = o.ig * bz, q = sqr(tz);
        const F2 s = rcp_f2(add_small(F2(1.f, 0.f), q));
        // (u' + u' x t) s = u' + (u' x z - t u') t s.  (Of six ways to write this sum, one that leaves the
        // 80-register window kernel of the thermal plasma as it was: 133.2 us a step against 138.)
        o.u = add_exact(up.x, (perp(up.x) + up.x * F2(-tz.h, -tz.l)) * (tz * s));
        o.u.l = o.u.l + up.l;
    } else {
        const D2 um = two_sum(u, eps);                                 // u^-
        const F2 g2 = one_plus_norm2(um);
        F2 tz;
        if (PUSHER == FETDPIC_HC) {
            const F2 bb = two_prod(bz, bz);
            const F2 sigma = normal(add_small(g2, F2(-bb.h, -bb.l)));
            const F2 root = sqrt_f2(add_small(sqr(sigma), scale(bb, 4.f)));
            tz = normal(rsqrt_f2(normal(scale(add_small(root, sigma), 0.5f))) * bz);
        } else {
            tz = normal(rsqrt_f2(normal(g2)) * bz);
        }
        F2 q = sqr(tz);
        if (PUSHER == FETDPIC_BORIS_TAN) {
            // tan t = t + t (t^2/3 + 2 t^4/15 + 17 t^6/315 + 62 t^8/2835 + ...): the first neglected
            // term is below 1e-15 of t for |t| < 0.04; 1/3 and 2/15 as double-floats
            const float c1 = 1.f / 3.f, c1l = (float)(1.0 / 3.0 - (double)c1);
            const float c2 = 2.f / 15.f, c2l = (float)(2.0 / 15.0 - (double)c2);
            const F2 r = add_small(F2(c2, c2l), q.h * (17.f / 315.f + q.h * (62.f / 2835.f)));
            tz = normal(add_small(tz, tz * (q * add_small(F2(c1, c1l), q * r))));
            q = sqr(tz);
        }
        // s = 2 t / (1 + t^2) = 2 t - 2 t t^2 / (1 + t^2); (u^- + u^- x t) x s = (u^- x z - t u^-) s
        const F2 t2 = scale(tz, 2.f), r = t2 * q * rcp_f2(add_small(F2(1.f, 0.f), q));
        const F2 sz = normal(add_small(t2, F2(-r.h, -r.l)));
        o.u = add_exact(two_sum(u, eps + eps), (perp(um) + um * F2(-tz.h, -tz.l)) * sz);
        o.ig = rsqrt_f2(one_plus_norm2(o.u.x));
    }
    return o;
}

}  // namespace fetdpic
