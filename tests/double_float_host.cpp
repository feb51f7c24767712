// double_float.h on the host: errors of the high-gamma push, and of the same push in FP64 with one
// Newton step to a root, against extended precision.  Single-precision seeds off by up to `ulps` units.
// Prints "pusher range quantity fp64_rms f2_rms fp64_max f2_max".
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "double_float.h"

using namespace fetdpic;
typedef long double real;

static unsigned long long state = 0x9e3779b97f4a7c15ull;
static unsigned long long rnd()
{
    state ^= state << 13; state ^= state >> 7; state ^= state << 17;
    return state;
}
static double uniform() { return (double)(rnd() >> 11) * 0x1p-53; }
static double spread(double a, double b) { return std::exp(std::log(a) + uniform() * std::log(b / a)); }
static int ulps = 1;
static float off(float v)
{
    for (int k = 0; k < ulps; ++k) {
        const int s = (int)(rnd() & 3);
        if (s < 2) v = std::nextafter(v, s ? 1e30f : 0.f);
    }
    return v;
}
namespace fetdpic {
float rsqrt_seed(float a) { return off((float)(1.0 / std::sqrt((double)a))); }
float rcp_seed(float a) { return off(1.0f / a); }
}

template <typename T> struct Result { T ux, uy, ig; };

template <typename T, int PUSHER, typename R, typename I>
static Result<T> push(T ux, T uy, T ex, T ey, T bz, R rsq, I rcp)
{
    const T bb = bz * bz;
    if (PUSHER == FETDPIC_VAY) {
        const T g0 = rsq(1 + ux * ux + uy * uy);
        const T px = ux + 2 * ex + uy * g0 * bz, py = uy + 2 * ey - ux * g0 * bz;
        const T sigma = 1 + px * px + py * py - bb, r2 = sigma * sigma + 4 * bb;
        const T ig = rsq((sigma + r2 * rsq(r2)) / 2), t = bz * ig, s = rcp(1 + t * t);
        return {s * (px + py * t), s * (py - px * t), ig};
    }
    const T mx = ux + ex, my = uy + ey, g2 = 1 + mx * mx + my * my;
    T t;
    if (PUSHER == FETDPIC_HC) {
        const T sigma = g2 - bb, r2 = sigma * sigma + 4 * bb;
        t = bz * rsq((sigma + r2 * rsq(r2)) / 2);
    } else {
        t = bz * rsq(g2);
        if (PUSHER == FETDPIC_BORIS_TAN) t = std::tan(t);
    }
    const T s = 2 * t * rcp(1 + t * t), rx = mx + my * t, ry = my - mx * t;
    const T x = mx + ry * s + ex, y = my - rx * s + ey;
    return {x, y, rsq(1 + x * x + y * y)};
}

struct Error {
    real sum = 0, top = 0;
    void add(real e) { sum += e * e; top = std::max(top, e); }
};

template <int PUSHER>
static void measure(const char *name, long long n, int range)
{
    static const double lim[4][4] = {{10.1, 3e8, 1e-9, 0.12}, {10.1, 1e3, 1e-4, 0.02}, {10.1, 1e3, 0.03, 0.12}, {10.1, 1e4, 1e-9, 1e-5}};
    const double *L = lim[range];
    Error e[3][2];
    for (long long k = 0; k < n; ++k) {
        const double g = spread(L[0], L[1]), p = std::sqrt(g * g - 1), th = 6.283185307179586 * uniform();
        const double kick = g * spread(L[2], L[3]), ph = 6.283185307179586 * uniform();
        const double top = PUSHER == FETDPIC_BORIS_TAN ? std::min(L[3], 0.031) : L[3];
        const float ux = (float)(p * std::cos(th)), uy = (float)(p * std::sin(th));
        const float ex = (float)(kick * std::cos(ph)), ey = (float)(kick * std::sin(ph));
        const float bz = (float)((rnd() & 1 ? 1 : -1) * g * spread(std::min(L[2], top / 4), top));
        const auto r = push<real, PUSHER>(ux, uy, ex, ey, bz, [](real v) { return 1 / std::sqrt(v); }, [](real v) { return 1 / v; });
        const auto d = push<double, PUSHER>(
            ux, uy, ex, ey, bz,
            [](double v) { const double y = rsqrt_seed((float)v); return y * (1.5 - 0.5 * v * (y * y)); },
            [](double v) { const double y = 1.0f / (float)v; return y * (2.0 - v * y); });
        const HighPush h = high_gamma_push<PUSHER>(ux, uy, ex, ey, bz);
        const D2 v = h.u.x * normal(h.ig);
        const real size = std::sqrt(r.ux * r.ux + r.uy * r.uy);
        const real fx = (real)h.u.x.h.x + h.u.x.l.x + h.u.l.x, fy = (real)h.u.x.h.y + h.u.x.l.y + h.u.l.y;
        const real hg = (real)h.ig.h + h.ig.l, vx = r.ux * r.ig, vy = r.uy * r.ig;
        e[0][0].add(std::hypot(d.ux - r.ux, d.uy - r.uy) / size);
        e[0][1].add(std::hypot(fx - r.ux, fy - r.uy) / size);
        e[1][0].add(std::fabs(d.ig / r.ig - 1));
        e[1][1].add(std::fabs(hg / r.ig - 1));
        e[2][0].add(std::hypot(d.ux * d.ig - vx, d.uy * d.ig - vy));
        e[2][1].add(std::hypot((real)v.h.x + v.l.x - vx, (real)v.h.y + v.l.y - vy));
    }
    const char *what[3] = {"u", "ig", "v"};
    for (int k = 0; k < 3; ++k)
        printf("%s %d %s %.3Le %.3Le %.3Le %.3Le\n", name, range, what[k], std::sqrt(e[k][0].sum / n), std::sqrt(e[k][1].sum / n),
               e[k][0].top, e[k][1].top);
}

int main(int argc, char **argv)
{
    const long long n = argc > 1 ? atoll(argv[1]) : 200000;
    ulps = argc > 2 ? atoi(argv[2]) : 1;
    for (int range = 0; range < 4; ++range) {
        measure<FETDPIC_BORIS>("boris", n, range);
        measure<FETDPIC_BORIS_TAN>("boris_tan", n, range);
        measure<FETDPIC_VAY>("vay", n, range);
        measure<FETDPIC_HC>("hc", n, range);
    }
    return 0;
}
