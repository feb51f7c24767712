// fp64_int.h on the host against the processor's IEEE arithmetic: random and
// edge operands, with the single-precision seeds off by up to `ulps` units.
// Prints the number of differing results of each operation.
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "fp64_int.h"

using namespace fetdpic;

static u64 state = 0x9e3779b97f4a7c15ull;
static u64 rnd()
{
    state ^= state << 13; state ^= state >> 7; state ^= state << 17;
    return state;
}
static int ulps = 0;
static float off(float v)
{
    if (!ulps) return v;
    const int k = (int)(rnd() % (u64)(2 * ulps + 1)) - ulps;
    return fetdpic::as_f32(fetdpic::as_u32(v) + (u32)k);
}
namespace fetdpic {
float seed_rcp(float a) { return off(1.0f / a); }
float seed_rsqrt(float a) { return off((float)(1.0 / std::sqrt((double)a))); }
}

// exponents in [-span, span]; a share of the significands with long runs of ones or zeros
static double value(int span)
{
    u64 m = rnd() & 0xfffffffffffffull;
    switch (rnd() % 6) {
    case 0: m &= ~0ull << (rnd() % 53); break;
    case 1: m |= (1ull << (rnd() % 53)) - 1; break;
    case 2: m = (1ull << (rnd() % 52)); break;
    case 3: m = 0xfffffffffffffull ^ (1ull << (rnd() % 52)); break;
    default: break;
    }
    m &= 0xfffffffffffffull;
    const u64 e = 1023 + (u64)((long long)(rnd() % (u64)(2 * span + 1)) - span);
    const u64 v = ((rnd() & 1) << 63) | (e << 52) | m;
    double a;
    std::memcpy(&a, &v, 8);
    return a;
}
static bool same(double a, double b) { return f64_bits(a) == f64_bits(b); }

int main(int argc, char **argv)
{
    const long long n = argc > 1 ? atoll(argv[1]) : 1000000;
    ulps = argc > 2 ? atoi(argv[2]) : 2;
    long long bm = 0, bd = 0, bs = 0, br = 0, bc = 0;
    for (long long k = 0; k < n; ++k) {
        double a = value(k & 1 ? 2 : 400), b = value(k & 2 ? 2 : 400);
        if (k % 13 == 0) b = a * (1.0 + 0x1p-52 * (double)(rnd() % 3));      // quotients next to 1
        if (k % 17 == 0) a = b * b;                                        // exact roots and quotients
        if (k % 101 == 0) a = k & 1 ? 0.0 : -0.0;
        if (a == 0.0 || std::isnormal(a * b)) bm += !same(mul_i(a, b), a * b);
        bd += !same(div_i(a, b), a / b);
        if (a != 0.0) bs += !same(sqrt_i(std::fabs(a)), std::sqrt(std::fabs(a)));
        bm += !same(scale_i<2>(b), 4.0 * b) + !same(scale_i<-1>(a), 0.5 * a) + (is_neg(a) != (a < 0.0));
        const double w = k % 23 == 0 ? a * 0.0 : value(k & 4 ? 2 : 160);
        const float f = (float)w, g = as_f32((u32)rnd());
        bc += as_u32(to_f32(w)) != as_u32(f) || !same(to_f64(f), (double)f);
        if (g == g) bc += !same(to_f64(g), (double)g);
        double c = value(61);
        if (k % 7 == 0) c = (double)((long long)(rnd() % 4000000) - 2000000) * 0.5;
        br += rint_i(c) != (long long)std::nearbyint(c);
        if (k % 1000 == 0) br += rint_i(0x1p63) != 0x7fffffffffffffffll || rint_i(-0x1p70) != -0x7fffffffffffffffll - 1 || rint_i(0.0) != 0;
    }
    printf("mul %lld div %lld sqrt %lld rint %lld convert %lld\n", bm, bd, bs, br, bc);
    return (bm | bd | bs | br | bc) != 0;
}
