// IEEE binary64 multiplication, division and square root, round to nearest
// even, in 32-bit integer arithmetic: the same bits as the hardware's operation
// for normal operands and results.
//
// Why: GB300 issues FP64 at 2 lanes per SM and clock, so one warp FP64
// instruction occupies the SM's FP64 pipe for 16 clocks while its four
// schedulers issue 64 other instructions.  Measured, SM clocks per warp
// operation with the SM full (24 warps): multiplication here 15 against 20,
// division 21 against 144, square root 27 against 173 (the hardware's
// sequences for these take 10-20 FP64 instructions); and they run beside the
// FP64 pipe, which keeps the additions.  Methods: schoolbook product; quotient
// and root from a single-precision seed, one Newton-Raphson step in 32-bit
// fixed point, one more 25-bit digit from the exact remainder, and a correction
// by the sign of the exact remainder of the rounded candidate (neither a
// quotient nor a root of 53-bit numbers falls halfway between two of them).
//
// Host code runs the same functions (tests/fp64_int_host.cpp compares them
// with the processor's arithmetic).
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define F64I_FN __device__ __forceinline__
#else
#define F64I_FN inline
#endif

namespace fetdpic {

typedef unsigned int u32;
typedef unsigned long long u64;

#ifdef __CUDACC__
F64I_FN u32 f64_hi(double a) { return (u32)__double2hiint(a); }
F64I_FN u32 f64_lo(double a) { return (u32)__double2loint(a); }
F64I_FN double f64_make(u32 hi, u32 lo) { return __hiloint2double((int)hi, (int)lo); }
F64I_FN u32 mulhi32(u32 a, u32 b) { return __umulhi(a, b); }
F64I_FN u32 shl_pair(u32 hi, u32 lo, u32 s) { return __funnelshift_l(lo, hi, s); }     // s in [0, 31]
// 64 x 64 -> 128 bits of (ah, al) (bh, bl), most significant word first.
F64I_FN void mul_128(u32 ah, u32 al, u32 bh, u32 bl, u32 &w3, u32 &w2, u32 &w1, u32 &w0)
{
    asm("{\n\t.reg .u32 t0, t1, t2;\n\t"
        "mul.lo.u32 %3, %4, %6;\n\tmul.hi.u32 t0, %4, %6;\n\t"
        "mad.lo.cc.u32 t0, %4, %7, t0;\n\tmadc.hi.u32 t1, %4, %7, 0;\n\t"
        "mad.lo.cc.u32 %2, %5, %6, t0;\n\tmadc.hi.cc.u32 t1, %5, %6, t1;\n\taddc.u32 t2, 0, 0;\n\t"
        "mad.lo.cc.u32 %1, %5, %7, t1;\n\tmadc.hi.u32 %0, %5, %7, t2;\n\t}"
        : "=&r"(w3), "=&r"(w2), "=&r"(w1), "=&r"(w0)
        : "r"(al), "r"(ah), "r"(bl), "r"(bh));
}
// (h, l) + (x, 0) + carry of r + c.
F64I_FN void add_round(u32 r, u32 c, u32 h, u32 x, u32 l, u32 &oh, u32 &ol)
{
    asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %2, %3;\n\taddc.cc.u32 %0, %4, 0;\n\taddc.u32 %1, %5, %6;\n\t}"
        : "=&r"(ol), "=&r"(oh)
        : "r"(r), "r"(c), "r"(l), "r"(h), "r"(x));
}
F64I_FN u32 as_u32(float a) { return __float_as_uint(a); }
F64I_FN float as_f32(u32 a) { return __uint_as_float(a); }
F64I_FN float seed_rcp(float a)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
F64I_FN float seed_rsqrt(float a)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
#else
F64I_FN u64 f64_bits(double a) { u64 v; std::memcpy(&v, &a, 8); return v; }
F64I_FN u32 f64_hi(double a) { return (u32)(f64_bits(a) >> 32); }
F64I_FN u32 f64_lo(double a) { return (u32)f64_bits(a); }
F64I_FN double f64_make(u32 hi, u32 lo) { const u64 v = ((u64)hi << 32) | lo; double a; std::memcpy(&a, &v, 8); return a; }
F64I_FN u32 mulhi32(u32 a, u32 b) { return (u32)(((u64)a * b) >> 32); }
F64I_FN u32 shl_pair(u32 hi, u32 lo, u32 s) { return s ? (hi << s) | (lo >> (32 - s)) : hi; }
F64I_FN void mul_128(u32 ah, u32 al, u32 bh, u32 bl, u32 &w3, u32 &w2, u32 &w1, u32 &w0)
{
    const u64 p0 = (u64)al * bl, p1 = (u64)al * bh + (p0 >> 32), p2 = (u64)ah * bl + (u32)p1;
    const u64 hi = (u64)ah * bh + (p1 >> 32) + (p2 >> 32);
    w3 = (u32)(hi >> 32); w2 = (u32)hi; w1 = (u32)p2; w0 = (u32)p0;
}
F64I_FN void add_round(u32 r, u32 c, u32 h, u32 x, u32 l, u32 &oh, u32 &ol)
{
    const u64 m = (((u64)h << 32) | l) + (((u64)r + c) >> 32);
    ol = (u32)m;
    oh = (u32)(m >> 32) + x;
}
F64I_FN u32 as_u32(float a) { u32 v; std::memcpy(&v, &a, 4); return v; }
F64I_FN float as_f32(u32 v) { float a; std::memcpy(&a, &v, 4); return a; }
float seed_rcp(float a);                      // the test supplies seeds with errors
float seed_rsqrt(float a);
#endif

constexpr u32 F64_EXP = 0x7ff00000u;          // exponent field of the high word
constexpr u32 F64_ONE = 0x3ff00000u;          // exponent field of 1.0

// True for zero and for 2^-LO <= |a| < 2^HI: the operands from which a chain of
// operations is started, LO and HI leaving room for the products formed of them.
template <int LO, int HI>
F64I_FN bool f64_within(double a)
{
    const u32 h = f64_hi(a) & 0x7fffffffu;
    return h - ((1023u - LO) << 20) < ((u32)(LO + HI) << 20) || (h | f64_lo(a)) == 0u;
}
F64I_FN bool f64_positive(double a)           // normal and above zero
{
    return f64_hi(a) - 0x100000u < 0x7fe00000u;
}
F64I_FN bool is_neg(double a)                 // a < 0 (not for NaN)
{
    const u32 h = f64_hi(a);
    return (h >> 31) != 0u && ((h << 1) | f64_lo(a)) != 0u;
}
// a 2^K for normal a and result, or zero.
template <int K>
F64I_FN double scale_i(double a)
{
    const u32 h = f64_hi(a);
    return f64_make((h & F64_EXP) != 0u ? h + ((u32)K << 20) : h, f64_lo(a));
}

// a b.  Normal operands and result, or a zero operand.
F64I_FN double mul_i(double a, double b)
{
    const u32 ha = f64_hi(a), la = f64_lo(a), hb = f64_hi(b), lb = f64_lo(b);
    const u32 ma = (ha & 0xfffffu) | 0x100000u, mb = (hb & 0xfffffu) | 0x100000u;
    // significands a (bit 52 set) and b 2^11 (bit 63 set): the product's upper 64 bits hold the
    // result's 53 or 52, the lower 64 what is rounded off
    u32 mh, ml, rh, rl;
    mul_128(ma, la, shl_pair(mb, lb, 11), lb << 11, mh, ml, rh, rl);
    const u32 s = (mh >> 20) ^ 1u;                                     // 1: one bit short
    mh = shl_pair(mh, ml, s);
    ml = shl_pair(ml, rh, s);
    rh = shl_pair(rh, rl, s);
    const u32 r = rh | (rl < 1u ? rl : 1u);                            // the rest as a sticky bit
    // sign and exponent: ha - ma and hb - mb are the operands' without their significands (and less
    // the implicit bit); the signs add up to their exclusive or modulo 2^32
    const u32 x = (ha - ma) + (hb - mb) - (s << 20) + (0x200000u - F64_ONE);
    // nearest even: carry of r + 2^31 - 1 + (last bit); mh brings its implicit bit along
    u32 oh, ol;
    add_round(r, 0x7fffffffu + (ml & 1u), mh, x, ml, oh, ol);
    const bool zero = (ha & F64_EXP) == 0u || (hb & F64_EXP) == 0u;
    return f64_make(zero ? (ha ^ hb) & 0x80000000u : oh, zero ? 0u : ol);
}

// a / b.  Normal operands and result, or a zero.
F64I_FN double div_i(double a, double b)
{
    const u32 ha = f64_hi(a), la = f64_lo(a), hb = f64_hi(b), lb = f64_lo(b);
    const u32 mah = (ha & 0xfffffu) | 0x100000u, mbh = (hb & 0xfffffu) | 0x100000u;
    const u64 ma = ((u64)mah << 32) | la, mb = ((u64)mbh << 32) | lb;
    const u32 at = shl_pair(mah, la, 11), bt = shl_pair(mbh, lb, 11);  // a, b in [1, 2) times 2^31
    // r ~ 2^32 / b from below: seed (reduced by 2^-20 so that it is), then one Newton step; the
    // truncations of the step are covered by the 4 units taken off
    const float fr = seed_rcp(as_f32(0x3f800000u | ((bt >> 8) & 0x7fffffu)));
    const u32 fb = as_u32(fr - fr * 0x1p-20f);
    u32 r = fb >= 0x3f000000u ? (fb << 8) | 0x80000000u : 0x80000000u;
    const u32 e = 0x80000000u - mulhi32(bt, r);
    r = r - 4u + mulhi32(r, e << 1);
    const u32 q1 = mulhi32(at, r);                                     // a/b 2^31, low by at most about 10
    const u64 rem = (ma << 31) - (u64)q1 * mb;                         // exact modulo 2^64, below 2^57
    const u32 q2 = mulhi32((u32)(rem >> 25), r) >> 2;                  // rem/b 2^25
    const u64 q = ((u64)q1 << 25) + q2;                                // a/b 2^56, low by at most about 3
    const u32 n = (u32)(q >> 56);                                      // 1: a >= b
    u64 c = (q + (4u << n)) >> (3u + n);                               // the candidate, 53 bits
    // a/b 2^(53 - n) - c, in units of 1/b: beyond half a unit either way the neighbour is nearer
    const long long d = (long long)((ma << (53u - n)) - c * mb);
    c += (u64)((long long)(2 * d > (long long)mb) - (long long)(2 * d < -(long long)mb));
    const u32 sign = (ha ^ hb) & 0x80000000u;
    const u32 oh = (u32)(c >> 32) + (ha & F64_EXP) - (hb & F64_EXP) + (n << 20) + (F64_ONE - 0x200000u);
    const bool zero = (ha & F64_EXP) == 0u;
    return f64_make((zero ? 0u : oh) | sign, zero ? 0u : (u32)c);
}

// sqrt(a).  a normal and positive.
F64I_FN double sqrt_i(double a)
{
    const u32 h = f64_hi(a), l = f64_lo(a);
    const u32 odd = ((h >> 20) & 1u) ^ 1u;                             // exponent of a odd: field even
    const u32 mh = (h & 0xfffffu) | 0x100000u;
    const u64 m = (((u64)mh << 32) | l) << odd;                        // m in [1, 4) times 2^52
    const u32 mt = (u32)(m >> 22);                                     // m 2^30
    // r ~ 2^32 / sqrt(m) from below
    const float fm = as_f32((odd ? 0x40000000u : 0x3f800000u) | shl_pair(h & 0xfffffu, l, 3));
    const float fr = seed_rsqrt(fm);
    const u32 fb = as_u32(fr - fr * 0x1p-20f);
    u32 r = fb >= 0x3f000000u ? (fb << 8) | 0x80000000u : 0x80000000u;
    const u32 e = 0x40000000u - mulhi32(mulhi32(mt, r), r);            // 2^30 (1 - m r^2)
    r = r - 4u + mulhi32(r, e << 1);
    const u32 s1 = mulhi32(mt, r) - 4u;                                // sqrt(m) 2^30 from below
    const u64 rem = (m << 8) - (u64)s1 * s1;                           // exact, below 2^36
    const u32 q2 = mulhi32((u32)(rem >> 4), r) >> 2;                   // rem / (2 s1) 2^25
    u64 c = (((u64)s1 << 25) + q2 + 4u) >> 3;                          // the candidate
    const long long d = (long long)((m << 52) - c * c);
    c += (u64)((long long)(d > (long long)c) - (long long)(d <= -(long long)c));
    const u32 oh = (u32)(c >> 32) + ((((h >> 20) + 1023u) >> 1) << 20) - 0x100000u;
    return f64_make(oh, (u32)c);
}

// round(a) to the nearest even integer, saturating at the ends of 64 bits.
F64I_FN long long rint_i(double a)
{
    const u32 h = f64_hi(a), l = f64_lo(a);
    const int e = (int)((h >> 20) & 0x7ffu) - 1075;                    // a = significand 2^e
    u64 m = ((u64)((h & 0xfffffu) | 0x100000u) << 32) | l;
    if (e > 10) return (h >> 31) ? (long long)0x8000000000000000ull : 0x7fffffffffffffffll;
    if (e >= 0) {
        m <<= e;
    } else {
        const int s = e < -54 ? 54 : -e;                               // below 2^-1 all bits leave
        m = (m + (1ull << (s - 1)) - 1ull + ((m >> s) & 1ull)) >> s;
    }
    return (h >> 31) ? -(long long)m : (long long)m;
}

// (float)a, nearest even, and (double)a, without the FP64 pipe (which does conversions too):
// normal results; others through the hardware's conversion.
F64I_FN float to_f32(double a)
{
    const u32 h = f64_hi(a), l = f64_lo(a);
    const u32 u = (h & 0x7fffffffu) - (896u << 20);                    // exponent field of the result
    if (u - 0x100000u >= (253u << 20)) return (float)a;
    const u32 b = shl_pair(u, l, 3);
    u32 o, carry;
    add_round(l << 3, 0x7fffffffu + (b & 1u), 0u, 0u, b, carry, o);
    return as_f32(o | (h & 0x80000000u));
}
F64I_FN double to_f64(float a)
{
    const u32 b = as_u32(a), m = b & 0x7fffffffu;
    if (m - 0x800000u >= 0x7f000000u) return (double)a;
    return f64_make(((m >> 3) + (896u << 20)) | (b & 0x80000000u), b << 29);
}

}  // namespace fetdpic
