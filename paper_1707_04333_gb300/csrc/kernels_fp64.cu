// Plain-FP64 kernels of the FETD-PIC step (Faraday update + the fused
// gather / push / walk / deposit particle kernel).
//
// This file is compiled with -fmad=false: every multiply and add rounds as
// written, in the order written, so a step from a given state reproduces a
// plain FP64 evaluation of the paper's formulas bit for bit (cells, crossed
// edges, positions, momenta).  Division and square root are IEEE
// correctly-rounded in CUDA and so also reproducible.
#include <cuda_runtime.h>

#include "fetdpic_internal.h"
#include "fp64_int.h"

namespace fetdpic {

// Faraday, Eq. (semi.dis.curl.1): b^{n+1/2} = b^{n-1/2} - dt C e^n, in place,
// fused with the per-triangle field record the particles gather from:
// (s_m e_m) for the three local edges and B_z^n = (b^{n+1/2}+b^{n-1/2})/(2A).
__global__ void k_faraday64(int F, const Geo64 *__restrict__ geo, const Topo *__restrict__ topo,
                            const double *__restrict__ e, double *__restrict__ b, Rec64 *__restrict__ rec, int E,
                            unsigned long long *__restrict__ ifix)
{
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    int3 w{};
    double dt = 0.0, inv2A = 0.0;
    if (f < F) {
        // static, loaded before the wait for the kernel that writes e
        w = make_int3(topo[f].ew[0], topo[f].ew[1], topo[f].ew[2]);
        dt = geo[f].dt; inv2A = geo[f].inv2A;
    }
    pdl_begin();
    for (int k = f; k < E; k += gridDim.x * blockDim.x) ifix[k] = 0ull;      // for the particle kernel
    if (f >= F) return;
    const int ew[3] = {w.x, w.y, w.z};
    double se[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const double v = e[ew[m] >> 1];
        se[m] = (ew[m] & 1) ? -v : v;
    }
    double ce = 0.0;
    ce = ce + se[0];
    ce = ce + se[1];
    ce = ce + se[2];
    const double bo = b[f];
    const double bn = bo - dt * ce;
    b[f] = bn;
    Rec64 r;
    r.se[0] = se[0]; r.se[1] = se[1]; r.se[2] = se[2];
    r.bz = (bn + bo) * inv2A;
    rec[f] = r;
}

void launch_faraday64(cudaStream_t st, int F, const Geo64 *geo, const Topo *topo, const double *e,
                      double *b, Rec64 *rec, int E, unsigned long long *ifix, bool pdl)
{
    if (F <= 0) return;
    launch_k(pdl, k_faraday64, dim3((F + 255) / 256), dim3(256), st, F, geo, topo, e, b, rec, E, ifix);
}

// ------------------------------------------------------------ arithmetic
// The particle kernel's arithmetic comes in two forms with the same bits: the
// hardware's FP64 instructions, and multiplication, division, square root and
// the conversion to integers in 32-bit integer instructions (fp64_int.h), with
// additions and a few products left on the FP64 pipe (about as many as balance
// the two).  GB300's FP64 pipe passes 2 lanes per SM and clock and bounded the
// hardware form (83 % busy, the schedulers 8 %).
// The integer form takes operands whose products and quotients stay normal;
// a particle with others (checked as they are loaded) takes the hardware form.
struct Hard {
    static constexpr bool SOFT = false;
    static __device__ __forceinline__ double mul(double a, double b) { return a * b; }
    static __device__ __forceinline__ double div(double a, double b) { return a / b; }
    static __device__ __forceinline__ double root(double a) { return sqrt(a); }
    static __device__ __forceinline__ double twice(double a) { return 2.0 * a; }
    static __device__ __forceinline__ double half(double a) { return 0.5 * a; }
    static __device__ __forceinline__ double four(double a) { return 4.0 * a; }
    static __device__ __forceinline__ long long round(double a) { return __double2ll_rn(a); }
    static __device__ __forceinline__ bool neg(double a) { return a < 0.0; }
};
// (Out of line, and the loops over the three nodes or edges left rolled: the
// straight-line form of a push is about 3,500 instructions, and its warps then
// wait for instructions more than for anything else.)
__device__ __noinline__ double div_call(double a, double b) { return div_i(a, b); }
__device__ __noinline__ double root_call(double a) { return sqrt_i(a); }
struct Soft {
    static constexpr bool SOFT = true;
    static __device__ __forceinline__ double mul(double a, double b) { return mul_i(a, b); }
    static __device__ __forceinline__ double div(double a, double b) { return div_call(a, b); }
    static __device__ __forceinline__ double root(double a) { return root_call(a); }
    static __device__ __forceinline__ double twice(double a) { return scale_i<1>(a); }
    static __device__ __forceinline__ double half(double a) { return scale_i<-1>(a); }
    static __device__ __forceinline__ double four(double a) { return scale_i<2>(a); }
    // an addition rounds |a| < 2^51 to an integer in its low bits
    static __device__ __forceinline__ long long round(double a)
    {
        if ((f64_hi(a) & 0x7fffffffu) >= ((1023u + 51u) << 20)) return rint_i(a);
        return __double_as_longlong(a + 0x1.8p52) - __double_as_longlong(0x1.8p52);
    }
    static __device__ __forceinline__ bool neg(double a) { return is_neg(a); }
};

// ------------------------------------------------------------------ push
// 2-D TE specialisation (u_z = 0, E_z = 0, B along z) of the 3-vector
// formulas of Sec. II.C; with u_z = 0 every dropped term is an exact zero,
// so the rounding equals the 3-vector evaluation.

struct Push { double ux, uy, g; };

template <class A>
__device__ __forceinline__ double gam2(double ux, double uy, double ic2)
{
    return A::root(1.0 + A::mul(A::mul(ux, ux) + A::mul(uy, uy), ic2));
}

// `ok` (integer form): cleared when u' or u^- leaves the range the rest is safe for, and where the
// gamma of the quartic is the root of exactly 0: sigma + sqrt(sigma^2 + 4 beta^2) cancels completely from
// |beta| of about 2^27 on, and sqrt_i takes positive numbers only.  (The FP64 instructions then find
// beta / 0 and report the particle as not finite.)
template <class A, int PUSHER>
__device__ __forceinline__ Push push64(double ux, double uy, double Ex, double Ey, double Bz,
                                       double alpha, double ic2, bool &ok)
{
    const double epsx = A::mul(alpha, Ex), epsy = A::mul(alpha, Ey);
    const double bz = A::mul(alpha, Bz);
    const double bb = A::mul(bz, bz);
    Push out;
    if (PUSHER == FETDPIC_VAY) {
        // Sec. II.C(b): u^n = u^{n-1/2} + eps + v^{n-1/2} x beta; u' = u^n + eps;
        // gamma^{n+1/2} from the quartic; u^{n+1/2} = s (u' + (u'.t) t + u' x t), s = 1/(1+t^2)
        const double g0 = gam2<A>(ux, uy, ic2);
        const double vx = A::div(ux, g0), vy = A::div(uy, g0);
        const double unx = (ux + epsx) + A::mul(vy, bz);
        const double uny = (uy + epsy) - A::mul(vx, bz);
        const double upx = unx + epsx, upy = uny + epsy;
        if (A::SOFT) ok = ok && f64_within<120, 64>(upx) && f64_within<120, 64>(upy);
        const double gp = gam2<A>(upx, upy, ic2);
        const double sigma = A::mul(gp, gp) - bb;
        const double gn2 = A::half(sigma + A::root(A::mul(sigma, sigma) + A::four(bb)));
        if (A::SOFT) ok = ok && f64_positive(gn2);
        const double gn = A::root(gn2);
        const double tz = A::div(bz, gn);
        const double s = A::div(1.0, 1.0 + A::mul(tz, tz));
        out.ux = A::mul(s, upx + A::mul(upy, tz));
        out.uy = A::mul(s, upy - A::mul(upx, tz));
        out.g = gn;
        return out;
    }
    // Boris family, Eqs. (Boris.u1-u4)
    const double umx = ux + epsx, umy = uy + epsy;
    if (A::SOFT) ok = ok && f64_within<120, 64>(umx) && f64_within<120, 64>(umy);
    const double gbar = gam2<A>(umx, umy, ic2);              // Eq. (gamma.middle)
    double tz;
    if (PUSHER == FETDPIC_HC) {
        // Sec. II.C(c): gamma_H from sigma = gamma_B^2 - |beta|^2 (u^- . beta = 0 in 2-D TE)
        const double sigma = A::mul(gbar, gbar) - bb;
        const double gh2 = A::half(sigma + A::root(A::mul(sigma, sigma) + A::four(bb)));
        if (A::SOFT) ok = ok && f64_positive(gh2);
        tz = A::div(bz, A::root(gh2));
    } else if (PUSHER == FETDPIC_BORIS_TAN) {
        // (sqrt(bz^2) and bz / |bz| are exact where bz^2 does not underflow)
        const double nb = A::SOFT ? fabs(bz) : sqrt(bb);
        if (A::SOFT) {
            const double t = tan(A::div(nb, gbar));
            tz = is_neg(bz) ? -t : t;
        } else {
            tz = (nb == 0.0) ? 0.0 : (bz / nb) * tan(nb / gbar);
        }
    } else {
        tz = A::div(bz, gbar);
    }
    const double den = 1.0 + A::mul(tz, tz);
    const double sz = A::div(A::twice(tz), den);
    const double uprx = umx + A::mul(umy, tz), upry = umy - A::mul(umx, tz);   // u' = u^- + u^- x t
    const double upx = umx + A::mul(upry, sz), upy = umy - A::mul(uprx, sz);   // u^+ = u^- + u' x s
    out.ux = upx + epsx;
    out.uy = upy + epsy;
    if (A::SOFT) ok = ok && f64_within<120, 64>(out.ux) && f64_within<120, 64>(out.uy);
    out.g = gam2<A>(out.ux, out.uy, ic2);
    return out;
}

// --------------------------------------------------------------- deposit

__device__ __forceinline__ void red_add_u64(unsigned long long *p, long long v)
{
    if (v != 0) atomicAdd(p, (unsigned long long)v);
}

// Fixed-point current of one sub-segment, Eq. (I.assign): for local edge m
// with (a, b) = (m+1, m+2), (Q/dt)(l_a^s l_b^f - l_a^f l_b^s), scaled by
// 2^shift/(Q_ref/dt) and rounded to the nearest integer.
template <class A>
__device__ __forceinline__ void seg_current(const double *ls, const double *lf, double w, long long *v)
{
    // l(m+1), l(m+2) of round m; the values rotate through registers
    double sa = ls[1], sb = ls[2], sc = ls[0], fa = lf[1], fb = lf[2], fc = lf[0];
#pragma unroll 1
    for (int m = 0; m < 3; ++m) {
        const double d = A::mul(sa, fb) - A::mul(fa, sb);
        const long long r = A::round(d * w);
        v[0] = v[1]; v[1] = v[2]; v[2] = r;
        const double s = sa, f = fa;
        sa = sb; sb = sc; sc = s;
        fa = fb; fb = fc; fc = f;
    }
}

// --------------------------------------------------------- particle kernel

// 32 bytes in one 256-bit load (read-only data).
__device__ __forceinline__ void ld_4d(const double *p, double &a, double &b, double &c, double &d)
{
    asm volatile("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(a), "=d"(b), "=d"(c), "=d"(d) : "l"(p));
}
struct Tri64 { double gx[3], gy[3], X[3], Y[3]; };
__device__ __forceinline__ Tri64 load_tri(const Geo64 *g)
{
    const double *d = reinterpret_cast<const double *>(g);
    Tri64 t;
    ld_4d(d, t.gx[0], t.gx[1], t.gx[2], t.gy[0]);
    ld_4d(d + 4, t.gy[1], t.gy[2], t.X[0], t.X[1]);
    ld_4d(d + 8, t.X[2], t.Y[0], t.Y[1], t.Y[2]);
    return t;
}
template <class A>
__device__ __forceinline__ void lambdas(const Tri64 &t, double x, double y, double *l)
{
#pragma unroll
    for (int m = 0; m < 3; ++m) {
        const int an = (m + 1) % 3;
        l[m] = A::mul(t.gx[m], x - t.X[an]) + A::mul(t.gy[m], y - t.Y[an]);
    }
}

// One particle's gather, push, end point and, if it stays in its triangle, its
// current.  ok: false when the integer form met an operand it does not take.
struct One64 {
    double xf, yf, ux, uy;
    long long v[3];
    bool stays, ok;
};

template <class A, int PUSHER>
__device__ __forceinline__ One64 one_particle64(const StepArgs64 &a, const Species *S, int f, double xs, double ys,
                                                double ux, double uy)
{
    One64 o;
    const Tri64 t = load_tri(a.geo + f);
    Rec64 R;
    ld_4d(a.rec[f].se, R.se[0], R.se[1], R.se[2], R.bz);
    o.ok = true;
    if (A::SOFT) {
        // E may be a far wave's tail (it enters linearly), B and the momentum are squared
        o.ok = f64_within<120, 64>(xs) && f64_within<120, 64>(ys) && f64_within<120, 64>(ux) &&
               f64_within<120, 64>(uy) && f64_within<400, 64>(R.se[0]) && f64_within<400, 64>(R.se[1]) &&
               f64_within<400, 64>(R.se[2]);
    }
    double lam[3];
    lambdas<A>(t, xs, ys, lam);
    // gather E^n (Sec. II.B): sum_m s_m e_m (l_a grad l_b - l_b grad l_a)
    double Ex = 0.0, Ey = 0.0;
    {
        double la = lam[1], lb = lam[2], lc = lam[0], xa = t.gx[1], xb = t.gx[2], xc = t.gx[0], ya = t.gy[1],
               yb = t.gy[2], yc = t.gy[0], ea = R.se[0], eb = R.se[1];
        const double ec = R.se[2];
#pragma unroll 1
        for (int m = 0; m < 3; ++m) {
            const double wx = A::mul(la, xb) - A::mul(lb, xa);
            const double wy = A::mul(la, yb) - A::mul(lb, ya);
            Ex = Ex + ea * wx;                                         // on the FP64 pipe in both forms
            Ey = Ey + ea * wy;
            const double l = la, x = xa, y = ya;
            la = lb; lb = lc; lc = l;
            xa = xb; xb = xc; xc = x;
            ya = yb; yb = yc; yc = y;
            ea = eb; eb = ec;
        }
    }
    double Bz = R.bz;
    if (a.ext_on) {
        // applied fields: (amplitude x E weight) E_ext, B weight x B_ext in this triangle
        double we = 1.0, wb = 1.0;
        if (a.extw) { const double2 wv = a.extw[f]; we = wv.x; wb = wv.y; }
        const double sa = a.ext_amp[S->inst] * we;
        Ex = Ex + sa * S->ext_ex;
        Ey = Ey + sa * S->ext_ey;
        Bz = R.bz + wb * S->ext_bz;
        if (A::SOFT) o.ok = o.ok && f64_within<700, 300>(Ex) && f64_within<700, 300>(Ey);
    }
    if (A::SOFT) o.ok = o.ok && f64_within<120, 64>(Bz);
    const Push u = push64<A, PUSHER>(ux, uy, Ex, Ey, Bz, S->alpha, S->ic2, o.ok);
    o.ux = u.ux; o.uy = u.uy;
    if (!A::SOFT) {
        if (!isfinite(u.g) || !isfinite(u.ux) || !isfinite(u.uy)) atomicOr(a.status, (unsigned)ST_NONFINITE);
    }
    const double ig = A::div(1.0, u.g);
    const double dt = S->dt;
    o.xf = xs + A::mul(A::mul(u.ux, ig), dt);                   // Eq. (eq.motion.dis)
    o.yf = ys + A::mul(A::mul(u.uy, ig), dt);
    // the geometry is read again (L1) rather than kept through the push: 24 registers
    double lf[3];
    lambdas<A>(load_tri(a.geo + f), o.xf, o.yf, lf);
    o.stays = !(A::neg(lf[0]) || A::neg(lf[1]) || A::neg(lf[2]));
    seg_current<A>(lam, lf, S->wfix, o.v);
    return o;
}

// The hardware form for a particle the integer form does not take (out of line: rare).
template <int PUSHER>
__device__ __noinline__ One64 one_particle64_hard(const StepArgs64 &a, const Species *S, int f, double xs, double ys,
                                                  double ux, double uy)
{
    return one_particle64<Hard, PUSHER>(a, S, f, xs, ys, ux, uy);
}

// A particle whose path leaves its starting triangle, queued per warp.
struct __align__(16) Walk64 {
    double xs, ys, xf, yf, ux, uy;
    unsigned p;                              // particle slot
    int f;                                   // starting triangle
    int soft, pad;                           // the integer form took its push
};
static_assert(sizeof(Walk64) == 64, "Walk64 layout");
constexpr int RING64 = 64;                   // 31 pending + 32 new fit

// Walk of a queued particle through the triangles it crosses: exit test,
// deposit of each sub-segment, hand-off to the neighbour or specular
// reflection at a PEC wall, and the final particle state.  The integer current
// of a crossed edge is carried to the next sub-segment, which ends on the same
// edge: one atomic, not two.
template <class A>
__device__ __forceinline__ void walk64(const StepArgs64 &a, const Walk64 &it)
{
    const unsigned p = it.p;
    const Species *S = a.sp + a.chunk_sp[p >> 5];
    // walk record slot: species storage offset + load index (unmoved by a later sort)
    const long long rp = a.rec_cap > 0 ? S->off + a.id[p] : 0;
    const int inst = S->inst;
    const double wfix = S->wfix;
    double xs = it.xs, ys = it.ys, xf = it.xf, yf = it.yf, ux = it.ux, uy = it.uy, tin = 0.0;
    double lin[3];
    int f = it.f, min = -1, ncross = 0;
    bool first = true, reflected = false;
    long long carry = 0;                     // current on the entry edge, not yet deposited
    for (;;) {
        const Tri64 t = load_tri(a.geo + f);
        const Topo *tp = a.topo + f;
        const int ew[3] = {__ldg(&tp->ew[0]), __ldg(&tp->ew[1]), __ldg(&tp->ew[2])};
        double ls[3], lf[3];
        lambdas<A>(t, xs, ys, ls);
        lambdas<A>(t, xf, yf, lf);
        if (first) { lin[0] = ls[0]; lin[1] = ls[1]; lin[2] = ls[2]; first = false; }
        // candidate exits in ascending order; a warp runs as many rounds as its worst lane has
        unsigned cand = (A::neg(lf[0]) ? 1u : 0u) | (A::neg(lf[1]) ? 2u : 0u) | (A::neg(lf[2]) ? 4u : 0u);
        if (min >= 0) cand &= ~(1u << min);
        int best = -1;
        double tb = 0.0;
        while (cand) {
            const int k = __ffs(cand) - 1;
            cand &= cand - 1u;
            const double s = k == 0 ? ls[0] : k == 1 ? ls[1] : ls[2];
            const double den = s - (k == 0 ? lf[0] : k == 1 ? lf[1] : lf[2]);
            double tk = den > 0.0 ? A::div(s, den) : tin;
            if (tk < tin) tk = tin;
            if (best < 0 || tk < tb) { best = k; tb = tk; }
        }
        double lout[3];
        if (best < 0) {
            lout[0] = lf[0]; lout[1] = lf[1]; lout[2] = lf[2];
        } else {
#pragma unroll
            for (int k = 0; k < 3; ++k) lout[k] = k == best ? 0.0 : ls[k] + A::mul(tb, lf[k] - ls[k]);
        }
        long long v[3];
        seg_current<A>(lin, lout, wfix, v);
        const long long cin = carry;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            long long s = (ew[m] & 1) ? -v[m] : v[m];
            if (m == min) s += cin;
            if (m == best) carry = s;
            else red_add_u64(a.ifix + (ew[m] >> 1), s);
        }
        if (best < 0) break;
        const int eg = (best == 0 ? ew[0] : best == 1 ? ew[1] : ew[2]) >> 1;
        if (ncross >= a.max_cross) {
            red_add_u64(a.ifix + eg, carry);
            xf = xs + A::mul(tb, xf - xs); yf = ys + A::mul(tb, yf - ys);
            atomicOr(a.status, (unsigned)ST_WALK);
            break;
        }
        const int nbw = __ldg(&tp->nb[best]);
        if (a.rec_cap > ncross) a.wrec[rp * a.rec_cap + ncross] = nbw < 0 ? -(eg - a.edge_off[inst] + 1) : eg - a.edge_off[inst];
        ++ncross;
        if (nbw < 0) {
            const double xw = xs + A::mul(tb, xf - xs), yw = ys + A::mul(tb, yf - ys);
            const double gxb = best == 0 ? t.gx[0] : best == 1 ? t.gx[1] : t.gx[2];
            const double gyb = best == 0 ? t.gy[0] : best == 1 ? t.gy[1] : t.gy[2];
            const double gg = gxb * gxb + gyb * gyb;
            const double pr = ((xf - xw) * gxb + (yf - yw) * gyb) / gg;
            xf = xf - 2.0 * pr * gxb;
            yf = yf - 2.0 * pr * gyb;
            const double pu = (ux * gxb + uy * gyb) / gg;
            ux = ux - 2.0 * pu * gxb;
            uy = uy - 2.0 * pu * gyb;
            xs = xw; ys = yw;
            tin = 0.0;
            min = best;
            lin[0] = lout[0]; lin[1] = lout[1]; lin[2] = lout[2];
            reflected = true;
        } else {
            // hand-off: the neighbour's node m2+1 is our node best+2, its m2+2 our best+1
            const int m2 = nbw & 3;
            const double la = best == 0 ? lout[2] : best == 1 ? lout[0] : lout[1];
            const double lb = best == 0 ? lout[1] : best == 1 ? lout[2] : lout[0];
            lin[0] = m2 == 0 ? 0.0 : (m2 == 2 ? la : lb);
            lin[1] = m2 == 1 ? 0.0 : (m2 == 0 ? la : lb);
            lin[2] = m2 == 2 ? 0.0 : (m2 == 1 ? la : lb);
            if (a.tshift) {
                // periodic wall: the rest of the segment continues from the other copy
                const int sc = a.tshift[3 * f + best];
                if (sc != 0) {
                    const double2 T = a.period[inst];
                    xs = xs + sc * T.x; ys = ys + sc * T.y;
                    xf = xf + sc * T.x; yf = yf + sc * T.y;
                }
            }
            f = nbw >> 2;
            min = m2;
            tin = tb;
        }
    }
    a.x[p] = xf; a.y[p] = yf;
    if (reflected) { a.ux[p] = ux; a.uy[p] = uy; }
    a.cell[p] = f;
    if (a.rec_cap > 0) a.rec_cnt[rp] = ncross;
}

__device__ __noinline__ void walk64_hard(const StepArgs64 &a, const Walk64 *it) { walk64<Hard>(a, *it); }
__device__ __noinline__ void walk64_soft(const StepArgs64 &a, const Walk64 *it) { walk64<Soft>(a, *it); }

__device__ __forceinline__ void walk64_any(const StepArgs64 &a, const Walk64 *it)
{
    if (it->soft) walk64_soft(a, it);
    else walk64_hard(a, it);
}

// Persistent warps, each over a contiguous range of 32-particle chunks (a chunk
// never straddles species), one particle per lane.  The current of the particles that
// stay in their triangle is summed over runs of equal triangle (particles are
// sorted by triangle) by shuffles, one lane per run issuing the three 64-bit
// integer additions; walkers go to the warp's ring in shared memory and are
// walked 32 at a time (a divergent walk per chunk ran the FP64 instructions of
// every chunk's two or three walkers on a whole warp's time).  Integer
// addition is associative, so the result does not depend on the order of
// particles or atomics: deposits are deterministic.
//
// Bound by the FP64 pipe (59 % busy with the additions and nine products) and
// the integer pipe (51 %) together.  128 registers and 16 warps per SM: at 80
// registers (24 warps) the spills cost what the warps bring.  2.05 M particles,
// Higuera-Cary: 1052 -> 390 us a launch; 327,680, Vay: 203 -> 76 us.
template <int PUSHER>
__global__ void __launch_bounds__(256, 2) k_particles64(StepArgs64 a)
{
    pdl_begin();
    extern __shared__ Walk64 rings[];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Walk64 *q = rings + warp * RING64;
    unsigned qhead = 0, qtail = 0;                        // warp-uniform ring positions
    const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
    const long long wid = (long long)blockIdx.x * (blockDim.x >> 5) + warp;
    long long c = wid * a.nchunks / nwarps;
    const long long cend = (wid + 1) * a.nchunks / nwarps;
    for (; c < cend; ++c) {
        const long long p = c * 32 + lane;
        const int f = a.cell[p];
        const double xs = a.x[p], ys = a.y[p], ux = a.ux[p], uy = a.uy[p];
        const Species *S = a.sp + a.chunk_sp[c];
        const bool live = f >= 0;
        One64 o;
        o.ok = false;
        if (a.soft && live) o = one_particle64<Soft, PUSHER>(a, S, f, xs, ys, ux, uy);
        const bool soft = o.ok;
        if (live && !soft) o = one_particle64_hard<PUSHER>(a, S, f, xs, ys, ux, uy);
        const bool stays = live && o.stays, walks = live && !o.stays;
        {
            const unsigned wm = __ballot_sync(full, walks);
            if (walks) {
                Walk64 &w = q[(qtail + __popc(wm & ((1u << lane) - 1u))) & (RING64 - 1)];
                w.xs = xs; w.ys = ys; w.xf = o.xf; w.yf = o.yf; w.ux = o.ux; w.uy = o.uy;
                w.p = (unsigned)p; w.f = f; w.soft = soft;
            }
            qtail += __popc(wm);
        }
        // segmented sum over runs of equal triangle; a level runs only when some run spans it
        {
            const int key = stays ? f : -1;
            long long v[3];
#pragma unroll
            for (int m = 0; m < 3; ++m) v[m] = stays ? o.v[m] : 0;
            const int kn = __shfl_down_sync(full, key, 1);
            const unsigned tails = __ballot_sync(full, (lane == 31) || (kn != key));
            const int seg_end = lane + __ffs(tails >> lane) - 1;
            const int kp = __shfl_up_sync(full, key, 1);
            const bool head = (lane == 0) || (kp != key);
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                if (!__any_sync(full, seg_end - lane >= off)) break;
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    const long long ov = __shfl_down_sync(full, v[m], off);
                    if (lane + off <= seg_end) v[m] += ov;
                }
            }
            if (head && key >= 0) {
                const int4 ew = __ldg(reinterpret_cast<const int4 *>(a.topo + f));       // edge words, neighbour 0
                red_add_u64(a.ifix + (ew.x >> 1), (ew.x & 1) ? -v[0] : v[0]);
                red_add_u64(a.ifix + (ew.y >> 1), (ew.y & 1) ? -v[1] : v[1]);
                red_add_u64(a.ifix + (ew.z >> 1), (ew.z & 1) ? -v[2] : v[2]);
            }
        }
        if (live) { a.ux[p] = o.ux; a.uy[p] = o.uy; }
        if (stays) {
            a.x[p] = o.xf; a.y[p] = o.yf;
            if (a.rec_cap > 0) a.rec_cnt[S->off + a.id[p]] = 0;
        }
        if (qtail - qhead >= 32) {
            __syncwarp();
            walk64_any(a, q + ((qhead + lane) & (RING64 - 1)));
            qhead += 32;
            __syncwarp();
        }
    }
    if (qtail > qhead) {
        __syncwarp();
        if ((unsigned)lane < qtail - qhead) walk64_any(a, q + ((qhead + lane) & (RING64 - 1)));
    }
}

template <int PUSHER>
static void launch_p64(cudaStream_t st, const StepArgs64 &a)
{
    // each thread keeps its own: contexts of different block sizes may step on several at once
    static thread_local int per_sm = 0, sms = 0, dev = -1, blk = 0;
    const size_t ring = (size_t)(a.block / 32) * RING64 * sizeof(Walk64);
    int d = 0;
    cudaGetDevice(&d);
    if (d != dev || blk != a.block) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_particles64<PUSHER>, a.block, ring);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d);
        dev = d; blk = a.block;
        if (per_sm < 1) per_sm = 1;
    }
    // few chunks go to as many SMs as there are, in blocks of fewer warps (4,000 particles: 125 chunks
    // in 16 blocks of 8 warps left 136 SMs idle)
    long long nw = (a.nchunks + sms - 1) / sms;
    if (nw > a.block / 32) nw = a.block / 32;
    const long long need = (a.nchunks + nw - 1) / nw;
    const long long grid = need < (long long)per_sm * sms ? need : (long long)per_sm * sms;
    launch_ks(a.pdl, k_particles64<PUSHER>, dim3((unsigned)grid), dim3((unsigned)nw * 32),
              (size_t)nw * RING64 * sizeof(Walk64), st, a);
}

void launch_particles64(cudaStream_t st, int pusher, const StepArgs64 &a)
{
    if (a.nchunks <= 0) return;
    switch (pusher) {
    case FETDPIC_BORIS: launch_p64<FETDPIC_BORIS>(st, a); break;
    case FETDPIC_BORIS_TAN: launch_p64<FETDPIC_BORIS_TAN>(st, a); break;
    case FETDPIC_VAY: launch_p64<FETDPIC_VAY>(st, a); break;
    default: launch_p64<FETDPIC_HC>(st, a); break;
    }
}

}  // namespace fetdpic
