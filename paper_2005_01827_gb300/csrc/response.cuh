// response.cuh -- A_lm, phi_lm and the TDI A/E/T transfer of Eqs. (5)-(10) of Katz et al.
// (2020) at one frequency, from constants computed once per walker and mode (source.cu).
//
// The constellation of model.cuh is a circular orbit with three spacecraft at fixed phases,
// so every scalar product of a fixed vector with an arm or a sum of spacecraft positions is
// a constant plus harmonics of the orbital angle a: o0 + o1 cos 2a + o2 sin 2a + o3 cos a +
// o4 sin a.  The arms are exactly one arm length L long and n_02 = n_01 + n_12; with the
// polarisation basis u, w of the wave (u in the ecliptic plane), n.e+.n = (u.n)^2 - (w.n)^2
// and n.ex.n = 2 (u.n)(w.n).  With x = pi f L, g = 1 -+ k.n and sin(x g) by angle addition,
// x sinc(x g) = sin(x g) / g, and the equal-arm delay e^{-2ix} factors out of the Michelson
// combinations: for an arm with link factors s1 (a -> c), s2 (c -> a) and common factor E,
// y_ca + D y_ac = e^{-ix} E ((s1 + s2) cos x + i (s2 - s1) sin x), and 1 - D^2 =
// 2i sin 2x e^{-2ix}.
#pragma once
#include "fixed.cuh"
#include "model.cuh"

namespace lisa {

constexpr double kInvCbrtPi = 0.68278406325529568;  // pi^(-1/3)

struct WalkerConst {
    double k128, ps2, ps3;     // inspiral phase
    double phj, c1, c2;        // late phase phj + c1 x - c2 / x
    double dphpk, tc, m2pi;    // slope at the peak, t_coal, M / 2 pi
    double al2, al3, ixrd;     // amplitude
    double kn[2][5], kq[2][5], wn[2][5];  // k.n, k.(q_a + q_c) / L, w.n of arms 01 and 12
    double un[2][3];           // u.n (no cos a, sin a terms)
    double dx, dy;             // delay phase f (dx cos a + dy sin a)
};

struct ModeConst {
    double are, aim, bre, bim;  // transfer of an arm: a ((u.n)^2 - (w.n)^2) + b (u.n)(w.n)
    double xf, v0, x160, s6;    // x / f; (pi x)^(1/3) and x^(1/6) at the first knot; step
    double amp, off, half_m;    // amplitude factor, phase offset, m / 2
    int power, pad;             // power of v in the mode's amplitude ratio
};
static_assert(sizeof(WalkerConst) % 8 == 0 && sizeof(WalkerConst) / 8 <= 96, "copied by a block");
static_assert(sizeof(ModeConst) % 8 == 0 && sizeof(ModeConst) / 8 <= 32, "copied by a warp");

__device__ __forceinline__ int amp_power(const Mode &md) {
    switch (mode_index(md.l, md.m)) {
        case 1: case 3: return 1;
        case 2: case 4: return 2;
        case 5: return 3;
        default: return 0;
    }
}

// sin(x g) / g for g = 1 -+ k.n near an arm direction (g < 1e-3), where the angle addition
// of the caller would lose digits; x in the limit g = 0
static __device__ __noinline__ double near_arm_link(double x, double g) {
    return g == 0.0 ? x : sin(x * g) / g;
}

// cos and sin of 2 pi turns on the integer units (fixed.cuh), with an absolute error of about
// 2e-16 beside the rounding of `turns` itself: like the rounding of a cosine near 1, but a sine or
// cosine near 0 has fewer correct bits than sincos() gives.  For unit phasors and angles, not
// where a small sine counts.  tab: the phasor table of kFxTab entries
__device__ __forceinline__ void phasor_turns(double turns, const FxTab *__restrict__ tab, double &sn, double &cs) {
    const double fr = turns - rint(turns);
    const i64 v = to_fixed(fr, 62);  // |fr| <= 1/2
    const unsigned long long ph = (unsigned long long)v << 2;
    const int4 e = __ldg(reinterpret_cast<const int4 *>(tab + fx_cell(ph)));
    i64 zr, zi;
    fx_rotate(ph, FxTab{Bal{e.x, e.y}, Bal{e.z, e.w}}, zr, zi);
    cs = (double)zr * 0x1p-60;
    sn = (double)zi * 0x1p-60;
}

// cos and sin of x radians, |x| < 1e9, likewise: x is reduced by the split of 2 pi, without the
// slow path that sincos() takes beyond 1e5
__device__ __forceinline__ void phasor_radians(double x, const FxTab *__restrict__ tab, double &sn, double &cs) {
    const double k = rint(x * kInvTwoPi);
    double r = fma(-k, kTwoPiHi, x);
    r = fma(-k, kTwoPiMid, r);
    r = fma(-k, kTwoPiLo, r);
    phasor_turns(r * kInvTwoPi, tab, sn, cs);
}

// sin and cos of |x| <= 0.35 by their Taylor series (the next terms are below 2e-17 of them): 15
// operations against about 25 of sincos()
__device__ __forceinline__ void sincos_small(double x, double &sn, double &cs) {
    const double y = x * x;
    double a = fma(y, 1.0 / 6227020800.0, -1.0 / 39916800.0);
    a = fma(y, a, 1.0 / 362880.0);
    a = fma(y, a, -1.0 / 5040.0);
    a = fma(y, a, 1.0 / 120.0);
    a = fma(y, a, -1.0 / 6.0);
    sn = fma(x * y, a, x);
    double b = fma(y, -1.0 / 87178291200.0, 1.0 / 479001600.0);
    b = fma(y, b, -1.0 / 3628800.0);
    b = fma(y, b, 1.0 / 40320.0);
    b = fma(y, b, -1.0 / 720.0);
    b = fma(y, b, 1.0 / 24.0);
    b = fma(y, b, -0.5);
    cs = fma(y, b, 1.0);
}

// What the modes of equal m share at one frequency: (m / 2) phi_22(2 f / m) with the
// constellation-centre delay, the amplitude up to the mode's factor, and the response up to
// the mode's polarisation weights.  Their modes add about 85 operations each to about 340.
struct ModeBase {
    double amp, v, phase;
    double P[3], C[3];     // (u.n)^2 - (w.n)^2 and (u.n)(w.n) of the arms
    cplx gu[3], gv[3];     // propagation phase times (s1 + s2) cos x +- i (s2 - s1) sin x
    cplx fac;              // 2 sin 2x e^{-4ix}
};

// v = (pi x)^(1/3) and x16 = x^(1/6) of the mapped frequency x = xf f; m: any mode of this m
__device__ __forceinline__ void mode_base(const WalkerConst &w, const ModeConst &m,
                                          const FxTab *__restrict__ tab, double f, double v, double x16,
                                          ModeBase &o) {
    const double x = m.xf * f;
    const double r = x * w.ixrd, r2 = r * r;
    const double v2 = v * v;
    // orbital angle from t_lm(f); its phase slope needs 1 / v
    const double iv = 1.0 / v;
    const double iv2 = iv * iv;
    const double ix = kPi * (iv2 * iv);
    double p, dp;
    if (x <= kXJoin) {
        const double b = iv * (iv2 + w.ps2);  // iv2 (iv2 iv + ps2 iv + ps3)
        p = -3.0 * w.k128 * (iv2 * (b + w.ps3));
        dp = w.k128 * ix * (iv2 * (iv * fma(3.0, w.ps2, 5.0 * iv2) + 2.0 * w.ps3));
    } else {
        p = fma(w.c1, x, w.phj) - w.c2 * ix;
        dp = fma(w.c2 * ix, ix, w.c1);
    }
    const double t = fma(-w.m2pi, dp - w.dphpk, w.tc);
    double sa, ca;
    phasor_turns((1.0 / kYearS) * t, tab, sa, ca);
    const double s2a = 2.0 * sa * ca, c2a = fma(-2.0 * sa, sa, 1.0);
    o.phase = fma(m.half_m, fma(-w.dphpk, x, p), m.off) + f * fma(w.dx, ca, w.dy * sa);
    auto harm5 = [&](const double *o) {
        return fma(o[4], sa, fma(o[3], ca, fma(o[2], s2a, fma(o[1], c2a, o[0]))));
    };
    auto harm3 = [&](const double *o) { return fma(o[2], s2a, fma(o[1], c2a, o[0])); };
    double kn[3], un[3], wn[3];
    kn[0] = harm5(w.kn[0]);
    kn[2] = harm5(w.kn[1]);
    kn[1] = kn[0] + kn[2];
    un[0] = harm3(w.un[0]);
    un[2] = harm3(w.un[1]);
    un[1] = un[0] + un[2];
    wn[0] = harm5(w.wn[0]);
    wn[2] = harm5(w.wn[1]);
    wn[1] = wn[0] + wn[2];
    const double kq0 = harm5(w.kq[0]), kq2 = harm5(w.kq[1]);

    const double xl = (kPi * (kArmM / kClight)) * f;  // pi f L
    // |k.n| <= 1, so every angle below but the propagation phases is at most x
    const bool small = xl <= 0.35;  // f < 13 mHz
    auto sine = [&](double a, double &sn, double &cs) {
        if (small)
            sincos_small(a, sn, cs);
        else
            sincos(a, &sn, &cs);
    };
    double sx, cx;
    sine(xl, sx, cx);
    // e^{-i x k.(q_a + q_c) / L}; the middle arm's is the conjugate product of the others
    cplx g[3];
    {
        double s0, c0, s2, c2;
        const double xt = xl * (1.0 / kTwoPi);
        phasor_turns(xt * kq0, tab, s0, c0);
        phasor_turns(xt * kq2, tab, s2, c2);
        g[0] = {c0, -s0};
        g[2] = {c2, -s2};
        g[1] = {c0 * c2 - s0 * s2, c0 * s2 + s0 * c2};
    }
    double sn[3], cn[3];
    sine(xl * kn[0], sn[0], cn[0]);
    sine(xl * kn[2], sn[2], cn[2]);
    sn[1] = sn[0] * cn[2] + cn[0] * sn[2];
    cn[1] = cn[0] * cn[2] - sn[0] * sn[2];

    // one division: the three 1 / (1 - (k.n)^2) and the amplitude's denominator
    double den[3], g1[3], g2[3];
#pragma unroll
    for (int e = 0; e < 3; e++) {
        g1[e] = 1.0 - kn[e];
        g2[e] = 1.0 + kn[e];
        const double q = g1[e] * g2[e];
        den[e] = fmin(g1[e], g2[e]) >= 1e-3 ? q : 1.0;
    }
    const double da = x16 * fma(r2 * r2, r2, 1.0);
    const double d01 = den[0] * den[1], d23 = den[2] * da;
    const double inv = 1.0 / (d01 * d23);
    const double i01 = inv * d23, i23 = inv * d01;
    const double iden[3] = {i01 * den[1], i01 * den[0], i23 * da};
    o.amp = ix * exp(v2 * fma(w.al3, v, w.al2)) * (i23 * den[2]);
    o.v = v;

#pragma unroll
    for (int e = 0; e < 3; e++) {
        o.P[e] = fma(un[e], un[e], -wn[e] * wn[e]);
        o.C[e] = un[e] * wn[e];
        const double a = sx * cn[e], c = cx * sn[e];
        double s1 = (a - c) * (g2[e] * iden[e]), s2 = (a + c) * (g1[e] * iden[e]);
        if (den[e] == 1.0) {  // within 1e-3 of the arm's direction (or k.n = 0: the same value)
            if (g1[e] < 1e-3) {
                s1 = near_arm_link(xl, g1[e]);
                s2 = (a + c) / g2[e];
            } else if (g2[e] < 1e-3) {
                s1 = (a - c) / g1[e];
                s2 = near_arm_link(xl, g2[e]);
            }
        }
        const double s = (s1 + s2) * cx, dd = (s2 - s1) * sx;
        const cplx gs = {g[e].re * s, g[e].im * s};
        o.gu[e] = {fma(-g[e].im, dd, gs.re), fma(g[e].re, dd, gs.im)};
        o.gv[e] = {fma(g[e].im, dd, gs.re), fma(-g[e].re, dd, gs.im)};
    }
    const double c2x = fma(-2.0 * sx, sx, 1.0), s2x = 2.0 * sx * cx;
    o.fac = {2.0 * s2x * fma(-2.0 * s2x, s2x, 1.0), -4.0 * s2x * s2x * c2x};
}

// amplitude and A, E, T transfer of one mode
__device__ __forceinline__ void mode_channels(const ModeBase &o, const ModeConst &m, double &amp,
                                              cplx T[3]) {
    amp = m.amp * o.amp;
    if (m.power & 1) amp *= o.v;
    if (m.power & 2) amp *= o.v * o.v;
    cplx U[3], V[3];
#pragma unroll
    for (int e = 0; e < 3; e++) {
        const cplx F = {fma(m.are, o.P[e], m.bre * o.C[e]), fma(m.aim, o.P[e], m.bim * o.C[e])};
        U[e] = cmul(F, o.gu[e]);
        V[e] = cmul(F, o.gv[e]);
    }
    // X = U_02 - U_01, Y = V_01 - U_12, Z = V_12 - V_02, times 2 sin 2x e^{-4ix}
    const cplx X = csub(U[1], U[0]), Y = csub(V[0], U[2]), Z = csub(V[2], V[1]);
    const double k2 = 0.70710678118654752440, k6 = 0.40824829046386301637, k3 = 0.57735026918962576451;
    T[0] = cmul(o.fac, cplx{(Z.re - X.re) * k2, (Z.im - X.im) * k2});
    T[1] = cmul(o.fac, cplx{(fma(-2.0, Y.re, X.re) + Z.re) * k6, (fma(-2.0, Y.im, X.im) + Z.im) * k6});
    T[2] = cmul(o.fac, cplx{(X.re + Y.re + Z.re) * k3, (X.im + Y.im + Z.im) * k3});
}

}  // namespace lisa
