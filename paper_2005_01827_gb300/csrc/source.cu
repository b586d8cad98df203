// source.cu -- everything that a walker's knots share, computed once per walker (Katz et al.
// 2020, Sec. II): the waveform constants, the peak of f^2 A_22, the band of every mode
// (the cut where t_lm(f) < 0 and the ringdown cut) with its integer dense-bin range, and
// the coefficients of the response in the constellation's orbital harmonics.
//
// One warp per walker.  What bounds it is the latency of FP64 operations one after another (about
// 40 clocks each), so the chain is kept short:
//  * both roots (the peak, and the frequency where the signal starts, which is one mapped
//    frequency x = 2 M f / m for all modes) are bracketed in FP32, 31 points a round, one per
//    lane, and finished by Newton steps in FP64 inside the whole range (quadratic: the step
//    that moves x by less than 1e-8 leaves 1e-16);
//  * what is needed at several places or angles is evaluated in one pass, a lane for each: the
//    ends of the peak's range, phase and slope at the band's ends and the peak, sines and cosines.
// One walker, one mode: 80 -> 29 us (98 -> 38 with cold caches; before, 31 points twice and up to
// six Newton steps in FP64 for each root, and all else one after another).
#include "fixed.cuh"
#include "kernels.h"
#include "model.cuh"
#include "response.cuh"

namespace lisa {

static_assert(sizeof(FxTab) * kFxTab == kFxTabBytes, "table size");

// f_j = f0 + j df, rounded as a separate product and sum (no fused multiply-add) so
// that band edges and knot-to-bin boundaries are decided exactly as written.
__device__ __forceinline__ double bin_freq(double f0, double df, int j) {
    return __dadd_rn(f0, __dmul_rn((double)j, df));
}

// index in [0, 31] of the interval that five bisections on the sign (true: the root lies
// above) of 31 interior points would end in; bit i of `above` belongs to point i, i = 1..31
__device__ __forceinline__ int bisect32(unsigned above) {
    int pos = 0;
    for (int step = 16; step > 0; step >>= 1)
        if ((above >> (pos + step)) & 1u) pos += step;
    return pos;
}

// the interval among 31 interior points of [lo, hi], equally spaced in the logarithm, that holds
// the root of f (above(x): the root lies above x), `rounds` times
template <class F>
__device__ __forceinline__ float bracket32(float lo, float hi, int rounds, int lane, F above) {
    float l0 = log2f(lo), st = log2f(hi) - l0;
    for (int r = 0; r < rounds; r++) {
        st *= 1.0f / 32.0f;
        const int p = bisect32(__ballot_sync(0xffffffffu, above(exp2f(fmaf(st, (float)lane, l0)))));
        l0 = fmaf(st, (float)p, l0);
    }
    return exp2f(l0 + 0.5f * st);
}

// peak of f^2 A_22 (t_coal is reached there, Sec. II): the zero of its log-derivative over
// [x_RD / 4, 2 x_RD], or the end of that range that it lies beyond
__device__ double find_peak_warp(const Source &s, double ixrd, int lane) {
    double lo = 0.25 * s.xrd, hi = 2.0 * s.xrd;
    const float al2 = (float)s.al2, al3 = (float)s.al3;
    // in units of x_RD
    const float v3 = (float)(kPi * s.xrd);
    auto equation = [&](float r) {
        const float v = cbrtf(v3 * r), r2 = r * r, r6 = r2 * r2 * r2;
        return 5.0f / 6.0f + v * v * fmaf(al3, v, (2.0f / 3.0f) * al2) - 6.0f * r6 / (1.0f + r6);
    };
    // the ends in FP32, and in FP64 where those could have the wrong sign
    if (!(equation(0.25f) > 1e-3f && equation(2.0f) < -1e-3f)) {
        const double ge = peak_equation(s, lane == 0 ? lo : hi);
        const double gl = __shfl_sync(0xffffffffu, ge, 0), gh = __shfl_sync(0xffffffffu, ge, 1);
        if (gl <= 0.0) return lo;
        if (gh >= 0.0) return hi;
    }
    double x = s.xrd * (double)bracket32(0.25f, 2.0f, 4, lane, [&](float r) { return equation(r) > 0.0f; });
    for (int it = 0; it < 100; it++) {
        const double v = cbrt(kPi * x), r = x * ixrd, r2 = r * r, r6 = r2 * r2 * r2;
        const double q2 = s.al2 * v * v, q3 = s.al3 * v * v * v, den = 1.0 / (1.0 + r6);
        const double g = 5.0 / 6.0 + (2.0 / 3.0) * q2 + q3 - 6.0 * r6 * den;
        const double gx = (4.0 / 9.0) * q2 + q3 - 36.0 * r6 * den * den;  // x dg/dx
        if (g > 0.0)
            lo = fmax(lo, x);
        else
            hi = fmin(hi, x);
        double nx = fma(-x, g / gx, x);
        if (!(nx >= lo && nx <= hi)) nx = 0.5 * (lo + hi);
        const double dx = fabs(nx - x);
        x = nx;
        if (dx <= 1e-8 * x) break;
    }
    return x;
}

// phase and slope of the (2,2) mode before its alignment, and the slope's derivative
__device__ __forceinline__ PhaseSet raw_set(const Source &s, double x) {
    PhaseSet r;
    if (x <= kXJoin) {
        r = inspiral_phase(s, x);
    } else {
        const double ix = 1.0 / x;
        r.p = s.phj + s.c1 * (x - kXJoin) - s.c2 * (ix - 1.0 / kXJoin);
        r.dp = s.c1 + s.c2 * (ix * ix);
        r.d2p = -2.0 * s.c2 * (ix * ix * ix);
    }
    return r;
}

// mapped frequency where t_22 = 0, inside [xa, xb] with t(xa) < 0 <= t(xb): t rises with x
__device__ double find_start_warp(const Source &s, double iM, double xa, double xb, int lane) {
    double lo = xa, hi = xb;
    const double target = s.tc * (kTwoPi * iM) + s.dphpk;  // the slope where t = 0
    const float want = (float)target, k = (float)s.k128, ps2 = (float)s.ps2, ps3 = (float)s.ps3;
    const float c1 = (float)s.c1, c2 = (float)s.c2;
    double x = (double)bracket32((float)xa, (float)xb, 4, lane, [&](float y) {
        const float iv = 1.0f / cbrtf((float)kPi * y), iv2 = iv * iv;
        const float dp = y <= (float)kXJoin
                             ? k / y * iv2 * fmaf(iv, fmaf(5.0f, iv2, 3.0f * ps2), 2.0f * ps3)
                             : c1 + c2 / (y * y);
        return dp > want;
    });
    x = fmin(hi, fmax(lo, x));
    for (int it = 0; it < 100; it++) {
        const PhaseSet r = raw_set(s, x);
        const double t = target - r.dp;  // 2 pi t / M
        if (t < 0.0)
            lo = fmax(lo, x);
        else
            hi = fmin(hi, x);
        double nx = x + t / r.d2p;
        if (!(nx >= lo && nx <= hi)) nx = 0.5 * (lo + hi);
        const double dx = fabs(nx - x);
        x = nx;
        if (dx <= 1e-8 * x) break;
    }
    return x;
}

// A vector's component along a combination of spacecraft positions, in units of the arm:
// v . sum_i g_i q_i / L as {1, cos 2a, sin 2a, cos a, sin a} coefficients, with
// cb = sum g_i cos b_i and sb = sum g_i sin b_i (b_i = 2 pi i / 3), a the orbital angle
__device__ __forceinline__ void harmonics(const double v[3], double cb, double sb, double o[5]) {
    constexpr double p = 0.14433756729740644113;  // 1 / (4 sqrt 3)
    o[0] = -3.0 * p * (v[0] * cb + v[1] * sb);
    o[1] = p * (v[0] * cb - v[1] * sb);
    o[2] = p * (v[0] * sb + v[1] * cb);
    o[3] = -0.5 * v[2] * cb;
    o[4] = -0.5 * v[2] * sb;
}

// x / (M f) of a mode's mapped frequency
__device__ __forceinline__ double md_scale(const Mode &md) {
    return md.m == 1 ? 2.0 : md.m == 2 ? 1.0 : md.m == 3 ? 2.0 / 3.0 : 0.5;
}

// One block more than the walkers need writes the phasor table of the fixed-point kernels.
__global__ void __launch_bounds__(128) source_kernel(StageDims d, StageBufs b) {
    if (blockIdx.x == gridDim.x - 1) {
        FxTab *tab = const_cast<FxTab *>(b.fxtab);
        for (int k = threadIdx.x; tab && k < kFxTab; k += blockDim.x) {
            double sn, cs;
            sincospi((double)k / (kFxTab / 2), &sn, &cs);
            tab[k] = FxTab{bal(to_fixed(cs, 62)), bal(to_fixed(sn, 62))};
        }
        return;
    }
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= d.B) return;
    Source src;
    const bool ok = make_source_core(b.params + (size_t)w * kNPar, d.t0, src);
    const double fmn = d.f0, fmx = bin_freq(d.f0, d.df, d.N - 1);
    // lanes 0 .. L-1: one mode each
    const bool mode = lane < d.L;
    Mode md = {2, 2};  // of lane % 8
#pragma unroll
    for (int i = 0; i < kMaxModes; i++)
        if (i == (lane & 7) && i < d.L) md = {d.ml[i], d.mm[i]};
    bool act = false, whole = false;
    double lo = 0.0, hi = 0.0, ixrd = 0.0, iM = 0.0, xf = 0.0;  // xf: x / f, this lane's mode
    if (ok) {
        ixrd = 1.0 / src.xrd;
        iM = 1.0 / src.M;
        xf = src.M * md_scale(md);
        const double xpk = find_peak_warp(src, ixrd, lane);
        const double fcut = 0.5 * md.m * kXCut * iM;
        hi = fmx < fcut ? fmx : fcut;
        // phase and slope at the first bin (lanes 0 .. 7), at the modes' ends and at the peak
        const PhaseSet at =
            raw_set(src, lane < 8 ? xf * fmn : lane < 16 ? xf * hi : xpk);
        src.xpk = xpk;
        src.phpk = __shfl_sync(0xffffffffu, at.p, 16);
        src.dphpk = __shfl_sync(0xffffffffu, at.dp, 16);
        const double t = src.tc - src.m2pi * (at.dp - src.dphpk);  // mode_time
        const double tend = __shfl_sync(0xffffffffu, t, (lane & 7) + 8);
        act = mode && hi > fmn * (1.0 + 1e-12);
        if (act) {
            whole = t >= 0.0;
            if (whole)
                lo = fmn;
            else if (tend < 0.0)
                act = false;  // the mode ends before the observation starts
        }
    }
    // the modes that start inside the observation share one mapped starting frequency
    const bool inside = act && !whole;
    if (__any_sync(0xffffffffu, inside)) {
        double xa = inside ? xf * fmn : INFINITY, xb = inside ? xf * hi : 0.0;
        for (int o = 16; o > 0; o >>= 1) {
            xa = fmin(xa, __shfl_xor_sync(0xffffffffu, xa, o));
            xb = fmax(xb, __shfl_xor_sync(0xffffffffu, xb, o));
        }
        const double x0 = find_start_warp(src, iM, xa, xb, lane);
        if (inside) lo = fmin(hi, fmax(fmn, 0.5 * md.m * x0 * iM));
    }
    int jl = 0, jh = -1;
    if (act && !(hi > lo * (1.0 + 1e-12))) act = false;
    if (act) {
        const double gl = ceil((lo - d.f0) / d.df - 1e-9);
        const double gh = floor((hi - d.f0) / d.df + 1e-9);
        jl = gl < 0.0 ? 0 : (int)gl;
        jh = gh > (double)(d.N - 1) ? d.N - 1 : (int)gh;
        if (jl > jh) act = false;
    }
    if (mode) {
        const size_t wm = (size_t)w * d.L + lane;
        int *bd = b.band + wm * 3;
        bd[0] = act ? 1 : 0;
        bd[1] = act ? jl : 0;
        bd[2] = act ? jh : -1;
        b.fedge[wm * 2] = lo;
        b.fedge[wm * 2 + 1] = hi;
    }
    if (lane == 0) {
        b.valid[w] = ok ? 1 : 0;
        b.tc[w] = ok ? src.tc : 0.0;
        b.xpk[w] = ok ? src.xpk : 0.0;
    }
    if (!ok) return;
    // sines and cosines: lanes 0 .. 8 one angle each, lanes 2 .. 5 are m = 1 .. 4
    double sn, cs;
    {
        double angle = src.phiref * (double)(lane - 1);
        if (lane == 0) angle = 0.5 * src.iota;
        if (lane == 1) angle = src.iota;
        if (lane == 6) angle = 2.0 * src.psi;
        if (lane == 7) angle = src.lam;
        if (lane >= 8) angle = src.beta;
        sincos(angle, &sn, &cs);
    }
    auto sine = [&](int i) { return __shfl_sync(0xffffffffu, sn, i); };
    auto cosine = [&](int i) { return __shfl_sync(0xffffffffu, cs, i); };
    const double shi = sine(0), chi = cosine(0), ci = cosine(1), s2 = sine(6), c2 = cosine(6);
    const double sl = sine(7), cl = cosine(7), sb = sine(8), cb = cosine(8);
    const double sm = sine(md.m + 1), cm = cosine(md.m + 1);
    if (act) {  // this lane's mode
        ModeConst c;
        cplx kp, kc;
        pol_weights(md, chi, shi, ci, cm, sm, kp, kc);
        c.are = kp.re * c2 - kc.re * s2;
        c.aim = kp.im * c2 - kc.im * s2;
        c.bre = 2.0 * (kp.re * s2 + kc.re * c2);
        c.bim = 2.0 * (kp.im * s2 + kc.im * c2);
        c.xf = xf;
        c.v0 = cbrt(kPi * (c.xf * lo));
        c.x160 = sqrt(c.v0 * kInvCbrtPi);
        c.s6 = log(hi / lo) / (6.0 * (double)(d.K - 1));
        c.amp = src.amp0 * amp_ratio(src, md, 1.0);
        c.off = phase_offset(md) - 0.5 * md.m * (src.phpk - src.dphpk * src.xpk);
        c.half_m = 0.5 * md.m;
        c.power = amp_power(md);
        c.pad = 0;
        b.mconst[(size_t)w * d.L + lane] = c;
    }
    WalkerConst *c = b.wconst + w;
    if (lane == 0) {
        c->k128 = src.k128;
        c->ps2 = src.ps2;
        c->ps3 = src.ps3;
        c->phj = src.phj - src.c1 * kXJoin + src.c2 * (1.0 / kXJoin);
        c->c1 = src.c1;
        c->c2 = src.c2;
        c->dphpk = src.dphpk;
        c->tc = src.tc;
        c->m2pi = src.m2pi;
        c->al2 = src.al2;
        c->al3 = src.al3;
        c->ixrd = ixrd;
        const double R = kAuM / kClight;
        c->dx = kTwoPi * R * (cb * cl);
        c->dy = kTwoPi * R * (cb * sl);
    }
    if (lane < 8) {
        // lanes 0 .. 7: kn, kq, wn, un, each for arms 0 -> 1 and 1 -> 2 (differences, or sums for kq)
        const int what = lane >> 1;
        const bool second = lane & 1;
        const double h = 0.8660254037844386467637;  // cos, sin of 0, 2 pi / 3, 4 pi / 3
        double v[3] = {-cb * cl, -cb * sl, -sb};  // k
        if (what == 2) v[0] = -sb * cl, v[1] = -sb * sl, v[2] = cb;
        if (what == 3) v[0] = sl, v[1] = -cl, v[2] = 0.0;
        const double gc = what == 1 ? (second ? -1.0 : 0.5) : (second ? 0.0 : -1.5);
        const double gs = what == 1 ? (second ? 0.0 : h) : (second ? -2.0 * h : h);
        double o[5];
        harmonics(v, gc, gs, o);
        double *dst = what == 0   ? c->kn[second]
                      : what == 1 ? c->kq[second]
                      : what == 2 ? c->wn[second]
                                  : c->un[second];
        const int n = what == 3 ? 3 : 5;
        for (int i = 0; i < n; i++) dst[i] = o[i];
    }
}

cudaError_t launch_source(const StageDims &d, const StageBufs &b, cudaStream_t s) {
    source_kernel<<<(d.B + 3) / 4 + 1, 128, 0, s>>>(d, b);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------- knots
// One thread per knot of the modes of one m, 128 knots per block: log-spaced frequencies
// (Sec. II.A: ~2^10 points) with A, phase + delay, and T, and the first dense bin at or
// above each.  kSplit: the same FP64 values, A (times 2^64) and T stored as FP32 (the
// split-precision layout).
//
// Bound by the FP64 pipe (2 lanes per clock per SM), so the count of FP64 operations per
// knot is what matters (about 270 an m and 85 a mode, against 730 a mode): the powers of f come from one
// exponential of the log-spaced step (f^(1/6) and its powers, no cube root or square root),
// one division serves v, the amplitude and the three arms, the response is in orbital
// harmonics, and the modes of equal m share all of it but their polarisation weights
// (response.cuh), whose unit phasors and orbital angle are evaluated on the integer units and the
// sines of small angles by series.  1024 walkers, six modes of 1024 knots: 8.4 -> 3.3 ms with the
// source kernel (5.4 with one mode per thread, 4.0 with sincos() throughout).  One block of 128
// threads per system left all but a few SMs idle in small
// calls (6 systems of 1024 knots: 246 us), hence one knot per thread.
template <bool kSplit>
__global__ void __launch_bounds__(128) knot_kernel(StageDims d, StageBufs b, double idf, double near) {
    const int w = blockIdx.x / d.L, first = blockIdx.x % d.L;
    if (d.same[first]) return;  // done with the first mode of its m
    const size_t wm = (size_t)w * d.L + d.ord[first];
    if (!b.band[wm * 3]) return;  // inactive modes (and invalid walkers) have no knots
    __shared__ WalkerConst wc;
    __shared__ ModeConst mc;
    {
        const double *src = reinterpret_cast<const double *>(b.wconst + w);
        double *dst = reinterpret_cast<double *>(&wc);
        if (threadIdx.x < sizeof(WalkerConst) / 8) dst[threadIdx.x] = src[threadIdx.x];
        const double *msrc = reinterpret_cast<const double *>(b.mconst + wm);
        double *mdst = reinterpret_cast<double *>(&mc);
        if (threadIdx.x >= 96 && threadIdx.x - 96 < sizeof(ModeConst) / 8)
            mdst[threadIdx.x - 96] = msrc[threadIdx.x - 96];
    }
    __syncthreads();
    const int K = d.K, k = blockIdx.y * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const double flo = b.fedge[wm * 2], fhi = b.fedge[wm * 2 + 1];
    const double e6 = exp(mc.s6 * (double)k), e3 = e6 * e6;
    const double f = (k == K - 1) ? fhi : flo * (e3 * e3 * e3);
    // first dense bin at or above this knot: a guess, then exact by the bin frequencies
    // themselves
    const double g = (f - d.f0) * idf, gc = ceil(g);
    int j = gc <= 0.0 ? 0 : (gc >= (double)d.N ? d.N : (int)gc);
    if (fabs(g - rint(g)) < near) {
        while (j > 0 && bin_freq(d.f0, d.df, j - 1) >= f) j--;
        while (j < d.N && bin_freq(d.f0, d.df, j) < f) j++;
    }
    ModeBase base;
    mode_base(wc, mc, b.fxtab, f, mc.v0 * e3, mc.x160 * e6, base);
    for (int i = first; i < d.L && (i == first || d.same[i]); i++) {
        const size_t m = (size_t)w * d.L + d.ord[i];
        double amp;
        cplx T[3];
        mode_channels(base, i == first ? mc : b.mconst[m], amp, T);
        b.fk[m * K + k] = f;
        b.kb[m * K + k] = j;
        double *vm = b.vals + m * kNSeries * (size_t)K;
        vm[1 * K + k] = base.phase;
        if (kSplit) {
            float *v32 = split_vals32(b.vals, m, K);
            v32[k] = (float)(amp * kAmpScale64);
            for (int c = 0; c < 3; c++) {
                v32[(1 + 2 * c) * K + k] = (float)T[c].re;
                v32[(2 + 2 * c) * K + k] = (float)T[c].im;
            }
        } else {
            vm[0 * K + k] = amp;
            for (int c = 0; c < 3; c++) {
                vm[(2 + 2 * c) * K + k] = T[c].re;
                vm[(3 + 2 * c) * K + k] = T[c].im;
            }
        }
    }
}

template <bool kSplit>
static cudaError_t launch_knots_t(const StageDims &d, const StageBufs &b, cudaStream_t s) {
    cudaError_t e = launch_source(d, b, s);
    if (e != cudaSuccess) return e;
    // how near to a whole number a knot's bin number may be wrong: numbers below 1e11 are right to 1e-4
    const double near = d.f0 / d.df + d.N < 1e11 ? 1e-3 : 1.0;
    knot_kernel<kSplit><<<dim3(d.B * d.L, (d.K + 127) / 128), 128, 0, s>>>(d, b, 1.0 / d.df, near);
    return cudaGetLastError();
}

cudaError_t launch_knots(const StageDims &d, const StageBufs &b, cudaStream_t s) {
    return launch_knots_t<false>(d, b, s);
}

cudaError_t launch_knots_split(const StageDims &d, const StageBufs &b, cudaStream_t s) {
    return launch_knots_t<true>(d, b, s);
}

}  // namespace lisa
