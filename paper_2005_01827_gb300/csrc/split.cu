// split.cu -- split-precision dense stage of the batched LISA likelihood (Katz et al.
// 2020, Sec. II.A): FP64 is kept for the knot phases (through the FP64 spline
// coefficients) and for the final cross-block sums; the in-segment evaluation, the
// sincos, amplitudes, transfer functions and per-thread partial sums run in FP32.
//
// Phase: per spline segment an FP64 prologue turns the cubic phase (including the
// -2 pi f t_coal ramp) into forward differences over one bin, Phi, D1, D2, D3, held as
// 64-bit fixed-point fractions of a turn (with extra low words for the differences).
// Each thread moves them to the first bin of its 8-bin chunk by Newton's formula in
// modular integer arithmetic, so no rounding accumulates along a segment, rounds them
// to 32-bit words and advances the phase by three 32-bit additions per bin; the top 8
// bits of the phase index a table of e^{2 pi i k / 256} (the nearest entry) and the
// next 23 bits give a small signed angle (|r| <= pi / 256) whose sine and cosine are
// short FP32 polynomials.
//
// What bounds the dense kernel is the instruction issue (64 % of the slots, FMA pipe 49 %; the
// rest waits on the segment records), so the work per bin is cut to what depends on the bin:
//  * modes of equal m share the phase, so per segment the preparation sums their A T (complex,
//    per channel) into one quartic; a thread re-expands it to a quadratic over its chunk, and a bin
//    costs two packed (f32x2) FMAs per channel, one phasor and one complex multiply-add per m:
//    34 instructions a bin and m, against 43 a bin and mode with A and T evaluated per mode;
//  * the segment and 64-bit phase anchor of all a group's (walker, m) in a warp's bins are found
//    by one lane each, once per item; warps with a segment's end in them, bands that end there
//    and short segments take a general path, thread by thread.  There a segment's bins alone are
//    evaluated where it has no quartics (a chunk may hold several such segments), and segments
//    without bins are passed over by their bounds, 4 bytes each: calls
//    of 128 heavy walkers on a week's grid of 12036 bins, 1024 knots 4.59 -> 1.77 ms, 4096 knots
//    21.5 -> 9.0 ms, of the 1024 walkers below 25.87 -> 25.56 ms.
// 1024 walkers, six modes, year's grid: prior 31.3 -> 20.2 ms, posterior 14.7 -> 9.9 ms;
// 8192 walkers 229 -> 147 ms.  128-thread blocks, four per SM: two blocks of 256 threads that
// share a tile took 23.5 against 22.1 ms (longer barrier waits).
#include "f32x2.cuh"
#include "fixed.cuh"
#include "kernels.h"
#include "model.cuh"
#include "split.h"
#include "tma.cuh"

namespace lisa {

// fraction of a turn of x radians as a 128-bit two's-complement fixed-point number:
// hi holds the turns scaled by 2^64 (modulo 2^64), lo the next 64 fractional bits
__device__ __forceinline__ void turns_fixed(double x, unsigned long long &hi,
                                            unsigned long long &lo) {
    const double k = rint(x * kInvTwoPi);
    double r = fma(-k, kTwoPiHi, x);
    r = fma(-k, kTwoPiMid, r);
    r = fma(-k, kTwoPiLo, r);
    const i64 b = double_bits(r * kInvTwoPi);  // in about [-0.5, 0.5]: m 2^sh units of 2^-64
    const int e = (int)((b >> 52) & 0x7ff), sh = e - 1075 + 64;
    const unsigned long long m = (b & 0xfffffffffffffLL) | 0x10000000000000LL;
    unsigned long long h = 0, l = 0;
    if (sh >= 0) {
        h = m << sh;
    } else if (sh > -117 && e != 0) {
        const int k = -sh;
        h = k < 64 ? m >> k : 0;
        l = k < 64 ? m << (64 - k) : m >> (k - 64);
    }
    if (b < 0) {  // two's complement of both words
        l = 0ull - l;
        h = ~h + (l == 0);
    }
    hi = h;
    lo = l;
}

__device__ __forceinline__ double bin_freq_s(double f0, double df, int j) {
    return __dadd_rn(f0, __dmul_rn((double)j, df));
}

// ------------------------------------------------------------------------ data prep
// Whitened FP32 data: s = sqrt(w) 2^-64 and -2 d_hat = -2 sqrt(w) d per channel,
// w = 4 df / S.
__global__ void __launch_bounds__(256) prep_split_kernel(const double *__restrict__ bins, int N,
                                                         float *__restrict__ out) {
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < N; j += gridDim.x * blockDim.x) {
        const double *b = bins + (size_t)j * kBinDoubles;
        float *o = out + (size_t)j * kBinFloats;
        for (int c = 0; c < 3; c++) {
            const double w = b[c];
            const double sw = sqrt(w);
            o[c] = (float)(sw * 5.421010862427522e-20);
            // (w d) / sqrt(w) = sqrt(w) d
            o[3 + 2 * c] = (float)(-2.0 * b[3 + 2 * c] / sw);
            o[4 + 2 * c] = (float)(-2.0 * b[4 + 2 * c] / sw);
        }
    }
}

cudaError_t launch_prep_split(const double *bins, int N, float *out, cudaStream_t s) {
    const int blocks = min((N + 255) / 256, 4096);
    prep_split_kernel<<<blocks, 256, 0, s>>>(bins, N, out);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------ segments
// FP32 cubics of mode wm over segment s in t (SegRec::c) from the knot values and second
// derivatives: the spline's x-polynomial on [f_s, f_s+1) re-expanded at x = a and scaled
// to t (x = a + t wd)
__device__ __forceinline__ void mode_cubics(const StageBufs &b, size_t wm, int K, int s, double a,
                                            double wd, float c[28]) {
    const float *f32 = split_fac32(b.mscratch, wm, K);
    const float ihs = f32[s], hs = f32[K + s];
    const float af = (float)a, wf = (float)wd;
#pragma unroll
    for (int q = 0; q < kSplitSeries32; q++) {
        const float *yv = split_vals32(b.vals, wm, K) + (size_t)q * K;
        const float *Mv = split_m32(b.mscratch, wm, K) + (size_t)q * K;
        const float ys = yv[s], ys1 = yv[s + 1], ms = Mv[s], ms1 = Mv[s + 1];
        const float e1 = (ys1 - ys) * ihs - hs * fmaf(2.0f, ms, ms1) * (1.0f / 6.0f);
        const float e2 = 0.5f * ms;
        const float e3 = (ms1 - ms) * ihs * (1.0f / 6.0f);
        const int base = q == 0 ? 0 : 4 + 8 * ((q - 1) >> 1) + ((q - 1) & 1);
        const int step = q == 0 ? 1 : 2;
        c[base] = fmaf(af, fmaf(af, fmaf(af, e3, e2), e1), ys);
        c[base + step] = fmaf(af, fmaf(3.0f * af, e3, 2.0f * e2), e1) * wf;
        c[base + 2 * step] = fmaf(3.0f * af, e3, e2) * wf * wf;
        c[base + 3 * step] = e3 * wf * wf * wf;
    }
}

// error-free sum of two floats: a + b = s + e exactly
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = a + b;
    const float bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// One thread per (walker, mode, segment).  Without kGroup (the FP64 path) it makes the
// fixed-point forward differences of the full phase at the segment's first bin.  With it
// (split precision) the first mode of every m makes the record of all modes of that m (split.h):
// the products A T, of degree 6 in t, are summed with an exact t^0 term (a rounding there
// would be common to the segment's bins), brought to degree 4 by replacing t^6 and t^5 by
// their best approximations of lower degree on [0, 1] (Chebyshev economisation: errors 1/2048
// and 1/512 of their coefficients), and scaled to bins.  The quartics are used if what
// was dropped, and the cubic term over half a chunk (half3 its cube) that the dense kernel
// drops, are below 2^-30 of S in each channel; with 1024 knots on a year's grid 98 % of the bins are in
// such segments (degree 3: 66 %, the response oscillates at high frequencies; 1024 walkers in
// the prior 27.6 against 20 ms).
template <bool kGroup>
__global__ void __launch_bounds__(256) segprep_kernel(StageDims d, StageBufs b, SegRec *segs,
                                                      unsigned long long *phases, float half3) {
    const int K = d.K;
    const long long total = (long long)d.B * d.L * (K - 1);
    for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < total;
         g += (long long)gridDim.x * blockDim.x) {
        const int s = (int)(g % (K - 1));
        const int w = (int)(g / (K - 1) / d.L), pos = (int)(g / (K - 1) % d.L);
        if (kGroup && d.same[pos]) continue;
        const size_t wm = (size_t)w * d.L + (kGroup ? d.ord[pos] : pos);
        const int *bd = b.band + wm * 3;
        if (!bd[0] || !b.valid[w]) continue;
        const int *kb = b.kb + wm * K;
        const int kb0 = kb[s];
        const int kb1 = (s < K - 2) ? kb[s + 1] : bd[2] + 1;
        const int W = max(kb1 - kb0, 1);
        const double fs = b.fk[wm * K + s];
        const double fj0 = bin_freq_s(d.f0, d.df, kb0);
        const double a = fj0 - fs;
        const double *cf = b.coef + (wm * (K - 1) + s) * 32 + 4;
        unsigned long long ph[kPhaseWords];
        {
            const double c0 = cf[0], c1 = cf[1], c2 = cf[2], c3 = cf[3];
            const double y = fma(a, fma(a, fma(a, c3, c2), c1), c0);
            const double y1 = fma(a, fma(3.0 * a, c3, 2.0 * c2), c1);
            const double y2 = fma(3.0 * a, c3, c2);  // y''/2
            const double tw = kTwoPi * b.tc[w];
            const double p0 = fma(-tw, fj0, y);
            const double p1 = (y1 - tw) * d.df;
            const double p2 = y2 * d.df * d.df;
            const double p3 = c3 * d.df * d.df * d.df;
            unsigned long long dummy;
            turns_fixed(p0, ph[0], dummy);
            turns_fixed(p1 + p2 + p3, ph[1], ph[4]);
            turns_fixed(2.0 * p2 + 6.0 * p3, ph[2], ph[5]);
            turns_fixed(6.0 * p3, ph[3], ph[6]);
            ph[7] = (unsigned int)((s < K - 2) ? kb[s + 1] : 0x7fffffff);
            int guess = 0;
            if (s <= 1) {  // the (walker, mode)'s segment-guess constants, read once per tile
                const double f_lo = b.fedge[2 * wm], f_hi = b.fedge[2 * wm + 1];
                const double scl = (double)(K - 1) / log2(f_hi / f_lo);
                guess = __float_as_int((float)(s == 0 ? log2(f_lo) * scl : scl));
            }
            ph[7] |= (unsigned long long)(unsigned int)guess << 32;
        }
        if (!kGroup) {
            ulonglong2 *o = reinterpret_cast<ulonglong2 *>(phases + kPhaseWords * (wm * (K - 1) + s));
            for (int q = 0; q < kPhaseWords / 2; q++) o[q] = make_ulonglong2(ph[2 * q], ph[2 * q + 1]);
            continue;
        }
        const double wd = (double)W * d.df;
        int end = pos + 1;
        while (end < d.L && d.same[end]) end++;
        float S[6][7], lo[6];  // (channel, re/im): t^0 .. t^6, and the rest of t^0
#pragma unroll
        for (int q = 0; q < 6; q++) {
            lo[q] = 0.0f;
#pragma unroll
            for (int k = 0; k < 7; k++) S[q][k] = 0.0f;
        }
        for (int p = pos; p < end; p++) {
            float c[28];
            mode_cubics(b, (size_t)w * d.L + d.ord[p], K, s, a, wd, c);
#pragma unroll
            for (int q = 0; q < 6; q++) {
                float t[4];
#pragma unroll
                for (int k = 0; k < 4; k++) t[k] = c[4 + 8 * (q >> 1) + (q & 1) + 2 * k];
                const float p0 = c[0] * t[0], e0 = fmaf(c[0], t[0], -p0);
                float sum, err;
                two_sum(S[q][0], p0, sum, err);
                S[q][0] = sum;
                lo[q] += err + e0;
#pragma unroll
                for (int k = 1; k < 7; k++)
#pragma unroll
                    for (int i = 0; i < 4; i++)
                        if (k - i >= 0 && k - i < 4) S[q][k] = fmaf(c[i], t[k - i], S[q][k]);
            }
        }
        const float iw = 1.0f / (float)W;
        GroupRec r;
        bool ok = true;
#pragma unroll
        for (int x = 0; x < 3; x++) {
            float drop = 0.0f, m0 = 0.0f, m1 = 0.0f;
#pragma unroll
            for (int q = 2 * x; q < 2 * x + 2; q++) {
                float *v = S[q];
                const float c6 = v[6], c5 = fmaf(3.0f, c6, v[5]);
                const float c4 = fmaf(2.5f, c5, fmaf(-3.375f, c6, v[4]));
                const float c3 = fmaf(-2.1875f, c5, fmaf(1.75f, c6, v[3]));
                const float c2 = fmaf(0.78125f, c5, fmaf(-0.41015625f, c6, v[2]));
                const float c1 = fmaf(-0.09765625f, c5, fmaf(0.03515625f, c6, v[1]));
                lo[q] += fmaf(1.0f / 512.0f, c5, -1.0f / 2048.0f * c6);
                const float w2 = iw * iw, w3 = w2 * iw;
                drop = fmaxf(drop, half3 * fmaf(4.0f, fabsf(c4), fabsf(c3)) * w3 +
                                       fabsf(c5) * (1.0f / 512.0f) + fabsf(c6) * (1.0f / 2048.0f));
                m0 = fmaxf(m0, fabsf(v[0]));
                m1 = fmaxf(m1, fabsf(v[0] + c1 + c2 + c3 + c4));
                float *o = &r.s[x][0].x + (q & 1);
                o[0] = v[0];
                o[2] = lo[q];
                o[4] = c1 * iw;
                o[6] = c2 * w2;
                o[8] = c3 * w3;
                o[10] = c4 * (w2 * w2);
            }
            ok = ok && drop <= 9.3132257e-10f * fminf(m0, m1);
        }
#pragma unroll
        for (int q = 0; q < kPhaseWords; q++) r.ph[q] = ph[q];
        r.kb0 = kb0;
        r.ok = ok ? 1 : 0;
        r.pad[0] = r.pad[1] = 0;
        *group_rec(b.coef, wm, K, s) = r;
        if (ok) continue;
        for (int p = pos; p < end; p++) {
            const size_t m = (size_t)w * d.L + d.ord[p];
            SegRec o;
            mode_cubics(b, m, K, s, a, wd, o.c);
            o.invw = 1.0f / (float)W;
            o.pad[0] = o.pad[1] = o.pad[2] = 0;
            segs[m * (K - 1) + s] = o;
        }
    }
}

cudaError_t launch_segprep(const StageDims &d, const StageBufs &b, SegRec *segs, int chunk,
                           cudaStream_t s) {
    const float half = 0.5f * (float)(chunk - 1);
    const long long total = (long long)d.B * d.L * (d.K - 1);
    const int blocks = (int)min((total + 255) / 256, (long long)152 * 32);
    segprep_kernel<true><<<blocks, 256, 0, s>>>(d, b, segs, nullptr, half * half * half);
    return cudaGetLastError();
}

cudaError_t launch_phaseprep(const StageDims &d, const StageBufs &b, unsigned long long *phases,
                             cudaStream_t s) {
    const long long total = (long long)d.B * d.L * (d.K - 1);
    const int blocks = (int)min((total + 255) / 256, (long long)152 * 32);
    segprep_kernel<false><<<blocks, 256, 0, s>>>(d, b, nullptr, phases, 0.0f);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------ dense
// segment of bin j from the log spacing of the knots: (log2 f - log2 f_lo) (K - 1) /
// log2(f_hi / f_lo) by one MUFU log2 and one FMA (l0 = scale log2 f_lo)
__device__ __forceinline__ int seg_index_guess(float fjf, float l0, float scale) {
    return (int)fmaf(__log2f(fjf), scale, -l0);
}

// the guess moved by the integer knot-to-bin boundaries so that kb[s] <= j < kb[s + 1]
__device__ __forceinline__ int seg_guess(const int *__restrict__ kb, int K, int j, float fjf,
                                         float l0, float scale) {
    int s = seg_index_guess(fjf, l0, scale);
    s = min(max(s, 0), K - 2);
    while (s > 0 && __ldg(kb + s) > j) s--;
    while (s < K - 2 && __ldg(kb + s + 1) <= j) s++;
    return s;
}

// phase and forward differences at one bin as 32-bit fractions of a turn; the phase is
// offset by half a table cell so that its top 8 bits name the nearest table entry
struct PhaseState {
    unsigned int ph, d1, d2, d3;
};

// x / 2^32 rounded to the nearest integer (modulo 2^32)
__device__ __forceinline__ unsigned int top_rn(unsigned long long x) {
    return (unsigned int)(x >> 32) + ((unsigned int)x >> 31);
}

// floor(c L / 2^64) from the top 32 bits of L: low by less than c / 2^32 + 2 (c < 2^63)
__device__ __forceinline__ unsigned long long mulhi_top32(unsigned long long c,
                                                          unsigned long long L) {
    const unsigned int lh = (unsigned int)(L >> 32);
    return (c >> 32) * lh + (((unsigned long long)(unsigned int)c * lh) >> 32);
}

// the fixed-point phase words of a segment record (the last one holds the next
// segment's first bin)
struct SegPhase {
    ulonglong2 a, b, c, e;
};

__device__ __forceinline__ int seg_next(const SegPhase &q) { return (int)(unsigned int)q.e.y; }

// record of segment i, counted over all (walker, mode)s
__device__ __forceinline__ const GroupRec *record_at(const double *coef, unsigned int i) {
    return reinterpret_cast<const GroupRec *>(coef + (size_t)i * 32);
}

__device__ __forceinline__ SegPhase load_phase(const GroupRec *__restrict__ r) {
    const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(r->ph);
    return SegPhase{__ldg(w), __ldg(w + 1), __ldg(w + 2), __ldg(w + 3)};
}

// the rest of a group record, and the first bin of the next segment
struct Segment {
    float2 s[3][6];
    int kb0, ok, next;
};

__device__ __forceinline__ void load_series(const GroupRec *__restrict__ r, Segment &o) {
    const float4 *v = reinterpret_cast<const float4 *>(&r->kb0);
    float4 x[10];
#pragma unroll
    for (int i = 0; i < 10; i++) x[i] = __ldg(v + i);
    o.kb0 = __float_as_int(x[0].x);
    o.ok = __float_as_int(x[0].y);
#pragma unroll
    for (int i = 0; i < 18; i++) {
        const float4 u = x[(i + 1) >> 1];
        o.s[i / 6][i % 6] = (i & 1) ? make_float2(u.x, u.y) : make_float2(u.z, u.w);
    }
}

// its first bin and ok alone
__device__ __forceinline__ void load_head(const GroupRec *__restrict__ r, Segment &o) {
    const int2 v = __ldg(reinterpret_cast<const int2 *>(&r->kb0));
    o.kb0 = v.x;
    o.ok = v.y;
}

// forward differences of the segment's phase moved from its first bin to bin n, which may
// lie up to a warp's bins before it (Newton's forward-difference formula in modular integer
// arithmetic).  The carries of the low words into the phase and the first difference are
// taken from their top 32 bits and the ones multiplied by n are dropped: the 64-bit anchor is
// low by at most a few n units of 2^-64 turn for n < 2^21.
struct __align__(16) Phase64 {
    unsigned long long ph, d1, d2, d3;
};

__device__ __forceinline__ Phase64 phase64(const SegPhase &q, int n) {
    const ulonglong2 a = q.a, b = q.b;
    const i64 sn = n;
    // n(n-1)/2 and n(n-1)(n-2)/6 (the product of three consecutive integers divided by 2
    // is a multiple of 3: multiplying by the inverse of 3 modulo 2^64 divides it exactly)
    const unsigned long long c2 = (unsigned long long)(sn * (sn - 1) / 2);
    const unsigned long long c3 = c2 * (unsigned long long)(sn - 2) * 0xAAAAAAAAAAAAAAABull;
    Phase64 p;
    p.ph = a.x + a.y * (unsigned long long)sn + c2 * b.x + c3 * b.y;
    p.d1 = a.y + b.x * (unsigned long long)sn + c2 * b.y;
    if (n >= 2) {
        p.ph += mulhi_top32(c2, q.c.y) + mulhi_top32(c3, q.e.x);
        p.d1 += mulhi_top32(c2, q.e.x);
    }
    p.d2 = b.x + b.y * (unsigned long long)sn;
    p.d3 = b.y;
    return p;
}

// The same rounded to 32-bit words, with which a thread advances its chunk: after i steps the
// phase is off by at most
// (1 + i + i(i-1)/2 + i(i-1)(i-2)/6) / 2 units of 2^-32 turn (32 units, 4.7e-8 rad, at
// i = 7), and every chunk starts again from the exact record.
__device__ __forceinline__ PhaseState phase_at(const SegPhase &q, int n) {
    const ulonglong2 a = q.a, b = q.b;
    const unsigned int un = (unsigned int)n;
    if (n < 65536) {
        // n(n-1)/2 fits 32 bits: the same sums from 32 x 32 -> 64 products
        const uint32_t m2 = un * (un - 1u) >> 1;
        const unsigned long long m3 =
            (unsigned long long)mad_s((int)m2, n - 2, 0) * 0xAAAAAAAAAAAAAAABull;
        const uint32_t m3l = (uint32_t)m3, m3h = (uint32_t)(m3 >> 32);
        const uint32_t d1l = (uint32_t)a.y, d1h = (uint32_t)(a.y >> 32);
        const uint32_t d2l = (uint32_t)b.x, d2h = (uint32_t)(b.x >> 32);
        const uint32_t d3l = (uint32_t)b.y, d3h = (uint32_t)(b.y >> 32);
        const uint32_t l2 = (uint32_t)(q.c.y >> 32), l3 = (uint32_t)(q.e.x >> 32);
        const uint32_t minus = (uint32_t)(n >> 31);  // un = n + 2^32 for n < 0
        i64 ph = mad_u(d1l, un, (i64)a.x);
        ph = mad_u(d2l, m2, ph);
        ph = mad_u(d3l, m3l, ph);
        if (n >= 0) ph += (i64)((unsigned long long)m3h * l3 + __umulhi(m3l, l3) + __umulhi(m2, l2));
        ph = add_hi(ph, d1h * un - (d1l & minus) + d2h * m2 + d3h * m3l + d3l * m3h);
        i64 d1 = mad_u(d2l, un, (i64)a.y);
        d1 = mad_u(d3l, m2, d1) + (i64)__umulhi(m2, l3);
        d1 = add_hi(d1, d2h * un - (d2l & minus) + d3h * m2);
        const i64 d2 = add_hi(mad_u(d3l, un, (i64)b.x), d3h * un - (d3l & minus));
        PhaseState p;
        p.ph = top_rn((unsigned long long)ph) + (1u << 23);  // + half a cell of the table
        p.d1 = top_rn((unsigned long long)d1);
        p.d2 = top_rn((unsigned long long)d2);
        p.d3 = top_rn(b.y);
        return p;
    }
    const Phase64 f = phase64(q, n);
    PhaseState p;
    p.ph = top_rn(f.ph) + (1u << 23);
    p.d1 = top_rn(f.d1);
    p.d2 = top_rn(f.d2);
    p.d3 = top_rn(f.d3);
    return p;
}

// the anchor of a warp's bins, m >= 0 bins on: c2 = m(m-1)/2, c3 = m(m-1)(m-2)/6
__device__ __forceinline__ PhaseState phase_from(const Phase64 *__restrict__ w, uint32_t m,
                                                 uint32_t c2, uint32_t c3) {
    const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(&w->ph);
    const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(&w->d2);
    const uint32_t d2l = (uint32_t)b.x, d2h = (uint32_t)(b.x >> 32);
    const uint32_t d3l = (uint32_t)b.y, d3h = (uint32_t)(b.y >> 32);
    i64 ph = mad_u((uint32_t)a.y, m, (i64)a.x);
    ph = mad_u(d2l, c2, ph);
    ph = mad_u(d3l, c3, ph);
    ph = add_hi(ph, (uint32_t)(a.y >> 32) * m + d2h * c2 + d3h * c3);
    const i64 d1 = add_hi(mad_u(d3l, c2, mad_u(d2l, m, (i64)a.y)), d2h * m + d3h * c2);
    const i64 d2 = add_hi(mad_u(d3l, m, (i64)b.x), d3h * m);
    PhaseState p;
    p.ph = top_rn((unsigned long long)ph) + (1u << 23);
    p.d1 = top_rn((unsigned long long)d1);
    p.d2 = top_rn((unsigned long long)d2);
    p.d3 = top_rn(b.y);
    return p;
}

// the FP32 cubic coefficients and 1/width of a mode's own record
struct SegCoef {
    float c[28];
    float invw;
};

__device__ __forceinline__ SegCoef seg_coef(const SegRec *__restrict__ rp) {
    SegCoef r;
    const float4 *v = reinterpret_cast<const float4 *>(rp->c);
#pragma unroll
    for (int q = 0; q < 7; q++) {
        const float4 x = __ldg(v + q);
        r.c[4 * q] = x.x;
        r.c[4 * q + 1] = x.y;
        r.c[4 * q + 2] = x.z;
        r.c[4 * q + 3] = x.w;
    }
    r.invw = __ldg(&rp->invw);
    return r;
}

// e^{2 pi i (ph - 2^23) / 2^32} for a phase word ph offset by half a cell: the table
// entry k = ph >> 24 (the nearest multiple of 2 pi / 256) times the rotation by the
// remaining signed angle r, |r| <= pi / 256, whose cosine 1 - r^2/2 is off by r^4/24 <
// 1e-9 and sine r - r^3/6 by r^5/120 < 3e-12.  (With 2048 entries two operations fewer are
// needed, but the mean norm of the rounded entries, common to all bins, is another: results
// move by 1.5e-9.)
__device__ __forceinline__ void phasor(unsigned int ph, const float2 *__restrict__ tab,
                                       float &zr, float &zi) {
    const float2 t = tab[ph >> 24];
    // x = 1 + (ph mod 2^24) / 2^24 from the next 23 bits; x - 1.5 is exact, and so is
    // 1.5 kStep (kStep is 2 pi / 256 rounded to 23 significant bits), so the FMA
    // rounds (x - 1.5) kStep once
    const float x = __uint_as_float(((ph >> 1) & 0x7fffffu) | 0x3f800000u);
    const float r = fmaf(x, 0.02454369142651558f, -0.03681553713977337f);
    const float r2 = r * r;
    const float sn = r * fmaf(r2, -0.16666666666666666f, 1.0f);
    const float cs = fmaf(r2, -0.5f, 1.0f);
    zr = t.x * cs - t.y * sn;
    zi = fmaf(t.x, sn, t.y * cs);
}

__device__ __forceinline__ int group_of_s(const int *__restrict__ item_start, int ng, int item) {
    int lo = 0, hi = ng - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (item_start[mid] <= item)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// FP32 (value, compensation) pairs, kept as an unevaluated hi + lo pair: this lane's and the
// one's o lanes up together, and the warp sum
__device__ __forceinline__ void pair_down(float &hi, float &lo, int o) {
    const float h2 = __shfl_down_sync(0xffffffffu, hi, o);
    const float l2 = __shfl_down_sync(0xffffffffu, lo, o);
    float s, e;
    two_sum(hi, h2, s, e);
    hi = s;
    lo = lo + l2 + e;
}

__device__ __forceinline__ void warp_sum_pair(float &hi, float &lo) {
    for (int o = 16; o > 0; o >>= 1) pair_down(hi, lo, o);
}

// the seven FP32 series of a record at in-segment coordinate tt = (t, t): the amplitude
// by scalar Horner, each channel's (Re, Im) transfer pair by packed Horner
__device__ __forceinline__ void eval_series(const SegCoef &r, float2 tt, float &amp,
                                            float2 tr[3]) {
    const float t = tt.x;
    amp = fmaf(t, fmaf(t, fmaf(t, r.c[3], r.c[2]), r.c[1]), r.c[0]);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const float *k = r.c + 4 + 8 * c;
        float2 x = fma2(tt, make_float2(k[6], k[7]), make_float2(k[4], k[5]));
        x = fma2(tt, x, make_float2(k[2], k[3]));
        tr[c] = fma2(tt, x, make_float2(k[0], k[1]));
    }
}

// h += T e^{i phi} (amp) for the three channels of one bin
__device__ __forceinline__ void add_mode(float zr, float zi, const float2 tr[3], float hr[3],
                                         float hm[3]) {
#pragma unroll
    for (int c = 0; c < 3; c++) {
        hr[c] = fmaf(tr[c].x, zr, fmaf(-tr[c].y, zi, hr[c]));
        hm[c] = fmaf(tr[c].x, zi, fmaf(tr[c].y, zr, hm[c]));
    }
}

// S^X at the chunk's bin i = m + u, m = (C - 1) / 2: s0 + u (s1 + u s2), re-expanded from the
// segment's quartic at its coordinate n of the chunk's middle
__device__ __forceinline__ void expand_at(const Segment &g, float n, float2 e[3][3]) {
    const float2 nn = make_float2(n, n);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const float2 *k = g.s[c];
        const float2 b3 = fma2(nn, k[5], k[4]);
        const float2 b2 = fma2(nn, b3, k[3]);
        const float2 b1 = fma2(nn, b2, k[2]);
        e[c][0] = add2(k[0], fma2(nn, b1, k[1]));
        const float2 d3 = fma2(nn, k[5], b3);
        const float2 d2 = fma2(nn, d3, b2);
        e[c][1] = fma2(nn, d2, b1);
        e[c][2] = fma2(nn, fma2(nn, k[5], d3), d2);
    }
}

__device__ __forceinline__ void phase_next(PhaseState &p) {
    p.ph += p.d1;
    p.d1 += p.d2;
    p.d2 += p.d3;
}

template <int C, int G>
__global__ void __launch_bounds__(128, 4) dense_split_kernel(StageDims d, StageBufs b,
                                                          const SegRec *__restrict__ segs,
                                                          const float *__restrict__ bins,
                                                          int tile_bins, float f0f, float dff) {
    extern __shared__ __align__(128) unsigned char smem[];
    float *sbin = reinterpret_cast<float *>(smem);  // [tile_bins][9]
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem + sizeof(float) * kBinFloats * tile_bins);
    __shared__ float2 tab[256];
    __shared__ int s_item, s_walker[G], s_here[G], s_lo[G][kMaxModes], s_hi[G][kMaxModes];
    __shared__ float s_flo[G][kMaxModes], s_scl[G][kMaxModes];
    __shared__ float4 red[G == 8 ? 1 : G][4];  // per slot, per warp: (ri, ri comp, hh, hh comp)
    // the first mode of each m (in the order of d.ord), their number; per walker and m the index
    // of segment 0 among all segments; and where a warp's bins of one m lie in one segment with
    // quartics, and in the band: the segment (-1 otherwise) and the phase at the warp's first bin
    __shared__ int s_first[kMaxModes], s_nm;
    __shared__ unsigned int s_base[G][kMaxModes];
    __shared__ int s_seg[4][G][kMaxModes];
    __shared__ Phase64 s_anchor[4][G][kMaxModes];
    // groups of 8 walkers: the (ri, ri comp, hh, hh comp) per slot of two threads together,
    // reduced once per item below instead of by warp shuffles per walker
    float4 *part_s = reinterpret_cast<float4 *>(bar + 2);  // [G][64], G = 8
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k = tid; k < 256; k += blockDim.x) {
        double sn, cs;
        sincospi((double)k / 128.0, &sn, &cs);
        tab[k] = make_float2((float)cs, (float)sn);
    }
    if (tid == 0) {
        mbar_init(bar, 1);
        int n = 0;
        for (int i = 0; i < d.L; i++)
            if (!d.same[i]) s_first[n++] = i;
        s_nm = n;
    }
    __syncthreads();
    const int nm = s_nm;
    const int ng = n_groups(d.B, G);
    const int total = b.item_start[ng];
    const int K = d.K;
    uint32_t parity = 0;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_item = atomicAdd(b.counter, 1);
        __syncthreads();
        const int item = s_item;
        if (item >= total) return;
        const int g = group_of_s(b.item_start, ng, item);
        const int J0 = b.grange[2 * g] + (item - b.item_start[g]) * tile_bins;
        const int Jend = min(J0 + tile_bins, b.grange[2 * g + 1] + 1);
        // whole groups of 4 rows (16-byte multiples) by one bulk copy, the last <= 3 rows
        // by plain loads, so nothing past the end of the data is read
        const int full = (Jend - J0) & ~3, tail = Jend - J0 - full;
        if (tid == 0 && full > 0) {
            const uint32_t bytes = (uint32_t)(full * kBinFloats * sizeof(float));
            fence_proxy_async();
            if (b.wait_test_polls == 0)
                tma_load_1d(sbin, bins + (size_t)J0 * kBinFloats, bytes, bar);
            else
                mbar_expect_tx(bar, bytes);  // test of the give-up path: no copy is issued
        }
        if (tid < tail * kBinFloats)
            sbin[full * kBinFloats + tid] = bins[((size_t)J0 + full) * kBinFloats + tid];
        if (tid < G) {
            const int i = g * G + tid, w = i < d.B ? b.order[i] : -1;
            s_walker[tid] = w;
            // not an empty slot, and a band that reaches into the tile
            s_here[tid] = w >= 0 && b.wrange[2 * w + 1] >= J0 && b.wrange[2 * w] < Jend;
        }
        if (tid < G * kMaxModes) {
            const int k = tid / kMaxModes, mi = tid % kMaxModes;
            const int i = g * G + k;
            int lo = 1, hi = 0;
            float flo = 0.0f, scl = 0.0f;  // scale log2 f_lo and the guess scale
            if (i < d.B && mi < nm) {
                const int w = b.order[i];
                const size_t wm = (size_t)w * d.L + d.ord[s_first[mi]];
                const int *bd = b.band + wm * 3;
                if (b.valid[w] && bd[0]) {
                    lo = bd[1];
                    hi = bd[2];
                    flo = __uint_as_float((unsigned int)(__ldg(&group_rec(b.coef, wm, K, 0)->ph[7]) >> 32));
                    scl = __uint_as_float((unsigned int)(__ldg(&group_rec(b.coef, wm, K, 1)->ph[7]) >> 32));
                }
                s_base[k][mi] = (unsigned int)(wm * (K - 1));
            }
            s_lo[k][mi] = lo;
            s_hi[k][mi] = hi;
            s_flo[k][mi] = flo;
            s_scl[k][mi] = scl;
        }
        __syncthreads();
        if (full > 0) {
            // every thread waits; the block leaves together if the copy never completed
            const uint32_t polls = b.wait_test_polls ? b.wait_test_polls : kWaitPolls;
            if (!__syncthreads_and(mbar_wait_bounded(bar, parity, b.err, polls))) return;
            parity ^= 1u;
        }

        // lane t: the t-th (walker, m) of the group in this warp's bins
        const int Jw = J0 + warp * 32 * C;
        for (int t = lane; t < G * nm; t += 32) {
            const int k = t / nm, mi = t % nm;
            int seg = -1;
            if (Jw + 32 * C <= Jend && s_lo[k][mi] <= Jw && s_hi[k][mi] >= Jw + 32 * C - 1) {
                const double *base = b.coef;
                const float fa = fmaf((float)Jw, dff, f0f);
                int s = seg_index_guess(fa, s_flo[k][mi], s_scl[k][mi]);
                s = min(max(s, 0), K - 2);
                const GroupRec *rec = record_at(base, s_base[k][mi] + s);
                int2 kk = __ldg(reinterpret_cast<const int2 *>(&rec->kb0));
                SegPhase q = load_phase(rec);
                if ((s > 0 && kk.x > Jw) || seg_next(q) <= Jw) {  // the guess missed: search
                    const int *kb = b.kb + ((size_t)s_walker[k] * d.L + d.ord[s_first[mi]]) * K;
                    s = seg_guess(kb, K, Jw, fa, s_flo[k][mi], s_scl[k][mi]);
                    rec = record_at(base, s_base[k][mi] + s);
                    kk = __ldg(reinterpret_cast<const int2 *>(&rec->kb0));
                    q = load_phase(rec);
                }
                if (kk.y && seg_next(q) >= Jw + 32 * C) {
                    seg = s;
                    s_anchor[warp][k][mi] = phase64(q, Jw - kk.x);
                }
            }
            s_seg[warp][k][mi] = seg;
        }
        __syncwarp();

        for (int k = 0; k < G; k++) {
            const int w = s_walker[k];
            if (!s_here[k]) continue;
            const int j0 = J0 + tid * C;
            float hr[C][3], hm[C][3];
#pragma unroll
            for (int i = 0; i < C; i++)
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    hr[i][c] = 0.0f;
                    hm[i][c] = 0.0f;
                }
            for (int mi = 0; mi < nm; mi++) {  // the modes of one m
                int s = s_seg[warp][k][mi];
                const unsigned int base = s_base[k][mi];
                Segment r;
                PhaseState p = {0, 0, 0, 0};
                float2 e[3][3];
                auto bin = [&](int i, bool in) {
                    const float u = (float)i - 0.5f * (C - 1);
                    const float2 uu = make_float2(u, u);
                    float2 tr[3];
#pragma unroll
                    for (int c = 0; c < 3; c++)
                        tr[c] = fma2(uu, fma2(uu, e[c][2], e[c][1]), e[c][0]);
                    float zr, zi;
                    phasor(p.ph, tab, zr, zi);
                    add_mode(in ? zr : 0.0f, in ? zi : 0.0f, tr, hr[i], hm[i]);
                    phase_next(p);
                };
                if (s >= 0) {  // one segment for the whole warp
                    load_series(record_at(b.coef, base + s), r);
                    const uint32_t m = lane * C, c2 = m * (m - 1) / 2;
                    p = phase_from(&s_anchor[warp][k][mi], m, c2, c2 * (m - 2) / 3);
                    expand_at(r, (float)(j0 - r.kb0) + 0.5f * (C - 1), e);
#pragma unroll
                    for (int i = 0; i < C; i++) bin(i, true);
                    continue;
                }
                int ja = max(j0, s_lo[k][mi]);
                const int jb = min(min(j0 + C, Jend), s_hi[k][mi] + 1);
                if (ja >= jb) continue;
                const float fa = fmaf((float)ja, dff, f0f);
                s = seg_index_guess(fa, s_flo[k][mi], s_scl[k][mi]);
                s = min(max(s, 0), K - 2);
                const GroupRec *rec = record_at(b.coef, base + s);
                SegPhase q = load_phase(rec);
                load_head(rec, r);
                // the record of the guessed segment is fetched with the bounds that check it (its
                // other cache line ahead of its use, which a segment without quartics has none for),
                // so a right guess (the usual case) costs no load from L2 after another
                asm volatile("prefetch.global.L1 [%0];" ::"l"(&rec->s[1][4]));
                if ((s > 0 && r.kb0 > ja) || seg_next(q) <= ja) {  // the guess missed: search
                    const int *kb = b.kb + ((size_t)w * d.L + d.ord[s_first[mi]]) * K;
                    s = seg_guess(kb, K, ja, fa, s_flo[k][mi], s_scl[k][mi]);
                    rec = record_at(b.coef, base + s);
                    q = load_phase(rec);
                    load_head(rec, r);
                }
                r.next = seg_next(q);
                p = phase_at(q, j0 - r.kb0);
                for (;;) {  // the chunk's segments, usually one
                    const int to = min(jb, r.next);
                    if (r.ok) {
                        load_series(rec, r);
                        expand_at(r, (float)(j0 - r.kb0) + 0.5f * (C - 1), e);
#pragma unroll
                        for (int i = 0; i < C; i++) bin(i, j0 + i >= ja && j0 + i < to);
                    } else {
                        const int pos = s_first[mi];
                        for (int m = pos; m < d.L && (m == pos || d.same[m]); m++) {
                            const SegCoef o =
                                seg_coef(segs + ((size_t)w * d.L + d.ord[m]) * (K - 1) + s);
                            PhaseState pm = p;
#pragma unroll
                            for (int i = 0; i < C; i++) {
                                const int j = j0 + i;
                                if (j >= ja && j < to) {
                                    const float t = (float)(j - r.kb0) * o.invw;
                                    float amp;
                                    float2 tr[3];
                                    eval_series(o, make_float2(t, t), amp, tr);
                                    float zr, zi;
                                    phasor(pm.ph, tab, zr, zi);
                                    add_mode(zr * amp, zi * amp, tr, hr[i], hm[i]);
                                }
                                phase_next(pm);
                            }
                        }
                    }
                    ja = max(ja, to);
                    if (ja >= jb) break;
                    const int *kb = b.kb + ((size_t)w * d.L + d.ord[s_first[mi]]) * K;
                    do
                        s++;
                    while (s < K - 2 && __ldg(kb + s + 1) <= ja);  // segments without bins
                    rec = record_at(b.coef, base + s);
                    q = load_phase(rec);
                    load_head(rec, r);
                    r.next = seg_next(q);
                    p = phase_at(q, j0 - r.kb0);
                }
            }

            // per-bin integrand |h|^2 - 2 Re(d h*) and |h|^2 in whitened units, packed as
            // (re, im) pairs per channel, then compensated (Kahan) sums over the chunk of
            // the pair (integrand, |h|^2)
            float2 sum = make_float2(0.0f, 0.0f), comp = make_float2(0.0f, 0.0f);
            auto bin_term = [&](const float *o, int i) {
                float2 ri = make_float2(0.0f, 0.0f), hh = make_float2(0.0f, 0.0f);
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const float sw = o[c];
                    const float2 x = mul2(make_float2(sw, sw), make_float2(hr[i][c], hm[i][c]));
                    const float2 e = add2(x, make_float2(o[3 + 2 * c], o[4 + 2 * c]));
                    ri = fma2(x, e, ri);
                    hh = fma2(x, x, hh);
                }
                const float2 y = sub2(make_float2(ri.x + ri.y, hh.x + hh.y), comp);
                const float2 t2 = add2(sum, y);
                comp = sub2(sub2(t2, sum), y);
                sum = t2;
            };
            if (j0 + C <= Jend) {
                // the chunk's C rows start on a 16-byte boundary ((j0 - J0) 36 bytes =
                // tid C 36): four rows at a time by nine 16-byte loads
                const float4 *o4 = reinterpret_cast<const float4 *>(sbin + tid * C * kBinFloats);
#pragma unroll
                for (int h4 = 0; h4 < C / 4; h4++) {
                    float rows[4 * kBinFloats];
#pragma unroll
                    for (int q = 0; q < kBinFloats; q++) {
                        const float4 v = o4[kBinFloats * h4 + q];
                        rows[4 * q] = v.x;
                        rows[4 * q + 1] = v.y;
                        rows[4 * q + 2] = v.z;
                        rows[4 * q + 3] = v.w;
                    }
#pragma unroll
                    for (int i = 0; i < 4; i++) bin_term(rows + kBinFloats * i, 4 * h4 + i);
                }
            } else {
#pragma unroll
                for (int i = 0; i < C; i++) {
                    const int j = j0 + i;
                    if (j >= Jend) continue;
                    bin_term(sbin + (j - J0) * kBinFloats, i);
                }
            }
            // FP32 (value, compensation) pairs summed error-free across the block below;
            // FP64 from the block's partial up
            if constexpr (G == 8) {
                float rs = sum.x, hs = sum.y, rl = -comp.x, hl = -comp.y;
                pair_down(rs, rl, 16);
                pair_down(hs, hl, 16);
                if (lane < 16) part_s[k * 64 + warp * 16 + lane] = make_float4(rs, rl, hs, hl);
            } else {
                float rs = sum.x, hs = sum.y, rl = -comp.x, hl = -comp.y;
                warp_sum_pair(rs, rl);
                warp_sum_pair(hs, hl);
                if ((tid & 31) == 0) red[k][tid >> 5] = make_float4(rs, rl, hs, hl);
            }
        }
        // one block barrier per item, then error-free FP32 sums (two-sum of the values,
        // compensations added) of every slot, once to FP64
        __syncthreads();
        if constexpr (G == 8) {
            // 16 sums (slot k, quantity q) of the 64 pairs, 8 threads each: 8 pairs per
            // thread, then the 8 threads' pairs by shuffles
            const int grp = tid >> 3, j = tid & 7, k = grp >> 1, q = grp & 1;
            float ps = 0.0f, pe = 0.0f;
            if (s_here[k]) {
                for (int i = 0; i < 8; i++) {
                    const float4 v = part_s[k * 64 + i * 8 + j];
                    float t, r;
                    two_sum(ps, q ? v.z : v.x, t, r);
                    ps = t;
                    pe += r + (q ? v.w : v.y);
                }
            }
            for (int o = 4; o > 0; o >>= 1) {
                const float s2 = __shfl_down_sync(0xffffffffu, ps, o, 8);
                const float e2 = __shfl_down_sync(0xffffffffu, pe, o, 8);
                float t, r;
                two_sum(ps, s2, t, r);
                ps = t;
                pe = pe + e2 + r;
            }
            if (j == 0 && s_walker[k] >= 0)
                b.part[2 * ((size_t)item * G + k) + q] = (double)ps + (double)pe;
        } else if (tid < G && s_walker[tid] >= 0) {
            const size_t slot = (size_t)item * G + tid;
            double a = 0.0, c = 0.0;
            if (s_here[tid]) {
                float4 v = red[tid][0];
                float as = v.x, ae = v.y, cs = v.z, ce = v.w;
                for (int q = 1; q < (int)(blockDim.x >> 5); q++) {
                    v = red[tid][q];
                    float t, e;
                    two_sum(as, v.x, t, e);
                    as = t;
                    ae += e + v.y;
                    two_sum(cs, v.z, t, e);
                    cs = t;
                    ce += e + v.w;
                }
                a = (double)as + (double)ae;
                c = (double)cs + (double)ce;
            }
            b.part[2 * slot] = a;
            b.part[2 * slot + 1] = c;
        }
    }
}

template <int C, int G>
size_t split_smem() {
    return sizeof(float) * kBinFloats * 128 * C + 16 + (G == 8 ? sizeof(float4) * G * 64 : 0);
}

template <int C, int G>
cudaError_t launch_split(const StageDims &d, const StageBufs &b, const SegRec *segs,
                         const float *bins, int blocks, cudaStream_t s) {
    const size_t smem = split_smem<C, G>();
    cudaError_t e = cudaFuncSetAttribute(dense_split_kernel<C, G>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    dense_split_kernel<C, G><<<blocks, 128, smem, s>>>(d, b, segs, bins, 128 * C, (float)d.f0,
                                                (float)d.df);
    return cudaGetLastError();
}

template <int C, int G>
int occ_split() {
    const size_t smem = split_smem<C, G>();
    if (cudaFuncSetAttribute(dense_split_kernel<C, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) != cudaSuccess)
        return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, dense_split_kernel<C, G>, 128, smem) != cudaSuccess)
        return 0;
    return n;
}

int dense_split_occupancy(int per_thread, int group) {
    if (per_thread == 8 && group == 8) return occ_split<8, 8>();
    if (per_thread == 8 && group == 1) return occ_split<8, 1>();
    if (per_thread == 16 && group == 8) return occ_split<16, 8>();
    if (per_thread == 4 && group == 8) return occ_split<4, 8>();
    return 0;
}

cudaError_t launch_dense_split(const StageDims &d, const StageBufs &b, const SegRec *segs,
                               const float *bins, const DenseTune &t, cudaStream_t s) {
    if (t.threads != 128) return cudaErrorInvalidValue;
    if (t.per_thread == 8 && t.group == 8) return launch_split<8, 8>(d, b, segs, bins, t.blocks, s);
    if (t.per_thread == 8 && t.group == 1) return launch_split<8, 1>(d, b, segs, bins, t.blocks, s);
    if (t.per_thread == 16 && t.group == 8)
        return launch_split<16, 8>(d, b, segs, bins, t.blocks, s);
    if (t.per_thread == 4 && t.group == 8) return launch_split<4, 8>(d, b, segs, bins, t.blocks, s);
    return cudaErrorInvalidValue;
}

}  // namespace lisa
