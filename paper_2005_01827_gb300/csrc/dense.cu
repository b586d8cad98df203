// dense.cu -- the fused dense kernel of the FP64 path of the batched LISA likelihood (Katz et
// al. 2020, Sec. II.A): spline interpolation of A, phase and T onto the dense bins, the mode
// sum, and the noise-weighted inner products of Eqs. (3) and (11), reduced to one
// (<d|h>, <h|h>) pair per (work item, walker).  The dense template is never stored.
//
// Arithmetic.  GB300's FP64 pipe does 2 operations per clock and SM, and a (walker, mode,
// bin) takes 47 of them, so evaluated in FP64 this kernel ran at that pipe's speed (94 %
// busy) and took 98 % of a call.  Here the per-bin work is in 64-bit fixed point on the
// integer multiply-add units (28 times the rate; fixed.cuh), with as many bits as FP64 has:
//   * the phase phi - 2 pi f t_coal advances from bin to bin by exact 64-bit forward
//     differences (anchored per spline segment by an FP64 prologue), and e^{i phase} comes
//     from a table and short polynomials, to 1e-16; modes with the same m have the same
//     phase and share it;
//   * the amplitude and the six transfer cubics are re-expanded in FP64 where a segment
//     enters a warp's block of 128 bins, scaled by a power of two that bounds them over its
//     bins there, and advance by 64-bit forward differences; A e^{i phase} T is summed over
//     the modes in 64 bits, in units of 2^-55 of the largest product of bounds of the block and
//     channel: 2^-49 of its largest mode on most segments.  Bounds further above their values
//     than kLoose bits are not used (dense_direct), so 2^-41 at worst;
//   * the integrand is summed in FP32 pairs over a thread's bins, and in FP64 from there up:
//     h rounded to 8 units of its sum (2^-46 of the largest mode, without a bias), w and w d to 48
//     bits; products with their errors and two-sums, what these leave summed in plain FP32
//     (2^-45 of a thread's sum).
// Terms are thus exact to about 2e-15 of the largest mode's on most segments, and the knots'
// FP64 phases (1e-12 to 1e-9 rad) set the error as they did: against 64-bit sums of the same splines the
// errors of ln L, <d|h> and <h|h> are those of the FP64 evaluation (1024 walkers: 7.1e-11
// both).  Where a warp's bins hold a segment of fewer than 8 bins or more than 14 segments
// of one mode, or a value is infinite, NaN or beyond the exponents handled, they are
// evaluated in FP64 (dense_direct).
//
// Work.  An item is (walker group, tile of consecutive bins inside the group's union band);
// blocks are persistent and pull items from a counter.  An item is split into units of 128
// bins and two walkers, one warp each; a lane has 4 consecutive bins.  Nothing but the
// phasor table (one TMA bulk copy per block) is shared between warps, so they meet only at
// the end of an item.  The mode sums of a warp's bins are kept in shared memory (6 KB): the
// loop over a lane's bins is then a loop in the code too, which stays within the
// instruction cache, and 128 registers hold the 7 cubics and the phase (16 warps per SM).
// With the sums in registers (the bins unrolled, 8 warps per SM, 255 registers) a third of
// all issue slots waited for instructions: 428 ms against 219 (below).  The data rows (76 bytes
// per bin, float pairs) are read from L2 by each walker.
//
// Bound by the multiply-add pipe and the waits between dependent instructions (pipe 67 % busy,
// 56 % of issue slots, 2.1 warps waiting per issue): per (walker, mode, bin) the method takes 84
// products, and 183 instructions of the multiply-add's opcode are executed, moves and parts of
// 64-bit additions among them.  1024 walkers, six modes, 1-yr grid: 951 -> 215.5 ms; 37 walkers,
// four modes, quarter-year grid: 2063 -> 887 us; one walker, (2,2), 30 days: 61 -> 35 us.
#include "f32x2.cuh"
#include "fixed.cuh"
#include "kernels.h"
#include "model.cuh"
#include "tma.cuh"

namespace lisa {

namespace {

constexpr int kC = kFxRows;    // consecutive bins of a thread
constexpr int kBlk = 32 * kC;  // bins of a warp: one block of expansions
constexpr int kWarps = 8;      // warps per block
constexpr int kTasks = 14;     // expansions a warp holds at a time
constexpr int kSer = 7;        // A, then Re/Im of T^A, T^E, T^T
constexpr int kABits = 62, kTBits = 61;  // A is scaled below 2^62, T below 2^61
constexpr int kNoScale = -10000;
// Shortest segment for the expansions: over a bin or more per segment the differences no
// longer fall with their order.
constexpr int kMinSeg = 8;
// Bits that the bounds of an amplitude and of a transfer together may lie above their values where
// the expansion begins: the sums' unit is then at most 2^(kLoose - 53) of that product.  4 bits on most
// segments and up to 9 from 64 knots up; with 4 to 32 knots and a few bins below the first bin
// (f0 / df < 30) up to 17.
constexpr int kLoose = 12;

// One (mode, segment) in a warp's block of bins, at the block's first bin or 3 bins before
// the segment's first one (a thread's 4 bins may begin there): value and forward differences of the
// seven series in fixed point, and (index kSer) of the phase in fractions of a turn scaled by
// 2^64; lo and low hold the next 32 bits of the differences.  A series is read by three loads, of 16, 16
// and 8 bytes (its differences in arrays of their own, by five: 218.3 against 215.5 ms of 1024
// walkers, 925 against 887 us of 37, and up to 15 % of calls with many short segments).
struct __align__(16) Expand {
    i64 vd[kSer + 1][2];  // value, first difference
    i64 dd[kSer + 1][2];  // second, third difference
    uint2 lo[kSer];       // of the second and the third
    uint32_t low[3];
    int org, kb, next;    // origin, first bin of the segment and of the next one
};
static_assert(sizeof(Expand) == 336, "16-byte loads of a series' value and first difference");

struct Phase64 {
    unsigned long long ph, d1, d2, d3;
};

// shared memory of a warp
struct WarpMem {
    i64 H[kC][6][32];  // the mode sums of each thread's bins
    i64 z[kC][2][32];  // e^{i phase} of each thread's bins, for modes with the same phase
    Expand ex[kTasks];
};

struct SmemF64 {
    FxTab tab[kFxTab];
    WarpMem w[kWarps];
};

}  // namespace

__device__ __forceinline__ double bin_freq_d(double f0, double df, int j) {
    return __dadd_rn(f0, __dmul_rn((double)j, df));
}

// fixed-point forward differences of a segment's phase moved to bin n of the segment
// (Newton's forward-difference formula in modular arithmetic; for n > 0 the low words
// add the carries of the 128-bit products; n >= -8)
__device__ __forceinline__ Phase64 phase64_at(const unsigned long long *__restrict__ r, int n) {
    const ulonglong2 a = __ldg(reinterpret_cast<const ulonglong2 *>(r));
    const ulonglong2 b = __ldg(reinterpret_cast<const ulonglong2 *>(r) + 1);
    const long long nn = n;
    const unsigned long long c1 = (unsigned long long)nn;
    const unsigned long long c2 = (unsigned long long)(nn * (nn - 1)) >> 1;
    const unsigned long long c3 = (c2 * (unsigned long long)(nn - 2)) * 0xAAAAAAAAAAAAAAABull;
    Phase64 p;
    p.ph = a.x + c1 * a.y + c2 * b.x + c3 * b.y;
    p.d1 = a.y + c1 * b.x + c2 * b.y;
    p.d2 = b.x + c1 * b.y;
    p.d3 = b.y;
    if (n > 0) {
        const ulonglong2 c = __ldg(reinterpret_cast<const ulonglong2 *>(r) + 2);
        const ulonglong2 e = __ldg(reinterpret_cast<const ulonglong2 *>(r) + 3);
        p.ph += __umul64hi(c1, c.x) + __umul64hi(c2, c.y) + __umul64hi(c3, e.x);
        p.d1 += __umul64hi(c1, c.y) + __umul64hi(c2, e.x);
        p.d2 += __umul64hi(c1, e.x);
    }
    return p;
}

// segment of bin j: kb[s] <= j < kb[s + 1] (the last one open), from the log spacing of the
// knots moved by the integer knot-to-bin boundaries
__device__ __forceinline__ int segment_at(const int *__restrict__ kb, int K, int j, float f, float l0,
                                          float scale) {
    int s = (int)fmaf(__log2f(f), scale, -l0);
    s = min(max(s, 0), K - 2);
    while (s > 0 && __ldg(kb + s) > j) s--;
    while (s < K - 2 && __ldg(kb + s + 1) <= j) s++;
    return s;
}

// group of a work item: largest g with item_start[g] <= item
__device__ __forceinline__ int group_of(const int *__restrict__ item_start, int ng, int item) {
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

// ------------------------------------------------------------------ FP64 evaluation
// Bins [j0, j1) of one walker in FP64 from the staged rows in global memory: segments too
// short for the expansions, and values outside them.
__device__ __noinline__ double2 dense_direct(const StageDims &d, const StageBufs &b,
                                             const unsigned long long *__restrict__ segs,
                                             const double *__restrict__ bins, int w, int j0, int j1,
                                             const int *slo, const int *shi) {
    double dh = 0.0, hh = 0.0;
    const int K = d.K;
    for (int j = j0; j < j1; j++) {
        const double f = bin_freq_d(d.f0, d.df, j);
        double h[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (int mi = 0; mi < d.L; mi++) {
            if (j < slo[mi] || j > shi[mi]) continue;
            const size_t wm = (size_t)w * d.L + mi;
            const int *kb = b.kb + wm * K;
            int lo = 0, hi = K - 2;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (kb[mid] <= j)
                    lo = mid;
                else
                    hi = mid - 1;
            }
            const unsigned long long *rec = segs + kPhaseWords * (wm * (K - 1) + lo);
            const double *c = b.coef + (wm * (K - 1) + lo) * 32;
            const double x = f - b.fk[wm * K + lo];
            double sn, cs;
            sincospi((double)(long long)phase64_at(rec, j - kb[lo]).ph * 0x1p-63, &sn, &cs);
            const double amp = fma(x, fma(x, fma(x, c[3], c[2]), c[1]), c[0]);
            const double zr = amp * cs, zi = amp * sn;
            for (int ch = 0; ch < 3; ch++) {
                const double *r = c + 8 + 8 * ch, *m = r + 4;
                const double tr = fma(x, fma(x, fma(x, r[3], r[2]), r[1]), r[0]);
                const double ti = fma(x, fma(x, fma(x, m[3], m[2]), m[1]), m[0]);
                h[2 * ch] = fma(tr, zr, fma(-ti, zi, h[2 * ch]));
                h[2 * ch + 1] = fma(tr, zi, fma(ti, zr, h[2 * ch + 1]));
            }
        }
        const double *o = bins + (size_t)j * kBinDoubles;
        for (int ch = 0; ch < 3; ch++) {
            const double hr = h[2 * ch], hi = h[2 * ch + 1];
            hh = fma(o[ch], fma(hr, hr, hi * hi), hh);
            dh = fma(o[3 + 2 * ch], hr, fma(o[4 + 2 * ch], hi, dh));
        }
    }
    return make_double2(dh, hh);
}

// ------------------------------------------------------------------ data rows
// A double scaled by 2^-e as a pair of floats, hi truncated to 24 bits and lo the next 24
// (|v| < 2^e; values below 2^-76 are dropped)
__device__ __forceinline__ void split_double(double v, int e, float &hi, float &lo) {
    const long long b = __double_as_longlong(v);
    const int de = (int)((b >> 52) & 0x7ff) - 1022 - e;  // <= 0; v = m 2^(de - 53) 2^e
    const unsigned int mh = (unsigned int)(b >> 29) & 0x7fffffu;
    const unsigned int ml = (unsigned int)b & 0x1fffffffu;
    const unsigned int sign = (unsigned int)(b >> 32) & 0x80000000u;
    const bool keep = de > -76 && ((b >> 52) & 0x7ff) != 0;
    hi = keep ? __uint_as_float(sign | (unsigned int)(126 + de) << 23 | mh) : 0.0f;
    const float l = (float)ml * __uint_as_float((unsigned int)max(126 + 1 + de - 53, 0) << 23);
    lo = keep ? __uint_as_float(__float_as_uint(l) | sign) : 0.0f;
}

// Rows of kFxRows bins of 9 doubles (w_A, w_E, w_T, (w d)_A re, im, ...) in the form the dense
// kernel uses: per row 18 floats, (w hi, w lo) of the three channels, then (re hi, im hi, re
// lo, im lo) of each w d, channel c scaled by 2^-ew[c] and 2^-ed[c], the largest exponents of
// the rows; and the exponents.  Rows past the data become zero.
struct FxRows {
    float v[kFxRows][2 * kBinDoubles];
    int ew[3], ed[3];
    bool ok;  // false: a value is infinite, NaN or out of range
};

__device__ __forceinline__ FxRows split_rows(const double *__restrict__ p, int rows) {
    FxRows f;
    f.ok = true;
    // a thread's rows are 288 contiguous bytes, the threads' 288 apart: 16-byte loads take half as
    // many passes through L1 as 8-byte ones, where the caller's rows are aligned to them (one walker
    // on the 1-yr grid with the caller's rows, one mode: 204 -> 163 us)
    double row[kFxRows * kBinDoubles];
    if (rows == kFxRows && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
#pragma unroll
        for (int i = 0; i < kFxRows * kBinDoubles / 2; i++) {
            const double2 v = __ldg(reinterpret_cast<const double2 *>(p) + i);
            row[2 * i] = v.x;
            row[2 * i + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < kFxRows * kBinDoubles; i++) row[i] = i < rows * kBinDoubles ? p[i] : 0.0;
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
        f.ew[c] = f.ed[c] = -2000;
#pragma unroll
        for (int r = 0; r < kFxRows; r++) {
            if (r >= rows) break;
            const double *o = row + r * kBinDoubles;
            f.ew[c] = max(f.ew[c], exponent_of(o[c]));
            f.ed[c] = max(f.ed[c], max(exponent_of(o[3 + 2 * c]), exponent_of(o[4 + 2 * c])));
        }
        f.ok = f.ok && max(f.ew[c], f.ed[c]) < 1025 && (f.ew[c] > -900 || f.ew[c] == -2000) &&
               (f.ed[c] > -900 || f.ed[c] == -2000);
    }
#pragma unroll
    for (int r = 0; r < kFxRows; r++)
#pragma unroll
        for (int q = 0; q < kBinDoubles; q++) {
            const int c = q < 3 ? q : (q - 3) >> 1, im = (q - 3) & 1;
            float h = 0.0f, l = 0.0f;
            if (f.ok && r < rows) split_double(row[r * kBinDoubles + q], q < 3 ? f.ew[c] : f.ed[c], h, l);
            if (q < 3) {
                f.v[r][2 * q] = h;
                f.v[r][2 * q + 1] = l;
            } else {
                f.v[r][6 + 4 * c + im] = h;
                f.v[r][6 + 4 * c + 2 + im] = l;
            }
        }
    return f;
}

// exponents as six signed 16-bit numbers and the flag, in one 16-byte word
__device__ __forceinline__ int4 pack_exponents(const FxRows &f) {
    auto two = [](int a, int b) { return (a & 0xffff) | (int)((unsigned int)b << 16); };
    return make_int4(two(f.ew[0], f.ew[1]), two(f.ew[2], f.ed[0]), two(f.ed[1], f.ed[2]), f.ok ? 1 : 0);
}

// One thread per kFxRows bins; 16-byte word u of rows c goes to ((c / 32) kFxWords + u) 32 + c % 32,
// so that a warp whose threads take consecutive rows reads every word coalesced.
__global__ void __launch_bounds__(128) prep_fx_kernel(const double *__restrict__ bins, int N,
                                                      float4 *__restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = c * kFxRows;
    if (c >= fx_chunks(N)) return;
    const FxRows f = split_rows(bins + (size_t)j * kBinDoubles, min(max(N - j, 0), kFxRows));
    const float *v = &f.v[0][0];
    float4 *o = out + (size_t)(c >> 5) * kFxWords * 32 + (c & 31);
#pragma unroll
    for (int u = 0; u < kFxWords - 1; u++) o[u * 32] = make_float4(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
    const int4 e = pack_exponents(f);
    o[(kFxWords - 1) * 32] = make_float4(__int_as_float(e.x), __int_as_float(e.y), __int_as_float(e.z),
                                         __int_as_float(e.w));
}

cudaError_t launch_prep_fx(const double *bins, int N, float4 *out, cudaStream_t s) {
    prep_fx_kernel<<<(fx_chunks(N) + 127) / 128, 128, 0, s>>>(bins, N, out);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ expansions
// A cubic of a segment, in x from its knot, and its forward differences over one bin at x
__device__ __forceinline__ void differences(const double2 *__restrict__ c2, int row, double x, double df,
                                            double d[4]) {
    const double2 lo = __ldg(c2 + 2 * row), hi = __ldg(c2 + 2 * row + 1);
    const double t = 3.0 * hi.y, df2 = df * df;
    const double p1 = fma(x, fma(x, t, hi.x + hi.x), lo.y) * df;
    const double p2 = fma(x, t, hi.x) * df2, p3 = hi.y * (df2 * df);
    d[0] = fma(x, fma(x, fma(x, hi.y, hi.x), lo.y), lo.x);
    d[1] = p1 + p2 + p3;
    d[2] = 2.0 * fma(3.0, p3, p2);
    d[3] = 6.0 * p3;
}

// m with |v| < 2^m over 2^n1 bins, |v| <= |d0| + n |d1| + n^2/2 |d2| + n^3/6 |d3|
__device__ __forceinline__ int bound_of(const double d[4], int n1) {
    return max(max(exponent_of(d[0]), exponent_of(d[1]) + n1),
               max(exponent_of(d[2]) + 2 * n1 - 1, exponent_of(d[3]) + 3 * n1 - 2)) +
           2;
}

// series q of an expansion, left as the doubles of differences() and their bound, in fixed
// point scaled by 2^s
__device__ __forceinline__ void series_put(Expand *e, int q, const double d[4], int bound) {
    e->vd[q][0] = __double_as_longlong(d[0]);
    e->vd[q][1] = __double_as_longlong(d[1]);
    e->dd[q][0] = __double_as_longlong(d[2]);
    e->dd[q][1] = __double_as_longlong(d[3]);
    e->lo[q].x = (uint32_t)bound;
}

__device__ __forceinline__ void series_fix(Expand *e, int q, int s) {
    e->vd[q][0] = to_fixed(__longlong_as_double(e->vd[q][0]), s);
    e->vd[q][1] = to_fixed(__longlong_as_double(e->vd[q][1]), s);
    uint2 lo;
    e->dd[q][0] = to_fixed96(__longlong_as_double(e->dd[q][0]), s, lo.x);
    e->dd[q][1] = to_fixed96(__longlong_as_double(e->dd[q][1]), s, lo.y);
    e->lo[q] = lo;
}

struct Diff {
    i64 v, d1, d2;
};

// series q n >= 0 bins from its origin; c2 = n(n-1)/2, c3 = n(n-1)(n-2)/6
__device__ __forceinline__ Diff series_at(const Expand *__restrict__ e, int q, uint32_t n, uint32_t c2,
                                          uint32_t c3) {
    const longlong2 a = *reinterpret_cast<const longlong2 *>(e->vd[q]);
    const longlong2 dd = *reinterpret_cast<const longlong2 *>(e->dd[q]);
    const i64 d2 = dd.x, d3 = dd.y;
    const uint2 lo = e->lo[q];
    Diff r;
    i64 v = mad_u((uint32_t)a.y, n, a.x);
    v = mad_u((uint32_t)d2, c2, v);
    v = mad_u((uint32_t)d3, c3, v);
    v += (i64)(__umulhi(c2, lo.x) + __umulhi(c3, lo.y));
    r.v = add_hi(v, (uint32_t)(a.y >> 32) * n + (uint32_t)(d2 >> 32) * c2 + (uint32_t)(d3 >> 32) * c3);
    i64 d1 = mad_u((uint32_t)d2, n, a.y);
    d1 = mad_u((uint32_t)d3, c2, d1);
    r.d1 = add_hi(d1, (uint32_t)(d2 >> 32) * n + (uint32_t)(d3 >> 32) * c2);
    r.d2 = add_hi(mad_u((uint32_t)d3, n, d2), (uint32_t)(d3 >> 32) * n);
    return r;
}

// the phase n >= 0 bins from its origin
__device__ __forceinline__ void phase_at(const Expand *__restrict__ e, uint32_t n, uint32_t c2, uint32_t c3,
                                         i64 p[4]) {
    const longlong2 a = *reinterpret_cast<const longlong2 *>(e->vd[kSer]);
    const longlong2 dd = *reinterpret_cast<const longlong2 *>(e->dd[kSer]);
    const i64 d2 = dd.x, d3 = dd.y;
    i64 v = mad_u((uint32_t)a.y, n, a.x);
    v = mad_u((uint32_t)d2, c2, v);
    v = mad_u((uint32_t)d3, c3, v);
    v += (i64)__umulhi(n, e->low[0]) + (i64)(__umulhi(c2, e->low[1]) + __umulhi(c3, e->low[2]));
    p[0] = add_hi(v, (uint32_t)(a.y >> 32) * n + (uint32_t)(d2 >> 32) * c2 + (uint32_t)(d3 >> 32) * c3);
    i64 d1 = mad_u((uint32_t)d2, n, a.y);
    d1 = mad_u((uint32_t)d3, c2, d1);
    p[1] = add_hi(d1, (uint32_t)(d2 >> 32) * n + (uint32_t)(d3 >> 32) * c2);
    p[2] = add_hi(mad_u((uint32_t)d3, n, d2), (uint32_t)(d3 >> 32) * n);
    p[3] = d3;
}

// ------------------------------------------------------------------ integrand
// Sums begin at half a unit of fixed_pair, which cuts off what is below: it rounds then
constexpr i64 kHalf = 4;

// x - kHalf as two floats, x 2^-27 = a + b 2^-24 to a unit of 2^3 in x.  |x| < 2^58: a cubic stays below
// 0.92 of its bound (bound_of), so a mode's |A T| below 1.2 2^55 units, and there are six
__device__ __forceinline__ void fixed_pair(i64 x, float &a, float &b) {
    const int hi = (int)(x >> 27);
    a = __int2float_rn(hi);
    const int rest = hi - __float2int_rn(a);  // |rest| <= 64
    // (rest 2^27 + low 27 bits) 2^-3, at most 2^30 + 2^24
    const int r = (int)(((unsigned int)rest << 24) + (((unsigned int)x & 0x7ffffffu) >> 3));
    b = __int2float_rn(r);
}

// q + e added to the pair sum + comp: the error of the sum is exact (two-sum)
__device__ __forceinline__ void add_pair(float2 &sum, float2 &comp, float2 q, float2 e) {
    const float2 t = add2(sum, q);
    const float2 z = sub2(t, sum);
    const float2 err = add2(sub2(sum, sub2(t, z)), sub2(q, z));
    comp = add2(comp, add2(err, e));
    sum = t;
}

// the two halves of a pair sum together, times 2^k
__device__ __forceinline__ double scaled_sum(float2 sum, float2 comp, int k) {
    const float t = sum.x + sum.y, z = t - sum.x;
    const float err = (sum.x - (t - z)) + (sum.y - z);
    const double v = (double)t + (double)(err + (comp.x + comp.y));
    return abs(k) < 1000 ? v * __hiloint2double((1023 + k) << 20, 0) : ldexp(v, k);
}

__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// G walkers per group; kRaw: data rows converted from the FP64 rows as they are used (callers
// that bring their own rows) instead of read in the dense kernel's form.
template <int G, bool kRaw>
__global__ void __launch_bounds__(32 * kWarps, 2) dense_f64_kernel(StageDims d, StageBufs b,
                                                                const unsigned long long *__restrict__ segs,
                                                                const double *__restrict__ bins,
                                                                const float4 *__restrict__ rows,
                                                                int tile_bins) {
    constexpr int NS = G == 1 ? 1 : 2;  // walkers expanded together: their modes share a warp
    extern __shared__ __align__(128) unsigned char smem[];
    SmemF64 &sm = *reinterpret_cast<SmemF64 *>(smem);
    __shared__ __align__(8) uint64_t bar;
    __shared__ int s_item, s_walker[G], s_wlo[G], s_whi[G], s_lo[G][kMaxModes], s_hi[G][kMaxModes];
    __shared__ float s_g0[G][kMaxModes], s_g1[G][kMaxModes];
    __shared__ int s_task[kWarps][kTasks];
    __shared__ int s_first[kWarps][kMaxModes * NS];  // first expansion of a (walker, mode), its count
    __shared__ double s_sum[kWarps][G][2];           // <d|h>, <h|h> of the item by each warp
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    WarpMem &wm_ = sm.w[warp];
    Expand *ex = wm_.ex;
    if (tid == 0) mbar_init(&bar, 1);
    __syncthreads();
    const int ng = n_groups(d.B, G);
    const int total = b.item_start[ng];
    const int K = d.K, L = d.L;
    const float f0f = (float)d.f0, dff = (float)d.df;
    bool staged = false;
    for (;;) {
        __syncthreads();
        if (tid == 0) s_item = atomicAdd(b.counter, 1);
        __syncthreads();
        const int item = s_item;
        if (item >= total) return;
        if (!staged) {
            // the phasor table by one bulk copy; every thread waits, and the block leaves
            // together if the copy never completed
            if (tid == 0) {
                if (b.wait_test_polls == 0)
                    tma_load_1d(sm.tab, b.fxtab, sizeof(sm.tab), &bar);
                else
                    mbar_expect_tx(&bar, sizeof(sm.tab));  // test of the give-up path: no copy is issued
            }
            const uint32_t polls = b.wait_test_polls ? b.wait_test_polls : kWaitPolls;
            if (!__syncthreads_and(mbar_wait_bounded(&bar, 0, b.err, polls))) return;
            staged = true;
        }
        const int g = group_of(b.item_start, ng, item);
        const int J0 = b.grange[2 * g] + (item - b.item_start[g]) * tile_bins;
        const int Jitem = min(J0 + tile_bins, b.grange[2 * g + 1] + 1);
        if (tid < G) {
            const int i = g * G + tid, w = i < d.B ? b.order[i] : -1;
            s_walker[tid] = w;
            s_wlo[tid] = w < 0 ? 0 : b.wrange[2 * w];
            s_whi[tid] = w < 0 ? -1 : b.wrange[2 * w + 1];
        }
        if (tid < G * kMaxModes) {
            const int k = tid / kMaxModes, mi = tid % kMaxModes;
            const int i = g * G + k;
            int lo = 1, hi = 0;
            float g0 = 0.0f, g1 = 0.0f;
            if (i < d.B && mi < L) {
                const int w = b.order[i];
                const size_t wm = (size_t)w * L + mi;
                const int *bd = b.band + wm * 3;
                if (b.valid[w] && bd[0]) {
                    lo = bd[1];
                    hi = bd[2];
                    const unsigned long long *r = segs + kPhaseWords * (wm * (K - 1)) + 7;
                    g0 = __uint_as_float((unsigned int)(__ldg(r) >> 32));
                    g1 = __uint_as_float((unsigned int)(__ldg(r + kPhaseWords) >> 32));
                }
            }
            s_lo[k][mi] = lo;
            s_hi[k][mi] = hi;
            s_g0[k][mi] = g0;
            s_g1[k][mi] = g1;
        }
        if (lane < G) s_sum[warp][lane][0] = s_sum[warp][lane][1] = 0.0;
        __syncthreads();

        const int nblk = (Jitem - J0 + kBlk - 1) / kBlk;
        for (int unit0 = warp; unit0 < nblk * (G / NS); unit0 += kWarps) {
            const int Jw = J0 + (unit0 % nblk) * kBlk, kp = unit0 / nblk * NS;
            const int Jend = min(Jw + kBlk, Jitem);
            const int j0 = Jw + lane * kC;
            {
                // lanes 0 .. NS L - 1: the segments that a walker's mode has in the warp's bins
                int s0 = 0, cnt = 0;
                if (lane < NS * L) {
                    const int k = kp + lane / L, mi = d.ord[lane % L];
                    const int ja = max(Jw, s_lo[k][mi]), jb = min(Jend, s_hi[k][mi] + 1);
                    if (ja < jb) {
                        const int *kb = b.kb + ((size_t)s_walker[k] * L + mi) * K;
                        s0 = segment_at(kb, K, ja, fmaf((float)ja, dff, f0f), s_g0[k][mi], s_g1[k][mi]);
                        int s1 = s0;
                        while (s1 < K - 2 && __ldg(kb + s1 + 1) < jb) s1++;
                        cnt = s1 - s0 + 1;
                    }
                }
                int upto = cnt;
                for (int o = 1; o < kMaxModes * NS; o <<= 1) {
                    const int u = __shfl_up_sync(0xffffffffu, upto, o);
                    if (lane >= o) upto += u;
                }
                int have = 0;  // (walker, mode) units expanded so far
                // scale of each channel's sums (units of 2^(E - 55)), of this walker and the next;
                // and whether a walker's bins here go to the FP64 evaluation
                int E[3] = {kNoScale, kNoScale, kNoScale}, En[3] = {kNoScale, kNoScale, kNoScale};
                bool direct = false, directn = false;
#pragma unroll 1
                for (int sub = 0; sub < NS; sub++) {
                    const int k = kp + sub, w = s_walker[k];
                    if (s_whi[k] < Jw || s_wlo[k] >= Jend) {  // nothing of this walker here
                        have = max(have, (sub + 1) * L);
                        continue;
                    }
#pragma unroll
                    for (int i = 0; i < kC; i++)
#pragma unroll
                        for (int q = 0; q < 6; q++) wm_.H[i][q][lane] = kHalf;
#pragma unroll 1
                    for (int pos = 0; pos < L; pos++) {
                        const int unit = sub * L + pos, mi = d.ord[pos];
                        if (direct) break;
                        if (unit >= have) {
                            // expand as many units from here on as fit
                            const int base = __shfl_sync(0xffffffffu, upto - cnt, unit);
                            const unsigned fit =
                                __ballot_sync(0xffffffffu, lane >= unit && lane < NS * L && upto - base <= kTasks);
                            if (!fit) {  // one mode alone has too many segments here
                                direct = true;
                                break;
                            }
                            have = unit + __popc(fit);
                            const int tasks = __shfl_sync(0xffffffffu, upto, have - 1) - base;
                            __syncwarp();
                            if (lane >= unit && lane < have) {
                                const int first = upto - cnt - base;
                                for (int i = 0; i < cnt; i++) s_task[warp][first + i] = lane | (s0 + i) << 4;
                                s_first[warp][lane] = first | cnt << 8;
                            }
                            __syncwarp();
                            if (lane < tasks) {
                                const int t = s_task[warp][lane], u = t & 15, seg = t >> 4;
                                const size_t wm = (size_t)s_walker[kp + u / L] * L + d.ord[u % L];
                                Expand *e = ex + lane;
                                const int *kb = b.kb + wm * K;
                                const int k0 = __ldg(kb + seg);
                                const int k1 =
                                    seg < K - 2 ? __ldg(kb + seg + 1) : s_hi[kp + u / L][d.ord[u % L]] + 1;
                                // a band may begin one bin below its first knot's (1e-9 bins of
                                // slack): no thread starts more than 3 bins before the lower of the two
                                const int b0 = min(k0, s_lo[kp + u / L][d.ord[u % L]]);
                                const int org = max(Jw, (seg == 0 ? b0 : k0) - (kC - 1)), nn = org - k0;
                                e->org = org;
                                e->kb = k0;
                                e->next = k1;
                                const unsigned long long *r = segs + kPhaseWords * (wm * (K - 1) + seg);
                                const Phase64 p = phase64_at(r, nn);
                                const i64 c2 = (i64)nn * (nn - 1) / 2;
                                e->vd[kSer][0] = p.ph;
                                e->vd[kSer][1] = p.d1;
                                e->dd[kSer][0] = p.d2;
                                e->dd[kSer][1] = p.d3;
                                e->low[0] = (uint32_t)((r[4] + (i64)nn * r[5] + c2 * r[6]) >> 32);
                                e->low[1] = (uint32_t)((r[5] + (i64)nn * r[6]) >> 32);
                                e->low[2] = (uint32_t)(r[6] >> 32);
                            }
                            __syncwarp();
                            // every lane one (expansion, series) at a time: FP64 instructions cost a
                            // full warp's time however few lanes take part
                            for (int i = lane; i < tasks * kSer; i += 32) {
                                Expand *e = ex + i / kSer;
                                const int q = i % kSer;
                                const int t = s_task[warp][i / kSer], u = t & 15, seg = t >> 4;
                                const size_t wm = (size_t)s_walker[kp + u / L] * L + d.ord[u % L];
                                const double x = bin_freq_d(d.f0, d.df, e->org) - __ldg(b.fk + wm * K + seg);
                                const double2 *cf =
                                    reinterpret_cast<const double2 *>(b.coef + (wm * (size_t)(K - 1) + seg) * 32);
                                double dd[4];
                                differences(cf, q == 0 ? 0 : q + 1, x, d.df, dd);  // series 1 is the phase
                                const int n1 = 32 - __clz(max(min(e->next, Jw + kBlk) - e->org - 1, 15));
                                series_put(e, q, dd, bound_of(dd, n1));
                            }
                            __syncwarp();
                            int ea = -5000, et[3] = {-5000, -5000, -5000}, ts = 0;
                            bool bad = false;
                            if (lane < tasks) {
                                const Expand *e = ex + lane;
                                ts = (s_task[warp][lane] & 15) / L;
                                ea = (int)e->lo[0].x;
                                auto at0 = [&](int q) { return exponent_of(__longlong_as_double(e->vd[q][0])); };
                                int top = ea, loose = 0;
#pragma unroll
                                for (int c = 0; c < 3; c++) {
                                    et[c] = max((int)e->lo[1 + 2 * c].x, (int)e->lo[2 + 2 * c].x);
                                    top = max(top, et[c]);
                                    if (et[c] > -1900)  // not all zero
                                        loose = max(loose, et[c] - max(at0(1 + 2 * c), at0(2 + 2 * c)));
                                }
                                // a short segment, an infinite or NaN coefficient, or bounds far
                                // above the values
                                if (ea > -1900) loose += ea - at0(0);
                                bad = e->next - e->kb < kMinSeg || top > 900 || loose > kLoose;
                            }
                            const unsigned wrong = __ballot_sync(0xffffffffu, bad);
                            const unsigned of_next = __ballot_sync(0xffffffffu, lane < tasks && ts > sub);
                            directn = directn || (wrong & of_next);
                            if (wrong & ~of_next) {
                                direct = true;
                                break;
                            }
                            int sc[3];
#pragma unroll
                            for (int c = 0; c < 3; c++) {
                                const int v = ea + et[c];
                                const int m = __reduce_max_sync(0xffffffffu, lane < tasks && ts == sub ? v : kNoScale);
                                const int mn = __reduce_max_sync(0xffffffffu, lane < tasks && ts > sub ? v : kNoScale);
                                if (m > E[c]) {
                                    if (pos > 0 && E[c] > kNoScale)
                                        for (int i = 0; i < kC; i++)
                                            for (int q = 2 * c; q < 2 * c + 2; q++) {
                                                i64 &h = wm_.H[i][q][lane];
                                                h = ((h - kHalf) >> min(m - E[c], 63)) + kHalf;
                                            }
                                    E[c] = m;
                                }
                                En[c] = max(En[c], mn);
                                sc[c] = ts > sub ? En[c] : E[c];
                            }
                            if (lane < tasks) {  // the binary scale of every series
                                Expand *e = ex + lane;
                                e->lo[0].x = (uint32_t)(kABits - ea);
#pragma unroll
                                for (int q = 1; q < kSer; q++)
                                    e->lo[q].x = (uint32_t)(kTBits - (sc[(q - 1) >> 1] - ea));
                            }
                            __syncwarp();
                            for (int i = lane; i < tasks * kSer; i += 32)
                                series_fix(ex + i / kSer, i % kSer, (int)ex[i / kSer].lo[i % kSer].x);
                            __syncwarp();
                        }
                        const int fc = s_first[warp][unit];
                        const Expand *e = ex + (fc & 0xff), *eend = e + (fc >> 8);
                        const int ja = max(j0, s_lo[k][mi]), jb = min(min(j0 + kC, Jend), s_hi[k][mi] + 1);
                        if (ja >= jb) continue;
                        while (e->next <= ja) e++;
                        int from = ja;
                        for (; from < jb && e < eend; e++) {  // usually one segment
                            const int to = min(jb, e->next), ka = from - j0, kz = to - j0;
                            if (ka >= kz) continue;  // a segment without bins
                            from = to;
                            const uint32_t n0 = j0 - e->org, c2 = n0 * (n0 - 1) / 2, c3 = c2 * (n0 - 2) / 3;
                            i64 ph[4] = {0, 0, 0, 0};
                            const bool same = d.same[pos] != 0;  // the phase of the mode before
                            if (!same) phase_at(e, n0, c2, c3, ph);
                            Diff s[kSer];
#pragma unroll
                            for (int q = 0; q < kSer; q++) s[q] = series_at(e, q, n0, c2, c3);
#pragma unroll 1
                            for (int i = 0; i < kC; i++) {
                                if (i >= ka && i < kz) {
                                    i64 pr, pi;
                                    if (same) {
                                        pr = wm_.z[i][0][lane];
                                        pi = wm_.z[i][1][lane];
                                    } else {
                                        fx_rotate(ph[0], sm.tab[fx_cell(ph[0])], pr, pi);
                                        wm_.z[i][0][lane] = pr;
                                        wm_.z[i][1][lane] = pi;
                                    }
                                    const Bal a = bal(s[0].v);
                                    const i64 ar = mulhi(a, bal(pr)), ai = mulhi(a, bal(pi));
                                    const Bal zr = bal(ar), zi = bal(ai), zn = bal(-ai);  // A e^{i phase}
#pragma unroll
                                    for (int c = 0; c < 3; c++) {
                                        const Bal r = bal(s[1 + 2 * c].v), m = bal(s[2 + 2 * c].v);
                                        i64 h0 = wm_.H[i][2 * c][lane], h1 = wm_.H[i][2 * c + 1][lane];
                                        i64 x0 = (i64)r.h * zr.l, x1 = (i64)r.h * zi.l;
                                        x0 = mad_s(r.l, zr.h, x0);
                                        x1 = mad_s(r.l, zi.h, x1);
                                        x0 = mad_s(m.h, zn.l, x0);
                                        x1 = mad_s(m.h, zr.l, x1);
                                        x0 = mad_s(m.l, zn.h, x0);
                                        x1 = mad_s(m.l, zr.h, x1);
                                        h0 += x0 >> 32;
                                        h1 += x1 >> 32;
                                        h0 = mad_s(r.h, zr.h, h0);
                                        h1 = mad_s(r.h, zi.h, h1);
                                        h0 = mad_s(m.h, zn.h, h0);
                                        h1 = mad_s(m.h, zr.h, h1);
                                        wm_.H[i][2 * c][lane] = h0;
                                        wm_.H[i][2 * c + 1][lane] = h1;
                                    }
                                }
                                // only what the bins to come need: six of twelve additions
                                if (i < kC - 1) {
                                    ph[0] += ph[1];
#pragma unroll
                                    for (int q = 0; q < kSer; q++) s[q].v += s[q].d1;
                                }
                                if (i < kC - 2) {
                                    ph[1] += ph[2];
#pragma unroll
                                    for (int q = 0; q < kSer; q++) s[q].d1 += s[q].d2;
                                }
                                if (i < kC - 3) {
                                    ph[2] += ph[3];
#pragma unroll
                                    for (int q = 0; q < kSer; q++) s[q].d2 += e->dd[q][1];
                                }
                            }
                        }
                    }

                    double dh = 0.0, hh = 0.0;
                    const int mine = min(max(Jend - j0, 0), kC);  // this thread's rows
                    bool here = !direct && mine > 0;
                    float2 hs[3], hc[3], ds[3], dc[3];
                    int ew[3] = {0, 0, 0}, ed[3] = {0, 0, 0};
                    FxRows raw;
                    const float4 *src = rows + (size_t)(j0 >> 7) * kFxWords * 32 + ((j0 >> 2) & 31);
                    if (here) {
                        if (kRaw) {
                            raw = split_rows(bins + (size_t)j0 * kBinDoubles, mine);
                            here = raw.ok;
#pragma unroll
                            for (int c = 0; c < 3; c++) {
                                ew[c] = raw.ew[c];
                                ed[c] = raw.ed[c];
                            }
                        } else {
                            const int4 e4 = __ldg(reinterpret_cast<const int4 *>(src) + (kFxWords - 1) * 32);
                            here = e4.w != 0;
                            ew[0] = (e4.x << 16) >> 16;
                            ew[1] = e4.x >> 16;
                            ew[2] = (e4.y << 16) >> 16;
                            ed[0] = e4.y >> 16;
                            ed[1] = (e4.z << 16) >> 16;
                            ed[2] = e4.z >> 16;
                        }
                    }
                    if (here) {
#pragma unroll
                        for (int c = 0; c < 3; c++) hs[c] = hc[c] = ds[c] = dc[c] = make_float2(0.0f, 0.0f);
#pragma unroll(kRaw ? 2 : 1)
                        for (int i2 = 0; i2 < kC / 2; i2++) {
                            // two rows: nine 16-byte words
                            float o[4 * kBinDoubles];
#pragma unroll
                            for (int q = 0; q < kBinDoubles; q++) {
                                if (kRaw) {
#pragma unroll
                                    for (int u = 0; u < 4; u++) o[4 * q + u] = (&raw.v[0][0])[36 * i2 + 4 * q + u];
                                } else {
                                    const float4 v = __ldg(src + (kBinDoubles * i2 + q) * 32);
                                    o[4 * q] = v.x;
                                    o[4 * q + 1] = v.y;
                                    o[4 * q + 2] = v.z;
                                    o[4 * q + 3] = v.w;
                                }
                            }
#pragma unroll
                            for (int ii = 0; ii < 2; ii++) {
                                const float *q = o + 2 * kBinDoubles * ii;
                                const int i = 2 * i2 + ii;
#pragma unroll
                                for (int c = 0; c < 3; c++) {
                                    float2 x, y;  // h = x + y
                                    fixed_pair(wm_.H[i][2 * c][lane], x.x, y.x);
                                    fixed_pair(wm_.H[i][2 * c + 1][lane], x.y, y.y);
                                    const float s24 = 5.9604644775390625e-8f;  // 2^-24
                                    y = mul2(y, make_float2(s24, s24));
                                    const float2 wh = make_float2(q[2 * c], q[2 * c]);
                                    const float2 wl = make_float2(q[2 * c + 1], q[2 * c + 1]);
                                    const float2 eh = make_float2(q[6 + 4 * c], q[7 + 4 * c]);
                                    const float2 el = make_float2(q[8 + 4 * c], q[9 + 4 * c]);
                                    // w |h|^2
                                    const float2 p = mul2(x, x);
                                    const float2 pe = fma2(add2(x, x), y, fma2(y, y, fma2(x, x, neg2(p))));
                                    const float2 u = mul2(wh, p);
                                    float2 ue = fma2(wh, p, neg2(u));
                                    ue = fma2(wl, p, ue);
                                    add_pair(hs[c], hc[c], u, fma2(wh, pe, ue));
                                    // Re((w d)* h)
                                    const float2 v = mul2(eh, x);
                                    float2 ve = fma2(eh, x, neg2(v));
                                    ve = fma2(el, x, ve);
                                    add_pair(ds[c], dc[c], v, fma2(eh, y, ve));
                                }
                            }
                        }
                        // h = (x + y) 2^(E - 28)
#pragma unroll
                        for (int c = 0; c < 3; c++) {
                            if (E[c] == kNoScale) continue;
                            hh += scaled_sum(hs[c], hc[c], ew[c] + 2 * (E[c] - 28));
                            dh += scaled_sum(ds[c], dc[c], ed[c] + E[c] - 28);
                        }
                    } else if (mine > 0) {
                        const double2 r = dense_direct(d, b, segs, bins, w, j0, j0 + mine, s_lo[k], s_hi[k]);
                        dh = r.x;
                        hh = r.y;
                    }
                    for (int o = 16; o > 0; o >>= 1) {
                        dh += __shfl_down_sync(0xffffffffu, dh, o);
                        hh += __shfl_down_sync(0xffffffffu, hh, o);
                    }
                    if (lane == 0) {
                        s_sum[warp][k][0] += dh;
                        s_sum[warp][k][1] += hh;
                    }
                    // after an early end the next walker's expansions are not in fixed point yet
                    have = direct ? (sub + 1) * L : max(have, (sub + 1) * L);
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        E[c] = direct ? kNoScale : En[c];
                        En[c] = kNoScale;
                    }
                    direct = directn;
                    directn = false;
                }
            }
        }
        __syncthreads();
        if (tid < 2 * G && s_walker[tid >> 1] >= 0) {
            const int k = tid >> 1, q = tid & 1;
            double t = 0.0;
            for (int i = 0; i < kWarps; i++) t += s_sum[i][k][q];
            b.part[2 * ((size_t)item * G + k) + q] = t;
        }
    }
}

template <int G, bool kRaw>
cudaError_t f64_attr() {
    return cudaFuncSetAttribute(dense_f64_kernel<G, kRaw>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(SmemF64));
}

template <int G, bool kRaw>
cudaError_t launch_f64(const StageDims &d, const StageBufs &b, const unsigned long long *segs,
                       const double *bins, const float4 *rows, const DenseTune &t, cudaStream_t s) {
    cudaError_t e = f64_attr<G, kRaw>();
    if (e != cudaSuccess) return e;
    dense_f64_kernel<G, kRaw><<<t.blocks, 32 * kWarps, sizeof(SmemF64), s>>>(d, b, segs, bins, rows,
                                                                             t.threads * t.per_thread);
    return cudaGetLastError();
}

template <int G, bool kRaw>
int occ_f64() {
    if (f64_attr<G, kRaw>() != cudaSuccess) return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, dense_f64_kernel<G, kRaw>, 32 * kWarps,
                                                      sizeof(SmemF64)) != cudaSuccess)
        return 0;
    return n;
}

// Blocks per SM of a tile shape: tiles of 512 or 1024 bins, groups of 1 or 8 walkers.
int dense_f64_occupancy(int per_thread, int group) {
    if ((per_thread != 4 && per_thread != 8) || (group != 1 && group != 8)) return 0;
    return group == 8 ? occ_f64<8, false>() : occ_f64<1, false>();
}

cudaError_t launch_dense_f64(const StageDims &d, const StageBufs &b,
                             const unsigned long long *segs, const double *bins, const float4 *rows,
                             const DenseTune &t, cudaStream_t s) {
    if (t.threads != 128 || (t.per_thread != 4 && t.per_thread != 8)) return cudaErrorInvalidValue;
    if (!rows) return t.group == 1 ? launch_f64<1, true>(d, b, segs, bins, rows, t, s) : cudaErrorInvalidValue;
    if (t.group == 8) return launch_f64<8, false>(d, b, segs, bins, rows, t, s);
    if (t.group == 1) return launch_f64<1, false>(d, b, segs, bins, rows, t, s);
    return cudaErrorInvalidValue;
}

}  // namespace lisa
