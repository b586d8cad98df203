// fixed.cuh -- 64-bit fixed-point arithmetic on the 32-bit integer units (internal).
//
// GB300 executes 2 FP64 operations per clock and SM but 56 multiply-adds of two 32-bit
// integers into a 64-bit one (measured), so a product of two 64-bit fixed-point numbers
// kept to 64 bits, three such multiply-adds, costs about a tenth of an FP64 multiply-add's
// time.  Numbers are split into a signed high and a signed low word ("balanced": low in
// [-2^31, 2^31)) so that every partial product is a signed 32 x 32 -> 64 multiply-add.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace lisa {

typedef long long i64;

struct Bal {
    int h, l;
};

// x = h 2^32 + l; |x| < 2^63 - 2^31
__host__ __device__ __forceinline__ Bal bal(i64 x) {
    Bal r;
    r.l = (int)x;
    r.h = (int)(x >> 32) + (int)((uint32_t)r.l >> 31);
    return r;
}

// cross terms h l' + l h' of a product, in units of 2^32
__host__ __device__ __forceinline__ i64 cross(Bal a, Bal b) {
    return (i64)a.h * b.l + (i64)a.l * b.h;
}

// a b 2^-64, low by less than 2 units (the l l' product and the fraction of the cross terms
// are dropped)
__host__ __device__ __forceinline__ i64 mulhi(Bal a, Bal b) {
    return (i64)a.h * b.h + (cross(a, b) >> 32);
}

__host__ __device__ __forceinline__ i64 double_bits(double v) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(v);
#else
    union {
        double d;
        i64 i;
    } u;
    u.d = v;
    return u.i;
#endif
}

// exponent e with 2^(e-1) <= |v| < 2^e (v finite and not subnormal); -2000 for v = 0 (and
// subnormal v); 1025 for infinities and NaN
__host__ __device__ __forceinline__ int exponent_of(double v) {
    const int e = (int)((double_bits(v) >> 52) & 0x7ff);
    return e == 0 ? -2000 : e - 1022;
}

// v 2^s rounded to the nearest integer, |v 2^s| < 2^62
__host__ __device__ __forceinline__ i64 to_fixed(double v, int s) {
    const i64 b = double_bits(v);
    const int e = (int)((b >> 52) & 0x7ff);
    const i64 m = (b & 0xfffffffffffffLL) | 0x10000000000000LL;
    const int sh = e - 1075 + s;  // m 2^sh
    i64 r;
    if (sh >= 0)
        r = m << (sh > 10 ? 10 : sh);
    else
        r = sh < -54 ? 0 : (m + (1LL << (-sh - 1))) >> -sh;
    if (e == 0) r = 0;
    return b < 0 ? -r : r;
}

// v 2^s as a 96-bit two's-complement number: the integer part (modulo 2^64) and the next 32
// bits, |v 2^s| < 2^62
__host__ __device__ __forceinline__ i64 to_fixed96(double v, int s, uint32_t &low) {
    const i64 b = double_bits(v);
    const int e = (int)((b >> 52) & 0x7ff);
    const i64 m = (b & 0xfffffffffffffLL) | 0x10000000000000LL;
    const int sh = e - 1075 + s;  // m 2^sh
    i64 r = 0;
    low = 0;
    if (e != 0) {
        if (sh >= 0) {
            r = m << (sh > 10 ? 10 : sh);
        } else if (sh > -86) {
            const int k = -sh;
            r = k < 54 ? m >> k : 0;
            low = (uint32_t)(k <= 32 ? m << (32 - k) : m >> (k - 32));
        }
    }
    if (b < 0) {  // -(r + low 2^-32)
        r = -r - (low != 0);
        low = 0u - low;
    }
    return r;
}

// c + a b
__device__ __forceinline__ i64 mad_u(uint32_t a, uint32_t b, i64 c) {
    i64 r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ i64 mad_s(int a, int b, i64 c) {
    i64 r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
// c + (a 2^32) (modulo 2^64)
__device__ __forceinline__ i64 add_hi(i64 c, uint32_t a) {
    return (i64)(((unsigned long long)((uint32_t)(c >> 32) + a) << 32) | (uint32_t)c);
}

// ------------------------------------------------------------------ e^{2 pi i ph}
// ph: a fraction of a turn scaled by 2^64.  The nearest of kFxTab multiples of 2 pi / 512
// comes from a table (cos, sin scaled by 2^62), the remaining angle t, |t| <= pi / 512, from
// cos t - 1 = -t^2/2 + t^4/24 (next term 7e-17) and sin t = t (1 - t^2/6 + t^4/120) (next term
// 6e-20); results scaled by 2^60, with an absolute error of about 1e-16.
constexpr int kFxTab = 512;

struct __align__(16) FxTab {
    Bal c, s;
};

__host__ __device__ __forceinline__ uint32_t umulhi32(uint32_t a, uint32_t b) {
    return (uint32_t)(((unsigned long long)a * b) >> 32);
}

__host__ __device__ __forceinline__ int fx_cell(unsigned long long ph) {
    return (int)((ph + (1ull << 54)) >> 55) & (kFxTab - 1);
}

__host__ __device__ __forceinline__ void fx_rotate(unsigned long long ph, FxTab t, i64 &zr, i64 &zi) {
    // remainder to the nearest cell, 55 signed bits, moved up by 8 bits
    const i64 r = (i64)(ph << 9) >> 1;
    // t 2^69 = r 2^8 (pi / 4): pi/4 2^63 as a signed balanced pair, product doubled
    constexpr i64 kQ = 7244019458077122842LL;  // pi/4 2^63
    const Bal q = {(int)(kQ >> 32) + (int)((uint32_t)(kQ & 0xffffffffLL) >> 31), (int)(uint32_t)(kQ & 0xffffffffLL)};
    const i64 th = mulhi(bal(r), q) << 1;
    const Bal tb = bal(th);
    // t^2 2^74
    const i64 t2 = (i64)tb.h * tb.h + (((i64)tb.h * tb.l) >> 31);
    const uint32_t t2a = (uint32_t)(t2 >> 32);   // t^2 2^42, below 2^27.4
    const uint32_t t2b = (uint32_t)(t2 >> 28);   // t^2 2^46, below 2^31.4
    const uint32_t t4 = (uint32_t)(((unsigned long long)t2a * t2a) >> 24);  // t^4 2^60
    // cos t - 1 (2^62): t^4 2^62 / 24 = t4 (2^34 / 24) 2^-32
    const i64 cm = -(t2 >> 13) + (i64)umulhi32(t4, 715827883u);
    // t^2/6 - t^4/120 (2^46): t2b (2^32 / 6) 2^-32, (t2b t2b 2^-32) (2^18 / 120) 2^-32
    const uint32_t s1 = umulhi32(t2b, 715827883u) - umulhi32(umulhi32(t2b, t2b), 2185u);
    const i64 sn = (th >> 7) - (((i64)tb.h * (int)s1) >> 21);
    const Bal c = bal((1LL << 62) + cm), q1 = bal(sn);
    zr = ((i64)t.c.h * c.h - (i64)t.s.h * q1.h) + ((cross(t.c, c) - cross(t.s, q1)) >> 32);
    zi = ((i64)t.s.h * c.h + (i64)t.c.h * q1.h) + ((cross(t.s, c) + cross(t.c, q1)) >> 32);
}

}  // namespace lisa
