// fx.cuh -- 64-bit fixed-point arithmetic with one exponent per line, the
// number type of the FP64 solve's transforms (fast_fx.cuh).
//
// Why: GB300's FP64 pipe does 1.6-1.9 operations per clock and SM (measured),
// its integer units 60 64-bit adds (two 32-bit instructions each) and 30
// 32 x 32 -> high-32 products.  A transform is three quarters additions, so in
// 64-bit integers it costs about a tenth of its FP64 time.
//
// A line (the n values one 1D transform works on) is a block floating-point
// vector: integers v with the value v 2^-ke, ke one number per line, chosen
// from the line's largest component and its 1-norm so that every partial sum
// of the transform has a modulus below 2^62 (fx_ke, tile_ke): such a sum is one
// of inputs times factors of modulus <= 1, so its modulus is at most the
// 1-norm and at most the number of terms times the largest modulus.  The
// butterflies form one value that is no such sum: x +- y of one complex value,
// for fx_w32's 45-degree factors, up to sqrt 2 2^62.  So no value is doubled to
// make room for a constant's 63 fraction bits (operator*, fx_w32), and every
// product states what it can take.
// A point charge reaches these bounds: one value carries its line's 1-norm.
// Twiddle products come out divided by 4, which takes back most of the growth
// of the radix before them, so the low bits stay in use through all stages:
// the rounding noise stays below what FP64 sums leave (about 2^-53 of the
// line's 2-norm): some 2^-61 of the 1-norm for inputs all alike, 2^-58 of it
// where a few inputs dominate.
//
// Products: a is split into signed halves (ah 2^32 + al), w likewise, and
//   a w / 2^64 = ah wh + (ah wl + al wh) / 2^32
// with the cross terms summed in 64 bits and rounded (the dropped low product
// is below half a unit).  All of it 32 x 32 + 64 multiply-adds: measured 0.49
// clocks per SM and complex product, against 0.61 with high-half products for
// the cross terms, whose floors would also have to be kept from adding up.
#pragma once
#include <cuda_runtime.h>

#include "fft_engine.cuh"

namespace fsp {

struct fx {
    long long v;
    fx() = default;
    __host__ __device__ constexpr explicit fx(long long q, int) : v(q) {}
    // a constant of modulus < 1 as the left factor of operator*: c 2^63
    __host__ __device__ constexpr explicit fx(double c) : v((long long)(c * 9223372036854775808.0)) {}
};
struct __align__(16) cfx {
    fx x, y;
};
template <> struct cx<fx> { using t = cfx; };

__device__ __forceinline__ fx operator+(fx a, fx b) { return fx(a.v + b.v, 0); }
__device__ __forceinline__ fx operator-(fx a, fx b) { return fx(a.v - b.v, 0); }
__device__ __forceinline__ fx operator-(fx a) { return fx(-a.v, 0); }

// A twiddle factor w, |w| <= 1, as round(w 2^62) split into signed halves.
struct __align__(16) fxw {
    int rh, rl, ih, il;
};
// signed halves: a = h 2^32 + l, l in [-2^31, 2^31)
__host__ __device__ constexpr int fx_hi(long long a) { return (int)((a + 0x80000000LL) >> 32); }
__host__ __device__ constexpr int fx_lo(long long a) { return (int)(unsigned)(a & 0xffffffffLL); }

// a b + c
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else  // the arithmetic compiled for the host (tests)
    return (long long)((unsigned long long)((long long)a * b) + (unsigned long long)c);
#endif
}
__device__ __forceinline__ long long fx_high(long long a) { return (long long)(int)(a >> 32); }
constexpr long long kFxHalf = 0x80000000LL;

// a w / 2^64, w in signed halves.  The cross terms are at most 2^31 (|ah| + |wh|),
// which must stay below 2^63: |a| + |w| < 2^64.
__device__ __forceinline__ long long fx_mul(long long a, int wh, int wl) {
    const int ah = fx_hi(a), al = fx_lo(a);
    return fx_mad(ah, wh, fx_high(fx_mad(ah, wl, fx_mad(al, wh, kFxHalf))));
}
// (x + i y) (wr + i wi) / 2^64, with u = -wi.  The cross terms are below
// 2^31 (|rh| + |ih|) + |x + i y| 2^-32 |rl + i il|, which must stay below 2^63:
// with twiddles (|w| <= 2^62) 0.71 of it at the largest modulus, 2^62.
__device__ __forceinline__ cfx fx_cmul(long long x, long long y, int rh, int rl, int ih, int il, int uh, int ul) {
    const int xh = fx_hi(x), xl = fx_lo(x), yh = fx_hi(y), yl = fx_lo(y);
    const long long p = fx_mad(xh, rl, fx_mad(xl, rh, fx_mad(yh, ul, fx_mad(yl, uh, kFxHalf))));
    const long long q = fx_mad(xh, il, fx_mad(xl, ih, fx_mad(yh, rl, fx_mad(yl, rh, kFxHalf))));
    return cfx{fx(fx_mad(xh, rh, fx_mad(yh, uh, fx_high(p))), 0), fx(fx_mad(xh, ih, fx_mad(yh, rh, fx_high(q))), 0)};
}
// Constants w of modulus < 1, with 63 fraction bits: twice w 2^63 wraps to
// (w - k) 2^64, k one of -1, 0, 1 (fx_whole), so w a = k a + a ((w - k) 2^64) / 2^64
// and a need not be doubled.
__host__ __device__ constexpr long long fx_twice(long long c) { return (long long)((unsigned long long)c << 1); }
__host__ __device__ constexpr int fx_whole(long long c) { return c >= 1LL << 62 ? 1 : c < -(1LL << 62) ? -1 : 0; }
// constant c times a, |a| < 2^63
__device__ __forceinline__ fx operator*(fx c, fx a) {
    const long long w = fx_twice(c.v), r = fx_mul(a.v, fx_hi(w), fx_lo(w));
    const int k = fx_whole(c.v);
    return fx(k > 0 ? r + a.v : k < 0 ? r - a.v : r, 0);
}

// x w / 4 (D < 0) or x conj(w) / 4 (D > 0)
template <int D> __device__ __forceinline__ cfx fx_twiddle(cfx x, fxw w) {
    if (D < 0) return fx_cmul(x.x.v, x.y.v, w.rh, w.rl, w.ih, w.il, -w.ih, -w.il);
    return fx_cmul(x.x.v, x.y.v, w.rh, w.rl, -w.ih, -w.il, w.ih, w.il);
}
__device__ __forceinline__ fx fx_quarter(fx a) { return fx((a.v + 2) >> 2, 0); }
// a / 2
__device__ __forceinline__ fx fx_halve(fx a) { return fx((a.v + 1) >> 1, 0); }
// as the generic engine calls them
template <> struct tw_of<fx> {
    using t = fxw;
    template <int D> static __device__ __forceinline__ cfx mul(cfx x, const fxw &w) { return fx_twiddle<D>(x, w); }
    static __device__ __forceinline__ cfx quarter(cfx a) { return cfx{fx_quarter(a.x), fx_quarter(a.y)}; }
};

// cos(2 pi m / 32) 2^63, rounded
__host__ __device__ constexpr long long fx_cos32(int m) {
    m &= 31;
    return m == 0                ? 9223372036854775807LL
           : m == 1              ? 9046147529429926059LL
           : m == 2              ? 8521284645587064995LL
           : m == 3              ? 7668953571605777421LL
           : m == 4              ? 6521908912666391106LL
           : m == 5              ? 5124230951741890994LL
           : m == 6              ? 3529631669043774883LL
           : m == 7              ? 1799390620744551094LL
           : m == 8              ? 0LL
           : m <= 16             ? -fx_cos32(16 - m)
           : m <= 24             ? -fx_cos32(m - 16)
                                 : fx_cos32(32 - m);
}

// multiply by exp(D 2 pi i m / 32), m not a multiple of 8
template <int D, int m> __device__ __forceinline__ cfx fx_w32(cfx a) {
    if constexpr (m % 8 == 4) {  // (+-1 +- i) / sqrt 2: two products
        constexpr int sx = m == 4 || m == 28 ? 1 : -1, sy = D * (m == 4 || m == 12 ? 1 : -1);
        constexpr fx c = fx(fx_cos32(4), 0);
        const fx u = sx > 0 ? (sy > 0 ? a.x - a.y : a.x + a.y) : (sy > 0 ? -(a.x + a.y) : a.y - a.x);
        const fx t = sx > 0 ? (sy > 0 ? a.y + a.x : a.y - a.x) : (sy > 0 ? a.x - a.y : -(a.y + a.x));
        return cfx{c * u, c * t};
    } else {
        // cross terms at a modulus of 2^62: 0.93 2^63 for the worst of the constants
        constexpr long long c = fx_cos32(m), s = D * fx_cos32(m - 8), wc = fx_twice(c), ws = fx_twice(s);
        constexpr int kc = fx_whole(c), ks = fx_whole(s);
        cfx r = fx_cmul(a.x.v, a.y.v, fx_hi(wc), fx_lo(wc), fx_hi(ws), fx_lo(ws), fx_hi(-ws), fx_lo(-ws));
        if constexpr (kc > 0) r = cfx{r.x + a.x, r.y + a.y};
        if constexpr (kc < 0) r = cfx{r.x - a.x, r.y - a.y};
        if constexpr (ks > 0) r = cfx{r.x - a.y, r.y + a.x};
        if constexpr (ks < 0) r = cfx{r.x + a.y, r.y - a.x};
        return r;
    }
}

// ------------------------------------------------ doubles <-> a line's scale --
// upper 32 bits of |x|
__device__ __forceinline__ int fx_habs(double x) { return __double2hiint(x) & 0x7fffffff; }
// |x| 2^-k as a float, from the upper word of |x| (truncated, relative error <
// 2^-20), for |x| 2^-k < 2^127; 0 below 2^-126.  -1023 <= k <= 1024.
__device__ __forceinline__ float fx_fabs(int h, int k = 0) {
    return __uint_as_float((unsigned)max(h, (896 + k) * 0x100000) * 8u - ((unsigned)(896 + k) << 23));
}
// ceil(log2 x) of a positive float
__device__ __forceinline__ int fx_clog2(float x) { return ((__float_as_int(x) + 0x7fffff) >> 23) - 127; }

// x 2^ke as an integer, |x| 2^ke < 2^62 (r >= 1 below)
__device__ __forceinline__ long long fx_of(double x, int ke) {
    const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
    const unsigned hm = (hi & 0xfffff) | 0x100000;
    const unsigned long long m = (((unsigned long long)hm << 32) | (unsigned)__double2loint(x)) << 10;
    const int r = min(1085 - ke - e, 64);
    const unsigned long long t = ((m >> (r - 1)) + 1) >> 1;
    const long long s = hi >> 31;
    return ((long long)t ^ s) - s;
}
// the same where the line's largest component may be subnormal
__device__ __forceinline__ long long fx_of_any(double x, int ke) {
    const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
    const unsigned hm = (hi & 0xfffff) | (e ? 0x100000 : 0);
    const unsigned long long m = (((unsigned long long)hm << 32) | (unsigned)__double2loint(x)) << 10;
    const int r = min(1085 - ke - (e ? e : 1), 64);
    const unsigned long long t = ((m >> (r - 1)) + 1) >> 1;
    const long long s = hi >> 31;
    return ((long long)t ^ s) - s;
}
// The same through the FP64 pipe, which the transforms leave idle: one of its
// instructions, the scaling done on the exponent field.  |ke| < 400.
__device__ __forceinline__ long long fx_of_p(double x, int ke) {
    const int hi = __double2hiint(x);
    const int hs = (hi & 0x7ff00000) < ((1022 - ke) << 20) ? 0 : hi + (ke << 20);  // below 1/4: zero
    return __double2ll_rn(__hiloint2double(hs, __double2loint(x)));
}
// v 2^eo, eo in [-1022, 961] (no result is subnormal or overflows)
__device__ __forceinline__ double fx_to(long long v, int eo) {
    const int sg = (int)(v >> 63);
    const unsigned long long a = (unsigned long long)((v ^ (long long)sg) - sg);
    const int lz = __clzll((long long)a);
    const unsigned long long m = a << (lz & 63);  // the leading bit to bit 63
    unsigned long long b = (m >> 11) + ((m >> 10) & 1);  // 53 bits, rounded; a carry moves the exponent
    b += (unsigned long long)(unsigned)((1023 + 63 - 1 + eo - lz) << 20) << 32;
    if (a == 0) b = 0;
    return __longlong_as_double((long long)(b | ((unsigned long long)(unsigned)(sg & 0x80000000) << 32)));
}
// The same through the FP64 pipe.
__device__ __forceinline__ double fx_to_p(long long v, int eo) {
    const double d = __ll2double_rn(v);
    const int hi = __double2hiint(d);
    return __hiloint2double(hi + (v == 0 ? 0 : eo << 20), __double2loint(d));
}
__device__ __forceinline__ double fx_to_any(long long v, int eo) {
    return v == 0 ? 0.0 : scalbn((double)v, eo);
}

}  // namespace fsp
