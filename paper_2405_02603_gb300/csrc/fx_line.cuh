// fx_line.cuh -- the scale of a fixed-point line (fx.cuh) from its largest
// component and its 1-norm, and the conversions between doubles and that scale.
#pragma once
#include "fx.cuh"

namespace fsp {

// bits by which a radix-R butterfly can grow a modulus; radices 3, 5 and 6
// rounded up, which also covers their partial differences
__host__ __device__ constexpr int fx_grow(int R) {
    return R <= 1 ? 0 : R == 2 ? 1 : R <= 4 ? 2 : R <= 8 ? 3 : R <= 16 ? 4 : 5;
}

// a complex double in the registers of a cfx until its line's scale is known
__device__ __forceinline__ cfx fx_raw(double2 q) {
    return cfx{fx(__double_as_longlong(q.x), 0), fx(__double_as_longlong(q.y), 0)};
}
// adds its modulus (within sqrt 2), in units of 2^k, to s, and the upper word of
// its larger component to the maximum h
__device__ __forceinline__ void fx_bound(const cfx &v, float &s, int &h, int k = 0) {
    const int hx = fx_habs(__longlong_as_double(v.x.v)), hy = fx_habs(__longlong_as_double(v.y.v));
    const int m = max(hx, hy);
    s += fx_fabs(m, k);
    h = max(h, m);
}

// The scale of a line: integers are x 2^ke.
struct FxScale {
    int ke;
    bool any;  // outside the range the fast conversions cover
    bool bad;  // an infinity or a NaN among the inputs
};
// components of a line are below 2^em, hmax the largest upper word
__device__ __forceinline__ int fx_em(int hmax) { return max(hmax >> 20, 1) - 1022; }
// outside the range of em in which sums of fx_fabs, fx_of and fx_of_p hold: below,
// values that count as zero would reach the 1-norm's last bits; above, it could
// overflow a float.  (Sources of 1e-30 .. 1e33: FP64 plans keep their spectra
// near 1.)  A line outside has the scale of its largest component alone in the
// specialised passes, at most 4 bits below the one of its 1-norm.
__device__ __forceinline__ bool fx_far(int em) { return em < -100 || em > 112; }

// ---- the scale of a line with a runtime schedule (kernels_impl.cuh)
// s <= 2^em * (some 2^12) in units of 2^(em - 16), rounded up; |em| < 100
__device__ __forceinline__ unsigned tile_units(float s, int em) {
    return (unsigned)(s * __int_as_float((127 + 16 - em) << 23)) + 1u;
}
// fx_ke of a runtime schedule (5s, 3s, 8s, last): modulus <= 2^B after every
// stage, each stage after the first dividing by 4 beforehand
__device__ __forceinline__ int tile_ke(const Stages &st, int em, int eL, int B) {
    int eb = -100000, g = 0, d = 0;
    auto stage = [&](int grow) {
        g += grow;
        eb = max(eb, min(em + 1 + g, eL) - d);
        d += 2;
    };
    for (int i = 0; i < st.n5; ++i) stage(3);
    for (int i = 0; i < st.n3; ++i) stage(2);
    for (int i = 0; i < st.n8; ++i) stage(3);
    if (st.last) stage(st.last == 4 ? 2 : 1);
    return B - max(eb, min(em + 1, eL));  // (a transform of length 1 has no stage)
}
__device__ __forceinline__ int tile_log2(const Stages &st) {
    return 3 * st.n5 + 2 * st.n3 + 3 * st.n8 + (st.last == 4 ? 2 : st.last == 2 ? 1 : 0) + 1;
}
// twice the number of stages that divide by 4
__device__ __forceinline__ int tile_div(const Stages &st) {
    return 2 * max(st.n5 + st.n3 + st.n8 + (st.last ? 1 : 0) - 1, 0);
}

// PX, PY: that component through the FP64 pipe.  A pass mixes the two ways so
// that neither pipe waits for the other.
template <bool PX, bool PY> __device__ __forceinline__ cfx fx_conv(const cfx &v, const FxScale &sc) {
    const double x = __longlong_as_double(v.x.v), y = __longlong_as_double(v.y.v);
    if (sc.any) return cfx{fx(fx_of_any(x, sc.ke), 0), fx(fx_of_any(y, sc.ke), 0)};
    return cfx{fx(PX ? fx_of_p(x, sc.ke) : fx_of(x, sc.ke), 0), fx(PY ? fx_of_p(y, sc.ke) : fx_of(y, sc.ke), 0)};
}
// back to doubles at 2^eo; bad lines become NaN
template <bool PX, bool PY> struct FxOut {
    int eo;
    bool slow, bad;
    __device__ __forceinline__ FxOut(int e, bool b) : eo(e), slow(b || e < -1022 || e > 961), bad(b) {}
    template <bool P> __device__ __forceinline__ double one(long long v) const {
        if (!slow) return P ? fx_to_p(v, eo) : fx_to(v, eo);
        return bad ? __longlong_as_double(0x7ff8000000000000LL) : fx_to_any(v, eo);
    }
    __device__ __forceinline__ double2 operator()(const cfx &v) const {
        return double2{one<PX>(v.x.v), one<PY>(v.y.v)};
    }
};

// ---- the product with the spectrum, rescaled for the inverse transform.
// v 2^eo are a line's coefficients, |v| < 2^61.  The 1-norm and the largest
// modulus of their products with S = +-m 2^(es - 1023), m in [1, 2), give the
// scale 2^ke of the inverse (the products' moduli below 2^60); then
//   v S 2^ke = ((v << (2 + max(-r, 0))) (m 2^61 >> max(r, 0))) / 2^64,
//   r = 1022 - ke - es
// (S is shifted rather than the products: one value, and its dropped bits are
// worth less than a unit of the result).
//
// The bounds are floats, which hold for |S| 2^-k in (2^-80, 2^80); a line outside
// has the bounds of the largest S and the largest possible v alone, 4 (N = 32)
// to 11 bits (N = 135) wider.  S scales with the square of the box (2^-100 in
// boxes of 1e-12, 2^114 in boxes of 1e20), so FP64 plans hold it divided by a
// power of two that P5 gives back, and k = 0 does.  A caller's bare spectrum,
// which only the generic engine meets, has the exponent of S(1, 1, 1) as its k:
// close to the largest of a potential's.
__device__ __forceinline__ int fx_base(double s) { return max(fx_habs(s) >> 20, 1) - 1023; }
__device__ __forceinline__ void fx_bound_mul(const cfx &v, double s, float &s2, float &m2, int &hS, int k = 0) {
    const int hs = fx_habs(s);
    // |v| <= f 2^32
    const float f = (float)(abs((int)(v.x.v >> 32)) + abs((int)(v.y.v >> 32)) + 2);
    const float q = f * fx_fabs(hs, k);
    s2 += q, m2 = fmaxf(m2, q), hS = max(hS, hs);
}
// exponent of the largest |S|, and whether the float bounds hold for it
__device__ __forceinline__ int fx_es(int hS) { return (hS >> 20) - 1022; }
__device__ __forceinline__ bool fx_near(int eS, int k = 0) { return eS - k > -80 && eS - k < 80; }
// neg: -1 to negate S; normal: the largest |S| is above 2^-900, so that a
// subnormal one gives a zero product whatever its leading bit
__device__ __forceinline__ cfx fx_mul_s(const cfx &v, double s, int ke, int neg, bool normal) {
    const int hi = __double2hiint(s), e = (hi >> 20) & 0x7ff, sh = 1022 - ke - max(e, 1);
    const int one = normal || e != 0 ? 0x100000 : 0;
    const unsigned long long m = ((unsigned long long)((hi & 0xfffff) | one) << 32) | (unsigned)__double2loint(s);
    const long long mr = (long long)(m << 9) >> min(max(sh, 0), 63), sg = (hi >> 31) ^ neg;
    const long long w = (mr ^ sg) - sg;
    const int wh = fx_hi(w), wl = fx_lo(w), up = 2 + min(max(-sh, 0), 60);
    return cfx{fx(fx_mul(v.x.v << up, wh, wl), 0), fx(fx_mul(v.y.v << up, wh, wl), 0)};
}

}  // namespace fsp
