// Double-float real and complex types for the FFT passes of FP64 plans
// (FFT engine arithmetic on the FP32 pipe).
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace nuasm {

// ---------------------------------------------------------------- double-float complex
// A real hi + lo of two floats (about 47 significant bits) and a complex of
// two of them, for FFT passes of FP64 plans on the FP32 pipe.  Sums use the
// two-sum of the high parts with the low parts added to its error term, and
// products the FMA errors of the high parts; both renormalise once (a complex
// product once per component, after the sum of its two real products).
struct dfr {
    float hi, lo;
    dfr() = default;
    __host__ __device__ constexpr dfr(float h, float l) : hi(h), lo(l) {}
    __host__ __device__ constexpr explicit dfr(double d) : hi(float(d)), lo(float(d - double(float(d)))) {}
};
__host__ __device__ constexpr dfr operator-(dfr a) { return dfr(-a.hi, -a.lo); }
// A complex of two double-floats, the high parts (re, im) and the low parts
// (re, im) each a register pair, so that a complex sum is one packed sequence.
// The double-float row passes were short of issue slots and instruction fetch,
// not of the FP32 pipe (42% busy): N' = 4096 row_t1 1.56 -> 1.17 ms, row_t2
// 1.49 -> 1.11 ms against scalar operations.
struct __align__(16) dfc {
    float2 h, l;
    __device__ __forceinline__ dfr x() const { return dfr(h.x, l.x); }
    __device__ __forceinline__ dfr y() const { return dfr(h.y, l.y); }
};
// s + e renormalised (|e| small against |s|)
__device__ __forceinline__ dfc dfc_renorm(float2 s, float2 e) {
    const float2 h = add2(s, e);
    return dfc{h, sub2(e, sub2(h, s))};
}
__device__ __forceinline__ dfc cadd(dfc a, dfc b) {
    const float2 s = add2(a.h, b.h), bb = sub2(s, a.h);
    const float2 e = add2(sub2(a.h, sub2(s, bb)), sub2(b.h, bb));
    return dfc_renorm(s, add2(e, add2(a.l, b.l)));
}
__device__ __forceinline__ dfc csub(dfc a, dfc b) {
    const float2 s = sub2(a.h, b.h), bb = sub2(s, a.h);
    const float2 e = sub2(sub2(a.h, sub2(s, bb)), add2(b.h, bb));
    return dfc_renorm(s, add2(e, sub2(a.l, b.l)));
}
// a + DIR i b: the products by +-1 are exact, so the multiplication by i costs
// only the swap
template <int DIR> __device__ __forceinline__ dfc cadd_i(dfc a, dfc b) {
    const float2 sg = DIR > 0 ? make_float2(-1.f, 1.f) : make_float2(1.f, -1.f);
    const float2 bh = f2_swap(b.h), bl = f2_swap(b.l);
    const float2 s = fma2(bh, sg, a.h), nb = sub2(a.h, s);
    const float2 e = add2(sub2(a.h, add2(s, nb)), fma2(bh, sg, nb));
    return dfc_renorm(s, add2(e, fma2(bl, sg, a.l)));
}
// a r for a real constant r (the product and its error in scalar FMAs: the
// packed fma of a, r and the packed product of a and -r came back as zero)
__device__ __forceinline__ dfc cscale(dfc a, dfr r) {
    const float2 p = make_float2(a.h.x * r.hi, a.h.y * r.hi);
    float2 e = make_float2(fmaf(a.h.x, r.hi, -p.x), fmaf(a.h.y, r.hi, -p.y));
    e = fma2(a.h, f2_dup(r.lo), e);
    return dfc_renorm(p, fma2(a.l, f2_dup(r.hi), e));
}
// the four products and their errors one by one (a packed form would need
// every factor in both halves of a pair), their sums packed
__device__ __forceinline__ dfc cmul(dfc a, dfc b) {
    const float2 p = make_float2(a.h.x * b.h.x, a.h.x * b.h.y);
    const float2 q = make_float2(-a.h.y * b.h.y, a.h.y * b.h.x);
    float2 ep = make_float2(fmaf(a.h.x, b.h.x, -p.x), fmaf(a.h.x, b.h.y, -p.y));
    float2 eq = make_float2(fmaf(-a.h.y, b.h.y, -q.x), fmaf(a.h.y, b.h.x, -q.y));
    ep = make_float2(fmaf(a.h.x, b.l.x, ep.x), fmaf(a.h.x, b.l.y, ep.y));
    eq = make_float2(fmaf(-a.h.y, b.l.y, eq.x), fmaf(a.h.y, b.l.x, eq.y));
    ep = make_float2(fmaf(a.l.x, b.h.x, ep.x), fmaf(a.l.x, b.h.y, ep.y));
    eq = make_float2(fmaf(-a.l.y, b.h.y, eq.x), fmaf(a.l.y, b.h.x, eq.y));
    const float2 s = add2(p, q), bb = sub2(s, p);
    const float2 e = add2(sub2(p, sub2(s, bb)), sub2(q, bb));
    return dfc_renorm(s, add2(e, add2(ep, eq)));
}
__device__ __forceinline__ dfc cconj(dfc a) {
    return dfc{make_float2(a.h.x, -a.h.y), make_float2(a.l.x, -a.l.y)};
}
__device__ __forceinline__ dfc cneg(dfc a) {
    return dfc{make_float2(-a.h.x, -a.h.y), make_float2(-a.l.x, -a.l.y)};
}
template <> struct CTraits<dfc> {
    using real = dfr;
    using tw = dfc;
    static constexpr int pad_shift = 3;   // 16-byte elements, as complex128
    __device__ static dfc zero() { return dfc{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
    __device__ static dfc make(dfr a, dfr b) { return dfc{make_float2(a.hi, b.hi), make_float2(a.lo, b.lo)}; }
};

// read-only cached load of a table entry (complex types of 8 or 16 bytes, reals)
template <typename T> __device__ __forceinline__ T ldgv(const T* p) { return __ldg(p); }
template <> __device__ __forceinline__ dfc ldgv<dfc>(const dfc* p) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(p));
    return dfc{make_float2(q.x, q.y), make_float2(q.z, q.w)};
}

// 2^k as a double for k in [-1022, 1023]
__device__ __forceinline__ double dfr_pow2(int k) {
    return __longlong_as_double(static_cast<long long>(k + 1023) << 52);
}

// x 2^-s (s in [-1022, 1023]) as a double-float by integer operations on the
// bits: hi the leading 24 significant bits of x (truncated), lo the next 23,
// relative error below 2^-46.  The caller picks s so that the result stays
// within the float range.  A subnormal x is first scaled by 2^-s in FP64
// (exact while the product is normal); zeros and values below 2^-100 after
// the scaling give zero, infinities and NaNs give themselves in hi.
__device__ __forceinline__ dfr dfr_split(double x, int s) {
    unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
    int ex = int(b >> 52) & 0x7ff;
    if (ex == 0x7ff) return dfr(__double2float_rn(x), 0.f);
    if (ex == 0) {   // zero or subnormal
        if ((b << 1) == 0 || s > -923) return dfr(0.f, 0.f);   // zero, or below 2^-100 of 2^s
        b = static_cast<unsigned long long>(__double_as_longlong(x * dfr_pow2(-s)));
        ex = int(b >> 52) & 0x7ff;
        s = 0;
    }
    const int e = ex - 1023 - s;
    if (e < -100) return dfr(0.f, 0.f);
    const unsigned sign = unsigned(b >> 32) & 0x80000000u;
    const unsigned hb = sign | (unsigned(e + 127) << 23) | unsigned((b >> 29) & 0x7fffffu);
    const unsigned r = unsigned(b) & 0x1fffffffu;   // the 29 mantissa bits below hi
    const unsigned lb = unsigned(e - 23 + 127) << 23;
    const float lo = __uint_as_float(lb | (r >> 6)) - __uint_as_float(lb);   // (r >> 6) 2^(e - 46), exact
    return dfr(__uint_as_float(hb), sign ? -lo : lo);
}

// (hi + lo) 2^s as a double by integer operations (the 53 leading bits of
// the exact sum, truncated), for a normalised pair (|lo| below ulp(hi)); a
// result outside the normal double range (subnormal, or beyond the largest
// double) is formed in FP64 arithmetic instead.  Zeros and subnormal hi give
// zero; infinities and NaNs give themselves.
__device__ __forceinline__ double dfr_to_double(dfr a, int s) {
    const unsigned hb = __float_as_uint(a.hi), lb = __float_as_uint(a.lo);
    const int eh = int(hb >> 23) & 0xff;
    if (eh == 0) return 0.0;
    if (eh == 0xff) return double(a.hi);
    // |hi| = Mh 2^(eh - 150); X = Mh 2^39 in units of 2^(eh - 189)
    long long X = static_cast<long long>((hb & 0x7fffffu) | 0x800000u) << 39;
    const int el = int(lb >> 23) & 0xff;
    if (el != 0) {
        const long long L = static_cast<long long>((lb & 0x7fffffu) | 0x800000u);
        const int d = eh - el;   // lo's mantissa sits d bits below hi's
        const long long Ls = d <= 39 ? (d >= 0 ? L << (39 - d) : 0) : (d - 39 < 63 ? L >> (d - 39) : 0);
        X = ((hb ^ lb) >> 31) ? X - Ls : X + Ls;
    }
    const int lz = __clzll(X);                  // leading bit at 63 - lz
    const int E = eh - 126 - lz + s;            // unbiased exponent of the result
    if (E < -1022 || E > 1023) {                // s is within [-1022, 1023]: two exact halves
        const int s1 = s / 2;
        return ((double(a.hi) + double(a.lo)) * dfr_pow2(s1)) * dfr_pow2(s - s1);
    }
    const unsigned long long m = lz <= 11 ? static_cast<unsigned long long>(X) >> (11 - lz)
                                          : static_cast<unsigned long long>(X) << (lz - 11);
    const unsigned long long bits = (static_cast<unsigned long long>(hb >> 31) << 63) |
                                    (static_cast<unsigned long long>(E + 1023) << 52) | (m & 0xfffffffffffffull);
    return __longlong_as_double(static_cast<long long>(bits));
}

}  // namespace nuasm
