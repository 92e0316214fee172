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
// a r for a real constant r.  The product and its error are scalar, which is no
// slower (row and column passes of the N = 2048 plane: the same 3.73 ms a solve with
// packed ones).  In a packed form the fma's addend has to be the product with its
// sign flipped: CUDA 13.0's assembler takes fma2(a, R, mul2(a, -R)), two exact
// operations on a and a constant, for zero (checked on 8192 values, alone in a
// kernel: off by 1.5e-8; fma2(a, R, -mul2(a, R)) and every scalar mix: 2e-15).
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

// The general conversions (infinities, NaNs, subnormals, exponents outside the
// float range), out of line.
static __device__ __noinline__ dfr dfr_split_any(double x, int s) {
    unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
    int ex = int(b >> 52) & 0x7ff;
    if (ex == 0x7ff) return dfr(__double2float_rn(x), 0.f);
    if (ex == 0) {   // zero or subnormal
        if ((b << 1) == 0 || s > -923) return dfr(0.f, 0.f);   // zero, or below 2^-100 of 2^s
        x *= dfr_pow2(-s);
        s = 0;
    } else {
        const int e = ex - 1023 - s;
        if (e < -100) return dfr(0.f, 0.f);
        x = scalbn(x, -s);
    }
    const float hi = float(x);
    return dfr(hi, float(x - double(hi)));
}
static __device__ __noinline__ double dfr_to_double_any(dfr a, int s) {
    if (a.hi == 0.f) return 0.0;
    if (!isfinite(a.hi)) return double(a.hi);
    return scalbn(double(a.hi) + double(a.lo), s);
}

// x 2^-s (s in [-1022, 1023]) as a double-float by integer operations on the
// bits: hi the leading 24 significant bits of x (truncated), lo the next 23,
// relative error below 2^-46.  Values below 2^-100 after the scaling give zero,
// infinities and NaNs give themselves in hi.  (An FP64 conversion holds the
// FP64 pipe for 64 cycles a warp.)
__device__ __forceinline__ dfr dfr_split(double x, int s) {
    const unsigned h = unsigned(__double2hiint(x)), l = unsigned(__double2loint(x));
    const int ex = int(h >> 20) & 0x7ff, e = ex - 1023 - s;
    if (e > 126 || ex == 0x7ff || s < -900) return dfr_split_any(x, s);
    const unsigned sign = h & 0x80000000u;
    const unsigned hb = sign | (unsigned(e + 127) << 23) | (__funnelshift_l(l, h, 3) & 0x7fffffu);
    const unsigned lb = unsigned(e + 104) << 23;   // 2^(e - 23); the mantissa bits below hi's go behind it
    const float lo = __uint_as_float(lb | ((l >> 6) & 0x7fffffu)) - __uint_as_float(lb);
    const bool tiny = e < -100;
    return dfr(tiny ? 0.f : __uint_as_float(hb), tiny ? 0.f : __uint_as_float(__float_as_uint(lo) ^ sign));
}

// (hi + lo) 2^s as a double: hi's bits, plus lo in units of 2^-29 ulp(hi) (of
// 2^-30 where a power of two loses to a lo of the other sign), for a
// normalised pair (|lo| at most an ulp of hi).  Infinities and NaNs give
// themselves.
__device__ __forceinline__ double dfr_to_double(dfr a, int s) {
    const unsigned u = __float_as_uint(a.hi), sign = u & 0x80000000u;
    const int eh = int(u >> 23) & 0xff, E = eh - 127 + 1023 + s;
    if (eh == 0) return 0.0;
    if (eh < 53 || eh == 255 || E < 2 || E > 2045) return dfr_to_double_any(a, s);
    // lo times +-2^29 / ulp(hi), the sign hi's
    int i = __float2int_rn(a.lo * __uint_as_float(sign | (unsigned(127 + 127 + 23 + 29 - eh) << 23)));
    const unsigned m = u & 0x7fffffu;
    if (m == 0 && i < 0) i *= 2;
    const unsigned bh = sign | (unsigned(E) << 20) | (m >> 3), bl = m << 29;
    return __longlong_as_double((static_cast<long long>((static_cast<unsigned long long>(bh) << 32) | bl)) + i);
}

}  // namespace nuasm
