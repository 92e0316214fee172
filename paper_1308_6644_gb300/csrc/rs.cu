// Rayleigh-Sommerfeld diffraction (Eq. 10) as a direct sum on the GPU: the
// O(M1 M2) reference the paper compares NU-ASM and NU-FRE against.
//
//   u2(x2) = (1/2 pi) sum_j a_j c_j (z/r)(1 - i k r) exp(i k r) / r^2,
//   r = sqrt(|x2 + o - x1_j|^2 + z^2),  k = 2 pi / lambda,
//
// with a_j the area element of source sample j.  The phase is split as
// k r = 2 pi (frac(z/lambda) + (r - z)/lambda), r - z = rho^2 / (r + z), so
// FP32 keeps ~1e-5-cycle accuracy for the geometries of the paper's
// experiments; the FP64 variant keeps every term to double precision.
//
// Work split: a CTA of 8 warps owns 64 (FP32) or 32 (FP64) destination points,
// all of its warps the same ones; the source samples stream through
// shared memory 256 at a time and each warp takes 32 of them.  Where that
// leaves the chip short of CTAs, a cluster of 2, 4 or 8 CTAs shares one set of
// points and splits the source tiles.  Partial sums meet in shared memory and
// are added in a fixed order (warps, then the cluster's CTAs), so results are
// reproducible.  One destination point per thread and all sources in turn (the
// earlier split) put 16384 points on 64 of the 152 SMs.  Measured (sources x
// points, before -> now): FP32 65536 x 65536 14.6 -> 6.0 ms, 30000 x 3000 5.2 ->
// 0.18 ms; FP64 16384 x 16384 83.6 -> 13.5 ms, 5001 x 1001 25.5 -> 0.39 ms.
//
// Lengths are scaled by the power of two that takes z into [1, 2), so the FP32
// seeds below neither overflow nor meet subnormals for any unit of length.  (The
// FP32 kernel's result takes the scaling back as a float: z from 2^-63 to 2^63.)
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "dfloat.cuh"
#include "nuasm_internal.h"

namespace nuasm {
namespace {

namespace cg = cooperative_groups;

constexpr int kThreads = 256, kWarps = kThreads / 32, kTile = 256;
constexpr int kMaxCluster = 8;

// exp(2 pi i j / 256), j < 256, and exp(2 pi i q / 2048), q < 8, from the host's math library
constexpr int kCoarse = 256, kFine = 2048;
struct PhaseTable {
    double2 e[kCoarse], f[kFine / kCoarse];
};

struct RsArgs {
    double scale;              // power of two with z scale in [1, 2); the lengths below are scaled
    double z, z2, ox, oy;      // ox, oy in the caller's units
    double il, k;              // 1 / lambda and 2 pi / lambda
    double zfrac;              // z / lambda mod 1
    double c0, s0;             // exp(2 pi i zfrac) / (2 pi), times what the scaling took out of 1 / r^2
    double norm;               // 1 / (2 pi), likewise
    unsigned rho2_max;         // FP64: high word of the rho^2 from which on (or from 2^40 turns) a pair takes
                               // the direct formulas
    float near;                // FP32: distance per axis up to which the phase is below 2^22 - 1 half-turns
    int64_t m1, m2;
};

__device__ __forceinline__ float rsqrt_fast(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_fast(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// The cluster's partial sums of `count` points, one complex value each in
// `part` of every CTA, added by the cluster's first CTA in rank order.
template <typename V, class StoreF>
__device__ __forceinline__ void cluster_sum(V* part, int count, StoreF store) {
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();   // every CTA's partial sums are in its shared memory
    if (cl.block_rank() == 0 && threadIdx.x < count) {
        V t = part[threadIdx.x];
        for (unsigned q = 1; q < cl.num_blocks(); ++q) {
            const V u = cl.map_shared_rank(part, q)[threadIdx.x];
            t.x += u.x;
            t.y += u.y;
        }
        store(int(threadIdx.x), t);
    }
    cl.sync();   // no CTA leaves while its shared memory is read
}

// ---------------------------------------------------------------- FP32
// Two destination points per lane, so that every operation is one f32x2
// instruction for the two.  The phase is rounded where the correctly rounded
// operations round it (r, r + z, the quotient, the product with 1/lambda), then
// reduced to half-turns by additions of 1.5 2^23, whose low bit is the sign of
// the half-turn.  That holds below 2^22 half-turns (2^21 wavelengths, where an FP32
// phase is down to half a turn); from there on only a pair's magnitude means
// anything, and its phase is taken mod 2 first, so that the sine and cosine stay
// within 1.  A warp asks once per 32 sources whether any may lie that far from the
// CTA's points and takes the reduced loop if so.  Sine and cosine are polynomials
// on [-1/4, 1/4] turn (Chebyshev-node fits, 1.5e-7 at most in FP32).  43 FP32
// operations and three MUFU ones per pair of points; the FP32 pipe bounds it (78%
// of its rate at 65536 x 65536).
struct Consts32 { float2 z, z2, il2, zf2, zk, nzk; };   // each in both halves; phases in half-turns
struct Sums32 { float2 rr, ii, im; };                   // of re re, im im and of the imaginary part
// one source's share for a lane's two points
template <bool FAR>
__device__ __forceinline__ void rs_pair32(float4 s, float4 v, float2 px, float2 py, const Consts32& k, Sums32& sum) {
    const float2 one = f2_dup(1.f), none = f2_dup(-1.f), half = f2_dup(0.5f), magic = f2_dup(12582912.f);
    const float2 dx = sub2(px, make_float2(s.x, s.y)), dy = sub2(py, make_float2(s.z, s.w));
    const float2 rho2 = fma2(dx, dx, mul2(dy, dy));
    const float2 d2 = add2(rho2, k.z2);
    // r = sqrt(d2) and d = rho^2 / (r + z), each an approximation and one
    // step with the exact remainder (Markstein)
    const float2 y = make_float2(rsqrt_fast(d2.x), rsqrt_fast(d2.y));
    const float2 r0 = mul2(d2, y);
    const float2 r = fma2(fma2(mul2(r0, none), r0, d2), mul2(y, half), r0);
    const float2 t = add2(r, k.z);
    const float2 rc = make_float2(rcp_fast(t.x), rcp_fast(t.y));
    const float2 g = mul2(rho2, rc);
    const float2 d = fma2(fma2(mul2(g, none), t, rho2), rc, g);
    // half-turns: the nearest integer n and the rest
    float2 ph = fma2(d, k.il2, k.zf2);
    if (FAR) ph = make_float2(fmaf(-2.f, rintf(0.5f * ph.x), ph.x), fmaf(-2.f, rintf(0.5f * ph.y), ph.y));
    const float2 kb = add2(ph, magic);
    const float2 x = sub2(ph, sub2(kb, magic));
    const float2 u = mul2(x, x);
    float2 cs = fma2(f2_dup(-0.024395931512117386f), u, f2_dup(0.23493707180023193f));
    cs = fma2(cs, u, f2_dup(-1.335211992263794f));
    cs = fma2(cs, u, f2_dup(4.058709144592285f));
    cs = fma2(cs, u, f2_dup(-4.934802055358887f));
    cs = fma2(cs, u, one);
    float2 sn = fma2(f2_dup(0.07765591144561768f), u, f2_dup(-0.5982903838157654f));
    sn = fma2(sn, u, f2_dup(2.550077438354492f));
    sn = fma2(sn, u, f2_dup(-5.167710304260254f));
    sn = mul2(x, fma2(sn, u, f2_dup(3.1415927410125732f)));
    // +- 1 / r^2, the sign (-1)^n
    float2 w = make_float2(rcp_fast(d2.x), rcp_fast(d2.y));
    w.x = __uint_as_float(__float_as_uint(w.x) ^ (__float_as_uint(kb.x) << 31));
    w.y = __uint_as_float(__float_as_uint(w.y) ^ (__float_as_uint(kb.y) << 31));
    // z/r^3 (1 - i k r)(cs + i sn) = (z/r^3 cs + z k/r^2 sn) + i (z/r^3 sn - z k/r^2 cs)
    const float2 A = mul2(mul2(w, make_float2(fabsf(w.x), fabsf(w.y))), mul2(r, k.z));
    const float2 kre = fma2(A, cs, mul2(mul2(w, k.zk), sn));
    const float2 kim = fma2(A, sn, mul2(mul2(w, k.nzk), cs));
    const float2 vr = make_float2(v.x, v.y), vi = make_float2(v.z, v.w);
    sum.rr = fma2(vr, kre, sum.rr);
    sum.ii = fma2(vi, kim, sum.ii);
    sum.im = fma2(vr, kim, fma2(vi, kre, sum.im));
}
// (out of line: a second copy of the loop beside the first made that one 2% slower)
__device__ __noinline__ Sums32 rs_far32(const float4* pos, const float4* val, int count, float2 px, float2 py,
                                        Consts32 k, Sums32 sum) {
#pragma unroll 1
    for (int q = 0; q < count; ++q) rs_pair32<true>(pos[q], val[q], px, py, k, sum);
    return sum;
}
constexpr int kPts32 = 64;
__global__ void __launch_bounds__(kThreads, 3) rs_f32_kernel(const double* __restrict__ x1, const double* __restrict__ y1,
                                                          const float2* __restrict__ c, const double* __restrict__ area,
                                                          const double* __restrict__ x2, const double* __restrict__ y2,
                                                          float2* __restrict__ out, RsArgs a, int split) {
    __shared__ float4 pos[kTile], val[kTile];   // {x, x, y, y} and {re, re, im, im} of a c
    __shared__ float2 acc[kWarps][kPts32];
    __shared__ float2 part[kPts32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rank = int(blockIdx.x) % split;
    const int64_t p0 = int64_t(blockIdx.x / split) * kPts32;
    // (lanes without a point of their own take the last one, which keeps them near the others)
    auto coord = [&](const double* v, double o, int64_t i) { return float((v[min(i, a.m2 - 1)] + o) * a.scale); };
    const float2 px = make_float2(coord(x2, a.ox, p0 + lane), coord(x2, a.ox, p0 + 32 + lane));
    const float2 py = make_float2(coord(y2, a.oy, p0 + lane), coord(y2, a.oy, p0 + 32 + lane));
    const float z = float(a.z), zk = float(a.z * a.k);
    const Consts32 k{f2_dup(z), f2_dup(z * z), f2_dup(float(2.0 * a.il)), f2_dup(float(2.0 * a.zfrac)), f2_dup(zk),
                     f2_dup(-zk)};
    Sums32 sum{make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    // the points lie within `reach` of the first one per axis (bits of magnitudes: a NaN tops all),
    // sources within `near` of it are near all of them
    const float cx = __shfl_sync(0xffffffffu, px.x, 0), cy = __shfl_sync(0xffffffffu, py.x, 0);
    auto off = [](float v, float c) { return __float_as_uint(v - c) & 0x7fffffffu; };
    const float reach = __uint_as_float(__reduce_max_sync(
        0xffffffffu, max(max(off(px.x, cx), off(px.y, cx)), max(off(py.x, cy), off(py.y, cy)))));
    const float near = a.near - reach;
    for (int64_t base = int64_t(rank) * kTile; base < a.m1; base += int64_t(split) * kTile) {
        const int64_t j = base + threadIdx.x;
        float4 ps = make_float4(cx, cx, cy, cy), vs = make_float4(0.f, 0.f, 0.f, 0.f);
        if (j < a.m1) {
            const float2 v = c[j];
            const float w = float(area[j]), sx = float(x1[j] * a.scale), sy = float(y1[j] * a.scale);
            ps = make_float4(sx, sx, sy, sy);
            vs = make_float4(v.x * w, v.x * w, v.y * w, v.y * w);
        }
        __syncthreads();
        pos[threadIdx.x] = ps;
        val[threadIdx.x] = vs;
        // (a warp's sources are those that its lanes loaded)
        const bool far = !__all_sync(0xffffffffu, fabsf(ps.x - cx) <= near && fabsf(ps.z - cy) <= near);
        __syncthreads();
        const int q0 = warp * 32, q1 = int(min(int64_t(q0 + 32), a.m1 - base));
        if (far) {
            sum = rs_far32(pos + q0, val + q0, q1 - q0, px, py, k, sum);
            continue;
        }
#pragma unroll 4
        for (int q = q0; q < q1; ++q) rs_pair32<false>(pos[q], val[q], px, py, k, sum);
    }
    acc[warp][lane] = make_float2(sum.rr.x - sum.ii.x, sum.im.x);
    acc[warp][32 + lane] = make_float2(sum.rr.y - sum.ii.y, sum.im.y);
    __syncthreads();
    if (threadIdx.x < kPts32) {
        float2 t = acc[0][threadIdx.x];
#pragma unroll
        for (int k = 1; k < kWarps; ++k) t = cadd(t, acc[k][threadIdx.x]);
        part[threadIdx.x] = t;
    }
    const float norm = float(a.norm);
    cluster_sum(part, kPts32, [&](int i, float2 t) {
        if (p0 + i < a.m2) out[p0 + i] = make_float2(t.x * norm, t.y * norm);
    });
}

// ---------------------------------------------------------------- FP64
// The FP64 pipe takes a warp instruction every 64 cycles of an SM
// sub-partition, so FP64 work is what a pair costs: about 80 FP64 operations
// with the library's sqrt, division and sincospi.  Here each function starts
// from FP32 or double-float on the FP32 pipe and is corrected in FP64:
//  * r - z: rho^2 / (r + z) in double-float (2^-44), then one Newton step on
//    d (2z + d) = rho^2 in FP64;
//  * 1 / r: rsqrt in FP32, then 1/r = y (1 + e + e^2), e = 1 - r y;
//  * the phase: rounded to 1/2048 turn by an addition of 1.5 2^41, the rest
//    (|theta| <= pi/2048) through short series in double-float: exp(i theta) - 1
//    times exp(2 pi i j / 2048) from shared memory, added to it in FP64.
// exp(2 pi i frac(z/lambda)) is one factor of the whole sum.  27 FP64 operations
// a pair, which bound it (33 with the series in FP64).
struct Src64 { double x, y, re, im; };
struct Pair64 { double re, im; };

// the direct formulas, for pairs whose rho^2 leaves the float range (or is not finite)
__device__ __noinline__ Pair64 rs_pair_direct(double dx, double dy, const double z, const double il, const double k) {
    const double rho2 = dx * dx + dy * dy;
    const double r = sqrt(rho2 + z * z);
    double ph = (rho2 / (r + z)) * il;
    ph -= rint(ph);
    double sn, cs;
    sincospi(2.0 * ph, &sn, &cs);
    const double amp = 1.0 / (r * r * r), kr = k * r;
    return {amp * (cs + kr * sn), amp * (sn - kr * cs)};
}

// The FP64 conversion instructions run at the FP64 rate, so values cross between
// the two by their bits (dfr_split, dfr_to_double, and here a float as a double, a
// zero as 2^-127).
__device__ __forceinline__ double wide(float x) {
    const unsigned u = __float_as_uint(x);
    return __hiloint2double(int((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), int(u << 29));
}
// (1 - i k r) exp(i k (r - z)) / r^3 of one pair
__device__ __forceinline__ Pair64 rs_pair(double dx, double dy, const RsArgs& a, const df z, const df z2,
                                          const double2* __restrict__ tab) {
    const double rho2 = fma(dx, dx, dy * dy);
    if (unsigned(__double2hiint(rho2)) >= a.rho2_max) return rs_pair_direct(dx, dy, a.z, a.il, a.k);
    // double-float: r and d = rho^2 / (r + z)
    const dfr rs = dfr_split(rho2, 0);
    const df rho = {rs.hi, rs.lo};
    const df q2 = df_add(rho, z2);
    const float yf = rsqrt_fast(q2.hi);
    const float r0 = q2.hi * yf;
    const df r1 = df_fast_two_sum(r0, 0.5f * yf * (fmaf(-r0, r0, q2.hi) + q2.lo));
    const df t1 = df_add(r1, z);
    const float rc = rcp_fast(t1.hi);
    const float g0 = rho.hi * rc;
    const df g = df_fast_two_sum(g0, rc * ((fmaf(-g0, t1.hi, rho.hi) + rho.lo) - g0 * t1.lo));
    // one Newton step in FP64 on d (2 z + d) = rho^2 (slope 2 r)
    const double yd = wide(yf);
    const double d1 = dfr_to_double(dfr(g.hi, g.lo), 0);
    const double d = fma(fma(-d1, fma(2.0, a.z, d1), rho2), wide(0.5f * yf), d1);
    const double r = a.z + d;
    const double e = fma(-r, yd, 1.0);
    const double y = fma(fma(e, e, e), yd, yd);
    // phase d / lambda: the nearest multiple of 1/2048 turn and the rest
    constexpr double magic = 3298534883328.0;   // 1.5 2^41: spacing 2^-11
    const double n = fma(d, a.il, magic);
    const double2 T = tab[__double2loint(n) & (kFine - 1)];
    // exp(i theta) - 1 as a double-float (2^-46 of it is 2^-55)
    const dfr dl = dfr_split(fma(d, a.il, magic - n), 0);
    const df th = df_mul({dl.hi, dl.lo}, {6.2831855f, -1.7484555e-7f});   // 2 pi
    const df h = df_mul(th, th);
    const df sn = df_fast_two_sum(th.hi, fmaf(th.hi * h.hi, fmaf(h.hi, 8.3333333e-3f, -0.16666667f), th.lo));
    const df c1 = df_fast_two_sum(-0.5f * h.hi, fmaf(h.hi * h.hi, fmaf(h.hi, -1.3888889e-3f, 4.1666667e-2f),
                                                     -0.5f * h.lo));
    const dfc C = cmul(CTraits<dfc>::make(dfr_split(T.x, 0), dfr_split(T.y, 0)),
                       CTraits<dfc>::make(dfr(c1.hi, c1.lo), dfr(sn.hi, sn.lo)));
    const double cr = T.x + dfr_to_double(C.x(), 0), ci = T.y + dfr_to_double(C.y(), 0);
    const double y2 = y * y, P = y2 * y, Q = y2 * a.k;
    return {fma(P, cr, Q * ci), fma(P, ci, -(Q * cr))};
}

constexpr int kPts64 = 32;
__global__ void __launch_bounds__(kThreads, 3) rs_f64_kernel(const double* __restrict__ x1, const double* __restrict__ y1,
                                                          const double2* __restrict__ c, const double* __restrict__ area,
                                                          const double* __restrict__ x2, const double* __restrict__ y2,
                                                          double2* __restrict__ out, const RsArgs a, int split,
                                                          const PhaseTable coarse) {
    __shared__ Src64 src[kTile];
    __shared__ double2 tab[kFine];
    __shared__ double2 acc[kWarps][kPts64];
    __shared__ double2 part[kPts64];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rank = int(blockIdx.x) % split;
    const int64_t p0 = int64_t(blockIdx.x / split) * kPts64;
    const bool live = p0 + lane < a.m2;
    const double px = live ? (x2[p0 + lane] + a.ox) * a.scale : 0.0, py = live ? (y2[p0 + lane] + a.oy) * a.scale : 0.0;
    {   // exp(2 pi i j / 2048): the coarse entries, times exp(2 pi i q / 2048) for q < 8
        const double2 b = coarse.e[threadIdx.x];
        tab[8 * threadIdx.x] = b;
#pragma unroll 1
        for (int q = 1; q < kFine / kCoarse; ++q) tab[8 * threadIdx.x + q] = cmul(b, coarse.f[q]);
    }
    const dfr zs = dfr(a.z), z2s = dfr(a.z2);
    const df zd = {zs.hi, zs.lo}, z2d = {z2s.hi, z2s.lo};
    double ar = 0.0, ai = 0.0;
    for (int64_t base = int64_t(rank) * kTile; base < a.m1; base += int64_t(split) * kTile) {
        const int64_t j = base + threadIdx.x;
        Src64 s{0.0, 0.0, 0.0, 0.0};
        if (j < a.m1) {
            const double2 v = c[j];
            s = Src64{x1[j] * a.scale, y1[j] * a.scale, v.x * area[j], v.y * area[j]};
        }
        __syncthreads();
        src[threadIdx.x] = s;
        __syncthreads();
        const int q0 = warp * 32, q1 = int(min(int64_t(q0 + 32), a.m1 - base));
#pragma unroll 1
        for (int q = q0; q < q1; ++q) {
            const Src64 sq = src[q];
            const Pair64 K = rs_pair(px - sq.x, py - sq.y, a, zd, z2d, tab);
            ar = fma(sq.re, K.re, fma(-sq.im, K.im, ar));
            ai = fma(sq.re, K.im, fma(sq.im, K.re, ai));
        }
    }
    acc[warp][lane] = make_double2(ar, ai);
    __syncthreads();
    if (threadIdx.x < kPts64) {
        double2 t = acc[0][threadIdx.x];
#pragma unroll
        for (int k = 1; k < kWarps; ++k) t = cadd(t, acc[k][threadIdx.x]);
        part[threadIdx.x] = t;
    }
    cluster_sum(part, kPts64, [&](int i, double2 t) {
        if (p0 + i < a.m2) out[p0 + i] = cmul(t, make_double2(a.c0, a.s0));
    });
}

PhaseTable make_phase_table() {
    PhaseTable t;
    for (int j = 0; j < kCoarse; ++j) {
        // the nearest multiple q of a quarter turn and the rest, at most pi/4
        const int q = ((j + kCoarse / 8) / (kCoarse / 4)) & 3;
        const double d = 2.0 * M_PI * double((j + kCoarse / 8) % (kCoarse / 4) - kCoarse / 8) / kCoarse;
        const double cs = std::cos(d), sn = std::sin(d);
        t.e[j] = q == 0 ? double2{cs, sn} : q == 1 ? double2{-sn, cs} : q == 2 ? double2{-cs, -sn} : double2{sn, -cs};
    }
    for (int q = 0; q < kFine / kCoarse; ++q) t.f[q] = double2{std::cos(2.0 * M_PI * q / kFine), std::sin(2.0 * M_PI * q / kFine)};
    return t;
}

// CTAs per set of destination points: doubled up to 8 while the grid holds fewer
// than four rounds of 3 CTAs on each of 152 SMs and every CTA keeps two source tiles
int source_split(int64_t sets, int64_t m1) {
    int split = 1;
    while (split < kMaxCluster && sets * split < 4 * 3 * 152 && m1 > int64_t(2) * split * kTile) split *= 2;
    return split;
}

template <typename... KArgs, typename... Args>
cudaError_t launch_split(void (*kernel)(KArgs...), int64_t sets, int split, cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(sets * split));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(split);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

bool on_device(const void* p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace
}  // namespace nuasm

extern "C" nuasm_status nuasm_rs_direct(const nuasm_params_t* p, int64_t m1, const double* x1, const double* y1,
                                        const void* c, const double* area, int64_t m2, const double* x2,
                                        const double* y2, void* out, void* stream) {
    using namespace nuasm;
    if (!p || m1 < 0 || m2 < 0) return NUASM_EINVAL;
    if (!std::isfinite(p->lambda) || !(p->lambda > 0) || !std::isfinite(p->z) || !(p->z > 0) ||
        !std::isfinite(p->ox) || !std::isfinite(p->oy))
        return NUASM_EINVAL;
    if (p->prec != NUASM_PREC_F32_F64PHASE && p->prec != NUASM_PREC_F64) return NUASM_EINVAL;
    if (m2 == 0) return NUASM_OK;
    if (!x2 || !y2 || !out || (m1 > 0 && (!x1 || !y1 || !c || !area))) return NUASM_EINVAL;
    const void* ptrs[] = {x2, y2, out};
    for (const void* q : ptrs)
        if (!on_device(q)) return NUASM_EINVAL;
    if (m1 > 0) {
        const void* sp[] = {x1, y1, c, area};
        for (const void* q : sp)
            if (!on_device(q)) return NUASM_EINVAL;
    }
    // z / lambda reduced mod 1 from a double-double quotient
    const double q = p->z / p->lambda;
    const double ql = std::fma(-q, p->lambda, p->z) / p->lambda;
    int ez;
    std::frexp(p->z, &ez);                                  // z in [2^(ez - 1), 2^ez)
    ez = ez - 1 < -1000 ? -1000 : ez - 1 > 1000 ? 1000 : ez - 1;
    RsArgs a{};
    a.scale = std::ldexp(1.0, -ez);
    a.z = p->z * a.scale;
    a.z2 = a.z * a.z;
    a.ox = p->ox;
    a.oy = p->oy;
    a.il = 1.0 / (p->lambda * a.scale);
    a.k = 2.0 * M_PI / (p->lambda * a.scale);
    a.zfrac = (q - std::nearbyint(q)) + ql;
    // z (1 - i k r) / r^3 is an inverse length squared; the FP64 kernel leaves out z
    a.norm = 0.5 / M_PI * a.scale * a.scale;
    a.c0 = a.norm * a.z * std::cos(2.0 * M_PI * a.zfrac);
    a.s0 = a.norm * a.z * std::sin(2.0 * M_PI * a.zfrac);
    const double dmax = 1099511627776.0 / a.il;   // r - z <= rho
    const double lim = dmax * dmax < 1e30 ? dmax * dmax : 1e30;
    uint64_t limbits;
    std::memcpy(&limbits, &lim, sizeof(limbits));
    a.rho2_max = unsigned(limbits >> 32);
    // |2 (d / lambda + zfrac)| < 2^22 - 1 up to d (2^-16 below it for FP32's roundings); rho^2 = d (d + 2 z)
    const double d = (4194302.0 - 64.0) / (2.0 * a.il);
    a.near = float(std::fmin(std::sqrt(0.5 * d) * std::sqrt(d + 2.0 * a.z), 1e19));
    a.m1 = m1;
    a.m2 = m2;
    const bool f64 = p->prec == NUASM_PREC_F64;
    const int64_t pts = f64 ? kPts64 : kPts32, sets = (m2 + pts - 1) / pts;
    const int split = source_split(sets, m1);
    if (sets * split > (int64_t(1) << 31) - 1) return NUASM_EUNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (f64) {
        static const PhaseTable table = make_phase_table();
        (void)launch_split(rs_f64_kernel, sets, split, st, x1, y1, static_cast<const double2*>(c), area, x2, y2,
                           static_cast<double2*>(out), a, split, table);
    } else {
        (void)launch_split(rs_f32_kernel, sets, split, st, x1, y1, static_cast<const float2*>(c), area, x2, y2,
                           static_cast<float2*>(out), a, split);
    }
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) return NUASM_OK;
    return e == cudaErrorMemoryAllocation ? NUASM_ENOMEM : NUASM_ECUDA;
}
