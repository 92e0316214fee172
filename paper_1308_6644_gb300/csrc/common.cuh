// Device-side helpers shared by the NU-ASM kernels: complex arithmetic on
// float2/double2, double-float (compensated FP32) arithmetic, padding.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace nuasm {

// ---------------------------------------------------------------- programmatic dependent launch
// The kernels of an execute chain after the first can be launched with
// programmatic stream serialisation (launch_chained): every kernel lets the
// next one launch as soon as all of its own CTAs are running
// (pdl_allow_next), and the next one runs its prologue -- index arithmetic,
// plan-constant loads -- before pdl_wait(), which returns once the previous
// grid has completed and its writes are visible.  Nothing before pdl_wait()
// reads what the previous kernel writes or writes what it reads.  Without the
// launch attribute both instructions return at once.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_allow_next() { asm volatile("griddepcontrol.launch_dependents;" :::); }

// 16-byte asynchronous global -> shared copies (both addresses 16-byte aligned).
// The issuing thread waits with cp_async_wait_all; a barrier after that wait
// makes the data visible to the block.
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A launch that may start before the stream's previous kernel has finished where
// `early` says so (launch_early in nuasm_internal.h): the kernel then waits with
// pdl_wait before it touches what the previous one writes.
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(bool early, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                           Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ---------------------------------------------------------------- debug bounds checks
// The debug library (built with NUASM_DEBUG_BOUNDS=1) checks the shared- and
// global-memory indices and the TMA coordinates its kernels compute against
// the extents of the buffers they address, skips any access that would fall
// outside, and records per translation unit how many were skipped and the
// first one (site, index, extent); nuasm_debug_bounds reads and clears the
// records.  It stands in for a memory checker.  In the normal build every
// check is the constant true and compiles away.
#ifndef NUASM_DEBUG_BOUNDS
#define NUASM_DEBUG_BOUNDS 0
#endif
namespace dbg {
enum Site : int {
    kFftLoad = 1, kFftStore = 2, kTmaLoad = 3, kTmaStore = 4,
    kColLoad = 10, kColStore = 11, kColRaw = 12, kColStage = 13,
    kRowLoad = 20, kRowStore = 21, kRowModes = 22,
    kBinRec = 30, kSpreadRec = 31, kSpreadValue = 32, kSpreadPlane = 33, kSpreadWindow = 34,
    kInterpRec = 40, kInterpTile = 41, kInterpOut = 42,
};
struct Record {
    unsigned int hits;
    int site;
    long long index, limit;
};
using Reader = cudaError_t (*)(Record*, bool reset);
int add_reader(Reader r);   // diag.cu: every translation unit's reader
}  // namespace dbg
#if NUASM_DEBUG_BOUNDS
namespace dbg {
static __device__ Record rec_;   // one per translation unit
static __device__ __noinline__ bool miss(long long i, long long n, int site) {
    if (atomicAdd(&rec_.hits, 1u) == 0) {
        rec_.site = site;
        rec_.index = i;
        rec_.limit = n;
    }
    return false;
}
__device__ __forceinline__ bool in_range(long long i, long long n, int site) {
    return (i >= 0 && i < n) ? true : miss(i, n, site);
}
static cudaError_t read_rec(Record* out, bool reset) {
    cudaError_t e = cudaMemcpyFromSymbol(out, rec_, sizeof(Record));
    if (e == cudaSuccess && reset) {
        const Record zero = {0, 0, 0, 0};
        e = cudaMemcpyToSymbol(rec_, &zero, sizeof(Record));
    }
    return e;
}
[[maybe_unused]] static const int registered_ = add_reader(&read_rec);
}  // namespace dbg
#define NUASM_IN_RANGE(i, n, site) ::nuasm::dbg::in_range((long long)(i), (long long)(n), (site))
#else
#define NUASM_IN_RANGE(i, n, site) true
#endif

// ---------------------------------------------------------------- packed FP32 pairs
// One f32x2 instruction does both halves of a register pair.  Its peak rate is
// the scalar one (measured: 126 against 121 lane operations per cycle and SM)
// at half the issue slots and half the code.
// The packing stays inside each asm statement: as 64-bit shifts and ors in C++
// it multiplied the compile time of the passes by ten.
#define NUASM_F2_OP2(name, op)                                                                       \
    __device__ __forceinline__ float2 name(float2 a, float2 b) {                                      \
        float2 r;                                                                                     \
        asm("{\n.reg .b64 a, b, r;\nmov.b64 a, {%2, %3};\nmov.b64 b, {%4, %5};\n" op                 \
            " r, a, b;\nmov.b64 {%0, %1}, r;\n}"                                                      \
            : "=f"(r.x), "=f"(r.y)                                                                    \
            : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));                                                \
        return r;                                                                                     \
    }
NUASM_F2_OP2(add2, "add.rn.f32x2")
NUASM_F2_OP2(sub2, "sub.rn.f32x2")
NUASM_F2_OP2(mul2, "mul.rn.f32x2")
#undef NUASM_F2_OP2
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{\n.reg .b64 a, b, c, r;\nmov.b64 a, {%2, %3};\nmov.b64 b, {%4, %5};\nmov.b64 c, {%6, %7};\n"
        "fma.rn.f32x2 r, a, b, c;\nmov.b64 {%0, %1}, r;\n}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ float2 f2_swap(float2 a) { return make_float2(a.y, a.x); }
__device__ __forceinline__ float2 f2_dup(float a) { return make_float2(a, a); }

// ---------------------------------------------------------------- complex
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 cneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 cneg(double2 a) { return make_double2(-a.x, -a.y); }
__device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }

template <typename V> struct CTraits;
template <> struct CTraits<float2> {
    using real = float;
    using tw = float2;   // element of the twiddle table
    static constexpr int pad_shift = 4;   // one pad slot per 16 elements (128 B)
    __device__ static float2 zero() { return make_float2(0.f, 0.f); }
    __device__ static float2 make(float a, float b) { return make_float2(a, b); }
};
template <> struct CTraits<double2> {
    using real = double;
    using tw = double2;
    static constexpr int pad_shift = 3;   // one pad slot per 8 elements (128 B)
    __device__ static double2 zero() { return make_double2(0.0, 0.0); }
    __device__ static double2 make(double a, double b) { return make_double2(a, b); }
};

// Two complex FP32 values, their real and their imaginary parts each a register
// pair: transforms of two sequences side by side, every operation one f32x2
// instruction for both and a multiplication by +-i free.
struct __align__(16) fp2 {
    float2 re, im;
};
__device__ __forceinline__ fp2 fp2_make(float2 a, float2 b) { return fp2{make_float2(a.x, b.x), make_float2(a.y, b.y)}; }
__device__ __forceinline__ float2 fp2_first(fp2 v) { return make_float2(v.re.x, v.im.x); }
__device__ __forceinline__ float2 fp2_second(fp2 v) { return make_float2(v.re.y, v.im.y); }
__device__ __forceinline__ fp2 cadd(fp2 a, fp2 b) { return fp2{add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ fp2 csub(fp2 a, fp2 b) { return fp2{sub2(a.re, b.re), sub2(a.im, b.im)}; }
__device__ __forceinline__ fp2 cscale(fp2 a, float s) { return fp2{mul2(a.re, f2_dup(s)), mul2(a.im, f2_dup(s))}; }
// one factor for both sequences, both halves of its register pairs the same
// (the scalar product's roundings)
__device__ __forceinline__ fp2 cmul(fp2 a, fp2 w) {
    return fp2{fma2(a.re, w.re, mul2(a.im, mul2(w.im, f2_dup(-1.f)))), fma2(a.re, w.im, mul2(a.im, w.re))};
}
__device__ __forceinline__ fp2 cmul_conj(fp2 a, fp2 w) {
    return fp2{fma2(a.re, w.re, mul2(a.im, w.im)), fma2(a.re, mul2(w.im, f2_dup(-1.f)), mul2(a.im, w.re))};
}
template <> struct CTraits<fp2> {
    using real = float;
    using tw = float2;
    // one pad slot per 16 elements: these transforms have radix 16, whose first
    // pass stores 16 elements apart
    static constexpr int pad_shift = 4;
    __device__ static fp2 zero() { return fp2{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }
    __device__ static fp2 make(float a, float b) { return fp2{f2_dup(a), f2_dup(b)}; }
};

// a + DIR i b
template <int DIR> __device__ __forceinline__ float2 cadd_i(float2 a, float2 b) {
    return DIR < 0 ? make_float2(a.x + b.y, a.y - b.x) : make_float2(a.x - b.y, a.y + b.x);
}
template <int DIR> __device__ __forceinline__ double2 cadd_i(double2 a, double2 b) {
    return DIR < 0 ? make_double2(a.x + b.y, a.y - b.x) : make_double2(a.x - b.y, a.y + b.x);
}
template <int DIR> __device__ __forceinline__ fp2 cadd_i(fp2 a, fp2 b) {
    return DIR < 0 ? fp2{add2(a.re, b.im), sub2(a.im, b.re)} : fp2{sub2(a.re, b.im), add2(a.im, b.re)};
}

// multiply by -i (DIR = -1) or +i (DIR = +1)
template <int DIR, typename V> __device__ __forceinline__ V mul_i(V a) {
    using C = CTraits<V>;
    return DIR < 0 ? C::make(a.y, -a.x) : C::make(-a.y, a.x);
}
template <int DIR> __device__ __forceinline__ fp2 mul_i(fp2 a) {
    const float2 n = f2_dup(-1.f);
    return DIR < 0 ? fp2{a.im, mul2(a.re, n)} : fp2{mul2(a.im, n), a.re};
}

// shared-memory padding: one spare slot every 128 bytes breaks the power-of-two
// strides of the first Stockham pass across banks
template <typename V> __host__ __device__ __forceinline__ constexpr int spad(int q) {
    return q + (q >> CTraits<V>::pad_shift);
}
template <typename V> __host__ __device__ constexpr int spad_size(int n) {
    return n + (n >> CTraits<V>::pad_shift) + 1;
}

// ---------------------------------------------------------------- double-float
// Unevaluated sums hi + lo of two floats (Dekker / Knuth error-free transforms).
struct df { float hi, lo; };

__device__ __forceinline__ df df_two_sum(float a, float b) {
    float s = a + b;
    float bb = s - a;
    float e = (a - (s - bb)) + (b - bb);
    return {s, e};
}
__device__ __forceinline__ df df_fast_two_sum(float a, float b) {
    float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ df df_add(df a, df b) {
    df s = df_two_sum(a.hi, b.hi);
    df t = df_two_sum(a.lo, b.lo);
    s.lo += t.hi;
    s = df_fast_two_sum(s.hi, s.lo);
    s.lo += t.lo;
    return df_fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ df df_mul(df a, df b) {
    float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
    return df_fast_two_sum(p, e);
}
__device__ __forceinline__ df df_div(df a, df b) {
    float q = a.hi / b.hi;
    // remainder a - q b, exact leading part through fma
    float r = fmaf(-q, b.hi, a.hi);
    r = r + a.lo - q * b.lo;
    float ql = r / b.hi;
    return df_fast_two_sum(q, ql);
}
__device__ __forceinline__ df df_sqrt(df a) {
    float y = sqrtf(a.hi);
    if (y == 0.f) return {0.f, 0.f};
    float e = fmaf(-y, y, a.hi) + a.lo;
    return df_fast_two_sum(y, e / (2.f * y));
}

}  // namespace nuasm
