// Row-pass instantiations of FP64 plans, in double-float arithmetic (dfc, on the
// FP32 pipe) or FP64 (fft_double_float): every supported N' is compiled here so
// that the radix schedule, the rows per CTA and the launch bounds are constants.
#include "passes.cuh"

namespace nuasm {

cudaError_t row_f64(const nuasm_plan_s* P, int type, cudaStream_t s) {
    auto run = [&](auto st) { return decltype(st)::row(P, type, s); };
    if (fft_double_float(P)) return passes::dispatch<dfc, 12>(P->g.lognp, run);
    return passes::dispatch<double2, 8>(P->g.lognp, run);
}

}  // namespace nuasm
