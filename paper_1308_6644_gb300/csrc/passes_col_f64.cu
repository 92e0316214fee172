// Column-pass instantiations of FP64 plans for every supported N', in
// double-float arithmetic (dfc, on the FP32 pipe) or FP64, as the row passes;
// the window and the caller's planes are FP64.
#include "passes.cuh"

namespace nuasm {

cudaError_t col_f64(const nuasm_plan_s* P, int mode, const void* ext, cudaStream_t s) {
    auto run = [&](auto st) -> cudaError_t {
        using S = decltype(st);
        switch (mode) {
            case passes::COL_FWD_FOLD: return S::col_fwd_fold(P, s);
            case passes::COL_INV: return S::col_inv(P, const_cast<void*>(ext), s);
            case passes::COL_FWD: return S::col_fwd(P, ext, s);
            default: return S::col_inv_fold(P, s);
        }
    };
    if (fft_double_float(P)) return passes::dispatch<dfc, 12>(P->g.lognp, run);
    return passes::dispatch<double2, 8>(P->g.lognp, run);
}

}  // namespace nuasm
