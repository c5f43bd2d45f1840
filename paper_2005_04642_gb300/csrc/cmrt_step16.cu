// Steps, fields and diagnostics of a lattice with 16-bit storage.
#include "cmrt_march.cuh"

namespace cmrt {
namespace {

template <Pass MODE>
cudaError_t launch_chain16(const void* src, void* dst, const StepParams& P, int rows, FieldOut fo, unsigned* flag,
                           double* partials, cudaStream_t s) {
    if (P.precision == kPrecF16) return launch_march<March16<__half2, kWin>, MODE>(src, dst, P, rows, fo, flag, partials, s);
    return launch_march<March16<__nv_bfloat162, kWin>, MODE>(src, dst, P, rows, fo, flag, partials, s);
}

}  // namespace

cudaError_t launch_step16(const void* src, void* dst, const StepParams& P, int rows, unsigned* flag, cudaStream_t s) {
    return launch_chain16<Pass::Step>(src, dst, P, rows, FieldOut{}, flag, nullptr, s);
}
cudaError_t launch_fields16(const void* src, const StepParams& P, int rows, FieldOut out, cudaStream_t s) {
    return launch_chain16<Pass::Fields>(src, nullptr, P, rows, out, nullptr, nullptr, s);
}
cudaError_t launch_diag_partials16(const void* src, const StepParams& P, int rows, double* partials, cudaStream_t s) {
    return launch_chain16<Pass::Diag>(src, nullptr, P, rows, FieldOut{}, nullptr, partials, s);
}

}  // namespace cmrt
