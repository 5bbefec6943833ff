// fast_f64_field.cu -- the field's P3 (the odd spectrum of E = -grad phi) in
// FP64, 64-bit fixed point, on cubic and non-cubic boxes, kept apart from the
// solve's passes so that the translation units compile in parallel.
#include "fast_field.h"
#include "fast_fx.cuh"

namespace fsp {
namespace fast {
template <> cudaError_t p3_odd<double>(int N, const ColArgs &a, int nb, cudaStream_t s) {
    return launch_fx_col<COL_FMO>(2 * N, a, nb, s);
}
template <> cudaError_t p3_odd_rg<double>(int n, const ColArgs &a, int nb, cudaStream_t s) {
    return launch_fx_col_rg<COL_FMO>(n, a, nb, s);
}
}  // namespace fast
}  // namespace fsp
