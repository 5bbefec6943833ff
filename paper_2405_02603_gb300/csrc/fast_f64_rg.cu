// fast_f64_rg.cu -- the FP64 column passes with runtime geometry (non-cubic
// boxes), 64-bit fixed point, apart from the cubic ones so that the
// translation units compile in parallel.
#include "fast_fx.cuh"

namespace fsp {
namespace fast {
template <> bool has_col_rg<double>(int n) {
    return n == 64 || n == 128 || n == 256 || n == 512 || n == 1024;
}
template <> cudaError_t col_rg<double>(int mode, int n, const ColArgs &a, int nb, cudaStream_t s) {
    switch (mode) {
    case COL_FWD: return launch_fx_col_rg<COL_FWD>(n, a, nb, s);
    case COL_INV: return launch_fx_col_rg<COL_INV>(n, a, nb, s);
    case COL_FMI: return launch_fx_col_rg<COL_FMI>(n, a, nb, s);
    }
    return cudaErrorInvalidValue;
}
}  // namespace fast
}  // namespace fsp
