// fast_f64.cu -- the FP64 passes of cubic boxes, in 64-bit fixed point
// (fast_fx.cuh).
#include "fast_fx.cuh"

namespace fsp {
namespace fast {
template <> bool has<double>(int N) {
    return N == 32 || N == 48 || N == 64 || N == 96 || N == 128 || N == 192 || N == 256 || N == 512;
}
template <> cudaError_t p1<double>(int N, const RowArgs &a, cudaStream_t s) { return launch_fx_row<true>(N, a, s); }
template <> cudaError_t p5<double>(int N, const RowArgs &a, cudaStream_t s) { return launch_fx_row<false>(N, a, s); }
template <> cudaError_t p2<double>(int N, const ColArgs &a, int nb, cudaStream_t s) {
    return launch_fx_col<COL_FWD>(2 * N, a, nb, s);
}
template <> cudaError_t p3<double>(int N, const ColArgs &a, int nb, cudaStream_t s) {
    return launch_fx_col<COL_FMI>(2 * N, a, nb, s);
}
template <> cudaError_t p4<double>(int N, const ColArgs &a, int nb, cudaStream_t s) {
    return launch_fx_col<COL_INV>(2 * N, a, nb, s);
}
}  // namespace fast
}  // namespace fsp
