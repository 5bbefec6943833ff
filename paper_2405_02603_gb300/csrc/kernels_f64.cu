// kernels_f64.cu -- double-precision instantiation of the line kernels (the
// FSP_F64 solve and every plan-time transform, which always runs in FP64):
// double arrays, transforms in 64-bit fixed point.
#include "kernels_impl.cuh"

namespace fsp {
// exp(-2 pi i e / n) to 62 fraction bits: the angle's octant, then the Taylor
// series of cos and sin on [0, pi/4] in 64-bit fractions (63 fraction bits).
__global__ void k_roots_fx(fxw *out, int n) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    typedef unsigned long long u64;
    const int oct = (int)(8LL * e / n);
    u64 num = (u64)(8LL * e - (long long)oct * n);
    if (oct & 1) num = n - num;
    const u64 one = 1ull << 63;
    const u64 g = one / n * num + one % n * num / n;                // num / n
    const u64 th = __umul64hi(g, 0xc90fdaa22168c235ull);            // times pi / 4
    const u64 x2 = __umul64hi(th << 1, th << 1);                    // 64 fraction bits
    u64 c = one, s = one;
    for (int k = 11; k >= 1; --k) {
        c = one - __umul64hi(x2, c) / (u64)((2 * k - 1) * (2 * k));
        s = one - __umul64hi(x2, s) / (u64)((2 * k) * (2 * k + 1));
    }
    s = __umul64hi(th << 1, s);
    long long ci = (long long)((c + 1) >> 1), si = (long long)((s + 1) >> 1);
    if (oct & 1) si = -si;  // the angle is the next quadrant's start minus th
    for (int q = ((oct + 1) >> 1) & 3; q > 0; --q) {
        const long long v = ci;
        ci = -si, si = v;
    }
    si = -si;
    out[e] = fxw{fx_hi(ci), fx_lo(ci), fx_hi(si), fx_lo(si)};
}
template <> cudaError_t launch_roots<double>(void *tw, int n, cudaStream_t s) {
    k_roots_fx<<<(n + 255) / 256, 256, 0, s>>>(reinterpret_cast<fxw *>(tw), n);
    return cudaGetLastError();
}
FSP_INSTANTIATE_PASSES(double)
// plan-time forms: DCT-I of real lines (Sec. 2.4), DST-I of real lines (the
// field kernels' odd axis) and the real part of the last inverse pass of the
// (4N)^3 transform (Sec. 2.3)
template cudaError_t launch_lines<double, IN_REAL_EVEN, OUT_REAL, M_FWD>(const LinesArgs &, cudaStream_t);
template cudaError_t launch_lines<double, IN_REAL_ODD, OUT_REAL, M_FWD>(const LinesArgs &, cudaStream_t);
template cudaError_t launch_lines<double, IN_CPLX, OUT_REAL, M_INV>(const LinesArgs &, cudaStream_t);
}  // namespace fsp
