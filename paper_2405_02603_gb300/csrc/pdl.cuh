// pdl.cuh -- programmatic dependent launch of the passes of a solve.
//
// A pass of a small box takes 2-6 us, of which the launch and the ramp-up are
// a large part.  Launched with this attribute, a pass is launched while the
// CTAs of the pass before it finish; pdl_wait, the first thing every kernel
// does, waits until everything before it in the stream is complete and
// visible.  Nothing is read or written before that wait, so the order of
// memory accesses is that of plain launches.
//
// No kernel triggers its dependents early: an early trigger packs the next
// pass's CTAs onto the SMs that happen to be free first, which unbalances
// grids of less than a wave.  Per solve, plain launches / triggered at the
// start / this: FP64 N = 32 26.6 / 22.9 / 17.7 us, FP32 N = 50 54.1 / 63.2 /
// 43.4, FP32 N = 64 24.6 / 22.3 / 17.2, N = 128 66.1 / 57.3 / 55.2, N = 256
// 427 / 415 / 415.
#pragma once
#include <cuda_runtime.h>

namespace fsp {

__device__ __forceinline__ void pdl_wait() {
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 900
    asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
}

inline cudaLaunchAttribute pdl_attribute() {
    cudaLaunchAttribute a{};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    return a;
}

// kern must begin with pdl_wait
template <typename A>
cudaError_t launch_pass(void (*kern)(const A), dim3 grid, unsigned threads, size_t smem, cudaStream_t s, const A &a) {
    cudaLaunchAttribute at = pdl_attribute();
    cudaLaunchConfig_t c{};
    c.gridDim = grid, c.blockDim = dim3(threads), c.dynamicSmemBytes = smem, c.stream = s;
    c.attrs = &at, c.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&c, kern, a);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace fsp
