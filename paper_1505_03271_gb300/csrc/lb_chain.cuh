// lb_chain.cuh -- kernels that overlap the end of the one before them in their
// stream: the wait, the launch, and the loads that follow the wait.
#pragma once

#include "lb_pair.cuh"

namespace lbgb {

// Steps chained by programmatic dependent launch: a kernel may be resident
// before the previous one in its stream has finished.  It reads only constant
// tables until chain_wait(), which returns when that kernel is complete and
// then lets the next one in; every CTA calls it, also one with nothing to do.
// What that kernel wrote is read by the plain loads of Chained<> (__ldg and its
// like promise that nobody writes the data while the kernel is resident, so
// the compiler may move them above the wait).
// The paired tiles use it, whose CTAs are short and stage tables first:
// channel 256 x 512 FP32 8.1 -> 7.7 us a step, 256 x 256 5.95 -> 5.4, 16
// served requests 16.9 -> 16.6 ms.  The block march, whose CTAs fill an SM
// and march for longer, lost by it (1000 x 375 thermal 30.0 -> 31.5 us).
__device__ __forceinline__ void chain_wait() {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
}
template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// Loads of the deviation storage (Store<>, PairIO<>) in a chained kernel.
template <typename S> struct Chained;
template <> struct Chained<double> {
    __device__ static double ld(const double* p) { return *p; }
};
template <> struct Chained<float> {
    __device__ static float ld(const float* p) { return *p; }
    __device__ static pairmath::V2 two(const float* p) { return {*reinterpret_cast<const float2*>(p)}; }
};
template <> struct Chained<__half> {
    __device__ static float ld(const __half* p) { return __half2float(*p) * (1.0f / kF16Scale); }
    __device__ static pairmath::V2 two(const __half* p) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(p));
        return {make_float2(f.x * (1.0f / kF16Scale), f.y * (1.0f / kF16Scale))};
    }
};
template <> struct Chained<__nv_bfloat16> {
    __device__ static float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }
    __device__ static pairmath::V2 two(const __nv_bfloat16* p) {
        return {__bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p))};
    }
};

}  // namespace lbgb
