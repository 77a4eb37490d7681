// lbpc_launch.cuh -- kernels that follow one another on a stream: overlapped starts.
#pragma once

#include <cuda_runtime.h>

#include "lbpc_internal.h"

#define LBPC_HD __host__ __device__ __forceinline__
#if defined(__CUDACC__)
#define LBPC_HD_CALL __host__ __device__ __noinline__  // kept out of its caller's registers
#else
#define LBPC_HD_CALL inline
#endif

namespace lbpc {

// Hides v's value from the compiler: the scatter addresses of an AA step are gather
// addresses (the same slots, in place), and without this the compiler keeps them all live
// across the collision.
template <class T>
LBPC_HD void opaque(T& v) {
#if defined(__CUDA_ARCH__)
    if constexpr (sizeof(T) == 8) asm volatile("" : "+l"(v));
    else asm volatile("" : "+r"(v));
#else
    (void)v;
#endif
}

#if defined(__CUDACC__)
// In the kernels that follow one another on a stream, before any access to their data: waits
// until the previous grid has completed and its stores are visible, then lets the next grid of
// the stream become resident while this one works.  In this order: a grid that let the next one
// in before it waits would have a whole call's grids queue up on the SMs, each of them putting its
// blocks where a waiting one left room (128 x 1 x 128 FP64 conduction, us a step: 4.8 in a call
// of 50 steps, 12.2 in one of 1000; in this order 3.7 and 3.9, without overlap 6.2).
// The pointers given go through the barrier.  A __restrict__ pointer has to: the compiler may
// take it that nothing else, the barrier included, touches its data, and move a load above.
// Others are held by the memory clobber; those that the pair kernels pass all the same are a
// measurement (addresses are then formed after the barrier: up to 8% of a 16-bit step either
// way).
// Why: between two dependent launches the GPU waits in steps of about 2 us; 64^3 FP32 took
// 10.3 us a step without the overlap and 8.1 us with it (4.1 -> 2.3 us for 32^3 conduction).
template <class... Ptr>
__device__ __forceinline__ void after_previous_grid(Ptr&... p) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    (opaque(p), ...);
}

// Launch of a kernel that begins with after_previous_grid(): with `early` its blocks may
// become resident before the stream's previous kernel has completed.
template <class... K, class... A>
inline void launch_after(void (*kern)(K...), const ItemGrid& g, bool early, cudaStream_t s,
                         A... args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = g.grid;
    c.blockDim = g.block;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&c, kern, K(args)...);
}
#endif  // __CUDACC__

}  // namespace lbpc
