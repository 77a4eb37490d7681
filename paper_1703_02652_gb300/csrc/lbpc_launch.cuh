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
// In the kernels that follow one another on a stream, before any access to their data: lets
// the next grid of the stream become resident while this one drains, then waits until the
// previous grid has completed and its stores are visible.  The pointers given go through the
// barrier.  A __restrict__ pointer has to: the compiler may take it that nothing else, the
// barrier included, touches its data, and move a load above.  Others are held by the memory
// clobber; those that the pair kernels pass all the same are a measurement (addresses are then
// formed after the barrier: up to 8% of a 16-bit step either way).
// Why: between two dependent launches the GPU waits in steps of about 2 us; 64^3 FP32 took
// 10.3 us a step without the overlap and 8.0 us with it (6.2 -> 3.1 us at 64 x 1 x 64).
template <class... Ptr>
__device__ __forceinline__ void after_previous_grid(Ptr&... p) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
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
