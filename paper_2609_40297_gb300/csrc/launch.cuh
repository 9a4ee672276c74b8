// Launches of a level's dependent kernels (cast, count, select, render) one behind the other. Each is
// launched as soon as every CTA of the one before it has started (programmatic stream serialization),
// sets up what does not depend on it, and waits on the device for its end: a small level's time is its
// chain of launches, and this takes the launch and the first CTAs' start out of the chain (338 -> 311 us
// for 24 launches over a 20-node tree, 10.3 -> 10.0 ms for 60 at paper scale).
// Every such kernel calls wait_previous() before its first access to memory that a kernel of the chain
// writes or reads, in all threads and on every way to its end, so that the end of a kernel implies the
// end of all before it. What it reads before that is the camera's yaw table, which no kernel of the chain
// writes: the copy or the kernels (noalloc.cu) that fill it come before the chain's first launch and never
// let a launch start early. Two neighbours' lifetimes overlap, so what one of the chain wrote is read by
// ld_written (dev_path.cuh), never through __ldg.
#pragma once

#include <cuda_runtime.h>

namespace mig {

template <class... P, class... A>
inline void launch_behind(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A &...args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, kernel, P(args)...);
}

#ifdef __CUDACC__
// Lets the next kernel of the stream be launched, and waits for the end of the one before.
__device__ __forceinline__ void wait_previous() {
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
}
#endif

}  // namespace mig
