// chain.cuh -- launches that overlap the end of the launch before them in the
// stream (programmatic dependent launch).
//
// A step is a chain of short launches, each reading what the one before it
// wrote.  Launched plainly, each starts only after the previous one has drained
// and the front end has set it up: 1.5 - 2 us per launch, of a dozen in a step.
// launch_chained lets the front end place the next launch's blocks as soon as
// every block of the previous launch has called chain_wait; chain_wait then
// holds them until the previous launch is complete and its writes are visible.
// Every kernel of the library's chains calls it before its first access to global
// memory that any launch writes, so completion is transitive: what the caller
// enqueued before the step is complete too.  One 256 x 512 matrix 163 -> 150 us
// per step, six odd-sized ones 222 -> 204, a GPT-2 Large layer 459 -> 449.
#pragma once
#include <cuda_runtime.h>
#include <utility>

namespace malt {

// Waits for the previous launch, then lets the next one be placed.  A no-op in a
// kernel that was launched plainly.
__device__ __forceinline__ void chain_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The index or pointer, opaque to the compiler: an access that it addresses cannot be
// moved above the wait before it.  The wait alone does not hold back accesses through
// a __restrict__ pointer, which the compiler may take for memory that nothing else
// changes: every access through one to what a launch of the chain writes goes by here.
__device__ __forceinline__ int after_wait(int i) {
    asm volatile("" : "+r"(i)::"memory");
    return i;
}
template <typename T>
__device__ __forceinline__ T* after_wait(T* p) {
    asm volatile("" : "+l"(p)::"memory");
    return p;
}

template <typename... Params, typename... Args>
cudaError_t launch_chained(void (*kernel)(Params...), unsigned blocks, unsigned threads, size_t smem,
                           cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
    if (e != cudaSuccess) cudaGetLastError();   // reported here, not by a later launch's check
    return e;
}

}  // namespace malt
