// launch.h -- chained kernel launches (programmatic dependent launch).
//
// A chain of short kernels on one stream pays at every boundary for draining,
// launching and filling the device.  Chained, a training step of 4,096 samples
// (10 kernels) takes 129 us instead of 133, a two-edit expansion round (4) 80
// instead of 83, a prediction of 20,736 orders (3) 71 instead of 72; the rest
// of such a call is its kernels and two synchronisations.  A chained kernel
// is put on the device while its predecessor still runs: it calls
// launch_next() once it holds what it allocates (tensor memory: a successor
// that took it first would wait for this kernel to end), and
// await_previous(), in every thread, before it touches global memory.  The
// latter returns when the predecessor has completed and its writes are
// visible; since every kernel of a chain waits so, all earlier ones have
// completed too.  Behind a kernel that is not part of a chain, a copy or a
// memset the launch is an ordinary one, and so is whatever follows a chain.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace comet {

__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void await_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);
    if (e != cudaSuccess) cudaGetLastError();  // reported here, not by a later call
    return e;
}

}  // namespace comet
