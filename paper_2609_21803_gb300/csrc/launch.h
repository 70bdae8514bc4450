// launch.h -- launches with attributes: chains of short kernels (programmatic
// dependent launch) and the persistent evaluators.
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
// completed too.  Its inputs may be written during its own lifetime, so it
// reads them by ordinary loads, not through the read-only path.  Behind a
// kernel that is not part of a chain, a copy or a memset the launch is an
// ordinary one, and so is whatever follows a chain.
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

// The CTA's barrier if `on` (uniform over the launch), as one predicated
// instruction: the persistent evaluators' warps in step.
__device__ __forceinline__ void cta_in_step(int on) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.s32 p, %0, 0;\n"
        "@p bar.sync 0;\n"
        "}\n" ::"r"(on)
        : "memory");
}

// Launch of a persistent evaluator, whose CTAs are all resident: the SM's
// on-chip memory is split between shared memory and L1 by what this launch
// puts on an SM, not by what the kernel's occupancy would allow (the default).
// Stage records come back through L1, and a launch that leaves SMs partly idle
// is bound by the latency of its slowest solves: 624 mixed pushing orders (N up
// to 145, a warp per CTA; the orders of launch_shape's table in api.cu) take
// 12.2 ms with the default split (28 KB of L1), 10.1 with this one, 150 orders
// 9.3 and 7.6; full launches keep their split.
// Shared memory keeps at least 44 % (100 KB), so that another stream's CTAs
// still fit beside a small launch; without that floor the times are the same.
template <class K, class A>
cudaError_t launch_persistent(K kernel, int blocks, unsigned threads, size_t smem, cudaStream_t s, const A& args) {
    int dev = 0, sms = 0, per_sm = 0, reserved = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (e != cudaSuccess) return e;
    const size_t need = (size_t)((blocks + sms - 1) / sms) * (smem + (size_t)reserved);
    const size_t percent = (100 * need + (size_t)per_sm - 1) / (size_t)per_sm;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    at.val.sharedMemCarveout = (unsigned)(percent < 44 ? 44 : percent > 100 ? 100 : percent);
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)blocks);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    e = cudaLaunchKernelEx(&c, kernel, args);
    if (e != cudaSuccess) cudaGetLastError();  // reported here, not by a later call
    return e;
}

}  // namespace comet
