// Launches that overlap with the end of the kernel before them in the stream (programmatic dependent
// launch): a chain of kernels of a few microseconds each, as in an operator application on a small lattice,
// then does not pay a launch latency per link (FP64 Qhat^2 + sigma, five kernels: 4^4 31 -> 23 us, 16^3x32
// 249 -> 240 us).  Not while the stream is being captured: between the nodes of a graph the plain
// dependency is the faster one (FP64 solve on 8^3x16 9.2 ms, 11.8 ms with programmatic edges), so kernels that run
// in the solvers' graphs only are launched plainly.
//
// A kernel started with launch_dependent() may begin as soon as every block of its predecessor has begun and
// there is room.  It calls dependent_begin() first: that lets its own successor be set up, and waits until
// everything launched before it has finished and can be seen.  Nothing that an earlier kernel writes is read,
// and nothing that an earlier kernel may still read is written, before that.  Such data change while the kernel
// runs: they are read by plain loads, never through the read-only path (__ldg, or a const __restrict__ kernel
// argument, which the compiler may turn into it and move above the wait).  The links, written once when the gauge
// handle is made, may take that path.  Plain loads do not pass earlier stores, so epilogues load before they store:
// then they cost nothing (FP64 Qhat^2 at 32^3x64 3.46 -> 3.44 ms, FP32 at 24^3x48 314 us either way; 404 us with loads
// between the stores).
#pragma once

#include <cuda_runtime.h>

// overlap = false: a plain launch; smem: bytes of dynamic shared memory
template <typename... P, typename... A>
inline void launch_dependent_smem(bool overlap, void (*kernel)(P...), dim3 grid, unsigned block, size_t smem,
                                  cudaStream_t s, A &&...args) {
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(s, &capture);
    c.attrs = &attr;
    c.numAttrs = overlap && capture == cudaStreamCaptureStatusNone ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);  // an error stays pending for the caller's check
}
template <typename... P, typename... A>
inline void launch_dependent_if(bool overlap, void (*kernel)(P...), dim3 grid, unsigned block, cudaStream_t s,
                                A &&...args) {
    launch_dependent_smem(overlap, kernel, grid, block, 0, s, static_cast<A &&>(args)...);
}
template <typename... P, typename... A>
inline void launch_dependent(void (*kernel)(P...), dim3 grid, unsigned block, cudaStream_t s, A &&...args) {
    launch_dependent_if(true, kernel, grid, block, s, static_cast<A &&>(args)...);
}

__device__ __forceinline__ void dependent_begin() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
