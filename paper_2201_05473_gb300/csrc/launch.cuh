// Launches of a chain of kernels on one stream, each overlapping its start
// with the tail of the one before (programmatic dependent launch).
//
// A chained kernel calls chain_begin() before it touches global memory. The
// hardware may bring its blocks up once every block of the kernel before has
// started (and called chain_begin), and holds them there until that kernel has
// completed and its writes are visible: the same order as a plain launch,
// without the launch latency and the ramp between the two. With chain_wait()
// alone a kernel does not let its successor in before it completes, which is
// the faster form ahead of the fluid kernel (faraday_kernel). Behind a kernel that is not
// chained, a copy or an event the launch is ordered as usual.
//
// What makes that order sound: griddepcontrol.wait holds a thread until the
// prerequisite grids have completed and their memory operations are performed
// and visible to its grid (PTX ISA, griddepcontrol); every thread of every
// chained kernel waits first thing, so the order carries over from kernel to
// kernel; the compiler keeps later accesses behind the wait (volatile, with a
// memory clobber); and what a predecessor may have written is read with
// coherent loads (ld_state or plain ones), not through the read-only path,
// whose data must not change while the kernel runs.
#pragma once

#include <utility>

#include <cuda_runtime.h>

namespace pwfa {

__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void chain_begin() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    chain_wait();
}

// Multiprocessors of the current device.
inline cudaError_t sm_count(int* n) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    return e == cudaSuccess ? cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev) : e;
}

template <class... P, class... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t s, A&&... args) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

}  // namespace pwfa
