// Programmatic dependent launch: a kernel's blocks may start while the kernel
// before it on the stream drains, do what needs none of its results, and wait
// for its completion (and the visibility of its writes) before they touch
// anything that it reads or writes.  A step of a small mesh is a chain of short
// kernels, and the launch latency between two of them is a good part of it.
// Without the attribute both instructions do nothing.
//
// Such a kernel is resident while the kernel before it still writes, so what any
// kernel writes (states, traces, partial sums, clocks) is read with ordinary
// coherent loads after the wait.  The read-only path (__ldg, or a const
// __restrict__ kernel parameter, which the compiler may take as one) is for the
// operator's tables, uploaded by blocking copies before any launch: its loads need
// data that stay the same for the kernel's whole life, and no wait orders them.
#pragma once

#include <cuda_runtime.h>

// Every thread of every block executes this before its first access to data
// that an earlier kernel writes, and before its first write.
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The next kernel's blocks may be scheduled from here on.
__device__ __forceinline__ void release_successor() { asm volatile("griddepcontrol.launch_dependents;"); }

template <class... P, class... A>
void launch_dependent(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, const A&... args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3((unsigned)threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute a[1] = {};
    a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = a;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}
