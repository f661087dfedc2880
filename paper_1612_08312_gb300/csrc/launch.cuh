// launch.cuh -- launches of a sweep's kernels that overlap the start of each
// with the end of the one before it.
//
// A sweep is six or seven dependent launches, and a small lattice's kernels
// run for a few microseconds each, so the gap between two of them is a good
// part of the sweep.  A kernel launched with launch_overlapped is placed on
// the SMs as soon as every block of its predecessor in the stream has called
// overlap_next (programmatic stream serialization), and waits there for the
// predecessor's end and its memory in overlap_wait.  Every thread of every
// such kernel calls overlap_wait before it touches global memory, so that the
// end of a kernel implies the end of all before it.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace pyro {

constexpr int GPU_SMS = 152;                // multiprocessors of a GB300
constexpr int GPU_THREADS = GPU_SMS * 2048;  // threads it holds at once

__device__ __forceinline__ void overlap_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void overlap_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void overlap_begin()
{
    overlap_wait();
    overlap_next();
}

// Errors are left for cudaGetLastError, as with <<< >>>.
template <typename... P, typename... A>
inline void launch_overlapped(void (*k)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A &&...args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = a;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, k, std::forward<A>(args)...);
}

}  // namespace pyro
