// Launches that overlap the end of the kernel before them in the stream
// (programmatic dependent launch).  A step is a chain of short dependent
// kernels; started the ordinary way each waits for the one before to drain and
// then for its own launch, about 4 us a kernel on this GPU.  Here a kernel's
// CTAs may take their places while the kernel before is finishing, and wait
// on the device for its results.
//
// Every kernel launched this way calls pdl_wait() in every thread before it
// writes global memory and before an early return (the next kernel's wait
// covers only kernels that have themselves waited), and pdl_launch() once its
// successor may take places.  What it reads before its wait is one of
//  - what only the host's copies write (hyetographs, inflow series, scenario
//    descriptors): a kernel after a copy starts when the copy has ended;
//  - a first reading that it takes again after the wait and acts on only if it
//    still holds: the plan kernels' clocks, maximum depths, rain multipliers
//    and window end.
// The first reading is of use because the clock is there by then: a step
// kernel calls pdl_wait_launch(), so the next plan starts only when the plan
// before has finished and its writes are visible.
#pragma once

#include <cuda_runtime.h>

namespace flood {

// Wait until every kernel before this one has finished and its writes are
// visible.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The kernel after this one may start to take places.
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// For a kernel whose successor reads ahead what the kernel before this one wrote.
__device__ __forceinline__ void pdl_wait_launch()
{
    pdl_wait();
    pdl_launch();
}

template <class... P, class... A>
inline cudaError_t launch_pdl(void (*f)(P...), dim3 grid, dim3 block, size_t shm, cudaStream_t s, const A&... a)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = shm;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, f, P(a)...);
}

}  // namespace flood
