// Programmatic dependent launch of the kernels of a solve's iteration.
//
// A kernel launched with launch_pdl may start while the one before it in the stream drains.  Every thread calls pdl_wait()
// before its first access to memory that the solve writes; it returns when the kernel before is complete with all its
// writes, and then lets the next one start.  (A kernel that lets the next one start has itself waited, so whatever lies
// further back is complete too, and a launch by other means waits for everything as always.)  So launch latency, the wait
// for free SMs and the set-up of tables overlap the tail before them.
//
// After anything that is not a kernel, or under a tool that serialises, the launch is an ordinary one and pdl_wait()
// returns at once.  FP16 defect correction on 16^3 elements of nx = 10 (1655 iterations of
// 5 launches): 160 -> 148 ms; 20 iterations on 24^3 elements 10.5 -> 10.2 ms.
#pragma once

#include <cuda_runtime.h>

namespace nek {

// p...: pointers that the wait redefines, so that no load through them, const __restrict__ or not, can be moved above
// it, or be made a read-only one.  A kernel gives its scalars, and what else the kernel just before it may still write
// while this one runs, where it is a const __restrict__ parameter (which may be read as data that nothing writes for as
// long as the kernel runs): k_alpha's and k_beta's partial sums.  What lies further back is complete before this kernel
// starts; it is read after a test of the scalars, or through pointers that are written in the same kernel.
// (Redefining all of k_ax_fx's DirUpdate takes it from the constant bank into registers: 10.25 -> 10.57 ms for the 20
// iterations.)
template <class... P>
__device__ __forceinline__ void pdl_wait(P&... p)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    (([&] { asm volatile("" : "+l"(p)::"memory"); }()), ...);
}

// Lets the next kernel start; after pdl_wait.
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;"); }

template <class... P, class... A>
void launch_pdl(void (*k)(P...), int grid, int block, size_t smem, cudaStream_t s, A... a)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, k, static_cast<P>(a)...);  // the error is read by check_launch
}

}  // namespace nek
