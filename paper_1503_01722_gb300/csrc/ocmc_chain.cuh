// ocmc_chain.cuh -- chained launches: a network pass is a chain of some twenty (forward) to a hundred
// (training) kernels of 5 to 100 us, each waiting for the one before it. Launched as programmatic
// dependents, a kernel's blocks are set up (barriers, tensor memory, weights) while the last blocks of the
// kernel before it still run, and the launch itself costs the chain nothing.
//
// What a kernel of a chain writes is thus still being written while the next ones are resident. They read it
// with ordinary loads, behind chain_wait: no __ldg and no const __restrict__ argument, which stand for data that
// does not change while the kernel lives (and which the compiler may load ahead of the wait). Those are for the
// caller's maps and the weights, which are complete before the chain starts.
#pragma once
#include <cuda_runtime.h>
#include <utility>

namespace ocmc {

// Returns once the kernel before this one in the stream has completed and its writes are visible; at once
// in a kernel that was launched plainly. Before it a kernel may only read what no kernel of its chain writes
// (a chain starts with a plain launch, so everything older has completed).
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel of the chain start once every block of this one has called it or ended.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_chained(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... a)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, k, std::forward<A>(a)...);
}

}  // namespace ocmc
