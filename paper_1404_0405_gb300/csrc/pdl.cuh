// Dependent launches without the gap between kernels (programmatic dependent launch).
//
// A step is a chain of 70 to 150 kernels, each needing all of the one before.  With an
// ordinary launch a kernel's blocks are scheduled only after the kernel before has
// drained (about 1 us of idle GPU inside a captured graph, 2-3 us between eager
// launches).  A kernel launched by launch_chain may be scheduled while its predecessor
// runs; every thread of it waits in chain_wait() until the predecessor has completed
// and its writes are visible.  So every kernel launched this way calls chain_wait()
// first, before any return and any memory access: completion then carries over the whole
// chain.
//
// It pays while the kernels are short: a step of 8 members at Jmax 7 takes 1.16 ms chained
// and 1.37 ms not.  Long kernels lose by it (64 members at Jmax 6..9: 8.5 ms chained, 7.9
// ms not): the successor's early blocks run in the predecessor's split of shared
// memory and L1.  So the caller says, from the size of the grid (CHAIN_PATCHES).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <utility>

namespace sww {

// active patches (of all members) up to which a step's launches are chained
constexpr int64_t CHAIN_PATCHES = 16384;

// (nothing to wait for in an ordinary launch)
__device__ __forceinline__ void chain_wait() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class... P, class... A>
cudaError_t launch_chain(bool chain, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid, cfg.blockDim = block, cfg.dynamicSmemBytes = smem, cfg.stream = s;
    cfg.attrs = attr, cfg.numAttrs = chain ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

}  // namespace sww
