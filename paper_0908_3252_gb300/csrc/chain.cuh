// chain.cuh -- kernels that follow each other on one stream without a gap
// (programmatic dependent launch).  A kernel launched by `chain` may be placed
// on the device before its predecessor has ended: from the predecessor's
// chain_next on, else as its blocks exit.  chain_enter, its first statement (or
// the first after a set-up that reads no global memory: barriers, tensor
// memory), waits until the predecessor has completed and its writes are visible.
// chain_next comes after chain_enter, or in a kernel with a plain launch, so at
// most two kernels of a chain overlap and everything from before the
// predecessor is complete when a kernel starts.
// What the predecessor wrote must not be read through the read-only path (__ldg,
// const __restrict__): the compiler may move such loads above the wait.
//
// The T apply of a small image and the minimisers' graphs are chains of kernels
// of a few microseconds.  Placing the next kernel early (chain_next) pays for
// the short row and column passes; it costs where a kernel fills the SMs once
// (four iterations at 2048^2: 1367 us, 1697 with chain_next in every kernel, as
// the next kernel's blocks then crowd on the SMs that empty first), so only
// those passes do it.
#pragma once

#include <cuda_runtime.h>

namespace spirec {

__device__ __forceinline__ void chain_enter() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// kern<<<grid, block, smem, st>>>(args...) as the next kernel of a chain; kern
// starts with chain_enter().
template <typename... P, typename... A>
void chain(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);  // errors: cudaGetLastError
}

}  // namespace spirec
