// smi_pdl.h -- programmatic dependent launch for the kernels of a time loop.
//
// A kernel launched with launch_pdl may start while the kernel before it on
// the stream is still running its last blocks; it calls pdl_wait before it
// touches anything that an earlier kernel of the loop writes (the wait
// returns when that kernel has finished and its writes are visible), and
// pdl_trigger after it, so that at most two kernels of the chain overlap:
// what was written two kernels ago or earlier may be read before the wait.
#pragma once

#include <cuda_runtime.h>

#include "smi_internal.h"

namespace smi {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
void launch_pdl(const LaunchCtx &lc, void (*kernel)(P...), dim3 grid, int block, size_t smem, A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = static_cast<cudaStream_t>(lc.stream);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
    ++*lc.launches;
}

}  // namespace smi
