// lbm_pdl.h -- programmatic dependent launch: a launch that may start while the previous launch of
// its stream drains, and the two instructions its kernel uses.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

// Programmatic dependent launch: let the next launch of the stream start; wait for the complete
// end of the previous one (no-ops in a launch without the attribute).
__device__ __forceinline__ void pdl_launch_next_() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait_() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A launch that may start while the previous launch of its stream drains (the kernel calls
// pdl_wait_ before it touches what that one wrote).
struct PdlLaunch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    PdlLaunch(dim3 grid, dim3 block, size_t smem, cudaStream_t s)
    {
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.gridDim = grid, cfg.blockDim = block, cfg.dynamicSmemBytes = smem, cfg.stream = s;
        cfg.attrs = at, cfg.numAttrs = 1;
    }
};

}  // namespace lbm
