// pdl.cuh -- programmatic dependent launch of the time-step kernels.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

// Programmatic dependent launch of the step kernels (LBM_PDL): a step kernel is launched
// so that its blocks may be scheduled while the kernel before it on the stream drains its
// last wave; every block first waits (griddepcontrol.wait) for that kernel's completion
// and memory -- before it reads or writes anything -- and then allows the next step's
// launch to begin (griddepcontrol.launch_dependents).  Launched without the attribute
// (the slab path) both instructions do nothing.
#ifndef LBM_PDL
#define LBM_PDL 1
#endif
__device__ __forceinline__ void pdl_begin() {
    if (LBM_PDL) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
}

template <typename... Params, typename... Args>
cudaError_t launch_pdl_smem(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                            Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = LBM_PDL ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename... Params, typename... Args>
cudaError_t launch_pdl(void (*kernel)(Params...), dim3 grid, dim3 block, cudaStream_t st, Args... args) {
    return launch_pdl_smem(kernel, grid, block, 0, st, args...);
}

}  // namespace lbm
