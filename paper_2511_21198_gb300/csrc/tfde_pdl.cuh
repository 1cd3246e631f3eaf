// Programmatic launches of the small kernels of the device-side loops: the next
// kernel's launch and block set-up run while the previous one drains.  At 16^3
// an iteration is 15 kernels of 1 to 2 us of work each (16^3 7.45 -> 7.33 ms per
// 16 steps, 40 x 32 x 24 10.4 -> 10.3 ms per 8).  Only for grids below one block
// per SM: the next kernel's waiting blocks take the place of the running one's
// (128^3 non-symmetric 29.8 -> 31.1 ms).
//
// A kernel launched so calls pdl_begin() before anything else.  Every kernel of
// a chain does, so when one has passed it, all but its direct predecessor had
// ended before and the predecessor has now: nothing older needs a wait.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace tfde {

__device__ __forceinline__ void pdl_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

constexpr int kPdlBlocks = 152;   // of a sweep over the grid's points: one per SM

template <typename... P, typename... A>
inline cudaError_t launch_pdl_smem(bool early, void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t s,
                                   A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(std::forward<A>(args))...);
}
template <typename... P, typename... A>
inline void launch_pdl(bool early, void (*kernel)(P...), int grid, int block, cudaStream_t s, A&&... args) {
    launch_pdl_smem(early, kernel, grid, block, 0, s, std::forward<A>(args)...);
}

}  // namespace tfde
