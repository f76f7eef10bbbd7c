// dvc_chain.cuh -- launches that start while the launch before them still runs.
//
// A chain of short kernels pays for each launch and for each kernel's prologue
// (barriers, TMEM, tables, weights) between the last block of one and the first
// work of the next.  launch_chained() lets a kernel's blocks start as soon as every
// block of the launch before it in the stream has called chain_next(); it calls
// chain_wait() before it touches anything that launch may write or still read, which
// returns when that launch has ended and its writes are visible.  Every kernel that is
// launched so, or before one that is, calls chain_wait() in every block, so that the
// end of one launch implies the end of all before it.  A kernel launched in the
// ordinary way waits for nothing there.
#pragma once
#include <cuda_runtime.h>

namespace dvc {

__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... KA, class... A>
cudaError_t launch_chained(void (*kernel)(KA...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                           A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KA(args)...);
}

}  // namespace dvc
