// Programmatic dependent launch: a kernel of a chain may be set up (its blocks scheduled, barriers
// initialised, tables read) while the kernel before it drains, instead of after it has ended.  Every
// block calls pdl_wait before it reads what an earlier kernel wrote, or writes what one may still
// read; until then it may only touch memory that no kernel writes (descriptors, tensor maps, tables,
// c^2).  pdl_trigger lets the next kernel of the chain start being set up.  Worth about 1.5 us a
// launch: a fifth of a pass on a single 601 x 301 shot.
#pragma once

#include <cuda_runtime.h>

namespace ewv {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
int launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...) == cudaSuccess ? 0 : -1;
}

}  // namespace ewv
