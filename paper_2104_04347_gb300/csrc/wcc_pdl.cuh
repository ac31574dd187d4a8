// wcc_pdl.cuh -- half-step launches that overlap the previous one's end
// (programmatic dependent launch).
//
// A half-step needs everything the previous one wrote, so its CTAs can only
// start working when that grid is complete; but they can be launched, placed on
// their SMs and waiting by then.  Every half-step kernel begins with
// pdl_begin(): wait for the previous grid (complete, its writes visible), then
// allow the next one to be placed.  Nothing that a half-step writes may be
// read before it, so the stages are read with ordinary loads: the read-only
// path (__ldg) lets the compiler move a load above the wait.
#pragma once

#include <cuda_runtime.h>

namespace wcc {

__device__ __forceinline__ void pdl_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// kernel<<<grid, block, smem, stream>>>(args) with programmatic stream
// serialisation (a programmatic edge when captured into a graph).
template <class A>
cudaError_t launch_pdl(void (*kernel)(A), dim3 grid, unsigned block, size_t smem, cudaStream_t stream, const A& args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args);
}

}  // namespace wcc
