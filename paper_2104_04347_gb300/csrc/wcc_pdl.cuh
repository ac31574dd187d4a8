// wcc_pdl.cuh -- half-step launches that overlap the previous one's end
// (programmatic dependent launch).
//
// A half-step needs everything the previous one wrote, so its CTAs can only
// start working when that grid is complete; but the launch itself is ready by
// then.  Every half-step kernel begins with pdl_begin(), which waits for the
// previous grid (complete, its writes visible).  Nothing that a half-step writes
// may be read before it, and stages are not read through the read-only path
// (__ldg), whose data must not change while the grid exists.
//
// No kernel asks for the next one to be placed early
// (griddepcontrol.launch_dependents): its waiting CTAs would fill the slots that a
// grid of less than one wave leaves free, unevenly over the SMs.  With the request
// at the start of the kernel and without: FP64 Euler P = 3 at 2^15 cells 47.6 and
// 33.7 us per half-step, FP32-mixed Euler P = 3 at 2^17 10.4 and 9.0 us (in pairs 8.4 and
// 7.0), P = 2 at 370 000 cells 16.2 and 13.9; elsewhere the request gained 6 % at most
// (FP64 advection P = 2 at 2^14 cells 6.0 and 6.3, FP32-mixed Euler P = 3 at 2^18 11.3 and
// 11.6, at 2^22 117.2 and 117.5).
#pragma once

#include <cuda_runtime.h>

namespace wcc {

__device__ __forceinline__ void pdl_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
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

// Position in the list of tiles of the i-th of n tiles to start: the stages are
// two buffers used in turn, and a half-step that reads the upper one walks the
// tiles backwards.  What the half-step before wrote last is then read first,
// while L2 (129 MB) still holds it; a stage larger than L2 walked always in one
// direction has lost those lines when it reaches them.  Parents are read once
// (one of a tile's 256 also by its neighbour), so their lines leave first
// (load_once).  FP32-mixed Euler, P = 3, per half-step: 2^22 cells
// (251 MB a stage) 125.5 -> 121.6 us, the batch of 768 meshes 248.0 -> 238.5 us
// (246.2 from the direction, the rest from the loads), 2^20 cells in pairs
// 23.2 -> 22.9 us.  Scalar systems (LARGE false: a third of the bytes) keep one
// direction and plain loads, which is the better choice for P = 1 at every size
// (Burgers at 2^22 cells, 67 MB a stage, 39.4 us, 40.8 with both) and up to 2^20 cells
// above (P = 4 at 250 007 cells 7.0 us, 7.3 with both; at 2^22, 100 MB, 78.0 and 76.6).
template <bool LARGE>
__device__ __forceinline__ long long sweep_index(const void* in, const void* out, long long i, long long n) {
    return LARGE && in > out ? n - 1 - i : i;
}
template <bool LARGE>
__device__ __forceinline__ float load_once(const float* p) { return LARGE ? __ldcs(p) : *p; }

}  // namespace wcc
