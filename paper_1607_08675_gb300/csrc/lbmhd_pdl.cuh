// lbmhd_pdl.cuh -- programmatic dependent launch of kernels that follow one
// another in a stream (a step after a step): the next grid is set up while this
// one runs and waits, in after_previous(), until it has completed and its
// stores are visible, so a step's launch latency is not paid between steps.
//
// A kernel launched with launch_after calls after_previous() before it
// touches memory, and takes its pointers without __restrict__: with it the
// compiler may read them as data that no one writes while the grid exists, by
// the non-coherent path or ahead of the wait, and the grid before this one
// writes them then.  No kernel triggers its successor early: blocks placed
// while the last ones still run pile up on the SMs that are free by then (FP64
// 256^2 28.8 us per step instead of 21.3).
//
// us per step, plain launches / this, by calls of 20 steps: FP32 256^2 4.5 /
// 2.7, 512^2 8.3 / 5.5, FP64 64^2 8.3 / 6.8; replayed from a graph: FP32 256^2
// 2.9 / 2.5, 512^2 5.6 / 5.1.
#pragma once

#include <cuda_runtime.h>

namespace lbmhd {

__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... Params, class... Args>
cudaError_t launch_after(void (*kernel)(Params...), unsigned grid, int block, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

}  // namespace lbmhd
