// Host side of the programmatic launches (see pdl_sync in cph_device.cuh).
#pragma once
#include <cuda_runtime.h>

namespace cph {

// A launch that may be set up while the one before it on the stream still runs
// (every kernel launched so begins with pdl_sync).  A step is a chain of launches
// of a few microseconds: 100 steps of the 160-atom FP64 walker 6.23 -> 5.35 ms, 20
// steps of one 2003-atom walker 2.13 -> 1.88 ms, 10 steps of 64 x 2400 atoms 10.45
// -> 10.21 ms.
template <class... P, class... A>
void launch_next(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...); // the caller checks cudaGetLastError
}

} // namespace cph
