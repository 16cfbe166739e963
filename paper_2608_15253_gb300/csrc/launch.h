// Launch with programmatic stream serialisation where kernels are short: the
// kernel is made ready while its predecessor on the stream drains, and waits
// in dep_wait() (common.cuh) until that has finished and its writes are
// visible.  Captured into a graph the edge stays programmatic.  Only for
// kernels that call dep_wait() before their first access to data of earlier
// kernels, and that read such data with plain loads: __ldg, and a const
// __restrict__ pointer, which lets the compiler make one of a load, are for
// data that is constant from the kernel's launch on, here the tables filled at
// setup (twiddles, tensor, materials), and may be moved above the wait.
#pragma once

#include <cuda_runtime.h>

#include "ctx.h"

namespace mm {

// Single instances up to 128 K cells: their kernels take a few microseconds
// (200x50, one step: 174 -> 167 us; 128x32 FP64 3.86 -> 3.78 ms; 256x256 at
// 300 K 1.65 -> 1.62).  Larger grids and ensembles lost 1 to 2 % to it (512x512
// film 1.53 -> 1.55 ms, uneven replicas 7.37 -> 7.52).
inline bool short_kernels(const mm_ctx* c) { return !c->batch && c->N <= 131072; }

template <typename... P, typename... A>
inline cudaError_t launch_dep(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, const mm_ctx* c, A&&... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cfg.attrs = &at;
    cfg.numAttrs = short_kernels(c) ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

}  // namespace mm
