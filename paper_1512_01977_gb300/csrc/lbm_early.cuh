#pragma once

#include <cuda_runtime.h>

namespace lbm {

// A launch that may start while its predecessor on the stream still runs; the
// kernel waits for it before it touches memory (griddepcontrol.wait).
template <typename... KA, typename... A>
static cudaError_t launch_early(void (*k)(KA...), unsigned grid, int nt, cudaStream_t s, const A&... a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(nt);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, a...);
}

}  // namespace lbm
