// Launch of a kernel of a chain: with programmatic stream serialization, so
// that its blocks are scheduled as the previous kernel's drain instead of
// after a full launch latency (about 2 us between dependent kernels without
// it).  The kernel starts with pdl_wait() (device_common.cuh).
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "grf_internal.h"

namespace grf {

template <class... P, class... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t st,
                                  A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(static_cast<unsigned>(block));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(std::forward<A>(args))...);
    if (e == cudaSuccess) count_launches(1);
    return e;
}

}  // namespace grf
