// Launch with programmatic dependent launch allowed: the kernel may start while
// the previous kernel on the stream finishes (every kernel launched this way
// executes griddepcontrol.wait before reading what its predecessor writes). A
// refused attribute falls back to a plain launch.
#pragma once
#include <cuda_runtime.h>

namespace mpr {

template <typename... KArgs, typename... Args>
void launch_pdl(void (*k)(KArgs...), dim3 grid, dim3 block, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, k, args...) != cudaSuccess) {
        cudaGetLastError();
        k<<<grid, block, 0, s>>>(args...);
    }
}

}  // namespace mpr
