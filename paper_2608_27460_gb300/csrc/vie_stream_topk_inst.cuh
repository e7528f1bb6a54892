// vie_stream_topk_inst.cuh - body shared by the per-width instantiation
// units: sets the shared-memory opt-in once per device and launches.
#pragma once

#include "vie_launch.h"

namespace vie {

template <int NB, int kR, bool Q8>
cudaError_t launch_one(const StreamTopkParams &p, int grid, uint32_t smem, cudaStream_t stream) {
    static bool configured[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        e = cudaFuncSetAttribute(stream_topk_kernel<NB, kR, Q8>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
        if (e != cudaSuccess) return e;
        configured[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(threads_for<NB>());
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, stream_topk_kernel<NB, kR, Q8>, p);
}

template <int NB, bool Q8>
cudaError_t launch_width(int r, const StreamTopkParams &p, int grid, uint32_t smem,
                         cudaStream_t stream) {
    switch (r) {
        case 1: return launch_one<NB, 1, Q8>(p, grid, smem, stream);
        case 2: return launch_one<NB, 2, Q8>(p, grid, smem, stream);
        case 4: return launch_one<NB, 4, Q8>(p, grid, smem, stream);
        case 8:  // narrow rows, one query: 64-row stages
            if constexpr (NB == 1) return launch_one<NB, 8, Q8>(p, grid, smem, stream);
            return cudaErrorInvalidValue;
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace vie
