// Instantiations of the streaming top-k kernel for query groups of 4.
#include "vie_stream_topk_inst.cuh"

namespace vie {
cudaError_t launch_stream_topk_nb4(int r, const StreamTopkParams &p, int grid,
                                   uint32_t smem, cudaStream_t stream) {
    return launch_width<4, false>(r, p, grid, smem, stream);
}
}  // namespace vie
