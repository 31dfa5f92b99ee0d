#include "moment_stream_impl.cuh"

namespace sobek {
cudaError_t moment_stream_dual(const MsArgs& a, int grid, int smem, bool loaders_edge, cudaStream_t s) {
    return loaders_edge ? moment_stream_launch<true, true>(a, grid, smem, s) : moment_stream_launch<true, false>(a, grid, smem, s);
}
}  // namespace sobek
