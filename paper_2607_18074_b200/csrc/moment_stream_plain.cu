#include "moment_stream_impl.cuh"

namespace sobek {
cudaError_t moment_stream_plain(const MsArgs& a, int grid, int smem, bool loaders_edge, cudaStream_t s) {
    return loaders_edge ? moment_stream_launch<false, true>(a, grid, smem, s) : moment_stream_launch<false, false>(a, grid, smem, s);
}
}  // namespace sobek
