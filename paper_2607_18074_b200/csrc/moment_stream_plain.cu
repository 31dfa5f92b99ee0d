#include "moment_stream_impl.cuh"

namespace sobek {
cudaError_t moment_stream_plain(const MsArgs& a, int grid, int smem, cudaStream_t s) { return moment_stream_launch<false>(a, grid, smem, s); }
}  // namespace sobek
