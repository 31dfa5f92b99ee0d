#include "moment_stream_impl.cuh"

namespace sobek {
cudaError_t moment_stream_dual(const MsArgs& a, int grid, int smem, cudaStream_t s) { return moment_stream_launch<true>(a, grid, smem, s); }
}  // namespace sobek
