// compress_coop_s4.cu -- instances of the block-per-chunk compression
// kernel for 4-byte symbols.
#include "compress_coop_launch.cuh"

namespace glz {
cudaError_t launch_coop_s4(const CompressArgs &A, uint32_t nw, unsigned grid,
                           cudaStream_t stream) {
  return launch_coop_t<4>(A, nw, grid, stream);
}
cudaError_t coop_blocks_s4(uint32_t nw, uint32_t smem, int *per_sm) {
  return coop_blocks_t<4>(nw, smem, per_sm);
}
}  // namespace glz
