// compress_coop_s1.cu -- instances of the block-per-chunk compression
// kernel for 1-byte symbols.
#include "compress_coop_launch.cuh"

namespace glz {
cudaError_t launch_coop_s1(const CompressArgs &A, uint32_t nw, unsigned grid,
                           cudaStream_t stream) {
  return launch_coop_t<1>(A, nw, grid, stream);
}
}  // namespace glz
