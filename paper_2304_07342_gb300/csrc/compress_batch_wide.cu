// compress_batch_wide.cu -- batches with a window beyond 256 symbols.
#include "compress_batch_launch.cuh"

namespace glz {
cudaError_t launch_batch_wide(const CompressArgs &A, uint32_t nj, int block, unsigned grid,
                              cudaStream_t stream) {
  switch (nj) {
    case 16: return launch_batch_nj<16>(A, block, grid, stream);
    case 32: return launch_batch_nj<32>(A, block, grid, stream);
    default: return cudaErrorInvalidValue;
  }
}
}  // namespace glz
