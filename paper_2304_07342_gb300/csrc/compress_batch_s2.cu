// compress_batch_s2.cu -- instances of the batch compression kernel for
// 2-byte symbols.
#include "compress_batch_launch.cuh"

namespace glz {
cudaError_t launch_batch_s2(const CompressArgs &A, uint32_t nj, bool mask, int block,
                            unsigned grid, cudaStream_t stream) {
  return launch_batch_t<2>(A, nj, mask, block, grid, stream);
}
}  // namespace glz
