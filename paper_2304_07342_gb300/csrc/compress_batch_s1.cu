// compress_batch_s1.cu -- instances of the batch compression kernel for
// 1-byte symbols.
#include "compress_batch_launch.cuh"

namespace glz {
cudaError_t launch_batch_s1(const CompressArgs &A, uint32_t nj, bool mask, int block,
                            unsigned grid, cudaStream_t stream) {
  return launch_batch_t<1>(A, nj, mask, block, grid, stream);
}
}  // namespace glz
