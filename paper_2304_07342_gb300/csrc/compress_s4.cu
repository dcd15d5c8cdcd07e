// compress_s4.cu -- instantiations of the compression and sampling kernels for
// 4-byte symbols (one translation unit per symbol size so that the
// variants compile in parallel).
#include "compress_launch.cuh"
#include "sample_launch.cuh"

namespace glz {
cudaError_t launch_compress_s4(const CompressArgs &A, uint32_t nj, bool mask, int block,
                               unsigned grid, cudaStream_t stream) {
  return launch_compress_t<4>(A, nj, mask, block, grid, stream);
}
cudaError_t launch_sample_s4(const CompressArgs &A, uint32_t nj, void *clear, uint64_t clear_bytes,
                             cudaStream_t stream) {
  return launch_sample_t<4>(A, nj, clear, clear_bytes, stream);
}
cudaError_t load_parses_s4(uint32_t nj) { return load_parses_t<4>(nj); }
}  // namespace glz
