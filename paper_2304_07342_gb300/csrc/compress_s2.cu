// compress_s2.cu -- instantiations of the compression and sampling kernels for
// 2-byte symbols (one translation unit per symbol size so that the
// variants compile in parallel).
#include "compress_launch.cuh"
#include "sample_launch.cuh"

namespace glz {
cudaError_t launch_compress_s2(const CompressArgs &A, uint32_t nj, bool mask, int block,
                               unsigned grid, cudaStream_t stream) {
  return launch_compress_t<2>(A, nj, mask, block, grid, stream);
}
cudaError_t launch_sample_s2(const CompressArgs &A, uint32_t nj, void *clear, uint64_t clear_bytes,
                             cudaStream_t stream) {
  return launch_sample_t<2>(A, nj, clear, clear_bytes, stream);
}
cudaError_t load_parses_s2(uint32_t nj) { return load_parses_t<2>(nj); }
}  // namespace glz
