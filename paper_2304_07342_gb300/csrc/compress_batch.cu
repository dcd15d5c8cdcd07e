// compress_batch.cu -- the launches of a compression batch: the headers of
// empty buffers and the launches of each class of buffers.
#include "compress_impl.cuh"

namespace glz {

cudaError_t launch_batch_s1(const CompressArgs &A, uint32_t nj, bool mask, int block,
                            unsigned grid, cudaStream_t stream);
cudaError_t launch_batch_s2(const CompressArgs &A, uint32_t nj, bool mask, int block,
                            unsigned grid, cudaStream_t stream);
cudaError_t launch_batch_s4(const CompressArgs &A, uint32_t nj, bool mask, int block,
                            unsigned grid, cudaStream_t stream);

// Empty buffers: their stream is the header alone.
__global__ void batch_empty_headers(const BufDesc *empties, uint32_t n) {
  const uint32_t lane = threadIdx.x & 31;
  for (uint32_t i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n;
       i += gridDim.x * (blockDim.x >> 5)) {
    const BufDesc B = empties[i];
    write_header(B, lane);
    if (lane == 0) *B.out_bytes = kHeaderBytes;
  }
}

cudaError_t launch_batch_empties(const BufDesc *empties, uint32_t n, cudaStream_t stream) {
  batch_empty_headers<<<(n + 7) / 8, 256, 0, stream>>>(empties, n);
  return cudaGetLastError();
}

cudaError_t launch_batch_class(const CompressArgs &A, uint32_t S, uint32_t nj, bool mask,
                               int block, unsigned grid, cudaStream_t stream) {
  switch (S) {
    case 1: return launch_batch_s1(A, nj, mask, block, grid, stream);
    case 2: return launch_batch_s2(A, nj, mask, block, grid, stream);
    default: return launch_batch_s4(A, nj, mask, block, grid, stream);
  }
}

}  // namespace glz
