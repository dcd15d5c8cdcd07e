// compress_batch.cu -- one persistent launch over the chunks of many buffers
// (each with its own parameters), plus the headers of empty buffers.
#include "compress_batch_launch.cuh"

namespace glz {

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

cudaError_t launch_compress_batch(const CompressArgs &A, const BufDesc *empties,
                                  uint32_t n_empty, uint32_t nj, int block, unsigned grid,
                                  cudaStream_t stream) {
  if (n_empty) {
    batch_empty_headers<<<(n_empty + 7) / 8, 256, 0, stream>>>(empties, n_empty);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (A.total_chunks == 0) return cudaSuccess;
  switch (nj) {
    case 1:
    case 2:
    case 4: return launch_batch_nj<4>(A, block, grid, stream);
    case 8: return launch_batch_nj<8>(A, block, grid, stream);
    default: return launch_batch_wide(A, nj, block, grid, stream);
  }
}

}  // namespace glz
