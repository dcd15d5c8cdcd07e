// compress_batch_launch.cuh -- host-side launch of compress_batch_kernel<NJ>
// (its instances are spread over two translation units to compile in parallel).
#pragma once

#include "compress_launch.cuh"

namespace glz {

template <int NJ>
static cudaError_t launch_batch_nj(const CompressArgs &A, int block, unsigned grid_req,
                                   cudaStream_t stream) {
  auto kern = compress_batch_kernel<NJ>;
  const size_t smem = static_cast<size_t>(A.sm.per_warp) * (block / 32);
  static LaunchCache lc;
  int per_sm = 0, sms = 0;
  cudaError_t e = resident_blocks(lc, kern, block, smem, &per_sm, &sms);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const uint64_t cap = static_cast<uint64_t>(per_sm) * sms;
  const unsigned grid = static_cast<unsigned>(grid_req < cap ? grid_req : cap);
  kern<<<grid, block, smem, stream>>>(A);
  return cudaGetLastError();
}

// Batches with a window beyond 256 symbols (compress_batch_wide.cu).
cudaError_t launch_batch_wide(const CompressArgs &A, uint32_t nj, int block, unsigned grid,
                              cudaStream_t stream);

}  // namespace glz
