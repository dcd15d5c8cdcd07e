// compress_launch.cuh -- host-side launch of compress_kernel<S, NJ, MASK>:
// dynamic shared-memory opt-in, occupancy-sized persistent grid.
#pragma once

#include <cuda_runtime.h>

#include "compress_impl.cuh"
#include "launch_cache.cuh"

namespace glz {

template <int S, int NJ, bool MASK>
static cudaError_t launch_compress_nj(const CompressArgs &A, int block, unsigned grid_req,
                                      cudaStream_t stream) {
  auto kern = compress_kernel<S, NJ, MASK>;
  const size_t smem = static_cast<size_t>(A.sm.per_warp) * (block / 32);
  static LaunchCache lc;
  int per_sm = 0, sms = 0;
  cudaError_t e = resident_blocks(lc, kern, block, smem, &per_sm, &sms);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // never more blocks than can be resident (the grid is persistent), never
  // more than the parking slots were sized for
  const uint64_t cap = static_cast<uint64_t>(per_sm) * sms;
  const unsigned grid = static_cast<unsigned>(grid_req < cap ? grid_req : cap);
  if (A.votes) return launch_dependent(kern, grid, block, smem, stream, A);
  kern<<<grid, block, smem, stream>>>(A);
  return cudaGetLastError();
}

template <int S, int NJ>
static cudaError_t launch_compress_mode(const CompressArgs &A, bool mask, int block, unsigned grid,
                                        cudaStream_t stream) {
  if constexpr (32 * NJ <= kMaskMaxWindow)
    if (mask) return launch_compress_nj<S, NJ, true>(A, block, grid, stream);
  return launch_compress_nj<S, NJ, false>(A, block, grid, stream);
}

template <int S>
static cudaError_t launch_compress_t(const CompressArgs &A, uint32_t nj, bool mask,
                                     int block, unsigned grid, cudaStream_t stream) {
  switch (nj) {
    case 1: return launch_compress_mode<S, 1>(A, mask, block, grid, stream);
    case 2: return launch_compress_mode<S, 2>(A, mask, block, grid, stream);
    case 4: return launch_compress_mode<S, 4>(A, mask, block, grid, stream);
    case 8: return launch_compress_mode<S, 8>(A, mask, block, grid, stream);
    case 16: return launch_compress_mode<S, 16>(A, mask, block, grid, stream);
    case 32: return launch_compress_mode<S, 32>(A, mask, block, grid, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace glz
