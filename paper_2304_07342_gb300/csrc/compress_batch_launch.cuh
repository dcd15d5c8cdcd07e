// compress_batch_launch.cuh -- host-side launch of compress_batch_kernel
// (its instances are spread over one translation unit per symbol size).
#pragma once

#include "compress_launch.cuh"

namespace glz {

template <int S, int NJ, bool MASK>
static cudaError_t launch_batch_nj(const CompressArgs &A, int block, unsigned grid_req,
                                   cudaStream_t stream) {
  auto kern = compress_batch_kernel<S, NJ, MASK>;
  const size_t smem = static_cast<size_t>(A.sm.per_warp) * (block / 32);
  static LaunchCache lc;
  int per_sm = 0, sms = 0;
  cudaError_t e = resident_blocks(lc, kern, block, smem, &per_sm, &sms);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const uint64_t cap = static_cast<uint64_t>(per_sm) * sms;
  const unsigned grid = static_cast<unsigned>(grid_req < cap ? grid_req : cap);
  if (A.votes) return launch_dependent(kern, grid, block, smem, stream, A);
  kern<<<grid, block, smem, stream>>>(A);
  return cudaGetLastError();
}

// One class of a batch: windows of at most 32 * nj symbols.  A mask word
// costs every position, so the mask parse has an instance for each class of
// windows; the chains only need one- or two-byte links, and an instance for
// each class where a sample chooses between the two.
template <int S>
static cudaError_t launch_batch_t(const CompressArgs &A, uint32_t nj, bool mask, int block,
                                  unsigned grid, cudaStream_t stream) {
  if (!mask && A.votes) {
    switch (nj) {
      case 4: return launch_batch_nj<S, 4, false>(A, block, grid, stream);
      case 8: return launch_batch_nj<S, 8, false>(A, block, grid, stream);
      default: return launch_batch_nj<S, 16, false>(A, block, grid, stream);
    }
  }
  if (!mask) {
    return nj <= 8 ? launch_batch_nj<S, 8, false>(A, block, grid, stream)
                   : launch_batch_nj<S, 32, false>(A, block, grid, stream);
  }
  switch (nj) {
    case 4: return launch_batch_nj<S, 4, true>(A, block, grid, stream);
    case 8: return launch_batch_nj<S, 8, true>(A, block, grid, stream);
    case 16: return launch_batch_nj<S, 16, true>(A, block, grid, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace glz
