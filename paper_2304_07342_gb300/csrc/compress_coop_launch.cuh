// compress_coop_launch.cuh -- host-side launch of compress_coop_kernel<S, NW>.
#pragma once

#include "compress_coop.cuh"
#include "launch_cache.cuh"

namespace glz {

template <int S, int NW>
static cudaError_t launch_coop_nw(const CompressArgs &A, unsigned grid_req, cudaStream_t stream) {
  auto kern = compress_coop_kernel<S, NW>;
  static LaunchCache lc;
  int per_sm = 0, sms = 0;
  cudaError_t e = resident_blocks(lc, kern, 32 * kCoopWarps, A.coop.total, &per_sm, &sms);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const uint64_t cap = static_cast<uint64_t>(per_sm) * sms;
  const unsigned grid = static_cast<unsigned>(grid_req < cap ? grid_req : cap);
  kern<<<grid, 32 * kCoopWarps, A.coop.total, stream>>>(A);
  return cudaGetLastError();
}

template <int S>
static cudaError_t launch_coop_t(const CompressArgs &A, uint32_t nw, unsigned grid,
                                 cudaStream_t stream) {
  switch (nw) {
    case 4: return launch_coop_nw<S, 4>(A, grid, stream);
    case 8: return launch_coop_nw<S, 8>(A, grid, stream);
    case 16: return launch_coop_nw<S, 16>(A, grid, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace glz
