// compress_coop_launch.cuh -- host-side launch of compress_coop_kernel<S, NW>.
#pragma once

#include "compress_coop.cuh"
#include "launch_cache.cuh"

namespace glz {

// The launch cache of a kernel instance, for its launch and for the question
// how many blocks run at once.
template <int S, int NW>
static LaunchCache &coop_cache() {
  static LaunchCache lc;
  return lc;
}

template <int S, int NW>
static cudaError_t coop_blocks_nw(uint32_t smem, int *per_sm) {
  int sms = 0;
  return resident_blocks(coop_cache<S, NW>(), compress_coop_kernel<S, NW>, 32 * kCoopWarps, smem,
                         per_sm, &sms);
}

template <int S>
static cudaError_t coop_blocks_t(uint32_t nw, uint32_t smem, int *per_sm) {
  switch (nw) {
    case 4: return coop_blocks_nw<S, 4>(smem, per_sm);
    case 8: return coop_blocks_nw<S, 8>(smem, per_sm);
    case 16: return coop_blocks_nw<S, 16>(smem, per_sm);
    default: return cudaErrorInvalidValue;
  }
}

template <int S, int NW>
static cudaError_t launch_coop_nw(const CompressArgs &A, unsigned grid_req, cudaStream_t stream) {
  auto kern = compress_coop_kernel<S, NW>;
  int per_sm = 0, sms = 0;
  cudaError_t e = resident_blocks(coop_cache<S, NW>(), kern, 32 * kCoopWarps, A.coop.total, &per_sm, &sms);
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
