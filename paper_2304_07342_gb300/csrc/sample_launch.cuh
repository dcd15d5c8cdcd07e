// sample_launch.cuh -- the sampling kernel (sample.cuh) and its launch.
#pragma once

#include "compress_impl.cuh"

namespace glz {

// Clears `words` 16-byte words at `clear` and samples the launch of A: block b
// < kSampleWarps / 8 takes pieces, every block clears.
template <int S, int NW>
__global__ void __launch_bounds__(kSampleBlock) sample_kernel(const __grid_constant__ CompressArgs A,
                                                             uint4 *clear, uint64_t words) {
  grid_launch_next();
  __shared__ __align__(16) uint8_t pieces[8][sample_symbols(NW) * S];
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < words;
       i += stride)
    clear[i] = make_uint4(0, 0, 0, 0);
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, w = blockIdx.x * 8 + warp;
  if (w >= kSampleWarps) return;
  const uint32_t h = sample_hash(w), first = A.first_ticket < A.end_chunk ? A.first_ticket : 0u;
  const uint32_t v = sample_piece<S, NW>(A.buf, first + __umulhi(h, A.end_chunk - first),
                                         sample_place(h), pieces[warp], lane);
  if (lane == 0) A.votes[w] = v;
}

// For launches with the parse by masks; `clear`: 16-byte aligned.
template <int S>
static cudaError_t launch_sample_t(const CompressArgs &A, uint32_t nj, void *clear,
                                   uint64_t clear_bytes, cudaStream_t stream) {
  const uint64_t words = clear_bytes / 16;
  uint64_t grid = (words + kSampleBlock - 1) / kSampleBlock;
  if (grid < kSampleWarps / 8) grid = kSampleWarps / 8;
  if (grid > 128) grid = 128;
  auto go = [&](auto kern) {
    kern<<<static_cast<unsigned>(grid), kSampleBlock, 0, stream>>>(A, static_cast<uint4 *>(clear),
                                                                   words);
    return cudaGetLastError();
  };
  // (the windows of the kernel instance decide: candidates outside W are
  // masked out)
  if (nj <= 4) return go(sample_kernel<S, 4>);
  if (nj <= 8) return go(sample_kernel<S, 8>);
  return go(sample_kernel<S, 16>);
}

// Load the code of every kernel that a call with symbols of S bytes and windows
// of 32 * nj symbols can launch (loading is lazy and takes device memory).
template <int S, int NJ>
static cudaError_t load_parses_nj() {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, compress_kernel<S, NJ, false>);
  if constexpr (32 * NJ <= kMaskMaxWindow) {
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, compress_kernel<S, NJ, true>);
    if (e == cudaSuccess)
      e = cudaFuncGetAttributes(&a, sample_kernel<S, (NJ <= 4 ? 4 : NJ)>);
  }
  return e;
}

template <int S>
static cudaError_t load_parses_t(uint32_t nj) {
  switch (nj) {
    case 1: return load_parses_nj<S, 1>();
    case 2: return load_parses_nj<S, 2>();
    case 4: return load_parses_nj<S, 4>();
    case 8: return load_parses_nj<S, 8>();
    case 16: return load_parses_nj<S, 16>();
    default: return load_parses_nj<S, 32>();
  }
}

}  // namespace glz
