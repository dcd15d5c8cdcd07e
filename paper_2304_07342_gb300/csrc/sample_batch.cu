// sample_batch.cu -- the sample of every class of a batch, in one launch.
#include "compress_impl.cuh"

namespace glz {

// Blocks 8 i .. 8 i + 7 sample class i (sample.cuh).
__global__ void __launch_bounds__(kSampleBlock)
    sample_batch_kernel(const __grid_constant__ SampleList L) {
  __shared__ __align__(16) uint8_t pieces[8][sample_symbols(16) * 4];
  const SampleClass &E = L.e[blockIdx.x / 8];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t w = 8 * (blockIdx.x % 8) + warp;
  const uint32_t h = sample_hash(w);
  CompressArgs A{};
  A.item_base = E.item_base;
  A.n_items = E.n_items;
  const uint64_t g = (E.total_chunks * h) >> 32;  // (fewer than 2^32 chunks)
  const BufDesc B = E.items[find_item(A, g, lane)];
  const uint32_t c = static_cast<uint32_t>(g - B.gbase), r = sample_place(h);
  uint8_t *piece = pieces[warp];
  uint32_t v = 0;
  switch (32 * E.S + E.nj) {
    case 32 + 4: v = sample_piece<1, 4>(B, c, r, piece, lane); break;
    case 32 + 8: v = sample_piece<1, 8>(B, c, r, piece, lane); break;
    case 32 + 16: v = sample_piece<1, 16>(B, c, r, piece, lane); break;
    case 64 + 4: v = sample_piece<2, 4>(B, c, r, piece, lane); break;
    case 64 + 8: v = sample_piece<2, 8>(B, c, r, piece, lane); break;
    case 64 + 16: v = sample_piece<2, 16>(B, c, r, piece, lane); break;
    case 128 + 4: v = sample_piece<4, 4>(B, c, r, piece, lane); break;
    case 128 + 8: v = sample_piece<4, 8>(B, c, r, piece, lane); break;
    case 128 + 16: v = sample_piece<4, 16>(B, c, r, piece, lane); break;
    default: break;
  }
  if (lane == 0) E.votes[w] = v;
}

cudaError_t launch_sample_batch(const SampleList &L, cudaStream_t stream) {
  sample_batch_kernel<<<8 * L.n, kSampleBlock, 0, stream>>>(L);
  return cudaGetLastError();
}

}  // namespace glz
