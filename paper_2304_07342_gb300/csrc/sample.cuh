// sample.cuh -- do a launch's symbols seldom repeat?  A sample of its data,
// taken by a small kernel before it, and the line between the parse by masks
// and the one by chains.
//
// kSampleWarps warps each take a chunk at random and count, for eight
// positions, the positions inside the window that carry the same key (the
// candidates that a hash chain would visit), and the bits in which the symbols
// around them differ.  The clearing of a single buffer's scratch rides along,
// so the sample costs no launch of its own there.  Chains and masks are then
// both launched, as dependent launches, and the one not chosen ends at once.
//
// Bound by latency (one round trip for a piece of each chunk).  Sample and
// second launch cost 2 to 3 us: uniform 4-byte values, all literals, 8 MiB 27.7
// us without, 29.5 with, 256 MiB of a float field 195.0 and 198.4.  What the
// choice gives is below (seldom_repeats).
#pragma once

#include <cstdint>

#include "glz_common.h"
#include "glz_device.cuh"
#include "mask_parse.cuh"

namespace glz {

constexpr uint32_t kSamplePositions = 8;  // per warp, four symbols apart
constexpr uint32_t kSampleCap = 48;       // candidates counted per position: a chain's walk ends
                                          // there and the rest costs no more
constexpr uint32_t kSampleBlock = 256;

// Symbols of a piece: the window before the positions, the positions and their
// keys.
__host__ __device__ constexpr uint32_t sample_symbols(int nw) { return 32 * nw + 4 * kSamplePositions + 32; }

// By sampling warp w: the chunk (in 2^32ths of all) and the place in it.
__device__ __forceinline__ uint32_t sample_hash(uint32_t w) { return (2 * w + 1) * 0x9E3779B1u; }
__device__ __forceinline__ uint32_t sample_place(uint32_t h) { return (h ^ (h >> 15)) * 0x85EBCA77u; }

// The number of positions inside the window of position p (>= 32 * NW) that
// carry its key, its first g symbols.
template <int S, int NW>
__device__ __forceinline__ uint32_t candidates(const typename SymType<S>::T *sym, uint32_t p,
                                               uint32_t g, uint32_t W, uint32_t lane) {
  using Sym = typename SymType<S>::T;
  uint32_t eq = 0;  // bit j: offset lane + 1 + 32 j
#pragma unroll
  for (int j = 0; j < NW; ++j) eq |= lane + 1 + 32 * j <= W ? 1u << j : 0u;
  const Sym *src = sym + p - 1 - lane;
#pragma unroll 1
  for (uint32_t x = 0; x < g && __any_sync(kFull, eq != 0); ++x) {
    const Sym c = sym[p + x];
    uint32_t e = 0;
#pragma unroll
    for (int j = 0; j < NW; ++j) e |= src[static_cast<int>(x) - 32 * j] == c ? 1u << j : 0u;
    eq &= e;
  }
  return __reduce_add_sync(kFull, __popc(eq));
}

// A word of the sample: candidates | varying bits << 16 | 1 << 24 (0: the chunk
// taken was shorter than a piece).
template <int S, int NW>
__device__ __forceinline__ uint32_t sample_piece(const BufDesc &B, uint32_t c, uint32_t r,
                                                 uint8_t *piece, uint32_t lane) {
  using Sym = typename SymType<S>::T;
  constexpr uint32_t kSyms = sample_symbols(NW), kBytes = kSyms * S;
  static_assert(kBytes % 16 == 0, "whole vectors");
  const uint64_t chunk_at = static_cast<uint64_t>(c) * B.C;
  const uint32_t bytes = (c + 1 < B.nc) ? B.C : static_cast<uint32_t>(B.n - chunk_at);
  const uint32_t k = bytes / S;
  if (k < kSyms) return 0;
  const uint32_t at = __umulhi(r, k - kSyms + 1) & ~15u;  // first symbol
  const uint8_t *src = B.in + chunk_at + at * S;
  if (B.in_aligned) {
#pragma unroll
    for (uint32_t i = lane; i < kBytes / 16; i += 32)
      reinterpret_cast<uint4 *>(piece)[i] = reinterpret_cast<const uint4 *>(src)[i];
  } else {
#pragma unroll 8
    for (uint32_t i = lane; i < kBytes; i += 32) piece[i] = src[i];
  }
  __syncwarp();
  const uint32_t g = min(B.m, 8u / S);
  uint32_t hits = 0;
#pragma unroll 1
  for (uint32_t i = 0; i < kSamplePositions; ++i)
    hits += min(candidates<S, NW>(reinterpret_cast<const Sym *>(piece), 32 * NW + 4 * i, g, B.W,
                                  lane),
                kSampleCap);
  return hits | (__popc(varying_bits<S>(piece, kSyms, lane)) << 16) | (1u << 24);
}

// Do the symbols of a launch seldom repeat, so that chains (of window class NW)
// cost less than masks of NW words?  A mask's cost grows with its words and with the bits in
// which symbols differ, a chain's with the candidates.  The lines lie between
// these, candidates per position (32 MiB in us, chains against masks):
//   S = 4, W = 256: text 0.53, 31 bits: 169, 423; codes 7.0, 5 bits: 756, 222
//   S = 4, W = 512: text 1.1: 339, 743; padded floats 31, 29 bits: 1657, 996
//   S = 2, W = 128: text 0.44, 15 bits: 297, 436; codes 0.83, 5 bits: 434, 297
//   S = 2, W = 512: text 1.8, 15 bits: 854, 1008; codes 3.1: 1791, 637
//   S = 1, W = 128: few repeats 0.06: 370, 580; floats 0.66: 798, 650
//   S = 1, W = 512: few repeats 0.06: 833, 1226; floats 0.66: 2095, 1406
// Both costs are about linear in these, so the means decide as the chunks one
// by one would, and all warps take one parse (an SM whose warps ran both took
// longer than with either: text, S = 2, W = 128: 478 us).  Both parses give
// the same bytes.
template <int S, int NW>
__device__ __forceinline__ bool seldom_repeats(const uint32_t *votes) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t hits = 0, bits = 0, n = 0;
#pragma unroll
  for (uint32_t i = 0; i < kSampleWarps; i += 32) {
    const uint32_t v = votes[i + lane];
    hits += v & 0xFFFFu;
    bits += (v >> 16) & 0xFFu;
    n += v >> 24;
  }
  hits = __reduce_add_sync(kFull, hits);
  bits = __reduce_add_sync(kFull, bits);
  n = __reduce_add_sync(kFull, n);
  // in 16ths of a candidate per position, times the pieces
  const uint32_t line = S == 4   ? 6 * n + bits
                        : S == 1 ? (NW <= 2 ? 4u : NW <= 8 ? 5u : 8u) * n
                        : NW <= 4  ? 3 * bits / 4
                        : NW <= 8  ? 2 * n + 5 * bits / 4
                                   : 4 * n + 2 * bits;
  return n != 0 && 16 / kSamplePositions * hits <= line;
}

}  // namespace glz
