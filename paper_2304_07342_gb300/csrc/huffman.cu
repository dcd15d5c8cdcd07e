// huffman.cu -- the Huffman stage that follows LZSS in the paper's use case
// (section 4.5: cuSZ Huffman-codes what gpuLZ produces).  Byte alphabet,
// an optimal prefix code limited to kHufMaxLen bits, canonical codes, and
// the "GHF1" stream described in include/lz.h.
//
//   huff_hist_kernel    256-bin histogram of the input; clears the block table
//   huff_book_kernel    one block: package-merge with every list built in
//                       parallel (each item finds its place in the merged
//                       list by a binary search in the other list), the
//                       selection walked level by level, canonical codes;
//                       writes the header and the code book
//   huff_encode_kernel  one thread block per 32 KiB block at a time: each
//                       warp packs four 1 KiB sub-blocks into shared memory,
//                       the block's place comes from a decoupled look-back
//                       over the block table itself, the words go out shifted
//   huff_decode_kernel  one warp per block, one lane per sub-block: a
//                       4096-entry table in shared memory maps the next 12
//                       bits to up to three symbols and their code bits
#include <cuda_runtime.h>

#include <cstdint>

#include "glz_common.h"
#include "glz_device.cuh"
#include "launch_cache.cuh"

namespace glz {

namespace {

constexpr uint32_t kHufMaxLen = 12;
constexpr uint32_t kHufBlock = 32768;
constexpr uint32_t kHufSub = 1024;
constexpr uint32_t kHufSubs = kHufBlock / kHufSub;  // 32: one per lane
constexpr uint32_t kHufLengthsAt = 16;
constexpr uint32_t kHufTableAt = 272;
constexpr uint32_t kHufInvalid = 0xFFFFu;

__host__ __device__ __forceinline__ uint64_t huf_subs_at(uint64_t nb) {
  return kHufTableAt + 8ull * nb;
}
__host__ __device__ __forceinline__ uint64_t huf_bits_at(uint64_t nb) {
  return kHufTableAt + 8ull * nb + 4ull * kHufSubs * nb;
}

__device__ __forceinline__ uint64_t ld_u64_le(const uint8_t *p) {
  uint64_t v = 0;
  for (int i = 0; i < 8; ++i) v |= static_cast<uint64_t>(p[i]) << (8 * i);
  return v;
}

// ---- histogram -----------------------------------------------------------------

// Bound by shared-memory atomics.  Each lane counts in a copy of its own
// (bin-major, so lane l always hits bank l): the high bytes of quantization
// codes take two or three values, and with one copy per warp most lanes of an
// atomic hit the same word, one after the other.
constexpr uint32_t kHistThreads = 512;

__global__ void __launch_bounds__(kHistThreads) huff_hist_kernel(const uint8_t *in, uint64_t n,
                                                                unsigned long long *hist,
                                                                unsigned long long *table,
                                                                uint64_t nb) {
  __shared__ uint32_t h[256 * 32];
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t tid = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * blockDim.x;
  for (uint64_t b = tid; b < nb; b += stride) table[b] = 0;  // look-back words, see the encoder
  for (uint32_t i = threadIdx.x; i < 256 * 32; i += blockDim.x) h[i] = 0;
  __syncthreads();
  uint32_t *mine = h + lane;
  auto count4 = [&](uint32_t v) {
    atomicAdd(mine + 32 * (v & 0xFF), 1u);
    atomicAdd(mine + 32 * ((v >> 8) & 0xFF), 1u);
    atomicAdd(mine + 32 * ((v >> 16) & 0xFF), 1u);
    atomicAdd(mine + 32 * (v >> 24), 1u);
  };
  const uint64_t mis = (16u - (reinterpret_cast<uintptr_t>(in) & 15u)) & 15u;
  const uint64_t head = n < mis ? n : mis;
  const uint64_t quads = (n - head) / 16;
  const uint4 *q = reinterpret_cast<const uint4 *>(in + head);
  for (uint64_t i = tid; i < quads; i += stride) {
    const uint4 v = q[i];
    count4(v.x);
    count4(v.y);
    count4(v.z);
    count4(v.w);
  }
  if (tid < head) atomicAdd(mine + 32 * in[tid], 1u);
  const uint64_t done = head + 16 * quads;
  if (tid < n - done) atomicAdd(mine + 32 * in[done + tid], 1u);
  __syncthreads();
  for (uint32_t s = threadIdx.x >> 5; s < 256; s += blockDim.x >> 5) {
    const uint32_t t = __reduce_add_sync(kFull, h[32 * s + lane]);
    if (lane == 0 && t) atomicAdd(&hist[s], static_cast<unsigned long long>(t));
  }
}

// ---- code book -------------------------------------------------------------------

// Canonical codes of lengths len[256] (one thread per symbol, blockDim >= 256,
// a multiple of 32): symbols in order of (length, value) take consecutive
// values, shifted left when the length grows.  A symbol's rank in its length
// is the number of lower lanes of its warp with that length plus those of the
// warps before.  first[] and cnt[] are shared scratch.
__device__ void canonical_codes(const uint32_t *len, uint32_t *first, uint32_t *cnt,
                                uint32_t *code_out) {
  __shared__ uint32_t warp_cnt[8][16];
  const uint32_t t = threadIdx.x, lane = t & 31, warp = t >> 5;
  uint32_t l = 0, rank = 0;
  if (warp < 8) {
    if (lane < 16) warp_cnt[warp][lane] = 0;
    __syncwarp();
    l = len[t];
    const uint32_t peers = __match_any_sync(kFull, l);
    rank = __popc(peers & lanemask_lt(lane));
    if (rank == 0) warp_cnt[warp][l] = __popc(peers);
  }
  __syncthreads();
  if (t >= 1 && t <= kHufMaxLen) {
    uint32_t c = 0;
    for (uint32_t w = 0; w < 8; ++w) c += warp_cnt[w][t];
    cnt[t] = c;
  }
  __syncthreads();
  if (t == 0) {
    uint32_t next = 0;
    for (uint32_t x = 1; x <= kHufMaxLen; ++x) {
      first[x] = next;
      next = (next + cnt[x]) << 1;
    }
  }
  __syncthreads();
  if (warp < 8) {
    for (uint32_t w = 0; w < warp; ++w) rank += warp_cnt[w][l];
    code_out[t] = l ? first[l] + rank : 0;
  }
  __syncthreads();
}

// Package-merge over the present symbols (at most 256, so every list has at
// most 511 items): leaves sorted by (count, value); list d (d = 0 the
// shallowest) merges the leaves with the packages of consecutive pairs of
// list d + 1, by weight, a leaf before a package of equal weight; the first
// 2n - 2 items of list 0 are selected and a selected package selects its two
// children.  A symbol's length is the number of lists where it is selected.
__global__ void __launch_bounds__(512) huff_book_kernel(const unsigned long long *hist,
                                                       uint64_t n_bytes, uint8_t *out,
                                                       uint32_t *book,
                                                       unsigned long long *out_bytes) {
  __shared__ unsigned long long hw[256], leafw[256];
  __shared__ unsigned long long w[2][512];
  __shared__ uint16_t ref[kHufMaxLen][512];  // 0x8000 | symbol, or package index
  __shared__ uint8_t sel[kHufMaxLen][512];
  __shared__ uint32_t leafsym[256], len[256], code[256], first[kHufMaxLen + 1],
      cnt[kHufMaxLen + 1], count[kHufMaxLen];
  const uint32_t t = threadIdx.x;
  if (t < 256) {
    hw[t] = hist[t];
    len[t] = 0;
  }
  for (uint32_t i = t; i < kHufMaxLen * 512; i += blockDim.x) (&sel[0][0])[i] = 0;
  __syncthreads();
  const uint32_t n = __syncthreads_count(t < 256 && hw[t] > 0);
  if (n == 1) {
    if (t < 256 && hw[t]) len[t] = 1;
  } else if (n > 1) {
    // a leaf's place: the present symbols before it by (count, value), each
    // lane of a warp comparing eight
    for (uint32_t x = t >> 5; x < 256; x += blockDim.x >> 5) {
      const unsigned long long mine = hw[x];
      if (!mine) continue;
      uint32_t r = 0;
      for (uint32_t s = t & 31; s < 256; s += 32)
        r += hw[s] && (hw[s] < mine || (hw[s] == mine && s < x));
      r = __reduce_add_sync(kFull, r);
      if ((t & 31) == 0) {
        leafsym[r] = x;
        leafw[r] = mine;
      }
    }
    __syncthreads();
    const uint32_t deep = kHufMaxLen - 1;
    if (t < n) {
      w[deep & 1][t] = leafw[t];
      ref[deep][t] = static_cast<uint16_t>(0x8000u | leafsym[t]);
    }
    if (t == 0) count[deep] = n;
    __syncthreads();
    for (int d = static_cast<int>(deep) - 1; d >= 0; --d) {
      const unsigned long long *below = w[(d + 1) & 1];
      unsigned long long *cur = w[d & 1];
      const uint32_t np = count[d + 1] / 2;
      if (t < n) {
        // leaf t: after every package strictly lighter
        const unsigned long long x = leafw[t];
        uint32_t lo = 0, hi = np;
        while (lo < hi) {
          const uint32_t mid = (lo + hi) / 2;
          if (below[2 * mid] + below[2 * mid + 1] < x) lo = mid + 1;
          else hi = mid;
        }
        cur[t + lo] = x;
        ref[d][t + lo] = static_cast<uint16_t>(0x8000u | leafsym[t]);
      } else if (t < n + np) {
        // package j: after every leaf of equal or smaller weight
        const uint32_t j = t - n;
        const unsigned long long x = below[2 * j] + below[2 * j + 1];
        uint32_t lo = 0, hi = n;
        while (lo < hi) {
          const uint32_t mid = (lo + hi) / 2;
          if (leafw[mid] <= x) lo = mid + 1;
          else hi = mid;
        }
        cur[j + lo] = x;
        ref[d][j + lo] = static_cast<uint16_t>(j);
      }
      if (t == 0) count[d] = n + np;
      __syncthreads();
    }
    for (uint32_t i = t; i < count[0] && i < 2 * n - 2; i += blockDim.x) sel[0][i] = 1;
    for (uint32_t d = 0; d < kHufMaxLen; ++d) {
      __syncthreads();
      for (uint32_t i = t; i < count[d]; i += blockDim.x) {
        if (!sel[d][i]) continue;
        const uint32_t r = ref[d][i];
        if (r & 0x8000u) {
          atomicAdd(&len[r & 0xFFu], 1u);
        } else if (d + 1 < kHufMaxLen) {
          sel[d + 1][2 * r] = 1;
          sel[d + 1][2 * r + 1] = 1;
        }
      }
    }
  }
  __syncthreads();
  canonical_codes(len, first, cnt, code);
  if (t < 256) {
    book[t] = code[t] | (len[t] << 24);
    out[kHufLengthsAt + t] = static_cast<uint8_t>(len[t]);
  }
  if (n_bytes == 0 && t == 0) *out_bytes = huf_bits_at(0);  // else the encoder's
  if (t < 16) {
    uint32_t b = 0;
    if (t < 4) b = "GHF1"[t];
    else if (t < 8) b = (kHufBlock >> (8 * (t - 4))) & 0xFF;
    else b = static_cast<uint32_t>(n_bytes >> (8 * (t - 8))) & 0xFF;
    out[t] = static_cast<uint8_t>(b);
  }
}

// ---- encode ------------------------------------------------------------------------

// This lane's sub-block of block b: [lo, hi) of the input (empty past n).
__device__ __forceinline__ void sub_range(uint64_t b, uint32_t lane, uint64_t n, uint64_t &lo,
                                          uint64_t &hi) {
  lo = b * kHufBlock + static_cast<uint64_t>(lane) * kHufSub;
  hi = lo + kHufSub < n ? lo + kHufSub : n;
  if (lo > n) lo = n;
}

// The 32 bytes of sub-block s of block b that lane `lane` handles, as eight
// little-endian words (zero past hi); 16-byte loads when `in` is aligned.
__device__ __forceinline__ void lane_bytes(const uint8_t *in, uint64_t at, uint64_t hi,
                                           bool in16, uint32_t (&w)[8]) {
  if (in16 && at + 32 <= hi) {
    const uint4 a = *reinterpret_cast<const uint4 *>(in + at);
    const uint4 c = *reinterpret_cast<const uint4 *>(in + at + 16);
    w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
    w[4] = c.x; w[5] = c.y; w[6] = c.z; w[7] = c.w;
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      uint32_t v = 0;
      for (int k = 0; k < 4; ++k) {
        const uint64_t idx = at + 4 * q + k;
        if (idx < hi) v |= static_cast<uint32_t>(in[idx]) << (8 * k);
      }
      w[q] = v;
    }
  }
}

// Encoding: one thread block takes a 32 KiB block at a time (in order, from a
// work counter); warp w codes sub-blocks 4w .. 4w + 3.  Each lane looks its 32
// consecutive bytes up once and joins the codes in pairs (at most 24 bits and
// their length in one word), a warp scan of the lanes' bit counts places them,
// and each lane packs its pairs into the words of the warp's own bit string in
// shared memory.  A full sub-block gives every lane at least 32 bits, so a
// word is shared by two lanes at most and the later one joins the earlier
// one's last bits (a shuffle).  Once the block's size is known it is published
// and the block's place found by a decoupled look-back; the warps' strings
// then go out as whole words, shifted to their bit offsets.
//
// The look-back words are the block table itself: 0 until published, size | 1
// (sizes are multiples of 4), at the end the end offset, which is what the
// stream holds.  So the sizes pass and the scan launch over the table that
// this replaces are gone, and with them one reading of the input.
constexpr uint32_t kEncWarps = kHufBlock / 4096;                        // 8
constexpr uint32_t kEncRegion = (4 * kHufSub * kHufMaxLen) / 32 + 4;    // words of a warp's string
constexpr uint32_t kEncSmem = kEncWarps * kEncRegion * 4;

// The pair of codes (a, b), each code | length << 24.
__device__ __forceinline__ uint32_t join_codes(uint32_t a, uint32_t b) {
  return ((a & 0xFFFFFFu) << (b >> 24)) + (a & 0xFF000000u) + b;
}

// Block b's end offset, from the published sizes and end offsets before it.
// False when a predecessor did not publish within `limit` polls.
__device__ __forceinline__ bool huf_lookback(const unsigned long long *table, uint64_t b,
                                             uint32_t lane, uint32_t limit, uint64_t &excl) {
  excl = 0;
  int64_t base = static_cast<int64_t>(b) - 1;
  uint32_t spins = 0;
  while (base >= 0) {
    const int64_t idx = base - static_cast<int64_t>(lane);
    const unsigned long long v = idx >= 0 ? ld_relaxed_u64(&table[idx]) : 4ull;  // any end
    const uint32_t ends = __ballot_sync(kFull, v != 0 && !(v & 1));
    const uint32_t empty = __ballot_sync(kFull, v == 0);
    const uint32_t limit_lane = ends ? __ffs(ends) - 1 : 31u;
    const uint32_t need = limit_lane == 31 ? kFull : ((2u << limit_lane) - 1u);
    if (empty & need) {
      if (++spins > limit) return false;
      __nanosleep(64);
      continue;
    }
    excl += warp_sum_u64(lane <= limit_lane && idx >= 0 ? (v & ~1ull) : 0ull);
    if (ends) return true;
    base -= 32;
  }
  return true;
}

__global__ void __launch_bounds__(256) huff_encode_kernel(const uint8_t *in, uint64_t n,
                                                         uint8_t *out, uint64_t out_cap,
                                                         const uint32_t *book, uint32_t *ticket,
                                                         unsigned long long *out_bytes,
                                                         uint32_t *err) {
  extern __shared__ __align__(16) uint32_t regions[];
  __shared__ uint32_t cl[256];  // code | length << 24
  __shared__ uint32_t sub_total[kHufSubs];
  __shared__ unsigned long long s_block, s_start;
  __shared__ uint32_t s_ok;
  for (uint32_t s = threadIdx.x; s < 256; s += blockDim.x) cl[s] = book[s];
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t *wb = regions + warp * kEncRegion;
  const uint64_t nb = (n + kHufBlock - 1) / kHufBlock;
  const uint64_t bits_at = huf_bits_at(nb);
  uint32_t *subs = reinterpret_cast<uint32_t *>(out + huf_subs_at(nb));
  unsigned long long *table = reinterpret_cast<unsigned long long *>(out + kHufTableAt);
  const bool in16 = (reinterpret_cast<uintptr_t>(in) & 15u) == 0;
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) s_block = atomicAdd(ticket, 1u);
    __syncthreads();
    const uint64_t b = s_block;
    if (b >= nb) break;
    uint32_t at = 0;     // bits of this warp's string so far
    uint32_t carry = 0;  // bits of its last, partial word (left-aligned)
    for (uint32_t i = 0; i < 4; ++i) {
      const uint32_t sb = 4 * warp + i;
      uint64_t lo, hi;
      sub_range(b, sb, n, lo, hi);
      uint32_t sub_bits = 0;
      if (hi - lo == kHufSub) {
        uint32_t w[8], pr[16], bits = 0;
        lane_bytes(in, lo + 32ull * lane, hi, in16, w);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          pr[2 * q] = join_codes(cl[w[q] & 0xFF], cl[(w[q] >> 8) & 0xFF]);
          pr[2 * q + 1] = join_codes(cl[(w[q] >> 16) & 0xFF], cl[w[q] >> 24]);
        }
#pragma unroll
        for (int q = 0; q < 16; ++q) bits += pr[q] >> 24;
        uint32_t incl = bits;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(kFull, incl, o);
          if (lane >= static_cast<uint32_t>(o)) incl += y;
        }
        sub_bits = __shfl_sync(kFull, incl, 31);
        const uint32_t p = at + incl - bits;
        uint32_t fill = p % 32, wi = p / 32;
        const uint32_t shared_bits = fill, wi0 = wi;
        uint64_t acc = 0;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const uint32_t l = pr[q] >> 24;
          acc = (acc << l) | (pr[q] & 0xFFFFFFu);
          fill += l;
          if (fill >= 32) {
            fill -= 32;
            if (GLZ_OK(wi < kEncRegion)) wb[wi] = static_cast<uint32_t>(acc >> fill);
            ++wi;
          }
        }
        // the last, partial word goes to the lane after (lane 31's is carried)
        const uint32_t part = fill ? static_cast<uint32_t>(acc << (32 - fill)) : 0u;
        uint32_t before = __shfl_up_sync(kFull, part, 1);
        if (lane == 0) before = carry;
        // (the first word also holds the low bits of a zero accumulator above
        // this lane's, so the joined bits are ORed into zeros)
        if (shared_bits) wb[wi0] |= before;
        carry = __shfl_sync(kFull, part, 31);
      } else if (hi > lo) {
        // the input's last, short sub-block: codes ORed in one by one
        const uint32_t room = ((at % 32) + kHufSub * kHufMaxLen + 31) / 32 + 1;
        __syncwarp();
        for (uint32_t j = lane; j < room && at / 32 + j < kEncRegion; j += 32)
          wb[at / 32 + j] = j == 0 ? carry : 0u;
        __syncwarp();
        const uint64_t from = lo + 32ull * lane;
        const uint32_t valid = from >= hi ? 0u : static_cast<uint32_t>(min(hi - from, uint64_t{32}));
        uint32_t bits = 0;
        for (uint32_t j = 0; j < valid; ++j) bits += cl[in[from + j]] >> 24;
        uint32_t incl = bits;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t y = __shfl_up_sync(kFull, incl, o);
          if (lane >= static_cast<uint32_t>(o)) incl += y;
        }
        sub_bits = __shfl_sync(kFull, incl, 31);
        uint32_t p = at + incl - bits;
        for (uint32_t j = 0; j < valid; ++j) {
          const uint32_t e = cl[in[from + j]], l = e >> 24, c = e & 0xFFFFFFu;
          const uint32_t end = p % 32 + l;  // l >= 1
          if (GLZ_OK(p / 32 + (end > 32) < kEncRegion)) {
            atomicOr(&wb[p / 32], end <= 32 ? c << (32 - end) : c >> (end - 32));
            if (end > 32) atomicOr(&wb[p / 32 + 1], c << (64 - end));
          }
          p += l;
        }
        __syncwarp();
        carry = (at + sub_bits) % 32 ? wb[(at + sub_bits) / 32] : 0u;
      }
      at += sub_bits;
      if (lane == 0) sub_total[sb] = sub_bits;
      __syncwarp();
    }
    if (lane == 0 && at % 32) wb[at / 32] = carry;
    __syncthreads();
    // sub-block offsets of the block (every warp scans them)
    const uint32_t mine = sub_total[lane];
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, incl, o);
      if (lane >= static_cast<uint32_t>(o)) incl += y;
    }
    const uint32_t total = __shfl_sync(kFull, incl, 31);
    const uint64_t size = static_cast<uint64_t>((total + 31) / 32) * 4;
    if (warp == 0) {
      subs[b * kHufSubs + lane] = incl - mine;
      if (b && lane == 0) st_relaxed_u64(&table[b], size | 1ull);
      uint64_t start = 0;
      const bool ok = huf_lookback(table, b, lane, kSpinLimit, start);
      if (lane == 0) {
        st_relaxed_u64(&table[b], start + size);
        if (!ok) atomicOr(err, kErrTimeout);
        const uint64_t end = bits_at + start + size;
        if (b + 1 == nb) {
          *out_bytes = end;
          if (end > out_cap) atomicOr(err, kErrSmall);
        }
        s_start = start;
        s_ok = ok && end <= out_cap;
      }
    }
    __syncthreads();
    if (!s_ok) continue;  // past the capacity: reported by the last block
    // this warp's string, from bit `bs` of the block; a word belongs to the
    // warp whose bits it starts with
    uint32_t *w32 = reinterpret_cast<uint32_t *>(out + bits_at + s_start);
    const uint32_t bs = __shfl_sync(kFull, incl - mine, 4 * warp), sh = bs % 32;
    const uint32_t touched = (sh + at + 31) / 32, held = (at + 31) / 32;
    const uint32_t over = (sh + at) % 32;  // bits of the last word that are this warp's
    uint32_t next0 = 0;                    // the next warp's first bits
    if (over && warp + 1 < kEncWarps && bs + at < total) next0 = wb[kEncRegion] >> over;
    if (at) {
      for (uint32_t j = lane + (sh ? 1u : 0u); j < touched; j += 32) {
        uint32_t v = j < held ? wb[j] : 0u;
        if (sh) v = (v >> sh) | (wb[j - 1] << (32 - sh));
        if (j + 1 == touched) v |= next0;
        if (GLZ_OK((bs / 32 + j) * 4ull < size)) w32[bs / 32 + j] = v;
      }
    }
  }
}

// ---- decode ------------------------------------------------------------------------

struct HufHeader {
  uint64_t n, nb, bits_at;
  bool ok;
};

__device__ __forceinline__ HufHeader huf_header(const uint8_t *in, uint64_t in_bytes) {
  HufHeader h{};
  h.ok = in_bytes >= kHufTableAt && in[0] == 'G' && in[1] == 'H' && in[2] == 'F' &&
         in[3] == '1' && in[4] == (kHufBlock & 0xFF) && in[5] == ((kHufBlock >> 8) & 0xFF) &&
         in[6] == 0 && in[7] == 0;
  if (!h.ok) return h;
  h.n = ld_u64_le(in + 8);
  h.nb = (h.n + kHufBlock - 1) / kHufBlock;
  h.bits_at = huf_bits_at(h.nb);
  h.ok = h.nb < (1ull << 40) && h.bits_at <= in_bytes;
  return h;
}

// Bound by instruction issue and, before, by each lane's own loads from its
// sub-block's words.  One lookup gives every symbol whose code ends inside
// the 12 bits (up to three); words come in and bytes go out 16 and 32 at a
// time through small rings in shared memory.
constexpr uint32_t kDecTables = 6u << kHufMaxLen;    // bytes of both tables
constexpr uint32_t kDecRing = (8 + 16) * 32;         // ring words of a warp
constexpr uint32_t kDecSmem = kDecTables + 8 * kDecRing * 4;

__global__ void __launch_bounds__(256) huff_decode_kernel(const uint8_t *in, uint64_t in_bytes,
                                                         uint8_t *out, uint64_t out_cap,
                                                         unsigned long long *out_bytes,
                                                         uint32_t *err) {
  extern __shared__ __align__(16) uint32_t dyn[];
  // next 12 bits -> up to three symbols, first lowest | their code bits << 24
  // | their number << 28 (an invalid code: length 15, one symbol)
  uint32_t *multi = dyn;
  uint16_t *dec = reinterpret_cast<uint16_t *>(dyn + (1u << kHufMaxLen));  // symbol | length << 8
  __shared__ uint32_t len[256], code[256], first[kHufMaxLen + 1], cnt[kHufMaxLen + 1];
  __shared__ uint32_t bad_code;
  const uint32_t t = threadIdx.x;
  const HufHeader h = huf_header(in, in_bytes);
  if (!h.ok) {
    if (blockIdx.x == 0 && t == 0) atomicOr(err, kErrCorrupt);
    return;
  }
  if (h.n > out_cap) {
    if (blockIdx.x == 0 && t == 0) atomicOr(err, kErrSmall);
    return;
  }
  if (blockIdx.x == 0 && t == 0) *out_bytes = h.n;
  if (t == 0) bad_code = 0;
  if (t < 256) len[t] = in[kHufLengthsAt + t];
  __syncthreads();
  // the lengths must form a complete code (or one symbol of length 1)
  uint32_t present = 0, kraft = 0;
  if (t < 256 && len[t]) {
    if (len[t] > kHufMaxLen) atomicOr(&bad_code, 1u);
    else kraft = 1u << (kHufMaxLen - len[t]);
    present = 1;
  }
  const uint32_t n_present = __syncthreads_count(present);
  __shared__ uint32_t kraft_sum;
  if (t == 0) kraft_sum = 0;
  __syncthreads();
  if (kraft) atomicAdd(&kraft_sum, kraft);
  __syncthreads();
  const bool complete = n_present == 1 ? kraft_sum == (1u << (kHufMaxLen - 1))
                                       : kraft_sum == (1u << kHufMaxLen);
  if (bad_code || (h.n > 0 && !complete)) {
    if (blockIdx.x == 0 && t == 0) atomicOr(err, kErrCorrupt);
    return;
  }
  canonical_codes(len, first, cnt, code);
  // symbols in canonical order: those of length l hold places off[l] ..
  // off[l] + cnt[l] - 1, by value
  __shared__ uint32_t off[kHufMaxLen + 2];
  __shared__ uint8_t order[256];
  if (t == 0) {
    off[1] = 0;
    for (uint32_t l = 1; l <= kHufMaxLen; ++l) off[l + 1] = off[l] + cnt[l];
  }
  __syncthreads();
  if (t < 256 && len[t]) order[off[len[t]] + code[t] - first[len[t]]] = static_cast<uint8_t>(t);
  __syncthreads();
  // entry e (the next 12 bits) belongs to the first length l whose codes,
  // left-aligned, end above e
  for (uint32_t e = t; e < (1u << kHufMaxLen); e += blockDim.x) {
    uint32_t l = 1;
#pragma unroll
    for (uint32_t x = 1; x <= kHufMaxLen; ++x)
      l += e >= ((first[x] + cnt[x]) << (kHufMaxLen - x)) ? 1u : 0u;
    uint32_t v = kHufInvalid;
    if (l <= kHufMaxLen) v = order[off[l] + (e >> (kHufMaxLen - l)) - first[l]] | (l << 8);
    dec[e] = static_cast<uint16_t>(v);
  }
  __syncthreads();
  // (no two codes in 12 bits, as for bytes that all occur about as often: a
  // lookup gives one symbol, and the table of several is not made)
  uint32_t shortest = 1;
  while (shortest < kHufMaxLen && cnt[shortest] == 0) ++shortest;
  const bool one_each = 2 * shortest > kHufMaxLen;
  for (uint32_t e = t; e < (1u << kHufMaxLen) && !one_each; e += blockDim.x) {
    const uint32_t a = dec[e];
    uint32_t v = (15u << 24) | (1u << 28);
    if (a != kHufInvalid) {
      uint32_t bits = a >> 8, num = 1;
      v = a & 0xFFu;
#pragma unroll
      for (uint32_t x = 1; x < 3; ++x) {
        // the code after: known when it ends inside the 12 bits
        const uint32_t c = dec[(e << bits) & ((1u << kHufMaxLen) - 1u)];
        const uint32_t l = c >> 8;
        if (num == x && c != kHufInvalid && bits + l <= kHufMaxLen) {
          v |= (c & 0xFFu) << (8 * x);
          bits += l;
          ++num;
        }
      }
      v |= (bits << 24) | (num << 28);
    }
    multi[e] = v;
  }
  __syncthreads();

  const uint32_t lane = t & 31;
  const uint64_t gw = (static_cast<uint64_t>(blockIdx.x) * blockDim.x + t) >> 5;
  const uint64_t nw = (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5;
  const uint32_t *subs = reinterpret_cast<const uint32_t *>(in + huf_subs_at(h.nb));
  const uint8_t *table = in + kHufTableAt;
  const bool out16 = (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
  uint32_t *ring_in = dyn + kDecTables / 4 + (t >> 5) * kDecRing + lane;  // 8 words per lane
  uint32_t *ring_out = ring_in + 8 * 32;                                  // 16 words per lane
  for (uint64_t b = gw; b < h.nb; b += nw) {
    const uint64_t start = b ? ld_u64_le(table + 8 * (b - 1)) : 0ull;
    const uint64_t end = ld_u64_le(table + 8 * b);
    const uint64_t bytes = end - start;
    bool bad = !huf_span_ok(start, end, h.bits_at, in_bytes);
    const uint32_t nbits = static_cast<uint32_t>(bytes * 8);
    uint64_t lo, hi;
    sub_range(b, lane, h.n, lo, hi);
    const uint32_t o = bad ? 0 : subs[b * kHufSubs + lane];
    const uint32_t o_down = __shfl_down_sync(kFull, o, 1);  // every lane takes part
    const uint32_t o_next = lane < 31 ? o_down : 0u;
    bad = bad || o > nbits || (lane == 0 && o != 0);
    if (__any_sync(kFull, bad)) {
      if (lane == 0) atomicOr(err, kErrCorrupt);
      continue;
    }
    const uint32_t nwords = static_cast<uint32_t>(bytes / 4);
    // This lane's words come 16 bytes at a time into a ring of eight words in
    // shared memory (word-major: lane l uses bank l), the next 16 held in
    // registers.  `wi` counts the words taken from the ring, `have` those put.
    const uint64_t first_at = h.bits_at + start + 4ull * (o / 32);  // byte of the first word
    const uint32_t skip = static_cast<uint32_t>((reinterpret_cast<uintptr_t>(in) + first_at) & 15u);
    const uint8_t *src = in + first_at - skip;  // (the stream's 272 leading bytes lie before)
    const uint8_t *src_end = in + in_bytes;
    auto load16 = [&](const uint8_t *a) -> uint4 {
      if (a + 16 <= src_end) return *reinterpret_cast<const uint4 *>(a);
      uint32_t x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        x[q] = a + 4 * q + 4 <= src_end ? *reinterpret_cast<const uint32_t *>(a + 4 * q) : 0u;
      return make_uint4(x[0], x[1], x[2], x[3]);
    };
    uint32_t have = 0, wi = skip / 4;
    uint4 ahead = load16(src);
    src += 16;
    auto top_up = [&]() {  // room for four words: put the 16 bytes held, fetch the next
      uint32_t *r = ring_in + 32 * (have & 7u);
      r[0] = ahead.x;
      r[32] = ahead.y;
      r[64] = ahead.z;
      r[96] = ahead.w;
      have += 4;
      ahead = load16(src);
      src += 16;
    };
    top_up();
    top_up();
    auto take = [&]() -> uint32_t {
      const uint32_t v = ring_in[32 * (wi & 7u)];
      ++wi;
      return v;
    };
    // bit buffer: the next `avail` bits, left-aligned
    const uint32_t b0 = take();
    uint64_t buf = ((static_cast<uint64_t>(b0) << 32) | take()) << (o % 32);
    uint32_t avail = 64 - o % 32;
    uint32_t used = 0;  // code bits so far
    bool invalid = false;
    auto refill = [&]() {  // afterwards at least 32 bits
      if (avail < 32) {
        buf |= static_cast<uint64_t>(take()) << (32 - avail);
        avail += 32;
      }
    };
    const uint32_t count = static_cast<uint32_t>(hi - lo);
    uint32_t done = 0;            // symbols decoded
    uint32_t flushed = 0;         // bytes stored to the output
    uint64_t acc = 0;             // decoded bytes not yet in the output ring
    uint32_t acc_bits = 0;        // (fewer than 32 between lookups)
    uint32_t *o_ring = ring_out;  // 16 words, word-major
    auto put = [&](uint32_t syms, uint32_t num) {
      acc |= static_cast<uint64_t>(syms) << acc_bits;
      acc_bits += 8 * num;
      done += num;
      if (acc_bits >= 32) {
        // the word that holds the bytes done - acc_bits / 8 .. + 3
        o_ring[32 * (((done * 8 - acc_bits) / 32) & 15u)] = static_cast<uint32_t>(acc);
        acc >>= 32;
        acc_bits -= 32;
      }
    };
    auto flush32 = [&]() {  // the next 32 bytes, a whole sector
      uint32_t x[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) x[q] = o_ring[32 * ((flushed / 4 + q) & 15u)];
      uint8_t *d = out + lo + flushed;
      if (out16) {
        // streaming stores: the output should not push the stream's lines,
        // which the other lanes of the warp still read, out of L2
        __stcs(reinterpret_cast<uint4 *>(d), make_uint4(x[0], x[1], x[2], x[3]));
        __stcs(reinterpret_cast<uint4 *>(d + 16), make_uint4(x[4], x[5], x[6], x[7]));
      } else {
#pragma unroll
        for (int q = 0; q < 32; ++q) d[q] = static_cast<uint8_t>(x[q / 4] >> (8 * (q & 3)));
      }
      flushed += 32;
    };
    // rounds of eight lookups: at most 96 bits (three words; the ring holds
    // five or more at the start of a round) and 24 symbols (the output ring
    // holds at most 31 bytes at the start of a round)
    constexpr uint32_t kLookups = 8;
    // one symbol each: a round gives two whole words of the output ring
    // (gathering them as below, uniform bytes took 94.6 us for 8 MiB, 86.4
    // before several symbols a lookup)
    while (one_each && done + kLookups <= count && !invalid) {
      if (have - wi <= 4) top_up();
#pragma unroll
      for (uint32_t h = 0; h < kLookups; h += 4) {
        uint32_t word = 0;
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q) {
          if (q % 2 == 0) refill();
          const uint32_t e = dec[static_cast<uint32_t>(buf >> (64 - kHufMaxLen))];
          const uint32_t l = (e >> 8) & 15u;
          invalid |= e == kHufInvalid;
          buf <<= l;
          avail -= l;
          used += l;
          word |= (e & 0xFFu) << (8 * q);
        }
        o_ring[32 * ((done / 4 + h / 4) & 15u)] = word;
      }
      done += kLookups;
      if (done - flushed >= 32) flush32();
    }
    while (!one_each && done + 3 * kLookups <= count && !invalid) {
      if (have - wi <= 4) top_up();
#pragma unroll
      for (uint32_t q = 0; q < kLookups; ++q) {
        if (q % 2 == 0) refill();  // 32 bits serve two lookups
        const uint32_t e = multi[static_cast<uint32_t>(buf >> (64 - kHufMaxLen))];
        const uint32_t l = (e >> 24) & 15u;  // an invalid entry reads as length 15
        invalid |= l > kHufMaxLen;
        buf <<= l;
        avail -= l;
        used += l;
        put(e & 0xFFFFFFu, e >> 28);
      }
      if (done - flushed >= 32) flush32();
    }
    // the rest, symbol by symbol
    while (done < count && !invalid) {
      if (have - wi <= 4) top_up();
      refill();
      const uint32_t e = dec[static_cast<uint32_t>(buf >> (64 - kHufMaxLen))];
      const uint32_t l = (e >> 8) & 15u;
      invalid |= e == kHufInvalid;
      buf <<= l;
      avail -= l;
      used += l;
      put(e & 0xFFu, 1);
      if (done - flushed >= 32 + 4) flush32();
    }
    if (!invalid) {
      while (done - flushed >= 32 && done * 8 - acc_bits >= 8 * (flushed + 32)) flush32();
      for (; flushed < done; ++flushed) {
        const uint32_t in_ring = done - acc_bits / 8;  // bytes before this lie in the ring
        const uint32_t v = flushed < in_ring
                               ? o_ring[32 * ((flushed / 4) & 15u)] >> (8 * (flushed & 3u))
                               : static_cast<uint32_t>(acc >> (8 * (flushed - in_ring)));
        out[lo + flushed] = static_cast<uint8_t>(v);
      }
    }
    const uint32_t pos = o + used;
    // each sub-block ends where the next begins; the block's words hold
    // exactly the bits used, rounded up to a word
    bool lane_bad = invalid || pos > nbits;
    if (lane < 31) lane_bad = lane_bad || pos != o_next;
    else lane_bad = lane_bad || (pos + 31) / 32 != nwords;
    if (__any_sync(kFull, lane_bad) && lane == 0) atomicOr(err, kErrCorrupt);
  }
}

}  // namespace

// `scratch`: 4096 bytes (histogram, code book, work counter), cleared here.
cudaError_t launch_huff_compress(const uint8_t *in, uint64_t n, uint8_t *out, uint64_t out_cap,
                                 unsigned long long *out_bytes, uint8_t *scratch, uint32_t *err,
                                 int sms, cudaStream_t st) {
  static LaunchCache lc;
  auto *hist = reinterpret_cast<unsigned long long *>(scratch);
  auto *book = reinterpret_cast<uint32_t *>(scratch + 2048);
  auto *ticket = reinterpret_cast<uint32_t *>(scratch + 3072);
  cudaError_t e = cudaMemsetAsync(scratch, 0, 4096, st);
  if (e != cudaSuccess) return e;
  const uint64_t nb = (n + kHufBlock - 1) / kHufBlock;
  if (n) {
    // four blocks per SM, fewer when each thread would not have 16 bytes
    const uint64_t want = (n + kHistThreads * 16 - 1) / (kHistThreads * 16);
    const unsigned grid = static_cast<unsigned>(want < 4ull * sms ? want : 4ull * sms);
    huff_hist_kernel<<<grid, kHistThreads, 0, st>>>(
        in, n, hist, reinterpret_cast<unsigned long long *>(out + kHufTableAt), nb);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  huff_book_kernel<<<1, 512, 0, st>>>(hist, n, out, book, out_bytes);
  if ((e = cudaGetLastError()) != cudaSuccess || nb == 0) return e;
  int per_sm = 0, dev_sms = 0;
  e = resident_blocks(lc, huff_encode_kernel, 256, kEncSmem, &per_sm, &dev_sms);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const uint64_t cap = static_cast<uint64_t>(per_sm) * dev_sms;
  const unsigned grid = static_cast<unsigned>(nb < cap ? nb : cap);
  huff_encode_kernel<<<grid, 256, kEncSmem, st>>>(in, n, out, out_cap, book, ticket, out_bytes,
                                                  err);
  return cudaGetLastError();
}

cudaError_t launch_huff_decompress(const uint8_t *in, uint64_t in_bytes, uint8_t *out,
                                   uint64_t out_cap, unsigned long long *out_bytes,
                                   uint32_t *err, cudaStream_t st) {
  static LaunchCache lc;
  int per_sm = 0, sms = 0;
  cudaError_t e = resident_blocks(lc, huff_decode_kernel, 256, kDecSmem, &per_sm, &sms);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // a warp per block of the largest stream that fits the output, at most
  // what is resident
  const uint64_t want = (out_cap / kHufBlock + 1 + 7) / 8;
  const uint64_t cap = static_cast<uint64_t>(per_sm) * sms;
  const unsigned grid = static_cast<unsigned>(want < cap ? want : cap);
  huff_decode_kernel<<<grid, 256, kDecSmem, st>>>(in, in_bytes, out, out_cap, out_bytes, err);
  return cudaGetLastError();
}

uint64_t huff_layout_bits_at(uint64_t n) {
  return huf_bits_at((n + kHufBlock - 1) / kHufBlock);
}

}  // namespace glz
