// glz_common.h -- launch-parameter structs shared by the host side of the
// C ABI and the kernels (product code only).
#pragma once

#include <cstdint>

namespace glz {

constexpr uint32_t kHeaderBytes = 32;   // GLZ1 header
constexpr uint32_t kTableEntry = 8;     // {u32 n_tokens, u32 payload_bytes}
constexpr uint32_t kIndexStride = 64;   // one u64 index entry per 64 chunks
constexpr uint32_t kMaxChunk = 32768;   // bytes
constexpr uint32_t kMaxWindow = 1024;   // symbols

// Matchers of the greedy parse (lz_match in lz.h).
constexpr uint32_t kMatchExact = 0;  // longest match, nearest offset on ties
constexpr uint32_t kMatchPaper = 1;  // the paper's forward scan (section 3.3.2)
constexpr uint32_t kMatchOverlap = 2;  // exact, a match may overlap its output

// Sticky device error bits (lz_sync maps them back to lz_status).
constexpr uint32_t kErrSmall = 1u << 0;
constexpr uint32_t kErrCorrupt = 1u << 1;
constexpr uint32_t kErrTimeout = 1u << 2;
constexpr uint32_t kErrInternal = 1u << 3;  // a device consistency check failed

// Bounded spins: a device wait that exceeds this many polls gives up and
// raises kErrTimeout instead of hanging the GPU.
constexpr uint32_t kSpinLimit = 1u << 22;

// Does a block of a GHF1 stream of `in_bytes` bytes, whose table says that it
// spans [start, end) of the bits at `bits_at` (<= in_bytes), lie inside the
// stream, as a whole number of words?  No sum is formed of values that come
// from the table (an end near 2^64 would wrap it past the check).
__host__ __device__ inline bool huf_span_ok(uint64_t start, uint64_t end, uint64_t bits_at,
                                            uint64_t in_bytes) {
  return start <= end && end <= in_bytes - bits_at && (end - start) % 4 == 0 &&
         end - start <= (1ull << 20);
}

// The parse by equality masks (mask_parse.cuh) takes the exact matchers when
// records can be written over the staged chunk (S * m >= 1 + offB), the first
// m rows of any position lie in the two slabs kept (m <= 32) and the window
// fits the widest instance (512 symbols: 16 mask words per lane; 32 would not
// leave registers for more than a few warps).  Everything else (the paper's
// matcher, other sizes) takes the hash chains.
constexpr uint32_t kMaskMaxWindow = 512;
__host__ __device__ inline bool mask_parse_takes(uint32_t S, uint32_t W, uint32_t m,
                                                 uint32_t match) {
  return match != kMatchPaper && W <= kMaskMaxWindow && m <= 32 &&
         S * m >= 1u + (W <= 256 ? 1u : 2u);
}
// Plane words of one slab of 32 symbols (one per symbol bit) and, for windows
// of 32 * nw symbols, the planes kept and the rows of two slabs for each one
// made at a time, and a spare row (bytes).
__host__ __device__ constexpr uint32_t mask_plane_words(uint32_t S) { return 8 * S; }
__host__ __device__ constexpr uint32_t mask_planes_bytes(uint32_t S, uint32_t nw) {
  return 2 * nw * mask_plane_words(S) * 4;
}
__host__ __device__ constexpr int mask_slabs_made(uint32_t nw) { return nw <= 8 ? 2 : 1; }
__host__ __device__ constexpr uint32_t mask_rows_bytes(uint32_t nw, uint32_t made) {
  return ((64 * made + 1) * nw * 4 + 15) & ~15u;
}

// The sample that chooses between masks and chains: one word per sampling warp.
constexpr uint32_t kSampleWarps = 64;

// Per-warp shared-memory layout of the compressor (byte offsets from the
// warp's slice; every region 16-byte aligned).
struct CompressSmem {
  uint32_t in_off;     // staged chunk, C bytes
  uint32_t prev_off;   // chain links; or the bit planes of the mask parse
  uint32_t flags_off;  // flag bits of up to k tokens
  uint32_t pay_off;    // hash table, then the pointer list; or the mask parse's rows
  uint32_t pay_bytes;  // size of the payload staging region
  uint32_t maybe_off;  // one bit per position: a match of >= m may exist
  uint32_t mbar_off;   // mbarrier for the TMA bulk copy
  uint32_t per_warp;   // total bytes per warp
  uint32_t hash_log2;  // hash table entries = 1 << hash_log2 (u16 each)
};

// Block of the compressor for few chunks (compress_coop.cuh): eight warps on
// one chunk.  Byte offsets of its shared memory after the staged chunk.
constexpr uint32_t kCoopWarps = 8;
struct CoopSmem {
  uint32_t planes_off;  // planes of the whole chunk, later the record's payload
  uint32_t rows_off;    // rows of each warp
  uint32_t info_off;    // per position: match length and offset (4 bytes)
  uint32_t reach_off;   // per position: tokens visited in its slab (4 bytes)
  uint32_t leave_off;   // per position: position after the slab (2 bytes)
  uint32_t slab_off;    // three words per slab
  uint32_t slabs;
  uint32_t flags_off;
  uint32_t total;
};
__host__ __device__ inline CoopSmem coop_layout(uint32_t S, uint32_t C, uint32_t nw) {
  const uint32_t k = C / S;
  CoopSmem L{};
  L.slabs = (k + 31) / 32;
  const uint32_t kk = 32 * L.slabs;  // whole slabs
  uint32_t at = (C + 31) & ~15u;
  L.planes_off = at;
  at += L.slabs * mask_plane_words(S) * 4 + 16;  // (>= C + 16)
  L.rows_off = at;
  at += kCoopWarps * mask_rows_bytes(nw, 1);
  L.info_off = at;
  at += 4 * kk;
  L.reach_off = at;
  at += 4 * kk;
  L.leave_off = at;
  at += 2 * kk;
  L.slab_off = at;
  at += 12 * L.slabs;
  at = (at + 15) & ~15u;
  L.flags_off = at;
  at += 4 * L.slabs + 16;
  L.total = (at + 127) & ~127u;
  return L;
}

// One buffer to compress (one stream): per-buffer parameters and places.
struct BufDesc {
  const uint8_t *in;
  uint64_t n;
  uint8_t *out;
  uint64_t cap;
  unsigned long long *out_bytes;
  uint32_t S, C, W, m, M, offB;
  uint32_t nc;          // chunks
  uint32_t in_aligned;  // in is 16-byte aligned: TMA bulk staging
  uint32_t match;       // kMatchExact, kMatchPaper or kMatchOverlap
  uint32_t version;     // stream version written: 1, or 2 (stored chunks); 0 reads as 1
  uint64_t records_at;  // byte offset of the records region
  uint64_t gbase;       // index of this buffer's chunk 0 among all chunks
};

// Shared memory of a batch's block beside its warps' slices: a descriptor for
// each of up to eight warps.
constexpr uint32_t kBatchDescBytes = 8 * sizeof(BufDesc);

struct CompressArgs {
  BufDesc buf;                 // single-buffer launch
  const BufDesc *items;        // batched launch (nullptr for a single buffer)
  const uint64_t *item_base;   // items[i].gbase, ascending (batched launch)
  uint32_t n_items;            // non-empty items
  uint64_t total_chunks;       // chunks over all items
  CompressSmem sm;             // per-warp layout (covers every item)
  CoopSmem coop;               // or the layout of a block per chunk
  unsigned long long *status;  // one look-back word per chunk (cleared per call)
  uint32_t *ticket;            // work counter (cleared per call)
  uint32_t *votes;             // kSampleWarps words, samples of the launch's data (sample.cuh);
                               // null: this kernel takes the launch whatever its data
  uint32_t *err;               // sticky error bits
  uint8_t *park;               // parking slots: grid warps x park_slots
  uint32_t park_slots;         // slots per warp (<= 32)
  uint32_t park_slot_bytes;    // one worst-case record, 16-byte multiple
  uint32_t spin_limit;         // polls before a device wait gives up (kSpinLimit normally)
  uint32_t first_ticket;       // first chunk handed out (0 normally)
  uint32_t end_chunk;          // single buffer: chunks [first_ticket, end_chunk) are taken
};

// The classes of a batch between whose parses a sample chooses: three symbol
// sizes, three window classes.
struct SampleClass {
  const BufDesc *items;
  const uint64_t *item_base;
  uint64_t total_chunks;
  uint32_t *votes;
  uint32_t n_items, S, nj;
};
struct SampleList {
  SampleClass e[9];
  uint32_t n;
};

// Placement of one shard stream inside a whole-input stream (lz_stitch).
struct StitchArgs {
  const uint8_t *shard;   // 8-byte aligned
  uint64_t shard_chunks;  // chunks in the shard
  uint64_t chunk_base;    // chunks before it (multiple of kIndexStride)
  uint64_t total_chunks;
  uint64_t total_bytes;
  uint64_t record_base;   // record bytes of the shards before it
  uint64_t src_records;   // byte offset of the shard's records
  uint64_t record_bytes;  // the shard's record bytes
  uint64_t dst_records;   // byte offset of this shard's records in out
  uint8_t *out;           // 8-byte aligned
  uint32_t *err;
};

struct DecompressArgs {
  const uint8_t *in;
  uint64_t in_bytes;
  uint8_t *out;
  uint64_t out_cap;
  unsigned long long *out_bytes;
  uint32_t *err;
  uint32_t smem_bytes;  // dynamic shared memory per block
  int out_aligned;      // out is 16-byte aligned
};

// One stream of a batched decompression.
struct DecItem {
  const uint8_t *in;
  uint64_t in_bytes;
  uint8_t *out;
  uint64_t out_cap;
  unsigned long long *out_bytes;
  uint64_t gbase;  // index of this stream's chunk 0 among all chunks
  uint32_t nc;
  uint32_t out_aligned;
};

// Per-warp shared-memory slice of the decoder (byte offsets, 16-byte
// aligned): an mbarrier, one mark byte per position of the chunk (0 inside
// a token, 1 where a literal starts, 2 where a pointer starts), a copy of
// the record's flag bytes, later a round's source distances, the high bytes of
// (offset - 1) when one-byte symbols carry two-byte offsets, then -- when they fit -- the io area:
// the chunk's output image from its start, with the record staged at its
// end.  When no pointer takes more payload bytes than the symbols it
// covers (S * m >= 1 + offB for every stream; `shared`), the output
// written so far never reaches a payload byte not yet read, so the area
// only needs room for the larger of the two; otherwise it holds both side
// by side.  Without the io area (`staged` false) a warp decodes straight
// into the output buffer and reads the record in place.
struct DecodeLayout {
  uint32_t marks_off;  // mark bytes, a multiple of 128 (a round of positions)
  uint32_t mark_bytes;
  uint32_t flags_off;  // flag bytes of one record (+ 16 slack)
  uint32_t flag_bytes;
  uint32_t dist_off;   // kDistBytes over the flag bytes (second phase)
  uint32_t hi_off;     // k bytes (one-byte symbols, two-byte offsets) or none
  uint32_t io_off;     // output image + staged record
  uint32_t io_bytes;
  uint32_t per_warp;
  uint32_t staged;
};

// Largest record of a chunk of k symbols: flags, payload and (stream version
// 2, last chunk) up to S - 1 tail bytes.
__host__ __device__ inline uint64_t decode_record_bound(uint64_t k, uint32_t S, uint32_t offB,
                                                       uint32_t m) {
  const uint64_t extra = (1u + offB > S * m) ? (1u + offB - S * m) : 0u;
  return (k + 7) / 8 + static_cast<uint64_t>(S) * k + extra * (k / m) + (S - 1);
}

// A round's source distances (128 u16) and a zero after them.
constexpr uint32_t kDistBytes = 256 + 16;

// Slack of the io area past the staged record (its end is at most this
// many bytes before the area's end, minus 15 for alignment).
constexpr uint32_t kIoSlack = 64;

// Slice for chunks of at most `kmax` symbols and `cmax` bytes whose records
// are at most `rmax` bytes; the full slice when `budget` bytes hold it,
// else without the io area.
__host__ __device__ inline DecodeLayout decode_layout(uint64_t kmax, uint64_t cmax,
                                                      uint64_t rmax, bool hi, bool shared,
                                                      uint64_t budget) {
  DecodeLayout L{};
  uint64_t at = 16;  // mbarrier
  L.marks_off = static_cast<uint32_t>(at);
  L.mark_bytes = static_cast<uint32_t>((kmax + 127) & ~127ull);
  at += L.mark_bytes;
  L.flags_off = static_cast<uint32_t>(at);
  // (the second phase reads no flags: its distances take their place, which
  // keeps 21 warps resident on streams of 8 KiB chunks, 20 beside them)
  L.flag_bytes = static_cast<uint32_t>(((kmax + 7) / 8 + 15) & ~15ull) + 16;
  if (L.flag_bytes < kDistBytes) L.flag_bytes = kDistBytes;
  L.dist_off = L.flags_off;
  at += L.flag_bytes;
  L.hi_off = static_cast<uint32_t>(at);
  if (hi) at += (kmax + 15) & ~15ull;
  const uint64_t base = at;
  L.io_off = static_cast<uint32_t>(at);
  const uint64_t c16 = ((cmax + 15) & ~15ull) + 16, r16 = (rmax + 15) & ~15ull;
  L.io_bytes = static_cast<uint32_t>((shared ? (c16 > r16 ? c16 : r16) : c16 + r16) + 32 +
                                     kIoSlack);
  at += L.io_bytes;
  L.staged = at <= budget;
  if (!L.staged) at = base;
  L.per_warp = static_cast<uint32_t>(at);
  return L;
}

struct DecompressBatchArgs {
  const DecItem *items;        // streams with at least one chunk
  const uint64_t *item_base;   // items[i].gbase, ascending
  uint32_t n_items;
  uint64_t total_chunks;
  const DecItem *empties;      // streams of zero bytes
  uint32_t n_empty;
  DecodeLayout lay;            // per-warp slice covering every stream
  uint32_t smem_bytes;         // dynamic shared memory per block
  uint32_t *err;
};

}  // namespace glz
