// decompress.cu -- the decompression kernel (one warp per chunk).
//
// The paper only reports decompression throughput (section 4.4) and gives
// no algorithm; this is the design used here.  The host knows nothing
// about the stream: every warp reads and checks the header itself, so the
// call needs no host synchronisation.  Per chunk:
//   * the record offset is the superblock index entry plus the record sizes
//     of the (at most 63) chunks before it in its superblock -- no scan
//     across the whole stream;
//   * the record (flags + payload) is staged into the warp's shared slice
//     with a TMA bulk copy; a chunk without pointers (or a stored chunk of
//     stream version 2) is copied straight out with 16-byte stores;
//   * otherwise the chunk is decoded into a shared-memory image of its
//     output in two phases, four tokens or positions per lane.  Phase 1
//     takes 128 tokens a round: flag bits give each token's payload offset by
//     popcount, a shuffle scan of the lanes' lengths its output position; a
//     literal writes its symbol there, a pointer writes (offset - 1) into the
//     slot of its first symbol, and both mark their first position (one byte
//     per position: literal or pointer start).  Phase 2 takes 128 output
//     positions a round: the owning token is the last marked position at or
//     before the position (in the lane, in the lanes before it by a vote, or
//     carried from the round before), a position inside a pointer copies from
//     position - offset, and sources inside the round that are pointer
//     symbols themselves are followed back through the round's offsets in
//     shared memory; earlier positions are final, later rounds read them;
//   * the image is copied out with 16-byte stores.
// Pointers never reach before their own chunk, so chunks are independent
// (section 3.3.1).  When the slice cannot hold the output image and the
// record window (very large chunks), the same two phases run on the output
// buffer itself and read the record in place.
#include <cuda_runtime.h>

#include "glz_common.h"
#include "glz_device.cuh"
#include "launch_cache.cuh"

namespace glz {

namespace {

struct Header {
  uint32_t version, overlap, S, offB, m, M, C, W, nc;
  uint64_t n;
};

__device__ __forceinline__ bool read_header(const uint8_t *in, Header &h) {
  const bool magic = in[0] == 'G' && in[1] == 'L' && in[2] == 'Z' &&
                     in[3] == '1' && (in[4] == 1 || in[4] == 2) &&
                     in[9] <= (in[4] == 2 ? 1 : 0) && in[10] == 0 && in[11] == 0;
  h.version = in[4];
  h.overlap = in[9];  // version 2: pointers may be longer than their offset
  h.S = in[5];
  h.offB = in[6];
  h.m = in[7];
  h.M = in[8];
  h.C = static_cast<uint32_t>(ld_le(in + 12, 4));
  h.W = static_cast<uint32_t>(ld_le(in + 16, 4));
  h.nc = static_cast<uint32_t>(ld_le(in + 20, 4));
  h.n = ld_le(in + 24, 8);
  bool ok = magic && (h.S == 1 || h.S == 2 || h.S == 4);
  ok = ok && h.C >= 16 && h.C <= kMaxChunk && h.C % 16 == 0;
  ok = ok && h.W >= 1 && h.W <= kMaxWindow;
  ok = ok && h.m >= 1 && h.m <= h.M && h.M <= 255;
  ok = ok && h.offB == (h.W <= 256 ? 1u : 2u);
  ok = ok && (h.version == 2 || h.n % h.S == 0);  // version 2 allows a tail
  ok = ok && static_cast<uint64_t>(h.nc) == (h.n + h.C - 1) / h.C;
  return ok;
}

// Eight bytes of the table or index: one load when the stream is 8-byte
// aligned (`aligned`, the same for every thread), else byte by byte.
__device__ __forceinline__ uint64_t ld_entry(const uint8_t *p, bool aligned) {
  return aligned ? *reinterpret_cast<const uint64_t *>(p) : ld_le(p, 8);
}

// Sum of the record sizes of chunks [lo, hi) (hi - lo <= 64).
__device__ __forceinline__ uint64_t record_bytes(const uint8_t *table,
                                                 uint32_t lo, uint32_t hi,
                                                 uint32_t lane, bool aligned) {
  uint64_t part = 0;
  for (uint32_t e = lo + lane; e < hi; e += 32) {
    const uint64_t v = ld_entry(table + 8ull * e, aligned);
    part += ((v & 0xFFFFFFFFu) + 7) / 8 + (v >> 32);
  }
  return warp_sum_u64(part);
}

// Worst-case record of a chunk of k symbols (flags + payload, no tail).
__device__ __forceinline__ uint64_t record_bound(uint64_t k, const Header &h) {
  const uint64_t extra = (1u + h.offB > h.S * h.m) ? (1u + h.offB - h.S * h.m) : 0u;
  return (k + 7) / 8 + static_cast<uint64_t>(h.S) * k + extra * (k / h.m);
}

// Little-endian 32-bit word at any byte address of shared memory (the two
// aligned words around it; may read up to 3 bytes past the addressed ones).
__device__ __forceinline__ uint32_t ld_u32_any(const uint8_t *p) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p);
  const uint32_t *w = reinterpret_cast<const uint32_t *>(a & ~static_cast<uintptr_t>(3));
  const uint32_t sh = 8u * static_cast<uint32_t>(a & 3u);
  return sh ? __funnelshift_r(w[0], w[1], sh) : w[0];
}

// Symbol slot j of an output image (S-byte aligned) or of an output buffer
// of any alignment.
template <int S>
__device__ __forceinline__ uint32_t ld_slot(const uint8_t *o, uint32_t j, bool aligned) {
  const uint8_t *p = o + static_cast<uint64_t>(j) * S;
  if constexpr (S == 1) return *p;
  if (aligned) {
    if constexpr (S == 2) return *reinterpret_cast<const uint16_t *>(p);
    else return *reinterpret_cast<const uint32_t *>(p);
  }
  return static_cast<uint32_t>(ld_le(p, S));
}

template <int S>
__device__ __forceinline__ void st_slot(uint8_t *o, uint32_t j, uint32_t v, bool aligned) {
  uint8_t *p = o + static_cast<uint64_t>(j) * S;
  if constexpr (S == 1) {
    *p = static_cast<uint8_t>(v);
    return;
  }
  if (aligned) {
    if constexpr (S == 2) *reinterpret_cast<uint16_t *>(p) = static_cast<uint16_t>(v);
    else *reinterpret_cast<uint32_t *>(p) = v;
    return;
  }
  for (uint32_t i = 0; i < S; ++i) p[i] = static_cast<uint8_t>(v >> (8 * i));
}

// Copy record bytes [src, src + n) to the end of the warp's io area (16-byte
// aligned, io_bytes long), ending at most kIoSlack bytes before it, so that
// the copy is 16-byte aligned on both sides: head and tail with plain
// loads, the middle with one TMA bulk copy.  Returns the shared address of
// byte 0.
__device__ __forceinline__ const uint8_t *stage_record(const uint8_t *src,
                                                       uint32_t n, uint8_t *io,
                                                       uint32_t io_bytes, uint64_t *bar,
                                                       uint32_t &phase,
                                                       uint32_t lane, bool &ok) {
  const uint32_t mis = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(src) & 15u);
  uint8_t *dst = io + ((io_bytes - kIoSlack - n - 15) & ~15u) + mis;
  const uint32_t head = min(n, (16u - mis) & 15u);
  const uint32_t bulk = (n - head) & ~15u;
  if (bulk && lane == 0) {
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(bar, bulk);
    bulk_g2s(dst + head, src + head, bulk, bar);
  }
  for (uint32_t i = lane; i < head; i += 32) dst[i] = src[i];
  for (uint32_t i = head + bulk + lane; i < n; i += 32) dst[i] = src[i];
  ok = true;
  if (bulk) {
    ok = mbar_wait_bounded(bar, phase);
    phase ^= 1u;
  }
  __syncwarp();
  return dst;
}

// 16 bytes of (a, b) starting at byte r (r uniform over the warp).
__device__ __forceinline__ uint4 bytes16(const uint4 &a, const uint4 &b, uint32_t r) {
  const uint32_t s = 8u * (r & 3u);
  uint32_t w0, w1, w2, w3, w4;
  switch (r >> 2) {
    case 0: w0 = a.x; w1 = a.y; w2 = a.z; w3 = a.w; w4 = b.x; break;
    case 1: w0 = a.y; w1 = a.z; w2 = a.w; w3 = b.x; w4 = b.y; break;
    case 2: w0 = a.z; w1 = a.w; w2 = b.x; w3 = b.y; w4 = b.z; break;
    default: w0 = a.w; w1 = b.x; w2 = b.y; w3 = b.z; w4 = b.w; break;
  }
  if (s == 0) return make_uint4(w0, w1, w2, w3);
  return make_uint4(__funnelshift_r(w0, w1, s), __funnelshift_r(w1, w2, s),
                    __funnelshift_r(w2, w3, s), __funnelshift_r(w3, w4, s));
}

// Warp copy of n bytes from shared src (any alignment, 16 bytes of slack
// readable past the end) to global dst, 16-byte stores where dst allows.
__device__ __forceinline__ void copy_s2g(uint8_t *dst, const uint8_t *src,
                                         uint32_t n, uint32_t lane) {
  const uint32_t head = min(
      n, (16u - static_cast<uint32_t>(reinterpret_cast<uintptr_t>(dst) & 15u)) & 15u);
  if (lane < head) dst[lane] = src[lane];
  const uint32_t body = (n - head) >> 4;
  const uint8_t *sb = src + head;
  const uint32_t r = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(sb) & 15u);
  const uint4 *s16 = reinterpret_cast<const uint4 *>(sb - r);
  uint4 *d16 = reinterpret_cast<uint4 *>(dst + head);
  for (uint32_t j = lane; j < body; j += 32) d16[j] = bytes16(s16[j], s16[j + 1], r);
  const uint32_t done = head + 16u * body;
  for (uint32_t i = done + lane; i < n; i += 32) dst[i] = src[i];
}


// A warp's shared-memory slice (see DecodeLayout).
struct Slice {
  uint64_t *bar;
  uint8_t *marks;           // per position: 0 inside a token, 1 literal start, 2 pointer start
  uint16_t *dist;           // per position of a round: how far back its source lies (over fl,
                            // which only the first phase reads)
  uint8_t *hi;              // high bytes of (offset - 1), or nullptr
  uint8_t *fl;              // a copy of the record's flag bytes
  uint8_t *io;              // output image + staged record, or nullptr (decode
                            // into the output, read the record in place)
  uint32_t io_bytes, flag_bytes, mark_bytes;  // region sizes
  uint32_t phase;           // parity of the next TMA completion on bar
};

__device__ __forceinline__ Slice make_slice(uint8_t *ws, const DecodeLayout &L, bool hi) {
  Slice sl;
  sl.bar = reinterpret_cast<uint64_t *>(ws);
  sl.marks = ws + L.marks_off;
  sl.dist = reinterpret_cast<uint16_t *>(ws + L.dist_off);
  sl.hi = hi ? ws + L.hi_off : nullptr;
  sl.fl = ws + L.flags_off;
  sl.io = L.staged ? ws + L.io_off : nullptr;
  sl.io_bytes = L.staged ? L.io_bytes : 0;
  sl.flag_bytes = L.flag_bytes;
  sl.mark_bytes = L.mark_bytes;
  sl.phase = 0;
  return sl;
}

// Symbols per lane and round of the two phases: a lane takes four consecutive
// tokens (phase 1) or positions (phase 2), so that votes, scans and the carry
// from lane to lane are paid once per 128 instead of once per 32, and slots,
// marks and payload move as words of four.  With one token or position per
// lane the quantization codes took 8.0 K warp instructions per 4 KiB chunk
// (issue-bound, 0.531 ms for 256 MiB).
constexpr uint32_t kPer = 4, kRound = 32 * kPer;

// The slots of positions j .. j + 3 (j a multiple of 4) of an output image.
template <int S>
__device__ __forceinline__ void ld_slots(const uint8_t *o, uint32_t j, uint32_t (&v)[kPer]) {
  if constexpr (S == 1) {
    const uint32_t w = *reinterpret_cast<const uint32_t *>(o + j);
    v[0] = w & 0xFFu;
    v[1] = (w >> 8) & 0xFFu;
    v[2] = (w >> 16) & 0xFFu;
    v[3] = w >> 24;
  } else if constexpr (S == 2) {
    const uint2 w = *reinterpret_cast<const uint2 *>(o + 2 * j);
    v[0] = w.x & 0xFFFFu;
    v[1] = w.x >> 16;
    v[2] = w.y & 0xFFFFu;
    v[3] = w.y >> 16;
  } else {
    const uint4 w = *reinterpret_cast<const uint4 *>(o + 4 * j);
    v[0] = w.x;
    v[1] = w.y;
    v[2] = w.z;
    v[3] = w.w;
  }
}

template <int S>
__device__ __forceinline__ void st_slots(uint8_t *o, uint32_t j, const uint32_t (&v)[kPer]) {
  if constexpr (S == 1) {
    *reinterpret_cast<uint32_t *>(o + j) =
        __byte_perm(__byte_perm(v[0], v[1], 0x0040), __byte_perm(v[2], v[3], 0x0040), 0x5410);
  } else if constexpr (S == 2) {
    *reinterpret_cast<uint2 *>(o + 2 * j) =
        make_uint2(__byte_perm(v[0], v[1], 0x5410), __byte_perm(v[2], v[3], 0x5410));
  } else {
    *reinterpret_cast<uint4 *>(o + 4 * j) = make_uint4(v[0], v[1], v[2], v[3]);
  }
}

// Phases 1 and 2 for a chunk of k symbols with ntok tokens whose payload
// holds pay_tok bytes of tokens: the symbols are written into `ob` (the
// output image, or the output itself).  The flag bytes are in sl.fl, bits
// past ntok cleared up to the next multiple of 128.  STAGED: the record is in
// shared memory (words may be read up to 12 bytes past it) and `ob` is the
// image.  False when the tokens are inconsistent (corrupt stream); nothing
// outside the chunk's output and the slice is written either way.
// SAME: a pointer's payload is S bytes like a literal's (1 + offB == S), so
// token t's payload starts at S * t without counting the pointers before it.
template <int S, bool STAGED, bool SAME = false>
__device__ __forceinline__ bool decode_tokens(const Header &h, const uint8_t *payload,
                                              uint32_t ntok, uint32_t pay_tok, uint32_t k,
                                              uint8_t *ob, bool aligned, const Slice &sl,
                                              uint32_t lane) {
  const uint32_t tsz = 1u + h.offB;
  const uint32_t offmask = h.offB == 2 ? 0xFFFFu : 0xFFu;
  const uint32_t lt = lanemask_lt(lane);
  uint8_t *marks = sl.marks;
  const uint32_t *fw = reinterpret_cast<const uint32_t *>(sl.fl);
  {
    uint4 *m16 = reinterpret_cast<uint4 *>(marks);
    const uint32_t n16 = ((k + kRound - 1) & ~(kRound - 1)) / 16;
    for (uint32_t i = lane; i < n16; i += 32) m16[i] = make_uint4(0, 0, 0, 0);
  }
  __syncwarp();

  // Phase 1: tokens.  A lane's four flag bits and, unless SAME, the pointers
  // before them in the round (popcounts of the round's four flag words) give
  // its tokens' payload offsets: S bytes per literal and 1 + offB per pointer
  // before it.  One scan of the lanes' lengths gives the output positions.
  // The payload must hold exactly the flagged tokens, checked before any
  // token is read.
  uint32_t np = 0;
  for (uint32_t g = lane; g < (ntok + 31) / 32; g += 32) np += __popc(fw[g]);
  np = __reduce_add_sync(kFull, np);
  if (S * (ntok - np) + tsz * np != pay_tok) return false;
  uint32_t pos = 0, pdone = 0;  // symbols produced; pointers in earlier rounds
#pragma unroll 1
  for (uint32_t t0 = 0; t0 < ntok; t0 += kRound) {
    const uint32_t t = t0 + kPer * lane;
    const uint32_t nv = t < ntok ? min(kPer, ntok - t) : 0u;
    const uint32_t own = fw[t0 / 32 + (lane >> 3)], at = kPer * (lane & 7u);
    const uint32_t f = own >> at;
    uint32_t w[kPer];
    if constexpr (SAME && STAGED) {
      if (nv && GLZ_OK(S * t < pay_tok)) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(payload + S * t);
        const uint32_t *p = reinterpret_cast<const uint32_t *>(a & ~static_cast<uintptr_t>(3));
        const uint32_t sh = 8u * static_cast<uint32_t>(a & 3u);  // 0 or 16
        const uint32_t x = p[0], y = p[1], z = p[2];
        const uint32_t lo = __funnelshift_r(x, y, sh), hi = __funnelshift_r(y, z, sh);
        w[0] = lo & 0xFFFFu;
        w[1] = lo >> 16;
        w[2] = hi & 0xFFFFu;
        w[3] = hi >> 16;
      } else {
        w[0] = w[1] = w[2] = w[3] = 0;
      }
    } else {
      const uint4 all = *reinterpret_cast<const uint4 *>(fw + t0 / 32);
      const uint32_t c0 = __popc(all.x), c1 = c0 + __popc(all.y), c2 = c1 + __popc(all.z);
      const uint32_t g = lane >> 3;
      uint32_t before = g == 0 ? 0u : g == 1 ? c0 : g == 2 ? c1 : c2;
      before += pdone + __popc(own & ((1u << at) - 1u));
      pdone += c2 + __popc(all.w);
      uint32_t o = S * (t - before) + tsz * before;
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) {
        const bool m = (f >> i) & 1u;
        w[i] = 0;
        if (i < nv && GLZ_OK(o < pay_tok)) {
          if constexpr (STAGED) w[i] = ld_u32_any(payload + o);
          else w[i] = static_cast<uint32_t>(ld_le(payload + o, m ? tsz : S));
        }
        o += m ? tsz : S;
      }
    }
    uint32_t len[kPer], off[kPer], sum = 0;
#pragma unroll
    for (uint32_t i = 0; i < kPer; ++i) {
      const bool m = (f >> i) & 1u;
      len[i] = m ? w[i] & 0xFFu : (i < nv ? 1u : 0u);
      off[i] = ((w[i] >> 8) & offmask) + 1u;
      sum += len[i];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, incl, o);
      if (lane >= static_cast<uint32_t>(o)) incl += y;
    }
    uint32_t st = pos + incl - sum;
    pos += __shfl_sync(kFull, incl, 31);
    // a pointer needs 1 <= length <= offset (any length <= 255 in overlap
    // mode) and offset <= min(W, its start): its source lies in the chunk
    bool bad = pos > k;
    uint32_t start[kPer];
#pragma unroll
    for (uint32_t i = 0; i < kPer; ++i) {
      start[i] = st;
      const uint32_t cap = h.overlap ? 256u : off[i];
      bad |= ((f >> i) & 1u) && !(len[i] - 1u < cap && off[i] <= min(h.W, st));
      st += len[i];
    }
    if (__any_sync(kFull, bad)) return false;
#pragma unroll
    for (uint32_t i = 0; i < kPer; ++i) {
      if (i >= nv || !GLZ_OK(start[i] < k && start[i] < sl.mark_bytes)) continue;
      const bool m = (f >> i) & 1u;
      marks[start[i]] = m ? 2 : 1;
      st_slot<S>(ob, start[i], m ? off[i] - 1u : w[i], aligned);
      if (S == 1 && sl.hi && m) sl.hi[start[i]] = static_cast<uint8_t>((off[i] - 1u) >> 8);
    }
  }
  if (pos != k) return false;
  __syncwarp();

  // Phase 2: positions.  A position's offset is that of the token it lies in
  // (0: a literal), carried from lane to lane by one vote and one shuffle per
  // round.  Offsets of the round go to sl.dist; a source inside the round
  // that is itself a pointer symbol is followed back through them until it is
  // a literal of the round or lies before it (2 to 3 turns on codes with 50
  // to 80 % pointer symbols).
  uint32_t carry = 0;  // offset owning the previous round's last position
  if (lane == 0) sl.dist[kRound] = 0;
#pragma unroll 1
  for (uint32_t r0 = 0; r0 < k; r0 += kRound) {
    const uint32_t x0 = kPer * lane, j = r0 + x0;
    const uint32_t nv = j < k ? min(kPer, k - j) : 0u;
    const uint32_t mk = *reinterpret_cast<const uint32_t *>(marks + j);  // zero past k
    uint32_t v[kPer] = {0, 0, 0, 0};
    if constexpr (STAGED) {
      if (nv) ld_slots<S>(ob, j, v);
    } else {
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i)
        if (i < nv) v[i] = ld_slot<S>(ob, j + i, aligned);
    }
    uint32_t s[kPer];  // offset of the token starting here (0: literal)
    if (S == 1 && sl.hi) {
      const uint32_t hw = nv ? *reinterpret_cast<const uint32_t *>(sl.hi + j) : 0u;
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) s[i] = (v[i] | (((hw >> (8 * i)) & 0xFFu) << 8)) + 1u;
    } else {
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) s[i] = v[i] + 1u;
    }
    uint32_t last = 0;  // that of the lane's last start
#pragma unroll
    for (uint32_t i = 0; i < kPer; ++i) {
      const uint32_t b = (mk >> (8 * i)) & 0xFFu;
      s[i] = b == 2 ? s[i] : 0u;
      last = b ? s[i] : last;
    }
    const uint32_t starts = __ballot_sync(kFull, mk != 0);
    const uint32_t prev = starts & lt;
    const uint32_t from_lane = __shfl_sync(kFull, last, (31u - __clz(prev)) & 31u);
    uint32_t own = prev ? from_lane : carry;
    uint32_t off[kPer], f[kPer];
#pragma unroll
    for (uint32_t i = 0; i < kPer; ++i) {
      own = (mk >> (8 * i)) & 0xFFu ? s[i] : own;
      off[i] = i < nv ? own : 0u;
      f[i] = j + i - off[i];
    }
    carry = __shfl_sync(kFull, own, 31);
    uint2 *mine = reinterpret_cast<uint2 *>(sl.dist + x0);
    *mine = make_uint2(__byte_perm(off[0], off[1], 0x5410), __byte_perm(off[2], off[3], 0x5410));
    __syncwarp();
    // one turn: every source in the round moves to its own source (by 0 at a
    // literal; sources before the round read the 0 after the round's entries)
    auto turn = [&]() -> bool {
      uint32_t moved = 0;
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) {
        const uint32_t d = sl.dist[min(f[i] - r0, kRound)];
        f[i] -= d;
        moved |= d;
      }
      return moved != 0;
    };
    bool again = true;
#pragma unroll 1
    for (uint32_t n = 0; again && n < 4; ++n) again = turn();
    // long chains (matches that overlap their output): the distances already
    // followed replace the offsets, which doubles the reach of a turn.  A
    // lane may see another's old or new distance; both lead back along the
    // same chain.
    while (__any_sync(kFull, again)) {
      uint32_t d[kPer];
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i) d[i] = j + i - f[i];
      *mine = make_uint2(__byte_perm(d[0], d[1], 0x5410), __byte_perm(d[2], d[3], 0x5410));
      __syncwarp();
      again = turn();
    }
    // (a literal is read from and written to its own slot: other lanes of the
    // round may be reading it)
    if constexpr (STAGED) {
      if (nv) {
#pragma unroll
        for (uint32_t i = 0; i < kPer; ++i)
          if (GLZ_OK(f[i] <= j + i)) v[i] = ld_slot<S>(ob, f[i], true);
        st_slots<S>(ob, j, v);
      }
    } else {
#pragma unroll
      for (uint32_t i = 0; i < kPer; ++i)
        if (off[i] && GLZ_OK(f[i] < j + i)) st_slot<S>(ob, j + i, ld_slot<S>(ob, f[i], aligned), aligned);
    }
    __syncwarp();
  }
  return true;
}

template <bool STAGED>
__device__ __forceinline__ bool decode_tokens_s(const Header &h, const uint8_t *payload,
                                                uint32_t ntok,
                                                uint32_t pay_tok, uint32_t k, uint8_t *ob,
                                                bool aligned, const Slice &sl, uint32_t lane) {
  switch (h.S) {
    case 1:
      return decode_tokens<1, STAGED>(h, payload, ntok, pay_tok, k, ob, aligned, sl, lane);
    case 2:
      if (h.offB == 1)  // a pointer (length, offset - 1) is two bytes, as a symbol
        return decode_tokens<2, STAGED, true>(h, payload, ntok, pay_tok, k, ob, aligned, sl,
                                              lane);
      return decode_tokens<2, STAGED>(h, payload, ntok, pay_tok, k, ob, aligned, sl, lane);
    default:
      return decode_tokens<4, STAGED>(h, payload, ntok, pay_tok, k, ob, aligned, sl, lane);
  }
}

// One chunk.  Returns false when a TMA copy did not complete in time (the
// warp must stop: its barrier phase is unknown).
__device__ __forceinline__ bool decode_chunk(const DecompressArgs &A, const Header &h,
                                             uint32_t c, uint64_t records_at, Slice &sl,
                                             uint32_t lane) {
  const uint8_t *in = A.in;
  const uint8_t *table = in + kHeaderBytes;
  const uint8_t *index = table + 8ull * h.nc;
  const uint32_t j = c / kIndexStride;
  const bool al = (reinterpret_cast<uintptr_t>(in) & 7u) == 0;
  const uint64_t idxv = ld_entry(index + 8ull * j, al);
  const uint64_t entry = ld_entry(table + 8ull * c, al);
  const uint64_t part = record_bytes(table, j * kIndexStride, c, lane, al);
  bool bad = false;
  if (c == 0) bad = idxv != 0;
  if (c % kIndexStride == 0 && c > 0) {
    const uint64_t prev = ld_entry(index + 8ull * (j - 1), al);
    const uint64_t sb = record_bytes(table, c - kIndexStride, c, lane, al);
    bad = bad || prev + sb != idxv;
  }
  const uint32_t ntok = static_cast<uint32_t>(entry);
  const uint32_t pay = static_cast<uint32_t>(entry >> 32);
  const uint64_t fb = (static_cast<uint64_t>(ntok) + 7) / 8;
  const uint64_t rec_at = records_at + idxv + part;
  const uint64_t chunk_at = static_cast<uint64_t>(c) * h.C;
  const uint32_t bytes_c = static_cast<uint32_t>((c + 1 < h.nc) ? h.C : h.n - chunk_at);
  const uint32_t k = bytes_c / h.S;
  const uint32_t tail = bytes_c - k * h.S;  // version 2, last chunk: bytes after the last symbol
  // version 2: a token count of 0 marks a stored chunk (its bytes as they are)
  const bool stored = h.version == 2 && ntok == 0;
  bad = bad || idxv > A.in_bytes || rec_at + fb + pay > A.in_bytes ||
        rec_at + fb + pay < rec_at || ntok > k || (ntok == 0 && !stored) ||
        (stored && pay != bytes_c) || (!stored && pay < tail) ||
        fb + pay > record_bound(k, h) + tail;
  if (bad) {
    if (lane == 0) atomicOr(A.err, kErrCorrupt);
    return true;
  }
  const uint8_t *flags = in + rec_at;  // read in place when there is no io area
  if (sl.io) {
    bool staged;
    if (!GLZ_OK(fb + pay + kIoSlack + 15 <= sl.io_bytes)) return true;
    flags = stage_record(in + rec_at, static_cast<uint32_t>(fb + pay), sl.io, sl.io_bytes,
                         sl.bar, sl.phase, lane, staged);
    if (!staged) {
      if (lane == 0) atomicOr(A.err, kErrTimeout);
      return false;
    }
  }
  const uint8_t *payload = flags + fb;
  uint8_t *dst = A.out + chunk_at;
  if (stored) {
    if (sl.io) {
      copy_s2g(dst, payload, pay, lane);  // the io area has slack past the record
    } else {
      for (uint32_t i = lane; i < pay; i += 32) dst[i] = payload[i];
    }
    return true;
  }
  // the flag words are copied out (the output image grows from the start of
  // the io area towards the record's flags), the bits past the last token
  // cleared up to a round of the token phase
  const uint32_t fwords = ((static_cast<uint32_t>(fb) + 15u) & ~15u) / 4;
  if (!GLZ_OK(4 * fwords <= sl.flag_bytes)) return true;
  uint32_t any = 0;
  for (uint32_t i = lane; i < fwords; i += 32) {
    uint32_t v = 0;
    if (32 * i < ntok) {
      if (sl.io) {
        v = ld_u32_any(flags + 4 * i);
      } else {
        for (uint32_t q = 0; q < 4; ++q)
          if (4 * i + q < fb) v |= static_cast<uint32_t>(flags[4 * i + q]) << (8 * q);
      }
      if (ntok - 32 * i < 32) v &= (1u << (ntok - 32 * i)) - 1u;
    }
    reinterpret_cast<uint32_t *>(sl.fl)[i] = v;
    any |= v;
  }
  // a chunk without pointers is its payload: copy it straight out
  if (!__any_sync(kFull, any != 0)) {
    if (ntok != k || pay != bytes_c) {
      if (lane == 0) atomicOr(A.err, kErrCorrupt);
      return true;
    }
    if (sl.io) {
      copy_s2g(dst, payload, pay, lane);
    } else {
      for (uint32_t i = lane; i < pay; i += 32) dst[i] = payload[i];
    }
    return true;
  }
  const uint32_t pay_tok = pay - tail;  // the tokens' payload; the tail follows it
  // the tail bytes, read before the output image may grow over the record
  const uint8_t tb = lane < tail ? payload[pay_tok + lane] : 0;
  bool ok;
  __syncwarp();
  if (sl.io) {
    ok = decode_tokens_s<true>(h, payload, ntok, pay_tok, k, sl.io, true, sl, lane);
  } else {
    const bool aligned = A.out_aligned != 0 && (h.C % 4) == 0;
    ok = decode_tokens_s<false>(h, payload, ntok, pay_tok, k, dst, aligned, sl, lane);
  }
  if (!ok) {
    if (lane == 0) atomicOr(A.err, kErrCorrupt);
    return true;
  }
  uint8_t *ob = sl.io ? sl.io : dst;
  if (lane < tail) ob[static_cast<uint64_t>(k) * h.S + lane] = tb;
  if (sl.io && GLZ_OK(bytes_c + 16 <= sl.io_bytes && chunk_at + bytes_c <= A.out_cap)) {
    __syncwarp();
    copy_s2g(dst, sl.io, bytes_c, lane);
  }
  __syncwarp();
  return true;
}

// Per-warp slice for a stream with header h.
__device__ __forceinline__ DecodeLayout layout_of(const Header &h, uint64_t budget) {
  const uint64_t k = h.C / h.S;
  return decode_layout(k, h.C, decode_record_bound(k, h.S, h.offB, h.m), h.S == 1 && h.offB == 2,
                       h.S * h.m >= 1 + h.offB, budget);
}

}  // namespace

__global__ void __launch_bounds__(1024, 1) decompress_kernel(const DecompressArgs A) {
  extern __shared__ __align__(128) uint8_t smem[];
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t warp = threadIdx.x >> 5;
  const uint32_t wpb = blockDim.x >> 5;

  Header h;
  const bool ok = read_header(A.in, h);
  const bool leader = blockIdx.x == 0 && threadIdx.x == 0;
  if (!ok) {
    if (leader) atomicOr(A.err, kErrCorrupt);
    return;
  }
  if (h.n > A.out_cap) {
    if (leader) atomicOr(A.err, kErrSmall);
    return;
  }
  const uint64_t records_at = kHeaderBytes + 8ull * h.nc +
                              8ull * ((h.nc + kIndexStride - 1) / kIndexStride);
  if (records_at > A.in_bytes) {
    if (leader) atomicOr(A.err, kErrCorrupt);
    return;
  }
  if (leader) *A.out_bytes = h.n;
  // per-warp slice, decided from the header; warps that do not fit sit out
  const DecodeLayout L = layout_of(h, A.smem_bytes);
  const uint32_t fit = A.smem_bytes / L.per_warp;
  const uint32_t active = fit < wpb ? fit : wpb;
  if (warp >= active) return;
  Slice sl = make_slice(smem + static_cast<uint64_t>(warp) * L.per_warp, L,
                        h.S == 1 && h.offB == 2);
  if (lane == 0) {
    mbar_init(sl.bar, 1);
    fence_mbar_init();
  }
  __syncwarp();
  // chunks that do not fill the GPU spread over all SMs (block by block, 256
  // chunks ran on 8: 1 MiB took 34.8 us, 19.0 spread); more go block by block
  // (neighbouring chunks on one SM: 512 MiB of literal chunks 186 us, 190
  // spread)
  const uint32_t nwarps = gridDim.x * active;
  const uint32_t gw = h.nc < nwarps ? warp * gridDim.x + blockIdx.x : blockIdx.x * active + warp;
  for (uint32_t c = gw; c < h.nc; c += nwarps)
    if (!decode_chunk(A, h, c, records_at, sl, lane)) break;
  if (lane == 0) checked_fold(A.err);
}

// Batched decompression: chunks of all streams in order, grid-stride; each
// warp finds its stream by a 32-way search over the streams' first chunks.
__global__ void __launch_bounds__(1024, 1) decompress_batch_kernel(const DecompressBatchArgs B) {
  extern __shared__ __align__(128) uint8_t smem[];
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t warp = threadIdx.x >> 5;
  const uint32_t wpb = blockDim.x >> 5;
  if (blockIdx.x == 0) {  // zero-byte streams: check the header, size 0
    for (uint32_t i = threadIdx.x; i < B.n_empty; i += blockDim.x) {
      Header h;
      if (!read_header(B.empties[i].in, h) || h.n != 0) atomicOr(B.err, kErrCorrupt);
      *B.empties[i].out_bytes = 0;
    }
  }
  const uint32_t fit = B.smem_bytes / B.lay.per_warp;
  const uint32_t active = fit < wpb ? fit : wpb;
  if (warp >= active) return;
  // the slice covers every stream; the high-byte area exists when any needs it
  Slice base = make_slice(smem + static_cast<uint64_t>(warp) * B.lay.per_warp, B.lay, false);
  if (lane == 0) {
    mbar_init(base.bar, 1);
    fence_mbar_init();
  }
  __syncwarp();
  const uint64_t stride = static_cast<uint64_t>(gridDim.x) * active;
  // (few chunks spread over the SMs, as above)
  for (uint64_t g = B.total_chunks < stride ? static_cast<uint64_t>(warp) * gridDim.x + blockIdx.x
                                            : static_cast<uint64_t>(blockIdx.x) * active + warp;
       g < B.total_chunks;
       g += stride) {
    uint32_t lo = 0, hi = B.n_items;
    while (hi - lo > 1) {
      const uint32_t step = (hi - lo + 31) / 32;
      const uint32_t idx = lo + lane * step;
      const bool le = idx < hi && B.item_base[idx] <= g;
      const uint32_t cnt = __popc(__ballot_sync(kFull, le));
      const uint32_t nlo = lo + (cnt - 1) * step;
      hi = min(hi, nlo + step);
      lo = nlo;
    }
    const DecItem it = B.items[lo];
    const uint32_t c = static_cast<uint32_t>(g - it.gbase);
    Header h{};
    const bool ok = it.in_bytes >= kHeaderBytes && read_header(it.in, h);
    const uint64_t records_at = kHeaderBytes + 8ull * h.nc +
                                8ull * ((h.nc + kIndexStride - 1) / kIndexStride);
    // the header must still be the one the plan sized the slices for
    const uint64_t kh = ok ? h.C / h.S : 0;
    const bool need_hi = ok && h.S == 1 && h.offB == 2;
    // the io area: a stream whose pointers may outgrow their symbols needs
    // the output image and the record side by side
    auto fits_io = [](const DecodeLayout &L, const Header &hh, uint64_t kk) {
      const uint64_t c16 = ((hh.C + 15) & ~15ull) + 16;
      const uint64_t r16 = (decode_record_bound(kk, hh.S, hh.offB, hh.m) + 15) & ~15ull;
      const bool sh = hh.S * hh.m >= 1 + hh.offB;
      return (sh ? (c16 > r16 ? c16 : r16) : c16 + r16) + 32 + kIoSlack <= L.io_bytes;
    };
    const bool fits = ok && h.nc == it.nc && kh <= B.lay.mark_bytes &&
                      (!need_hi || B.lay.io_off - B.lay.hi_off >= kh) &&
                      (kh + 7) / 8 + 8 <= B.lay.flag_bytes &&
                      (!B.lay.staged || fits_io(B.lay, h, kh)) &&
                      records_at <= it.in_bytes && h.n <= it.out_cap;
    if (!fits) {
      if (lane == 0) atomicOr(B.err, h.n > it.out_cap && ok ? kErrSmall : kErrCorrupt);
      continue;
    }
    if (c == 0 && lane == 0) *it.out_bytes = h.n;
    DecompressArgs A{};
    A.in = it.in;
    A.in_bytes = it.in_bytes;
    A.out = it.out;
    A.out_cap = it.out_cap;
    A.out_bytes = it.out_bytes;
    A.err = B.err;
    A.out_aligned = static_cast<int>(it.out_aligned);
    base.hi = need_hi ? smem + static_cast<uint64_t>(warp) * B.lay.per_warp + B.lay.hi_off
                      : nullptr;
    if (!decode_chunk(A, h, c, records_at, base, lane)) break;
  }
  if (lane == 0) checked_fold(B.err);
}

cudaError_t launch_decompress_batch(DecompressBatchArgs B, int block, cudaStream_t stream) {
  static LaunchCache lc;
  const size_t smem = B.smem_bytes;
  int per_sm = 0, sms = 0;
  cudaError_t e = resident_blocks(lc, decompress_batch_kernel, block, smem, &per_sm, &sms);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const uint64_t warps = block / 32;
  uint64_t want = (B.total_chunks + warps - 1) / warps;
  if (want == 0) want = 1;
  const uint64_t cap = static_cast<uint64_t>(per_sm) * sms;
  const unsigned grid = static_cast<unsigned>(want < cap ? want : cap);
  decompress_batch_kernel<<<grid, block, smem, stream>>>(B);
  return cudaGetLastError();
}

cudaError_t launch_decompress(DecompressArgs A, int block, cudaStream_t stream) {
  static LaunchCache lc;
  const size_t smem = A.smem_bytes;
  int per_sm = 0, sms = 0;
  cudaError_t e = resident_blocks(lc, decompress_kernel, block, smem, &per_sm, &sms);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // enough blocks for the largest stream the input could hold, capped at the
  // resident limit (the grid cannot depend on the header: it is on the GPU)
  const uint64_t max_chunks = A.in_bytes / kTableEntry + 1;
  const uint64_t warps = block / 32;
  const uint64_t want = (max_chunks + warps - 1) / warps;
  const uint64_t cap = static_cast<uint64_t>(per_sm) * sms;
  const unsigned grid = static_cast<unsigned>(want < cap ? want : cap);
  decompress_kernel<<<grid, block, smem, stream>>>(A);
  return cudaGetLastError();
}

}  // namespace glz
