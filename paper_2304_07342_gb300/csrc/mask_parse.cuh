// mask_parse.cuh -- the greedy parse of one chunk by equality masks (one
// warp), for windows of at most 32 * NW symbols.
//
// For every position p the warp forms the bit mask E(p) over the window:
// bit d - 1 is set when symbol p equals symbol p - d (d = 1 .. W).  A match
// of length l at p from offset d exists exactly when bit d - 1 is set in
// E(p), E(p + 1), .., E(p + l - 1), so the longest match is found by ANDing
// masks until nothing is left, and the nearest offset among the longest is
// the lowest set bit of the last non-zero AND.  Length <= offset (section
// 3.3.2) clears bit l - 1 and those below before a match may reach l + 1.
//
// Masks come from bit planes.  Symbols of a slab (32 positions) are written
// as Gray codes, whose neighbours differ in one bit, so codes around a mean
// vary in few bits; the bits that vary inside the chunk (`act`) are taken in
// groups of eight, and one ballot per bit gives the plane word of the slab.
// A lane's 32 comparisons with a slab are then one three-input logic
// instruction per plane: acc &= ~(plane ^ my bit).  Lane i holds position
// 31 - i of the slab, so that a plane word lists the slab's positions from
// the last to the first: in the words of slab s, s - 1, s - 2, .. bit
// 32 t + i is position 32 s + 31 - 32 t - i, and shifting them right by
// lane + 1 puts offset d at bit d - 1.
//
// What bounds it: instruction issue.  The hash chains this replaces took
// 20 of 32 lanes and one dependent shared-memory load per hop; here every
// instruction of the mask and match steps runs on all lanes and the loads
// are broadcasts or 16-byte rows.  The work per position grows with the
// window's words and with the bits that vary in the chunk, up to four groups of
// planes for 4-byte symbols, and hardly with the matches: where symbols seldom
// repeat, the chains cost less and a sample of the data sends the launch there
// (sample.cuh).
#pragma once

#include <cstdint>

#include "glz_common.h"
#include "glz_device.cuh"

namespace glz {

template <int S>
struct SymType;
template <>
struct SymType<1> {
  using T = uint8_t;
};
template <>
struct SymType<2> {
  using T = uint16_t;
};
template <>
struct SymType<4> {
  using T = uint32_t;
};

// Number of words of a vectorised row access.
template <int NW>
__device__ __forceinline__ void load_row(const uint32_t *row, uint32_t (&v)[NW]) {
  if constexpr (NW == 1) {
    v[0] = row[0];
  } else if constexpr (NW == 2) {
    const uint2 t = *reinterpret_cast<const uint2 *>(row);
    v[0] = t.x;
    v[1] = t.y;
  } else {
#pragma unroll
    for (int j = 0; j < NW; j += 4) {
      const uint4 t = *reinterpret_cast<const uint4 *>(row + j);
      v[j] = t.x;
      v[j + 1] = t.y;
      v[j + 2] = t.z;
      v[j + 3] = t.w;
    }
  }
}

template <int NW>
__device__ __forceinline__ void store_row(uint32_t *row, const uint32_t (&v)[NW]) {
  if constexpr (NW == 1) {
    row[0] = v[0];
  } else if constexpr (NW == 2) {
    *reinterpret_cast<uint2 *>(row) = make_uint2(v[0], v[1]);
  } else {
#pragma unroll
    for (int j = 0; j < NW; j += 4)
      *reinterpret_cast<uint4 *>(row + j) = make_uint4(v[j], v[j + 1], v[j + 2], v[j + 3]);
  }
}

template <int NW>
__device__ __forceinline__ bool any_bit(const uint32_t (&v)[NW]) {
  uint32_t o = 0;
#pragma unroll
  for (int j = 0; j < NW; ++j) o |= v[j];
  return o != 0;
}

// Clears the bits of offsets up to `l` (the first l bits).
template <int NW>
__device__ __forceinline__ void drop_offsets(uint32_t (&v)[NW], uint32_t l) {
#pragma unroll
  for (int j = 0; j < NW; ++j) {
    const uint32_t at = 32u * j;
    if (l >= at + 32) v[j] = 0;
    else if (l > at) v[j] &= kFull << (l - at);
  }
}

// 1 + index of the lowest set bit of v (v has one).
template <int NW>
__device__ __forceinline__ uint32_t lowest_bit(const uint32_t (&v)[NW]) {
  uint32_t w = v[NW - 1], at = 32 * (NW - 1);
#pragma unroll
  for (int j = NW - 2; j >= 0; --j)
    if (v[j]) {
      w = v[j];
      at = 32 * j;
    }
  return at + __ffs(w);
}

// The bits in which the k symbols of a staged chunk differ, as Gray codes (one
// warp).
template <int S>
__device__ __forceinline__ uint32_t varying_bits(const uint8_t *inb, uint32_t k, uint32_t lane) {
  using Sym = typename SymType<S>::T;
  constexpr uint32_t kBelow = S == 1 ? 0x7F7F7F7Fu : S == 2 ? 0x7FFF7FFFu : 0x7FFFFFFFu;
  auto gray = [](uint32_t v) { return v ^ ((v >> 1) & kBelow); };  // of every symbol in v
  const uint32_t first = reinterpret_cast<const Sym *>(inb)[0];
  const uint32_t g0 = gray(S == 1 ? first * 0x01010101u : S == 2 ? first * 0x00010001u : first);
  const uint32_t words = k * S / 4, quads = words / 4;  // whole words of symbols
  uint32_t d = 0;
#pragma unroll 1
  for (uint32_t i = lane; i < quads; i += 32) {
    const uint4 v = reinterpret_cast<const uint4 *>(inb)[i];
    d |= (gray(v.x) ^ g0) | (gray(v.y) ^ g0) | (gray(v.z) ^ g0) | (gray(v.w) ^ g0);
  }
  if (lane < words - 4 * quads)
    d |= gray(reinterpret_cast<const uint32_t *>(inb)[4 * quads + lane]) ^ g0;
  if constexpr (S < 4) {
    const uint32_t p = words * (4 / S) + lane;  // symbols after the last whole word
    const uint32_t one = S == 1 ? 0xFFu : 0xFFFFu;
    if (p < k) d |= (gray(reinterpret_cast<const Sym *>(inb)[p]) ^ g0) & one;
  }
  if constexpr (S == 1) d |= d >> 16, d |= d >> 8, d &= 0xFFu;
  if constexpr (S == 2) d |= d >> 16, d &= 0xFFFFu;
  return __reduce_or_sync(kFull, d);
}

// WHOLE: planes of every slab of the chunk are kept, else of the last 2 * NW.
// COUNT: slabs made at a time; two share the plane words of the slabs before
// them and the work around them (windows of 512 keep one: four slabs of their
// rows would take the shared memory of three warps in thirteen).
template <int S, int NW, bool WHOLE = false>
struct MaskParser {
  static constexpr int COUNT = WHOLE ? 1 : mask_slabs_made(NW);
  using Sym = typename SymType<S>::T;
  static constexpr uint32_t kPlanes = mask_plane_words(S);  // plane words per slab
  static constexpr uint32_t kRing = NW > 1 ? 2 * NW : 4;    // slabs of planes kept
  static constexpr uint32_t kRows = 64 * COUNT;             // rows kept: two slabs, or four
  static constexpr uint32_t kPart = NW < 4 ? NW : 4;        // words of a row side by side

  const uint8_t *inb;
  uint32_t k, act, ngroups, lane;
  uint32_t lift0[8];  // the first eight varying bits, see next_lifts
  uint32_t *planes, *rows;

  // Plane words of slab n - t (any slab's when it lies before the chunk).
  __device__ __forceinline__ uint32_t *slab_planes(uint32_t n, uint32_t t) const {
    if constexpr (WHOLE) return planes + (t <= n ? n - t : 0u) * kPlanes;
    else return planes + ((n - t) & (kRing - 1)) * kPlanes;
  }

  __device__ __forceinline__ uint32_t symbol(uint32_t p) const {
    return p < k ? static_cast<uint32_t>(reinterpret_cast<const Sym *>(inb)[p]) : 0u;
  }

  __device__ __forceinline__ void find_varying_bits() {
    act = varying_bits<S>(inb, k, lane);
    ngroups = (__popc(act) + 7) / 8;
    uint32_t rest = act;
    next_lifts(rest, lift0);
  }

  // The next eight set bits of `rest`: factors that lift each to bit 31 (0
  // when none is left).
  static __device__ __forceinline__ void next_lifts(uint32_t &rest, uint32_t (&lift)[8]) {
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const uint32_t low = rest & (0u - rest);
      lift[b] = low ? 1u << __clz(low) : 0u;
      rest &= rest - 1u;
    }
  }

  // Planes FIRST .. FIRST + N - 1 of a group of eight of slabs n .. n + COUNT
  // - 1: the plane words go to the ring, and acc[c][t] keeps the bits of slab
  // n + c - t whose symbols agree with this lane's in slab n + c.  (A lane's
  // bit as a mask comes from a multiplication and an arithmetic shift:
  // selected by a predicate, the compiler turned each logic instruction below
  // into two.)
  template <int FIRST, int N, bool ROWS>
  __device__ __forceinline__ void some_planes(uint32_t n, uint32_t group,
                                              const uint32_t (&g)[COUNT],
                                              const uint32_t (&lift)[8],
                                              uint32_t (&acc)[COUNT][NW + 1]) const {
    static_assert(N == 2 || N == 4, "one vector store");
    const uint32_t at = 8 * group + FIRST;
    uint32_t my[COUNT][N], own[COUNT][N];
#pragma unroll
    for (int c = 0; c < COUNT; ++c) {
#pragma unroll
      for (int b = 0; b < N; ++b) {
        const int32_t t = static_cast<int32_t>(g[c] * lift[FIRST + b]);
        own[c][b] = __ballot_sync(kFull, t < 0);
        my[c][b] = static_cast<uint32_t>(t >> 31);
      }
      if (lane == 0) store_row<N>(slab_planes(n + c, 0) + at, own[c]);
    }
    if constexpr (!ROWS) return;
#pragma unroll
    for (int c = 0; c < COUNT; ++c)
#pragma unroll
      for (int o = 0; o <= c; ++o)
#pragma unroll
        for (int b = 0; b < N; ++b) acc[c][c - o] &= ~(own[o][b] ^ my[c][b]);
#pragma unroll
    for (int t = 1; t <= NW; ++t) {
      uint32_t x[N];
      load_row<N>(slab_planes(n, t) + at, x);
#pragma unroll
      for (int c = 0; c < COUNT; ++c)
        if (t + c <= NW)
#pragma unroll
          for (int b = 0; b < N; ++b) acc[c][t + c] &= ~(x[b] ^ my[c][b]);
    }
  }

  template <bool ROWS>
  __device__ __forceinline__ void plane_group(uint32_t n, uint32_t group,
                                              const uint32_t (&g)[COUNT],
                                              const uint32_t (&lift)[8],
                                              uint32_t (&acc)[COUNT][NW + 1]) const {
    some_planes<0, 4, ROWS>(n, group, g, lift, acc);
    // (codes around a mean vary in 5 to 7 Gray bits: the last pair is often idle)
    if (lift[4]) some_planes<4, 2, ROWS>(n, group, g, lift, acc);
    if (lift[6]) some_planes<6, 2, ROWS>(n, group, g, lift, acc);
  }

  // Planes of slabs n .. n + COUNT - 1, and with ROWS the masks E(p) of their
  // positions (for the full 32 * NW offsets; the window is applied by the
  // reader).
  template <bool ROWS>
  __device__ __forceinline__ void make_slabs(uint32_t n) const {
    __syncwarp();  // rows and planes of the slabs these replace have been read
    const uint32_t p = 32 * n + 31 - lane;
    uint32_t g[COUNT], acc[COUNT][NW + 1];
#pragma unroll
    for (int c = 0; c < COUNT; ++c) {
      const uint32_t v = symbol(p + 32 * c);
      g[c] = v ^ (v >> 1);
#pragma unroll
      for (int t = 0; t <= NW; ++t) acc[c][t] = kFull;
    }
    if (ngroups) plane_group<ROWS>(n, 0, g, lift0, acc);
    if (ngroups > 1) {
      uint32_t rest = act, lift[8];
      next_lifts(rest, lift);
#pragma unroll 1
      for (uint32_t group = 1; group < ngroups; ++group) {
        next_lifts(rest, lift);
        plane_group<ROWS>(n, group, g, lift, acc);
      }
    }
    if constexpr (ROWS) {
      if (n < NW) {  // slabs before the chunk
#pragma unroll
        for (int c = 0; c < COUNT; ++c)
#pragma unroll
          for (int t = 1; t <= NW; ++t)
            if (static_cast<uint32_t>(t) > n + c) acc[c][t] = 0;
      }
#pragma unroll
      for (int c = 0; c < COUNT; ++c) {
        uint32_t e[NW];
#pragma unroll
        for (int j = 0; j < NW; ++j) e[j] = __funnelshift_rc(acc[c][j], acc[c][j + 1], lane + 1);
        set_row(p + 32 * c, e);
      }
    }
    __syncwarp();
  }

  // E(p), a position of the last two slabs made with rows.  Rows of more than
  // four words are split into parts of 16 bytes, part-major: neighbouring
  // lanes then read neighbouring 16 bytes (whole rows of 32 and 64 bytes put
  // the lanes of a 16-byte access 2 and 4 deep on the same banks).
  __device__ __forceinline__ void row(uint32_t p, uint32_t (&e)[NW]) const {
    const uint32_t *at = rows + (p & (kRows - 1)) * kPart;
    if constexpr (NW <= 4) {
      load_row<NW>(at, e);
    } else {
#pragma unroll
      for (int j = 0; j < NW; j += 4) {
        const uint4 t = *reinterpret_cast<const uint4 *>(at + j * kRows);
        e[j] = t.x;
        e[j + 1] = t.y;
        e[j + 2] = t.z;
        e[j + 3] = t.w;
      }
    }
  }
  // Word j of E(p).
  __device__ __forceinline__ uint32_t row_word(uint32_t p, uint32_t j) const {
    const uint32_t at = (p & (kRows - 1)) * kPart;
    return rows[NW <= 4 ? at + j : at + (j & ~3u) * kRows + (j & 3u)];
  }
  __device__ __forceinline__ void set_row(uint32_t p, const uint32_t (&e)[NW]) const {
    uint32_t *at = rows + (p & (kRows - 1)) * kPart;
    if constexpr (NW <= 4) {
      store_row<NW>(at, e);
    } else {
#pragma unroll
      for (int j = 0; j < NW; j += 4)
        *reinterpret_cast<uint4 *>(at + j * kRows) = make_uint4(e[j], e[j + 1], e[j + 2], e[j + 3]);
    }
  }
  __device__ __forceinline__ void and_row(uint32_t p, uint32_t (&a)[NW]) const {
    uint32_t e[NW];
    row(p, e);
#pragma unroll
    for (int j = 0; j < NW; ++j) a[j] &= e[j];
  }
};

// The longest match of the position p of this lane (place r of its slab) when
// p >= from: its length (0: none of m symbols) and nearest offset; a = the
// offsets that match over that length.  `open`: it still matches at the last
// row kept and may be longer.
template <int S, int NW, bool WHOLE>
__device__ __forceinline__ void longest_match(const MaskParser<S, NW, WHOLE> &P, uint32_t p,
                                              uint32_t r, uint32_t cur, uint32_t m, uint32_t M,
                                              uint32_t W, bool overlap, uint32_t (&a)[NW],
                                              uint32_t &len, uint32_t &off, bool &open) {
  const uint32_t k = P.k;
  len = 0;
  off = 0;
  open = false;
  P.row(p, a);
  if (W != 32u * NW) {
#pragma unroll
    for (int j = 0; j < NW; ++j)
      a[j] &= W >= 32u * (j + 1) ? kFull : W <= 32u * j ? 0u : (1u << (W - 32u * j)) - 1u;
  }
  if (m >= 2) P.and_row(p + 1, a);
  if (m >= 3) P.and_row(p + 2, a);
#pragma unroll 1
  for (uint32_t l = 3; l < m; ++l) P.and_row(p + l, a);
  if (!overlap) a[0] &= kFull << (m - 1);
  if (p >= cur && p + m <= k && any_bit<NW>(a)) {
    const uint32_t lim = min(M, k - p), stop = min(lim, 64 - r), stop0 = min(stop, 32u);
    uint32_t l = m;
    bool more = true;
#pragma unroll 1
    while (l < stop0) {
      uint32_t e[NW];
      P.row(p + l, e);
#pragma unroll
      for (int j = 0; j < NW; ++j) e[j] &= a[j];
      if (!overlap) e[0] &= kFull << l;
      if (!any_bit<NW>(e)) {
        more = false;
        break;
      }
#pragma unroll
      for (int j = 0; j < NW; ++j) a[j] = e[j];
      ++l;
    }
#pragma unroll 1
    while (more && l < stop) {
      uint32_t e[NW];
      P.row(p + l, e);
      drop_offsets<NW>(e, overlap ? 0u : l);
#pragma unroll
      for (int j = 0; j < NW; ++j) e[j] &= a[j];
      if (!any_bit<NW>(e)) {
        more = false;
        break;
      }
#pragma unroll
      for (int j = 0; j < NW; ++j) a[j] = e[j];
      ++l;
    }
    len = l;
    off = lowest_bit<NW>(a);
    open = more && l < lim;
  }
}

// The greedy parse of a slab from each of its positions: `tok` = the lanes
// of the token starts it visits, `last` = the lane of the last of them.  A
// lane's successor is the lane of the next token start (itself when that lies
// past the slab); joining the sets reached by the successors, twice as far
// each time, takes five rounds of two shuffles (following one pointer after
// the other took 20 instructions each).
__device__ __forceinline__ void parse_from_every_lane(uint32_t step, uint32_t lane, uint32_t &tok,
                                                      uint32_t &last) {
  last = step <= lane ? lane - step : lane;
  tok = 1u << lane;
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    tok |= __shfl_sync(kFull, tok, last);
    last = __shfl_sync(kFull, last, last);
  }
}

// The greedy parse (section 2.2 steps 1-6) of the staged chunk of k symbols
// and the record it gives: the flags are left in `flags`, the payload (and a
// stream-version-2 tail) over the staged chunk itself, which is unchanged
// when the parse has no pointer (np == 0: the record is k literals).  In
// place because S * m >= 1 + offB (the caller's condition): a token's payload
// never starts after its own input, a literal's ends with it, and a
// pointer's ends before the next token's input; pointer payloads are at most
// three bytes, so no symbol beyond the next slab is touched, whose planes are
// made before the slab's tokens are written.  Requires m <= 32 and
// W <= 32 * NW.
//
// The rows of slabs s and s + 1 are kept: a match that starts in slab s is followed
// through slab s + 1 by its own lane.  A longer one that the parse takes is
// left open: its offsets wait in one more row, and the whole warp follows it
// through the slabs after s + 1 as they are made.  It covers every position
// before them, so the rows given up are not asked for again.
template <int S, int NW>
__device__ __forceinline__ void mask_parse(uint8_t *inb, uint32_t k, uint32_t tail,
                                           const BufDesc &B, uint32_t *planes, uint32_t *rows,
                                           uint32_t *flags, uint32_t flag_bytes, uint32_t lane,
                                           uint32_t &ntok_out, uint32_t &pay_out,
                                           uint32_t &nptr_out) {
  const bool overlap = B.match == kMatchOverlap;
  const uint32_t tsz = 1 + B.offB, m = B.m, M = B.M, W = B.W, nslab = (k + 31) / 32;
  for (uint32_t i = lane; i < nslab; i += 32)
    if (GLZ_OK(4 * i + 4 <= flag_bytes)) flags[i] = 0;
  MaskParser<S, NW> P;
  P.inb = inb;
  P.k = k;
  P.lane = lane;
  P.planes = planes;
  P.rows = rows;
  P.find_varying_bits();
  const uint32_t earlier = lane == 31 ? 0u : kFull << (lane + 1);  // lanes of earlier positions
  const uint32_t r = 31 - lane;           // this lane's place in a slab
  uint32_t made = 0;                      // slabs whose planes exist
  uint32_t cur = 0;                       // next position to parse
  uint32_t pbase = 0, tbase = 0, np = 0;  // payload bytes, tokens, pointers so far
  // a pointer whose match is still open: its position (or kNone), the length
  // so far, the place of its payload bytes
  constexpr uint32_t kNone = kFull;
  uint32_t long_p = kNone, long_len = 0, long_at = 0;
#pragma unroll 1
  for (uint32_t s = 0; s < nslab; ++s) {
#pragma unroll 1
    while (made < nslab && made < s + 2) {
      P.template make_slabs<true>(made);  // (also inside a long match: rare)
      made += P.COUNT;
    }
    if (long_p != kNone) {
      // the open match, through the rows of slabs s and s + 1: lane j < NW
      // holds word j of its offsets (each lane holding all words took a
      // hundred instructions a symbol at 16 words: 32 MiB of zero words,
      // W = 512, 2,780 us, 758 so)
      const uint32_t lim = min(M, k - long_p), stop = min(lim, 32 * made - long_p);
      const uint32_t word = min(lane, static_cast<uint32_t>(NW - 1));
      uint32_t b = lane < NW ? rows[P.kRows * NW + word] : 0u;
      bool more = true;
#pragma unroll 1
      while (long_len < stop) {
        uint32_t e = P.row_word(long_p + long_len, word) & b;
        if (!overlap) {  // offsets up to the length drop out
          const uint32_t gone = long_len > 32 * word ? min(long_len - 32 * word, 32u) : 0u;
          e &= __funnelshift_lc(0u, kFull, gone);
        }
        more = __any_sync(kFull, e != 0);
        if (!more) break;
        b = e;
        ++long_len;
      }
      cur = long_p + long_len;
      if (more && long_len < lim) {  // still open
        __syncwarp();
        if (lane < NW) rows[P.kRows * NW + word] = b;
        __syncwarp();
        continue;
      }
      const uint32_t at = __ffs(__ballot_sync(kFull, b != 0)) - 1;
      const uint32_t low = 32 * at + __ffs(__shfl_sync(kFull, b, at));  // its nearest offset
      const uint32_t v = long_len | ((low - 1) << 8);
      if (lane < tsz && GLZ_OK(long_at + lane < S * k))
        inb[long_at + lane] = static_cast<uint8_t>(v >> (8 * lane));
      long_p = kNone;
    }
    if (cur >= 32 * (s + 1)) continue;  // the slab lies inside a pointer
    const uint32_t p = 32 * s + r;

    uint32_t a[NW], len, off;
    bool open;
    longest_match(P, p, r, cur, m, M, W, overlap, a, len, off, open);

    // the parse through the slab from `cur`
    const uint32_t has = __ballot_sync(kFull, len != 0), opened = __ballot_sync(kFull, open);
    const uint32_t step = len ? len : 1u;
    uint32_t tok, last;
    parse_from_every_lane(step, lane, tok, last);
    tok = __shfl_sync(kFull, tok, 31 - (cur - 32 * s));
    const uint32_t ptr = tok & has;
    const uint32_t lv = __ffs(tok) - 1;  // lane of the last token
    if ((opened >> lv) & 1u) {
      // longer than the rows kept: its offsets wait in the spare row
      if (lane == lv) store_row<NW>(rows + P.kRows * NW, a);
      long_p = 32 * s + 31 - lv;
      long_len = __shfl_sync(kFull, len, lv);
      cur = 32 * (s + 1);
    } else {
      cur = 32 * s + 31 - lv + __shfl_sync(kFull, step, lv);
    }
    if (k - 32 * s < 32) tok &= kFull << (32 - (k - 32 * s));


    // the slab's tokens: payload offsets and token indices by popcounts over
    // the slab (the local prefix sum of section 3.2.2).  Until the first
    // pointer the payload is the input itself.
    if (np | ptr) {
      const bool is_tok = (tok >> lane) & 1u, is_ptr = (ptr >> lane) & 1u;
      const uint32_t t = __popc(tok & earlier), pb = __popc(ptr & earlier);
      const uint32_t po = pbase + S * (t - pb) + tsz * pb;
      const uint32_t v = is_ptr ? len | ((off - 1) << 8) : P.symbol(p);
      __syncwarp();  // every read of the slab before any write (in place)
      if (is_tok && GLZ_OK(po + (is_ptr ? tsz : S) <= S * k)) {
        uint8_t *o = inb + po;
        if (S != 1 && tsz == 2) {  // every token is a whole number of 16-bit words
          *reinterpret_cast<uint16_t *>(o) = static_cast<uint16_t>(v);
          if (S == 4 && !is_ptr)
            *reinterpret_cast<uint16_t *>(o + 2) = static_cast<uint16_t>(v >> 16);
        } else {
          const uint32_t n = is_ptr ? tsz : S;
#pragma unroll
          for (uint32_t i = 0; i < (S > 3 ? S : 3); ++i)
            if (i < n) o[i] = static_cast<uint8_t>(v >> (8 * i));
        }
      }
      if (long_p == p) long_at = po;
      if (long_p != kNone) long_at = __shfl_sync(kFull, long_at, 31 - (long_p & 31));
      if (is_ptr) {
        const uint32_t ti = tbase + t;
        if (GLZ_OK(4 * (ti >> 5) + 4 <= flag_bytes)) atomicOr(&flags[ti >> 5], 1u << (ti & 31));
      }
    }
    const uint32_t nt = __popc(tok), nptr = __popc(ptr);
    pbase += S * (nt - nptr) + tsz * nptr;
    tbase += nt;
    np += nptr;
  }
  __syncwarp();
  const uint8_t tb = lane < tail ? inb[k * S + lane] : 0;
  __syncwarp();
  if (lane < tail) inb[pbase + lane] = tb;
  __syncwarp();
  ntok_out = tbase;
  pay_out = pbase;
  nptr_out = np;
}

}  // namespace glz
