// compress_coop.cuh -- compression of few chunks: one block of eight warps per
// chunk.
//
// With one warp per chunk (compress_impl.cuh) a launch takes at least the
// time of one chunk: about 1.5 us for a slab of 32 positions, 97 us for
// 4 KiB of 2-byte symbols, however many SMs are idle (1 MiB: 256 warps for 152
// SMs).  Here the warps of a block share the chunk's slabs:
//   1. planes of all slabs (mask_parse.cuh), the warps taking every eighth;
//   2. rows and longest matches, each warp a run of slabs; for every position
//      also the tokens that a parse from it visits in its slab and where it
//      leaves the slab;
//   3. one warp follows the parse from slab to slab, one load each, and scans
//      the slabs' token counts;
//   4. the tokens are written, each warp every eighth slab, beside the chunk
//      (over the planes), and the record copied out by all warps once the
//      look-back has its place.
// A match that runs on past the rows of step 2 is measured by step 3's warp
// from the symbols.  The total work per chunk is a little more than with one
// warp, so launches that fill the GPU with one warp per chunk stay there.
#pragma once

#include "compress_impl.cuh"

namespace glz {

// The literal pre-check of compress_impl.cuh (literal_chunk) by the whole
// block: true only when no position of the chunk can start a match of >= m
// symbols.  All keys are ORed into one Bloom filter of a word per position, in
// no order between warps, so of two positions with one key the one ORed later
// is flagged: a flagged position is checked exactly as the target of a match
// and as the source of one, over the whole window.  Every thread returns the
// same answer.  For each flagged position one more full scan than
// literal_chunk's, but about one chunk in two has none.
constexpr uint32_t kCoopMaxFlagged = 16;

template <int S>
__device__ __forceinline__ bool literal_chunk_block(const typename SymType<S>::T *sym, uint32_t k,
                                                    const BufDesc &B, uint32_t *bm,
                                                    uint32_t nwords, uint32_t *flagged,
                                                    uint32_t *count, uint32_t warp,
                                                    uint32_t lane) {
  for (uint32_t i = threadIdx.x; i < nwords / 4; i += blockDim.x)
    reinterpret_cast<uint4 *>(bm)[i] = make_uint4(0, 0, 0, 0);
  if (threadIdx.x == 0) *count = 0;
  __syncthreads();
  const uint8_t *in = reinterpret_cast<const uint8_t *>(sym);
  const uint32_t kb = S * min(B.m, 8u / S);  // key bytes, as in build_chains
  const uint32_t mlo = kb >= 4 ? kFull : (1u << (8 * kb)) - 1u;
  const uint32_t mhi = kb <= 4 ? 0u : (kb >= 8 ? kFull : (1u << (8 * (kb - 4))) - 1u);
  const volatile uint32_t *seen = count;
  for (uint32_t p0 = 32 * warp; p0 < k && *seen <= kCoopMaxFlagged; p0 += 32 * kCoopWarps) {
    const uint32_t p = p0 + lane;
    if (p + B.m > k) continue;
    uint32_t lo, hi;
    key_at<S>(in, p, mlo, mhi, lo, hi);
    const uint32_t h = ((hi * 0x85EBCA77u) ^ lo) * 0x9E3779B1u, g = h * 0xC2B2AE3Du;
    const uint32_t mask = (1u << (g >> 27)) | (1u << ((g >> 22) & 31u)) |
                          (1u << ((g >> 17) & 31u)) | (1u << ((g >> 12) & 31u));
    const uint32_t at = __umulhi(h, nwords);
    if (GLZ_OK(at < nwords) && (atomicOr(&bm[at], mask) & mask) == mask) {
      const uint32_t i = atomicAdd(count, 1u);
      if (i < kCoopMaxFlagged) flagged[i] = p;
    }
  }
  __syncthreads();
  const uint32_t n = *count;
  bool hit = n > kCoopMaxFlagged;
  if (!hit) {
    for (uint32_t i = warp; i < n && !hit; i += kCoopWarps) {
      const uint32_t p = flagged[i];
      hit = match_near<S>(sym, k, B, p, p + 1, lane);  // p as the target
      bool eq_any = false;                             // p as the source
      const uint32_t end = min(k, p + B.W + 1);
      for (uint32_t q = p + 1 + lane; q < end; q += 32) {
        bool eq = (q - p >= B.m || B.match == kMatchOverlap) && q + B.m <= k;
        for (uint32_t x = 0; eq && x < B.m; ++x) eq = sym[q + x] == sym[p + x];
        eq_any |= eq;
      }
      hit |= __any_sync(kFull, eq_any) != 0;
    }
  }
  return !__syncthreads_or(hit);
}

template <int S, int NW>
__global__ void __launch_bounds__(32 * kCoopWarps, NW <= 8 ? 3 : 2)
    compress_coop_kernel(const CompressArgs A) {
  using Sym = typename SymType<S>::T;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ BufDesc B;
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t s_ticket, s_totals, s_flagged[kCoopMaxFlagged], s_count;
  __shared__ uint8_t *s_out;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const CoopSmem &L = A.coop;
  uint8_t *inb = smem, *pay = smem + L.planes_off;
  uint32_t *planes = reinterpret_cast<uint32_t *>(smem + L.planes_off);
  uint32_t *rows = reinterpret_cast<uint32_t *>(smem + L.rows_off + warp * mask_rows_bytes(NW, 1));
  uint32_t *info = reinterpret_cast<uint32_t *>(smem + L.info_off);    // length | offset << 8
  uint32_t *reach = reinterpret_cast<uint32_t *>(smem + L.reach_off);  // tokens of the slab
  uint16_t *leave = reinterpret_cast<uint16_t *>(smem + L.leave_off);  // position after it
  uint32_t *has = reinterpret_cast<uint32_t *>(smem + L.slab_off);     // per slab: matches,
  uint32_t *toks = has + L.slabs, *base = toks + L.slabs;  // token starts, counts before it
  uint32_t *flags = reinterpret_cast<uint32_t *>(smem + L.flags_off);
  constexpr uint32_t kOpen = 0x8000;  // in `leave`: the last match is not finished
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
    if (!A.items) B = A.buf;
  }
  uint32_t phase = 0;
  bool try_literal = true;  // the block's previous chunk was all literals
  const uint64_t end_ticket = A.items ? A.total_chunks : A.end_chunk;
  while (true) {
    __syncthreads();
    if (threadIdx.x == 0) s_ticket = atomicAdd(A.ticket, 1u) + A.first_ticket;
    __syncthreads();
    const uint32_t g = s_ticket;
    if (g >= end_ticket) break;
    if (A.items) {
      if (warp == 0) {
        const uint32_t item = find_item(A, g, lane);
        if (lane < sizeof(BufDesc) / 4)
          reinterpret_cast<uint32_t *>(&B)[lane] =
              reinterpret_cast<const uint32_t *>(A.items + item)[lane];
      }
      __syncthreads();
    }
    const uint32_t c = static_cast<uint32_t>(g - B.gbase);
    if (c == 0 && warp == 0) write_header(B, lane);

    // stage the chunk
    const uint64_t chunk_at = static_cast<uint64_t>(c) * B.C;
    const uint32_t bytes = (c + 1 < B.nc) ? B.C : static_cast<uint32_t>(B.n - chunk_at);
    const uint32_t k = bytes / S, tail = bytes - k * S, nslab = (k + 31) / 32;
    const uint8_t *src = B.in + chunk_at;
    const uint32_t bulk = B.in_aligned ? (bytes & ~15u) : 0u;
    if (bulk && threadIdx.x == 0) {
      fence_proxy_async_smem();
      mbar_arrive_expect_tx(&bar, bulk);
      bulk_g2s(inb, src, bulk, &bar);
    }
    for (uint32_t i = bulk + threadIdx.x; i < bytes; i += blockDim.x) inb[i] = src[i];
    for (uint32_t i = threadIdx.x; i < nslab; i += blockDim.x) {
      flags[i] = 0;
      toks[i] = 0;
    }
    bool staged = true;
    if (bulk) {
      staged = mbar_wait_bounded(&bar, phase, A.spin_limit);
      // a copy given up may still write the chunk: it is waited for (bounded
      // again) before the block moves on to leave
      if (!staged) mbar_wait_bounded(&bar, phase);
      phase ^= 1u;
    }
    staged = __syncthreads_and(staged);
    if (!staged && threadIdx.x == 0) atomicOr(A.err, kErrTimeout);

    // A chunk that was not staged is not parsed (its symbols may change under
    // the parse): it is published as literals and nothing of it is placed.
    // (The pre-check is tried after a chunk without pointers, as with one warp
    // per chunk; the filter takes the place of `info`.)
    const bool literal =
        !staged ||
        (try_literal && literal_chunk_block<S>(reinterpret_cast<const Sym *>(inb), k, B, info,
                                               32 * nslab, s_flagged, &s_count, warp, lane));
    const bool overlap = B.match == kMatchOverlap;
    const uint32_t m = B.m, M = B.M, W = B.W, tsz = 1 + B.offB;
    const uint32_t r = 31 - lane;
    if (!literal) {
      // 1. planes
      MaskParser<S, NW, true> P;
      P.inb = inb;
      P.k = k;
      P.lane = lane;
      P.planes = planes;
      P.rows = rows;
      P.find_varying_bits();
      for (uint32_t n = warp; n < nslab; n += kCoopWarps) P.template make_slabs<false>(n);
      __syncthreads();

      // 2. longest matches and the parse through each slab
      {
        const uint32_t per = (nslab + kCoopWarps - 1) / kCoopWarps;
        const uint32_t s1 = min(nslab, (warp + 1) * per);
        uint32_t made = warp * per;
#pragma unroll 1
        for (uint32_t s = warp * per; s < s1; ++s) {
#pragma unroll 1
          while (made < nslab && made < s + 2) P.template make_slabs<true>(made++);
          const uint32_t p = 32 * s + r;
          uint32_t a[NW], len, off;
          bool open;
          longest_match(P, p, r, 0, m, M, W, overlap, a, len, off, open);
          const uint32_t step = len ? len : 1u;
          uint32_t tok, last;
          parse_from_every_lane(step, lane, tok, last);
          const uint32_t out = 32 * s + 31 - last + __shfl_sync(kFull, step, last);
          const uint32_t any = __ballot_sync(kFull, len != 0);
          const uint32_t opened = __ballot_sync(kFull, open);
          if (p < k) {
            info[p] = len | (off << 8);
            reach[p] = tok;
            leave[p] = static_cast<uint16_t>(out | ((opened >> last) & 1u ? kOpen : 0u));
          }
          if (lane == 0) has[s] = any;
        }
      }
      __syncthreads();

      // 3. the parse from slab to slab; token and pointer counts before each
      if (warp == 0) {
        uint32_t cur = 0;
        bool stuck = false;
        while (cur < k) {
          const uint32_t s = cur >> 5, tok = reach[cur];
          uint32_t next = leave[cur];
          if (lane == 0) toks[s] = tok;
          if (next & kOpen) {
            const uint32_t q = 32 * s + 31 - (__ffs(tok) - 1);
            uint32_t l, d;
            window_match<S, NW>(reinterpret_cast<const Sym *>(inb), k, B, q, lane, l, d);
            if (lane == 0) info[q] = l | (d << 8);
            // The parse always moves on.  An empty match here, which the rows
            // rule out, is reported after the loop: with the report inside it,
            // or a look at the rows' own length, the whole kernel was up to 9 %
            // slower (95,020 bytes of codes, S = 2, C = 16384, W = 64: 80 us
            // against 74).
            stuck |= l == 0;
            next = q + (l != 0 ? l : 1);
          }
          cur = next;
        }
        if (stuck && lane == 0) atomicOr(A.err, kErrInternal);
        __syncwarp();
        uint32_t before = 0;  // tokens | pointers << 16
        for (uint32_t b0 = 0; b0 < nslab; b0 += 32) {
          const uint32_t s = b0 + lane;
          uint32_t t = 0, x = 0;
          if (s < nslab) {
            t = toks[s];
            if (k - 32 * s < 32) t &= kFull << (32 - (k - 32 * s));
            toks[s] = t;
            x = __popc(t) | (__popc(t & has[s]) << 16);
          }
          uint32_t total;
          const uint32_t excl = warp_excl_scan(x, lane, total);
          if (s < nslab) base[s] = before + excl;
          before += total;
        }
        if (lane == 0) s_totals = before;
      }
      __syncthreads();

    }

    // 4. the record
    uint32_t ntok = literal ? k : s_totals & 0xFFFFu;
    const uint32_t np = literal ? 0u : s_totals >> 16;
    try_literal = np == 0;
    uint32_t pb = S * (ntok - np) + tsz * np + tail, fb = (ntok + 7) / 8;
    const bool stored = B.version == 2 && fb + pb >= bytes;  // the chunk as it is
    if (stored) {
      ntok = 0;
      fb = 0;
      pb = bytes;
    }
    const uint64_t rec = static_cast<uint64_t>(fb) + pb;
    // (published before the record is written, so that later chunks wait less)
    if (c != 0 && warp == 0) publish(A.status + B.gbase, c, kAgg, rec, lane);
    if (!stored && !literal) {
      const uint32_t earlier = lane == 31 ? 0u : kFull << (lane + 1);
      for (uint32_t s = warp; s < nslab; s += kCoopWarps) {
        const uint32_t tok = toks[s], ptr = tok & has[s], b = base[s];
        if (!((tok >> lane) & 1u)) continue;
        const bool is_ptr = (ptr >> lane) & 1u;
        const uint32_t t = (b & 0xFFFFu) + __popc(tok & earlier);
        const uint32_t q = (b >> 16) + __popc(ptr & earlier);
        const uint32_t p = 32 * s + r, po = S * (t - q) + tsz * q;
        uint32_t v = reinterpret_cast<const Sym *>(inb)[p];
        if (is_ptr) {
          const uint32_t x = info[p];
          v = (x & 0xFFu) | (((x >> 8) - 1) << 8);
          if (GLZ_OK(t < 32 * L.slabs)) atomicOr(&flags[t >> 5], 1u << (t & 31));
        }
        const uint32_t n = is_ptr ? tsz : S;
        if (!GLZ_OK(po + n <= S * k)) continue;
        uint8_t *o = pay + po;
        if (S != 1 && tsz == 2) {  // every token is a whole number of 16-bit words
          *reinterpret_cast<uint16_t *>(o) = static_cast<uint16_t>(v);
          if (S == 4 && !is_ptr)
            *reinterpret_cast<uint16_t *>(o + 2) = static_cast<uint16_t>(v >> 16);
        } else {
#pragma unroll
          for (uint32_t i = 0; i < (S > 3 ? S : 3); ++i)
            if (i < n) o[i] = static_cast<uint8_t>(v >> (8 * i));
        }
      }
      if (threadIdx.x < tail) pay[pb - tail + threadIdx.x] = inb[k * S + threadIdx.x];
    }
    if (warp == 0) {
      uint8_t *tab = B.out + kHeaderBytes + static_cast<uint64_t>(kTableEntry) * c;
      if (lane < 4) tab[lane] = static_cast<uint8_t>(ntok >> (8 * lane));
      else if (lane < 8) tab[lane] = static_cast<uint8_t>(pb >> (8 * (lane - 4)));
      uint64_t excl;
      const bool ok = lookback_wait(A.status + B.gbase, c, lane, A.err, excl, A.spin_limit);
      uint8_t *o = place_meta(A, B, c, excl, rec, staged && ok, lane);
      if (lane == 0) s_out = o;
    }
    __syncthreads();
    if (uint8_t *o = s_out) {
      if (warp == 0 && fb) warp_copy(o, reinterpret_cast<const uint8_t *>(flags), fb, lane);
      const uint8_t *from = stored || literal ? inb : pay;
      const uint32_t part = (pb / kCoopWarps + 16) & ~15u;
      const uint32_t at = min(pb, warp * part), n = min(pb - at, part);
      if (n) warp_copy(o + fb + at, from + at, n, lane);
    }
    if (!staged) break;  // the barrier's phase is unknown
  }
  if (threadIdx.x == 0) checked_fold(A.err);
}

}  // namespace glz
