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

template <int S, int NW>
__global__ void __launch_bounds__(32 * kCoopWarps, NW <= 8 ? 3 : 2)
    compress_coop_kernel(const CompressArgs A) {
  using Sym = typename SymType<S>::T;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ BufDesc B;
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t s_ticket, s_totals;
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
      phase ^= 1u;
    }
    staged = __syncthreads_and(staged);
    if (!staged && threadIdx.x == 0) atomicOr(A.err, kErrTimeout);

    // 1. planes
    MaskParser<S, NW, true> P;
    P.inb = inb;
    P.k = k;
    P.lane = lane;
    P.planes = planes;
    P.rows = rows;
    P.find_varying_bits();
    for (uint32_t n = warp; n < nslab; n += kCoopWarps) P.make_slabs(n, false);
    __syncthreads();

    // 2. longest matches and the parse through each slab
    const bool overlap = B.match == kMatchOverlap;
    const uint32_t m = B.m, M = B.M, W = B.W, tsz = 1 + B.offB;
    const uint32_t r = 31 - lane;
    {
      const uint32_t per = (nslab + kCoopWarps - 1) / kCoopWarps;
      const uint32_t s1 = min(nslab, (warp + 1) * per);
      uint32_t made = warp * per;
#pragma unroll 1
      for (uint32_t s = warp * per; s < s1; ++s) {
#pragma unroll 1
        while (made < nslab && made < s + 2) P.make_slabs(made++, true);
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
      while (cur < k) {
        const uint32_t s = cur >> 5, tok = reach[cur];
        uint32_t next = leave[cur];
        if (lane == 0) toks[s] = tok;
        if (next & kOpen) {
          const uint32_t q = 32 * s + 31 - (__ffs(tok) - 1);
          uint32_t l, d;
          window_match<S, NW>(reinterpret_cast<const Sym *>(inb), k, B, q, lane, l, d);
          if (lane == 0) info[q] = l | (d << 8);
          next = q + l;
        }
        cur = next;
      }
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

    // 4. the record
    uint32_t ntok = s_totals & 0xFFFFu;
    const uint32_t np = s_totals >> 16;
    uint32_t pb = S * (ntok - np) + tsz * np + tail, fb = (ntok + 7) / 8;
    const bool stored = B.version == 2 && fb + pb >= bytes;  // the chunk as it is
    if (!stored) {
      const uint32_t earlier = lane == 31 ? 0u : kFull << (lane + 1);
      for (uint32_t s = warp; s < nslab; s += kCoopWarps) {
        const uint32_t tok = toks[s], ptr = tok & has[s], b = base[s];
        if (!((tok >> lane) & 1u)) continue;
        const bool is_ptr = (ptr >> lane) & 1u;
        const uint32_t t = (b & 0xFFFFu) + __popc(tok & earlier);
        const uint32_t q = (b >> 16) + __popc(ptr & earlier);
        const uint32_t p = 32 * s + r, po = S * (t - q) + tsz * q;
        uint32_t v = P.symbol(p);
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
    } else {
      ntok = 0;
      fb = 0;
      pb = bytes;
    }
    const uint64_t rec = static_cast<uint64_t>(fb) + pb;
    if (warp == 0) {
      if (c != 0) publish(A.status + B.gbase, c, kAgg, rec, lane);
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
      const uint8_t *from = stored ? inb : pay;
      const uint32_t part = (pb / kCoopWarps + 16) & ~15u;
      const uint32_t at = min(pb, warp * part), n = min(pb - at, part);
      if (n) warp_copy(o + fb + at, from + at, n, lane);
    }
    if (!staged) break;  // the barrier's phase is unknown
  }
  if (threadIdx.x == 0) checked_fold(A.err);
}

}  // namespace glz
