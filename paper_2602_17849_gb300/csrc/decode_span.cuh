// decode_span.cuh -- the split decoder (Section 7): a warp decodes a span of
// consecutive chunks of one group, up to 4096 symbols, with every lane on a
// piece of its own of about 128 symbols.
//
// The codes are not self-synchronising, but they resynchronise quickly: a
// reader that starts at a wrong bit soon lands on a true codeword boundary
// and stays on the true boundaries from there.  So
//   load     the span's bits go to shared memory, byte-swapped;
//   guess    each lane but a chunk's first starts kWarm bits before its piece
//            and steps over codewords (the 3-bit area code fixes the length)
//            until it enters its piece;
//   decode   each lane decodes from there to the end of its piece into its
//            column of a staging table, and notes where it left the piece
//            (its exit) and how many symbols it found;
//   check    a piece's true entry is the exit of the piece before it.  Lanes
//            whose guess was another one decode again from there, until
//            entries and exits agree all along every chunk: then, from each
//            chunk's first lane on, every entry is the true one.  At most as
//            many rounds as a chunk has pieces; nearly always none or one;
//   flush    a prefix sum of the counts places the lanes' symbols, which meet
//            in shared memory and leave in whole lines.
// A chunk is valid when its last piece ends at its last bit and its counts
// add up to its symbols, which is when decoding it serially ends at its last
// bit after that many symbols.
//
// One lane per chunk (decode.cu) issues fewer instructions per symbol, but a
// chunk is a chain of up to 4096 dependent steps (79 us) however few chunks
// there are, and a group occupies one warp.
#pragma once

#include "decode_common.cuh"

namespace qlc {

constexpr int kSpanCtasPerSm = 5;                     // resident: bounded by shared memory
constexpr uint32_t kSpanSyms = 32 * kPiece;           // symbols per warp at most
constexpr uint32_t kSpanVecs = (127 + kSpanSyms * kMaxCode + 127) / 128;  // 16-byte vectors that hold a span's bits
constexpr uint32_t kSpanWords = 4 * kSpanVecs + 4;    // and words read past the end (never consumed)
constexpr uint32_t kStageWords = 38;                  // staged words (4 symbols each) per lane
constexpr uint32_t kOutWords = kSpanSyms / 4 + kSpanSyms / 128;  // output words, one more after every 32
static_assert(kOutWords <= kSpanWords, "the output words take the place of the span's bits");

struct SpanWarp {
  __align__(16) uint32_t bits[kSpanWords];  // the span's bits; later its symbols, word i at i + i / 32
  uint32_t col[kStageWords][32];              // word k of lane l at col[k][l]
};
// The 64 bits of a span from bit p on: x the first 32, y the next.  Four
// codewords take at most 44, so one read of three words serves four of them;
// keeping a running window instead costs a test and several moves every two.
struct SpanBits {
  uint32_t x, y;
  __device__ __forceinline__ SpanBits(const uint32_t* bits, uint32_t p) {
    const uint32_t j = p >> 5;
    const bool ok = QLC_GUARD(j + 2 < kSpanWords, nullptr);
    const uint32_t w0 = ok ? bits[j] : 0u, w1 = ok ? bits[j + 1] : 0u, w2 = ok ? bits[j + 2] : 0u;
    x = __funnelshift_l(w1, w0, p);
    y = __funnelshift_l(w2, w1, p);
  }
};

// The ends p[0..3] of the four codewords from bit at on.
__device__ __forceinline__ void four_ends(const uint32_t* bits, uint32_t at, uint32_t len_lo, uint32_t len_hi,
                                          uint32_t (&p)[4]) {
  const SpanBits w(bits, at);
  const uint32_t la = code_len(w.x, len_lo, len_hi);
  const uint32_t lab = la + code_len(w.x << la, len_lo, len_hi);
  const uint32_t x = __funnelshift_l(w.y, w.x, lab);
  const uint32_t lc = code_len(x, len_lo, len_hi);
  const uint32_t lcd = lc + code_len(x << lc, len_lo, len_hi);
  p[0] = at + la;
  p[1] = at + lab;
  p[2] = p[1] + lc;
  p[3] = p[1] + lcd;
}

// The four symbols from bit p on, packed, the first lowest; p moves past them.
__device__ __forceinline__ uint32_t four_symbols(const uint32_t* bits, uint32_t& p, const uint8_t* T, uint32_t len_lo,
                                                 uint32_t len_hi) {
  auto symbol = [&](uint32_t x, uint32_t len) {  // of the codeword of len bits at the top of x
    const uint32_t i = __funnelshift_l(x, 0u, len);
    return QLC_GUARD(i < 2048u, nullptr) ? (uint32_t)T[i] : 0u;
  };
  const SpanBits w(bits, p);
  const uint32_t la = code_len(w.x, len_lo, len_hi);
  const uint32_t xb = w.x << la;
  const uint32_t lb = code_len(xb, len_lo, len_hi);
  const uint32_t xc = __funnelshift_l(w.y, w.x, la + lb);
  const uint32_t lc = code_len(xc, len_lo, len_hi);
  const uint32_t xd = xc << lc;
  const uint32_t ld = code_len(xd, len_lo, len_hi);
  p += la + lb + (lc + ld);
  const uint32_t ab = mad_lo(symbol(xb, lb), 256u, symbol(w.x, la));
  const uint32_t cd = mad_lo(symbol(xd, ld), 256u, symbol(xc, lc));
  return __byte_perm(ab, cd, 0x5410);
}

// Bits of warm-up before a piece.  Under Table 1 a reader is on the true
// boundaries after 37 codewords (264 bits) in 99.7 % of cases.  A scheme whose
// lengths are all even but the last area's keeps a wrong parity until such a
// code comes by, and gets twice as much (Table 2: 99 %).
constexpr uint32_t kWarm = 264;
__device__ __forceinline__ bool mixed_parity(uint32_t len_lo, uint32_t len_hi) {
  return ((len_lo | (len_hi & 0xFFFFFFu)) & 0x01010101u) != 0;
}
__device__ __forceinline__ uint32_t warm_bits(uint32_t len_lo, uint32_t len_hi) {
  return mixed_parity(len_lo, len_hi) ? kWarm : 2 * kWarm;
}

// Whether to decode a container split, where `total` symbols are decoded in
// this launch.  A lane per chunk takes at least the time of its chain, about 19
// us per 1024 symbols of chunk, and hardly more up to 40 Mi symbols; split, the
// time goes with the size, and is longer where readers are slow to find the
// true boundaries: in schemes of one parity, and in streams of mostly the
// shortest codeword.  Measured (us, split / lane per chunk): chunk 4096,
// Student-t 1 Mi 15 / 79, 16 Mi 27 / 80, 64 Mi 72 / 85, half zeros under Table 2
// 43 Mi 77 / 81; chunk 2048, Student-t 32 Mi 43 / 53, half zeros under Table 2
// 16 Mi 40 / 45, 32 Mi 58 / 53; chunk 1024, Student-t 8 Mi 19 / 27, 16 Mi 29 /
// 31, 32 Mi 44 / 33, half zeros 8 Mi 25 / 27, 16 Mi 39 / 31; chunk 512,
// Student-t 2 Mi 15 / 17, 8 Mi 19.1 / 18.4, half zeros 2 Mi 19 / 17.  Values:
// chunk 4096, fp32, half zeros 29 Mi 70 / 109; chunk 1024, bf16, Student-t 8 Mi
// 25 / 31, 12 Mi 37 / 33, 16 Mi 40 / 36, half zeros 8 Mi 29 / 31, 16 Mi 46 / 36;
// chunk 2048, bf16, Student-t 24 Mi 52 / 58, fp32, half zeros 19 Mi 63 / 58; chunk 4096, bf16, Student-t 47 Mi 83
// / 105, 48 Mi 98 / 105, 60 Mi 121 / 109.
// Hence the lines, proportional to the chunk; and streams of hardly anything
// but the shortest codeword (fewer than 1/32 bit per symbol above it) never,
// since they do not find the boundaries from a wrong phase, and their pieces
// are corrected one after the other (64 Mi equal symbols 1216 us).
template <int kOut>
__device__ __forceinline__ bool split_pays(const DecHeader& h, uint64_t total) {
  const uint64_t bits = 8 * h.payload_bytes, least = h.n * (h.len_lo & 0xFFu);
  const uint64_t excess = bits > least ? bits - least : 0;
  const bool fast = mixed_parity(h.len_lo, h.len_hi) && excess >= h.n / 16 * 7;
  const uint64_t cs = h.cs, line = (cs << 13) + (cs << 12);
  const uint64_t values = cs < 1024 ? cs << 12 : min(line, (cs << 14) + (cs << 12) - (12u << 20));
  const uint64_t slow = (kOut == kOutCodes ? line : (cs << 13) + (cs << 11)) - (3ull << 20);
  const uint64_t most = fast ? (cs < 512 ? 0 : kOut == kOutCodes ? cs << 14 : values) : cs < 1024 ? 0 : slow;
  return excess >= h.n / 32 && total <= most;
}

// Decodes a span of a validated container: chunks c0 .. c0 + shape.chunks - 1
// of group g.  One warp; k and seg are the lane's chunk in the span and its
// piece of the chunk.
template <int kOut>
__device__ __forceinline__ void decode_span(const DecHeader& h, const SpanShape& shape, const uint8_t* __restrict__ in,
                                            void* __restrict__ out, const float* __restrict__ scales, uint64_t g,
                                            uint32_t c0, uint32_t k, uint32_t seg, SpanWarp& sm, const uint8_t* T,
                                            uint32_t warm, uint32_t* status, int lane) {
  const unsigned long long* group_off = reinterpret_cast<const unsigned long long*>(in + kIndexOff);
  const uint16_t* chunk_bits = reinterpret_cast<const uint16_t*>(in + kIndexOff + 8 * h.n_groups);
  const uint64_t cg = g * kGroupChunks + lane;
  const uint32_t cbits =
      cg < h.n_chunks && QLC_GUARD(kIndexOff + 8 * h.n_groups + 2 * (cg + 1) <= h.in_bytes, status) ? chunk_bits[cg] : 0u;
  const uint64_t goff = QLC_GUARD(kIndexOff + 8 * (g + 1) <= h.in_bytes, status) ? group_off[g] : 0ull;
  const uint64_t gnext = g + 1 < h.n_groups
                             ? (QLC_GUARD(kIndexOff + 8 * (g + 2) <= h.in_bytes, status) ? group_off[g + 1] : 0ull)
                             : h.payload_bytes;
  uint32_t incl = cbits;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const uint32_t gbits = __shfl_sync(0xffffffffu, incl, 31);
  const bool group_ok = (g != 0 || goff == 0) && (goff & 15u) == 0 && goff <= gnext && gnext <= h.payload_bytes &&
                        gnext - goff == align16((gbits + 7u) / 8u);
  // this lane's chunk and piece
  const uint32_t ck = min(c0 + k, kGroupChunks - 1);
  const uint64_t c = g * kGroupChunks + ck;
  const bool mine = k < shape.chunks && c0 + k < kGroupChunks && c < h.n_chunks;
  const uint32_t nsym = mine ? (uint32_t)min((uint64_t)h.cs, h.n - c * h.cs) : 0u;
  const uint32_t ck_bits = __shfl_sync(0xffffffffu, cbits, ck);
  const uint32_t E = __shfl_sync(0xffffffffu, incl, ck);  // the chunk's end within the group
  const uint32_t B = mine ? ck_bits : 0u;
  // a chunk of nsym codewords has at most kMaxCode bits for each, which
  // bounds the span's bits
  if (!group_ok || __any_sync(0xffffffffu, mine && B > kMaxCode * nsym)) {
    if (lane == 0) set_status(status, QLC_ERR_CORRUPT);
    return;
  }
  if (!__any_sync(0xffffffffu, mine)) return;  // past a last group's chunks
  const uint32_t S0 = __shfl_sync(0xffffffffu, E - B, 0);  // the span's first bit
  const uint32_t E0 = __reduce_max_sync(0xffffffffu, mine ? E : 0u);
  const uint32_t v0 = S0 >> 7, nv = (E0 + 127) / 128 - v0;
  {
    const uint4* gp = reinterpret_cast<const uint4*>(in + h.P + goff) + v0;
    for (uint32_t v = lane; v < nv; v += 32) {
      if (!QLC_GUARD(v < kSpanVecs && h.P + goff + 16 * (uint64_t)(v0 + v + 1) <= h.in_bytes, status)) continue;
      const uint4 q = ldg_nc_v4(gp + v);
      reinterpret_cast<uint4*>(sm.bits)[v] = make_uint4(bswap32(q.x), bswap32(q.y), bswap32(q.z), bswap32(q.w));
    }
  }
  __syncwarp();
  const uint32_t cb = (mine ? E - B : S0) - 128u * v0;  // the chunk's first bit within sm.bits
  // Pieces of an odd number of words: lanes that have come equally far read 32
  // different banks (a stride of 27.4 words, for one, has four of them on one).
  const uint32_t B_max = __reduce_max_sync(0xffffffffu, B);
  const uint32_t piece = 32u * ((B_max + 32 * shape.lanes - 1) / (32 * shape.lanes) | 1u);
  const uint32_t beg = cb + min(B, piece * seg), end = cb + min(B, piece * (seg + 1));
  const uint32_t len_lo = h.len_lo, len_hi = h.len_hi;
  uint32_t p[4];
  uint32_t entry = cb;
  if (mine && seg > 0) {
    if (beg > cb + warm) entry = beg - warm;
    while (entry < beg) {
      four_ends(sm.bits, entry, len_lo, len_hi, p);
      entry = p[0] >= beg ? p[0] : p[1] >= beg ? p[1] : p[2] >= beg ? p[2] : p[3];
    }
  }
  uint32_t exit = cb, count = 0;
  bool again = mine;
  while (true) {
    if (again) {
      uint32_t n4 = 0, at = entry, last = entry;
      while (at < end) {
        last = at;
        const uint32_t w = four_symbols(sm.bits, at, T, len_lo, len_hi);
        if (n4 < kStageWords) sm.col[n4][lane] = w;
        n4++;
      }
      exit = at;
      count = 4 * n4;
      if (n4) {  // the last word may reach past the piece
        four_ends(sm.bits, last, len_lo, len_hi, p);
        exit = p[0] >= end ? p[0] : p[1] >= end ? p[1] : p[2] >= end ? p[2] : p[3];
        count -= (p[0] >= end) + (p[1] >= end) + (p[2] >= end);
      }
    }
    __syncwarp();
    const uint32_t before = __shfl_up_sync(0xffffffffu, exit, 1);
    again = mine && seg > 0 && before != entry;
    if (!__any_sync(0xffffffffu, again)) break;
    if (again) entry = before;
  }
  // positions of the lanes' symbols within the span
  uint32_t off = count;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, off, o);
    if (lane >= o) off += t;
  }
  const uint32_t upto = off;  // counts up to and with this lane
  off -= count;
  const uint32_t chunk_off = __shfl_sync(0xffffffffu, off, lane - (int)seg);
  const bool bad = mine && seg == shape.lanes - 1 && (exit != cb + B || upto - chunk_off != nsym);
  if (__any_sync(0xffffffffu, bad)) {
    if (lane == 0) set_status(status, QLC_ERR_CORRUPT);
    return;
  }
  const uint64_t base = (g * kGroupChunks + c0) * h.cs;  // the span's first symbol
  const uint32_t total = __shfl_sync(0xffffffffu, upto, 31);
  if (__any_sync(0xffffffffu, count > 4 * kStageWords)) {
    // a piece with more symbols than its column holds (a run of short codes
    // in a chunk of long ones): symbol by symbol, straight to the output
    if (mine) {
      uint32_t at = entry;
      for (uint32_t i = 0; i < count; i++) {
        const SpanBits w(sm.bits, at);
        const uint32_t la = code_len(w.x, len_lo, len_hi), ia = __funnelshift_l(w.x, 0u, la);
        const uint32_t sym = QLC_GUARD(ia < 2048u, nullptr) ? T[ia] : 0u;
        at += la;
        if (QLC_GUARD(base + off + i < h.out_cap, status)) put1<kOut>(out, scales, base + off + i, sym);
      }
    }
    __syncwarp();
    return;
  }
  // The symbols, shifted to their place.  A lane's first and last words may
  // be shared with its neighbours: they start from zero and are OR-ed.
  uint32_t* ow = sm.bits;
  auto slot = [](uint32_t i) { return mad_hi(i, 1u << 27, i); };  // i + i / 32
  const uint32_t w0 = off >> 2, nout = ((off & 3u) + count + 3) >> 2;
  const bool fits = QLC_GUARD(w0 + nout <= kSpanSyms / 4, status);
  __syncwarp();  // every lane is done with the bits
  if (nout && fits) ow[slot(w0)] = ow[slot(w0 + nout - 1)] = 0u;
  __syncwarp();
  if (nout && fits) {
    const uint32_t sh = (off & 3u) * 8u, nin = (count + 3) >> 2;
    uint32_t prev = sm.col[0][lane];
    uint32_t tail = prev;  // the last staged word
    uint32_t t = 1;
    for (; t + 1 < nout; t++) {
      const uint32_t cur = sm.col[t][lane];
      ow[slot(w0 + t)] = __funnelshift_l(prev, cur, sh);
      prev = cur;
    }
    // prev is word t - 1; the last output word holds the rest of it and, when
    // there is one, of word t
    tail = t < nin ? sm.col[t][lane] : 0u;
    const uint32_t keep = 0xFFFFFFFFu >> ((32u - 8u * (off + count)) & 31u);  // the bytes of the last output word
    const uint32_t head = sm.col[0][lane] << sh;
    if (nout == 1) {
      atomicOr(&ow[slot(w0)], head & keep);
    } else {
      atomicOr(&ow[slot(w0)], head);
      atomicOr(&ow[slot(w0 + nout - 1)], __funnelshift_l(prev, tail, sh) & keep);
    }
  }
  __syncwarp();
  if (kOut == kOutCodes && total == kSpanSyms && QLC_GUARD(base + kSpanSyms <= h.out_cap, status)) {
    // word 4 lane + m of the k-th 512 bytes sits in bank 4 lane + m + lane / 8: no two lanes share one
    uint4* dst = reinterpret_cast<uint4*>(static_cast<uint8_t*>(out) + base) + lane;
    const uint32_t* src = ow + slot(4 * lane);
#pragma unroll
    for (int q = 0; q < (int)kSpanSyms / 512; q++)
      st_cs_v4(dst + 32 * q, make_uint4(src[132 * q], src[132 * q + 1], src[132 * q + 2], src[132 * q + 3]));
  } else {
    for (uint32_t i = lane; i < (total + 3) / 4; i += 32) {
      const uint32_t v = ow[slot(i)];
      const uint64_t at = base + 4 * i;
      if (4 * i + 4 <= total) {
        if (QLC_GUARD(at + 4 <= h.out_cap, status)) put4<kOut>(out, scales, at, v);
      } else {
        for (uint32_t b = 0; b < total - 4 * i; b++)
          if (QLC_GUARD(at + b < h.out_cap, status)) put1<kOut>(out, scales, at + b, (v >> (8 * b)) & 0xFFu);
      }
    }
  }
  __syncwarp();
}

}  // namespace qlc
