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
//            until it enters its piece; in a chunk whose codewords all have
//            one length, as in padding, the boundaries are known;
//   decode   each lane decodes from there to the end of its piece into its
//            column of a staging table, and notes where it left the piece
//            (its exit) and how many symbols it found;
//   check    a piece's true entry is the exit of the piece before it.  Lanes
//            whose guess was another one decode again from there, until
//            entries and exits agree all along every chunk: then, from each
//            chunk's first lane on, every entry is the true one.  At most as
//            many rounds as a chunk has pieces; nearly always none or one.  In
//            a run of one symbol nobody resynchronises: pieces that repeat
//            one codeword take their boundaries from where the run begins,
//            all at once, and need no decoding;
//   flush    a prefix sum of the counts places the lanes' symbols, which meet
//            in shared memory and leave in whole lines.
// Half of a tensor zeros (Student-t, Table 1, chunks of 4096): 1 Mi 103 -> 15 us,
// 16 Mi 156 -> 27; the second half of every chunk 1 Mi 56 -> 19; one chunk of zeros
// in 64 Mi 191 -> 74 (none: 74); 64 Mi equal symbols under ranks of other data 900
// -> 68, since runs are not corrected piece after piece.  What still does not
// resynchronise (sparse data, repeated patterns) is found by samples, and larger
// containers of it are decoded a lane per chunk (split_rule.cuh).
// A chunk is valid when its last piece ends at its last bit and its counts
// add up to its symbols, which is when decoding it serially ends at its last
// bit after that many symbols.
//
// One lane per chunk (decode.cu) issues fewer instructions per symbol, but a
// chunk is a chain of up to 4096 dependent steps (79 us) however few chunks
// there are, and a group occupies one warp.
#pragma once

#include "decode_common.cuh"
#include "split_rule.cuh"

namespace qlc {

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
constexpr int kRounds = 64;  // of corrections, twice as many as there can be
__device__ __forceinline__ uint32_t warm_bits(uint32_t len_lo, uint32_t len_hi) {
  return mixed_parity(len_lo, len_hi) ? kWarm : 2 * kWarm;
}

// A lane's piece: bits [beg, end) of the chunk [cb, ce), positions in the span's
// bits; piece number seg of the chunk.
struct Piece {
  uint32_t cb, ce, beg, end, seg;
};

// The first codeword boundary at or after `end`, from the boundary at.
__device__ __forceinline__ uint32_t walk_to(const uint32_t* bits, uint32_t at, uint32_t end, uint32_t len_lo,
                                            uint32_t len_hi) {
  uint32_t p[4];
  while (at < end) {
    four_ends(bits, at, len_lo, len_hi, p);
    at = p[0] >= end ? p[0] : p[1] >= end ? p[1] : p[2] >= end ? p[2] : p[3];
  }
  return at;
}

// Corrections (see decode_span).  A run of one symbol repeats its codeword: a
// reader that starts at a wrong bit stays on the wrong boundaries as long as the
// run lasts, and the true ones are known only from where the run begins.
//
// The period, up to kMaxCode, of the bits from the tenth bit of the piece to the
// tenth behind it, or to the chunk's end; 0 if they have none.  The first 32 bits
// rule nearly every piece out that is no run.
__device__ __forceinline__ uint32_t run_period(const uint32_t* bits, const Piece& pc) {
  const uint32_t from = pc.beg + kMaxCode - 1, to = min(pc.end + kMaxCode - 1, pc.ce);
  if (from + 32 + kMaxCode > to) return 0;  // hardly longer than what it would save
  const SpanBits w(bits, from);
  uint32_t period = 0;
#pragma unroll
  for (uint32_t p = kMaxCode; p > 0; p--) period = w.x == __funnelshift_l(w.y, w.x, p) ? p : period;
  if (period) {
    // bit t against bit t + period, the last one below the chunk's end
    const uint32_t stop = min(to, pc.ce - period);
    for (uint32_t t = from + 32; t < stop; t += 32) {
      const SpanBits v(bits, t);
      uint32_t differ = v.x ^ __funnelshift_l(v.y, v.x, period);
      if (stop - t < 32) differ >>= 32 - (stop - t);
      if (differ) return 0;
    }
  }
  return period;
}

// What a lane learns from a run that its piece goes on with from the piece
// before: its entry, and the run's codeword length and symbol.
struct Run {
  uint32_t entry, len, sym;  // len 0: no run
};

// Called by all lanes, with the boundary x that the piece before leaves to this
// one.  The boundaries of a run are those of its first piece.  A function of its
// own, so that its registers and code are not the decoder's (inlined it cost 3 %).
static __device__ __noinline__ Run follow_run(const uint32_t* bits, const uint8_t* T, Piece pc, bool mine, uint32_t x,
                                       uint32_t len_lo, uint32_t len_hi, int lane) {
  const uint32_t period = mine ? run_period(bits, pc) : 0u;
  if (!__any_sync(0xffffffffu, period != 0)) return {0u, 0u, 0u};
  const uint32_t period_before = __shfl_up_sync(0xffffffffu, period, 1);
  const bool goes_on = period != 0 && pc.seg != 0 && period_before == period;
  const uint32_t heads = ~__ballot_sync(0xffffffffu, goes_on);
  const int head = 31 - __clz(heads & (0xFFFFFFFFu >> (31 - lane)));
  // a boundary within the run, the length there and the symbol (of use in heads)
  uint32_t len = 0, sym = 0;
  if (period) {
    x = walk_to(bits, x, pc.beg + kMaxCode - 1, len_lo, len_hi);
    const SpanBits w(bits, x);
    len = code_len(w.x, len_lo, len_hi);
    const uint32_t code = __funnelshift_l(w.x, 0u, len);
    sym = QLC_GUARD(code < 2048u, nullptr) ? T[code] : 0u;
  }
  x = __shfl_sync(0xffffffffu, x, head);
  len = __shfl_sync(0xffffffffu, len, head);
  sym = __shfl_sync(0xffffffffu, sym, head);
  if (!goes_on || len % period != 0 || x > pc.beg) return {0u, 0u, 0u};
  return {x + (pc.beg - x + len - 1) / len * len, len, sym};
}

// Whether readers are slow to find the boundaries at sample i of a container: in
// a group's first chunk, somewhere, readers from three bits in a row have not met
// after `warm` bits.  A chunk of one codeword length has its boundaries known.
// Nothing is taken for granted of the container but its n_chunks and payload
// being inside it.  words: kSampleWords of shared memory.
constexpr uint32_t kSampleVecs = 5, kSampleWords = 4 * kSampleVecs + 1;
__device__ __forceinline__ bool sample_is_slow(const uint8_t* in, const SplitData& d, uint64_t n_chunks, uint32_t i,
                                               uint32_t* words) {
  const uint64_t n_groups = n_groups_of(n_chunks), g = i * n_groups / kSamples, first = g * kGroupChunks * d.cs;
  if (n_groups == 0 || first >= d.n) return false;
  const uint64_t goff = reinterpret_cast<const unsigned long long*>(in + kIndexOff)[g];
  const uint32_t bits = reinterpret_cast<const uint16_t*>(in + kIndexOff + 8 * n_groups)[g * kGroupChunks];
  const uint32_t nsym = (uint32_t)min((uint64_t)d.cs, d.n - first);
  bool even = false;
#pragma unroll
  for (int k = 0; k < 4; k++)
    even |= bits == nsym * (d.len_lo >> (8 * k) & 0xFFu) || bits == nsym * (d.len_hi >> (8 * k) & 0xFFu);
  if (even || bits < 128 * kSampleVecs) return false;
  const uint32_t v = (i * 0x9E3779B1u >> 16) % (bits / 128 - kSampleVecs + 1);
  if ((goff & 15u) != 0 || goff > d.payload_bytes || d.payload_bytes - goff < 16 * (v + kSampleVecs)) return false;
  const uint4* p = reinterpret_cast<const uint4*>(in + payload_start(n_chunks) + goff) + v;
#pragma unroll
  for (uint32_t k = 0; k < kSampleVecs; k++) {
    const uint4 q = ldg_nc_v4(p + k);
    words[4 * k] = bswap32(q.x);
    words[4 * k + 1] = bswap32(q.y);
    words[4 * k + 2] = bswap32(q.z);
    words[4 * k + 3] = bswap32(q.w);
  }
  const uint32_t end = warm_bits(d.len_lo, d.len_hi);
  uint32_t at[3] = {0, 1, 2}, e[4];  // side by side: a walk is a chain of latencies
  while (min(at[0], min(at[1], at[2])) < end) {
#pragma unroll
    for (int k = 0; k < 3; k++) {
      four_ends(words, at[k], d.len_lo, d.len_hi, e);
      const uint32_t to = e[0] >= end ? e[0] : e[1] >= end ? e[1] : e[2] >= end ? e[2] : e[3];
      at[k] = at[k] < end ? to : at[k];
    }
  }
  return at[0] != at[1] || at[0] != at[2];
}
static_assert((2 * kWarm + kMaxCode) / 32 + 2 < 4 * kSampleVecs, "readers stay within the sample");

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
  auto load_bits = [&]() {
    const uint4* gp = reinterpret_cast<const uint4*>(in + h.P + goff) + v0;
    for (uint32_t v = lane; v < nv; v += 32) {
      if (!QLC_GUARD(v < kSpanVecs && h.P + goff + 16 * (uint64_t)(v0 + v + 1) <= h.in_bytes, status)) continue;
      const uint4 q = ldg_nc_v4(gp + v);
      reinterpret_cast<uint4*>(sm.bits)[v] = make_uint4(bswap32(q.x), bswap32(q.y), bswap32(q.z), bswap32(q.w));
    }
  };
  load_bits();
  __syncwarp();
  const uint32_t cb = (mine ? E - B : S0) - 128u * v0;  // the chunk's first bit within sm.bits
  // Pieces of an odd number of words: lanes that have come equally far read 32
  // different banks (a stride of 27.4 words, for one, has four of them on one).
  const uint32_t B_max = __reduce_max_sync(0xffffffffu, B);
  const uint32_t piece = 32u * ((B_max + 32 * shape.lanes - 1) / (32 * shape.lanes) | 1u);
  const Piece pc = {cb, cb + B, cb + min(B, piece * seg), cb + min(B, piece * (seg + 1)), seg};
  const uint32_t beg = pc.beg, end = pc.end;
  const uint32_t len_lo = h.len_lo, len_hi = h.len_hi;
  uint32_t p[4];
  uint32_t entry = cb;
  if (mine && seg > 0) {
    const uint32_t len = code_len(SpanBits(sm.bits, cb).x, len_lo, len_hi);
    if (B == nsym * len) {  // codewords of one length, as in a chunk of one symbol
      entry = cb + (beg - cb + len - 1) / len * len;
    } else {
      if (beg > cb + warm) entry = beg - warm;
      entry = walk_to(sm.bits, entry, beg, len_lo, len_hi);
    }
  }
  uint32_t exit = cb, count = 0;
  bool again = mine, run = false;  // run: the piece is count times the symbol of run_word, and nothing is staged
  uint32_t run_word = 0;
  int round = 0;
  for (; round <= kRounds; round++) {
    if (again) {
      uint32_t n4 = 0, at = entry, last = entry;
      while (at < end && n4 < kStageWords) {
        last = at;
        sm.col[n4][lane] = four_symbols(sm.bits, at, T, len_lo, len_hi);
        n4++;
      }
      while (at < end) {  // more than the column holds: decoded again at the end
        last = at;
        four_symbols(sm.bits, at, T, len_lo, len_hi);
        n4++;
      }
      exit = at;
      count = 4 * n4;
      if (n4) {  // the last word may reach past the piece
        four_ends(sm.bits, last, len_lo, len_hi, p);
        exit = p[0] >= end ? p[0] : p[1] >= end ? p[1] : p[2] >= end ? p[2] : p[3];
        count -= (p[0] >= end) + (p[1] >= end) + (p[2] >= end);
      }
      run = false;
    }
    __syncwarp();
    const uint32_t before = __shfl_up_sync(0xffffffffu, exit, 1);
    again = mine && seg > 0 && before != entry;
    if (!__any_sync(0xffffffffu, again)) break;
    if (again) entry = before;
    if (round == 0) continue;  // nearly always all it takes
    const Run r = follow_run(sm.bits, T, pc, mine, entry, len_lo, len_hi, lane);
    if (r.len) {  // needs no decoding
      entry = r.entry;
      count = entry < end ? (end - entry + r.len - 1) / r.len : 0u;
      exit = entry + count * r.len;
      again = false;
      run = true;
      run_word = r.sym * 0x01010101u;
    }
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
  if (round > kRounds || __any_sync(0xffffffffu, bad)) {
    if (lane == 0) set_status(status, QLC_ERR_CORRUPT);
    return;
  }
  const uint64_t base = (g * kGroupChunks + c0) * h.cs;  // the span's first symbol
  const uint32_t total = __shfl_sync(0xffffffffu, upto, 31);
  // The symbols, shifted to their place.  A lane's first and last words may
  // be shared with its neighbours: they start from zero and are OR-ed.
  uint32_t* ow = sm.bits;
  auto slot = [](uint32_t i) { return mad_hi(i, 1u << 27, i); };  // i + i / 32
  const uint32_t w0 = off >> 2, nout = ((off & 3u) + count + 3) >> 2;
  const bool fits = QLC_GUARD(w0 + nout <= kSpanSyms / 4, status);
  __syncwarp();  // every lane is done with the bits
  if (nout && fits) ow[slot(w0)] = ow[slot(w0 + nout - 1)] = 0u;
  __syncwarp();
  const uint32_t nin = (count + 3) >> 2;
  auto place = [&](auto word) {  // word(i): the lane's word i
    const uint32_t sh = (off & 3u) * 8u;
    uint32_t prev = word(0u);
    const uint32_t head = prev << sh;
    uint32_t t = 1;
    for (; t + 1 < nout; t++) {
      const uint32_t cur = word(t);
      ow[slot(w0 + t)] = __funnelshift_l(prev, cur, sh);
      prev = cur;
    }
    // prev is word t - 1; the last output word holds the rest of it and, when
    // there is one, of word t
    const uint32_t tail = t < nin ? word(t) : 0u;
    const uint32_t keep = 0xFFFFFFFFu >> ((32u - 8u * (off + count)) & 31u);  // the bytes of the last output word
    if (nout == 1) {
      atomicOr(&ow[slot(w0)], head & keep);
    } else {
      atomicOr(&ow[slot(w0)], head);
      atomicOr(&ow[slot(w0 + nout - 1)], __funnelshift_l(prev, tail, sh) & keep);
    }
  };
  const uint32_t held = run ? 0u : kStageWords;  // words that are staged
  const bool unstaged = __any_sync(0xffffffffu, nin > held);
  if (unstaged) {
    if (nout && fits) place([&](uint32_t i) { return i < held ? sm.col[i][lane] : run_word; });
  } else if (nout && fits) {
    place([&](uint32_t i) { return sm.col[i][lane]; });
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
  // A piece with more symbols than its column holds (short codewords in a chunk
  // of long ones): the rest of them, byte by byte over what was written there.
  if (unstaged) {
    const bool rest = !run && count > 4 * kStageWords;
    if (!__any_sync(0xffffffffu, rest)) return;
    load_bits();
    __syncwarp();
    uint32_t at = entry;
    for (uint32_t i = 0; rest && i < count; i += 4) {
      const uint32_t w = four_symbols(sm.bits, at, T, len_lo, len_hi);
      if (i < 4 * kStageWords) continue;
      for (uint32_t b = 0; b < 4 && i + b < count; b++)
        if (QLC_GUARD(base + off + i + b < h.out_cap, status)) put1<kOut>(out, scales, base + off + i + b, w >> (8 * b) & 0xFFu);
    }
    __syncwarp();
  }
}

}  // namespace qlc
