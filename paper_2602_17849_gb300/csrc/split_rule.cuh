// split_rule.cuh -- when a container is decoded split (decode_span.cuh) and when
// a lane per chunk (decode.cu).  One rule for single containers, for the shards
// of a batch and for the plan of a batch; host and device.
#pragma once

#include "qlc_common.cuh"

namespace qlc {

constexpr uint32_t kSamples = 32;  // places looked at, see sample_is_slow

// What is decoded: one container to codes or to values, or a batch to codes.
enum SplitInto { kSplitCodes = 0, kSplitValues = 1, kSplitBatch = 2 };

// What the rule looks at: the header's chunk size, code lengths (len_lo, len_hi:
// of areas 0-3 and 4-7, one byte each), symbols and payload.
struct SplitData {
  uint32_t cs, len_lo, len_hi;
  uint64_t n, payload_bytes;
};

// Reads them, and the number of chunks, from a container's first 64 bytes (16-byte
// aligned).  False for a container that the decoder refuses: else the lengths are
// 3 to 11 bits, the chunk size is one and index and payload are inside in_bytes.
__host__ __device__ inline bool split_data(const uint8_t* hdr, uint64_t in_bytes, SplitData* d, uint64_t* n_chunks) {
  const uint32_t b_lo = *reinterpret_cast<const uint32_t*>(hdr + 40), b_hi = *reinterpret_cast<const uint32_t*>(hdr + 44);
  d->cs = *reinterpret_cast<const uint32_t*>(hdr + 16);
  d->len_lo = b_lo + 0x03030303u;
  d->len_hi = b_hi + 0x03030303u;
  d->n = *reinterpret_cast<const unsigned long long*>(hdr + 8);
  d->payload_bytes = *reinterpret_cast<const unsigned long long*>(hdr + 48);
  *n_chunks = *reinterpret_cast<const uint32_t*>(hdr + 20);
  const uint64_t P = payload_start(*n_chunks);
  const uint32_t wide = (b_lo + 0x07070707u) | (b_hi + 0x07070707u);  // a width above 8 sets one of its upper four bits
  return ((b_lo | b_hi) & 0xF0F0F0F0u) == 0 && (wide & 0xF0F0F0F0u) == 0 && chunk_symbols_ok(d->cs) && P <= in_bytes &&
         d->payload_bytes <= in_bytes - P;
}

// Whether the lengths below the last area's are not all even.
__host__ __device__ inline bool mixed_parity(uint32_t len_lo, uint32_t len_hi) {
  return ((len_lo | (len_hi & 0xFFFFFFu)) & 0x01010101u) != 0;
}

// Bits of the payload above those of the shortest codewords alone.  (Per symbol:
// Table 1, Student-t 0.86, normal 0.62, half zeros 0.06 to 0.45; Table 2, 3.0, 2.8
// and 1.1 to 1.5.)
__host__ __device__ inline uint64_t excess_bits(const SplitData& d) {
  const uint64_t bits = 8 * d.payload_bytes, least = d.n * (d.len_lo & 0xFFu);
  return bits > least ? bits - least : 0;
}
// Whether readers may be slow to find the boundaries in many places: most
// codewords are near the shortest length.
__host__ __device__ inline bool split_unsure(const SplitData& d) {
  return excess_bits(d) < (mixed_parity(d.len_lo, d.len_hi) ? d.n / 16 * 9 : 2 * d.n);
}

// The most symbols decoded in one launch for which splitting pays; slow: of
// kSamples samples, in data that is unsure.
// A lane per chunk takes at least the time of its chain, about 19 us per 1024
// symbols of chunk, and hardly more up to 40 Mi symbols; split, the time goes
// with the size, and with how often pieces are corrected.
// Measured on 152 SMs (us, split / lane per chunk), no slow places: chunk 4096,
// Student-t 1 Mi 15 / 79, 16 Mi 31 / 80, 64 Mi 74 / 85; chunk 2048, 32 Mi 43 /
// 53; chunk 1024, 8 Mi 19 / 27, 16 Mi 31 / 31; chunk 512, 2 Mi 15 / 17, 8 Mi 19 /
// 18.  Values: chunk 1024, bf16, 8 Mi 25 / 31, 12 Mi 37 / 33; chunk 2048, bf16,
// 24 Mi 52 / 58; chunk 4096, fp32, 40 Mi 83 / 107, bf16, 47 Mi 83 / 105, 60 Mi
// 121 / 109.  One parity, or up to a quarter of slow places: chunk 4096, Table 2,
// normal 40 Mi 62 / 81, a fifth nonzero 16 Mi 50 / 79, 45 Mi 90 / 81; chunk 1024,
// half zeros 8 Mi 25 / 27.  More (chunk 4096): the second half of every chunk
// zeros, 13 of 32, 16 Mi 45 / 78, 45 Mi 92 / 78; a twentieth nonzero, 26 of 32,
// 16 Mi 70 / 79, 45 Mi 141 / 79; a hundredth, 31 of 32, 1 Mi 125 / 74.
// Hence lines proportional to the chunk, less what a launch takes in any case.  A
// batch is split with more to do besides (headers, tables and barriers for every
// four spans): 40 shards, chunk 4096, 40 Mi 72 / 82, 50 Mi 83 / 84, chunk 2048, 12 Mi
// 40 / 47, 24 Mi 53 / 49, chunk 1024, 2 Mi 29 / 31, 6 Mi 33 / 31, chunk 512, 2 Mi 29 /
// 23; 300 shards, chunk 4096, 40 Mi 82 / 84, chunk 2048, 12 Mi 48 / 49.
__host__ __device__ inline uint64_t split_most(const SplitData& d, SplitInto into, uint32_t slow) {
  const uint64_t cs = d.cs, batch = cs < 1024 ? 0 : (cs - 768) * 14336;
  uint64_t most = 0;
  if (mixed_parity(d.len_lo, d.len_hi) && !split_unsure(d)) {
    const uint64_t a = (cs << 13) + (cs << 12), b = (cs << 14) + (cs << 12) - (12u << 20);
    if (cs < 512)
      most = 0;
    else if (into != kSplitValues)
      most = cs << 14;
    else
      most = cs < 1024 ? cs << 12 : (a < b ? a : b);
  } else if (cs >= 1024 && slow <= kSamples / 4 * 3) {
    if (slow <= kSamples / 4)
      most = (cs << 13) + (into == kSplitValues ? cs << 11 : cs << 12) - (3u << 20);
    else if (slow <= kSamples / 8 * 3)
      most = (cs - 1024) * 10240;
    else if (cs > 2048)
      most = (cs - 2048) * 5120;
  }
  return into == kSplitBatch && most > batch ? batch : most;
}

// Whether it takes a look at samples to tell for a container, where `total`
// symbols are decoded in this launch: not in data that is sure; nor where it would
// not be split in any case; nor up to 8 Mi in chunks of 4096, where every span has
// a warp of its own and the slowest takes about as long as a lane per chunk (1 Mi,
// a twentieth nonzero 43 us, two symbols in turn 56 to 78, the chain 79), unless
// nearly all symbols are the same.  The look takes 2 us, or 4 with one parity (half
// zeros, Table 1, 40 Mi 65 us without it, 67.8 with it).
__host__ __device__ inline bool split_samples(const SplitData& d, SplitInto into, uint64_t total) {
  return split_unsure(d) && total <= split_most(d, into, 0) &&
         (total > (uint64_t)d.cs << 11 || excess_bits(d) < d.n / 32 * (mixed_parity(d.len_lo, d.len_hi) ? 1 : 10));
}

}  // namespace qlc
