// split_rule.cuh -- when a container is decoded split (decode_span.cuh) and when
// a lane per chunk (decode.cu).  One rule for single containers, for the shards
// of a batch and for the plan of a batch; host and device.
#pragma once

#include "qlc_common.cuh"

namespace qlc {

constexpr uint32_t kSamples = 32;  // places looked at, see sample_is_slow

// What the rule looks at: the header's chunk size, code lengths (len_lo, len_hi:
// of areas 0-3 and 4-7, one byte each), symbols and payload.
struct SplitData {
  uint32_t cs, len_lo, len_hi;
  uint64_t n, payload_bytes;
};

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

// The most symbols decoded in one launch for which splitting pays; values: the
// output is values, not codes; slow: of kSamples samples, in data that is unsure.
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
// Hence lines proportional to the chunk, less what a launch takes in any case.
__host__ __device__ inline uint64_t split_most(const SplitData& d, bool values, uint32_t slow) {
  const uint64_t cs = d.cs;
  const bool mixed = mixed_parity(d.len_lo, d.len_hi);
  if (mixed && !split_unsure(d)) {
    if (cs < 512) return 0;
    if (!values) return cs << 14;
    const uint64_t a = (cs << 13) + (cs << 12), b = (cs << 14) + (cs << 12) - (12u << 20);
    return cs < 1024 ? cs << 12 : (a < b ? a : b);
  }
  if (cs < 1024 || slow > kSamples / 4 * 3) return 0;
  if (slow <= kSamples / 4) return (cs << 13) + (values ? cs << 11 : cs << 12) - (3u << 20);
  if (slow <= kSamples / 8 * 3) return (cs - 1024) * 10240;
  return cs < 2048 ? 0 : (cs - 2048) * 5120;
}

// Whether it takes a look at samples to tell for a container, where `total`
// symbols are decoded in this launch: not in data that is sure; nor where it would
// not be split in any case; nor up to 8 Mi in chunks of 4096, where every span has
// a warp of its own and the slowest takes about as long as a lane per chunk (1 Mi,
// a twentieth nonzero 43 us, two symbols in turn 56 to 78, the chain 79), unless
// nearly all symbols are the same.  The look takes 2 us, or 4 with one parity (half
// zeros, Table 1, 40 Mi 65 us without it, 67.8 with it).
__host__ __device__ inline bool split_samples(const SplitData& d, bool values, uint64_t total) {
  return split_unsure(d) && total <= split_most(d, values, 0) &&
         (total > (uint64_t)d.cs << 11 || excess_bits(d) < d.n / 32 * (mixed_parity(d.len_lo, d.len_hi) ? 1 : 10));
}

}  // namespace qlc
