// lut.cuh -- LUT construction by one CTA (Section 7), with the scheme chosen
// among candidates (Section 6).
#pragma once

#include "qlc_common.cuh"

namespace qlc {

// Rank of a symbol (Section 7): symbols with a larger count, or the same
// count and a smaller value, come first.  With key(t) = count(t) * 256 +
// (255 - t), which is unique and orders exactly that way (counts stay below
// 2^56), the rank of s is the number of keys above key(s): no sort, one
// comparison per key.  One thread per symbol; all threads read the same key
// at a time (a broadcast).
constexpr int kLutThreads = 256;

// From L2: the kernel before may have just written the counts.
__device__ __forceinline__ unsigned long long load_key(const unsigned long long* __restrict__ hist, int s) {
  return (__ldcg(hist + s) << 8) | (unsigned long long)(255 - s);
}

// The rank of symbol s.  Keys of a tensor below 2^24 symbols fit in 32 bits
// (small): a comparison and an add per key, where 64 bits take three operations
// and twice the loads.
__device__ __forceinline__ int rank_of(const unsigned long long* key, int s) {
  const unsigned long long k = key[s];
  int r = 0;
#pragma unroll 16
  for (int t = 0; t < 256; t++) r += key[t] > k;
  return r;
}
__device__ __forceinline__ int rank_of_small(const uint32_t* key, int s) {
  const uint32_t k = key[s];
  int r = 0;
#pragma unroll 8
  for (int t = 0; t < 64; t++) {
    const uint4 q = reinterpret_cast<const uint4*>(key)[t];
    r += (q.x > k) + (q.y > k) + (q.z > k) + (q.w > k);
  }
  return r;
}

// Codeword of a rank under a scheme (Section 5): area code i, then the
// rank's position in area i in area_bits[i] bits; 8-bit areas store the rank.
__host__ __device__ inline uint32_t lut_entry(const qlc_scheme& sc, int r) {
  uint32_t base = 0;
  for (int i = 0; i < 8; i++) {
    const uint32_t n = sc.area_n[i];
    if ((uint32_t)r < base + n) {
      const uint32_t b = sc.area_bits[i];
      const uint32_t suffix = b == 8 ? (uint32_t)r : (uint32_t)r - base;
      const uint32_t code = ((uint32_t)i << b) | suffix;
      return (code << 4) | (3 + b);
    }
    base += n;
  }
  return 0;
}

struct SchemeSet {
  qlc_scheme s[8];
  int count;
};

// What one CTA of kLutThreads threads knows after ranking: its symbol's
// (thread's) rank and entry, and the scheme.
struct LutRow {
  int rank;
  uint32_t entry;  // codeword << 4 | length
  int scheme;      // index in the set
};

// Ranks the symbols of a histogram and picks the scheme (Section 6: the scheme
// can be adapted to the distribution): each candidate is scored by its payload
// bits sum_s count[s] * len(rank[s]) and the smallest wins (ties: the earlier
// candidate).  Thread s is symbol s.  key (256 entries, 16-byte aligned) and bits are scratch.
__device__ __forceinline__ LutRow rank_and_choose(const unsigned long long* __restrict__ hist, const SchemeSet& set,
                                                  unsigned long long* key,
                                                  unsigned long long (&bits)[8][kLutThreads / 32], int tid) {
  // (the counts are bounded by their sum, but the caller's histogram may be any)
  const unsigned long long own = load_key(hist, tid);
  const bool small = !__syncthreads_or(own >> 32 != 0);
  if (small)
    reinterpret_cast<uint32_t*>(key)[tid] = (uint32_t)own;
  else
    key[tid] = own;
  __syncthreads();
  LutRow row;
  row.rank = small ? rank_of_small(reinterpret_cast<const uint32_t*>(key), tid) : rank_of(key, tid);
  row.scheme = 0;
  if (set.count > 1) {
    const int warp = tid >> 5, lane = tid & 31;
    const unsigned long long count = own >> 8;
    for (int k = 0; k < set.count; k++) {
      unsigned long long v = count * (unsigned long long)(lut_entry(set.s[k], row.rank) & 15u);
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) bits[k][warp] = v;
    }
    __syncthreads();
    unsigned long long best_bits = ~0ull;
    for (int k = 0; k < set.count; k++) {
      unsigned long long t = 0;
      for (int w = 0; w < kLutThreads / 32; w++) t += bits[k][w];
      if (t < best_bits) {
        best_bits = t;
        row.scheme = k;
      }
    }
  }
  row.entry = lut_entry(set.s[row.scheme], row.rank);
  return row;
}

// Writes thread tid's row of the LUT, and the scheme.
__device__ __forceinline__ void write_lut(qlc_lut* lut, const LutRow& row, const SchemeSet& set, int tid) {
  lut->enc[tid] = (uint16_t)row.entry;
  lut->dec[row.rank] = (uint8_t)tid;
  if (tid < (int)(sizeof(qlc_scheme) / 4))
    reinterpret_cast<uint32_t*>(&lut->scheme)[tid] = reinterpret_cast<const uint32_t*>(&set.s[row.scheme])[tid];
}

// Host parts of the entry points, for the calls that chain them.
bool scheme_set(const qlc_scheme* h_schemes, int n_schemes, SchemeSet* set);  // false: a bad scheme or count
// Zeroes or adds to d_hist; the counting kernel is launched as usual.
qlc_status launch_histogram(const uint8_t* d_in, size_t n, uint64_t* d_hist, int accumulate, cudaStream_t st);
// n_luts LUTs; after: directly behind another kernel of the same call.
qlc_status launch_luts(const uint64_t* d_hists, int n_luts, const SchemeSet& set, qlc_lut* d_luts, bool after,
                       cudaStream_t st);

}  // namespace qlc
