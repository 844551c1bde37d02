// encode.cu -- QLC encoder (Sections 5 and 7) writing container v1.
//
// encode_kernel, one persistent kernel: teams of eight warps, two to a CTA, take
// groups (32 chunks) in ticket order; the LUT is staged in shared memory once per
// team and tensor, one copy per lane, so every lookup is free of bank conflicts.
//   pass 1  each warp sums the code lengths of four chunks in a row -> chunk_bits;
//   look-back  warp 0 publishes the group's padded byte size and finds the sum of
//           all earlier groups' sizes (decoupled look-back, bounded waits), while
//           the other warps pack their first step;
//   pass 2  each warp re-reads its four chunks (about two thirds from L2) and
//           packs them as one run of the group's bit stream, 1024 symbols per
//           step: codeword pairs, a warp scan of the lanes' bit counts, per-lane
//           word accumulation into a per-warp staging window (completed words
//           are plain stores, a lane's partial last word one shared OR), and
//           16-byte streaming stores of every completed 16-byte block.
// Small tensors take lengths_kernel and pack_kernel instead.
//
// 256 Mi symbols, t4 data: 184 us (217 with three CTAs of 8 warps, 512 symbols a
// step, a chunk at a time with blocks merged by the CTA).  16.8 instructions per
// symbol (22 before): 4 for a length, 12 for packing.  It is bound by the shared-
// memory pipe (34.7 M wavefronts, 72 % busy: two lookups per symbol, and word
// stores at 1.7 wavefronts) and the integer pipe (71 %), and loses about a fifth
// of its warps' time to the look-back and its barriers.  Measured and left out:
// teams of 16 warps 201 us; the next group's pass 1 before this group's pass 2
// 223 us (the re-reads then miss L2); pass 1 and pass 2 as two kernels 78 + 140
// us; shift and OR by one wide multiply-add 193 us (fewer integer instructions,
// more in all).
#include <mutex>
#include <unordered_map>
#include <utility>

#define QLC_FILE_ID 2
#include "hist_cols.cuh"
#include "lut.cuh"
#include "../../include/qlc_testing.h"

namespace qlc {

constexpr int kPartThreads = 256;  // of lengths_kernel and pack_kernel
constexpr int kPartWarps = kPartThreads / 32;
constexpr int kPackCtasPerSm = 3;
constexpr int kTeams = 2;  // of a CTA of encode_kernel
constexpr int kTeamThreads = 256;
constexpr int kTeamWarps = kTeamThreads / 32;
constexpr int kRun = kGroupChunks / kTeamWarps;  // chunks of a group that a warp takes
constexpr int kEncCtasPerSm = 2;
constexpr uint32_t kBatch = 2048;  // symbols whose lengths a warp sums while it fetches the next ones
// Shared address of encode_kernel's tables; dynamic shared memory starts at or below it.
constexpr uint32_t kTableAddr = 2048;
constexpr int kHalf = 32 * 16;  // symbols of half a step, 16 per lane
// words of a warp's staging window: a block carried over, one step's bits, one spare block
constexpr int kWStage = 4 + (2 * kHalf * kMaxCode + 31) / 32 + 4;
constexpr int kPass1Unroll = 8;
// Tensors of up to this many chunks are encoded in parts (lengths_kernel, pack_kernel).
constexpr uint64_t kPartMaxChunks = 4096;

constexpr unsigned long long kFlagAgg = 1ull << 62;
constexpr unsigned long long kFlagPrefix = 2ull << 62;
constexpr unsigned long long kFlagError = 3ull << 62;
constexpr unsigned long long kValMask = (1ull << 62) - 1;
constexpr uint64_t kWaitLimitNs = 1000000000ull;  // 1 s per look-back wait

// OR v into a shared word.
__device__ __forceinline__ void red_or(uint32_t saddr, uint32_t v) {
  asm volatile("red.shared.or.b32 [%0], %1;" ::"r"(saddr), "r"(v) : "memory");
}

__device__ __forceinline__ uint32_t ld_shared_u32(uint32_t saddr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(saddr) : "memory");
  return v;
}
__device__ __forceinline__ void st_shared_u32(uint32_t saddr, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(saddr), "r"(v) : "memory");
}

// Appends the MSB-aligned bits P (at most 22) to the accumulator: hi holds the
// bits of the current word, at shared address wa.  at is the stream position
// before P and next the one after it; only their low six bits count.  When the
// word is complete it is stored and hi gets what spills over: one predicate,
// no branch.
__device__ __forceinline__ void append(uint32_t& hi, uint32_t& wa, uint32_t P, uint32_t at, uint32_t next) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      ".reg .b32 t, lo;\n\t"
      "shf.r.wrap.b32 t, %2, 0, %3;\n\t"   // P >> (at & 31)
      "shf.r.wrap.b32 lo, 0, %2, %3;\n\t"  // P << (32 - (at & 31)), 0 when that is 32
      "or.b32 %0, %0, t;\n\t"
      "xor.b32 t, %3, %4;\n\t"
      "and.b32 t, t, 32;\n\t"
      "setp.ne.u32 q, t, 0;\n\t"
      "@q st.shared.u32 [%1], %0;\n\t"
      "selp.b32 %0, lo, %0, q;\n\t"
      "@q add.u32 %1, %1, 4;\n\t"
      "}"
      : "+r"(hi), "+r"(wa)
      : "r"(P), "r"(at), "r"(next)
      : "memory");
}

// Inclusive sum over the warp's lanes.
__device__ __forceinline__ uint32_t warp_scan(uint32_t v) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1)
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b32 t;\n\t"
        "shfl.sync.up.b32 t|p, %0, %1, 0, 0xffffffff;\n\t"
        "@p add.u32 %0, %0, t;\n\t}"
        : "+r"(v)
        : "r"(o));
  return v;
}

__device__ __forceinline__ uint32_t warp_sum_u32(uint32_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The encoder table holds one copy per lane, so the 32 lanes of a lookup always
// hit 32 different banks.
struct PartTable {  // rows of 128 bytes
  const uint8_t* col;  // this lane's word of row 0
  __device__ __forceinline__ uint32_t at(uint32_t s) const {
    return *reinterpret_cast<const uint32_t*>(col + (s << 7));
  }
  // entry of byte j of w
  __device__ __forceinline__ uint32_t of(uint32_t w, int j) const { return at(__byte_perm(w, 0, 0x4440 + j)); }
};
// Two teams' tables side by side in rows of 256 bytes, at a constant address: one
// byte permute makes the whole offset (symbol << 8 | col), where rows of 128
// bytes take two instructions.
struct WideTable {
  uint32_t col;  // 128 * team + 4 * lane
  __device__ __forceinline__ uint32_t load(uint32_t offset) const {
    uint32_t e;
    asm volatile("ld.shared.u32 %0, [%1 + %2];" : "=r"(e) : "r"(offset), "n"(kTableAddr));
    return e;
  }
  __device__ __forceinline__ uint32_t at(uint32_t s) const { return load((s << 8) | col); }
  __device__ __forceinline__ uint32_t of(uint32_t w, int j) const {
    return load(__byte_perm(w, col, 0x5504 | (j << 4)));
  }
};

// Sum of the encoder entries of 16 symbols.  An entry is
// codeword << (32 - len) | len with len <= 11, so its bits below 21 are the
// length alone, and the low 21 bits of a sum of entries are the sum of the
// lengths as long as that stays below 2^21.
template <class Table>
__device__ __forceinline__ uint32_t entry_sum16(const Table& tab, uint4 q) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < 4; k++)
#pragma unroll
    for (int j = 0; j < 4; j++) s += tab.of(w[k], j);
  return s;
}

// Decoupled look-back over groups (warp-wide).  Publishes this group's size,
// returns the byte offset of the group (sum of all earlier groups' sizes).
// Every wait is bounded; on timeout *err is set and an error flag is
// published so that later groups stop waiting too.
__device__ unsigned long long lookback(unsigned long long* gstat, uint64_t g, uint64_t first,
                                       uint64_t gbytes, int lane, bool* err) {
  *err = false;
  if (g == first) {
    if (lane == 0) st_release_u64(&gstat[g], kFlagPrefix | gbytes);
    return 0;
  }
  if (lane == 0) st_release_u64(&gstat[g], kFlagAgg | gbytes);
  unsigned long long excl = 0;
  int64_t idx = (int64_t)g - 1 - lane;
  const uint64_t t0 = globaltimer_ns();
  while (true) {
    unsigned long long v = kFlagPrefix;  // before the shard's first group: prefix 0
    if (idx >= (int64_t)first) {
      while (true) {
        v = ld_acquire_u64(&gstat[idx]);
        if (v >> 62) break;
        if (globaltimer_ns() - t0 > kWaitLimitNs) {
          v = kFlagError;
          break;
        }
        __nanosleep(64);
      }
    }
    const unsigned flag = (unsigned)(v >> 62);
    const unsigned stop = __ballot_sync(0xffffffffu, flag >= 2);
    if (stop) {
      const int k = __ffs(stop) - 1;  // nearest earlier group with a full prefix
      const unsigned bad = __ballot_sync(0xffffffffu, flag == 3 && lane <= k);
      excl += warp_sum_u64(lane <= k ? (v & kValMask) : 0ull);
      *err = bad != 0;
      break;
    }
    excl += warp_sum_u64(v & kValMask);
    idx -= 32;
  }
  if (lane == 0) st_release_u64(&gstat[g], (*err ? kFlagError : kFlagPrefix) | (excl + gbytes));
  return excl;
}

// The header but its dec; 256 threads call it.
__device__ void write_header_of(uint8_t* out, uint64_t n, uint32_t cs, uint64_t n_chunks, const qlc_scheme* scheme,
                                int tid) {
  if (tid == 0) {
    *reinterpret_cast<uint32_t*>(out + 0) = 0x31434C51u;  // "QLC1"
    *reinterpret_cast<uint16_t*>(out + 4) = QLC_VERSION;
    out[6] = scheme->id;
    out[7] = 0;
    *reinterpret_cast<unsigned long long*>(out + 8) = n;
    *reinterpret_cast<uint32_t*>(out + 16) = cs;
    *reinterpret_cast<uint32_t*>(out + 20) = (uint32_t)n_chunks;
    *reinterpret_cast<unsigned long long*>(out + 56) = 0;
  }
  if (tid < 8) {
    *reinterpret_cast<uint16_t*>(out + 24 + 2 * tid) = scheme->area_n[tid];
    out[40 + tid] = scheme->area_bits[tid];
  }
  const uint64_t idx_end = kIndexOff + 8 * n_groups_of(n_chunks) + 2 * n_chunks;
  const uint64_t P = payload_start(n_chunks);
  if (idx_end + tid < P) out[idx_end + tid] = 0;
}
__device__ void write_header(uint8_t* out, uint64_t n, uint32_t cs, uint64_t n_chunks, const qlc_lut* lut, int tid) {
  write_header_of(out, n, cs, n_chunks, &lut->scheme, tid);
  if (tid < 256) out[64 + tid] = lut->dec[tid];
}

// Work source of the encode kernel: one tensor (descs == nullptr), or the
// shards of a batch, whose groups are numbered consecutively shard after
// shard (item_base[s] = first item of shard s, item_base[n_shards] = total).
struct EncArgs {
  const uint8_t* in;
  uint64_t n;
  const qlc_lut* lut;
  uint8_t* out;
  unsigned long long* out_bytes;
  uint64_t n_items;  // one tensor: its groups
  const qlc_desc* descs;
  const unsigned long long* item_base;
  int n_shards;
  uint32_t cs;
  unsigned int* ticket;
  unsigned long long* gstat;
  uint32_t* status;
  uint64_t out_cap;    // one tensor: bytes at out (batches: each descriptor's)
  uint64_t gstat_cap;  // look-back words at gstat
};

// Packing state of one warp within a run of chunks.  A step appends 512 or 1024
// symbols, 16 per lane and half, to the bit stream in the warp's staging
// window; completed 16-byte blocks go to the payload, and the block in work
// moves to the window's front.
// Where a run goes: its group's payload (null: nowhere, the group is given up) and
// the 16-byte blocks there (for the checked build).
struct Place {
  uint4* dst;
  uint32_t blk_lim;
};

template <class Table, class Find>
struct Packer {
  Table tab;
  const Find& find;  // the place, asked for when the first step's blocks are there
  uint32_t* stage;   // the warp's window
  uint32_t stage_s;  // its shared address
  uint4* dst;        // the window's block `lane` in the payload
  uint32_t off;      // bits in the window, below 128 between steps
  uint32_t blk;      // the window's first block within the payload
  uint32_t blk_lim;  // 16-byte blocks of the payload (checked build)
  bool shared;       // the run's first block starts before it
  int lane;

  __device__ __forceinline__ void put_block(uint32_t b, uint32_t nblk, bool skip) const {
    if (b < nblk && !skip && QLC_GUARD(blk + b < blk_lim, nullptr)) {
      const uint4 v = reinterpret_cast<const uint4*>(stage)[b];
      st_cs_v4(dst + (b - lane), make_uint4(bswap32(v.x), bswap32(v.y), bswap32(v.z), bswap32(v.w)));
    }
  }

  // kHalves 1 or 2: symbols in q[0 .. kHalves).  kRagged: the lane's first cnt
  // symbols of q[0] alone (total_cnt over all lanes), and no block from blk_end
  // on.  first: the run's first step.  False when the group is given up.
  template <int kHalves, bool kRagged>
  __device__ __forceinline__ bool step(const uint4 (&q)[kHalves], int cnt, bool first, uint32_t total_cnt,
                                       uint32_t blk_end) {
    // codeword pairs: P MSB-aligned (at most 22 bits); c the running sum of the
    // entries, whose low 21 bits are the bits so far
    uint32_t P[kHalves][8], c[kHalves][8];
#pragma unroll
    for (int h = 0; h < kHalves; h++) {
      const uint32_t w[4] = {q[h].x, q[h].y, q[h].z, q[h].w};
      uint32_t sum = 0;
#pragma unroll
      for (int k = 0; k < 8; k++) {
        uint32_t e0 = tab.of(w[k / 2], 2 * k & 3), e1 = tab.of(w[k / 2], (2 * k & 3) + 1);
        if (kRagged) {
          e0 = 2 * k < cnt ? e0 : 0u;
          e1 = 2 * k + 1 < cnt ? e1 : 0u;
        }
        // the second code right after the first: e1 >> len0 (a shift takes the
        // low five bits of e0) also moves e1's length down to bits 0..3, which
        // the mask clears with e0's
        P[h][k] = (e0 | __funnelshift_r(e1, 0u, e0)) & ~31u;
        sum += e0 + e1;
        c[h][k] = sum;
      }
    }
    // one scan for both halves, of at most 32 * 176 bits each
    const uint32_t len = kHalves == 2 ? __byte_perm(c[0][7], c[kHalves - 1][7], 0x5410) : c[0][7] & 0xFFFFu;
    const uint32_t incl = warp_scan(len);
    const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t excl = incl - len;
    const uint32_t end = off + (tot & 0xFFFFu) + (tot >> 16);
    // Each lane packs its pairs from its bit of the stream on; lane 0 goes on
    // with the word in work.  A completed word is stored whole: a lane's first
    // one lacks the previous lane's last bits, which that lane ORs in when all
    // words are stored.  16 codes have at least 48 bits, so each lane completes
    // a word, no two lanes store the same one and nothing has to be zero
    // before; only the last lane's last word is still to be written.  In a
    // ragged step a lane may have few bits or none, so there the words it can
    // reach are zeroed and every last word is OR-ed.
    if (kRagged) {
      const uint32_t words = ((off + total_cnt * kMaxCode) >> 5) + 1;
      for (uint32_t i = (off >> 5) + 1 + lane; i <= words; i += 32)
        if (QLC_GUARD(i < (uint32_t)kWStage, nullptr)) stage[i] = 0;
      __syncwarp();
    }
    uint32_t hi[kHalves], wa[kHalves];
#pragma unroll
    for (int h = 0; h < kHalves; h++) {
      uint32_t p = off + (excl & 0xFFFFu);
      if (h == 1) p = off + (tot & 0xFFFFu) + (excl >> 16);
      wa[h] = stage_s + (p >> 5) * 4;
      hi[h] = 0;
      if (h == 0 && lane == 0) hi[0] = ld_shared_u32(wa[0]);
      if (QLC_GUARD(((p + (c[h][7] & 0xFFFFu)) >> 5) < (uint32_t)kWStage, nullptr)) {
        uint32_t at = p;
#pragma unroll
        for (int k = 0; k < 8; k++) {
          const uint32_t next = p + c[h][k];
          append(hi[h], wa[h], P[h][k], at, next);
          at = next;
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < kHalves; h++) {
      if (!kRagged && h == kHalves - 1 && lane == 31)
        st_shared_u32(wa[h], hi[h]);
      else
        red_or(wa[h], hi[h]);
    }
    __syncwarp();
    uint32_t nblk = end >> 7;
    if (kRagged) nblk = min(nblk, blk_end - blk);
    bool skip = false;
    if (first) {
      const Place p = find();
      if (!p.dst) return false;
      dst = p.dst + blk + lane;
      blk_lim = p.blk_lim;
      skip = lane == 0 && shared;
    }
    put_block(lane, nblk, skip);
    if (kHalves == 2 || nblk > 32) put_block(lane + 32, nblk, false);
    if (kHalves == 2 && nblk > 64) put_block(lane + 64, nblk, false);
    uint32_t carry = 0;
    if (lane < 4) carry = stage[4 * nblk + lane];
    __syncwarp();
    if (lane < 4) stage[lane] = carry;
    dst += nblk;
    blk += nblk;
    off = end & 127u;
    __syncwarp();
    return true;
  }
};

// A LUT entry as the kernels keep it, codeword << (32 - len) | len, or 0 for
// one that is not a codeword of 3..11 bits (a LUT not made by qlc_build_lut*),
// which would overrun the staging window and the output bound.
__device__ __forceinline__ uint32_t table_entry(uint32_t e) {
  const uint32_t len = e & 15u, code = e >> 4;
  return len < 3 || len > kMaxCode || (code >> len) != 0 ? 0u : (code << (32 - len)) | len;
}
// Stages entry v of symbol s at its row, one copy per lane; pieces in an order
// that spreads the threads' stores over the banks.
__device__ __forceinline__ void stage_entry(uint8_t* row, int s, uint32_t v) {
#pragma unroll
  for (int k = 0; k < 8; k++) reinterpret_cast<uint4*>(row)[(k + s) & 7] = make_uint4(v, v, v, v);
}

// Bits of m symbols at p (16-byte aligned; m <= 4096, so that a lane's sum
// stays below 2^21), the same in every lane.
template <class Table>
__device__ __forceinline__ uint32_t chunk_length(const Table& tab, const uint8_t* p, uint32_t m, int lane) {
  uint32_t bits = 0;
  const uint32_t nv = m / 16;
  const uint4* v = reinterpret_cast<const uint4*>(p);
  uint32_t k = lane;
  for (; k + (kPass1Unroll - 1) * 32 < nv; k += kPass1Unroll * 32) {
    uint4 q[kPass1Unroll];
#pragma unroll
    for (int u = 0; u < kPass1Unroll; u++) q[u] = ldg_nc_v4(v + k + 32 * u);
#pragma unroll
    for (int u = 0; u < kPass1Unroll; u++) bits += entry_sum16(tab, q[u]);
  }
  for (; k < nv; k += 32) bits += entry_sum16(tab, ldg_nc_v4(v + k));
  for (uint32_t t = nv * 16 + lane; t < m; t += 32) bits += tab.at(p[t]);
  return warp_sum_u32(bits & ((1u << 21) - 1));
}

// The first step's symbols of a run of m at p.
__device__ __forceinline__ void load_first(uint4 (&q)[2], const uint8_t* p, uint32_t m, int lane) {
#pragma unroll
  for (uint32_t h = 0; h < 2; h++)
    q[h] = h < m / kHalf ? ldg_nc_v4(reinterpret_cast<const uint4*>(p) + lane + 32 * h) : make_uint4(0, 0, 0, 0);
}

// Packs a run of a group's chunks: m symbols at p (next: load_first of them),
// group-relative bits [S, E), rest more symbols of the group behind them, to the
// place that find() tells, which every run calls once.  A 16-byte block belongs
// to the run that its first bit falls in: the run also encodes the symbols after
// it that reach into its last block (48 have 144 bits or more; a run ends on a
// multiple of 128 symbols or with its tensor, so they never fill a step), and
// leaves its first block out when that starts before the run.  Runs need nothing
// from one another, and no barrier.
template <class Table, class Find>
__device__ __forceinline__ void pack_run(const Table& tab, uint32_t* stage, const uint8_t* p, uint32_t m, uint64_t rest,
                                         uint32_t S, uint32_t E, uint4 (&next)[2], const Find& find, int lane) {
  const uint32_t blk_end = (E + 127u) >> 7;
  if ((S + 127u) >> 7 >= blk_end) {  // the last symbols of a tensor, in another run's block
    find();
    return;
  }
  if (E & 127u) m += (uint32_t)min(rest, (uint64_t)48);
  Packer<Table, Find> pk = {tab, find, stage};
  pk.stage_s = (uint32_t)__cvta_generic_to_shared(stage);
  pk.off = S & 127u;
  pk.blk = S >> 7;
  pk.shared = pk.off != 0;
  pk.lane = lane;
  bool first = true;
  if (lane < 4) stage[lane] = 0;
  __syncwarp();
  // full steps, with the input of the next one in flight
  const uint32_t n_half = m / kHalf;
  const uint4* src = reinterpret_cast<const uint4*>(p) + lane;
  uint32_t i = 0;
  for (; i + 2 <= n_half; i += 2) {
    const uint4 q[2] = {next[0], next[1]};
#pragma unroll
    for (uint32_t h = 0; h < 2; h++)
      if (i + 2 + h < n_half) next[h] = ldg_nc_v4(src + 32 * (i + 2 + h));
    if (!pk.template step<2, false>(q, 16, first, 0, 0)) return;
    first = false;
  }
  if (i < n_half) {
    const uint4 q[1] = {next[0]};
    if (!pk.template step<1, false>(q, 16, first, 0, 0)) return;
    first = false;
  }
  // what is left, 16 symbols a lane
  if (m % kHalf) {
    const uint32_t at = n_half * kHalf + 16u * lane;
    const int cnt = at < m ? (int)min(16u, m - at) : 0;
    uint4 q[1] = {make_uint4(0, 0, 0, 0)};
    if (cnt == 16) {
      q[0] = ldg_nc_v4(reinterpret_cast<const uint4*>(p + at));
    } else {
      uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
      for (int j = 0; j < 16; j++)
        if (j < cnt) w[j >> 2] |= (uint32_t)p[at + j] << (8 * (j & 3));
      q[0] = make_uint4(w[0], w[1], w[2], w[3]);
    }
    if (!pk.template step<1, true>(q, cnt, first, m % kHalf, blk_end)) return;
  }
  // the group's zero-padded end
  if (pk.blk < blk_end && lane == 0 && QLC_GUARD(pk.blk < pk.blk_lim, nullptr)) {
    uint32_t v[4];
#pragma unroll
    for (uint32_t k = 0; k < 4; k++) v[k] = k <= pk.off >> 5 ? bswap32(stage[k]) : 0u;
    st_cs_v4(pk.dst, make_uint4(v[0], v[1], v[2], v[3]));
  }
  __syncwarp();
}

struct TeamShared {
  unsigned long long item, first, excl;
  const uint8_t* in;
  uint64_t n;
  const qlc_lut* lut;
  uint8_t* out;
  uint64_t cap;
  unsigned long long* ob;
  int err;
  uint32_t chunk_bits[kGroupChunks];
};
struct EncShared {
  uint8_t table[256 << 8];  // codeword << (32 - len) | len, one copy per team and lane
  __align__(16) uint32_t stage[kTeams * kTeamWarps][kWStage];
  TeamShared team[kTeams];
};
constexpr size_t kEncSharedBytes = fixed_smem_bytes(kTableAddr, sizeof(EncShared));

// Barriers of a team's threads.  The second one is for a group's offset, which
// warp 0 tells the others.
__device__ __forceinline__ void team_sync(int team) {
  asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(kTeamThreads) : "memory");
}
__device__ __forceinline__ void offset_tell(int team) {
  asm volatile("bar.arrive %0, %1;" ::"r"(team + 1 + kTeams), "n"(kTeamThreads) : "memory");
}
__device__ __forceinline__ void offset_wait(int team) {
  asm volatile("bar.sync %0, %1;" ::"r"(team + 1 + kTeams), "n"(kTeamThreads) : "memory");
}
__device__ __forceinline__ bool team_or(int team, bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, %2, %3, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(team + 1), "n"(kTeamThreads)
      : "memory");
  return r != 0;
}

// The next group and, in a batch, its tensor (warp-wide).
__device__ __forceinline__ void take_item(const EncArgs& A, uint64_t n_items, TeamShared& ts, int lane) {
  unsigned long long t = 0;
  if (lane == 0) t = atomicAdd(A.ticket, 1u);
  t = __shfl_sync(0xffffffffu, t, 0);
  const int shard = A.descs && t < n_items ? shard_of_warp(A.item_base, A.n_shards, t, lane) : 0;
  if (lane != 0) return;
  ts.item = t;
  if (t >= n_items) return;
  if (A.descs) {
    const qlc_desc d = A.descs[shard];
    ts.first = A.item_base[shard];
    ts.in = static_cast<const uint8_t*>(d.in);
    ts.n = d.in_bytes;
    ts.lut = d.lut;
    ts.out = static_cast<uint8_t*>(d.out);
    ts.cap = d.out_cap;
    ts.ob = reinterpret_cast<unsigned long long*>(d.out_bytes);
  } else {
    ts.first = 0;
    ts.in = A.in;
    ts.n = A.n;
    ts.lut = A.lut;
    ts.out = A.out;
    ts.cap = A.out_cap;
    ts.ob = A.out_bytes;
  }
}

// Lengths of a warp's kRun full chunks, cs symbols each from p on, to put(chunk
// of the run, bits): the next kBatch symbols are on their way while a batch is
// summed.  kPer 1: cs is a multiple of kBatch; 2: half of it (200 Mi symbols 275
// -> 248 us, a chunk at a time before; the end of a chunk looked for after every
// 512 symbols, for all sizes alike, costs 9 % at 4096).
template <int kPer, class Put>
__device__ __forceinline__ void run_lengths(const WideTable& tab, const uint8_t* p, uint32_t cs, int lane, Put put) {
  constexpr int kV = kBatch / 512;
  const uint4* src = reinterpret_cast<const uint4*>(p) + lane;
  const uint32_t per = cs / kBatch, total = kPer == 2 ? kRun / 2 : per * kRun;
  uint4 q[2][kV];
  uint32_t bits = 0, left = per, c = 0;
  auto fetch = [&](uint4 (&d)[kV]) {
#pragma unroll
    for (int u = 0; u < kV; u++) d[u] = ldg_nc_v4(src + 32 * u);
    src += 32 * kV;
  };
  auto add = [&](const uint4 (&d)[kV]) {
#pragma unroll
    for (int u = 0; u < kV; u++) {
      bits += entry_sum16(tab, d[u]);
      if (kPer == 2 && u % 2 == 1) {
        put(c++, warp_sum_u32(bits & ((1u << 21) - 1)));
        bits = 0;
      }
    }
    if (kPer == 1 && --left == 0) {
      put(c++, warp_sum_u32(bits & ((1u << 21) - 1)));
      bits = 0;
      left = per;
    }
  };
  fetch(q[0]);
  for (uint32_t j = 0; j < total; j += 2) {  // total is even: kRun is
    fetch(q[1]);
    add(q[0]);
    if (j + 2 < total) fetch(q[0]);
    add(q[1]);
  }
}

// A team's work on one group.
__device__ __forceinline__ void encode_group(const EncArgs& A, EncShared& sh, TeamShared& ts, int team,
                                             const qlc_lut*& cur_lut) {
  const int tid = threadIdx.x % kTeamThreads, lane = tid & 31, warp = tid >> 5;
  const uint32_t cs = A.cs;
  const uint64_t group_syms = (uint64_t)kGroupChunks * cs;
  const WideTable tab = {128u * team + 4u * lane};
  const uint64_t n = ts.n, item = ts.item, g = item - ts.first;  // g: the group within its tensor
  uint8_t* out = ts.out;
  const qlc_lut* lut = ts.lut;
  if (lut != cur_lut) {
    const uint32_t e = tid < 256 ? table_entry(lut->enc[tid]) : 1u;
    if (team_or(team, e == 0)) {  // the tensor is refused
      if (tid == 0) {
        set_status(A.status, QLC_ERR_ARG);
        st_release_u64(&A.gstat[item], kFlagError);
      }
      cur_lut = nullptr;
      return;
    }
    if (tid < 256) stage_entry(sh.table + 256 * tid + 128 * team, tid, e);
    cur_lut = lut;
    team_sync(team);
  }
  const uint64_t n_chunks = (n + cs - 1) / cs;
  const uint64_t n_groups = n_groups_of(n_chunks);
  if (g == 0) write_header(out, n, cs, n_chunks, lut, tid);
  if (n == 0) {  // an empty shard of a batch: header-only container
    if (tid == 0) {
      *reinterpret_cast<unsigned long long*>(out + 48) = 0;
      if (ts.ob) *ts.ob = payload_start(n_chunks);
    }
    return;
  }
  const uint64_t gbeg = g * group_syms;
  const uint64_t gend = min(gbeg + group_syms, n);
  const uint32_t c0 = warp * kRun;  // the warp's chunks
  const uint64_t beg = gbeg + (uint64_t)c0 * cs, end = min(beg + (uint64_t)kRun * cs, gend);
  const uint8_t* p = ts.in + beg;

  // ---- pass 1: bits of each chunk
  {
    uint16_t* chunk_bits = reinterpret_cast<uint16_t*>(out + kIndexOff + 8 * n_groups);
    auto put = [&](uint32_t i, uint32_t bits) {
      const uint32_t c = c0 + i;
      if (lane != 0) return;
      ts.chunk_bits[c] = bits;
      if (QLC_GUARD(g * kGroupChunks + c < n_chunks, A.status)) chunk_bits[g * kGroupChunks + c] = (uint16_t)bits;
    };
    if (gend - gbeg == group_syms && cs % kBatch == 0) {
      run_lengths<1>(tab, p, cs, lane, put);
    } else if (gend - gbeg == group_syms && cs == kBatch / 2) {
      run_lengths<2>(tab, p, cs, lane, put);
    } else {
      for (uint32_t i = 0; i < kRun; i++) {
        const uint64_t cbeg = beg + (uint64_t)i * cs;
        if (cbeg < gend)
          put(i, chunk_length(tab, ts.in + cbeg, (uint32_t)(min(cbeg + cs, gend) - cbeg), lane));
        else if (lane == 0)
          ts.chunk_bits[c0 + i] = 0;
      }
    }
  }
  uint4 next[2] = {};
  if (beg < gend) load_first(next, p, (uint32_t)(end - beg), lane);
  team_sync(team);

  const uint32_t cb = ts.chunk_bits[lane];
  const uint32_t incl = warp_scan(cb);  // group-relative bit of each chunk's end
  // ---- look-back, by warp 0: this group's byte offset in the payload.  The other
  // warps pack their first step meanwhile.
  if (warp == 0) {
    const uint64_t gbytes = align16((__shfl_sync(0xffffffffu, incl, 31) + 7) / 8);
    bool err = !QLC_GUARD(item < A.gstat_cap, A.status);
    const unsigned long long excl = err ? 0ull : lookback(A.gstat, item, ts.first, gbytes, lane, &err);
    if (lane == 0) {
      ts.excl = excl;
      ts.err = err;
      if (err) {
        set_status(A.status, QLC_ERR_TIMEOUT);
      } else {
        if (QLC_GUARD(g < n_groups, A.status)) reinterpret_cast<unsigned long long*>(out + kIndexOff)[g] = excl;
        if (g == n_groups - 1) {
          *reinterpret_cast<unsigned long long*>(out + 48) = excl + gbytes;
          if (ts.ob) *ts.ob = payload_start(n_chunks) + excl + gbytes;
        }
      }
    }
    __syncwarp();
    offset_tell(team);
  }
  const auto find = [&]() -> Place {
    if (warp != 0) offset_wait(team);
    if (ts.err) return {nullptr, 0};
    const uint64_t start = payload_start((ts.n + cs - 1) / cs) + ts.excl;
    return {reinterpret_cast<uint4*>(ts.out + start), (uint32_t)min((ts.cap - start) / 16, (uint64_t)0xFFFFFFFEu)};
  };

  // ---- pass 2: the warp's chunks, one run of the group's bit stream
  if (beg >= gend || !QLC_GUARD(end <= n, A.status)) {
    find();
    return;
  }
  const uint32_t S = __shfl_sync(0xffffffffu, incl - cb, c0), E = __shfl_sync(0xffffffffu, incl, c0 + kRun - 1);
  pack_run(tab, sh.stage[threadIdx.x >> 5], p, (uint32_t)(end - beg), gend - end, S, E, next, find, lane);
}

__global__ void __launch_bounds__(kTeams* kTeamThreads, kEncCtasPerSm)
encode_kernel(EncArgs A) {
  extern __shared__ __align__(16) uint8_t enc_smem[];
  const uint32_t smem_s = (uint32_t)__cvta_generic_to_shared(enc_smem);
  if (smem_s > kTableAddr) {  // does not happen
    if (threadIdx.x == 0) set_status(A.status, QLC_ERR_CUDA);
    return;
  }
  EncShared& sh = *reinterpret_cast<EncShared*>(enc_smem + (kTableAddr - smem_s));
  const int team = threadIdx.x / kTeamThreads, lane = threadIdx.x & 31, warp = threadIdx.x % kTeamThreads / 32;
  const qlc_lut* cur_lut = nullptr;
  dependency_wait();
  const uint64_t n_items = A.descs ? A.item_base[A.n_shards] : A.n_items;
  if (team > 0 && n_items <= gridDim.x) return;  // a CTA per group
  TeamShared& ts = sh.team[team];
  while (true) {
    team_sync(team);
    // taken early (by a warp that is done before the others) a group would be
    // waited for longer by those after it: 1152 tensors 2680 us instead of 2570
    if (warp == 0) take_item(A, n_items, ts, lane);
    team_sync(team);
    if (ts.item >= n_items) break;
    encode_group(A, sh, ts, team, cur_lut);
  }
}

// ------------------------------------------------------- tensors of few groups
//
// A team per group leaves most of the GPU idle below a few hundred groups, and
// a team takes about 20 us for a group of 32 x 4096 symbols.  Up to
// kPartMaxChunks chunks the work is cut finer, in two kernels without
// look-back (and without the memset of its words).  Histogram, LUT and encode
// of Student-t symbols, us, by groups / in parts: in chunks of 4096 4 Mi symbols
// 34 / 23.3, 12 Mi 37.6 / 35, 16 Mi 40 / 37.6, 24 Mi 48.2 / 46.5, 32 Mi 49.3 /
// 54.7, 40 Mi 73.5 / 64.9, 64 Mi 80.8 / 91.6, 256 Mi 245 / 309; in chunks of 1024
// 4 Mi 28.7 / 29.4, 8 Mi 29.1 / 33.9, 64 Mi 99.8 / 142; in chunks of 128 0.5 Mi
// 23.6 / 21.8, 1 Mi 23.9 / 27.8, 8 Mi 67 / 93: the line lies at 4096 chunks.
//   lengths  a warp per chunk: chunk_bits (and the container's header);
//   pack     a CTA per part of kPartWarps chunks, a chunk per warp. The sizes of
//            the groups before a part's are summed from chunk_bits (2 bytes per
//            chunk, from L2), so a CTA needs nothing from the others.
// With kBuild every CTA ranks the histogram itself (about 1 us), and the first
// writes the LUT: no kernel of its own between the histogram and this one.
template <bool kBuild>
__global__ void __launch_bounds__(kPartThreads)
lengths_kernel(const uint8_t* __restrict__ in, uint64_t n, const unsigned long long* __restrict__ hist, SchemeSet set,
               qlc_lut* lut, uint32_t cs, uint8_t* out, uint32_t* status) {
  static_assert(kPartThreads == kLutThreads, "a thread per symbol");
  __shared__ __align__(16) uint8_t s_enc[256 << 7];
  __shared__ __align__(16) unsigned long long s_key[kBuild ? 256 : 2];
  __shared__ unsigned long long s_bits[8][kLutThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n_chunks = ((uint32_t)n + cs - 1) / cs;  // <= kPartMaxChunks
  dependents_may_start();
  uint32_t e;
  if constexpr (kBuild) {
    dependency_wait();
    const LutRow row = rank_and_choose(hist, set, s_key, s_bits, tid);
    if (blockIdx.x == 0) {
      write_lut(lut, row, set, tid);
      write_header_of(out, n, cs, n_chunks, &set.s[row.scheme], tid);
      out[64 + row.rank] = (uint8_t)tid;
    }
    e = table_entry(row.entry);
  } else {
    e = table_entry(lut->enc[tid]);
  }
  stage_entry(s_enc + 128 * tid, tid, e);
  if (__syncthreads_or(e == 0)) {  // not a LUT of this library: refused
    if (blockIdx.x == 0 && tid == 0) set_status(status, QLC_ERR_ARG);
    return;
  }
  if (!kBuild && blockIdx.x == 0) write_header(out, n, cs, n_chunks, lut, tid);
  uint16_t* chunk_bits = reinterpret_cast<uint16_t*>(out + kIndexOff + 8 * n_groups_of(n_chunks));
  for (uint64_t c = (uint64_t)blockIdx.x * kPartWarps + warp; c < n_chunks; c += (uint64_t)gridDim.x * kPartWarps) {
    const uint64_t beg = c * cs;
    const uint32_t bits = chunk_length(PartTable{s_enc + 4 * lane}, in + beg, (uint32_t)min((uint64_t)cs, n - beg), lane);
    if (lane == 0) chunk_bits[c] = (uint16_t)bits;
  }
}

constexpr uint32_t kParts = kGroupChunks / kPartWarps;  // parts per group

__global__ void __launch_bounds__(kPartThreads, kPackCtasPerSm)
pack_kernel(const uint8_t* __restrict__ in, uint64_t n, const qlc_lut* lut, uint32_t cs, uint8_t* out,
            uint64_t out_cap, unsigned long long* out_bytes, uint32_t* status) {
  __shared__ __align__(16) uint8_t s_enc[256 << 7];
  __shared__ __align__(16) uint32_t s_stage[kPartWarps][kWStage];
  __shared__ unsigned long long s_sum[kPartWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  dependency_wait();
  const uint32_t e = table_entry(__ldcg(&lut->enc[tid]));
  stage_entry(s_enc + 128 * tid, tid, e);
  if (__syncthreads_or(e == 0)) return;  // lengths_kernel has set the status
  const PartTable tab = {s_enc + 4 * lane};
  const uint32_t n_chunks = ((uint32_t)n + cs - 1) / cs;  // <= kPartMaxChunks
  const uint32_t n_groups = (uint32_t)n_groups_of(n_chunks);
  const uint64_t P = payload_start(n_chunks);
  unsigned long long* group_off = reinterpret_cast<unsigned long long*>(out + kIndexOff);
  const uint16_t* chunk_bits = reinterpret_cast<const uint16_t*>(out + kIndexOff + 8 * (uint64_t)n_groups);
  unsigned long long excl = 0;  // payload offset of group g_at
  uint32_t g_at = 0;
  for (uint32_t item = blockIdx.x; item < n_groups * kParts; item += gridDim.x) {
    const uint32_t g = item / kParts, first = (item % kParts) * kPartWarps;  // the part's first chunk in the group
    const uint32_t c = first + warp;
    const uint64_t gbeg = (uint64_t)g * kGroupChunks * cs;
    const uint64_t gend = min(gbeg + (uint64_t)kGroupChunks * cs, n);
    const uint64_t beg = gbeg + (uint64_t)c * cs, end = min(beg + cs, gend);
    uint4 next[2] = {};
    if (beg < gend) load_first(next, in + beg, (uint32_t)(end - beg), lane);
    // the sizes of groups g_at .. g - 1 (all of 32 chunks): 8 lanes per group, 4 chunks each
    unsigned long long sum = 0;
    for (uint32_t b = 8 * g_at + 32 * warp; b < 8 * g; b += 32 * kPartWarps) {
      uint32_t bits = 0;
      if (b + lane < 8 * g) {
        const uint2 q = __ldcg(reinterpret_cast<const uint2*>(chunk_bits + 4 * (b + lane)));
        bits = (q.x & 0xFFFFu) + (q.x >> 16) + (q.y & 0xFFFFu) + (q.y >> 16);
      }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) bits += __shfl_xor_sync(0xffffffffu, bits, o);
      if ((lane & 7) == 0) sum += align16((bits + 7) / 8);
    }
    sum = warp_sum_u64(sum);
    // the group's chunks: bit offsets, in every warp
    const uint32_t cg = g * kGroupChunks + lane;
    const uint32_t cb = cg < n_chunks ? __ldcg(&chunk_bits[cg]) : 0u;
    uint32_t incl = cb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    const uint32_t gbits = __shfl_sync(0xffffffffu, incl, 31);
    __syncthreads();  // the previous part's sums are done with
    if (lane == 0) s_sum[warp] = sum;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kPartWarps; w++) excl += s_sum[w];
    g_at = g;
    if (first == 0 && tid == 0) {
      const unsigned long long gbytes = align16((gbits + 7) / 8);
      if (QLC_GUARD(g < n_groups, status)) group_off[g] = excl;
      if (g == n_groups - 1) {
        *reinterpret_cast<unsigned long long*>(out + 48) = excl + gbytes;
        *out_bytes = P + excl + gbytes;
      }
    }
    const uint32_t E = __shfl_sync(0xffffffffu, incl, c), S = E - __shfl_sync(0xffffffffu, cb, c);
    if (beg < gend)
      pack_run(tab, s_stage[warp], in + beg, (uint32_t)(end - beg), gend - end, S, E, next,
               [&]() -> Place {
                 return {reinterpret_cast<uint4*>(out + P + excl),
                         (uint32_t)min((uint64_t)((out_cap - P - excl) / 16), (uint64_t)0xFFFFFFFEu)};
               },
               lane);
  }
}

// ------------------------------------------------------- one CTA
//
// Histogram, LUT and encode of a tensor of up to 16 chunks (64 KiB) in one CTA, a
// warp per chunk: up to this size the three kernels that a larger tensor takes
// are little but their own latency.  Back to back, us, three kernels / this one:
// chunks of 4096, 4 KiB 13.7 / 9.4, 16 KiB 14.7 / 10.6, 64 KiB 16.8 / 14.8, 92 KiB
// 18.6 / 17.9, 128 KiB 18.1 / 21.1; 32 chunks of 1024 12.1 / 12.4, of 2048 15.2 /
// 17: one SM packs longer than the rest saves, hence 16 chunks.
constexpr uint32_t kOneChunks = 16;
struct OneShared {
  union {
    uint32_t cols[kHcColWords];     // the histogram's counters, then
    uint8_t table[256 << 7];        // the encoder table
  };
  __align__(16) uint32_t key[256];
  __align__(16) uint32_t stage[kOneChunks][kWStage];
  uint32_t chunk_bits[kGroupChunks];
  unsigned long long bits[8][kHcWarps];
};
static_assert(kHcWarps == (int)kGroupChunks && kOneChunks <= kGroupChunks, "a warp for every chunk of a group");

__global__ void __launch_bounds__(kHcThreads)
encode_one_kernel(const uint8_t* __restrict__ in, uint32_t n, SchemeSet set, uint32_t cs, unsigned long long* hist,
                  qlc_lut* lut, uint8_t* out, uint64_t out_cap, unsigned long long* out_bytes) {
  extern __shared__ __align__(16) uint8_t one_smem[];
  OneShared& sh = *reinterpret_cast<OneShared*>(one_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n_chunks = (n + cs - 1) / cs;
  const uint32_t beg = warp * cs, end = min(beg + cs, n);
  uint4 next[2] = {};
  if (beg < n) load_first(next, in + beg, end - beg, lane);
  // ---- counts: thread tid has that of symbol tid / 4
  zero_cols(sh.cols, tid);
  __syncthreads();
  const uint32_t col = lane_col(sh.cols, lane);
  count_span(reinterpret_cast<const uint4*>(in), n / 16, col, tid);
  count_bytes(in + n / 16 * 16, n % 16, col, tid);
  __syncthreads();
  const uint32_t count = sum_cols(sh.cols, tid), sym = tid >> 2, part = tid & 3;
  const uint32_t key = count << 8 | (255u - sym);  // fits: n < 2^24
  if (part == 0) {
    hist[sym] = count;
    sh.key[sym] = key;
  }
  __syncthreads();
  // ---- rank (see rank_of): four threads per symbol, 64 keys each
  int rank = 0;
#pragma unroll
  for (int t = 0; t < 16; t++) {
    const uint4 q = reinterpret_cast<const uint4*>(sh.key)[4 * t + part];
    rank += (q.x > key) + (q.y > key) + (q.z > key) + (q.w > key);
  }
  rank += __shfl_xor_sync(0xffffffffu, rank, 1);
  rank += __shfl_xor_sync(0xffffffffu, rank, 2);
  // ---- scheme (see rank_and_choose)
  int scheme = 0;
  if (set.count > 1) {
    for (int k = 0; k < set.count; k++) {
      const uint32_t len = lut_entry(set.s[k], rank) & 15u;
      const uint32_t v = warp_sum_u32(part == 0 ? count * len : 0u);  // at most 11 * 2^17
      if (lane == 0) sh.bits[k][warp] = v;
    }
    __syncthreads();
    unsigned long long best = ~0ull;
    for (int k = 0; k < set.count; k++) {
      unsigned long long t = 0;
      for (int w = 0; w < kHcWarps; w++) t += sh.bits[k][w];
      if (t < best) {
        best = t;
        scheme = k;
      }
    }
  }
  const uint32_t entry = lut_entry(set.s[scheme], rank);
  if (part == 0) {
    lut->enc[sym] = (uint16_t)entry;
    lut->dec[rank] = (uint8_t)sym;
    out[64 + rank] = (uint8_t)sym;
  }
  if (tid < (int)(sizeof(qlc_scheme) / 4))
    reinterpret_cast<uint32_t*>(&lut->scheme)[tid] = reinterpret_cast<const uint32_t*>(&set.s[scheme])[tid];
  write_header_of(out, n, cs, n_chunks, &set.s[scheme], tid);
  {
    const uint32_t e = table_entry(entry);
    uint4* row = reinterpret_cast<uint4*>(sh.table + 128 * sym);
#pragma unroll
    for (uint32_t k = 0; k < 2; k++) row[(2 * part + k + sym) & 7] = make_uint4(e, e, e, e);
  }
  __syncthreads();
  // ---- chunk lengths
  const PartTable tab = {sh.table + 4 * lane};
  uint16_t* chunk_bits = reinterpret_cast<uint16_t*>(out + kIndexOff + 8);
  uint32_t bits = 0;
  if (beg < n) {
    bits = chunk_length(tab, in + beg, end - beg, lane);
    if (lane == 0) chunk_bits[warp] = (uint16_t)bits;
  }
  if (lane == 0) sh.chunk_bits[warp] = bits;
  __syncthreads();
  // ---- packing
  const uint32_t cb = sh.chunk_bits[lane], incl = warp_scan(cb);
  const uint64_t P = payload_start(n_chunks);
  if (tid == 31) {  // the last lane of the scan
    const unsigned long long bytes = align16((incl + 7) / 8);
    *reinterpret_cast<unsigned long long*>(out + kIndexOff) = 0;
    *reinterpret_cast<unsigned long long*>(out + 48) = bytes;
    *out_bytes = P + bytes;
  }
  const uint32_t E = __shfl_sync(0xffffffffu, incl, warp), S = E - __shfl_sync(0xffffffffu, cb, warp);
  if (beg < n)
    pack_run(tab, sh.stage[warp], in + beg, end - beg, n - end, S, E, next,
             [&]() -> Place {
               return {reinterpret_cast<uint4*>(out + P), (uint32_t)min((out_cap - P) / 16, (uint64_t)0xFFFFFFFEu)};
             },
             lane);
}

// n = 0: a header-only container.
__global__ void header_only_kernel(uint8_t* out, uint32_t cs, const qlc_lut* lut,
                                   unsigned long long* out_bytes) {
  const int tid = threadIdx.x;
  write_header(out, 0, cs, 0, lut, tid);
  if (tid == 0) {
    *reinterpret_cast<unsigned long long*>(out + 48) = 0;
    *out_bytes = payload_start(0);
  }
}

}  // namespace qlc

using namespace qlc;

extern "C" {

size_t qlc_encoded_size(size_t n, uint32_t chunk_symbols) {
  if (!chunk_symbols_ok(chunk_symbols)) return 0;
  const uint64_t n_chunks = (n + chunk_symbols - 1) / chunk_symbols;
  const uint64_t group_syms = (uint64_t)kGroupChunks * chunk_symbols;
  const uint64_t full = n / group_syms, rest = n % group_syms;
  uint64_t total = payload_start(n_chunks);
  total += full * align16((group_syms * kMaxCode + 7) / 8);
  if (rest) total += align16((rest * kMaxCode + 7) / 8);
  return (size_t)total;
}

size_t qlc_encode_workspace_size(size_t n, uint32_t chunk_symbols) {
  if (!chunk_symbols_ok(chunk_symbols)) return 0;
  const uint64_t n_chunks = (n + chunk_symbols - 1) / chunk_symbols;
  return (size_t)(16 + 8 * n_groups_of(n_chunks));
}

// Resident encode CTAs per SM.
static int encode_ctas(const qlc_launch* launch) {
  const int n = launch ? launch->encode_ctas_per_sm : 0;
  return n > 0 && n < kEncCtasPerSm ? n : kEncCtasPerSm;
}

// Launches encode_kernel for up to `items` groups, after the previous kernel of
// the same call (pdl) or by itself.
static qlc_status launch_groups(const EncArgs& A, uint64_t items, const qlc_launch* launch, bool pdl, cudaStream_t st) {
  static OncePerContext done;
  if (!smem_ok(encode_kernel, kEncSharedBytes, done)) return QLC_ERR_CUDA;
  const uint64_t cap = (uint64_t)sm_count() * encode_ctas(launch);
  const int grid = (int)(items < 1 ? 1 : (items < cap ? items : cap));
  if (pdl)
    launch_after(encode_kernel, grid, kTeams * kTeamThreads, kEncSharedBytes, st, A);
  else
    encode_kernel<<<grid, kTeams * kTeamThreads, kEncSharedBytes, st>>>(A);
  return cudaGetLastError() == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
}

// Argument checks of the single-tensor encoders.
static qlc_status check_encode(const uint8_t* d_in, size_t n, const qlc_lut* d_lut, uint32_t chunk_symbols,
                               const uint8_t* d_out, size_t out_cap, const void* d_ws, size_t ws_bytes,
                               const uint64_t* d_out_bytes, const uint32_t* d_status) {
  if (!d_lut || !d_out || !d_out_bytes || (n > 0 && (!d_in || !d_ws))) return QLC_ERR_ARG;
  if (!chunk_symbols_ok(chunk_symbols)) return QLC_ERR_ARG;
  if (!aligned(d_in, 16) || !aligned(d_out, 16) || !aligned(d_lut, 16) || !aligned(d_ws, 16) ||
      !aligned(d_out_bytes, 8) || !aligned(d_status, 4))
    return QLC_ERR_ARG;
  if ((n + chunk_symbols - 1) / chunk_symbols > 0xFFFFFFFFull) return QLC_ERR_ARG;
  if (out_cap < qlc_encoded_size(n, chunk_symbols)) return QLC_ERR_CAPACITY;
  if (n > 0 && ws_bytes < qlc_encode_workspace_size(n, chunk_symbols)) return QLC_ERR_CAPACITY;
  return QLC_OK;
}

// Launches the encoder behind the histogram of the same call, building the LUT
// from it (hist), or with the caller's LUT (hist NULL).  Look-back words are
// cleared by the caller where clear_lookback says so.
static bool looks_back(size_t n, uint32_t cs) { return (n + cs - 1) / cs > kPartMaxChunks; }
static qlc_status clear_lookback(size_t n, uint32_t cs, void* d_ws, cudaStream_t st) {
  if (!looks_back(n, cs)) return QLC_OK;
  return cudaMemsetAsync(d_ws, 0, qlc_encode_workspace_size(n, cs), st) == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
}
static qlc_status launch_encode(const uint8_t* d_in, size_t n, const uint64_t* d_hist, const SchemeSet& set, qlc_lut* d_lut,
                                uint32_t cs, uint8_t* d_out, size_t out_cap, void* d_ws, size_t ws_bytes,
                                uint64_t* d_out_bytes, uint32_t* d_status, cudaStream_t st) {
  unsigned long long* ob = reinterpret_cast<unsigned long long*>(d_out_bytes);
  const unsigned long long* hist = reinterpret_cast<const unsigned long long*>(d_hist);
  const uint64_t n_chunks = (n + cs - 1) / cs;
  if (n > 0 && !looks_back(n, cs)) {
    const int sms = sm_count(), parts = (int)(n_groups_of(n_chunks) * kParts);
    const int want = (int)((n_chunks + kPartWarps - 1) / kPartWarps), grid = want < 6 * sms ? want : 6 * sms;
    if (hist)
      launch_after(lengths_kernel<true>, grid, kPartThreads, 0, st, d_in, n, hist, set, d_lut, cs, d_out, d_status);
    else
      lengths_kernel<false><<<grid, kPartThreads, 0, st>>>(d_in, n, nullptr, set, d_lut, cs, d_out, d_status);
    if (cudaGetLastError() != cudaSuccess) return QLC_ERR_CUDA;
    launch_after(pack_kernel, parts < kPackCtasPerSm * sms ? parts : kPackCtasPerSm * sms, kPartThreads, 0, st, d_in, n, d_lut,
                 cs, d_out, out_cap, ob, d_status);
    return cudaGetLastError() == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
  }
  if (hist) {
    const qlc_status s = launch_luts(d_hist, 1, set, d_lut, n > 0, st);
    if (s != QLC_OK) return s;
  }
  if (n == 0) {
    header_only_kernel<<<1, 256, 0, st>>>(d_out, cs, d_lut, ob);
    return cudaGetLastError() == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
  }
  EncArgs A = {};
  A.in = d_in;
  A.n = n;
  A.lut = d_lut;
  A.out = d_out;
  A.out_bytes = ob;
  A.n_items = n_groups_of(n_chunks);
  A.cs = cs;
  A.ticket = static_cast<unsigned int*>(d_ws);
  A.gstat = reinterpret_cast<unsigned long long*>(static_cast<uint8_t*>(d_ws) + 16);
  A.status = d_status;
  A.out_cap = out_cap;
  A.gstat_cap = (ws_bytes - 16) / 8;
  return launch_groups(A, A.n_items, nullptr, hist != nullptr, st);
}

qlc_status qlc_encode(const uint8_t* d_in, size_t n, const qlc_lut* d_lut, uint32_t chunk_symbols,
                      uint8_t* d_out, size_t out_cap, void* d_ws, size_t ws_bytes,
                      uint64_t* d_out_bytes, uint32_t* d_status, qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_encode");
  qlc_status s = check_encode(d_in, n, d_lut, chunk_symbols, d_out, out_cap, d_ws, ws_bytes, d_out_bytes, d_status);
  if (s != QLC_OK) return s;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  s = clear_lookback(n, chunk_symbols, d_ws, st);
  if (s != QLC_OK) return s;
  SchemeSet none;
  none.count = 0;
  return launch_encode(d_in, n, nullptr, none, const_cast<qlc_lut*>(d_lut), chunk_symbols, d_out, out_cap, d_ws, ws_bytes,
                       d_out_bytes, d_status, st);
}

qlc_status qlc_encode_tensor(const uint8_t* d_in, size_t n, const qlc_scheme* h_schemes, int n_schemes,
                             uint32_t chunk_symbols, uint64_t* d_hist, qlc_lut* d_lut, uint8_t* d_out, size_t out_cap,
                             void* d_ws, size_t ws_bytes, uint64_t* d_out_bytes, uint32_t* d_status,
                             qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_encode_tensor");
  SchemeSet set;
  if (!d_hist || !aligned(d_hist, 8) || !scheme_set(h_schemes, n_schemes, &set)) return QLC_ERR_ARG;
  qlc_status s = check_encode(d_in, n, d_lut, chunk_symbols, d_out, out_cap, d_ws, ws_bytes, d_out_bytes, d_status);
  if (s != QLC_OK) return s;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (n > 0 && n <= (size_t)kOneChunks * chunk_symbols) {
    static OncePerContext done;
    if (!smem_ok(encode_one_kernel, sizeof(OneShared), done)) return QLC_ERR_CUDA;
    encode_one_kernel<<<1, kHcThreads, sizeof(OneShared), st>>>(
        d_in, (uint32_t)n, set, chunk_symbols, reinterpret_cast<unsigned long long*>(d_hist), d_lut, d_out, out_cap,
        reinterpret_cast<unsigned long long*>(d_out_bytes));
    return cudaGetLastError() == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
  }
  s = clear_lookback(n, chunk_symbols, d_ws, st);  // before the kernels, which then follow one another directly
  if (s == QLC_OK) s = launch_histogram(d_in, n, d_hist, 0, st);
  if (s != QLC_OK) return s;
  return launch_encode(d_in, n, d_hist, set, d_lut, chunk_symbols, d_out, out_cap, d_ws, ws_bytes, d_out_bytes, d_status,
                       st);
}

int qlc_test_encode_ctas(const qlc_launch* h_launch) { return encode_ctas(h_launch); }

void qlc_test_encode_smem(uint32_t* addr, uint32_t* size, uint32_t* requested) {
  *addr = kTableAddr;
  *size = (uint32_t)sizeof(EncShared);
  *requested = (uint32_t)kEncSharedBytes;
}

qlc_status qlc_test_encode_stalled_lookback(const uint8_t* d_in, size_t n, const qlc_lut* d_lut,
                                            uint32_t chunk_symbols, uint8_t* d_out, size_t out_cap,
                                            void* d_ws, size_t ws_bytes, uint64_t* d_out_bytes,
                                            uint32_t* d_status, qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_test_encode_stalled_lookback");
  if (!d_in || !d_lut || !d_out || !d_ws || !chunk_symbols_ok(chunk_symbols)) return QLC_ERR_ARG;
  if (!aligned(d_in, 16) || !aligned(d_out, 16) || !aligned(d_lut, 16) || !aligned(d_ws, 16) ||
      !aligned(d_out_bytes, 8) || !aligned(d_status, 4))
    return QLC_ERR_ARG;
  const uint64_t n_chunks = (n + chunk_symbols - 1) / chunk_symbols;
  if (n_groups_of(n_chunks) < 2) return QLC_ERR_ARG;
  if (out_cap < qlc_encoded_size(n, chunk_symbols)) return QLC_ERR_CAPACITY;
  const size_t ws_need = qlc_encode_workspace_size(n, chunk_symbols);
  if (ws_bytes < ws_need) return QLC_ERR_CAPACITY;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (cudaMemsetAsync(d_ws, 0, ws_need, st) != cudaSuccess) return QLC_ERR_CUDA;
  if (cudaMemsetAsync(d_ws, 1, 1, st) != cudaSuccess) return QLC_ERR_CUDA;  // group counter = 1
  EncArgs A = {};
  A.in = d_in;
  A.n = n;
  A.lut = d_lut;
  A.out = d_out;
  A.out_bytes = reinterpret_cast<unsigned long long*>(d_out_bytes);
  A.n_items = n_groups_of(n_chunks);
  A.cs = chunk_symbols;
  A.ticket = static_cast<unsigned int*>(d_ws);
  A.gstat = reinterpret_cast<unsigned long long*>(static_cast<uint8_t*>(d_ws) + 16);
  A.status = d_status;
  A.out_cap = out_cap;
  A.gstat_cap = (ws_bytes - 16) / 8;
  return launch_groups(A, A.n_items, nullptr, false, st);
}

qlc_status qlc_encode_batch(const qlc_desc* d_descs, int n_shards, uint32_t chunk_symbols, void* d_ws,
                            size_t ws_bytes, uint32_t* d_status, const qlc_launch* h_launch,
                            qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_encode_batch");
  if (!d_descs || n_shards < 1 || !d_ws || !chunk_symbols_ok(chunk_symbols)) return QLC_ERR_ARG;
  if (!aligned(d_ws, 16) || !aligned(d_descs, 16) || !aligned(d_status, 4)) return QLC_ERR_ARG;
  BatchWs w;
  if (!batch_ws_layout(d_ws, ws_bytes, n_shards, &w)) return QLC_ERR_CAPACITY;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (!launch_plan(kPlanEncode, d_descs, n_shards, chunk_symbols, w, d_status, st)) return QLC_ERR_CUDA;
  EncArgs A = {};
  A.descs = d_descs;
  A.item_base = w.item_base;
  A.n_shards = n_shards;
  A.cs = chunk_symbols;
  A.ticket = w.ticket;
  A.gstat = w.gstat;
  A.status = d_status;
  A.gstat_cap = w.gstat_cap;
  // the item count is only known on the device: launch the full resident grid
  return launch_groups(A, ~0ull, h_launch, true, st);
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Encoding without any device allocation by the caller or the library.
//
// Some callers cannot allocate device memory: a plugin running inside a host
// framework whose allocator owns all of the GPU's memory, or a request path
// that must not call cudaMalloc (which can synchronise the device).  For them
// the look-back state that qlc_encode keeps in a caller-provided workspace
// lives instead in this file-scope device array, sized for up to
// kNoAllocMaxGroups groups of 32 chunks.  Every GPU that loads the library
// holds these bytes until the process exits.
namespace qlc {
constexpr uint64_t kNoAllocMaxGroups = 65536;
constexpr size_t kNoAllocScratchBytes = 16 + 8 * kNoAllocMaxGroups;  // 512 KiB + 16 B
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

// Device address of g_noalloc_scratch in the current device's context (the
// host-side symbol is not a device address).  It is looked up with the
// device current on the first call, and again whenever the device's context
// has changed since (a reset destroys the old context, and the array moves
// with the new one); without a context id from the driver it is looked up
// on every call.  The cache is shared by all host threads and guarded by a
// mutex.
static void* noalloc_scratch_ptr(qlc_status* err) {
  static std::mutex mu;
  static std::unordered_map<int, std::pair<unsigned long long, void*>> cache;  // device -> (context id, address)
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    *err = QLC_ERR_CUDA;
    return nullptr;
  }
  const unsigned long long id = current_context_id();
  std::lock_guard<std::mutex> lock(mu);
  const auto it = cache.find(dev);
  if (it != cache.end() && id != 0 && it->second.first == id) return it->second.second;
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
    *err = QLC_ERR_CUDA;
    return nullptr;
  }
  // the lookup makes the device's primary context current if none was
  cache[dev] = {current_context_id(), p};
  return p;
}
}  // namespace qlc

extern "C" qlc_status qlc_encode_noalloc(const uint8_t* d_in, size_t n, const qlc_lut* d_lut,
                                          uint32_t chunk_symbols, uint8_t* d_out, size_t out_cap,
                                          uint64_t* d_out_bytes, uint32_t* d_status,
                                          qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_encode_noalloc");
  if (!chunk_symbols_ok(chunk_symbols)) return QLC_ERR_ARG;
  const uint64_t n_chunks = (n + chunk_symbols - 1) / chunk_symbols;
  if (n_groups_of(n_chunks) > kNoAllocMaxGroups) return QLC_ERR_CAPACITY;
  qlc_status err = QLC_OK;
  void* ws = noalloc_scratch_ptr(&err);
  if (!ws) return err;
  // qlc_encode clears the part of the array it uses before its kernel runs.
  return qlc_encode(d_in, n, d_lut, chunk_symbols, d_out, out_cap, ws, kNoAllocScratchBytes,
                    d_out_bytes, d_status, stream);
}

namespace qlc {
QLC_DEFINE_CHECK_TAKE(check_take_encode)
}  // namespace qlc
