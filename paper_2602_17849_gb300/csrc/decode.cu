// decode.cu -- QLC decoder (Section 7) for container v1.
//
// A container is decoded in one of two ways, which decode_span.cuh chooses: split,
// where each chunk is cut into pieces that lanes decode beside one another
// (decode_span.cuh), or, in this file, a warp per group of 32 chunks with a lane
// per chunk: each lane starts at its chunk's bit offset (group offset + exclusive
// scan of the group's chunk_bits) and decodes its chunk serially.  Per symbol: the
// top 3 bits of a 32-bit window are the area code; the code length 3 + bits[area]
// comes from a byte permute of two registers (no memory access); the whole
// codeword (area code and suffix, right-aligned) indexes a 2048-entry code ->
// symbol table in shared memory built from the LUT and the area table.  The rank
// is never formed explicitly: for every code of every area the table holds
// dec[offset + suffix] (offset 0 for 8-bit areas), exactly the paper's rule.
// Input: each lane's bytes arrive by cp.async in 16-byte vectors into a
// staging ring, and once per block of 32 symbols the lane moves the vectors it
// will need next, byte-swapped, into its column of a word ring (word k of lane
// l in bank l, so the lanes' reads never collide).  The lane decodes from a
// 64-bit register buffer: two symbols per round from the 32-bit window at its
// bit position (one funnel shift); when the position crosses a word the
// buffer moves up and the next word comes from the ring, read one word ahead
// of its use so that no memory access lies on the round-to-round chain.
// Output: symbols by one 32-byte streaming store per lane and block; values
// through a tile in shared memory, so that a store covers few lines.
// Work is dealt out so that every SM, and every quarter of one, has the same
// share: a container by one CTA per SM (decode_kernel), batches in three ways
// (decode_few_kernel, decode_batch_kernel).
//
// 256 Mi symbols, t4: 168 us (180 with a CTA per warp); bound by the integer
// pipe, the shared-memory pipe (table lookups by random codes) and, with 13.5
// groups per SM, by the chain of a lane's own rounds.  1152 tensors (3.4 GB)
// 1757 us.
#define QLC_FILE_ID 1
#include "decode_common.cuh"
#include "decode_span.cuh"
#include "../../include/qlc_testing.h"

namespace qlc {

constexpr int kDecCtasPerSm = 20;  // 20 x (8.3 KB + 1 KB reserved); at 24 the register cap (80) spills
// cp.async (global -> shared, 16 bytes, bypassing L1) and its groups.
__device__ __forceinline__ void cp_async16(uint32_t smem, const void* g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

constexpr uint32_t kBlk = 32;       // symbols per lane per block
constexpr uint32_t kStageVec = 8;   // 16-byte vectors staged per lane (128 B of its stream)
constexpr uint32_t kColRows = 16;   // words in each lane's column ring

// How a lane reads its column ring: in shared memory at a constant address, or
// at an address in registers, which costs no add when the ring is aligned to
// its 2 KB (kRingMany, kRingFew; the latter for few warps per SM, see step_to).
enum Ring { kRingStatic, kRingMany, kRingFew };
constexpr uint32_t kRingBytes = kColRows * 128;

// Shared memory of one warp decoding a group: the lanes' staging ring and
// column ring.
struct LaneShared {
  uint32_t col[kColRows][32];  // word k of lane l at col[k % 16][l]
  uint4 stage[kStageVec][32];  // vector v of lane l at stage[v % 8][l]
};
// ... and of a CTA of one such warp: with its code table and header.
struct DecShared {
  LaneShared lanes;
  uint8_t T[2048];                // code -> symbol
  __align__(16) uint8_t hdr[kIndexOff];  // the container's header and dec
  uint32_t seen[64];
};

// A lane's bit stream, positions group-relative.  The stream's words j and
// j + 1 sit in a 64-bit buffer (hi:lo, most significant bit first) and word
// j + 2 in nxt, where j = p / 32; the window at bit p is one funnel shift of
// the buffer.  When a round crosses into the next word the buffer moves up
// by one word and word j + 3 is read from the column ring, so no memory
// access lies on the chain from one round to the next.
struct LaneDec {
  uint32_t p;      // bit position of the next codeword
  uint32_t hi, lo, nxt;
  uint32_t tv;     // next vector to move from the staging ring to the column ring
  uint32_t fv;     // next vector to fetch
  uint32_t vend;   // vectors of this stream in the group
  uint64_t vlim;   // vectors from the group's start to the end of the container (checked build)
  const uint4* gp; // the group's payload
  uint32_t lane4;      // byte offset of col[0][lane] in the column ring
  uint32_t col_s;      // shared address of col[0][lane]
  uint32_t stage_s;    // shared address of stage[0][lane]

  // Fetches (cp.async, 16 bytes each) vector fv into its staging slot when
  // fv < want, k times, with no branch; the caller commits the group.
  template <int k>
  __device__ __forceinline__ void fetch(uint32_t want) {
#pragma unroll
    for (int i = 0; i < k; i++) {
      const uint32_t q = fv < want && QLC_GUARD(fv < vlim, nullptr);
      asm volatile(
          "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q cp.async.cg.shared.global [%0], [%1], 16;\n\t}" ::"r"(
              stage_s + (fv % kStageVec) * 512),
          "l"(gp + fv), "r"(q)
          : "memory");
      fv += q;
    }
  }
  // Moves vector tv from the staging ring to the column ring (byte-swapped,
  // so each word reads most significant bit first) when its first word is
  // at most `need` and it exists.
  __device__ __forceinline__ void move(uint32_t need) {
    const uint32_t q = (tv * 4 <= need) & (tv < vend);
    const uint32_t src = stage_s + (tv % kStageVec) * 512;
    const uint32_t dst = col_s + (tv % 4) * 512;
      asm volatile(
          "{\n\t.reg .pred q;\n\t.reg .b32 a, b, c, d;\n\t"
          "setp.ne.u32 q, %2, 0;\n\t"
          "@q ld.shared.v4.u32 {a, b, c, d}, [%0];\n\t"
          "prmt.b32 a, a, 0, 0x0123;\n\t"
          "prmt.b32 b, b, 0, 0x0123;\n\t"
          "prmt.b32 c, c, 0, 0x0123;\n\t"
          "prmt.b32 d, d, 0, 0x0123;\n\t"
          "@q st.shared.u32 [%1], a;\n\t"
          "@q st.shared.u32 [%1+128], b;\n\t"
          "@q st.shared.u32 [%1+256], c;\n\t"
          "@q st.shared.u32 [%1+384], d;\n\t"
          "}" ::"r"(src),
          "r"(dst), "r"(q)
          : "memory");
    tv += q;
  }
  template <Ring kRing>
  __device__ __forceinline__ uint32_t ring(const LaneShared& sm, uint32_t k) const {
    if constexpr (kRing == kRingStatic) {
      return *reinterpret_cast<const uint32_t*>(reinterpret_cast<const uint8_t*>(sm.col) + (((k << 7) & 0x780u) | lane4));
    } else {
      uint32_t v;
      asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(((k << 7) & 0x780u) | col_s) : "memory");
      return v;
    }
  }
  // Set-up at bit S of the group: fill the staging ring, wait for it, move
  // the words the first block can read, load the buffer, refill.  Words
  // j .. j + 2 (at most two vectors) go to the buffer before the rest is
  // moved: the ring holds 16 words, and word j + 16 shares word j's row.
  template <Ring kRing>
  __device__ __forceinline__ void start(const LaneShared& sm, uint32_t S) {
    p = S;
    tv = fv = min(S >> 7, vend);
    fetch<kStageVec>(min(tv + kStageVec, vend));
    cp_async_commit();
    cp_async_wait<0>();
    const uint32_t j = S >> 5;
    move(j + 2);
    move(j + 2);
    hi = ring<kRing>(sm, j);
    lo = ring<kRing>(sm, j + 1);
    nxt = ring<kRing>(sm, j + 2);
#pragma unroll
    for (int i = 0; i < 3; i++) move(j + 13);
    fetch<5>(min(tv + kStageVec, vend));
    cp_async_commit();
  }
  // Before each block of at most 32 symbols (at most 352 bits, so the ring
  // is read up to word p/32 + 13): move up to three vectors (the position
  // moved at most 11 words since the last block) and refetch as many.
  // Vectors moved now were fetched two blocks ago at the latest, so waiting
  // for all but the latest cp.async group suffices.
  __device__ __forceinline__ void advance() {
    cp_async_wait<1>();
    const uint32_t need = (p >> 5) + 13;
#pragma unroll
    for (int i = 0; i < 3; i++) move(need);
    fetch<3>(min(tv + kStageVec, vend));
    cp_async_commit();
  }
  // Advances the position to pn (less than 32 bits on): when it crosses into
  // the next word the buffer moves up a word and the word after nxt is read.
  // With kRingFew as predicated instructions, which shortens the chain of a
  // warp that has a quarter of an SM nearly to itself (16 Mi equal symbols 85
  // -> 79 us, 1814 groups of a batch 167 -> 161 us); the compiler's form issues
  // less, which counts with many warps (256 Mi symbols 181 us, not 188).
  template <Ring kRing>
  __device__ __forceinline__ void step_to(const LaneShared& sm, uint32_t pn) {
    if constexpr (kRing == kRingFew) {
      asm volatile(
          "{\n\t.reg .pred q;\n\t.reg .b32 t;\n\t"
          "xor.b32 t, %3, %4;\n\t"
          "and.b32 t, t, 32;\n\t"
          "setp.ne.u32 q, t, 0;\n\t"
          "@q mov.b32 %0, %1;\n\t"
          "@q mov.b32 %1, %2;\n\t"
          "@q ld.shared.u32 %2, [%5];\n\t"
          "}"
          : "+r"(hi), "+r"(lo), "+r"(nxt)
          : "r"(pn), "r"(p), "r"((((pn << 2) + 256u) & 0x780u) | col_s)  // row (pn / 32 + 2) % 16
          : "memory");
    } else if ((pn ^ p) & 32u) {
      hi = lo;
      lo = nxt;
      nxt = ring<kRing>(sm, (pn >> 5) + 2);
    }
    p = pn;
  }
  // Two symbols (at most 22 bits) from the window, packed as s0 | s1 << 8.
  template <Ring kRing>
  __device__ __forceinline__ uint32_t round2(const LaneShared& sm, const uint8_t* T, uint32_t len_lo, uint32_t len_hi) {
    const uint32_t x = __funnelshift_l(lo, hi, p);
    const uint32_t la = code_len(x, len_lo, len_hi);
    const uint32_t ia = __funnelshift_l(x, 0u, la);
    const uint32_t a = QLC_GUARD(ia < 2048u, nullptr) ? (uint32_t)T[ia] : 0u;
    const uint32_t x2 = x << la;
    const uint32_t lb = code_len(x2, len_lo, len_hi);
    const uint32_t ib = __funnelshift_l(x2, 0u, lb);
    const uint32_t b = QLC_GUARD(ib < 2048u, nullptr) ? (uint32_t)T[ib] : 0u;
    step_to<kRing>(sm, p + la + lb);
    return mad_lo(b, 256u, a);
  }
  // One symbol (ragged chunk ends only).
  template <Ring kRing>
  __device__ __forceinline__ uint32_t round1(const LaneShared& sm, const uint8_t* T, uint32_t len_lo, uint32_t len_hi) {
    const uint32_t x = __funnelshift_l(lo, hi, p);
    const uint32_t la = code_len(x, len_lo, len_hi);
    const uint32_t ia = __funnelshift_l(x, 0u, la);
    const uint32_t a = QLC_GUARD(ia < 2048u, nullptr) ? (uint32_t)T[ia] : 0u;
    step_to<kRing>(sm, p + la);
    return a;
  }
};

// Streaming 32-byte store (dst 32-byte aligned) or two 16-byte stores.
__device__ __forceinline__ void st_cs_32(uint8_t* dst, const uint32_t w[8], bool aligned32) {
  if (aligned32) {
    asm volatile("st.global.cs.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(dst), "r"(w[0]), "r"(w[1]),
                 "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
  } else {
    asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                 : "memory");
    asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(dst + 16), "r"(w[4]), "r"(w[5]), "r"(w[6]),
                 "r"(w[7])
                 : "memory");
  }
}

// One block of 32 symbols of each of the group's 32 chunks (all of them whole)
// as values: the lanes' words pass through a tile (at shared address
// tile_s, a multiple of 1 KB; word k of lane l is word 32 k + (l ^ 4 k): no two
// lanes of a write or a read share a bank), so that
// eight lanes write the 128 (or 64) bytes of a chunk's block and a store covers
// 4 lines.  With each lane writing its own block in pieces of 32 bytes a store
// touched 32 lines, and those stores were half of the L1 data pipe's work (256
// Mi fp32 values 328 us).  first: index of the first chunk's block in the
// tensor; sc: the scale of this lane's block.
template <int kOut>
__device__ __forceinline__ void put_tile(void* out, uint32_t tile_s, float sc, uint64_t first, uint32_t cs,
                                         const uint32_t w[8], int lane) {
  const uint32_t at = tile_s | 4u * lane;
#pragma unroll
  for (int k = 0; k < 8; k++)
    asm volatile("st.shared.u32 [%0], %1;" ::"r"((at ^ 16u * k) + 128u * k), "r"(w[k]) : "memory");
  __syncwarp();
  const uint32_t j = (uint32_t)lane >> 3, k = (uint32_t)lane & 7u;  // chunk 4 q + j, symbols 4 k ..
  const uint32_t from = tile_s | 128u * k | 16u * k | 4u * j;
  uint32_t v[8];
#pragma unroll
  for (uint32_t q = 0; q < 8; q++) asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v[q]) : "r"(from ^ 16u * q) : "memory");
  constexpr uint32_t kElem = kOut == QLC_DTYPE_F32 ? 4 : 2;
  uint8_t* dst = static_cast<uint8_t*>(out) + (first + j * cs + 4 * k) * kElem;
#pragma unroll
  for (uint32_t q = 0; q < 8; q++)
    put4_values<kOut>(dst + (size_t)(4 * q * cs * kElem), __shfl_sync(0xffffffffu, sc, 4 * q + j), v[q]);
  __syncwarp();
}

// Decodes group g of a validated container (one warp; lane = chunk).  With
// out_slot the output pointer is read from that shared word at each block
// instead of out: a pointer that is not a kernel parameter would otherwise
// hold two registers across the decoding loop, which then issued about 10 %
// more instructions (the batch decoder, 124.3 M against 112.8 M on 256 MiB).
template <int kOut, Ring kRing, bool kTile = true>
__device__ __forceinline__ void decode_group(const DecHeader& h, const uint8_t* __restrict__ in, void* __restrict__ out,
                             const float* __restrict__ scales, uint64_t g, LaneShared& sm, const uint8_t* T, LaneDec& d,
                             uint32_t* status, int lane, bool aligned32, bool sc_vec = false,
                             uint32_t tile_s = 0, void* const volatile* out_slot = nullptr) {
  const unsigned long long* group_off = reinterpret_cast<const unsigned long long*>(in + kIndexOff);
  const uint16_t* chunk_bits = reinterpret_cast<const uint16_t*>(in + kIndexOff + 8 * h.n_groups);
  const uint4* vbase = reinterpret_cast<const uint4*>(in + h.P);
  const uint32_t cs = h.cs;
  const uint32_t len_lo = h.len_lo, len_hi = h.len_hi;
  const uint64_t c = g * kGroupChunks + lane;
  const bool exists = c < h.n_chunks;
  const uint32_t nsym = exists ? (uint32_t)min((uint64_t)cs, h.n - c * cs) : 0u;
  const uint32_t bits =
      exists && QLC_GUARD(kIndexOff + 8 * h.n_groups + 2 * (c + 1) <= h.in_bytes, status) ? chunk_bits[c] : 0u;
  uint32_t incl = bits;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const uint32_t gbits = __shfl_sync(0xffffffffu, incl, 31);
  const uint64_t goff = QLC_GUARD(kIndexOff + 8 * (g + 1) <= h.in_bytes, status) ? group_off[g] : 0ull;
  const uint64_t gnext = g + 1 < h.n_groups
                             ? (QLC_GUARD(kIndexOff + 8 * (g + 2) <= h.in_bytes, status) ? group_off[g + 1] : 0ull)
                             : h.payload_bytes;
  const bool group_ok = (g != 0 || goff == 0) && (goff & 15u) == 0 && goff <= gnext &&
                        gnext <= h.payload_bytes && gnext - goff == align16((gbits + 7u) / 8u);
  if (!group_ok) {
    if (lane == 0) set_status(status, QLC_ERR_CORRUPT);
    return;
  }
  // lane start bit (group-relative) and ring set-up
  const uint32_t S = incl - bits;
  d.gp = vbase + goff / 16;
  d.vend = (uint32_t)((gnext - goff) / 16);
  d.vlim = (h.in_bytes - h.P - goff) / 16;  // goff <= payload_bytes <= in_bytes - P (validated)
  d.template start<kRing>(sm, S);
  const uint64_t i_chunk = c * cs;  // the chunk's first symbol
  const uint32_t nmax = __reduce_max_sync(0xffffffffu, nsym);
  // dequantising outputs: the scales of the chunk's whole blocks, four per
  // 16-byte load (a lane's loads hit lines of their own, so four scales per
  // load cut the load traffic of the L1 data pipe fourfold), each four
  // loaded four blocks before their use
  const uint32_t nfull = nsym / kBlk;
  const float* sc_chunk = kOut != kOutCodes ? scales + i_chunk / 32 : nullptr;
  auto scales4 = [&](uint32_t q) {  // scales of whole blocks 4q .. 4q + 3 (0 past the last)
    float4 r = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (kOut == kOutCodes) return r;
    if (4 * q + 4 <= nfull && sc_vec) return __ldg(reinterpret_cast<const float4*>(sc_chunk + 4 * q));
    if (4 * q < nfull) r.x = sc_chunk[4 * q];
    if (4 * q + 1 < nfull) r.y = sc_chunk[4 * q + 1];
    if (4 * q + 2 < nfull) r.z = sc_chunk[4 * q + 2];
    if (4 * q + 3 < nfull) r.w = sc_chunk[4 * q + 3];
    return r;
  };
  float4 sc_cur = make_float4(0.0f, 0.0f, 0.0f, 0.0f), sc_nxt = scales4(0);
  for (uint32_t i0 = 0; i0 < nmax; i0 += kBlk) {
    d.advance();
    const uint32_t b = i0 / kBlk;  // the same block index in every lane
    if (kOut != kOutCodes && (b & 3u) == 0) {
      sc_cur = sc_nxt;
      sc_nxt = scales4(b / 4 + 1);
    }
    const float sc = (b & 3u) == 0 ? sc_cur.x : (b & 3u) == 1 ? sc_cur.y : (b & 3u) == 2 ? sc_cur.z : sc_cur.w;
    const uint32_t cnt = nsym > i0 ? min(kBlk, nsym - i0) : 0u;
    void* o = out_slot ? *out_slot : out;
    const bool whole = kOut != kOutCodes && kTile && __all_sync(0xffffffffu, cnt == kBlk);
    if (cnt == kBlk) {
      uint32_t w[8];
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const uint32_t p0 = d.template round2<kRing>(sm, T, len_lo, len_hi);
        const uint32_t p1 = d.template round2<kRing>(sm, T, len_lo, len_hi);
        w[j] = __byte_perm(p0, p1, 0x5410);
      }
      if constexpr (kOut == kOutCodes) {
        if (QLC_GUARD(i_chunk + i0 + kBlk <= h.out_cap, status)) st_cs_32(static_cast<uint8_t*>(o) + i_chunk + i0, w, aligned32);
      } else if (whole) {
        if (QLC_GUARD(g * kGroupChunks * cs + 31ull * cs + i0 + kBlk <= h.out_cap, status))
          put_tile<kOut>(o, tile_s, sc, g * kGroupChunks * cs + i0, cs, w, lane);
      } else if (QLC_GUARD(i_chunk + i0 + kBlk <= h.out_cap, status)) {  // a tensor's last group
        constexpr uint32_t kElem = kOut == QLC_DTYPE_F32 ? 4 : 2;
#pragma unroll
        for (uint32_t j = 0; j < 8; j++)
          put4_values<kOut>(static_cast<uint8_t*>(o) + (i_chunk + i0 + 4 * j) * kElem, sc, w[j]);
      }
    } else {
      for (uint32_t k = 0; k < cnt; k++) {
        const uint32_t sym = d.template round1<kRing>(sm, T, len_lo, len_hi);
        if (QLC_GUARD(i_chunk + i0 + k < h.out_cap, status)) put1<kOut>(o, scales, i_chunk + i0 + k, sym);
      }
    }
  }
  cp_async_wait<0>();
  if (exists && d.p - S != bits) set_status(status, QLC_ERR_CORRUPT);
}

// Lane set-up shared by the kernels; false if the staging ring's vectors are not
// on 16 bytes.  Column rings that are addressed in registers lie on their own
// size by construction (ring_aligned, and the sizes that are asserted there); a
// check of that here cost 24 shards 1.2 of 165 us.
__device__ __forceinline__ bool lane_init(LaneShared& sm, LaneDec& d, int lane) {
  d.lane4 = 4u * lane;
  d.col_s = (uint32_t)__cvta_generic_to_shared(&sm.col[0][lane]);
  d.stage_s = (uint32_t)__cvta_generic_to_shared(&sm.stage[0][lane]);
  return (__cvta_generic_to_shared(sm.stage) & 15u) == 0;
}

// One container: one CTA per SM of up to dec_warps warps, which validate the header and
// build the code table once, then decode spans (decode_span.cuh) where that
// pays and else groups, a lane per chunk.  Spans and groups are dealt out warp
// by warp over the SMs, so that every SM, and every quarter of an SM, has the
// same number of them, give or take one.  (With a CTA per warp or per four, the
// block scheduler puts up to 16 of 2048 working warps on some SMs, unless the
// grid is as large as the groups; the host, which does not know the chunk,
// could then be four times off: 50 Mi symbols in chunks of 1024 took 85 us.)
constexpr int dec_warps(int out) { return out == kOutCodes ? 20 : 16; }  // 96 or 128 registers: values spill at 96
struct LaneWarp {  // a warp that decodes groups
  LaneShared lanes;
  uint32_t tile[256];
  uint8_t pad[1024];
};
static_assert(sizeof(LaneWarp) % kRingBytes == 0 && sizeof(LaneWarp) <= sizeof(SpanWarp), "");
constexpr size_t one_bytes(int warps) { return warps * sizeof(SpanWarp) + kRingBytes; }
// The first address at or after p that a column ring can have.
__device__ __forceinline__ uint8_t* ring_aligned(uint8_t* p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  return p + ((kRingBytes - a % kRingBytes) % kRingBytes);
}
template <int kOut>
__global__ void __launch_bounds__(32 * dec_warps(kOut), 1)
decode_kernel(const uint8_t* __restrict__ in, uint64_t in_bytes, void* __restrict__ out,
              const float* __restrict__ scales, uint64_t out_cap, unsigned long long* __restrict__ n_out,
              uint32_t* __restrict__ status) {
  constexpr int kWarps = dec_warps(kOut);
  extern __shared__ __align__(16) uint8_t one_sm[];
  __shared__ uint8_t T[2048];                       // code -> symbol
  __shared__ __align__(16) uint8_t hdr[kIndexOff];  // the container's header and dec
  __shared__ uint32_t seen[kWarps][64], s_slow;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // so known to be the same in all lanes
  const uint32_t warps = blockDim.x / 32;
  load_header(in, in_bytes, hdr, tid, blockDim.x);
  __syncthreads();
  DecHeader h;
  const uint32_t err = parse_header(hdr, in_bytes, out_cap, &h, seen[warp], lane);
  if (blockIdx.x == 0 && tid == 0) {
    if (!err || err == QLC_ERR_CAPACITY) *n_out = h.n;
    if (err) set_status(status, err);
  }
  if (err) return;
  const SplitData sd = {h.cs, h.len_lo, h.len_hi, h.n, h.payload_bytes};
  constexpr SplitInto kInto = kOut == kOutCodes ? kSplitCodes : kSplitValues;
  const bool ask = split_samples(sd, kInto, h.n);
  if (ask && warp == 0) {  // every CTA looks at the same samples
    static_assert(kSamples == 32 && 4 * 32 * kSampleWords <= sizeof(SpanWarp), "a sample per lane");
    const bool slow = sample_is_slow(in, sd, h.n_chunks, lane, reinterpret_cast<uint32_t*>(one_sm) + lane * kSampleWords);
    const unsigned all = __ballot_sync(0xffffffffu, slow);
    if (lane == 0) s_slow = __popc(all);
  }
  build_table(hdr, T, tid, blockDim.x);
  __syncthreads();
  const uint32_t first = (uint32_t)warp * gridDim.x + blockIdx.x;
  if (h.n <= split_most(sd, kInto, ask ? s_slow : 0)) {
    const uint32_t stride = warps * gridDim.x;
    const SpanShape shape(h.cs);
    const uint32_t warm = warm_bits(h.len_lo, h.len_hi);
    const uint32_t k = (uint32_t)lane / shape.lanes, seg = (uint32_t)lane - k * shape.lanes;
    // span s is span r of group g; the step to the warp's next span is made in both
    const uint32_t dg = stride / shape.per_group, dr = stride % shape.per_group;
    uint64_t g = first / shape.per_group;
    uint32_t r = first % shape.per_group;
    while (g < h.n_groups) {
      decode_span<kOut>(h, shape, in, out, scales, g, r * shape.chunks, k, seg, reinterpret_cast<SpanWarp*>(one_sm)[warp], T,
                        warm, status, lane);
      g += dg;
      r += dr;
      if (r >= shape.per_group) {
        r -= shape.per_group;
        g++;
      }
    }
    return;
  }
  LaneWarp& sm = reinterpret_cast<LaneWarp*>(ring_aligned(one_sm))[warp];
  LaneDec d;
  if (!lane_init(sm.lanes, d, lane)) {
    if (lane == 0) set_status(status, QLC_ERR_CUDA);
    return;
  }
  const bool aligned32 = (reinterpret_cast<uintptr_t>(out) & 31u) == 0;
  const bool sc_vec = (reinterpret_cast<uintptr_t>(scales) & 15u) == 0;  // scales read four at a time
  // as many rounds of groups as the warps need, and no more warps than these
  // rounds need: a last round that is nearly empty costs as much as a full one
  // (200 Mi symbols in chunks of 2048, 3200 groups on 3040 warps: 158 us)
  const uint64_t rounds = (h.n_groups + (uint64_t)warps * gridDim.x - 1) / ((uint64_t)warps * gridDim.x);
  const uint32_t used = (uint32_t)((h.n_groups + rounds * gridDim.x - 1) / (rounds * gridDim.x));
  if ((uint32_t)warp >= used) return;
  const uint32_t stride = used * gridDim.x;
  const uint32_t tile_s = (uint32_t)__cvta_generic_to_shared(sm.tile);
  if (kOut != kOutCodes && kOut != QLC_DTYPE_F32 && used <= 3) {
    // with so few warps what counts is a warp's own chain, which is shorter
    // without the tile for 2-byte values (26 Mi in chunks of 2048 60.6 -> 56 us;
    // at four warps 111 us with it, 126 without)
    for (uint64_t g = first; g < h.n_groups; g += stride)
      decode_group<kOut, kRingFew, false>(h, in, out, scales, g, sm.lanes, T, d, status, lane, aligned32, sc_vec);
  } else if (used <= (kOut == kOutCodes ? 8 : 4)) {
    for (uint64_t g = first; g < h.n_groups; g += stride)
      decode_group<kOut, kRingFew>(h, in, out, scales, g, sm.lanes, T, d, status, lane, aligned32, sc_vec, tile_s);
  } else {
    for (uint64_t g = first; g < h.n_groups; g += stride)
      decode_group<kOut, kRingMany>(h, in, out, scales, g, sm.lanes, T, d, status, lane, aligned32, sc_vec, tile_s);
  }
}

// Shared memory of a team of kSpanWarps warps that decode spans, or groups, of
// one shard.
struct SpanShared {
  union {
    SpanWarp span;
    LaneShared lanes;
  } w[kSpanWarps];
  uint8_t T[2048];                          // code -> symbol
  __align__(16) uint8_t hdr[kIndexOff];     // the container's header and dec
  uint32_t seen[kSpanWarps][64];
};

// ---------------------------------------------------------------- batches
//
// Three ways (plan_kernel decides, on the device): split, where that pays for its
// shards (split_rule.cuh); else a lane per chunk, with a group for every warp dealt
// out evenly while there are no more groups than warps, and above with all groups
// from a counter.

// The shard an item belongs to changed: reads its header and builds its table.
// Reports a bad one and returns its status.
__device__ __forceinline__ uint32_t enter_shard(const qlc_desc& dd, DecHeader* h, uint8_t* hdr, uint8_t* T,
                                                uint32_t* seen, uint32_t* status, int lane) {
  __syncwarp();  // every lane is done with the previous shard's header
  load_header(static_cast<const uint8_t*>(dd.in), dd.in_bytes, hdr, lane, 32);
  __syncwarp();
  const uint32_t err = parse_header(hdr, dd.in_bytes, dd.out_cap, h, seen, lane);
  if (err) {
    if (lane == 0) {
      if (err == QLC_ERR_CAPACITY && dd.out_bytes) *dd.out_bytes = h->n;
      set_status(status, err);
    }
    return err;
  }
  build_table(hdr, T, lane, 32);
  __syncwarp();
  return 0;
}

// Many groups: warps take (shard, group) items from a device counter.  A CTA is
// one warp, so that the table's address is a constant (an add less for every
// lookup than with several tables per CTA: 1152 shards 1764 us, not 1790-1830).
__global__ void __launch_bounds__(32, kDecCtasPerSm)
decode_batch_kernel(const qlc_desc* __restrict__ descs, int n_shards,
                    const unsigned long long* item_base, unsigned int* ticket,
                    uint32_t* __restrict__ status) {
  __shared__ DecShared sm;
  __shared__ void* volatile s_out;  // the current item's output
  dependency_wait();
  if (ticket[kTicketWay] != kWayGroups) return;
  const int lane = threadIdx.x;
  LaneDec d;
  if (!lane_init(sm.lanes, d, lane)) {
    if (lane == 0) set_status(status, QLC_ERR_CUDA);
    return;
  }
  const unsigned long long total = item_base[n_shards];
  int cur = -1, bad = -1;
  DecHeader h;
  // Items t + 1 .. t_end - 1 are taken.  While more than eight per warp are left
  // a warp takes several in a row, mostly of one shard, whose table it then
  // builds once: 48000 groups 3379 -> 3357 us, 25600 in 400 shards 1855 -> 1848;
  // with twice as many at a time the last ones take too long (1897).
  unsigned long long t = 0, t_end = 0;
  while (true) {
    if (++t >= t_end) {
      const uint32_t left = t < total ? (uint32_t)min(total - t, 0xFFFFFFFFull) : 0u;
      const uint32_t k = min(max(left / (4 * gridDim.x), 1u), 4u);
      uint32_t first = 0;
      if (lane == 0) first = atomicAdd(ticket, k);
      t = __shfl_sync(0xffffffffu, first, 0);
      t_end = t + k;
    }
    if (t >= total) break;
    const int sh = shard_of_warp(item_base, n_shards, t, lane);
    if (sh == bad) continue;
    const qlc_desc dd = descs[sh];
    const uint64_t g = t - item_base[sh];
    if (sh != cur) {
      if (enter_shard(dd, &h, sm.hdr, sm.T, sm.seen, status, lane)) {
        bad = sh;
        cur = -1;
        continue;
      }
      cur = sh;
    }
    if (g == 0 && lane == 0 && dd.out_bytes) *dd.out_bytes = h.n;
    const bool aligned32 = (reinterpret_cast<uintptr_t>(dd.out) & 31u) == 0;
    __syncwarp();  // every lane is done with the previous item's output
    if (lane == 0) s_out = dd.out;
    __syncwarp();
    if (g < h.n_groups)
      decode_group<kOutCodes, kRingStatic>(h, static_cast<const uint8_t*>(dd.in), nullptr, nullptr, g, sm.lanes, sm.T, d, status, lane,
                              aligned32, false, 0u, &s_out);
  }
}

// The barrier of a team of kSpanWarps warps within its CTA.
__device__ __forceinline__ void team_sync(int team) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(32 * kSpanWarps) : "memory");
}

// Few groups: one CTA per SM, of up to kFewWarps warps, in teams of kSpanWarps
// where the batch is decoded split.
constexpr int kFewTeams = 5;
constexpr int kFewWarps = kSpanWarps * kFewTeams;
static_assert(kFewWarps == kDecCtasPerSm, "both bounded by qlc_launch.decode_ctas_per_sm");
struct FewOwn {
  LaneShared lanes;
  uint8_t T[2048];
  __align__(16) uint8_t hdr[kRingBytes - 256];  // kIndexOff bytes of it
  uint32_t seen[64];
};
static_assert(sizeof(FewOwn) % kRingBytes == 0, "");
// Shared memory: a SpanShared for every team, or a FewOwn for every warp, behind
// what aligns it.
constexpr size_t few_bytes(int warps) {
  const size_t teams = (size_t)(warps / kSpanWarps) * sizeof(SpanShared), own = warps * sizeof(FewOwn);
  return (teams > own ? teams : own) + kRingBytes;
}
__global__ void __launch_bounds__(32 * kFewWarps, 1)
decode_few_kernel(const qlc_desc* __restrict__ descs, int n_shards, const unsigned long long* item_base,
                  unsigned int* ticket, uint32_t* __restrict__ status) {
  extern __shared__ __align__(16) uint8_t few_sm[];
  __shared__ void* volatile s_out[kFewWarps];  // the warps' current outputs
  __shared__ volatile unsigned long long s_item[kFewTeams];
  dependents_may_start();
  dependency_wait();
  const uint32_t way = ticket[kTicketWay];
  const uint64_t batch_symbols = ticket[kTicketSymbols];
  const uint32_t batch_slow = ticket[kTicketSlow];
  if (way == kWayGroups) return;
  const int lane = threadIdx.x % 32;
  const int wid = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0);  // so known to be the same in all lanes
  const unsigned long long total = item_base[n_shards];
  DecHeader h;
  if (way == kWayEven) {
    // A group for every warp at most: item t goes to warp t / SMs of SM t mod
    // SMs, so every SM, and every quarter of an SM, has the same number, give
    // or take one.  From the counter, the CTAs that an SM got first took items
    // that others lacked: 24 shards of 4 KiB - 64 MiB (1814 groups) 256 us,
    // now 165.
    const unsigned long long t = (unsigned long long)wid * gridDim.x + blockIdx.x;
    if (t >= total) return;
    FewOwn& sm = reinterpret_cast<FewOwn*>(ring_aligned(few_sm))[wid];
    LaneDec d;
    if (!lane_init(sm.lanes, d, lane)) {
      if (lane == 0) set_status(status, QLC_ERR_CUDA);
      return;
    }
    const int sh = shard_of_warp(item_base, n_shards, t, lane);
    const qlc_desc dd = descs[sh];
    const uint64_t g = t - item_base[sh];
    if (enter_shard(dd, &h, sm.hdr, sm.T, sm.seen, status, lane)) return;
    if (g == 0 && lane == 0 && dd.out_bytes) *dd.out_bytes = h.n;
    if (lane == 0) s_out[wid] = dd.out;
    __syncwarp();
    if (g < h.n_groups)
      decode_group<kOutCodes, kRingFew>(h, static_cast<const uint8_t*>(dd.in), nullptr, nullptr, g, sm.lanes, sm.T, d, status, lane,
                              (reinterpret_cast<uintptr_t>(dd.out) & 31u) == 0, false, 0u, &s_out[wid]);
    return;
  }
  // Split: items are kSpanWarps spans of one shard, which a team decodes with a
  // table that its warps share.
  const int team = wid / kSpanWarps, warp = wid % kSpanWarps, tid = 32 * warp + lane;
  const uint32_t teams = blockDim.x / (32 * kSpanWarps);
  if (team >= (int)teams) return;  // warps that make no team
  SpanShared& sm = reinterpret_cast<SpanShared*>(few_sm)[team];
  int cur = -1;
  uint32_t err = 0;
  for (unsigned long long t = (unsigned long long)team * gridDim.x + blockIdx.x; t < total;) {
    const int sh = shard_of_warp(item_base, n_shards, t, lane);  // the same in every warp of the team
    const qlc_desc dd = descs[sh];
    const uint8_t* in = static_cast<const uint8_t*>(dd.in);
    const uint32_t q = (uint32_t)(t - item_base[sh]);
    if (sh != cur) {
      load_header(in, dd.in_bytes, sm.hdr, tid, 32 * kSpanWarps);
      team_sync(team);
      err = parse_header(sm.hdr, dd.in_bytes, dd.out_cap, &h, sm.seen[warp], lane);
      if (!err) build_table(sm.hdr, sm.T, tid, 32 * kSpanWarps);
      team_sync(team);
      cur = sh;
    }
    if (q == 0 && tid == 0) {
      if ((!err || err == QLC_ERR_CAPACITY) && dd.out_bytes) *dd.out_bytes = h.n;
      if (err) set_status(status, err);
    }
    if (!err) {
      const uint64_t s = (uint64_t)q * kSpanWarps + warp;
      const SplitData sd = {h.cs, h.len_lo, h.len_hi, h.n, h.payload_bytes};
      if (batch_symbols <= split_most(sd, kSplitBatch, split_samples(sd, kSplitBatch, batch_symbols) ? batch_slow : 0)) {
        const SpanShape shape(h.cs);
        const uint32_t k = (uint32_t)lane / shape.lanes, seg = (uint32_t)lane - k * shape.lanes;
        const uint64_t g = s / shape.per_group;
        const uint32_t r = (uint32_t)(s - g * shape.per_group);
        if (g < h.n_groups)
          decode_span<kOutCodes>(h, shape, in, dd.out, nullptr, g, r * shape.chunks, k, seg, sm.w[warp].span, sm.T,
                                 warm_bits(h.len_lo, h.len_hi), status, lane);
      } else if (s < h.n_groups) {
        LaneDec d;
        if (lane_init(sm.w[warp].lanes, d, lane))
          decode_group<kOutCodes, kRingStatic>(h, in, dd.out, nullptr, s, sm.w[warp].lanes, sm.T, d, status, lane,
                                  (reinterpret_cast<uintptr_t>(dd.out) & 31u) == 0);
        else if (lane == 0)
          set_status(status, QLC_ERR_CUDA);
      }
    }
    if (tid == 0) s_item[team] = teams * gridDim.x + (unsigned long long)atomicAdd(ticket, 1u);
    team_sync(team);  // ... and every warp is done with the header and the table
    t = s_item[team];
    team_sync(team);
  }
}

}  // namespace qlc

using namespace qlc;

template <int kOut>
static qlc_status launch_decode(const uint8_t* d_in, size_t in_bytes, void* d_out, const float* d_scales,
                                size_t out_cap, uint64_t* d_n_out, uint32_t* d_status, cudaStream_t st) {
  static OncePerContext done;
  if (!smem_ok(decode_kernel<kOut>, one_bytes(dec_warps(kOut)), done)) return QLC_ERR_CUDA;
  // a warp for every span there can be, four at least (a CTA of all warps and
  // their shared memory starts 1 to 3 us later)
  const uint64_t spans = out_cap / (kSpanSyms / 2) + 1, sms = (uint64_t)sm_count();
  const uint64_t per_sm = (spans + sms - 1) / sms;
  const int warps = per_sm >= dec_warps(kOut) ? dec_warps(kOut) : (int)((per_sm + 3) / 4 * 4);
  decode_kernel<kOut><<<(int)(spans < sms ? spans : sms), 32 * warps, one_bytes(warps), st>>>(
      d_in, in_bytes, d_out, d_scales, out_cap, reinterpret_cast<unsigned long long*>(d_n_out), d_status);
  return cudaGetLastError() == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
}

extern "C" qlc_status qlc_decode(const uint8_t* d_in, size_t in_bytes, uint8_t* d_out, size_t out_cap,
                                 uint64_t* d_n_out, uint32_t* d_status, qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_decode");
  if (!d_in || !d_n_out || (out_cap > 0 && !d_out)) return QLC_ERR_ARG;
  if (!aligned(d_in, 16) || !aligned(d_out, 16) || !aligned(d_n_out, 8) || !aligned(d_status, 4))
    return QLC_ERR_ARG;
  return launch_decode<kOutCodes>(d_in, in_bytes, d_out, nullptr, out_cap, d_n_out, d_status,
                                  reinterpret_cast<cudaStream_t>(stream));
}

extern "C" qlc_status qlc_decode_dequantize(const uint8_t* d_in, size_t in_bytes, const float* d_scales,
                                            void* d_out, qlc_dtype dtype, size_t out_cap, uint64_t* d_n_out,
                                            uint32_t* d_status, qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_decode_dequantize");
  if (dtype != QLC_DTYPE_F32 && dtype != QLC_DTYPE_BF16) return QLC_ERR_ARG;
  if (!d_in || !d_n_out || (out_cap > 0 && (!d_out || !d_scales))) return QLC_ERR_ARG;
  if (!aligned(d_in, 16) || !aligned(d_out, 16) || !aligned(d_scales, 4) || !aligned(d_n_out, 8) ||
      !aligned(d_status, 4))
    return QLC_ERR_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (dtype == QLC_DTYPE_F32)
    return launch_decode<QLC_DTYPE_F32>(d_in, in_bytes, d_out, d_scales, out_cap, d_n_out, d_status, st);
  return launch_decode<QLC_DTYPE_BF16>(d_in, in_bytes, d_out, d_scales, out_cap, d_n_out, d_status, st);
}

// Resident decode warps per SM of a batch.
static int decode_warps(const qlc_launch* launch) {
  const int n = launch ? launch->decode_ctas_per_sm : 0;
  return n > 0 && n < kDecCtasPerSm ? n : kDecCtasPerSm;
}

extern "C" int qlc_test_decode_warps(const qlc_launch* h_launch) { return decode_warps(h_launch); }

extern "C" qlc_status qlc_decode_batch(const qlc_desc* d_descs, int n_shards, void* d_ws, size_t ws_bytes,
                                       uint32_t* d_status, const qlc_launch* h_launch, qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_decode_batch");
  if (!d_descs || n_shards < 1 || !d_ws) return QLC_ERR_ARG;
  if (!aligned(d_ws, 16) || !aligned(d_descs, 16) || !aligned(d_status, 4)) return QLC_ERR_ARG;
  BatchWs w;
  if (!batch_ws_layout(d_ws, ws_bytes, n_shards, &w)) return QLC_ERR_CAPACITY;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int per_sm = decode_warps(h_launch), sms = sm_count();
  static OncePerContext done;
  if (!smem_ok(decode_few_kernel, few_bytes(kFewWarps), done)) return QLC_ERR_CUDA;
  if (!launch_plan(per_sm < kSpanWarps ? kPlanDecodeGroups : kPlanDecode, d_descs, n_shards, (uint32_t)(per_sm * sms), w,
                   d_status, st))
    return QLC_ERR_CUDA;
  // which of the two has the work is decided on the device; the other returns at once
  launch_after(decode_few_kernel, sms, 32 * per_sm, few_bytes(per_sm), st, d_descs, n_shards, w.item_base, w.ticket, d_status);
  launch_after(decode_batch_kernel, sms * per_sm, 32, 0, st, d_descs, n_shards, w.item_base, w.ticket, d_status);
  return cudaGetLastError() == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
}

namespace qlc {
QLC_DEFINE_CHECK_TAKE(check_take_decode)
}  // namespace qlc
