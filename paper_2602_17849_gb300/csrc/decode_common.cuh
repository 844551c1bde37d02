// decode_common.cuh -- what the decoders share: the container's header, the
// code table and the outputs of single symbols (Section 7; container v1).
#pragma once

#include <cuda_bf16.h>

#include "qlc_common.cuh"

namespace qlc {

struct DecHeader {
  uint64_t n, payload_bytes, P, n_chunks, n_groups;
  uint64_t in_bytes, out_cap;  // the caller's buffers (bounds of the checked build)
  uint32_t cs;
  uint32_t len_lo, len_hi;  // code length of areas 0-3 / 4-7, one byte each
};

__constant__ uint16_t c_table_n[2][8] = {{8, 8, 8, 8, 8, 16, 32, 168}, {2, 8, 8, 8, 8, 32, 32, 158}};
__constant__ uint8_t c_table_b[2][8] = {{3, 3, 3, 3, 3, 4, 5, 8}, {1, 3, 3, 3, 3, 5, 5, 8}};

// Copies the container's header and dec (kIndexOff bytes; fewer in a container
// that is shorter, which parse_header refuses) to shared memory: one round of
// loads, where reading the fields one by one waited for several.  The caller
// synchronises.
__device__ __forceinline__ void load_header(const uint8_t* in, uint64_t in_bytes, uint8_t* hdr, int tid, int threads) {
  if (in_bytes < kIndexOff) return;
  for (uint32_t i = tid; i < kIndexOff / 16; i += threads)
    reinterpret_cast<uint4*>(hdr)[i] = reinterpret_cast<const uint4*>(in)[i];
}

// Parses and validates the header (all lanes, redundantly) from its copy in
// shared memory; same checks, in the same order of kinds, as the container
// rules: 0 = ok, else a status.  s_seen: 64 words of scratch.
static __device__ uint32_t parse_header(const uint8_t* in, uint64_t in_bytes, uint64_t out_cap,
                                 DecHeader* h, uint32_t* s_seen, int lane) {
  if (in_bytes < kIndexOff) return QLC_ERR_CORRUPT;
  const uint32_t w0 = *reinterpret_cast<const uint32_t*>(in);
  const uint32_t w1 = *reinterpret_cast<const uint32_t*>(in + 4);
  const unsigned long long reserved = *reinterpret_cast<const unsigned long long*>(in + 56);
  bool ok = w0 == 0x31434C51u && (w1 & 0xFFFFu) == QLC_VERSION && (w1 >> 24) == 0 && reserved == 0;
  const uint32_t id = (w1 >> 16) & 0xFFu;
  uint16_t an[8];
  uint8_t ab[8];
  for (int i = 0; i < 8; i++) {
    an[i] = *reinterpret_cast<const uint16_t*>(in + 24 + 2 * i);
    ab[i] = in[40 + i];
  }
  ok = ok && scheme_ok(an, ab);
  if (id == 1 || id == 2) {
    for (int i = 0; i < 8; i++) ok = ok && an[i] == c_table_n[id - 1][i] && ab[i] == c_table_b[id - 1][i];
  } else {
    ok = ok && id == 0;
  }
  h->n = *reinterpret_cast<const unsigned long long*>(in + 8);
  h->cs = *reinterpret_cast<const uint32_t*>(in + 16);
  h->n_chunks = *reinterpret_cast<const uint32_t*>(in + 20);
  // n_chunks == (n + cs - 1) / cs, without the division
  const uint64_t up = h->n + h->cs - 1;
  ok = ok && chunk_symbols_ok(h->cs) && (uint64_t)h->n_chunks * h->cs <= up && up < ((uint64_t)h->n_chunks + 1) * h->cs;
  // dec must be a permutation of 0..255: marks the 256 places it names and looks
  // whether all are marked (with bits set by atomics this took most of the
  // header's time where an SM's warps all do it; unrolled it slows the loops
  // behind it, 24 shards by 1.7 %)
  s_seen[lane] = s_seen[lane + 32] = 0;
  __syncwarp();
#pragma unroll 1
  for (int i = lane; i < 256; i += 32) reinterpret_cast<uint8_t*>(s_seen)[in[64 + i]] = 1;
  __syncwarp();
  ok = __all_sync(0xffffffffu, s_seen[lane] == 0x01010101u && s_seen[lane + 32] == 0x01010101u) && ok;
  h->n_groups = n_groups_of(h->n_chunks);
  h->P = payload_start(h->n_chunks);
  h->payload_bytes = *reinterpret_cast<const unsigned long long*>(in + 48);
  ok = ok && h->P <= in_bytes && h->payload_bytes <= in_bytes - h->P;
  if (!ok) return QLC_ERR_CORRUPT;
  if (out_cap < h->n) return QLC_ERR_CAPACITY;
  h->in_bytes = in_bytes;
  h->out_cap = out_cap;
  h->len_lo = h->len_hi = 0;
  for (int i = 0; i < 4; i++) {
    h->len_lo |= (3u + ab[i]) << (8 * i);
    h->len_hi |= (3u + ab[i + 4]) << (8 * i);
  }
  return 0;
}

__device__ __forceinline__ uint32_t mad_hi(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
// prmt.b32 in its default mode; a selector nibble with bit 3 set yields the
// sign of the selected byte replicated (0x00 for bytes below 0x80).
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}
__device__ __forceinline__ uint32_t mad_lo(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t d;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// Code length of the codeword at the top of x (Section 7: the area code,
// i.e. the top 3 bits, fixes it): a byte permute of two registers; the
// selector's sign-mode nibbles make bytes 1-3 zero.
__device__ __forceinline__ uint32_t code_len(uint32_t x, uint32_t len_lo, uint32_t len_hi) {
  return prmt(len_lo, len_hi, mad_hi(x, 8u, 0x8880u));
}

// code -> symbol table: every code (i << bits[i]) | s of every area i maps to
// dec[offset_i + s] (offset 0 for 8-bit areas); hdr is the header's copy in
// shared memory.  The caller synchronises.
__device__ __forceinline__ void build_table(const uint8_t* hdr, uint8_t* T, int tid, int threads) {
  uint32_t base = 0;
  for (int i = 0; i < 8; i++) {
    const uint32_t b = hdr[40 + i];
    for (uint32_t s = tid; s < (1u << b); s += threads)
      if (QLC_GUARD(((i << b) | s) < 2048u && (b == 8 ? s : base + s) < 256u, nullptr))
        T[(i << b) | s] = hdr[64 + (b == 8 ? s : base + s)];
    base += *reinterpret_cast<const uint16_t*>(hdr + 24 + 2 * i);
  }
}

// Output of the decoder: the symbols themselves (kOutCodes), or their
// block-32 dequantised values (value(code) * scale, fp32 or rounded to bf16).
constexpr int kOutCodes = -1;

// One decoded symbol s at index i of the tensor.
template <int kOut>
__device__ __forceinline__ void put1(void* out, const float* scales, uint64_t i, uint32_t s) {
  if (kOut == kOutCodes) {
    static_cast<uint8_t*>(out)[i] = (uint8_t)s;
  } else {
    const float y = e4m3_to_f32(s) * scales[i / 32];
    if (kOut == QLC_DTYPE_F32)
      static_cast<float*>(out)[i] = y;
    else
      static_cast<__nv_bfloat16*>(out)[i] = __float2bfloat16_rn(y);
  }
}

// Four symbols w of one block as values at dst, one streaming store; a warp's
// 32 stores cover few lines.
template <int kOut>
__device__ __forceinline__ void put4_values(uint8_t* dst, float sc, uint32_t w) {
  float y[4];
#pragma unroll
  for (int j = 0; j < 4; j++) y[j] = __uint_as_float(e4m3_scaled_bits(w, j)) * 0x1p120f * sc;
  if (kOut == QLC_DTYPE_F32) {
    __stcs(reinterpret_cast<float4*>(dst), make_float4(y[0], y[1], y[2], y[3]));
  } else {
    const __nv_bfloat162 a = __floats2bfloat162_rn(y[0], y[1]), b = __floats2bfloat162_rn(y[2], y[3]);
    __stcs(reinterpret_cast<uint2*>(dst),
           make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b)));
  }
}
// Four decoded symbols w starting at index i of the tensor (a multiple of 4).
template <int kOut>
__device__ __forceinline__ void put4(void* out, const float* __restrict__ scales, uint64_t i, uint32_t w) {
  if (kOut == kOutCodes)
    __stcs(reinterpret_cast<unsigned int*>(static_cast<uint8_t*>(out) + i), w);
  else
    put4_values<kOut>(static_cast<uint8_t*>(out) + i * (kOut == QLC_DTYPE_F32 ? 4 : 2), __ldg(scales + i / 32), w);
}

}  // namespace qlc
