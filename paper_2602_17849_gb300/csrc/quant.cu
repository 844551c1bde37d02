// quant.cu -- block-32 e4m3 quantisation fused with the byte histogram, and
// dequantisation (Section 3: the tensors are all-finite eXmY e4m3 with one
// scale per block of 32 elements; Section 4: the 256-bin histogram).
//
// Quantisation reads the wide input once and writes the codes and scales; the
// histogram the LUT needs (Section 7) is counted in the same pass, so the
// codes are not read again before encoding.  Rule per block of 32 (the last
// may be shorter): scale = absmax / 480 in fp32; code = the e4m3 byte nearest
// to x / scale (fp32 division), ties to the even code, saturating at 480, sign
// kept; a block whose scale is 0 (absmax 0, or absmax / 480 rounding to 0 in
// fp32) gets codes 0x00.
//
// A warp handles 1 KiB of input per step: 32 contiguous bytes per lane, 8
// fp32 (or 16 bf16) elements, so one block of 32 is 4 (or 2) lanes and its
// absmax is a 2 (or 1) step butterfly.  Codes leave as one 8- (or 16-) byte
// store per lane.
//
// One CTA of up to 32 warps per SM, which count into one table of a column per
// lane (word of code c and lane l at 256 c + 4 l: the 32 lanes of a warp update 32
// different banks, whatever the codes, and a byte permute makes the address).
// With a histogram per warp of 8 an update took 2.9 wavefronts of the shared-
// memory pipe, which was 81 % busy with 16-bit input.  Quantise, LUT and encode,
// us, before / now: fp32, 256 Mi elements 428 / 405, bf16, 61 Mi 112 / 109.5; 4 Mi
// fp32 32.4 / 30.5; the kernel alone 220 / 193 and 38 / 33.  Input in flight: three
// slots per warp (two 413 / 112, four 418 / 110).  fp32 is bound by HBM, bf16 by instruction issue (16 an element).
#include <cuda_bf16.h>

#define QLC_FILE_ID 5
#include "qlc_common.cuh"
#include "../../include/qlc_testing.h"

namespace qlc {

constexpr int kQuantWarps = 32;  // at most, of the one CTA per SM
constexpr int kQuantThreads = kQuantWarps * 32;
constexpr int kQuantDepth = 3;  // input ring slots (warp steps) per warp
constexpr int kQuantVec = 2;    // 16-byte input vectors per lane and step
// Shared address of the histogram; dynamic shared memory starts at or below it.
constexpr uint32_t kColAddr = 2048;
constexpr size_t quant_used(int warps) { return (256u << 8) + (size_t)warps * kQuantDepth * kQuantVec * 512; }
constexpr size_t quant_smem(int warps) { return fixed_smem_bytes(kColAddr, quant_used(warps)); }

// The e4m3 byte nearest to v, ties to the even code, saturating (|v| finite).
// With k = max(exponent of |v|, -6), the grid of e4m3 values around |v| is
// (q / 8) 2^k for integer q (q in [8, 16] for normals, [0, 8] below 2^-6), so
// q = |v| 2^(3-k) rounded to nearest even (the scaling is exact) and the
// code is 8 k + 48 + q, which also carries q = 16 into the next exponent.
__device__ __forceinline__ uint32_t e4m3_rne(float v) {
  const uint32_t u = __float_as_uint(v);
  const int e = (int)((u >> 23) & 0xFFu) - 127;
  const int k = max(e, -6);
  const float t = fabsf(v) * __uint_as_float((uint32_t)(130 - k) << 23);
  const uint32_t code = (uint32_t)(8 * k + 48) + __float2uint_rn(t);
  return min(code, 0x7Fu) | ((u >> 24) & 0x80u);
}

// x / scale rounded to nearest, from y = 1 / scale rounded to nearest: the
// product q0 = x y and one correction by its fused-multiply-add residual
// (Markstein's correction step).  It equals the fp32 division for every scale
// mantissa with every x whose quotient lies within three floats of a value or
// a rounding midpoint of the format (checked exhaustively on the host with
// IEEE fmaf), and elsewhere lies on the same side of every midpoint; so the
// code taken from it is the rule's.  Scales from 2^-80 on: below, the residual
// of an element that matters could be subnormal.  The residual is formed as
// q0 scale - x and multiplied by -y, which keeps -0.
// Three FMA-pipe operations per element (bf16, 61 M elements with the
// histogram: 38 us, 33 with the table of columns; fp32, 256 Mi: 220 and 193 us)
// replaced a bracket (two conversions of
// the product moved up and down by 2^-20, an exact division where they
// differed): bf16 elements, whose quotients often lie on midpoints, sent
// nearly every warp step to that division (59 us; fp32 234 us).
__device__ __forceinline__ float quotient(float x, float scale, float y) {
  const float q0 = x * y;
  return fmaf(fmaf(q0, scale, -x), -y, q0);
}
// Codes of four quotients, the first lowest, from the hardware conversion to
// e4m3 (round to nearest even).  Below 448 its grid is this format's grid
// (subnormals m 2^-9, normals (1 + m/8) 2^(e-7), sign bit 7), so the codes
// agree there; it saturates at 448 (0x7E), and this format goes on to 480
// (0x7F), the code of every magnitude above the midpoint 464.  So the code's
// low bit is set by a flag computed on the FMA pipe: (|v| - 464) 2^20 clamped
// to [0, 1] is 1.0 above 464 (the fp32 neighbours of 464 are 2^-15 away) and
// 0.0 up to it, and f0 + 256 f1 + 2^23 holds two flags in its low bits, one
// per byte.
__device__ __forceinline__ uint32_t sat_flags(float a, float b) {
  const float fa = __saturatef(fmaf(fabsf(a), 0x1p20f, -464.0f * 0x1p20f));
  const float fb = __saturatef(fmaf(fabsf(b), 0x1p20f, -464.0f * 0x1p20f));
  return __float_as_uint(fmaf(fb, 256.0f, fa + 0x1p23f));
}
__device__ __forceinline__ uint32_t e4m3x4(float a, float b, float c, float d) {
  uint16_t lo, hi;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(lo) : "f"(b), "f"(a));
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(hi) : "f"(d), "f"(c));
  const uint32_t flags = __byte_perm(sat_flags(a, b), sat_flags(c, d), 0x5410) & 0x01010101u;
  return __byte_perm(lo, hi, 0x5410) | flags;  // 0x7E -> 0x7F above 464
}

// amax / 480 rounded to nearest.  For amax in [2^-100, FLT_MAX] a product
// with 1/480 (rounded) and one correction by its fused-multiply-add residual
// (Markstein's correction step) give the correctly rounded quotient; checked
// against the division for every float with an exponent in that range (the
// quotient's pattern repeats from binade to binade there).  Other values
// (zero, tiny, non-finite) take the division.
__device__ __forceinline__ float scale_of(float amax) {
  constexpr float c = 1.0f / 480.0f;
  if (amax >= 0x1p-100f && amax <= 3.40282347e38f) {
    const float q0 = amax * c;
    return fmaf(fmaf(-q0, 480.0f, amax), c, q0);
  }
  return amax / 480.0f;
}

// max(a, b) that returns NaN when either is NaN.
__device__ __forceinline__ float fmax_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

template <int kDtype>
struct QuantIo;

template <>
struct QuantIo<QLC_DTYPE_F32> {
  static constexpr int kPerVec = 4;
  __device__ static void unpack(uint4 q, float* v) {
    v[0] = __uint_as_float(q.x), v[1] = __uint_as_float(q.y), v[2] = __uint_as_float(q.z),
    v[3] = __uint_as_float(q.w);
  }
  __device__ static void load_tail(const void* x, uint64_t i, uint64_t n, float* v) {
    const float* p = static_cast<const float*>(x);
    for (int j = 0; j < 4 * kQuantVec; j++) v[j] = i + j < n ? p[i + j] : 0.0f;
  }
};

template <>
struct QuantIo<QLC_DTYPE_BF16> {
  static constexpr int kPerVec = 8;
  __device__ static void unpack(uint4 q, float* v) {
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int j = 0; j < 4; j++) {
      v[2 * j] = __uint_as_float(w[j] << 16);
      v[2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
    }
  }
  __device__ static void load_tail(const void* x, uint64_t i, uint64_t n, float* v) {
    const uint16_t* p = static_cast<const uint16_t*>(x);
    for (int j = 0; j < 8 * kQuantVec; j++) v[j] = i + j < n ? __uint_as_float((uint32_t)p[i + j] << 16) : 0.0f;
  }
};

__device__ __forceinline__ void q_cp_async16(uint32_t smem, const void* g, bool pred) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q cp.async.cg.shared.global [%0], [%1], 16;\n\t}" ::"r"(smem),
      "l"(g), "r"((uint32_t)pred)
      : "memory");
}
__device__ __forceinline__ void q_cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void q_cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Steps per launch: step indices and their products stay in 32 bits.
constexpr uint64_t kQuantMaxSteps = 1ull << 30;

// Scale and codes of one lane's E elements v (its block of 32 spans
// 32 / E lanes, whose absmax the shuffles combine).  Sets bad for NaN or
// infinity among v.  w receives the codes, 4 per word, element 4t + b in
// byte b of w[t].
template <int E>
__device__ __forceinline__ float lane_codes(const float (&v)[E], uint32_t (&w)[E / 4], bool& bad) {
  constexpr int kLanesPerBlock = 32 / E;
  constexpr int kWords = E / 4;
  float amax = 0.0f;
#pragma unroll
  for (int j = 0; j < E; j++) amax = fmax_nan(amax, fabsf(v[j]));
  bad |= !(amax <= 3.402823466e38f);  // NaN or infinity in this lane
#pragma unroll
  for (int o = 1; o < kLanesPerBlock; o <<= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  const float scale = scale_of(amax);
  const float y = __frcp_rn(scale);
#pragma unroll
  for (int t = 0; t < kWords; t++)
    w[t] = e4m3x4(quotient(v[4 * t], scale, y), quotient(v[4 * t + 1], scale, y), quotient(v[4 * t + 2], scale, y),
                  quotient(v[4 * t + 3], scale, y));
  if (!(scale >= 0x1p-80f)) {  // rare: exact division, or codes 0x00 for a scale of 0
#pragma unroll
    for (int t = 0; t < kWords; t++) {
      w[t] = 0u;
      if (scale > 0.0f)
        for (int j = 0; j < 4; j++) w[t] |= e4m3_rne(v[4 * t + j] / scale) << (8 * j);
    }
  }
  return scale;
}

// Input pipeline: warp step s covers elements [s kStep, (s + 1) kStep),
// 1 KiB of input, 32 contiguous bytes per lane; warps take steps s = first,
// first + W, ... (W warps in the grid).  A warp keeps its next
// kQuantDepth - 1 steps in flight: its k-th step goes by cp.async into its
// 1 KiB of shared slot k mod kQuantDepth, each copy instruction 512
// contiguous bytes (one commit group per step; in a ragged last step only
// the 16-byte vectors wholly inside are copied).  About 100 bytes per thread
// are in flight without holding registers.  Lanes read bytes other lanes
// copied, so each step starts with the lane's wait on its own groups and a
// warp barrier; a slot is refilled after that barrier, when every lane has
// finished the step that read it.  Every step but a ragged last one takes
// the short path; there a lane whose 32 bytes are not wholly inside reads
// its elements with plain loads.
template <int kDtype>
__global__ void __launch_bounds__(kQuantThreads)
quantize_kernel(const void* __restrict__ x, uint64_t n, uint8_t* __restrict__ codes, float* __restrict__ scales,
                unsigned long long* __restrict__ hist, uint32_t* __restrict__ status) {
  constexpr int E = QuantIo<kDtype>::kPerVec * kQuantVec;  // elements per lane
  constexpr int kLanesPerBlock = 32 / E;
  constexpr uint32_t kStep = 32 * E;             // elements per warp step
  constexpr uint32_t kWords = E / 4;             // code words per lane
  constexpr uint32_t kSlot = kQuantVec * 512u;  // bytes of a ring slot
  extern __shared__ __align__(16) uint8_t quant_sm[];
  const uint32_t smem_s = (uint32_t)__cvta_generic_to_shared(quant_sm);
  if (smem_s > kColAddr) {  // does not happen
    if (threadIdx.x == 0) set_status(status, QLC_ERR_CUDA);
    return;
  }
  uint8_t* cols = quant_sm + (kColAddr - smem_s);
  if (hist) {  // the half of each row that is counted in
    for (uint32_t i = threadIdx.x; i < 256 * 8; i += blockDim.x)
      reinterpret_cast<uint4*>(cols)[i / 8 * 16 + i % 8] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t cta_warps = blockDim.x / 32;
  uint4* ring = reinterpret_cast<uint4*>(cols + (256 << 8)) + warp * kQuantDepth * kQuantVec * 32;
  const uint32_t n_steps = (uint32_t)((n + kStep - 1) / kStep);  // <= kQuantMaxSteps
  const uint32_t warps = gridDim.x * cta_warps;
  const uint32_t first = blockIdx.x * cta_warps + warp;
  const uint32_t cnt = first < n_steps ? (n_steps - first + warps - 1) / warps : 0;  // this warp's steps
  // this warp's steps whose whole 1 KiB lies inside: all but a ragged last
  const uint32_t nfw = cnt > 0 && first + (cnt - 1) * warps == n_steps - 1 && (uint64_t)n_steps * kStep > n
                           ? cnt - 1 : cnt;
  const uint64_t n_bytes = n * (16 / QuantIo<kDtype>::kPerVec);
  uint8_t* c_lane = codes + lane * E;
  float* s_lane = scales + lane / kLanesPerBlock;
  const bool scale_lane = lane % kLanesPerBlock == 0;
  // copy instruction u of lane l: bytes [512 u + 16 l, + 16) of the step
  const uint8_t* x_copy = static_cast<const uint8_t*>(x) + lane * 16;
  const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring + lane);
  auto fetch = [&](uint32_t k, uint32_t slot) {  // step k of this warp into slot k mod kQuantDepth
    const uint32_t d = ring_s + slot * kSlot;
    const uint64_t b = (uint64_t)(first + k * warps) * (512u * kQuantVec);
    if (k < nfw) {
#pragma unroll
      for (int u = 0; u < kQuantVec; u++)
        q_cp_async16(d + 512u * u, x_copy + b + 512u * u,
                     QLC_GUARD(b + lane * 16 + 512u * u + 16 <= n_bytes, status));
    } else if (k < cnt) {  // the ragged last step: the vectors wholly inside
#pragma unroll
      for (int u = 0; u < kQuantVec; u++) {
        const bool in = b + lane * 16 + 512u * u + 16 <= n_bytes;
        q_cp_async16(d + 512u * u, in ? x_copy + b + 512u * u : x_copy, in);
      }
    }
    q_cp_async_commit();
  };
  auto count = [&](const uint32_t (&w)[kWords], int m) {  // the first m codes into the histogram
#pragma unroll
    for (int j = 0; j < E; j++) {
      if (j < m) {
        const uint32_t at = __byte_perm(w[j / 4], 4u * lane, 0x5504 | (j % 4) << 4);  // code << 8 | 4 lane
        asm volatile("red.shared.add.u32 [%0 + %1], %2;" ::"r"(at), "n"(kColAddr), "r"(1u) : "memory");
      }
    }
  };
#pragma unroll
  for (uint32_t d = 0; d + 1 < kQuantDepth; d++) fetch(d, d);
  bool bad = false;
  uint32_t s = first, k = 0, slot = 0;  // slot: k mod kQuantDepth
  for (; k < nfw; k++, s += warps) {
    // groups committed so far: kQuantDepth - 1 + k; step k's is complete
    // when at most kQuantDepth - 2 are pending
    q_cp_async_wait<kQuantDepth - 2>();
    __syncwarp();
    fetch(k + kQuantDepth - 1, slot == 0 ? kQuantDepth - 1 : slot - 1);  // the slot step k - 1 was read from
    float v[E];
    const uint4* r = ring + slot * kQuantVec * 32 + lane * kQuantVec;
#pragma unroll
    for (int u = 0; u < kQuantVec; u++) QuantIo<kDtype>::unpack(r[u], v + u * QuantIo<kDtype>::kPerVec);
    slot = slot + 1 == kQuantDepth ? 0 : slot + 1;
    uint32_t w[kWords];
    const float scale = lane_codes<E>(v, w, bad);
    if (scale_lane && QLC_GUARD((uint64_t)s * kStep + lane * E < n, status)) s_lane[(uint64_t)s * (kStep / 32)] = scale;
    if (QLC_GUARD((uint64_t)s * kStep + (lane + 1) * E <= n, status)) {
      if constexpr (kWords == 2)
        *reinterpret_cast<uint2*>(c_lane + (uint64_t)s * kStep) = make_uint2(w[0], w[1]);
      else
        *reinterpret_cast<uint4*>(c_lane + (uint64_t)s * kStep) = make_uint4(w[0], w[1], w[2], w[3]);
      if (hist) count(w, E);
    }
  }
  if (k < cnt) {  // the ragged last step
    q_cp_async_wait<0>();
    __syncwarp();
    const uint64_t i = (uint64_t)s * kStep + (uint64_t)lane * E;
    float v[E];
    if (i + E <= n) {
      const uint4* r = ring + slot * kQuantVec * 32 + lane * kQuantVec;
#pragma unroll
      for (int u = 0; u < kQuantVec; u++) QuantIo<kDtype>::unpack(r[u], v + u * QuantIo<kDtype>::kPerVec);
    } else {
      QuantIo<kDtype>::load_tail(x, i, n, v);  // zeros past the end
    }
    uint32_t w[kWords];
    const float scale = lane_codes<E>(v, w, bad);
    if (scale_lane && i < n && QLC_GUARD(i / 32 < (n + 31) / 32, status)) scales[i / 32] = scale;
    for (int j = 0; j < E; j++)
      if (i + j < n) codes[i + j] = (uint8_t)(w[j / 4] >> (8 * (j % 4)));
    if (hist && i < n) count(w, (int)(n - i < (uint64_t)E ? n - i : E));
  }
  q_cp_async_wait<0>();
  if (__syncthreads_or(bad) && threadIdx.x == 0) set_status(status, QLC_ERR_ARG);
  if (hist) {
    for (uint32_t b = threadIdx.x; b < 256; b += blockDim.x) {
      uint32_t t = 0;
#pragma unroll 8
      for (uint32_t l = 0; l < 32; l++) t += reinterpret_cast<const uint32_t*>(cols + 256 * b)[(l + b) & 31];
      if (t) atomicAdd(&hist[b], (unsigned long long)t);
    }
  }
}

// out[i] = value(codes[i]) * scales[i / 32].  Warp step s covers codes
// [512 s, 512 s + 512); in part k (0..3) lane l takes codes
// [512 s + 128 k + 4 l, + 4), so each load and store instruction of the warp
// covers contiguous bytes (128 bytes of codes, 512 of fp32 or 256 of bf16).
template <int kDtype>
__global__ void __launch_bounds__(256)
dequantize_kernel(const uint8_t* __restrict__ codes, const float* __restrict__ scales, uint64_t n,
                  void* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const uint64_t n_steps = (n + 511) / 512;
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x / 32);
  for (uint64_t s = (uint64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; s < n_steps; s += warps) {
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const uint64_t i = s * 512 + 128 * k + 4 * lane;
      if (i >= n) continue;
      const float sc = scales[i / 32];
      uint32_t w = 0;
      if (i + 4 <= n) {
        w = __ldg(reinterpret_cast<const unsigned int*>(codes + i));
      } else {
        for (int j = 0; j < 4; j++)
          if (i + j < n) w |= (uint32_t)codes[i + j] << (8 * j);
      }
      float y[4];
#pragma unroll
      for (int j = 0; j < 4; j++) y[j] = __uint_as_float(e4m3_scaled_bits(w, j)) * 0x1p120f * sc;
      if (kDtype == QLC_DTYPE_F32) {
        float* o = static_cast<float*>(out) + i;
        if (i + 4 <= n) {
          __stcs(reinterpret_cast<float4*>(o), make_float4(y[0], y[1], y[2], y[3]));
        } else {
          for (int j = 0; j < 4; j++)
            if (i + j < n) o[j] = y[j];
        }
      } else {
        __nv_bfloat16* o = static_cast<__nv_bfloat16*>(out) + i;
        if (i + 4 <= n) {
          const __nv_bfloat162 h0 = __floats2bfloat162_rn(y[0], y[1]), h1 = __floats2bfloat162_rn(y[2], y[3]);
          __stcs(reinterpret_cast<uint2*>(o), make_uint2(*reinterpret_cast<const uint32_t*>(&h0),
                                                         *reinterpret_cast<const uint32_t*>(&h1)));
        } else {
          for (int j = 0; j < 4; j++)
            if (i + j < n) o[j] = __float2bfloat16_rn(y[j]);
        }
      }
    }
  }
}

}  // namespace qlc

namespace qlc {
template <int kDtype>
static qlc_status launch_quantize(const void* x, uint64_t n, uint64_t steps, uint8_t* codes, float* scales,
                                  unsigned long long* hist, uint32_t* status, cudaStream_t st) {
  static OncePerContext done;
  if (!smem_ok(quantize_kernel<kDtype>, quant_smem(kQuantWarps), done)) return QLC_ERR_CUDA;
  // one CTA per SM, each warp looping over its steps with its copies in flight;
  // small inputs over all SMs, in CTAs of four warps at least
  const uint64_t sms = sm_count(), per_sm = (steps + sms - 1) / sms;
  const int warps = per_sm >= kQuantWarps ? kQuantWarps : (int)((per_sm + 3) / 4 * 4);
  const uint64_t want = (steps + warps - 1) / warps;
  quantize_kernel<kDtype><<<(int)(want < sms ? want : sms), 32 * warps, quant_smem(warps), st>>>(x, n, codes, scales, hist,
                                                                                            status);
  return cudaGetLastError() == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
}
}  // namespace qlc

using namespace qlc;

extern "C" void qlc_test_quantize_smem(int warps, uint32_t* addr, uint32_t* size, uint32_t* requested) {
  *addr = kColAddr;
  *size = (uint32_t)quant_used(warps);
  *requested = (uint32_t)quant_smem(warps);
}

extern "C" qlc_status qlc_quantize_e4m3(const void* d_x, qlc_dtype dtype, size_t n, uint8_t* d_codes,
                                        float* d_scales, uint64_t* d_hist, int accumulate, uint32_t* d_status,
                                        qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_quantize_e4m3");
  if (dtype != QLC_DTYPE_F32 && dtype != QLC_DTYPE_BF16) return QLC_ERR_ARG;
  if (n > 0 && (!d_x || !d_codes || !d_scales)) return QLC_ERR_ARG;
  if (!aligned(d_x, 16) || !aligned(d_codes, 16) || !aligned(d_scales, 16) || !aligned(d_hist, 8) ||
      !aligned(d_status, 4))
    return QLC_ERR_ARG;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (d_hist && !accumulate && cudaMemsetAsync(d_hist, 0, 256 * sizeof(uint64_t), st) != cudaSuccess)
    return QLC_ERR_CUDA;
  if (n == 0) return QLC_OK;
  // inputs above kQuantMaxSteps steps go in several launches (slices of whole
  // blocks, the histogram accumulating)
  const uint64_t step = (uint64_t)32 * kQuantVec * (dtype == QLC_DTYPE_F32 ? 4 : 8);  // elements per warp step
  const uint64_t elem = dtype == QLC_DTYPE_F32 ? 4 : 2;
  const uint64_t slice = kQuantMaxSteps * step;
  unsigned long long* h = reinterpret_cast<unsigned long long*>(d_hist);
  for (uint64_t off = 0; off < n; off += slice) {
    const uint64_t m = n - off < slice ? n - off : slice;
    const void* xs = static_cast<const uint8_t*>(d_x) + off * elem;
    const uint64_t steps = (m + step - 1) / step;
    const qlc_status s =
        dtype == QLC_DTYPE_F32
            ? launch_quantize<QLC_DTYPE_F32>(xs, m, steps, d_codes + off, d_scales + off / 32, h, d_status, st)
            : launch_quantize<QLC_DTYPE_BF16>(xs, m, steps, d_codes + off, d_scales + off / 32, h, d_status, st);
    if (s != QLC_OK) return s;
  }
  return QLC_OK;
}

extern "C" qlc_status qlc_dequantize_e4m3(const uint8_t* d_codes, const float* d_scales, size_t n, void* d_out,
                                          qlc_dtype dtype, qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_dequantize_e4m3");
  if (dtype != QLC_DTYPE_F32 && dtype != QLC_DTYPE_BF16) return QLC_ERR_ARG;
  if (n > 0 && (!d_codes || !d_scales || !d_out)) return QLC_ERR_ARG;
  if (!aligned(d_codes, 16) || !aligned(d_out, 16) || !aligned(d_scales, 4)) return QLC_ERR_ARG;
  if (n == 0) return QLC_OK;
  const uint64_t want = ((n + 511) / 512 + 7) / 8;  // warp steps of 512 codes, 8 warps per CTA
  const uint64_t cap = (uint64_t)sm_count() * 8;
  const int grid = (int)(want < cap ? want : cap);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (dtype == QLC_DTYPE_F32)
    dequantize_kernel<QLC_DTYPE_F32><<<grid, 256, 0, st>>>(d_codes, d_scales, n, d_out);
  else
    dequantize_kernel<QLC_DTYPE_BF16><<<grid, 256, 0, st>>>(d_codes, d_scales, n, d_out);
  return cudaGetLastError() == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
}

namespace qlc {
QLC_DEFINE_CHECK_TAKE(check_take_quant)
}  // namespace qlc
