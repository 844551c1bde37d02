// hist_cols.cuh -- byte counting for the histogram kernels (Section 4: the
// symbol statistics every code is built from).
//
// A CTA of 32 warps counts into one 256 x 32 table of 32-bit counters: value
// b seen by lane l of any warp goes to word 32 b + l.  The 32 lanes of a warp
// therefore always update 32 different banks and 32 different words, whatever
// bytes they hold, so one byte per lane costs one shared reduction of one
// wavefront; lanes with the same number in different warps share a word, which
// the reductions keep exact.  What bounds it is the LSU pipe (a wavefront per
// 32 bytes, and a quarter more for the loads) together with HBM.
// One table for all warps, because the table limits the warps: with a table
// per warp (32 KB each) only 7 warps fit on an SM, and they could not keep the
// pipe busy.  256 MiB of Student-t bytes, one CTA per SM: 7 warps with 7
// tables 62-69 us, 28 warps with 7 tables 67 us, with 4 tables 48.5 us, 32
// warps with 4 / 2 / 1 tables 48.5 / 46.4 / 44.9 us; 16 and 8 warps with one
// table 50.7 and 77 us.  (Back to back; by itself, with a cold cache, the
// kernel takes 47.7 us, 5.6 TB/s, 83 % of a device copy's rate.)
#pragma once

#include "qlc_common.cuh"

namespace qlc {

constexpr int kHcWarps = 32;                    // one CTA per SM
constexpr int kHcThreads = kHcWarps * 32;
constexpr int kHcUnroll = 4;                    // 16-byte loads per lane per batch, two batches in flight
constexpr uint32_t kHcColWords = 256 * 32;      // the CTA's table

__device__ __forceinline__ void red_add_one(uint32_t saddr) {
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(saddr), "r"(1u) : "memory");
}

// col: shared address of this lane's column (value 0); value b is b * 128 bytes on.
__device__ __forceinline__ void count_word(uint32_t col, uint32_t w) {
#pragma unroll
  for (int j = 0; j < 4; j++) {
    const uint32_t b = __byte_perm(w, 0, 0x4440 + j);
    if (QLC_GUARD(b < 256u, nullptr)) red_add_one(col + (b << 7));
  }
}
__device__ __forceinline__ void count_vec(uint32_t col, uint4 q) {
  count_word(col, q.x);
  count_word(col, q.y);
  count_word(col, q.z);
  count_word(col, q.w);
}

// Counts nvec 16-byte vectors at v; thread t of the CTA takes t, t + T, ...
// Loads of the next batch are issued before the current batch is counted.
__device__ __forceinline__ void count_span(const uint4* __restrict__ v, uint64_t nvec, uint32_t col, int tid) {
  constexpr int U = kHcUnroll;
  constexpr uint64_t T = kHcThreads;
  uint64_t i = (uint64_t)tid;
  if (i + (U - 1) * T < nvec) {
    uint4 a[U], b[U];
#pragma unroll
    for (int u = 0; u < U; u++) a[u] = ldg_nc_v4(v + i + u * T);
    i += U * T;
    while (true) {
      if (i + (U - 1) * T >= nvec) {
#pragma unroll
        for (int u = 0; u < U; u++) count_vec(col, a[u]);
        break;
      }
#pragma unroll
      for (int u = 0; u < U; u++) b[u] = ldg_nc_v4(v + i + u * T);
      i += U * T;
#pragma unroll
      for (int u = 0; u < U; u++) count_vec(col, a[u]);
      if (i + (U - 1) * T >= nvec) {
#pragma unroll
        for (int u = 0; u < U; u++) count_vec(col, b[u]);
        break;
      }
#pragma unroll
      for (int u = 0; u < U; u++) a[u] = ldg_nc_v4(v + i + u * T);
      i += U * T;
#pragma unroll
      for (int u = 0; u < U; u++) count_vec(col, b[u]);
    }
  }
  for (; i < nvec; i += T) count_vec(col, ldg_nc_v4(v + i));
  QLC_GUARD(i >= nvec && i - nvec < T, nullptr);  // the loop ended at the span's end
}

// Counts m single bytes at p (a ragged end), CTA-strided.
__device__ __forceinline__ void count_bytes(const uint8_t* __restrict__ p, uint64_t m, uint32_t col, int tid) {
  for (uint64_t i = (uint64_t)tid; i < m; i += kHcThreads) red_add_one(col + ((uint32_t)p[i] << 7));
}

// Zeroes the table (callers synchronise).
__device__ __forceinline__ void zero_cols(uint32_t* cols, int tid) {
  uint4* c4 = reinterpret_cast<uint4*>(cols);
#pragma unroll
  for (uint32_t i = 0; i < kHcColWords / 4; i += kHcThreads) c4[i + tid] = make_uint4(0u, 0u, 0u, 0u);
}

// The CTA's count of value tid / 4, in the value's first thread (tid % 4 ==
// 0).  Called by every thread, after a barrier.  Four threads sum a value's 32
// counters, eight each, in an order rotated by the value so that the 32 lanes
// read 32 different banks.
__device__ __forceinline__ uint32_t sum_cols(const uint32_t* cols, int tid) {
  const uint32_t* row = cols + 32 * (tid >> 2) + 8 * (tid & 3);
  uint32_t acc = 0;
#pragma unroll
  for (int k = 0; k < 8; k++) acc += row[(k + (tid >> 2)) & 7];
  acc += __shfl_xor_sync(0xffffffffu, acc, 1);
  acc += __shfl_xor_sync(0xffffffffu, acc, 2);
  return acc;
}

// Adds the CTA's counts to hist[0..255], one 64-bit global atomic per value
// with a nonzero count, and zeroes the table when more is to be counted.
// Called by every thread of the CTA.  A counter stays below 2^32 as long as a
// CTA counts fewer than 2^32 bytes between flushes, which the launches
// guarantee.
__device__ __forceinline__ void flush_cols(uint32_t* cols, unsigned long long* __restrict__ hist, int tid, bool more) {
  __syncthreads();
  const uint32_t t = sum_cols(cols, tid);
  if ((tid & 3) == 0 && t) atomicAdd(&hist[tid >> 2], (unsigned long long)t);
  if (more) {
    __syncthreads();
    zero_cols(cols, tid);
    __syncthreads();
  }
}

// The column address of this lane.
__device__ __forceinline__ uint32_t lane_col(const uint32_t* cols, int lane) {
  return (uint32_t)__cvta_generic_to_shared(cols + lane);
}

}  // namespace qlc
