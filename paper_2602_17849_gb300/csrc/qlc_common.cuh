// qlc_common.cuh -- shared definitions of the libqlc CUDA kernels (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include <atomic>

#include "../../include/qlc.h"

namespace qlc {

constexpr uint32_t kGroupChunks = QLC_CHUNKS_PER_GROUP;  // chunks per group
constexpr uint32_t kIndexOff = QLC_INDEX_OFFSET;         // header 64 + dec 256
constexpr uint32_t kMaxCode = 11;                        // 3 + 8 suffix bits

__host__ __device__ __forceinline__ uint64_t align16(uint64_t v) {
  return (v + 15u) & ~uint64_t(15);
}
__host__ __device__ __forceinline__ uint64_t n_groups_of(uint64_t n_chunks) {
  return (n_chunks + kGroupChunks - 1) / kGroupChunks;
}
__host__ __device__ __forceinline__ uint64_t payload_start(uint64_t n_chunks) {
  return align16(kIndexOff + 8 * n_groups_of(n_chunks) + 2 * n_chunks);
}
__host__ __device__ __forceinline__ bool chunk_symbols_ok(uint64_t cs) {
  return cs >= QLC_MIN_CHUNK && cs <= QLC_MAX_CHUNK && cs % 128 == 0;
}

// Scheme validity (qlc.h): counts sum to 256, widths never decrease, an area
// with b < 8 bits is complete (2^b ranks), an 8-bit area holds 1..256 ranks.
__host__ __device__ inline bool scheme_ok(const uint16_t n[8], const uint8_t b[8]) {
  uint32_t total = 0;
  for (int i = 0; i < 8; i++) {
    if (b[i] > 8) return false;
    if (i > 0 && b[i] < b[i - 1]) return false;
    if (b[i] < 8) {
      if (n[i] != (1u << b[i])) return false;
    } else if (n[i] < 1 || n[i] > 256) {
      return false;
    }
    total += n[i];
  }
  return total == 256;
}

// Alignment of a caller's pointer to a bytes (a power of two); NULL counts as
// aligned, the entry points check NULL where it matters.
__host__ __device__ __forceinline__ bool aligned(const void* p, uintptr_t a) {
  return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0;
}

// First error wins.
__device__ __forceinline__ void set_status(uint32_t* st, uint32_t code) {
  if (st) atomicCAS(st, 0u, code);
}

// Unique id of the calling thread's current CUDA context, 0 if there is none
// or the driver cannot report it (hist_lut.cu).
unsigned long long current_context_id();

// Something that has to be done once in every context, by device: the id of
// the context it was last done in.  A context's id is never given out again, so
// a device reset or another context on the device is seen; without an id it is
// done every time.  Any number of threads may call at once.
class OncePerContext {
 public:
  template <class Id, class Do>
  bool ensure(int dev, Id id_of, Do act) {
    const unsigned long long id = id_of();
    const bool kept = dev >= 0 && dev < kDevices;
    if (kept && id != 0 && at_[dev].load(std::memory_order_relaxed) == id) return true;
    if (!act()) return false;
    // act makes the device's primary context current if none was
    if (kept) at_[dev].store(id_of(), std::memory_order_relaxed);
    return true;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<unsigned long long> at_[kDevices] = {};
};

// Raises a kernel's shared-memory limit (a function attribute of the context,
// allowed inside stream capture).
template <typename K>
static bool smem_ok(K kernel, size_t bytes, OncePerContext& done) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return false;
  return done.ensure(dev, current_context_id, [&] {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
  });
}

// Dynamic shared memory to ask for when `size` bytes are used from the shared
// address `addr` on.  Where dynamic shared memory starts is up to the driver
// (at 1024 on GB300, behind its own kilobyte), so the bytes below addr are asked
// for too: the end is inside whatever the start, and the kernel itself refuses
// a start above addr.
constexpr size_t fixed_smem_bytes(uint32_t addr, size_t size) { return addr + size; }

// Checked build (-DQLC_CHECKED): QLC_GUARD(cond, status) is false when an
// index check fails; the caller then skips the access.  The first failure of
// each .cu file is recorded in that file's g_check_site (file number << 16 |
// line) and, where a status word is at hand, as QLC_ERR_CHECK.  In a normal
// build the guard is the constant true and compiles away.
#ifndef QLC_FILE_ID
#define QLC_FILE_ID 0
#endif
#ifdef QLC_CHECKED
static __device__ uint32_t g_check_site = 0;
#endif
__device__ __forceinline__ bool guard(bool ok, uint32_t* status, uint32_t site) {
#ifdef QLC_CHECKED
  if (!ok) {
    atomicCAS(&g_check_site, 0u, site);
    set_status(status, QLC_ERR_CHECK);
  }
  return ok;
#else
  (void)status;
  (void)site;
  return true;
#endif
}
#define QLC_GUARD(cond, status) (::qlc::guard((cond), (status), ((uint32_t)QLC_FILE_ID << 16) | __LINE__))

// Host side of the checked build: reads and clears this file's record.
// Each .cu file defines its own with QLC_DEFINE_CHECK_TAKE(name).
#ifdef QLC_CHECKED
#define QLC_DEFINE_CHECK_TAKE(name)                                       \
  uint32_t name() {                                                       \
    uint32_t v = 0, z = 0;                                                \
    if (cudaDeviceSynchronize() != cudaSuccess) return 0xFFFFFFFEu;       \
    if (cudaMemcpyFromSymbol(&v, g_check_site, 4) != cudaSuccess) return 0xFFFFFFFEu; \
    cudaMemcpyToSymbol(g_check_site, &z, 4);                              \
    return v;                                                             \
  }
#else
#define QLC_DEFINE_CHECK_TAKE(name) \
  uint32_t name() { return 0; }
#endif
uint32_t check_take_decode();
uint32_t check_take_encode();
uint32_t check_take_hist();
uint32_t check_take_batch();
uint32_t check_take_quant();

// Big-endian view of a little-endian 32-bit word: byte 0 becomes bits 31..24,
// so the first bit of the stream is the word's most significant bit.
__device__ __forceinline__ uint32_t bswap32(uint32_t w) { return __byte_perm(w, 0, 0x0123); }

__device__ __forceinline__ uint4 ldg_nc_v4(const uint4* p) {
  uint4 r;
  asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// Streaming (evict-first) 16-byte store: what is written once should not push
// out of L2 what is read again (the encoder's second pass over its input).
__device__ __forceinline__ void st_cs_v4(uint4* p, uint4 v) {
  asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

__device__ __forceinline__ uint64_t ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// The value of an e4m3 byte (Section 3, all-finite eXmY): its sign and
// magnitude bits placed at fp32 bits 31 and 26..20 read as (1 + m/8) 2^(e-127)
// for e >= 1 and m 2^-129 for e = 0 (an fp32 subnormal); one exact
// multiplication by 2^120 gives the value.
__device__ __forceinline__ float e4m3_to_f32(uint32_t c) {
  return __uint_as_float(((c & 0x80u) << 24) | ((c & 0x7Fu) << 20)) * 0x1p120f;
}
// The same bit pattern (value 2^-120 times) for byte j of w: the byte moved
// to the top (sign at bit 31), an arithmetic shift right by 4 (the
// magnitude to bits 26..20, the sign repeated above it), bits 30..27 cleared.
__device__ __forceinline__ uint32_t e4m3_scaled_bits(uint32_t w, int j) {
  const uint32_t t = __byte_perm(w, 0u, 0x0444u | ((uint32_t)j << 12));
  return (uint32_t)((int32_t)t >> 4) & 0x87F00000u;
}

// The shard holding work item t of a batch: the largest s < n_shards with
// item_base[s] <= t (item_base is non-decreasing and item_base[0] = 0, so
// shards without items are skipped).  Warp-wide: each round the 32 lanes
// probe 32 evenly spaced entries of the remaining range and the last lane
// whose entry is <= t narrows it, so 1152 shards take 3 rounds of loads
// instead of the 11 dependent loads of a binary search.  Every lane returns
// the same shard.
__device__ __forceinline__ int shard_of_warp(const unsigned long long* item_base, int n_shards,
                                             unsigned long long t, int lane) {
  int lo = 0, hi = n_shards;  // item_base[lo] <= t; the shard lies in [lo, hi)
  while (hi - lo > 1) {
    const int step = (hi - lo + 31) / 32;
    const int idx = lo + lane * step;
    const unsigned le = __ballot_sync(0xffffffffu, idx < hi && item_base[idx] <= t);
    lo += (31 - __clz(le)) * step;  // lane 0 always qualifies
    hi = min(lo + step, hi);
  }
  return lo;
}

// Number of SMs of the current device (cached per device).
int sm_count();

// Programmatic dependent launch, between kernels of one call.  A kernel started
// with launch_after, directly behind another kernel of the same call, may have
// its CTAs resident, and the launch itself behind it, while that kernel still
// runs: that one calls dependents_may_start(), and this one touches no memory
// before dependency_wait(), which returns when that kernel is complete, and
// reads what that kernel wrote without the read-only cache (no __restrict__ on
// such pointers, or __ldcg).  The
// first kernel of a call is launched as usual: what comes before it in the
// stream is not known (behind a memset node of a captured graph, the wait does
// not hold).
__device__ __forceinline__ void dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dependents_may_start() { asm volatile("griddepcontrol.launch_dependents;"); }
template <typename... P, typename... A>
inline bool launch_after(void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...) == cudaSuccess;
}

// A named NVTX range around a host entry point: profilers (nsys, ncu with
// --nvtx) show the kernels a call launches under the call's name.  Without a
// profiler attached a push or pop is a call through an empty slot.
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

// --------------------------------------------- the split decoder's geometry
constexpr int kSpanWarps = 4;                    // warps of a team of the batch decoder; they share a code table
constexpr uint32_t kPiece = 128;                 // symbols per lane, about
constexpr uint64_t kSplitMax = 64ull << 20;      // symbols of a batch decoded split, at most: see split_most

// Geometry of a container's spans: a chunk takes `lanes` lanes, a warp
// `chunks` chunks (of one group), a group `per_group` spans.
struct SpanShape {
  uint32_t lanes, chunks, per_group;
  __device__ __forceinline__ explicit SpanShape(uint32_t cs) {
    lanes = (cs + kPiece - 1) / kPiece;
    chunks = 32 / lanes;
    per_group = (kGroupChunks + chunks - 1) / chunks;
  }
};

// ----------------------------------------------------------------- batches
// Batch workspace: 64 bytes of counters, item_base[n_shards + 1] (first work
// item of each shard; the last entry is the total), then one look-back word
// per encode work item.
// Counter word that says how a batch is decoded (decode.cu).
constexpr int kTicketWay = 1;
constexpr int kTicketSymbols = 2;  // the batch's symbols, in kWaySplit
constexpr int kTicketSlow = 3;     // of kSamples samples of its unsure shards (split_rule.cuh), in kWaySplit
enum DecodeWay : uint32_t { kWayGroups = 0, kWaySplit = 1, kWayEven = 2 };
struct BatchWs {
  unsigned int* ticket;                // [0] shared by encode / decode
  unsigned long long* item_base;
  unsigned long long* gstat;
  unsigned long long gstat_cap;        // look-back words available
};
inline bool batch_ws_layout(void* ws, size_t bytes, int n_shards, BatchWs* w) {
  const size_t head = 64 + 8 * (size_t)(n_shards + 1);
  if (bytes < head) return false;
  uint8_t* p = static_cast<uint8_t*>(ws);
  w->ticket = reinterpret_cast<unsigned int*>(p);
  w->item_base = reinterpret_cast<unsigned long long*>(p + 64);
  w->gstat = reinterpret_cast<unsigned long long*>(p + head);
  w->gstat_cap = (bytes - head) / 8;
  return true;
}

// kPlanDecodeGroups: decoding by warps too few for the split way.
enum PlanKind { kPlanEncode = 1, kPlanDecode = 2, kPlanDecodeGroups = 3 };
constexpr int kPlanThreads = 1024;
constexpr uint64_t kHistItem = 64 * 1024;  // symbols per histogram work item

// Launches plan_kernel (batch.cu), one CTA: the number of work items of every shard
// (encode: groups of 32 chunks; decode: the container's groups, or in a batch that
// is decoded split sets of kSpanWarps spans or groups), their exclusive prefix in
// item_base, and zeroed counters / look-back words.  Shards that cannot be
// processed get no items and set *status.  cs: the chunk size (encode), or the
// warps of decode_few_kernel (decode): up to as many groups are dealt out evenly.
bool launch_plan(PlanKind kind, const qlc_desc* descs, int n_shards, uint32_t cs, const BatchWs& w, uint32_t* status,
                 cudaStream_t st);

}  // namespace qlc
