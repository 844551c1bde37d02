// batch.cu -- planning and histogram kernels for batches of shards.
//
// A batch is an array of qlc_desc in device memory (the paper's own workload
// is 1152 shards per tensor type, Section 3).  plan_kernel turns the shard
// sizes into work items (encode / decode: groups of 32 chunks) with a
// block-wide prefix sum; the persistent kernels then take items from a device
// counter, so shards of very different sizes share the GPU evenly and no host
// round trip is needed.  The histogram kernel scans the sizes itself.
#define QLC_FILE_ID 4
#include "decode_span.cuh"
#include "hist_cols.cuh"

namespace qlc {

__host__ __device__ inline uint64_t encoded_bound(uint64_t n, uint32_t cs) {
  const uint64_t n_chunks = (n + cs - 1) / cs;
  const uint64_t group_syms = (uint64_t)kGroupChunks * cs;
  const uint64_t full = n / group_syms, rest = n % group_syms;
  uint64_t total = payload_start(n_chunks);
  total += full * align16((group_syms * kMaxCode + 7) / 8);
  if (rest) total += align16((rest * kMaxCode + 7) / 8);
  return total;
}

__device__ __forceinline__ bool al16(const void* p) {
  return (reinterpret_cast<uintptr_t>(p) & 15u) == 0;
}

// Inclusive prefix sums of the CTA's kHcThreads values v (thread t's at
// s_incl[t]); returns their total.  Called by every thread; s_warp holds a
// value per warp.
__device__ __forceinline__ unsigned long long cta_scan(unsigned long long v, unsigned long long* s_incl,
                                                       unsigned long long* s_warp, int tid) {
  static_assert(kHcWarps == 32, "the warps' totals are scanned by one warp");
  const int lane = tid & 31, warp = tid >> 5;
  auto warp_scan = [&](unsigned long long x) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long t = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += t;
    }
    return x;
  };
  const unsigned long long incl = warp_scan(v);
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  const unsigned long long w = warp_scan(s_warp[lane]);  // every warp for itself
  const unsigned long long before = __shfl_sync(0xffffffffu, w, (warp + 31) & 31);
  s_incl[tid] = incl + (warp ? before : 0ull);
  const unsigned long long total = __shfl_sync(0xffffffffu, w, 31);
  __syncthreads();
  return total;
}

// A shard's work: its groups (a shard that cannot be run has none and sets a
// status), and for decoding its symbols.
struct ShardWork {
  uint64_t groups, symbols;
};
__device__ ShardWork shard_work(PlanKind kind, const qlc_desc& d, uint32_t cs, uint32_t* status) {
  ShardWork w = {0, 0};
  if (kind == kPlanEncode) {
    const uint64_t n = d.in_bytes;
    const uint64_t n_chunks = (n + cs - 1) / cs;
    if (!d.out || !d.lut || !al16(d.out) || !al16(d.lut) || !aligned(d.out_bytes, 8) ||
        (n > 0 && (!d.in || !al16(d.in))) || n_chunks > 0xFFFFFFFFull) {
      set_status(status, QLC_ERR_ARG);
    } else if (d.out_cap < encoded_bound(n, cs)) {
      set_status(status, QLC_ERR_CAPACITY);
    } else {
      w.groups = n == 0 ? 1 : n_groups_of(n_chunks);
    }
    return w;
  }
  // decode: the container's groups, from a header that at least parses
  if (!d.in || !al16(d.in) || !aligned(d.out_bytes, 8) || (d.out_cap > 0 && (!d.out || !al16(d.out)))) {
    set_status(status, QLC_ERR_ARG);
    return w;
  }
  if (d.in_bytes < kIndexOff) {
    set_status(status, QLC_ERR_CORRUPT);
    return w;
  }
  const uint4 h0 = *static_cast<const uint4*>(d.in);                    // magic .. n
  const uint2 h1 = *reinterpret_cast<const uint2*>(static_cast<const uint8_t*>(d.in) + 16);  // chunk_symbols, n_chunks
  const uint64_t groups = n_groups_of(h1.y);
  if (h0.x != 0x31434C51u || groups > d.in_bytes / 16) {  // every group takes at least 16 payload bytes
    set_status(status, QLC_ERR_CORRUPT);
    return w;
  }
  w.groups = groups ? groups : 1;  // an empty container still gets its header checked
  w.symbols = min((uint64_t)h0.z | (uint64_t)h0.w << 32, (uint64_t)d.out_cap);
  return w;
}

// What the split rule looks at of a shard that has groups.
__device__ __forceinline__ bool shard_data(const qlc_desc& d, SplitData* sd, uint64_t* n_chunks) {
  return split_data(static_cast<const uint8_t*>(d.in), d.in_bytes, sd, n_chunks) && *n_chunks > 0;
}

// Of kSamples samples of the batch's shards that are looked at (split_samples):
// those that are slow.  Called by all threads; at most kSampleThreads samples, as
// many of every shard.
constexpr int kSampleThreads = 256;
__device__ uint32_t slow_samples(const qlc_desc* descs, int n_shards, const unsigned long long* item_base, uint64_t total,
                                 int tid) {
  __shared__ uint32_t words[kSampleThreads * kSampleWords];
  const int per = min(max(kSampleThreads / n_shards, 1), (int)kSamples);  // samples of a shard
  bool asked = false, slow = false;
  if (tid < kSampleThreads) {
    const int s = n_shards <= kSampleThreads ? tid / per : (int)((int64_t)tid * n_shards / kSampleThreads);
    SplitData sd;
    uint64_t n_chunks;
    if (s < n_shards && item_base[s] != 0 && shard_data(descs[s], &sd, &n_chunks) && split_samples(sd, kSplitBatch, total)) {
      asked = true;
      const uint32_t i = per > 1 ? tid % per * kSamples / per : tid % kSamples;
      slow = sample_is_slow(static_cast<const uint8_t*>(descs[s].in), sd, n_chunks, i, words + tid * kSampleWords);
    }
  }
  const uint32_t tries = __syncthreads_count(asked), found = __syncthreads_count(slow);
  return tries ? (found * kSamples + tries - 1) / tries : 0;
}

template <bool kDecode>
__global__ void __launch_bounds__(kPlanThreads, 1)
plan_kernel(PlanKind kind, const qlc_desc* descs, int n_shards, uint32_t cs, BatchWs w, uint32_t* status) {
  static_assert(kPlanThreads == kHcThreads, "cta_scan");
  __shared__ unsigned long long s_incl[kPlanThreads], s_warp[kPlanThreads / 32];
  __shared__ uint32_t s_chunk[2];
  const int tid = threadIdx.x;
  dependents_may_start();
  if (tid < 2) s_chunk[tid] = 0;  // published by the scan's barriers
  // every thread keeps its shards' groups, and the items they make in a split
  // batch, in item_base until the number of symbols has settled which it is
  unsigned long long symbols = 0;
  for (int s = tid; s < n_shards; s += kPlanThreads) {
    const ShardWork sw = shard_work(kind, descs[s], cs, status);
    symbols += sw.symbols;
    w.item_base[s] = sw.groups;
  }
  bool split = false;
  uint32_t slow = 0;
  if constexpr (kDecode) {
    symbols = cta_scan(symbols, s_incl, s_warp, tid);
    split = kind == kPlanDecode && symbols <= kSplitMax;
    if (split) {
      // Split where that pays for every shard: one that it does not pay for is
      // decoded a lane per chunk, which takes its chunk's chain, and that is what the
      // whole batch takes when it is dealt out evenly.  Only shards of chunks less
      // than half as long as the longest hold nothing up.
      uint32_t longest = 0, held = 0;  // chunks: of all shards, and of those that are not split
      bool asked = false;
      auto settle = [&](bool look) {
        for (int s = tid; s < n_shards; s += kPlanThreads) {
          SplitData sd;
          uint64_t n_chunks;
          const unsigned long long groups = w.item_base[s] & 0xFFFFFFFFu;
          if (groups == 0 || !shard_data(descs[s], &sd, &n_chunks)) continue;  // (nothing or a refusal to decode)
          const bool ask = split_samples(sd, kSplitBatch, symbols);
          asked = asked || ask;
          longest = max(longest, sd.cs);
          if (ask && look) continue;  // not yet known
          const bool pays = symbols <= split_most(sd, kSplitBatch, ask ? slow : 0);
          if (!pays) held = max(held, sd.cs);
          // items of kSpanWarps spans, or of as many groups
          const uint64_t parts = pays ? groups * SpanShape(sd.cs).per_group : groups;
          w.item_base[s] = groups | (parts + kSpanWarps - 1) / kSpanWarps << 32;
        }
      };
      settle(true);
      if (__syncthreads_or(asked)) {
        slow = slow_samples(descs, n_shards, w.item_base, symbols, tid);
        settle(false);
      }
      longest = __reduce_max_sync(0xffffffffu, longest);
      held = __reduce_max_sync(0xffffffffu, held);
      if (tid % 32 == 0) {
        atomicMax(&s_chunk[0], longest);
        atomicMax(&s_chunk[1], held);
      }
      __syncthreads();
      split = 2 * s_chunk[1] <= s_chunk[0];
    }
  }
  // the 64 bytes of counters
  if (tid < 16) w.ticket[tid] = !split ? 0u : tid == kTicketSymbols ? (uint32_t)symbols : tid == kTicketSlow ? slow : 0u;
  unsigned long long total = 0;
  for (int base = 0; base < n_shards; base += kPlanThreads) {
    const int s = base + tid;
    unsigned long long cnt = 0;
    if (s < n_shards) {
      const unsigned long long v = w.item_base[s], groups = v & 0xFFFFFFFFu;
      cnt = split && v >> 32 ? v >> 32 : groups;
    }
    const unsigned long long part = cta_scan(cnt, s_incl, s_warp, tid);
    if (s < n_shards) w.item_base[s] = total + s_incl[tid] - cnt;
    total += part;
  }
  if (kind == kPlanEncode && total > w.gstat_cap) {
    if (tid == 0) set_status(status, QLC_ERR_CAPACITY);
    total = 0;
  }
  if (tid == 0) {
    w.item_base[n_shards] = total;
    if (kDecode) w.ticket[kTicketWay] = split ? kWaySplit : total <= cs ? kWayEven : kWayGroups;
  }
  if (kind == kPlanEncode)
    for (unsigned long long i = tid; i < total; i += kPlanThreads) w.gstat[i] = 0;
}

bool launch_plan(PlanKind kind, const qlc_desc* descs, int n_shards, uint32_t cs, const BatchWs& w, uint32_t* status,
                 cudaStream_t st) {
  if (kind == kPlanEncode)
    plan_kernel<false><<<1, kPlanThreads, 0, st>>>(kind, descs, n_shards, cs, w, status);
  else
    plan_kernel<true><<<1, kPlanThreads, 0, st>>>(kind, descs, n_shards, cs, w, status);
  return cudaGetLastError() == cudaSuccess;
}

// ------------------------------------------------------------- histograms

// Histogram work items of shard s: its 64 KiB pieces, and one more without
// bytes that stands for the flush after it (about as long as a piece), so that
// a run of small shards is not all one CTA's.  0 for a shard that is empty or
// cannot be read (its encode reports it: histograms have no status word).
__device__ __forceinline__ unsigned long long hist_items(const qlc_desc* descs, int n_shards, int s) {
  if (s >= n_shards) return 0;
  const qlc_desc* d = descs + s;
  return d->in && al16(d->in) && d->in_bytes ? (d->in_bytes + kHistItem - 1) / kHistItem + 1 : 0;
}

// Each CTA (32 warps, hist_cols.cuh; one per SM) takes a contiguous run of
// items.  Its items of one shard are one contiguous byte range, counted in a
// single streaming pass; the table is flushed into a shard's histogram when
// the target histogram changes (never, for one shared histogram).  A run is
// 1 / SMs of the batch's items, so a counter stays below 2^32 for any batch
// smaller than 2^32 x SMs bytes, far above the device's memory.
// Every CTA scans the shard sizes itself, kHcThreads at a time (once for a
// batch of up to 1024 shards, else once for the total and once for its run):
// a load and two warp scans, where a planning kernel of its own and the search
// in its prefix cost a launch and a chain of dependent loads.  24 shards of
// 4 KiB - 64 MiB (139 MB): 30 us, from 4.5 us of planning and 43.5 us; 1152
// shards (3.4 GB): 541-547 us (6.2 TB/s), from 600 us.
__global__ void __launch_bounds__(kHcThreads, 1)
hist_batch_kernel(const qlc_desc* descs, int n_shards, unsigned long long* hists, int shared) {
  __shared__ __align__(16) uint32_t cols[kHcColWords];
  __shared__ unsigned long long s_incl[kHcThreads], s_warp[kHcWarps];
  const int tid = threadIdx.x, lane = tid & 31;
  zero_cols(cols, tid);  // published by the scan's barriers
  unsigned long long cnt = hist_items(descs, n_shards, tid), total = cta_scan(cnt, s_incl, s_warp, tid);
  for (int base = kHcThreads; base < n_shards; base += kHcThreads)
    total += cta_scan(hist_items(descs, n_shards, base + tid), s_incl, s_warp, tid);
  const unsigned long long per = (total + gridDim.x - 1) / gridDim.x;
  const unsigned long long t0 = (unsigned long long)blockIdx.x * per;
  const unsigned long long t1 = min(t0 + per, total);
  if (t0 >= t1) return;
  const uint32_t col = lane_col(cols, lane);
  int target = -1;  // the histogram the table's counts belong to
  unsigned long long first = 0;  // first item of the scanned shards
  for (int base = 0; base < n_shards && first < t1; base += kHcThreads) {
    unsigned long long part = s_incl[kHcThreads - 1];
    if (n_shards > kHcThreads) {
      __syncthreads();
      part = cta_scan(hist_items(descs, n_shards, base + tid), s_incl, s_warp, tid);
    }
    if (first + part > t0) {
      // the first shard here with an item at or after t0: the number of
      // shards that end at or before it
      int j = 0;
      {
        const unsigned long long rel = t0 > first ? t0 - first : 0;
        for (int half = kHcThreads / 2; half > 0; half >>= 1)
          if (s_incl[j + half - 1] <= rel) j += half;
      }
      for (; j < kHcThreads && base + j < n_shards; j++) {
        const unsigned long long sb = first + (j ? s_incl[j - 1] : 0ull), se = first + s_incl[j];  // the shard's items
        if (sb >= t1) break;
        if (sb == se) continue;
        const int tgt = shared ? 0 : base + j;
        if (target >= 0 && tgt != target)
          flush_cols(cols, hists + (size_t)(QLC_GUARD(target < n_shards, nullptr) ? target : 0) * 256, tid, true);
        target = tgt;
        const uint8_t* in = static_cast<const uint8_t*>(descs[base + j].in);
        const uint64_t n = descs[base + j].in_bytes;
        const uint64_t beg = min((uint64_t)((max(t0, sb) - sb) * kHistItem), n);  // a multiple of 16, or the end
        const uint64_t end = min((uint64_t)((min(t1, se) - sb) * kHistItem), n);
        const uint64_t vb = beg / 16, ve = end / 16;
        if (beg < end) {
          count_span(reinterpret_cast<const uint4*>(in) + vb, ve - vb, col, tid);
          count_bytes(in + ve * 16, end - ve * 16, col, tid);
        }
      }
    }
    first += part;
  }
  if (target >= 0) flush_cols(cols, hists + (size_t)target * 256, tid, false);
}

}  // namespace qlc

using namespace qlc;

extern "C" {

size_t qlc_batch_workspace_size(int n_shards, uint64_t total_symbols, uint32_t chunk_symbols) {
  if (n_shards < 1 || !chunk_symbols_ok(chunk_symbols)) return 0;
  const uint64_t group_syms = (uint64_t)kGroupChunks * chunk_symbols;
  const uint64_t items = (total_symbols + group_syms - 1) / group_syms + (uint64_t)n_shards;
  return (size_t)(64 + 8 * (uint64_t)(n_shards + 1) + 8 * items);
}

qlc_status qlc_histogram_batch(const qlc_desc* d_descs, int n_shards, uint64_t* d_hists, int shared,
                               void* d_ws, size_t ws_bytes, qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_histogram_batch");
  if (!d_descs || n_shards < 1 || !d_hists || !d_ws) return QLC_ERR_ARG;
  if (!aligned(d_ws, 16) || !aligned(d_descs, 16) || !aligned(d_hists, 8)) return QLC_ERR_ARG;
  BatchWs w;
  if (!batch_ws_layout(d_ws, ws_bytes, n_shards, &w)) return QLC_ERR_CAPACITY;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const size_t hist_bytes = (size_t)(shared ? 1 : n_shards) * 256 * sizeof(uint64_t);
  if (cudaMemsetAsync(d_hists, 0, hist_bytes, st) != cudaSuccess) return QLC_ERR_CUDA;
  hist_batch_kernel<<<sm_count(), kHcThreads, 0, st>>>(d_descs, n_shards,
                                                       reinterpret_cast<unsigned long long*>(d_hists), shared ? 1 : 0);
  return cudaGetLastError() == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
}

}  // extern "C"

namespace qlc {
QLC_DEFINE_CHECK_TAKE(check_take_batch)
}  // namespace qlc
