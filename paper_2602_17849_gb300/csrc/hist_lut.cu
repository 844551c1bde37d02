// hist_lut.cu -- byte histogram (Section 4) and LUT construction (Section 7)
// kernels of libqlc, plus their C-ABI entry points.
#define QLC_FILE_ID 3
#include "hist_cols.cuh"
#include "lut.cuh"
#include "split_rule.cuh"
#include "../../include/qlc_testing.h"

#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <functional>
#include <mutex>

namespace qlc {

// One CTA of 32 warps per SM counts a contiguous slice of the tensor
// (hist_cols.cuh); the last CTA also counts the bytes after the last whole
// 16-byte vector.  A single CTA (small tensors) can write the counts itself
// (overwrite): no memset has to run before it.
__global__ void __launch_bounds__(kHcThreads, 1)
hist_kernel(const uint8_t* __restrict__ in, uint64_t n, unsigned long long* __restrict__ hist, bool overwrite) {
  __shared__ __align__(16) uint32_t cols[kHcColWords];
  const int tid = threadIdx.x, lane = tid & 31;
  dependents_may_start();
  zero_cols(cols, tid);
  __syncthreads();
  const uint32_t col = lane_col(cols, lane);
  const uint64_t nvec = n / 16;
  const uint64_t per = (nvec + gridDim.x - 1) / gridDim.x;
  const uint64_t beg = (uint64_t)blockIdx.x * per;
  const uint64_t end = min(beg + per, nvec);
  if (beg < end) count_span(reinterpret_cast<const uint4*>(in) + beg, end - beg, col, tid);
  if (blockIdx.x == gridDim.x - 1) count_bytes(in + nvec * 16, n - nvec * 16, col, tid);
  if (overwrite) {
    __syncthreads();
    const uint32_t t = sum_cols(cols, tid);
    if ((tid & 3) == 0) hist[tid >> 2] = t;
  } else {
    flush_cols(cols, hist, tid, false);
  }
}

// Fewest vectors per histogram CTA (64 KiB): up to there one CTA counts alone
// and no memset precedes it.
constexpr uint64_t kHistCtaVecs = 4096;

// One CTA per histogram: CTA b builds luts[b] from hists[b * 256 ...].
__global__ void __launch_bounds__(kLutThreads)
lut_best_kernel(const unsigned long long* __restrict__ hists, SchemeSet set, qlc_lut* __restrict__ luts) {
  __shared__ __align__(16) unsigned long long key[256];
  __shared__ unsigned long long bits[8][kLutThreads / 32];
  const int tid = threadIdx.x;
  dependents_may_start();
  dependency_wait();
  const LutRow row = rank_and_choose(hists + (size_t)blockIdx.x * 256, set, key, bits, tid);
  write_lut(luts + blockIdx.x, row, set, tid);
}

// The driver entry points come through the runtime, so the library needs no
// link to the driver library.
unsigned long long current_context_id() {
  using GetCurrent = CUresult (*)(CUcontext*);
  using GetId = CUresult (*)(CUcontext, unsigned long long*);
  static GetCurrent get_current = nullptr;
  static GetId get_id = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_current = reinterpret_cast<GetCurrent>(f);
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_id = reinterpret_cast<GetId>(f);
  });
  CUcontext ctx = nullptr;
  unsigned long long id = 0;
  if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx || get_id(ctx, &id) != CUDA_SUCCESS)
    return 0;
  return id;
}

int sm_count() {
  // one atomic slot per device below 64 (any thread may fill it; all write
  // the same value); other devices ask the runtime each time
  static std::atomic<int> cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 148;
  if (dev < 64) {
    const int c = cached[dev].load(std::memory_order_relaxed);
    if (c > 0) return c;
  }
  int v = 0;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 148;
  if (dev < 64) cached[dev].store(v, std::memory_order_relaxed);
  return v;
}

}  // namespace qlc

using namespace qlc;

static const qlc_scheme kTable1 = {{8, 8, 8, 8, 8, 16, 32, 168}, {3, 3, 3, 3, 3, 4, 5, 8}, 1, {0}};
static const qlc_scheme kTable2 = {{2, 8, 8, 8, 8, 32, 32, 158}, {1, 3, 3, 3, 3, 5, 5, 8}, 2, {0}};

static bool scheme_valid(const qlc_scheme* s) {
  if (!s || !scheme_ok(s->area_n, s->area_bits)) return false;
  if (s->id == 1 || s->id == 2) {
    const qlc_scheme& t = s->id == 1 ? kTable1 : kTable2;
    for (int i = 0; i < 8; i++)
      if (t.area_n[i] != s->area_n[i] || t.area_bits[i] != s->area_bits[i]) return false;
  } else if (s->id != 0) {
    return false;
  }
  return true;
}

static qlc_scheme clean_scheme(const qlc_scheme* s) {
  qlc_scheme c = *s;
  for (int i = 0; i < 7; i++) c.reserved[i] = 0;
  return c;
}

namespace qlc {

bool scheme_set(const qlc_scheme* h_schemes, int n_schemes, SchemeSet* set) {
  if (!h_schemes || n_schemes < 1 || n_schemes > 8) return false;
  set->count = n_schemes;
  for (int k = 0; k < n_schemes; k++) {
    if (!scheme_valid(&h_schemes[k])) return false;
    set->s[k] = clean_scheme(&h_schemes[k]);
  }
  return true;
}

qlc_status launch_histogram(const uint8_t* d_in, size_t n, uint64_t* d_hist, int accumulate, cudaStream_t st) {
  // One CTA per SM, at least kHistCtaVecs vectors each; a CTA counts under
  // 2^31 bytes.
  const uint64_t nvec = n / 16;
  uint64_t grid = (nvec + kHistCtaVecs - 1) / kHistCtaVecs;
  const uint64_t cap = (uint64_t)sm_count();
  if (grid > cap) grid = cap;
  const uint64_t floor_grid = (nvec >> 27) + 1;
  if (grid < floor_grid) grid = floor_grid;
  if (grid > 0x7fffffffu) return QLC_ERR_ARG;
  const bool overwrite = !accumulate && n > 0 && grid == 1;
  if (!accumulate && !overwrite && cudaMemsetAsync(d_hist, 0, 256 * sizeof(uint64_t), st) != cudaSuccess)
    return QLC_ERR_CUDA;
  if (n == 0) return QLC_OK;
  hist_kernel<<<(int)grid, kHcThreads, 0, st>>>(d_in, n, reinterpret_cast<unsigned long long*>(d_hist), overwrite);
  return cudaGetLastError() == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
}

qlc_status launch_luts(const uint64_t* d_hists, int n_luts, const SchemeSet& set, qlc_lut* d_luts, bool after,
                       cudaStream_t st) {
  const unsigned long long* h = reinterpret_cast<const unsigned long long*>(d_hists);
  if (after)
    launch_after(lut_best_kernel, n_luts, kLutThreads, 0, st, h, set, d_luts);
  else
    lut_best_kernel<<<n_luts, kLutThreads, 0, st>>>(h, set, d_luts);
  return cudaGetLastError() == cudaSuccess ? QLC_OK : QLC_ERR_CUDA;
}

}  // namespace qlc

extern "C" {

int qlc_version(void) { return QLC_VERSION; }

const char* qlc_status_string(qlc_status s) {
  switch (s) {
    case QLC_OK: return "ok";
    case QLC_ERR_ARG: return "invalid argument";
    case QLC_ERR_CAPACITY: return "buffer too small";
    case QLC_ERR_CORRUPT: return "corrupt container";
    case QLC_ERR_TIMEOUT: return "device wait timed out";
    case QLC_ERR_CUDA: return "CUDA error";
    case QLC_ERR_CHECK: return "index check failed";
  }
  return "unknown status";
}

qlc_status qlc_scheme_table(int id, qlc_scheme* out) {
  if (!out || (id != 1 && id != 2)) return QLC_ERR_ARG;
  *out = id == 1 ? kTable1 : kTable2;
  return QLC_OK;
}

int qlc_scheme_check(const qlc_scheme* s) { return scheme_valid(s) ? 1 : 0; }

qlc_status qlc_histogram(const uint8_t* d_in, size_t n, uint64_t* d_hist, int accumulate,
                         qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_histogram");
  if (!d_hist || (n > 0 && !d_in)) return QLC_ERR_ARG;
  if (!aligned(d_in, 16) || !aligned(d_hist, 8)) return QLC_ERR_ARG;
  return launch_histogram(d_in, n, d_hist, accumulate, reinterpret_cast<cudaStream_t>(stream));
}

qlc_status qlc_build_lut(const uint64_t* d_hist, const qlc_scheme* h_scheme, qlc_lut* d_lut,
                         qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_build_lut");
  if (!d_hist || !d_lut || !scheme_valid(h_scheme)) return QLC_ERR_ARG;
  if (!aligned(d_hist, 8) || !aligned(d_lut, 16)) return QLC_ERR_ARG;
  SchemeSet set;
  set.count = 1;
  set.s[0] = clean_scheme(h_scheme);
  return launch_luts(d_hist, 1, set, d_lut, false, reinterpret_cast<cudaStream_t>(stream));
}

qlc_status qlc_build_lut_best(const uint64_t* d_hist, const qlc_scheme* h_schemes, int n_schemes,
                              qlc_lut* d_lut, qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_build_lut_best");
  if (!d_hist || !d_lut || !h_schemes || n_schemes < 1 || n_schemes > 8) return QLC_ERR_ARG;
  if (!aligned(d_hist, 8) || !aligned(d_lut, 16)) return QLC_ERR_ARG;
  SchemeSet set;
  if (!scheme_set(h_schemes, n_schemes, &set)) return QLC_ERR_ARG;
  return launch_luts(d_hist, 1, set, d_lut, false, reinterpret_cast<cudaStream_t>(stream));
}

qlc_status qlc_build_lut_batch(const uint64_t* d_hists, int n_luts, const qlc_scheme* h_schemes,
                               int n_schemes, qlc_lut* d_luts, qlc_stream_t stream) {
  NvtxRange nvtx_range("qlc_build_lut_batch");
  if (!d_hists || !d_luts || !h_schemes || n_luts < 1 || n_schemes < 1 || n_schemes > 8)
    return QLC_ERR_ARG;
  if (!aligned(d_hists, 8) || !aligned(d_luts, 16)) return QLC_ERR_ARG;
  SchemeSet set;
  if (!scheme_set(h_schemes, n_schemes, &set)) return QLC_ERR_ARG;
  return launch_luts(d_hists, n_luts, set, d_luts, false, reinterpret_cast<cudaStream_t>(stream));
}

qlc_status qlc_build_lut_host(const uint64_t* h_hist, const qlc_scheme* h_scheme, qlc_lut* h_lut) {
  if (!h_hist || !h_lut || !scheme_valid(h_scheme)) return QLC_ERR_ARG;
  h_lut->scheme = clean_scheme(h_scheme);
  for (int s = 0; s < 256; s++) {
    int r = 0;
    for (int t = 0; t < 256; t++) r += (h_hist[t] > h_hist[s]) || (h_hist[t] == h_hist[s] && t < s);
    h_lut->enc[s] = (uint16_t)lut_entry(h_lut->scheme, r);
    h_lut->dec[r] = (uint8_t)s;
  }
  return QLC_OK;
}

// Section 8 leaves the choice of areas, symbols per area and code lengths as
// future work.  Within the family this library codes (qlc_scheme), the best
// scheme for a histogram is found exhaustively: areas 1..7 are complete
// (2^b ranks, b non-decreasing in 0..7), area 8 takes the remaining ranks,
// either raw (8 bits) or complete when their number is a power of two.  Cost
// = sum over ranks of count * code length, counts taken in decreasing order.
qlc_status qlc_scheme_search(const uint64_t* h_hist, qlc_scheme* out, uint64_t* out_bits) {
  if (!h_hist || !out) return QLC_ERR_ARG;
  uint64_t c[256];
  for (int i = 0; i < 256; i++) c[i] = h_hist[i];
  std::sort(c, c + 256, std::greater<uint64_t>());
  uint64_t pre[257];
  pre[0] = 0;
  for (int i = 0; i < 256; i++) pre[i + 1] = pre[i] + c[i];
  uint64_t best = ~0ull;
  uint8_t best_b[8] = {0};
  uint16_t best_n[8] = {0};
  uint8_t b[8];
  // depth-first over b[0] <= b[1] <= ... <= b[6]
  struct Rec {
    static void go(int i, uint32_t base, uint64_t cost, uint8_t* b, const uint64_t* pre, uint64_t* best,
                   uint8_t* best_b, uint16_t* best_n) {
      if (i == 7) {
        const uint32_t rem = 256 - base;
        uint32_t last_bits = 8;
        if ((rem & (rem - 1)) == 0 && rem <= 128) {  // power of two: complete area
          uint32_t lb = 0;
          while ((1u << lb) < rem) lb++;
          if (lb >= b[6]) last_bits = lb;
        }
        const uint64_t total = cost + (3 + last_bits) * (pre[256] - pre[base]);
        if (total < *best) {
          *best = total;
          for (int k = 0; k < 7; k++) {
            best_b[k] = b[k];
            best_n[k] = (uint16_t)(1u << b[k]);
          }
          best_b[7] = (uint8_t)last_bits;
          best_n[7] = (uint16_t)rem;
        }
        return;
      }
      for (uint32_t bi = i ? b[i - 1] : 0; bi <= 7; bi++) {
        const uint32_t n = 1u << bi;
        if (base + n > 255) break;  // area 8 keeps at least one rank
        b[i] = (uint8_t)bi;
        go(i + 1, base + n, cost + (3 + bi) * (pre[base + n] - pre[base]), b, pre, best, best_b, best_n);
      }
    }
  };
  Rec::go(0, 0, 0, b, pre, &best, best_b, best_n);
  qlc_scheme sc = {};
  for (int i = 0; i < 8; i++) {
    sc.area_n[i] = best_n[i];
    sc.area_bits[i] = best_b[i];
  }
  sc.id = 0;
  for (int id = 1; id <= 2; id++) {
    const qlc_scheme& t = id == 1 ? kTable1 : kTable2;
    bool same = true;
    for (int i = 0; i < 8; i++) same = same && t.area_n[i] == sc.area_n[i] && t.area_bits[i] == sc.area_bits[i];
    if (same) sc.id = (uint8_t)id;
  }
  *out = sc;
  if (out_bits) *out_bits = best;
  return QLC_OK;
}

qlc_status qlc_peek_header(const void* h_hdr, size_t hdr_bytes, uint64_t* n, uint64_t* container_bytes) {
  if (!h_hdr || hdr_bytes < QLC_HEADER_BYTES) return QLC_ERR_ARG;
  const uint8_t* p = static_cast<const uint8_t*>(h_hdr);
  auto le = [&](int off, int bytes) {
    uint64_t v = 0;
    for (int i = 0; i < bytes; i++) v |= (uint64_t)p[off + i] << (8 * i);
    return v;
  };
  if (p[0] != 'Q' || p[1] != 'L' || p[2] != 'C' || p[3] != '1' || le(4, 2) != QLC_VERSION)
    return QLC_ERR_CORRUPT;
  const uint64_t nn = le(8, 8);
  const uint64_t n_chunks = le(20, 4);
  if (n) *n = nn;
  if (container_bytes) *container_bytes = payload_start(n_chunks) + le(48, 8);
  return QLC_OK;
}

}  // extern "C"

namespace qlc {
QLC_DEFINE_CHECK_TAKE(check_take_hist)
}  // namespace qlc

extern "C" uint32_t qlc_test_check_take(void) {
#ifdef QLC_CHECKED
  const uint32_t v[5] = {qlc::check_take_decode(), qlc::check_take_encode(), qlc::check_take_hist(),
                         qlc::check_take_batch(), qlc::check_take_quant()};
  for (uint32_t x : v)
    if (x) return x;
  return 0;
#else
  return 0xFFFFFFFFu;
#endif
}

extern "C" int qlc_test_once_per_context(const int* dev, const uint64_t* id, const uint64_t* id_after, int calls) {
  qlc::OncePerContext once;
  int done = 0;
  for (int i = 0; i < calls; i++) {
    bool acted = false;
    once.ensure(dev[i], [&] { return acted ? (unsigned long long)id_after[i] : (unsigned long long)id[i]; },
                [&] { return acted = true; });
    done += acted;
  }
  return done;
}

static qlc::SplitData split_data_of(const void* h_hdr) {
  const uint8_t* p = static_cast<const uint8_t*>(h_hdr);
  qlc::SplitData d = {};
  memcpy(&d.cs, p + 16, 4);
  memcpy(&d.n, p + 8, 8);
  memcpy(&d.payload_bytes, p + 48, 8);
  memcpy(&d.len_lo, p + 40, 4);
  memcpy(&d.len_hi, p + 44, 4);
  d.len_lo += 0x03030303u;
  d.len_hi += 0x03030303u;
  return d;
}
extern "C" uint64_t qlc_test_split_most(const void* h_hdr, int into, uint32_t slow) {
  return qlc::split_most(split_data_of(h_hdr), (qlc::SplitInto)into, slow);
}
extern "C" int qlc_test_split_samples(const void* h_hdr, int into, uint64_t total) {
  return qlc::split_samples(split_data_of(h_hdr), (qlc::SplitInto)into, total);
}
