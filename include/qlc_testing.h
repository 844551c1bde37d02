/*
 * qlc_testing.h -- test hooks of libqlc (not part of the codec's API).
 *
 * The paper has no counterpart to these; they exist so that tests can drive
 * the library's failure paths on a GPU without faulting, trapping or hanging
 * it.
 */
#ifndef QLC_TESTING_H
#define QLC_TESTING_H

#include "qlc.h"

#ifdef __cplusplus
extern "C" {
#endif

/* Runs qlc_encode's kernel with its group counter starting at 1 instead of 0,
 * so group 0 is never encoded and group 1's look-back waits for a value that
 * nobody writes.  Every device-side wait is bounded (about 1 s); the call
 * must end with QLC_ERR_TIMEOUT in *d_status, later groups giving up at once
 * through the propagated error flag, and leave the GPU usable.  Arguments as
 * for qlc_encode; n must span at least two groups of 32 chunks. */
qlc_status qlc_test_encode_stalled_lookback(const uint8_t *d_in, size_t n, const qlc_lut *d_lut,
                                            uint32_t chunk_symbols, uint8_t *d_out, size_t out_cap,
                                            void *d_ws, size_t ws_bytes, uint64_t *d_out_bytes,
                                            uint32_t *d_status, qlc_stream_t stream);

/* The checked build of the library (compiled with -DQLC_CHECKED) guards every
 * index into global and shared memory that its kernels compute from data: an
 * index out of its range skips the access, sets *d_status to QLC_ERR_CHECK
 * where the call has a status word, and records where it happened.  This
 * returns that record for the first failed check since the last call
 * (file number << 16 | source line; 0 if no check failed) and clears it.
 * Synchronises the device.  In a normal build it returns 0xFFFFFFFF. */
uint32_t qlc_test_check_take(void);

/* How often the library would raise a kernel's shared-memory limit over a
 * sequence of calls, call i on device dev[i] in the context with the id id[i] (0:
 * none), which is id_after[i] once the runtime has been called.  Host only. */
int qlc_test_once_per_context(const int *dev, const uint64_t *id, const uint64_t *id_after, int calls);

/* Shared-memory use of the encode kernel, and of the quantise kernel with
 * `warps` warps: `size` bytes from the fixed shared address `addr` on, out of
 * `requested` bytes of dynamic shared memory, whose start may be any address up
 * to addr.  Host only. */
void qlc_test_encode_smem(uint32_t *addr, uint32_t *size, uint32_t *requested);
void qlc_test_quantize_smem(int warps, uint32_t *addr, uint32_t *size, uint32_t *requested);

/* What a batch is launched with for these knobs (NULL: the defaults): encode CTAs
 * and decode warps per SM.  Host only. */
int qlc_test_encode_ctas(const qlc_launch *h_launch);
int qlc_test_decode_warps(const qlc_launch *h_launch);

/* The rule by which containers are decoded split, for a host copy of a
 * container's first 64 bytes, decoded to codes (into 0), to values (1) or as a
 * shard of a batch (2): the most symbols of one launch for which it is, when `slow`
 * of 32 samples are places where readers are slow to find the codeword
 * boundaries; and whether samples are taken when `total` symbols are decoded in
 * the launch (without them slow counts as 0).  Host only. */
uint64_t qlc_test_split_most(const void *h_hdr, int into, uint32_t slow);
int qlc_test_split_samples(const void *h_hdr, int into, uint64_t total);

/* Counter words that qlc_decode_batch leaves at the start of its workspace: how
 * the batch was decoded (0: a warp per group, from a counter; 1: split; 2: a warp
 * per group, dealt out evenly), its symbols, and its slow samples (both 0 unless
 * split). */
#define QLC_TEST_WS_WAY 1
#define QLC_TEST_WS_SYMBOLS 2
#define QLC_TEST_WS_SLOW 3

#ifdef __cplusplus
}
#endif
#endif /* QLC_TESTING_H */
