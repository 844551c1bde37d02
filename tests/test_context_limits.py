"""What is set up once in a CUDA context is set up again in the next one: after
a device reset, or in a second context on the device.  The ids are made up, so
no context is touched; two contexts in turn are tested on a GPU."""
import ctypes
import os
import subprocess
import sys

import pytest

from paper_2602_17849_gb300 import _build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _times(dev, ids, after=None):
    lib = ctypes.CDLL(_build.build())
    n = len(dev)
    return lib.qlc_test_once_per_context((ctypes.c_int * n)(*dev), (ctypes.c_uint64 * n)(*ids),
                                         (ctypes.c_uint64 * n)(*(after or ids)), n)


@pytest.mark.parametrize("dev,ids,want", [
    ([0, 0, 0], [7, 7, 7], 1),
    ([0, 0, 0], [7, 8, 8], 2),           # the device was reset: a new context
    ([0, 0, 0, 0], [7, 8, 7, 8], 4),     # two contexts in turn
    ([0, 1, 0, 1], [7, 8, 7, 8], 2),     # two devices
    ([0, 0], [0, 0], 2),                 # no id: every time
    ([64, 64, 200], [7, 7, 9], 3),       # devices past the table
])
def test_once_in_every_context(dev, ids, want):
    assert _times(dev, ids) == want


def test_first_call_makes_the_context():
    assert _times([0, 0, 0], [0, 7, 7], [7, 7, 7]) == 1


TWO = r"""
import ctypes, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
import torch  # the library's binding loads it; it makes no context here
from paper_2602_17849_gb300 import qlc
rt = ctypes.CDLL("libcuda.so.1")
dev, u64 = ctypes.c_int(), ctypes.c_uint64
def ok(r):
    assert r == 0, r
ok(rt.cuInit(0)); ok(rt.cuDeviceGet(ctypes.byref(dev), 0))
def once():
    # 4100 chunks: the kernel with a raised limit; buffers by the driver, in the current context
    n, cs = 4100 * 128, 128
    x = np.random.default_rng(1).integers(0, 256, n, dtype=np.uint8)
    def alloc(b):
        p = u64(); ok(rt.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(b))); return p.value
    cap = qlc.qlc_encoded_size(n, cs)
    d_in, d_hist, d_lut, d_out, d_res = alloc(n), alloc(2048), alloc(qlc.LUT_BYTES), alloc(cap), alloc(32)
    d_back = alloc(n)
    ok(rt.cuMemcpyHtoD_v2(u64(d_in), x.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(n)))
    ok(rt.cuMemsetD8_v2(u64(d_res), 0, ctypes.c_size_t(32)))
    L, s = qlc.lib, qlc.qlc_scheme_table(1)
    P, sz = ctypes.c_void_p, ctypes.c_size_t
    L.qlc_encode_noalloc.argtypes = [P, sz, P, ctypes.c_uint32, P, sz, P, P, P]
    assert L.qlc_histogram(d_in, n, d_hist, 0, 0) == 0
    assert L.qlc_build_lut(d_hist, ctypes.byref(s), d_lut, 0) == 0
    r = L.qlc_encode_noalloc(d_in, n, d_lut, cs, d_out, cap, d_res, d_res + 16, 0)
    assert r == 0, f"encode: {r}"
    r = L.qlc_decode(d_out, cap, d_back, n, d_res + 8, d_res + 16, 0)
    assert r == 0, f"decode: {r}"
    ok(rt.cuCtxSynchronize())
    res, back = np.zeros(4, np.uint64), np.zeros(n, np.uint8)
    ok(rt.cuMemcpyDtoH_v2(res.ctypes.data_as(P), u64(d_res), sz(32)))
    ok(rt.cuMemcpyDtoH_v2(back.ctypes.data_as(P), u64(d_back), sz(n)))
    assert res[2] == 0 and res[1] == n and np.array_equal(back, x)
ctx = ctypes.c_void_p()
ok(rt.cuDevicePrimaryCtxRetain(ctypes.byref(ctx), dev)); ok(rt.cuCtxSetCurrent(ctx))
once()
other = ctypes.c_void_p()
ok(rt.cuCtxCreate_v2(ctypes.byref(other), 0, dev))  # current from here on
once()
ok(rt.cuCtxSetCurrent(ctx))
once()
print("both contexts")
"""


@pytest.mark.gpu
def test_encode_and_decode_in_two_contexts():
    _build.build()
    r = subprocess.run([sys.executable, "-c", TWO, ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "both contexts" in r.stdout, r.stdout + r.stderr
