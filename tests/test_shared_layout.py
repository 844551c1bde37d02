"""Kernels that address shared memory by constants stay inside what the host
asks for, wherever the driver lets dynamic shared memory start."""
import ctypes

import pytest

from paper_2602_17849_gb300 import _build

SM_BYTES = 228 * 1024      # shared memory of an SM
RESERVED = 1024            # taken by the driver for every resident CTA
CTA_MOST = 227 * 1024


@pytest.fixture(scope="module")
def lib():
    return ctypes.CDLL(_build.build())


def _use(call):
    v = [ctypes.c_uint32() for _ in range(3)]
    call(*[ctypes.byref(x) for x in v])
    return [x.value for x in v]


def _inside_for_every_start(addr, size, requested):
    # the kernels refuse a start above addr; from any other the used bytes must fit
    return all(start + requested >= addr + size for start in range(0, addr + 1, 16))


def test_encode_kernel(lib):
    addr, size, requested = _use(lib.qlc_test_encode_smem)
    assert size > 0 and _inside_for_every_start(addr, size, requested)
    assert 2 * (requested + RESERVED) <= SM_BYTES  # two CTAs per SM


@pytest.mark.parametrize("warps", [4, 8, 32])
def test_quantise_kernel(lib, warps):
    addr, size, requested = _use(lambda *a: lib.qlc_test_quantize_smem(warps, *a))
    assert size > 0 and _inside_for_every_start(addr, size, requested)
    assert requested <= CTA_MOST
