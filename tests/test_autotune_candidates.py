"""The autotuner's candidates are different launches, the library's own among them."""
import ctypes

from paper_2602_17849_gb300 import _build, autotune


class Launch(ctypes.Structure):
    _fields_ = [("encode_ctas_per_sm", ctypes.c_uint16), ("decode_ctas_per_sm", ctypes.c_uint16),
                ("reserved", ctypes.c_uint32)]


def test_candidates_are_distinct_and_hold_the_default():
    lib = ctypes.CDLL(_build.build())
    enc = [lib.qlc_test_encode_ctas(ctypes.byref(Launch(v, 0, 0))) for v in autotune.ENC_CTAS]
    dec = [lib.qlc_test_decode_warps(ctypes.byref(Launch(0, v, 0))) for v in autotune.DEC_CTAS]
    assert enc == list(autotune.ENC_CTAS) and len(set(enc)) == len(enc)
    assert dec == list(autotune.DEC_CTAS) and len(set(dec)) == len(dec)
    assert lib.qlc_test_encode_ctas(None) == max(enc) and lib.qlc_test_decode_warps(None) == max(dec)
    assert lib.qlc_test_encode_ctas(ctypes.byref(Launch(0, 0, 0))) == max(enc)
    assert lib.qlc_test_decode_warps(ctypes.byref(Launch(9, 65535, 0))) == max(dec)
