"""The split decoder's cases against the checked build (QLC_LIBRARY names it):
no index check may fail, on sound and on corrupt containers."""
import ctypes
import os
import sys

import numpy as np
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import oracle  # noqa: E402
from paper_2602_17849_gb300 import qlc  # noqa: E402
from tests import _split_cases as S  # noqa: E402

qlc.lib.qlc_test_check_take.restype = ctypes.c_uint32


def decode(cont, n):
    y = torch.zeros(max(n, 1), dtype=torch.uint8, device="cuda")
    n_out = torch.zeros(1, dtype=torch.int64, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    qlc.qlc_decode(torch.from_numpy(cont).cuda(), y, n_out, st, out_cap=n)
    site = int(qlc.lib.qlc_test_check_take())
    assert site == 0, f"file {site >> 16} line {site & 0xFFFF}"
    return int(st.item()), y[:n].cpu().numpy()


assert int(qlc.lib.qlc_test_check_take()) == 0
rng = np.random.default_rng(5)
cases = 0
for name, x, cont in S.containers():
    st, y = decode(cont, x.size)
    assert st == 0 and np.array_equal(x, y), name
    for pos in [int(v) for v in rng.integers(320, cont.size, 8)]:
        c = cont.copy()
        c[pos] ^= np.uint8(1 << int(rng.integers(0, 8)))
        assert decode(c, x.size)[0] == oracle.decode(c, cap=x.size)[0], (name, pos)
        cases += 1
    cases += 1
print(f"checked build: {cases} cases, no index check failed")
