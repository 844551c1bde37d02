"""A container whose dec is no permutation of 0..255 is refused: one value twice,
at every lane's first and last place, by each of the decoders."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_17849_gb300 import inputs

pytestmark = pytest.mark.gpu
PLACES = [0, 1, 6, 7, 8, 15, 127, 128, 247, 248, 254, 255]


@pytest.fixture(scope="module")
def qlc():
    from paper_2602_17849_gb300 import _build
    _build.build()
    from paper_2602_17849_gb300 import qlc as q
    return q


@pytest.mark.parametrize("n,cs", [(50, 128), (70_001, 1024), (140_000, 4096)])
def test_one_value_twice(qlc, n, cs):
    x = inputs.make_e4m3("t4", n, seed=1).numpy()
    good = oracle.encode(x, chunk_symbols=cs)
    scales = torch.ones((n + 31) // 32, device="cuda")
    for place in PLACES:
        for other in (place ^ 1, (place + 131) % 256):
            c = good.copy()
            c[64 + place] = c[64 + other]
            assert oracle.decode(c, cap=n)[0] == oracle.ERR_CORRUPT
            d = torch.from_numpy(c).cuda()
            y, v = torch.zeros(n, dtype=torch.uint8, device="cuda"), torch.zeros(n, device="cuda")
            words = torch.full((2,), -1, dtype=torch.int64, device="cuda")
            st = torch.zeros(2, dtype=torch.int32, device="cuda")
            qlc.qlc_decode(d, y, words[:1], st[:1])
            qlc.qlc_decode_dequantize(d, scales, v, words[1:], st[1:])
            assert st.tolist() == [qlc.ERR_CORRUPT] * 2 and words.tolist() == [-1, -1], (place, other)


@pytest.mark.parametrize("warps", [0, 3, 1])
def test_shards_of_batches(qlc, warps):
    """Split, dealt out evenly and from the counter: the other shards are decoded."""
    sizes = [20 << 20, 300_001, 9 << 20]
    shards = [inputs.make_e4m3("t4", n, seed=i, device="cuda") for i, n in enumerate(sizes)]
    b = qlc.Batch(shards, 4096, launch=(0, warps))
    b.encode()
    for place in (0, 100, 255):
        c = b.container(1)
        keep = c[64 + place].clone()
        c[64 + place] = c[64 + (place + 1) % 256]
        b.decoded.zero_()
        b.decode()
        assert int(b.status.item()) == qlc.ERR_CORRUPT
        b.status.zero_()
        c[64 + place] = keep
        for i in (0, 2):
            assert torch.equal(b.output(i), shards[i]), (place, i)
    b.decode()
    b.check()
    assert torch.equal(b.output(1), shards[1])
