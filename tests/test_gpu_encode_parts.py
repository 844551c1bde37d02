"""The encoder of tensors of few chunks (parts of eight chunks, blocks shared
between them) against the oracle: sizes around parts, groups and the line to
the look-back encoder, and a last chunk that lies within one 16-byte block
(bytes: no tolerance)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_17849_gb300 import inputs
from tests import _split_cases as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qlc():
    from paper_2602_17849_gb300 import _build
    _build.build()
    from paper_2602_17849_gb300 import qlc as q
    return q


def _check(qlc, x, cs, scheme, want):
    codec = qlc.Codec(x.size, cs, scheme)
    out = torch.full((codec.cap,), 0x5A, dtype=torch.uint8, device="cuda")
    codec.encode_into(torch.from_numpy(x).cuda(), out)
    torch.cuda.synchronize()
    codec.check()
    nb = int(codec.out_bytes.item())
    out = out.cpu().numpy()
    assert nb == want.size and np.array_equal(out[:nb], want)
    assert np.all(out[nb:] == 0x5A)  # nothing written past the container


@pytest.mark.parametrize("cs", [128, 1024, 1280, 4096])
@pytest.mark.parametrize("kind", ["t4", "uniform_bytes", "constant", "two"])
def test_part_and_group_boundaries(qlc, cs, kind):
    for chunks in (1, 7, 8, 9, 16, 24, 31, 32, 33, 40, 64, 72):
        for extra in (0, 1, 17):
            n = chunks * cs + extra
            x = S.data(kind, n, chunks + extra)
            sid = 1 + chunks % 2
            _check(qlc, x, cs, sid, oracle.encode(x, scheme_id=sid, chunk_symbols=cs))


def test_three_bit_codewords(qlc):
    """42 codewords after a part reach into its last block."""
    for cs in (128, 4096):
        x = S.data("constant", 41 * cs + 5, 1).copy()
        x[::7 * cs + 3] = 9  # shifts the later chunks' first bits
        _check(qlc, x, cs, S.SHORT, oracle.encode(x, scheme_id=0, area=S.SHORT, chunk_symbols=cs))


@pytest.mark.parametrize("chunks", [16383, 16384, 16385])
def test_line_to_the_look_back_encoder(qlc, chunks):
    n = chunks * 128 - 3
    x = inputs.make_e4m3("laplace", n, seed=chunks).numpy()
    _check(qlc, x, 128, 1, oracle.encode(x, chunk_symbols=128))


def test_refused_lut(qlc):
    codec = qlc.Codec(5000, 1024)
    codec.lut.zero_()
    x = torch.zeros(5000, dtype=torch.uint8, device="cuda")
    codec.encode_into(x, codec.new_container(), build_lut=False)
    assert int(codec.status.item()) == qlc.ERR_ARG
