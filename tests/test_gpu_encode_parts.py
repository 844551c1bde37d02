"""The two encoders (parts of eight chunks for tensors of few chunks, groups with
look-back for the others) against the oracle: sizes around parts, runs, groups
and the line between the two, and a last chunk that lies within one 16-byte
block (bytes: no tolerance)."""
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


@pytest.mark.parametrize("chunks", [4095, 4096, 4097, 16383, 16384, 16385])
def test_line_to_the_look_back_encoder(qlc, chunks):
    n = chunks * 128 - 3
    x = inputs.make_e4m3("laplace", n, seed=chunks).numpy()
    _check(qlc, x, 128, 1, oracle.encode(x, chunk_symbols=128))


@pytest.mark.parametrize("cs", [128, 640, 1024, 2048])
@pytest.mark.parametrize("kind", ["t4", "uniform_bytes", "constant", "two"])
def test_runs_of_groups(qlc, cs, kind):
    """Last groups of 1, 4, 5, 31 and 32 chunks (a warp takes 4), chunks of a part
    of a step, half steps and whole ones, and last chunks of a few symbols."""
    for chunks, extra in ((4097, 0), (4100, 1), (4101, 17), (4127, 3), (4128, 0), (4128, 47)):
        n = chunks * cs + extra
        x = S.data(kind, n, chunks + extra)
        sid = 1 + chunks % 2
        _check(qlc, x, cs, sid, oracle.encode(x, scheme_id=sid, chunk_symbols=cs))


def test_three_bit_codewords_in_groups(qlc):
    for cs in (128, 512):
        x = S.data("constant", 4101 * cs + 5, 1).copy()
        x[::7 * cs + 3] = 9
        _check(qlc, x, cs, S.SHORT, oracle.encode(x, scheme_id=0, area=S.SHORT, chunk_symbols=cs))


@pytest.mark.parametrize("cs", [128, 2048])
def test_shards_with_their_own_tables(qlc, cs):
    """Teams change tables from group to group, beside one another: 700 tensors of
    one to three groups, each with its own LUT, and empty ones."""
    rng = np.random.default_rng(cs)
    sizes = [0 if i % 97 == 5 else int(rng.integers(1, 3 * 32 * cs)) for i in range(700 if cs == 128 else 120)]
    xs = [S.data("uniform_bytes" if i % 3 else "two", n, i) for i, n in enumerate(sizes)]
    b = qlc.Batch([torch.from_numpy(x).cuda() for x in xs], cs)
    b.encode()
    torch.cuda.synchronize()
    b.check()
    for i, x in enumerate(xs):
        got = b.container(i)[:int(b.c_bytes[i])].cpu().numpy()
        assert np.array_equal(got, oracle.encode(x, scheme_id=1, chunk_symbols=cs)), i


def test_refused_lut(qlc):
    codec = qlc.Codec(5000, 1024)
    codec.lut.zero_()
    x = torch.zeros(5000, dtype=torch.uint8, device="cuda")
    codec.encode_into(x, codec.new_container(), build_lut=False)
    assert int(codec.status.item()) == qlc.ERR_ARG
