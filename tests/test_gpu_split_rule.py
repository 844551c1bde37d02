"""Which containers and batches are decoded split: sizes on both sides of the
lines, taken from the rule itself, and the way that a batch's plan left in its
workspace.  Bytes and values: no tolerance."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2602_17849_gb300 import inputs

pytestmark = pytest.mark.gpu
M = 1 << 20
CODES, VALUES, BATCH = 0, 1, 2
GROUPS, SPLIT, EVEN = 0, 1, 2


@pytest.fixture(scope="module")
def qlc():
    from paper_2602_17849_gb300 import _build
    _build.build()
    from paper_2602_17849_gb300 import qlc as q
    q.lib.qlc_test_split_most.argtypes = [ctypes.c_char_p, ctypes.c_int, ctypes.c_uint32]
    q.lib.qlc_test_split_most.restype = ctypes.c_uint64
    q.lib.qlc_test_split_samples.argtypes = [ctypes.c_char_p, ctypes.c_int, ctypes.c_uint64]
    return q


def _encode(qlc, kind, n, cs, scheme):
    x = inputs.make_e4m3(kind, n, seed=n % 89, device="cuda")
    codec = qlc.Codec(n, cs, scheme)
    cont = codec.new_container()
    codec.encode_into(x, cont)
    return x, codec, cont


def _header(cont):
    return cont[:64].cpu().numpy().tobytes()


@pytest.mark.parametrize("into", [CODES, VALUES])
@pytest.mark.parametrize("kind,scheme,cs", [("t4", 1, 4096), ("ffn2", 2, 4096), ("t4", 1, 2048), ("gauss", 2, 1024),
                                            ("laplace", 1, 512), ("gauss", 1, 640)])
def test_containers_on_both_sides(qlc, kind, scheme, cs, into):
    line = qlc.lib.qlc_test_split_most(_header(_encode(qlc, kind, 1 << 18, cs, scheme)[2]), into, 0)
    assert line >= M
    for n in (line - 45, line, line + 32 * cs + 7 * cs + 45):  # the last group, chunk and block ragged
        x, codec, cont = _encode(qlc, kind, n, cs, scheme)
        assert qlc.lib.qlc_test_split_most(_header(cont), into, 0) == line
        assert not qlc.lib.qlc_test_split_samples(_header(cont), into, n)
        if into == CODES:
            y = torch.empty_like(x)
            codec.decode_into(cont, y)
            codec.check()
            assert torch.equal(x, y), n
            continue
        scales = torch.rand((n + 31) // 32, device="cuda") + 0.01
        for dtype in (torch.float32, torch.bfloat16):
            y, want = torch.zeros(n, dtype=dtype, device="cuda"), torch.zeros(n, dtype=dtype, device="cuda")
            qlc.qlc_decode_dequantize(cont, scales, y, codec.n_out, codec.status)
            qlc.qlc_dequantize_e4m3(x, scales, want)
            codec.check()
            assert torch.equal(y.view(torch.int16), want.view(torch.int16)), (n, dtype)


@pytest.mark.parametrize("n", [4 * M, 12 * M, 33 * M + 77])
def test_containers_that_samples_decide(qlc, n):
    """Sparse and half-zero data: whatever the samples say, the bytes are right."""
    for cs, scheme in ((4096, 1), (4096, 2), (1024, 1)):
        for density in (0.02, 0.1, 0.3, 0.5):
            x, codec, cont = _encode(qlc, "t4", n, cs, scheme)
            x[torch.rand(n, device="cuda", generator=torch.Generator("cuda").manual_seed(n)) > density] = 0
            codec.encode_into(x, cont)
            y = torch.empty_like(x)
            codec.decode_into(cont, y)
            codec.check()
            assert torch.equal(x, y), (cs, scheme, density)


def _decode_batch(b):
    b.decode()
    torch.cuda.synchronize()
    return int(b.ws[:64].view(torch.int32)[1].item())  # the way


@pytest.mark.parametrize("total,cs,way", [(2, 1024, SPLIT), (16, 2048, SPLIT), (30, 4096, SPLIT), (20, 2048, EVEN),
                                          (60, 4096, EVEN), (500, 4096, GROUPS)])
def test_batches_in_each_way(qlc, total, cs, way):
    """With an empty, a constant, a nearly constant and a corrupt shard."""
    sizes = [0, 5, 4096 * 33 + 1, M // 4, 40_000, M // 8 + 13]
    sizes += [(total * M - sum(sizes)) // 4 // 16 * 16] * 4
    kinds = ["t4", "gauss", "laplace", "constant", "t4", "constant", "t4", "laplace_outliers", "gauss", "laplace"]
    _, shards = inputs.make_shards(sizes, kinds, list(range(len(sizes))), "cuda")
    shards[5][::3000] = 17
    b = qlc.Batch(shards, cs)
    b.encode()
    assert _decode_batch(b) == way
    b.check()
    assert b.n_out.tolist() == sizes
    for i, x in enumerate(shards):
        assert torch.equal(b.output(i), x), i
    b.container(4)[330] ^= 0x11  # its index
    b.decoded.zero_()
    assert _decode_batch(b) == way
    assert int(b.status.item()) == qlc.ERR_CORRUPT
    b.status.zero_()
    for i, x in enumerate(shards):
        if i != 4:
            assert torch.equal(b.output(i), x), i


# lengths all even but the last area's, and not one of the paper's tables
EVEN_LENGTHS = ([2, 2, 8, 8, 32, 32, 128, 44], [1, 1, 3, 3, 5, 5, 7, 8])


@pytest.mark.parametrize("kind,total,cs,way", [("t4", 16, 4096, SPLIT), ("relu_t4", 12, 1024, EVEN), ("even", 50, 4096, EVEN),
                                               ("even", 12, 1024, EVEN), ("sparse", 16, 4096, EVEN),
                                               ("constant", 16, 4096, SPLIT), ("t4", 16, 1024, EVEN)])
def test_plan_and_decoder_agree(qlc, kind, total, cs, way):
    """A batch that its shards would not be decoded split in is dealt out evenly."""
    m = 40
    sizes = [total * M * 2 * (i + 1) // (m * (m + 1)) // 16 * 16 for i in range(m)]
    gen = torch.Generator("cuda").manual_seed(5)
    xs = []
    for i, n in enumerate(sizes):
        x = inputs.make_e4m3("t4" if kind in ("even", "sparse") else kind, n, seed=i, device="cuda")
        if kind == "sparse":
            x[torch.rand(n, device="cuda", generator=gen) > 0.02] = 0
        xs.append(x)
    scheme = qlc.make_scheme(*EVEN_LENGTHS) if kind == "even" else 1
    b = qlc.Batch(xs, cs, schemes=[scheme])
    b.encode()
    got = _decode_batch(b)
    b.check()
    for i, x in enumerate(xs):
        assert torch.equal(b.output(i), x), i
    assert got == way
    slow = int(b.ws[:64].view(torch.int32)[3].item())
    pays = [total * M <= qlc.lib.qlc_test_split_most(
        b.container(i)[:64].cpu().numpy().tobytes(), BATCH,
        slow if qlc.lib.qlc_test_split_samples(b.container(i)[:64].cpu().numpy().tobytes(), BATCH, sum(sizes)) else 0)
        for i in (0, m // 2, m - 1)]
    assert way == EVEN or all(pays)
