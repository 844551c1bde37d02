"""The split decoder against the oracle's containers (bytes: no tolerance), its
values against the oracle's dequantisation, corrupt containers' statuses, and
the choice between it and a lane per chunk."""
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


def _decode(qlc, cont, n):
    y = torch.full((n + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    n_out = torch.zeros(1, dtype=torch.int64, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    qlc.qlc_decode(torch.from_numpy(cont).cuda(), y, n_out, st, out_cap=n)
    assert int(st.item()) == 0 and int(n_out.item()) == n
    y = y.cpu().numpy()
    assert np.all(y[n:] == 0xA5)  # nothing written past the symbols
    return y[:n]


def test_containers_of_the_oracle(qlc):
    for name, x, cont in S.containers():
        assert np.array_equal(_decode(qlc, cont, x.size), x), name


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_values(qlc, dtype):
    for i, (n, cs) in enumerate([(33, 128), (4097, 4096), (70_001, 1024), (300_013, 4096)]):
        codes = S.data(("runs", "t4")[i % 2], n, i)
        scales = np.random.default_rng(i).uniform(0.01, 3.0, (n + 31) // 32).astype(np.float32)
        cont = torch.from_numpy(oracle.encode(codes, chunk_symbols=cs)).cuda()
        y = torch.zeros(n, dtype=dtype, device="cuda")
        n_out = torch.zeros(1, dtype=torch.int64, device="cuda")
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        qlc.qlc_decode_dequantize(cont, torch.from_numpy(scales).cuda(), y, n_out, st)
        assert int(st.item()) == 0
        want = torch.from_numpy(oracle.dequantize_block32(codes, scales)).to(dtype)
        assert torch.equal(y.cpu().view(torch.int16), want.view(torch.int16)), (n, cs)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_values_on_both_sides_of_the_choice(qlc, dtype):
    """Above 33 Mi symbols groups are decoded with a lane per chunk; the last
    group, chunk and block are ragged."""
    for n in (33 << 20, (33 << 20) + 4096 * 7 + 45):
        codes = inputs.make_e4m3("t4", n, seed=1, device="cuda")
        scales = torch.rand((n + 31) // 32, device="cuda") + 0.01
        codec = qlc.Codec(n)
        cont = codec.new_container()
        codec.encode_into(codes, cont)
        y, want = torch.zeros(n, dtype=dtype, device="cuda"), torch.zeros(n, dtype=dtype, device="cuda")
        qlc.qlc_decode_dequantize(cont, scales, y, codec.n_out, codec.status)
        qlc.qlc_dequantize_e4m3(codes, scales, want)
        codec.check()
        assert torch.equal(y.view(torch.int16), want.view(torch.int16)), n


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("n", [8 << 20, (8 << 20) + 32, 400 * 32768 + 45, 540 * 32768, 700 * 32768 + 77])
def test_values_by_groups_per_sm(qlc, dtype, n):
    """Chunks of 1024: both sides of the choice, then up to 3, 4 and 5 groups per SM."""
    codes = inputs.make_e4m3("t4", n, seed=n % 97, device="cuda")
    scales = torch.rand((n + 31) // 32, device="cuda") + 0.01
    codec = qlc.Codec(n, 1024)
    cont = codec.new_container()
    codec.encode_into(codes, cont)
    y, want = torch.zeros(n, dtype=dtype, device="cuda"), torch.zeros(n, dtype=dtype, device="cuda")
    qlc.qlc_decode_dequantize(cont, scales, y, codec.n_out, codec.status)
    qlc.qlc_dequantize_e4m3(codes, scales, want)
    codec.check()
    assert torch.equal(y.view(torch.int16), want.view(torch.int16))


def test_batch_warps_that_take_several_groups(qlc):
    """4900 groups on one warp per SM: four at a time, across shards, then fewer."""
    sizes = [(1 << 16) * i + 16 * i for i in range(50)]
    xs = [inputs.make_e4m3("t4", n, seed=i, device="cuda") for i, n in enumerate(sizes)]
    assert sum(sizes) > 64 << 20
    b = qlc.Batch(xs, 512, launch=(0, 1))
    b.encode()
    b.decode()
    torch.cuda.synchronize()
    b.check()
    for i, x in enumerate(xs):
        assert torch.equal(b.output(i), x), i


def test_corrupt_payload_and_index_statuses(qlc):
    rng = np.random.default_rng(3)
    for sid, cs in ((1, 4096), (2, 1024), (1, 1280)):
        x = S.data("t4", 3 * 32 * 1024 + 999, sid)
        cont = oracle.encode(x, scheme_id=sid, chunk_symbols=cs)
        for pos in [int(v) for v in rng.integers(320, cont.size, 60)]:
            c = cont.copy()
            c[pos] ^= np.uint8(1 << int(rng.integers(0, 8)))
            ost, oy, _ = oracle.decode(c, cap=x.size)
            y = torch.zeros(x.size, dtype=torch.uint8, device="cuda")
            n_out = torch.zeros(1, dtype=torch.int64, device="cuda")
            st = torch.zeros(1, dtype=torch.int32, device="cuda")
            qlc.qlc_decode(torch.from_numpy(c).cuda(), y, n_out, st)
            assert int(st.item()) == ost, (sid, cs, pos)
            if ost == oracle.OK:
                assert np.array_equal(y.cpu().numpy(), oy), (sid, cs, pos)


@pytest.mark.parametrize("kind,n", [("t4", 44 << 20), ("t4", (44 << 20) + 128), ("relu_t4", 44 << 20),
                                    ("relu_t4", (44 << 20) + 128)])
def test_both_sides_of_the_choice(qlc, kind, n):
    x = inputs.make_e4m3(kind, n, seed=2, device="cuda")
    codec = qlc.Codec(n)
    cont = codec.new_container()
    codec.encode_into(x, cont)
    y = torch.empty_like(x)
    codec.decode_into(cont, y)
    codec.check()
    assert torch.equal(x, y)


def test_checked_build():
    import os
    import subprocess
    import sys

    from paper_2602_17849_gb300 import _build
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, QLC_LIBRARY=_build.build(checked=True))
    r = subprocess.run([sys.executable, os.path.join(root, "tests", "_checked_split.py")], env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "no index check failed" in r.stdout


@pytest.mark.parametrize("total", [40 << 20, 70 << 20, 500 << 20])
def test_batches_decoded_in_each_of_three_ways(qlc, total):
    """Split up to 44 Mi symbols, a warp per group up to 20 per SM, and above;
    with an empty, a nearly constant and a corrupt shard among them."""
    sizes = [0, 5, 4096 * 33 + 1, 3 << 20, 40_000]
    sizes += [(total - sum(sizes)) // 4 // 16 * 16] * 4
    kinds = ["t4", "gauss", "laplace", "constant", "t4", "t4", "relu_t4", "gauss", "laplace"]
    _, shards = inputs.make_shards(sizes, kinds, list(range(len(sizes))), "cuda")
    b = qlc.Batch(shards, 4096 if total > 100 << 20 else 2048)
    b.encode()
    b.decode()
    torch.cuda.synchronize()
    b.check()
    assert b.n_out.tolist() == sizes
    for i, x in enumerate(shards):
        assert torch.equal(b.output(i), x), i
    b.container(4)[330] ^= 0x11  # its index
    b.decoded.zero_()
    b.decode()
    assert int(b.status.item()) == qlc.ERR_CORRUPT
    b.status.zero_()
    for i, x in enumerate(shards):
        if i != 4:
            assert torch.equal(b.output(i), x), i


@pytest.mark.parametrize("scheme", [1, 2, [1, 2]])
@pytest.mark.parametrize("cs,total", [(256, 6), (512, 7), (512, 9), (1024, 9), (1024, 10), (1024, 15), (1024, 18), (2048, 34)])
def test_batches_on_both_sides_of_the_choice(qlc, cs, total, scheme):
    """Mebisymbols around the sizes up to which a batch of such chunks is split."""
    m, kinds = 40, ("t4", "relu_t4", "gauss", "ffn2")
    sizes = [(total << 20) * (i + 1) // (m * (m + 1) // 2) // 16 * 16 for i in range(m)]
    xs = [inputs.make_e4m3(kinds[i % 4], n, seed=i, device="cuda") for i, n in enumerate(sizes)]
    b = qlc.Batch(xs, cs, schemes=scheme)
    b.encode()
    b.decode()
    torch.cuda.synchronize()
    b.check()
    for i, x in enumerate(xs):
        assert torch.equal(b.output(i), x), i
