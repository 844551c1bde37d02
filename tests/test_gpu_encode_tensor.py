"""qlc_encode_tensor against the three calls it stands for: the same histogram,
LUT, container and sizes (bytes: no tolerance) in every way it is launched,
also captured in a CUDA graph and on several streams, and the same refusals."""
import pytest
import torch

from paper_2602_17849_gb300 import inputs
from tests import _split_cases as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qlc():
    from paper_2602_17849_gb300 import _build
    _build.build()
    from paper_2602_17849_gb300 import qlc as q
    return q


def _separate(qlc, x, scheme, cs):
    c = qlc.Codec(max(x.numel(), 1), cs, scheme)
    out = torch.full((c.cap,), 0x5A, dtype=torch.uint8, device="cuda")
    qlc.qlc_histogram(x, c.hist, n=x.numel())
    if isinstance(scheme, list):
        qlc.qlc_build_lut_best(c.hist, scheme, c.lut)
    else:
        qlc.qlc_build_lut(c.hist, scheme, c.lut)
    qlc.qlc_encode(x, c.lut, cs, out, c.ws, c.out_bytes, c.status, n=x.numel())
    torch.cuda.synchronize()
    c.check()
    return c, out


# one CTA for up to 16 chunks; one histogram CTA and several; parts and look-back; no symbols at all
@pytest.mark.parametrize("n,cs", [(0, 4096), (1, 128), (15, 4096), (127, 128), (129, 128), (4096, 4096), (4097, 4096),
                                  (16 * 128 - 1, 128), (16 * 128, 128), (16 * 128 + 1, 128), (15 * 640 + 3, 640),
                                  (16 * 1024 - 1023, 1024), (16 * 4096 - 17, 4096), (16 * 4096, 4096),
                                  (16 * 4096 + 1, 4096), (32 * 4096, 4096), (4096 * 128, 128), (4096 * 128 + 1, 128), (65536, 1024), (65537, 4096), (300_077, 1024),
                                  (16384 * 128, 128), (16384 * 128 + 1, 128), (5_000_011, 256)])
@pytest.mark.parametrize("scheme", [1, [1, 2], [2]])
def test_equals_the_three_calls(qlc, n, cs, scheme):
    x = inputs.make_e4m3("ffn2", n, seed=n).cuda() if n else torch.zeros(16, dtype=torch.uint8, device="cuda")[:0]
    want, want_out = _separate(qlc, x, scheme, cs)
    c = qlc.Codec(max(n, 1), cs, scheme)
    out = torch.full((c.cap,), 0x5A, dtype=torch.uint8, device="cuda")
    c.hist.fill_(9)
    c.encode_into(x, out)
    torch.cuda.synchronize()
    c.check()
    assert torch.equal(c.hist, want.hist) and torch.equal(c.lut, want.lut)
    assert torch.equal(c.out_bytes, want.out_bytes) and torch.equal(out, want_out)


@pytest.mark.parametrize("kind", ["uniform_bytes", "constant", "two"])
def test_one_cta_of_other_bytes(qlc, kind):
    """Counts with many ties, one symbol alone and two, against the three calls."""
    for n, cs in ((777, 128), (16 * 512 - 5, 512), (60_003, 4096)):
        x = torch.from_numpy(S.data(kind, n, n)).cuda()
        for scheme in (1, [1, 2]):
            want, want_out = _separate(qlc, x, scheme, cs)
            c = qlc.Codec(n, cs, scheme)
            out = torch.full((c.cap,), 0x5A, dtype=torch.uint8, device="cuda")
            c.encode_into(x, out)
            torch.cuda.synchronize()
            c.check()
            assert torch.equal(c.hist, want.hist) and torch.equal(c.lut, want.lut), (n, scheme)
            assert torch.equal(c.out_bytes, want.out_bytes) and torch.equal(out, want_out), (n, scheme)


@pytest.mark.parametrize("n,cs", [(9_000, 1024), (40_000, 1024), (700_001, 4096), (3 << 20, 128)])
def test_captured_in_a_graph(qlc, n, cs):
    c = qlc.Codec(n, cs, [1, 2])
    out = c.new_container()
    x = inputs.make_e4m3("t4", n, seed=1, device="cuda")
    y = torch.zeros_like(x)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        c.encode_into(x, out)
    torch.cuda.current_stream().wait_stream(s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        c.encode_into(x, out)
        c.decode_into(out, y)
    for seed, kind in ((5, "gauss"), (6, "relu_t4"), (7, "uniform_bytes")):
        x.copy_(inputs.make_e4m3(kind, n, seed=seed, device="cuda"))
        out.fill_(0x5A)
        y.zero_()
        g.replay()
        torch.cuda.synchronize()
        c.check()
        want, want_out = _separate(qlc, x, [1, 2], cs)
        nb = int(want.out_bytes.item())
        assert int(c.out_bytes.item()) == nb and torch.equal(out[:nb], want_out[:nb])
        assert torch.equal(x, y)


def test_several_streams(qlc):
    n = 900_001
    streams = [torch.cuda.Stream() for _ in range(4)]
    xs = [inputs.make_e4m3("laplace", n, seed=i, device="cuda") for i in range(4)]
    cs = [qlc.Codec(n) for _ in xs]
    outs = [c.new_container() for c in cs]
    ys = [torch.zeros_like(x) for x in xs]
    torch.cuda.synchronize()
    for _ in range(5):
        for s, x, c, o, y in zip(streams, xs, cs, outs, ys):
            c.encode_into(x, o, stream=s)
            c.decode_into(o, y, stream=s)
    torch.cuda.synchronize()
    for x, c, y in zip(xs, cs, ys):
        c.check()
        assert torch.equal(x, y)


def test_refusals(qlc):
    x = torch.zeros(5000, dtype=torch.uint8, device="cuda")
    c = qlc.Codec(5000, 1024)
    out = c.new_container()

    def call(**kw):
        a = dict(d_in=x, schemes=1, chunk_symbols=1024, d_hist=c.hist, d_lut=c.lut, d_out=out, d_ws=c.ws,
                 d_out_bytes=c.out_bytes, d_status=c.status)
        a.update(kw)
        qlc.qlc_encode_tensor(**a)

    call()
    bad = qlc.make_scheme([8] * 8, [3] * 8)
    for kw, status in ((dict(chunk_symbols=100), qlc.ERR_ARG), (dict(d_hist=None), qlc.ERR_ARG),
                       (dict(d_lut=None), qlc.ERR_ARG), (dict(d_in=x[1:]), qlc.ERR_ARG), (dict(d_out=out[8:]), qlc.ERR_ARG),
                       (dict(schemes=bad), qlc.ERR_ARG), (dict(schemes=[]), qlc.ERR_ARG), (dict(schemes=[1] * 9), qlc.ERR_ARG),
                       (dict(d_out=out[:-16]), qlc.ERR_CAPACITY), (dict(d_ws=c.ws[:16]), qlc.ERR_CAPACITY)):
        with pytest.raises(qlc.QlcError) as e:
            call(**kw)
        assert e.value.status == status, kw
    torch.cuda.synchronize()
    c.check()


def test_oneshot_calls(qlc):
    for n, scheme in ((1, 1), (300_077, [1, 2]), (70_000, 2)):
        x = inputs.make_e4m3("t4", n, seed=n, device="cuda")
        cont = qlc.encode(x, scheme, 1024)
        want, out = _separate(qlc, x, scheme, 1024)
        assert torch.equal(cont, out[: int(want.out_bytes.item())])
        assert torch.equal(qlc.decode(cont), x)
    cont[64] = cont[65]  # dec is no permutation any more
    with pytest.raises(qlc.QlcError):
        qlc.decode(cont)
