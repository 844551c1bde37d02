"""Streams whose readers do not resynchronise: runs of one symbol that begin and
end anywhere in a chunk, under codewords of every length, patterns of several
symbols, sparse data, and more short codewords in a piece than it has room for.
Run as a script it decodes them, sound and corrupt, with the library that
QLC_LIBRARY names (the checked build): no index check may fail."""
import ctypes
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import oracle  # noqa: E402
from paper_2602_17849_gb300 import inputs  # noqa: E402

# all lengths but the last area's even, and 3-bit codewords
EVEN = (np.array([2, 2, 8, 8, 32, 32, 128, 44], np.uint16), np.array([1, 1, 3, 3, 5, 5, 7, 8], np.uint8))
SHORT = (np.array([1, 1, 2, 4, 8, 16, 32, 192], np.uint16), np.array([0, 0, 1, 2, 3, 4, 5, 8], np.uint8))


def data(kind, n, cs, seed):
    rng = np.random.default_rng(seed)
    x = inputs.make_e4m3("t4", n, seed=seed).numpy().copy()
    for c in range(0, n, cs):
        m = min(cs, n - c)
        if kind == "run":            # one run, its ends and symbol anywhere
            a, b = sorted(int(v) for v in rng.integers(0, m + 1, 2))
            x[c + a:c + b] = rng.integers(0, 256)
        elif kind == "runs":         # several runs that follow one another
            a = 0
            while a < m:
                b = min(m, a + int(rng.integers(1, 700)))
                if rng.random() < 0.7:
                    x[c + a:c + b] = rng.integers(0, 256)
                a = b
        elif kind == "pattern":      # symbols in turn
            p = rng.integers(0, 256, int(rng.integers(2, 9)), dtype=np.uint8)
            x[c + m // 3:c + m] = np.resize(p, m - m // 3)
        elif kind == "sparse":
            x[c:c + m][rng.random(m) > 0.03] = 0
        elif kind == "one":          # all of the chunk
            x[c:c + m] = rng.integers(0, 256)
    return x


def containers():
    """(name, symbols, container); containers are the oracle's."""
    i = 0
    for cs in (512, 1024, 1152, 2176, 4096):
        for kind in ("run", "runs", "pattern", "sparse", "one"):
            for scheme in (1, 2, EVEN, SHORT):
                i += 1
                n = (33 * cs + 5, 3 * cs + 127, 40 * cs)[i % 3]
                x = data(kind, n, cs, i)
                kw = dict(scheme_id=scheme) if isinstance(scheme, int) else dict(scheme_id=0, area=scheme)
                if i % 2:  # ranks of other data: the run's codeword may have any length
                    other = inputs.make_e4m3("t4", 1 << 14, seed=i).numpy()
                    kw["sym_of_rank"] = oracle.rank(oracle.histogram(other))[0]
                yield f"{kind} n={n} chunk={cs} scheme {i % 4}", x, oracle.encode(x, chunk_symbols=cs, **kw)


def main():
    import torch

    from paper_2602_17849_gb300 import qlc
    qlc.lib.qlc_test_check_take.restype = ctypes.c_uint32

    def decode(cont, n):
        y = torch.zeros(n, dtype=torch.uint8, device="cuda")
        words = torch.zeros(2, dtype=torch.int64, device="cuda")
        qlc.qlc_decode(torch.from_numpy(cont).cuda(), y, words[:1], words[1:].view(torch.int32)[:1])
        site = int(qlc.lib.qlc_test_check_take())
        assert site == 0, f"file {site >> 16} line {site & 0xFFFF}"
        return int(words[1].item()), y.cpu().numpy()

    assert int(qlc.lib.qlc_test_check_take()) == 0
    rng = np.random.default_rng(5)
    cases = 0
    for name, x, cont in containers():
        st, y = decode(cont, x.size)
        assert st == 0 and np.array_equal(x, y), name
        for pos in [int(v) for v in rng.integers(320, cont.size, 6)]:
            c = cont.copy()
            c[pos] ^= np.uint8(1 << int(rng.integers(0, 8)))
            st, y = decode(c, x.size)
            ost, oy, _ = oracle.decode(c, cap=x.size)
            assert st == ost and (ost != 0 or np.array_equal(y, oy)), (name, pos)
            cases += 1
        cases += 1
    print(f"checked build: {cases} cases, no index check failed")


if __name__ == "__main__":
    main()
