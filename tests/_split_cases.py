"""Inputs for the split decoder: sizes around its pieces, spans and groups at
every kind of chunk size, and data whose readers are slow to find the codeword
boundaries (runs, two-symbol patterns, schemes of one parity)."""
import numpy as np

import oracle
from paper_2602_17849_gb300 import inputs

# a complete 3-bit-suffix-and-up scheme with 3-bit codewords (area widths 0, 0, 1, 2, ...) and the raw last area
SHORT = (np.array([1, 1, 2, 4, 8, 16, 32, 192], np.uint16), np.array([0, 0, 1, 2, 3, 4, 5, 8], np.uint8))
CHUNKS = (128, 256, 384, 1024, 1280, 2176, 2048, 3968, 4096)


def data(kind, n, seed):
    rng = np.random.default_rng(seed)
    if kind == "runs":          # long runs of one symbol between random stretches
        x = inputs.make_e4m3("t4", n, seed=seed).numpy().copy()
        i = 0
        while i < n:
            i += int(rng.integers(1, 3000))
            m = int(rng.integers(1, 5000))
            x[i:i + m] = x[i % n]
            i += m
        return x
    if kind == "sparse":        # nearly constant
        x = np.full(n, 7, np.uint8)
        at = rng.integers(0, n, max(1, n // 150))
        x[at] = rng.integers(0, 256, at.size)
        return x
    if kind == "two":           # two symbols in turn
        return np.tile(np.array([200, 3], np.uint8), n // 2 + 1)[:n]
    return inputs.make_e4m3(kind, n, seed=seed).numpy()


def containers():
    """(name, symbols, container) of every case; containers are the oracle's."""
    sizes = [1, 127, 128, 129, 4095, 4096, 4097, 32 * 1024 + 1, 32 * 4096, 32 * 4096 + 777, 300_077]
    kinds = ("t4", "gauss", "ffn2", "relu_t4", "uniform_bytes", "constant", "runs", "sparse", "two")
    i = 0
    for cs in CHUNKS:
        for n in sizes:
            kind = kinds[i % len(kinds)]
            sid = 1 + (i // 2) % 2
            i += 1
            x = data(kind, n, i)
            yield f"{kind} n={n} chunk={cs} table={sid}", x, oracle.encode(x, scheme_id=sid, chunk_symbols=cs)
    shared = oracle.rank(oracle.histogram(inputs.make_e4m3("t4", 1 << 16, seed=1).numpy()))[0]
    for kind in kinds:
        x = data(kind, 150_001, 77)
        yield f"{kind} short codes", x, oracle.encode(x, scheme_id=0, area=SHORT, chunk_symbols=4096)
        # ranked by other data: runs of codewords that are not the shortest
        for sid in (1, 2):
            yield (f"{kind} table={sid} foreign ranks", x,
                   oracle.encode(x, scheme_id=sid, sym_of_rank=shared, chunk_symbols=4096))
