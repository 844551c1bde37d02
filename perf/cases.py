"""What this library is asked to do, as timed cases.

A user hands the codec e4m3 bytes (activations, weights or gradients of one
tensor, or of a batch of shards) and gets containers, or hands it containers
and gets the bytes back; or starts from fp32 / bf16 values and ends with them.
Sizes are those of the repository's own workloads: requests of 4 KiB - 64 MiB
(the server), shards of 64 KiB - 16 MiB (the 1152-shard batch), the 256 MiB
activation tensor, and the 1 Mi-symbol tensor, with ragged sizes among them.

A case: op, n (symbols) or n_shards / lo / hi / size_seed, chunk, scheme
(1 = Table 1, 2 = Table 2, 0 = the better of both), kind (the distribution),
dtype and, for batches, shared (one LUT for all shards).
"""
import math

import numpy as np
import torch

from paper_2602_17849_gb300 import inputs, qlc

KIB, MIB = 1 << 10, 1 << 20
MAX_N = 256 * MIB
# container bytes per input byte under Table 1 (measured on each distribution)
RATIO = {"t4": 0.857, "gauss": 0.828, "laplace": 0.873, "laplace_outliers": 0.908, "ffn2": 0.81, "relu_t4": 0.79,
         "mixed": 0.853}
KINDS = ("t4", "t4", "gauss", "laplace", "laplace_outliers", "ffn2", "relu_t4")
BATCH_KINDS = ("t4", "gauss", "laplace")


def _one(name, op, n, chunk=4096, scheme=1, kind="t4", dtype="e4m3"):
    return {"name": name, "op": op, "n": n, "chunk": chunk, "scheme": scheme, "kind": kind, "dtype": dtype}


def _many(name, op, n_shards, lo, hi, size_seed, chunk=4096, scheme=1, shared=False):
    return {"name": name, "op": op, "n_shards": n_shards, "lo": lo, "hi": hi, "size_seed": size_seed, "chunk": chunk,
            "scheme": scheme, "shared": shared, "kind": "mixed", "dtype": "e4m3"}


def listed():
    return [
        # the smallest request the server takes, coded and decoded with the buffers of a kept Codec
        _one("roundtrip_4KiB", "roundtrip", 4 * KIB),
        # one ordinary tensor of 1 Mi symbols through a kept Codec
        _one("roundtrip_1MiB", "roundtrip", MIB),
        # one call each of encode() and decode() on a tensor of an odd size: allocations, size read-backs and
        # checks included, the better of both tables
        _one("oneshot_odd_300077", "oneshot", 300_077, chunk=1024, scheme=0, kind="ffn2"),
        # a [16384 x 16384] activation tensor: histogram, LUT and container ...
        _one("encode_256MiB", "encode", 256 * MIB),
        # ... and back
        _one("decode_256MiB", "decode", 256 * MIB),
        # 1152 shards (18 layers x 64 devices) of activations, weights and gradients, a LUT each
        _many("batch_encode_1152", "batch_encode", 1152, 64 * KIB, 16 * MIB, 1000),
        _many("batch_decode_1152", "batch_decode", 1152, 64 * KIB, 16 * MIB, 1000),
        # what the server has in hand at one time: a few dozen requests of 4 KiB - 64 MiB
        _many("serve_encode_24", "batch_encode", 24, 4 * KIB, 64 * MIB, 3000),
        _many("serve_decode_24", "batch_decode", 24, 4 * KIB, 64 * MIB, 3001),
        # fp32 activations to a container (the histogram counted while quantising)
        _one("quantise_encode_f32_256Mi", "quantise", 256 * MIB, dtype="float32"),
        # bf16 gradients of an odd size to a container
        _one("quantise_encode_bf16_odd", "quantise", 61_234_567, kind="laplace", chunk=2048, dtype="bfloat16"),
        # a container straight back to fp32 values
        _one("decode_values_f32_256Mi", "values", 256 * MIB, dtype="float32"),
    ]


def _log_uniform(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    op = rng.choice(("roundtrip", "oneshot", "encode", "decode", "batch_encode", "batch_decode", "quantise", "values"))
    chunk = rng.choice((1024, 2048, 4096, 4096))
    scheme = rng.choice((1, 1, 2, 0))
    if op.startswith("batch"):
        lo, hi = rng.choice(((4 * KIB, 64 * MIB), (64 * KIB, 16 * MIB), (4 * KIB, 1 * MIB)))
        mean = (hi - lo) / math.log(hi / lo)
        n_shards = _log_uniform(rng, 4, max(8, min(1152, int(2 ** 31 / mean))))
        c = _many("", op, n_shards, lo, hi, rng.randrange(1 << 30), chunk, scheme, rng.random() < 0.3)
    else:
        n = _log_uniform(rng, 4 * KIB, MAX_N if op != "oneshot" else 64 * MIB)
        if rng.random() < 0.3:
            n = max(4 * KIB, n // 4096 * 4096)
        dtype = rng.choice(("float32", "bfloat16")) if op in ("quantise", "values") else "e4m3"
        c = _one("", op, n, chunk, scheme, rng.choice(KINDS), dtype)
    del c["name"]
    return c


def _schemes(case):
    return [1, 2] if case["scheme"] == 0 else case["scheme"]


def _sizes(case):
    """Shard sizes, log-uniform in [lo, hi]; multiples of 16 (a server's requests) or of 128."""
    r = np.random.Generator(np.random.PCG64(case["size_seed"]))
    v = np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), case["n_shards"]))
    step = 16 if case["hi"] > 16 * MIB else 128
    return [max(step, int(x) // step * step) for x in v]


def _shards(case, seed):
    """The shards as views of one pool per distribution (kinds cycle activations, weights, gradients)."""
    sizes = _sizes(case)
    starts, total = [], [0, 0, 0]
    for i, n in enumerate(sizes):
        starts.append(total[i % 3])
        total[i % 3] += (n + 31) // 32 * 32
    pools = [inputs.make_e4m3(k, max(t, 32), seed=3 * seed + j, device="cuda")
             for j, (k, t) in enumerate(zip(BATCH_KINDS, total))]
    return [pools[i % 3][s:s + n] for i, (s, n) in enumerate(zip(starts, sizes))]


def _codec(case):
    c = qlc.Codec(case["n"], case["chunk"], _schemes(case))
    return c, torch.zeros(c.cap, dtype=torch.uint8, device="cuda")


def _values(case, seed):
    x = inputs.make_f32(case["kind"], case["n"], seed=seed, device="cuda")
    return x.to(getattr(torch, case["dtype"]))


def _block_scales(x):
    """absmax / 480 of every block of 32 (the last may be shorter)."""
    a = x.float().abs()
    pad = (-a.numel()) % 32
    if pad:
        a = torch.cat([a, a.new_zeros(pad)])
    return a.view(-1, 32).amax(dim=1)


def prepare(case, seed):
    op = case["op"]
    if op.startswith("batch"):
        b = qlc.Batch(_shards(case, seed), case["chunk"], _schemes(case), case["shared"])
        b.containers.zero_()
        b.decoded.zero_()
        if op == "batch_decode":
            b.encode()
        return {"op": op, "batch": b}
    codec, cont = _codec(case)
    st = {"op": op, "codec": codec, "cont": cont, "case": case}
    if op in ("roundtrip", "oneshot", "encode", "decode"):
        st["x"] = inputs.make_e4m3(case["kind"], case["n"], seed=seed, device="cuda")
        st["y"] = torch.zeros(case["n"], dtype=torch.uint8, device="cuda")
        if op == "decode":
            codec.encode_into(st["x"], cont)
            codec.check()
            st["cont"] = cont[:int(codec.out_bytes.item())].clone()
            st["x"] = None
        return st
    x = _values(case, seed)
    n_scales = (case["n"] + 31) // 32
    if op == "quantise":
        st["x"] = x
        st["codes"] = torch.zeros(case["n"], dtype=torch.uint8, device="cuda")
        st["scales"] = torch.zeros(n_scales, dtype=torch.float32, device="cuda")
        return st
    # values: a container and the block scales, as the sender wrote them
    codes = inputs.quantize_block32(x)
    codec.encode_into(codes, cont)
    codec.check()
    st["cont"] = cont[:int(codec.out_bytes.item())].clone()
    st["scales"] = _block_scales(x) / 480.0
    st["values"] = torch.zeros(case["n"], dtype=x.dtype, device="cuda")
    return st


def run(state):
    op = state["op"]
    if op == "batch_encode":
        b = state["batch"]
        b.encode()
        return {"containers": b.containers, "bytes": b.c_bytes, "luts": b.luts, "status": b.status}
    if op == "batch_decode":
        b = state["batch"]
        b.decode()
        return {"symbols": b.decoded, "n": b.n_out, "status": b.status}
    codec, cont = state["codec"], state["cont"]
    if op == "encode":
        codec.encode_into(state["x"], cont)
        return {"container": cont, "bytes": codec.out_bytes, "lut": codec.lut, "hist": codec.hist,
                "status": codec.status}
    if op == "decode":
        codec.decode_into(cont, state["y"])
        return {"symbols": state["y"], "n": codec.n_out, "status": codec.status}
    if op == "roundtrip":
        codec.encode_into(state["x"], cont)
        codec.decode_into(cont, state["y"])
        return {"container": cont, "bytes": codec.out_bytes, "symbols": state["y"], "n": codec.n_out,
                "status": codec.status}
    if op == "oneshot":
        c = state["case"]
        container = qlc.encode(state["x"], _schemes(c), c["chunk"])
        cont[:container.numel()].copy_(container)  # a container's size varies with the data: it goes into a kept slot
        return {"container": cont, "symbols": qlc.decode(container)}
    if op == "quantise":
        qlc.qlc_quantize_e4m3(state["x"], state["codes"], state["scales"], codec.hist, codec.status)
        if isinstance(codec.scheme, list):
            qlc.qlc_build_lut_best(codec.hist, codec.scheme, codec.lut)
        else:
            qlc.qlc_build_lut(codec.hist, codec.scheme, codec.lut)
        codec.encode_into(state["codes"], cont, build_lut=False)
        return {"codes": state["codes"], "scales": state["scales"], "container": cont, "bytes": codec.out_bytes,
                "status": codec.status}
    qlc.qlc_decode_dequantize(cont, state["scales"], state["values"], codec.n_out, codec.status)
    return {"values": state["values"], "n": codec.n_out, "status": codec.status}


def work(case):
    """Bytes in and out of one pass; the path is integer bit work and counts no flops."""
    op, r = case["op"], RATIO[case["kind"]]
    n = sum(_sizes(case)) if op.startswith("batch") else case["n"]
    elem = {"e4m3": 1, "float32": 4, "bfloat16": 2}[case["dtype"]]
    if op in ("roundtrip", "oneshot"):
        b = 2 * (1 + r) * n
    elif op == "quantise":
        b = (elem + 1 + 1 / 8 + r) * n
    elif op == "values":
        b = (r + 1 / 8 + elem) * n
    else:
        b = (1 + r) * n
    return {"bytes": int(b), "flops": 0}


def _e4m3_values():
    v = torch.arange(128, dtype=torch.float64)
    e, m = torch.floor(v / 8), v % 8
    mag = torch.where(e == 0, m * 2.0 ** -9, (1 + m / 8) * torch.pow(torch.tensor(2.0, dtype=torch.float64), e - 7))
    return torch.cat([mag, -mag]).cuda()


def exact(case, seed):
    """Block scales and decoded values in 64 bits; everything else is bytes and counts."""
    if case["op"] == "quantise":
        s = _block_scales(_values(case, seed)).double() / 480.0
        return {"codes": None, "scales": s, "container": None, "bytes": None, "status": None}
    if case["op"] == "values":
        x = _values(case, seed)
        codes, scales = inputs.quantize_block32(x), (_block_scales(x) / 480.0).double()
        del x
        v = _e4m3_values()[codes.long()]
        v *= scales.repeat_interleave(32)[:case["n"]]
        return {"values": v, "n": None, "status": None}
    return None
