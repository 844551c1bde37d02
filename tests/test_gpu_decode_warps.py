"""qlc_launch.decode_ctas_per_sm bounds the resident decode warps of every batch,
also of those that are decoded split or dealt out evenly, and changes no byte."""
import pytest
import torch

from paper_2602_17849_gb300 import inputs

pytestmark = pytest.mark.gpu
M = 1 << 20
GROUPS, SPLIT, EVEN = 0, 1, 2


@pytest.fixture(scope="module")
def qlc():
    from paper_2602_17849_gb300 import _build
    _build.build()
    from paper_2602_17849_gb300 import qlc as q
    return q


# 16 Mi in chunks of 4096 (131 groups and more) is decoded split by teams of four
# warps; 3 warps make no team.  60 Mi are 500 groups, 200 Mi in chunks of 2048 3240.
@pytest.mark.parametrize("total,cs,warps,way", [
    (16, 4096, 0, SPLIT), (16, 4096, 20, SPLIT), (16, 4096, 65535, SPLIT), (16, 4096, 9, SPLIT), (16, 4096, 4, SPLIT),
    (16, 4096, 3, EVEN), (16, 4096, 1, EVEN), (60, 4096, 4, EVEN), (60, 4096, 3, None), (60, 4096, 1, GROUPS),
    (200, 2048, 0, None), (200, 2048, 12, GROUPS), (200, 2048, 1, GROUPS)])
def test_way_and_bytes(qlc, total, cs, warps, way):
    sizes = [0, 77, 3 * 4096 + 1] + [total * M // 8 - 16 * i for i in range(8)]
    _, shards = inputs.make_shards(sizes, ["t4"] * len(sizes), list(range(len(sizes))), "cuda")
    b = qlc.Batch(shards, cs, launch=(0, warps))
    b.encode()
    b.decode()
    torch.cuda.synchronize()
    b.check()
    for i, x in enumerate(shards):
        assert torch.equal(b.output(i), x), i
    groups = sum(-(-n // (32 * cs)) for n in sizes) + 1  # the empty shard counts as one
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if way != SPLIT:
        bound = warps if 0 < warps < 20 else 20
        want = EVEN if groups <= bound * sms else GROUPS
        assert way in (None, want)
        way = want
    assert int(b.ws[:64].view(torch.int32)[1].item()) == way
