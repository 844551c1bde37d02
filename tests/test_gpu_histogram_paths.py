"""The histogram kernels where their work is split: one CTA writing the counts
itself against several adding to a cleared array, and batches around the 1024
shards a CTA scans at a time (counts are whole numbers: no tolerance)."""
import numpy as np
import pytest
import torch

from paper_2602_17849_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qlc():
    from paper_2602_17849_gb300 import _build
    _build.build()
    from paper_2602_17849_gb300 import qlc as q
    return q


@pytest.mark.parametrize("n", [1, 15, 16, 65535, 65536, 65551, 65552, 131072 + 5])
@pytest.mark.parametrize("accumulate", [False, True])
def test_one_and_several_ctas(qlc, n, accumulate):
    x = inputs.make_e4m3("t4", n, seed=n).cuda()
    h = torch.full((256,), 7, dtype=torch.int64, device="cuda")
    qlc.qlc_histogram(x, h, accumulate=accumulate)
    want = torch.bincount(x.long(), minlength=256) + (7 if accumulate else 0)
    assert torch.equal(h, want)


@pytest.mark.parametrize("n_shards", [1, 31, 1023, 1024, 1025, 2500])
@pytest.mark.parametrize("shared", [False, True])
def test_batches_around_a_scan(qlc, n_shards, shared):
    rng = np.random.default_rng(n_shards)
    sizes = [int(v) for v in rng.choice([0, 0, 1, 16, 17, 5000, 65536, 65537], n_shards)]
    sizes[-1] = 200_003
    pool = inputs.make_e4m3("laplace", sum((s + 15) // 16 * 16 for s in sizes), seed=5, device="cuda")
    views, off = [], 0
    for s in sizes:
        views.append(pool[off:off + s])
        off += (s + 15) // 16 * 16
    b = qlc.Batch(views, 1024, shared_lut=shared)
    b.hists.fill_(3)
    qlc.qlc_histogram_batch(b.enc_descs, b.n, b.hists, b.shared, b.ws)
    per = torch.stack([torch.bincount(v.long(), minlength=256) for v in views])
    want = per.sum(0) if shared else per.reshape(-1)
    assert torch.equal(b.hists, want)
