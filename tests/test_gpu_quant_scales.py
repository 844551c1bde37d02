"""Quantisation on both sides of the smallest scale whose quotients are
computed by the corrected product (2^-80), with quotients on and next to every
rounding midpoint and zeros of both signs, against the oracle (bit for bit)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("e", [-82, -81, -80, -79, -78, 0, 60, 118])
def test_scales_around_the_line(dtype, e):
    from paper_2602_17849_gb300 import _build
    _build.build()
    from paper_2602_17849_gb300 import qlc
    rng = np.random.default_rng(e + 200)
    n = 32 * 2048 + 19
    scale = rng.uniform(1.0, 2.0, (n + 31) // 32) * 2.0 ** e
    grid = np.array([m * 2.0 ** -9 for m in range(8)] + [(1 + m / 8) * 2.0 ** k for k in range(-6, 9) for m in range(8)])
    mids = np.concatenate([grid, (grid[1:] + grid[:-1]) / 2])
    x = (rng.choice(mids, n) * rng.choice([-1.0, 1.0], n) * np.repeat(scale, 32)[:n]).astype(np.float32)
    side = rng.integers(-1, 2, n)  # on it, or the float next to it
    x = np.where(side == 0, x, np.nextafter(x, np.where(side > 0, np.float32(1e38), np.float32(-1e38)), dtype=np.float32))
    x[5::37] = np.float32(-0.0)
    x[::32] = (480.0 * scale).astype(np.float32)[: x[::32].size]  # the block's absmax
    xt = torch.from_numpy(x).to(dtype).cuda()
    xh = xt.float().cpu().numpy()
    codes = torch.empty(n, dtype=torch.uint8, device="cuda")
    scales = torch.empty((n + 31) // 32, dtype=torch.float32, device="cuda")
    hist = torch.zeros(256, dtype=torch.int64, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    qlc.qlc_quantize_e4m3(xt, codes, scales, hist, st)
    ost, oc, osc = oracle.quantize_block32(xh)
    assert int(st.item()) == ost == 0
    assert np.array_equal(scales.cpu().numpy().view(np.uint32), osc.view(np.uint32))
    assert np.array_equal(codes.cpu().numpy(), oc)
    assert torch.equal(hist, torch.bincount(codes.long(), minlength=256))


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("per_sm", [1, 4, 5, 31, 32, 33, 65])
def test_warps_per_cta(dtype, per_sm):
    """Around the numbers of warp steps where the CTAs grow and where a warp takes
    a second and third one; the histogram adds to what is there."""
    from paper_2602_17849_gb300 import _build
    _build.build()
    from paper_2602_17849_gb300 import qlc
    step = 256 if dtype == torch.float32 else 512
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (per_sm * sms * step, per_sm * sms * step + 1, per_sm * sms * step - 37):
        x = torch.randn(n, generator=torch.Generator().manual_seed(n)).to(dtype)
        xd = x.cuda()
        codes = torch.empty(n, dtype=torch.uint8, device="cuda")
        scales = torch.empty((n + 31) // 32, dtype=torch.float32, device="cuda")
        hist = torch.ones(256, dtype=torch.int64, device="cuda")
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        qlc.qlc_quantize_e4m3(xd, codes, scales, hist, st, accumulate=True)
        ost, oc, osc = oracle.quantize_block32(x.float().numpy())
        assert int(st.item()) == ost == 0
        assert np.array_equal(scales.cpu().numpy().view(np.uint32), osc.view(np.uint32))
        assert np.array_equal(codes.cpu().numpy(), oc)
        assert torch.equal(hist, torch.bincount(codes.long(), minlength=256) + 1)
