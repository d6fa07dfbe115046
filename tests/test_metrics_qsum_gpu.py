"""Sums of Q over windows are exact: more windows than 40 fractional bits of an
int64 leave room for (2^23), and Q values of a window far below 2^-40.

Bars: Q = 1 in every window sums and divides exactly, so the figures of a
constant scene are exact.  A single Q is one FP32 expression of nine roundings
over exact integers: 9 * 2^-24 < 1e-6 relative, and the mean of equal Qs keeps it.
"""
import pytest
import torch

from paper_1803_00737_gb300 import HAAR, _C

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("call", ["metrics", "fuse_metrics"])
def test_more_windows_than_2_to_23(call):
    side = 92704  # 2897^2 = 8,392,609 windows
    pan = torch.full((side, side), 7, dtype=torch.uint8, device=DEV)
    ms = torch.full((1, side // 2, side // 2), 7, dtype=torch.uint8, device=DEV)
    ws = torch.zeros(_C.dwtfuse_metrics_workspace_size(), dtype=torch.uint8, device=DEV)
    res = torch.zeros(4, dtype=torch.float64, device=DEV)
    if call == "metrics":
        _C.dwtfuse_metrics(pan[None], ms, pan, ws, res)
    else:
        out = torch.zeros((1, side, side), dtype=torch.uint8, device=DEV)
        _C.dwtfuse_fuse_metrics(pan, ms, HAAR, None, out, ws, res)
    assert res.tolist() == [0.0, 1.0, 0.0, 0.0]


@pytest.mark.parametrize("bands", range(2, 9))
@pytest.mark.parametrize("W", [160, 162])
def test_q_far_below_2_to_minus_40(bands, W):
    H = 128
    # x: half 0, half 255 but for three pixels, so that its covariance with y (one pixel of 1) is -1 / n^2.
    x = torch.zeros(1024, dtype=torch.int64)
    x[512:] = 255
    x[512], x[513], x[514] = 127, 0, 127
    y = torch.zeros(1024, dtype=torch.int64)
    y[512] = 1
    n, sx, sy = 1024, int(x.sum()), 1
    cov, vx, vy = n * int((x * y).sum()) - sx * sy, n * int((x * x).sum()) - sx * sx, n - 1
    assert cov == -1
    q = 4 * cov * sx * sy / ((vx + vy) * (sx * sx + sy * sy))
    assert abs(q) < 2.0 ** -48
    fused = torch.zeros((bands, H, W), dtype=torch.uint8, device=DEV)
    for b in range(bands):
        fused[b, :, :160] = (y if b else x).view(32, 32).to(torch.uint8).repeat(H // 32, 5)
    ms = torch.full((bands, H // 2, W // 2), 9, dtype=torch.uint8, device=DEV)
    ms[0] = 5  # Q(MS_0, MS_b) = 0, every other pair 1, as in the product
    pan = torch.full((H, W), 3, dtype=torch.uint8, device=DEV)
    ws = torch.zeros(_C.dwtfuse_metrics_workspace_size(), dtype=torch.uint8, device=DEV)
    res = torch.zeros(4, dtype=torch.float64, device=DEV)
    _C.dwtfuse_metrics(fused, ms, pan, ws, res)
    want = 2.0 * abs(q) / bands
    assert abs(res[2].item() - want) <= 1e-6 * want
