"""The forward with a uint8 output alone: it has kernel instances of its own for
uint8 images (walker modes per band count, 192-thread CTAs for 8 bands, no float
stores for fewer).

Each band count on every row layout (4-pixel rows, rows shifted by 2 pixels,
pixel pairs on planes off the vector grid), strips at the image edges and
inside, fewer and more items than the launch has warps.  The product equals the
uint8 plane of the call with both outputs bit for bit: paired and scalar FP32
round alike and the order of operations is the same.  It is checked against the
FP64 oracle with the bars of test_fuse_gpu.py.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1803_00737_gb300 import _C, fuse
from test_fuse_gpu import check
from test_fuse_strips_gpu import _scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wav", [O.HAAR, O.D4])
@pytest.mark.parametrize("bands", range(1, 9))
@pytest.mark.parametrize("W,offset", [(130, 0), (388, 0), (390, 0), (388, 2), (390, 2)])
def test_u8_alone(wav, bands, W, offset):
    pan, ms, p, m = _scene(22, W, bands, np.uint8, 7 * W + bands, offset)
    f, u = fuse(p, m, wav, f32=True, u8=True)
    _, only = fuse(p, m, wav, f32=False, u8=True)
    torch.cuda.synchronize()
    assert torch.equal(only, u)
    check(pan, ms, wav, f.cpu().numpy(), only.cpu().numpy())


@pytest.mark.parametrize("bands", [3, 8])
@pytest.mark.parametrize("W", [2052, 2054])
def test_u8_alone_more_items_than_warps(bands, W):
    _, _, p, m = _scene(2200, W, bands, np.uint8, W + bands, 0)
    _, u = fuse(p, m, O.D4, f32=True, u8=True)
    only = torch.zeros_like(u)
    _C.dwtfuse_set_rows_per_item(1)
    try:
        _C.dwtfuse_fuse(p, m, O.D4, None, only)
    finally:
        _C.dwtfuse_set_rows_per_item(0)
    torch.cuda.synchronize()
    assert torch.equal(only, u)
