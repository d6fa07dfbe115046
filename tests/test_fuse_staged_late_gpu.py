"""The staged forward's aligned instances of 5 and 6 bands against the
warp-strip kernel bit for bit: both sides of the rule that stores the uint8
pixels behind the row barrier (6 bands and a uint8 output; D4 on rows on the
128-byte line grid, Haar on uint8 images), inner and edge strips, more rows
than the two slots hold.  The staged kernel takes these rows at every size."""
import pytest
import torch

from paper_1803_00737_gb300 import D4, HAAR, _C

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("wav", [HAAR, D4])
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
@pytest.mark.parametrize("bands", [5, 6])
@pytest.mark.parametrize("W", [1024, 1020, 2048 - 96, 2044])
@pytest.mark.parametrize("u8", [True, False])
def test_staged_equals_warp_strips(wav, dtype, bands, W, u8):
    H = 46
    g = torch.Generator(device=DEV).manual_seed(W + bands)
    pan = torch.randint(0, 256, (H, W), generator=g, device=DEV, dtype=torch.uint8).to(dtype)
    ms = torch.randint(0, 256, (bands, H // 2, W // 2), generator=g, device=DEV, dtype=torch.uint8).to(dtype)
    got = []
    for staging in (True, False):
        f = torch.full((bands, H, W), float("nan"), device=DEV)
        u = torch.zeros((bands, H, W), dtype=torch.uint8, device=DEV) if u8 else None
        _C.dwtfuse_set_fuse_staging(staging)
        try:
            _C.dwtfuse_fuse(pan, ms, wav, f, u)
        finally:
            _C.dwtfuse_set_fuse_staging(True)
        got.append((f, u))
    assert torch.equal(got[0][0], got[1][0])
    assert u8 is False or torch.equal(got[0][1], got[1][1])
