"""The staged forward (float rows as bulk copies) on shifted rows (W = 2 mod 4)
and on more than 6 bands, against the warp-strip kernel bit for bit: full and
ragged last strips, and the last columns' pixel pairs.  The sizes are those
where the staged kernel is taken (output over 700 MB)."""
import pytest
import torch

from paper_1803_00737_gb300 import D4, HAAR, _C

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("wav", [HAAR, D4])
@pytest.mark.parametrize("W,bands,dtype,u8", [(1022, 4, torch.uint8, True), (2046, 7, torch.uint8, False),
                                              (1922, 3, torch.float32, True), (3070, 8, torch.float32, False),
                                              (1026 * 4 - 14, 6, torch.uint8, True), (2048, 9, torch.uint8, True)])
def test_staged_equals_warp_strips(wav, W, bands, dtype, u8):
    H = 2 * (700_000_000 // (W * bands * 8)) + 2
    g = torch.Generator(device=DEV).manual_seed(W)
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
