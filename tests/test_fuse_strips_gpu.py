"""The row walkers' instances: strips at the image edges (wrapped columns)
against strips inside, the three row layouts (4-pixel rows, rows shifted by 2
pixels, pixel pairs on planes off the vector grid), both input types, and a
batch table that mixes all of them.

Bars as in test_fuse_gpu.py: Haar exact on integer inputs, D4 within 5e-4 of
the FP64 oracle on the 0-255 scale (FP32 sums of 20 products of values below
2^10: 20 * 2^-24 * 2^10 ~ 1.2e-3 worst case, a quarter of it reached), uint8
off by one only within 5e-4 of a rounding boundary.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1803_00737_gb300 import _C, fuse
from test_fuse_gpu import check

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _plane(a, offset):
    """The array on the GPU, `offset` elements past a 256-byte boundary."""
    buf = torch.zeros(a.size + offset, dtype=torch.uint8 if a.dtype == np.uint8 else torch.float32, device=DEV)
    out = buf[offset:].view(a.shape)
    out.copy_(torch.from_numpy(a))
    return out


def _scene(H, W, B, dtype, seed, offset):
    rng = np.random.default_rng(seed)
    pan = rng.integers(0, 256, (H, W)).astype(dtype)
    ms = rng.integers(0, 256, (B, H // 2, W // 2)).astype(dtype)
    return pan, ms, _plane(pan, offset), [_plane(m, offset // 2) for m in ms]


@pytest.mark.parametrize("wav", [O.HAAR, O.D4])
@pytest.mark.parametrize("dtype,bands", [(np.uint8, 3), (np.uint8, 8), (np.float32, 4)])
@pytest.mark.parametrize("W", [128, 130, 256, 258, 260, 384, 386, 390, 516])
@pytest.mark.parametrize("offset", [0, 2])
def test_strips(wav, dtype, bands, W, offset):
    pan, ms, p, m = _scene(22, W, bands, dtype, W + bands, offset)
    f, u = fuse(p, m, wav, f32=True, u8=True)
    torch.cuda.synchronize()
    check(pan, ms, wav, f.cpu().numpy(), u.cpu().numpy())


def test_batch_of_all_bodies_equals_single_scenes():
    """Types, widths of 1-4 and 5-8 bands, wavelets and layouts in one table."""
    table, keep = [], []
    for i in range(48):
        wav, dtype = (O.HAAR, O.D4)[i % 2], (np.uint8, np.float32)[(i // 2) % 2]
        B, W = 1 + (i * 5) % 8, (260, 386, 512)[i % 3]
        _, _, p, m = _scene(18 + 2 * (i % 5), W, B, dtype, i, 2 * (i % 4 == 3))
        f = torch.full((B, *p.shape), float("nan"), device=DEV)
        u = torch.zeros((B, *p.shape), dtype=torch.uint8, device=DEV)
        table.append(_C.make_scene(p, m, wav, f, u))
        keep.append((wav, p, m, f, u))
    ws = torch.zeros(_C.dwtfuse_batched_workspace_size(), dtype=torch.uint8, device=DEV)
    _C.dwtfuse_fuse_batched(table, ws)
    torch.cuda.synchronize()
    assert _C.dwtfuse_get_last_device_status(ws) == _C.OK
    for wav, p, m, f, u in keep:
        ef, eu = fuse(p, m, wav, f32=True, u8=True)
        assert torch.equal(f, ef) and torch.equal(u, eu), (wav, p.shape, len(m))
