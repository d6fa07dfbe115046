"""Row staging of the 8-bit metric passes: planes off the 16-byte grid, whose
first and last rows reach chunks outside the plane (clipped) and whose inner
rows do not, several items per warp and fewer items than warps (more ring
slots per warp), against the FP64 oracle.

Bars as in test_metrics_gpu.py: exact integer sums, one FP32 ratio per window
(2e-6 on QNR, D_lambda, D_s), ERGAS to 1e-12 (its sums are exact integers); the
fixed-point sums of Q add at most 2^-41 per window.
"""
import pytest
import torch

import scenegen
from paper_1803_00737_gb300 import _C, fuse
from test_metrics_gpu import check, gpu_metrics, ref_metrics

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _at(t, offset):
    buf = torch.empty(t.numel() + offset, dtype=t.dtype, device=DEV)
    out = buf[offset:].view(t.shape)
    out.copy_(t)
    return out


@pytest.mark.parametrize("bands", [1, 4, 6, 8])
@pytest.mark.parametrize("H,W,offset", [(64, 64, 2), (66, 514, 14), (34 * 2, 1030, 6), (1100, 130, 0),
                                        (2050, 2070, 0), (96, 2048, 2)])
def test_metrics_of_planes_off_the_grid(bands, H, W, offset):
    ws = torch.empty(_C.dwtfuse_metrics_workspace_size(), dtype=torch.uint8, device=DEV)
    pan, ms = scenegen.make_scene(H, W, bands, seed=H + W + bands)
    pan, ms = _at(pan.to(DEV), offset), [_at(m.to(DEV), offset + 1) for m in ms]
    _, u8 = fuse(pan, ms, 1, f32=False, u8=True)
    u8 = _at(u8, offset)
    check(gpu_metrics(u8, ms, pan, ws), ref_metrics(u8, torch.stack(ms), pan), False)
