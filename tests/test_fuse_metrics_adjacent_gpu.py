"""Scoring forward on shifted rows (W = 2 mod 4), 5-7 bands: the item order at
both sides of "every warp has an item" (64 strips by 16-row items: 38 item
rows fill 152 SMs of 16 warps once), a ragged last item row, several items a
warp, and the neighbouring band counts that keep the other order.

Bars as in test_fuse_metrics_gpu.py: outputs and ERGAS equal to the separate
calls', Q sums (another summation order) within 1e-6.
"""
import pytest
import torch

import oracle as O
from paper_1803_00737_gb300 import _C
from test_fuse_metrics_gpu import agree, fused_path, scene, separate_path

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wav,B", [(O.D4, 4), (O.D4, 5), (O.D4, 6), (O.HAAR, 6), (O.D4, 7), (O.D4, 8)])
@pytest.mark.parametrize("H", [1152, 1210, 1216, 2434])
def test_item_order_of_shifted_rows(wav, B, H):
    ws = torch.empty(_C.dwtfuse_metrics_workspace_size(), dtype=torch.uint8, device="cuda")
    pan, ms = scene(H, 8190, B, seed=H + B)
    f1, u1, r1 = fused_path(pan, ms, wav, ws)
    f2, u2, r2 = separate_path(pan, ms, wav, ws)
    assert torch.equal(f1, f2) and torch.equal(u1, u2)
    agree(r1, r2)
